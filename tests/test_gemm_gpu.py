"""GPU parity of the tensor-core weight-streaming GEMM (sjd_gemm through the C-ABI) against a plain
fp64 matrix product of the same bf16 weights and fp32 activations."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2410_01699_b200 import binding as B
from tests.parity_util import run_in_threads

pytestmark = pytest.mark.gpu


def _case(m, n, k, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(m, k, generator=g, dtype=torch.float32)
    w = (torch.randn(n, k, generator=g, dtype=torch.float32) * 0.05).to(torch.bfloat16)
    ref = x.to(torch.float64).numpy() @ w.to(torch.float64).numpy().T      # the definition, fp64
    return x, w, ref


def _tolerance(x, w, k):
    # activations carry bf16 hi + lo (relative 2^-17 per element), products accumulate in fp32
    scale = float(np.sqrt(k) * x.abs().max() * w.to(torch.float32).abs().max())
    return 3e-5 * scale + 1e-6


@pytest.mark.parametrize("m,n,k", [
    (32, 128, 64),        # one tile, one k-block
    (32, 256, 4096),      # two tiles over all CTAs: every segment partial
    (32, 4096, 4096),     # the attention output projection of the 7B shape
    (32, 1024, 11008),    # long K (SwiGLU down projection), 172 k-blocks
    (17, 384, 512),       # ragged row count (padded to 32 columns of the MMA)
    (1, 128, 128),        # single row
    (64, 2048, 1024),     # W = 64
    (48, 4096, 4096),     # W = 48: three activation stages beside four of weights, K split
    (33, 19200, 640),     # the same with whole K, two CTAs on some SMs
    (128, 512, 256),      # widest supported window batch
    (32, 65536, 512),     # 512 tiles (vocabulary-sized N)
    (112, 768, 1024),     # 112 rows in one slab: accumulators of 224 columns
    (128, 22016, 4096),   # four images x W = 32 on the gate|up projection: 172 tiles on 148 SMs
    (129, 256, 512),      # first row count cut into token slabs: two of 72 rows (the second holds 57)
    (256, 1024, 1024),    # two full slabs of 128 rows
    (300, 384, 640),      # three ragged slabs of 104 rows (the last holds 92)
    (512, 4096, 4096),    # 8 images x W = 64 on the attention output projection: 4 slabs x 32 tiles x K splits
    (1024, 256, 256),     # most rows covered: eight slabs
    (65, 128, 64),            # CTA pairs: one tile (the second CTA has none), one k-block
    (130, 384, 1088),         # three tiles (an odd pair), two slabs of 72 rows, K over several splits
    (257, 19200, 256),        # more units than pairs, three slabs, few k-blocks per unit
    (72, 384, 1088),          # slabs whose rows are not a multiple of 16: one of 72,
    (200, 1024, 512),         # two of 104,
    (258, 256, 320),          # three of 88 (the last holds 82)
])
def test_gemm_matches_fp64_product(m, n, k):
    x, w, ref = _case(m, n, k, seed=m + n + k)
    out, status = B.sjd_gemm(x.cuda(), w.cuda())
    torch.cuda.synchronize()
    assert int(status.item()) == 0, "a device-side wait ran out"
    got = out.cpu().to(torch.float64).numpy()
    err = np.abs(got - ref).max()
    assert err <= _tolerance(x, w, k), f"max |err| {err:.3e}"


def test_gemm_wide_rows_do_not_mix():
    """Each token row of a many-row product depends on its own activations only: rows of a 512-row call
    equal the same rows computed in a call of their own slab size (catches a wrong slab offset)."""
    x, w, _ = _case(512, 512, 1024, seed=5)
    full, st = B.sjd_gemm(x.cuda(), w.cuda())
    part, _ = B.sjd_gemm(x[256:].contiguous().cuda(), w.cuda())
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert torch.equal(full[256:], part)


def test_gemm_accumulates_and_is_deterministic():
    x, w, ref = _case(32, 1024, 2048, seed=9)
    base = torch.full((32, 1024), 0.5, dtype=torch.float32, device="cuda")
    out, status = B.sjd_gemm(x.cuda(), w.cuda(), out=base.clone(), accumulate=True)
    out2, _ = B.sjd_gemm(x.cuda(), w.cuda(), out=base.clone(), accumulate=True)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(out, out2)
    assert np.abs(out.cpu().to(torch.float64).numpy() - (ref + 0.5)).max() <= _tolerance(x, w, 2048)


def test_gemm_rejects_uncovered_shapes():
    x = torch.zeros(8, 96, device="cuda")
    w = torch.zeros(128, 96, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(B.SJDError) as e:
        B.sjd_gemm(x, w)                      # K not a multiple of 64
    assert e.value.status == B.SJD_ERR_UNSUPPORTED
    assert B.lib().sjd_gemm_workspace_bytes(1025, 128, 64) == 0


def test_gemm_threads_with_different_sizes():
    """Threads whose launches ask for different amounts of shared memory (80 and 128 token rows: rings of eight and of seven
    stages): none lowers the limit under another's launch."""
    x, w, _ = _case(128, 256, 512, seed=3)
    x, w = x.cuda(), w.cuda()
    want = {m: B.sjd_gemm(x[:m], w)[0] for m in (80, 128)}

    def calls(m):
        out = torch.empty(m, 256, device="cuda")
        ws = torch.empty(int(B.lib().sjd_gemm_workspace_bytes(m, 256, 512)), dtype=torch.uint8, device="cuda")
        args = [m, 256, 512, *(C.c_void_p(t.data_ptr()) for t in (x, w, out)), 0, C.c_void_p(ws.data_ptr()), ws.numel(),
                C.c_void_p(torch.cuda.current_stream().cuda_stream)]
        call = B.lib().sjd_gemm
        assert all(call(*args) == B.SJD_OK for _ in range(10000))
        assert torch.equal(out, want[m])

    run_in_threads(*[lambda m=m: calls(m) for m in (80, 128, 80, 128)])
