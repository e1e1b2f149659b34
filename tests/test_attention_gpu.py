"""GPU parity of the tensor-core window attention (sjd_attention through the C-ABI) against the
definition in fp64: softmax(q k^T / sqrt(d)) v over the cache rows each query may see."""
import numpy as np
import pytest
import torch

from paper_2410_01699_b200 import binding as B

pytestmark = pytest.mark.gpu


def _reference(q, kv, pos, window, n_kv_heads):
    m, h, hd = q.shape
    group = h // n_kv_heads
    out = np.zeros((m, h, hd))
    q64, kv64 = q.double().numpy(), kv.to(torch.float64).numpy()
    for r in range(m):
        b, p = r // window, int(pos[r])
        if p < 0:
            continue
        for head in range(h):
            k = kv64[b, 0, head // group, :p + 1]
            v = kv64[b, 1, head // group, :p + 1]
            s = k @ q64[r, head] / np.sqrt(hd)
            w = np.exp(s - s.max())
            out[r, head] = (w / w.sum()) @ v
    return out


@pytest.mark.parametrize("batch,window,prefix,heads,kv_heads,hd", [
    (1, 32, 100, 32, 32, 128),    # the 7B shape early in an image
    (1, 32, 1500, 4, 4, 128),     # long prefix: many tiles per split (few heads keep the fp64 check cheap)
    (2, 64, 300, 8, 2, 128),      # grouped-query heads, W = 64, two sequences
    (3, 16, 70, 8, 2, 64),        # head_dim 64
    (1, 5, 1, 4, 4, 64),          # first step after a one-token prompt: query k sees k + 1 rows
    (1, 24, 64, 4, 1, 128),       # window not a multiple of 16, one kv head
    (5, 16, 90, 32, 8, 64),       # 160 (head, sequence) pairs: one key range each, output written without a merge
    (10, 32, 130, 32, 32, 128),   # the same at the 7B head shape, W = 32
])
def test_attention_matches_definition(batch, window, prefix, heads, kv_heads, hd):
    g = torch.Generator().manual_seed(prefix + window)
    max_seq = prefix + window + 3
    q = torch.randn(batch * window, heads, hd, generator=g)
    kv = torch.randn(batch, 2, kv_heads, max_seq, hd, generator=g).to(torch.bfloat16)
    pos = (prefix - 1 + torch.arange(window, dtype=torch.int32)).repeat(batch)
    if window > 8:
        pos[-3:] = -1                       # inactive rows (a window shortened at the end of the image)
    out, status = B.sjd_attention(q.cuda(), kv.cuda(), pos.cuda(), window, kv_heads)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = _reference(q, kv, pos, window, kv_heads)
    err = np.abs(out.cpu().double().numpy() - ref).max()
    # q and the probabilities carry bf16 hi + lo parts (2^-17 relative), accumulation in fp32
    assert err <= 2e-4, f"max |err| {err:.3e}"
    assert torch.all(out[pos.cuda() < 0] == 0)


def test_attention_rejects_uncovered_shapes():
    assert B.lib().sjd_attention_workspace_bytes(1, 32, 8, 96) == 0
    assert B.lib().sjd_attention_workspace_bytes(1, 65, 8, 128) == 0


@pytest.mark.parametrize("batch,window,keys,heads,kv_heads,hd,grow", [
    (1, 32, 128, 2, 2, 128, 0.0),     # a tile of 128 keys, full
    (2, 17, 129, 2, 1, 128, 0.0),     # one key more
    (1, 16, 65, 4, 4, 64, 0.0),       # one key in the second box of a tile
    (1, 33, 64, 2, 2, 64, 0.0),       # first window of 64 columns; a tile with one box
    (51, 3, 140, 3, 3, 64, 0.0),      # an odd number of (head, sequence) pairs with one key range each
    (20, 64, 400, 8, 2, 128, 1.0),    # scores grow along the keys past every reference: output rescaled, 64 columns, one range
    (10, 32, 700, 32, 32, 128, 1.0),  # the same with 32 columns, two output accumulators
    (1, 20, 900, 2, 2, 64, 1.0),      # and over several key ranges
])
def test_attention_tiles_and_growing_scores(batch, window, keys, heads, kv_heads, hd, grow):
    g = torch.Generator().manual_seed(keys + window)
    n = keys - window
    q = torch.randn(batch * window, heads, hd, generator=g)
    kv = torch.randn(batch, 2, kv_heads, keys + 1, hd, generator=g)
    if grow:   # key j adds grow * j / 2 to every score: sum(q * u) / sqrt(hd) = 1 for u along q's common direction
        q += 4.0
        kv[:, 0] += (grow * 0.125 / hd ** 0.5) * torch.arange(keys + 1)[:, None]
    kv = kv.to(torch.bfloat16)
    pos = (n + torch.arange(window, dtype=torch.int32)).repeat(batch)
    out, status = B.sjd_attention(q.cuda(), kv.cuda(), pos.cuda(), window, kv_heads)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    rows = torch.cat([torch.arange(window), torch.arange((batch - 1) * window, batch * window)]).unique()   # first and last sequence
    some = sorted({0, batch - 1})
    ref = _reference(q[rows], kv[some], pos[rows], window, kv_heads)
    # as above, and a score's own error: q is off by 2^-17 of each entry, and 4 * |score error| * max|v| bounds the output's
    bound = (q[rows].abs().amax(0).amax(0).double() @ kv[some][:, 0].double().abs().amax((0, 1)).T / hd ** 0.5).max().item()
    tol = 2e-4 + 4 * 2.0 ** -17 * bound * kv[some][:, 1].abs().max().item()
    err = np.abs(out.cpu()[rows].double().numpy() - ref).max()
    assert err <= tol, f"max |err| {err:.3e} (bound {tol:.3e})"


# batch, window, keys, heads, kv_heads, head_dim, ramp: scores grow by a quarter per key over `ramp` keys and start again
TILE_CASES = [
    (1, 32, 128, 2, 2, 128, 0),       # a tile of 128 keys, full
    (2, 17, 129, 2, 1, 128, 0),       # one key more
    (1, 16, 65, 4, 4, 64, 0),         # one key in the second box of a tile
    (1, 33, 64, 2, 2, 64, 0),         # first window of 64 columns; a tile with one box
    (51, 3, 140, 3, 3, 64, 0),        # an odd number of (head, sequence) pairs with one key range each
    (5, 40, 4000, 32, 8, 128, 0),     # 64 columns, one range: the longest chain of additions, in one output accumulator
    (20, 64, 400, 8, 2, 128, 400),    # scores pass every reference: output rescaled, 64 columns, one range
    (10, 32, 700, 32, 32, 128, 400),  # the same with 32 columns, two output accumulators
    (4, 20, 700, 32, 8, 64, 316),     # two ranges of three tiles, both with a peak that carries weight
    (4, 40, 700, 32, 8, 128, 316),    # the same with 64 columns
    (1, 20, 900, 2, 2, 64, 316),      # a tile per range
]


def tile_case(batch, window, keys, heads, kv_heads, hd, ramp):
    g = torch.Generator().manual_seed(keys + window)
    q = torch.randn(batch * window, heads, hd, generator=g)
    kv = torch.randn(batch, 2, kv_heads, keys + 1, hd, generator=g)
    if ramp:   # all entries of q lean the same way, and key j of a ramp leans j / 4 that way
        q += 4.0
        kv[:, 0] += (0.25 / (4.0 * hd ** 0.5)) * (torch.arange(keys + 1) % ramp)[:, None]
    pos = (keys - window + torch.arange(window, dtype=torch.int32)).repeat(batch)
    return q, kv.to(torch.bfloat16), pos


def _planes(x, lo):
    hi = x.to(torch.bfloat16).double()
    return hi + (x.double() - hi).to(torch.bfloat16).double() if lo else hi


def definition_and_bound(q, kv, pos, window, seqs, q_lo=None, p_lo=None):
    """Rows of the sequences `seqs` by the definition in fp64, [seq][head][row][hd], and the largest error that a correct kernel
    shows.  A product's operand is off by 2^-17 of itself (bf16 hi + lo), and each of its additions of 16 products in the tensor
    core by 2^-22 of the sum of magnitudes; a score that is off by d_j moves the output by w_j d_j (v_j - o) to first order.
    With q_lo or p_lo given: the output as computed from these planes (True: hi and lo, False: hi only) instead."""
    group, hd = q.shape[1] // kv.shape[2], q.shape[2]
    outs, bounds = [], []
    for b in seqs:
        rows = slice(b * window, (b + 1) * window)
        k, v = (kv[b, i].double().repeat_interleave(group, 0) for i in (0, 1))
        qh = q[rows].transpose(0, 1)
        if q_lo is None:
            s = qh.double() @ k.transpose(1, 2) / hd ** 0.5
        else:
            s = _planes(qh * (1.4426950408889634 / hd ** 0.5), q_lo) @ k.transpose(1, 2) * np.log(2.0)
        s = s.masked_fill(torch.arange(k.shape[1])[None] > pos[rows].long()[:, None], -np.inf)
        p = torch.exp(s - s.amax(-1, keepdim=True))
        total = p.sum(-1, keepdim=True)
        if q_lo is not None:
            outs.append(_planes(p.float(), p_lo) @ v / total)
            continue
        w = p / total
        o = w @ v
        wd = w * (2.0 ** -17 + hd / 16 * 2.0 ** -22) * (qh.double().abs() @ k.abs().transpose(1, 2)) / hd ** 0.5
        outs.append(o)
        bounds.append(wd @ v.abs() + wd.sum(-1, keepdim=True) * o.abs() + (2.0 ** -17 + k.shape[1] / 16 * 2.0 ** -22) * (w @ v.abs()))
    return torch.stack(outs), torch.stack(bounds) if bounds else None


@pytest.mark.parametrize("case", TILE_CASES)
def test_attention_entries_within_their_own_bounds(case):
    """(tests/test_attention_bound.py: the bound notices a lost plane of Q or of the probabilities in every one of these.)"""
    batch, window, kv_heads = case[0], case[1], case[4]
    q, kv, pos = tile_case(*case)
    out, status = B.sjd_attention(q.cuda(), kv.cuda(), pos.cuda(), window, kv_heads)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    seqs = sorted({0, batch - 1})
    ref, bound = definition_and_bound(q, kv, pos, window, seqs)
    got = out.cpu().view(batch, window, *out.shape[1:])[seqs].double().transpose(1, 2)
    worst = ((got - ref).abs() / bound).max().item()
    assert worst <= 1.0, f"largest error is {worst:.2f} of its bound"


@pytest.mark.parametrize("window,heads,hd", [(5, 4, 64), (32, 2, 128), (48, 4, 64), (64, 2, 128)])
def test_attention_takes_queries_that_start_on_eight_bytes(window, heads, hd):
    """They are loaded in pairs instead of in fours: the same values, so the same output."""
    g = torch.Generator().manual_seed(window)
    q = torch.randn(2 * window, heads, hd, generator=g).cuda()
    kv = torch.randn(2, 2, heads, 200, hd, generator=g).to(torch.bfloat16).cuda()
    pos = (200 - window + torch.arange(window, dtype=torch.int32)).repeat(2).cuda()
    pos[-2:] = -1
    shifted = torch.full((q.numel() + 2,), float("nan"), device="cuda")[2:].view(q.shape)
    shifted.copy_(q)
    assert q.data_ptr() % 16 == 0 and shifted.data_ptr() % 16 == 8
    want, _ = B.sjd_attention(q, kv, pos, window, heads)
    got, status = B.sjd_attention(shifted, kv, pos, window, heads)
    assert int(status.item()) == 0 and torch.equal(got, want)


@pytest.mark.parametrize("batch,window,keys,heads,kv_heads,hd", [
    (20, 40, 300, 8, 4, 128),    # one key range: the kernel writes the rows itself
    (20, 24, 300, 8, 8, 64),
    (2, 20, 600, 4, 2, 128),     # several key ranges and the merge; the bad key is in the first, the window in the last
    (1, 64, 150, 2, 1, 64),      # more ranges than tiles
])
def test_attention_shows_scores_that_are_not_numbers(batch, window, keys, heads, kv_heads, hd):
    """A NaN in a key reaches every row that sees it and no other, one in a query its own row."""
    g = torch.Generator().manual_seed(keys + window)
    n, group = keys - window, heads // kv_heads
    q = torch.randn(batch * window, heads, hd, generator=g)
    kv = torch.randn(batch, 2, kv_heads, keys, hd, generator=g).to(torch.bfloat16)
    pos = (n + torch.arange(window, dtype=torch.int32)).repeat(batch)
    pos[:2] = -1
    clean, _ = B.sjd_attention(q.cuda(), kv.cuda(), pos.cuda(), window, kv_heads)
    b = batch - 1
    for key in (70, n + window // 2):
        bad = kv.clone()
        bad[b, 0, kv_heads - 1, key, 3] = float("nan")
        out, status = B.sjd_attention(q.cuda(), bad.cuda(), pos.cuda(), window, kv_heads)
        sees = torch.zeros(batch * window, heads, dtype=torch.bool)
        sees[b * window:, heads - group:] = (pos[b * window:] >= key)[:, None]
        assert int(status.item()) == 0 and sees.any()
        assert torch.all(out.cpu()[sees].isnan())
        assert torch.equal(out.cpu()[~sees], clean.cpu()[~sees])
    q[window // 2, 0, 5] = float("nan")
    out, status = B.sjd_attention(q.cuda(), kv.cuda(), pos.cuda(), window, kv_heads)
    hit = torch.zeros(batch * window, heads, dtype=torch.bool)
    hit[window // 2, 0] = True
    assert int(status.item()) == 0
    assert torch.all(out.cpu()[hit].isnan())
    assert torch.equal(out.cpu()[~hit], clean.cpu()[~hit])
