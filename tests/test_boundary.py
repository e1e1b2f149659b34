"""Host-side checks of the C-ABI: the library loads, exports every function include/sjd.h declares,
and rejects bad arguments before touching a device.  No GPU."""
import ctypes as C
import os
import re

import pytest

from paper_2410_01699_b200 import binding as B
from paper_2410_01699_b200.inputs import WORKLOADS

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "sjd.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(sjd_[a-z_]+)\s*\(", text)))


def test_library_exports_every_declared_function():
    names = _declared_functions()
    assert "sjd_init" in names and "sjd_step" in names and "sjd_verify" in names and len(names) >= 12
    lib = B.lib()
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(B.EXPORTS) == sorted(n for n in names)


def test_struct_sizes_match_the_header_layout():
    assert C.sizeof(B.sjd_model_cfg) == 15 * 4
    assert C.sizeof(B.sjd_weights) == 14 * 8
    assert C.sizeof(B.sjd_sample_cfg) == 48
    assert B.sjd_sample_cfg.guidance.offset == 36 and B.sjd_sample_cfg.schedule.offset == 40
    assert B.sjd_sample_cfg.seed.offset == 8 and B.sjd_sample_cfg.window.offset == 16
    assert C.sizeof(B.sjd_step_out) == 8 * 8


def test_strerror_and_status_codes():
    lib = B.lib()
    seen = set()
    for code in (0, -1, -2, -3, -4, -5, -6):
        msg = lib.sjd_strerror(code).decode()
        assert msg and msg not in seen
        seen.add(msg)
    assert "unknown" in lib.sjd_strerror(-99).decode()


def test_workspace_size_query():
    wl = WORKLOADS["7b"]
    cfg = B.make_model_cfg(wl, max_batch=1, max_seq=2432, max_window=32)
    nbytes = B.sjd_workspace_bytes(cfg)
    kv = 32 * 2 * 32 * 128 * 2432 * 2
    logits = 2 * 32 * 65536 * 2
    assert kv + logits < nbytes < kv + logits + (256 << 20)
    # paged cache: the pool (plus its spare page) replaces max_batch x max_seq rows
    paged = B.make_model_cfg(wl, max_batch=8, max_seq=2432, max_window=32, kv_pages=40)
    pool = 41 * 32 * 2 * 32 * 64 * 128 * 2
    rest = B.sjd_workspace_bytes(B.make_model_cfg(wl, 8, 2432, 32)) - 8 * kv
    assert pool + rest <= B.sjd_workspace_bytes(paged) < pool + rest + (1 << 20)
    for field, bad in (("n_layers", 0), ("head_dim", 63), ("n_kv_heads", 5), ("max_window", 0), ("dtype", 7),
                       ("kv_pages", -1)):
        c = B.make_model_cfg(wl, 1, 2432, 32)
        setattr(c, field, bad)
        assert B.sjd_workspace_bytes(c) == 0, field


def test_calls_reject_bad_arguments_without_a_device():
    lib = B.lib()
    s = B.make_sample_cfg(top_k=10, window=4)
    out = B.sjd_step_out()
    one = C.c_void_p(256)  # never dereferenced: validation fails first
    assert lib.sjd_verify(0, 4, 16, 0, one, one, one, None, None, C.byref(s), 0, C.byref(out), one, 1 << 20, None) == B.SJD_ERR_BAD_ARG
    assert lib.sjd_verify(1, 4, 16, 9, one, one, one, None, None, C.byref(s), 0, C.byref(out), one, 1 << 20, None) == B.SJD_ERR_UNSUPPORTED
    assert lib.sjd_verify(1, 65, 16, 0, one, one, one, None, None, C.byref(s), 0, C.byref(out), one, 1 << 20, None) == B.SJD_ERR_CAPACITY
    assert lib.sjd_verify(1, 4, 16, 0, one, one, one, None, None, C.byref(s), 0, C.byref(out), one, 8, None) == B.SJD_ERR_CAPACITY
    assert lib.sjd_verify(1, 4, 16, 0, None, one, one, None, None, C.byref(s), 0, C.byref(out), one, 1 << 20, None) == B.SJD_ERR_BAD_ARG
    # queries are loaded in pairs of floats: any other address is refused before the device is asked for
    def attention(q):
        return lib.sjd_attention(1, 4, 2, 2, 64, 32, C.c_void_p(q), one, one, one, one, 1 << 20, None)
    assert attention(256 + 4) == B.SJD_ERR_BAD_ARG and attention(256 + 2) == B.SJD_ERR_BAD_ARG
    ctx = C.c_void_p()
    cfg = B.make_model_cfg(WORKLOADS["tiny"], 1, 64, 8)
    assert lib.sjd_init(C.byref(ctx), C.byref(cfg), None, one, 1 << 30) == B.SJD_ERR_BAD_ARG
    assert lib.sjd_step(None, None, None) == B.SJD_ERR_BAD_ARG
    assert lib.sjd_prefill(None, 1, one, 4, C.byref(s), None) == B.SJD_ERR_BAD_ARG
    assert lib.sjd_last_device_status(None) == B.SJD_ERR_BAD_ARG
    lib.sjd_destroy(None)
    assert B.sjd_verify_workspace_bytes(0, 4) == 0 and B.sjd_verify_workspace_bytes(32, 32) >= 32 * 32 * 64


def test_every_entry_point_of_the_tensor_core_kernels_asks_for_the_same_device():
    """tcgen05 and tensor memory exist on compute capability 10.x only: sjd_gemm, sjd_attention and sjd_init (which takes the
    generic kernels elsewhere) test for it, and the header promises nothing else.  Read from the source: no device to ask here."""
    csrc = os.path.join(ROOT, "paper_2410_01699_b200", "csrc")
    tests = {f: re.findall(r"\bcc_major\s*([<>=!]=|[<>])\s*(\d+)", open(os.path.join(csrc, f)).read()) for f in ("api.cu", "engine.cu")}
    assert tests == {"api.cu": [("!=", "10"), ("!=", "10")], "engine.cu": [("==", "10")]}
    header = open(os.path.join(ROOT, "include", "sjd.h")).read()
    assert re.findall(r"compute\s[\s*]*capability\s([^;]*?);", header) == ["10.x", "10.x"]


def test_tensor_core_roles_wait_as_a_warp():
    """The lanes of a warp may leave a polling loop in different rounds; the tcgen05 loads and named barriers that follow the waits are
    defined for a converged warp.  So no kernel calls the wait of a single thread."""
    csrc = os.path.join(ROOT, "paper_2410_01699_b200", "csrc")
    calls = {f: len(re.findall(r"\bmbar_wait\(", open(os.path.join(csrc, f)).read())) for f in ("attention_tc.cu", "gemm_tc.cu", "tcgen05.cuh")}
    assert calls == {"attention_tc.cu": 0, "gemm_tc.cu": 0, "tcgen05.cuh": 2}   # its definition and warp_wait


def test_missing_library_fails_loudly(monkeypatch):
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "LIB_PATH", "/nonexistent/libsjd.so")
    with pytest.raises(RuntimeError, match="not built"):
        B.lib()
