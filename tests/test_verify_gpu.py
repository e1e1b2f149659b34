"""GPU parity of the fused verify-and-resample kernel (sjd_verify through the C-ABI) against the
CPU checker, element by element on the same seeded inputs."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2410_01699_b200 import binding as B
from paper_2410_01699_b200.inputs import make_verify_case, round_bf16
from tests.parity_util import ParityStats, compare_window, oracle_verify_case, run_in_threads

pytestmark = pytest.mark.gpu


def _run_gpu(case, logits_prev=True):
    dt = torch.bfloat16 if case.dtype == "bf16" else torch.float32
    cur = torch.from_numpy(case.logits_cur).to("cuda").to(dt)
    prev = torch.from_numpy(case.logits_prev).to("cuda").to(dt) if logits_prev else None
    draft = torch.from_numpy(case.draft).cuda()
    kind = torch.from_numpy(case.q_kind.astype(np.int32)).cuda()
    base = torch.from_numpy(case.base_pos).cuda()
    out = B.StepOut(case.batch, case.window)
    sample = B.make_sample_cfg(temperature=case.temperature, top_k=case.top_k, seed=case.seed, window=case.window)
    B.sjd_verify(cur, prev, draft, kind, base, sample, case.step, out)
    return out.host()


def _check_case(case, prob_tol=1e-5, max_flag_frac=0.03):
    got = _run_gpu(case)
    stats = ParityStats()
    for b in range(case.batch):
        vr, qdescs = oracle_verify_case(case, b)
        gpu = dict(n_accepted=got["n_accepted"][b], committed=got["committed"][b], draft=got["draft"][b],
                   q_draft=got["q_draft"][b])
        st = compare_window(vr, gpu, case.logits_cur[b].astype(np.float64), case.draft[b], qdescs, case.temperature,
                            case.top_k, prob_tol, where=f"seq {b}")
        stats.merge(st)
        if st.skipped_sequences == 0:
            assert got["n_committed"][b] == len(vr.committed)
            assert got["total_committed"][b] == case.base_pos[b] + len(vr.committed)
            kept = len(vr.redraft)
            assert list(got["q_kind"][b][:kept]) == [B.SJD_Q_ROW] * kept
            assert all(x == -1 for x in got["draft"][b][kept:]) and all(x == -1 for x in got["q_kind"][b][kept:])
    assert stats.flagged <= max(2, max_flag_frac * stats.decisions), f"too many near-ties: {stats}"
    return stats


@pytest.mark.parametrize("batch", [1, 4])
def test_verify_workload_shape(batch):
    """The isolated-verification workload: W = 32 rows over a 16384 vocabulary, bf16, top-k 2000."""
    _check_case(make_verify_case(batch))


def test_verify_full_batch():
    """Largest batch of the workload in the launch configuration the benchmark times (32 sequences of
    32 rows): every sequence is re-computed by the checker."""
    stats = _check_case(make_verify_case(32))
    assert stats.sequences == 32


# Few rows run on a thread-block cluster each, bf16 rows in more blocks than the device has SMs (148) on a block per row: the
# corner cases below take both routes.
@pytest.mark.parametrize("batch", [3, 40])
def test_verify_ratio_corner_cases(batch):
    """Eq. 1 where q(d) or p(d) vanishes (drafts whose law is a logits row, top-k 200 of 4096):
    q(d) = 0 < p(d) accepts for any uniform, p(d) = 0 < q(d) rejects, p(d) = q(d) = 0 rejects.  Rows
    around the corner rows have identical current and previous logits (ratio exactly 1: accepted), so the
    scan reaches each corner row and the number of accepted drafts is known without any checker."""
    case = make_verify_case(batch, window=6, vocab=4096, top_k=200, seed=77)
    case.logits_prev = case.logits_cur.copy()
    order = np.argsort(-case.logits_cur, axis=-1, kind="stable")   # tokens of each row, largest logit first

    def put(b, k, p_in, q_in):
        """Draft of row k of sequence b: a token of p's top-k set (or not), q's entry raised / lowered."""
        d = int(order[b, k, 50 if p_in else 3000])
        case.draft[b, k] = d
        if p_in and not q_in:
            case.logits_prev[b, k, d] = np.float32(-30.0)     # out of q's set; q's set takes the 201st entry in
        if q_in and not p_in:
            case.logits_prev[b, k, d] = np.float32(12.0)      # in q's set only
        return d

    for b in range(batch):
        for k in range(6):
            case.draft[b, k] = int(order[b, k, 20])           # p == q on the draft: always accepted
    put(0, 2, True, False)     # q(d) = 0 < p(d): accepted, the scan goes on
    put(0, 4, False, False)    # 0 / 0: rejected
    put(1, 0, True, False)     # accepted
    put(1, 1, False, True)     # p(d) = 0 < q(d): rejected
    put(2, 0, False, False)    # 0 / 0 on the very first row
    got = _run_gpu(case)
    assert list(got["n_accepted"]) == [4, 1, 0] + [6] * (batch - 3)
    assert list(got["n_committed"]) == [5, 2, 1] + [6] * (batch - 3)
    stats = _check_case(case)
    assert stats.flagged == 0


@pytest.mark.parametrize("batch,dtype,vocab,window,top_k", [
    (2, "bf16", 16001, 29, 2000),    # ragged: rows not 16-byte aligned, odd window
    (6, "bf16", 16001, 29, 2000),    # the same, a staged block per row
    (2, "f32", 1024, 16, 64),        # the tiny end-to-end model's head
    (2, "f32", 1000, 7, 1000),       # top_k == V: no filtering
    (22, "f32", 1000, 7, 1000),      # the same, a block per row
    (2, "bf16", 4099, 5, 1),         # top-1
    (30, "bf16", 4099, 5, 1),
    (2, "bf16", 65536, 4, 2000),     # 128 KB rows (the 7B head)
    (38, "bf16", 65536, 4, 2000),    # the same in the registers of a block
    (2, "bf16", 184320, 2, 2048),    # the longest bf16 rows of a cluster (the 8B head)
    (10, "bf16", 184320, 2, 2048),   # longer than a block's registers: streamed in three segments
    (2, "bf16", 100000, 5, 2000),
    (8, "bf16", 100000, 5, 2000),    # two segments, the second partial (12500 vectors against 8192)
    (2, "bf16", 184320, 3, 184320),  # top_k == V: no threshold
    (7, "bf16", 184320, 3, 184320),  # the same on streamed rows
    (2, "bf16", 262000, 2, 4000),
    (10, "bf16", 262000, 2, 4000),   # the longest row the chunk table covers: four segments
    (2, "f32", 50000, 3, 500),       # fp32 rows beyond the staging buffer
])
def test_verify_shapes(batch, dtype, vocab, window, top_k):
    """Row lengths, alignments and filters at a few rows (a cluster per row) and at many (a block per row)."""
    case = make_verify_case(batch, window=window, vocab=vocab, dtype=dtype, top_k=top_k, seed=7 + vocab)
    _check_case(case, max_flag_frac=0.06)


@pytest.mark.parametrize("batch,window,vocab,dtype,top_k", [
    (1, 3, 65537, "f32", 900),       # rows that start off 16 bytes, the last vector partly outside
    (1, 2, 131056, "f32", 2000),     # close to the longest row: eight blocks, eight vectors per thread
    (2, 2, 513, "f32", 1),           # one block, the last vector partly outside
    (15, 5, 2050, "f32", 100),       # one block whose rows reach past the first vector of every thread
    (5, 32, 3000, "f32", 100),       # more rows than SMs: Eq. 2 left to the sequence's last block
    (2, 5, 60001, "bf16", 700),      # bf16 rows at four alignments
    (1, 3, 32776, "bf16", 40000),    # no filter (top-k above the vocabulary), odd tail
])
def test_verify_cluster_rows(batch, window, vocab, dtype, top_k):
    """A thread-block cluster per row: slice sizes, alignments and the rules between it and a block per row."""
    _check_case(make_verify_case(batch, window=window, vocab=vocab, dtype=dtype, top_k=top_k, mixed_kinds=True, seed=9))


@pytest.mark.parametrize("levels", [3, 4000])
def test_verify_cluster_ties(levels):
    """fp32 rows of few distinct values: thousands of entries tie at the threshold (more than a block lists at 3 levels)."""
    case = make_verify_case(1, window=3, vocab=40000, dtype="f32", top_k=1500, seed=11)
    for rows in (case.logits_cur, case.logits_prev):
        rows[...] = np.floor(rows * (levels / 60.0)) * np.float32(60.0 / levels)
    _check_case(case)


def _awkward(case, mode, seed=0):
    """Rows whose threshold a histogram of the codes next to the maximum does not reach, or whose entries are not all finite."""
    rng = np.random.default_rng(seed)
    for rows in (case.logits_cur, case.logits_prev):
        if mode == "below zero":            # positive maximum, negative threshold
            rows -= np.float32(9.0)
        elif mode.startswith("masked"):     # nine entries in ten hold one value, the threshold among them
            rows[rng.random(rows.shape) > 0.1] = np.float32(-np.inf if mode == "masked -inf" else -1e9)
        elif mode == "dense":               # a third of the row within one step of the 16 leading bits of a key
            pick = rng.random(rows.shape) < 0.33
            rows[pick] = (8.0 + 0.03 * rng.random(int(pick.sum()))).astype(np.float32)
        elif mode == "levels":
            rows[...] = np.floor(rows / 8.0) * np.float32(8.0)
    if mode == "nan":                       # in this row, the earlier one, both
        case.logits_cur[:, 0::3, 7] = np.nan
        case.logits_prev[:, 1::3, 9] = np.inf
        case.logits_cur[:, 2::3, 11] = np.inf
        case.logits_prev[:, 2::3, 11] = np.nan
    if mode == "none finite":
        case.logits_cur[::2, case.window // 2, :] = -np.inf
        case.logits_prev[1::2, 0, :] = -np.inf
        if case.batch == 1:
            case.logits_prev[:, 0, :] = -np.inf
    if case.dtype == "bf16":
        case.logits_cur, case.logits_prev = round_bf16(case.logits_cur), round_bf16(case.logits_prev)
    for b in range(case.batch):             # drafts that have mass in both rows
        for k in range(case.window):
            both = np.nan_to_num(case.logits_cur[b, k], nan=-1e30, posinf=-1e30, neginf=-1e30)
            case.draft[b, k] = int(np.argsort(-both, kind="stable")[3])
    return case


@pytest.mark.parametrize("mode", ["below zero", "masked -1e9", "masked -inf", "dense", "levels", "nan", "none finite"])
@pytest.mark.parametrize("batch,window,vocab,dtype", [
    (1, 4, 1024, "f32"), (1, 3, 4000, "f32"), (1, 4, 8001, "f32"), (1, 3, 40000, "f32"),         # clusters of 1, 2, 4, 8 blocks
    (1, 4, 4096, "bf16"), (1, 3, 8000, "bf16"), (1, 3, 16001, "bf16"), (1, 3, 40000, "bf16"),
    (19, 8, 4096, "f32"), (150, 1, 3000, "f32"),                                                # more rows than SMs
    (19, 8, 4096, "bf16"), (75, 2, 3001, "bf16"),                                               # and a block per row
    (7, 3, 140000, "bf16"),                                                                     # whose rows are streamed
])
def test_verify_awkward_rows(batch, window, vocab, dtype, mode):
    """Thresholds far below the maximum, masked entries, thousands of ties, entries that are not finite: on every size of cluster
    and with a block per row."""
    case = make_verify_case(batch, window=window, vocab=vocab, dtype=dtype, top_k=vocab // 4, seed=41)
    _check_case(_awkward(case, mode), max_flag_frac=0.06)
    if mode == "nan" and window > 2:
        assert all(f & B.SJD_FLAG_NONFINITE for f in _run_gpu(case)["flags"])


def test_verify_mixed_laws():
    """Slots whose draft came from a uniform initialisation (q = 1/V) or a copy (point mass)."""
    case = make_verify_case(6, window=16, vocab=4096, top_k=300, seed=11, mixed_kinds=True)
    _check_case(case)


@pytest.mark.parametrize("batch", [3, 7])   # a cluster per row; streamed through the registers of a block
def test_verify_mixed_laws_on_long_rows(batch):
    """The same on rows too long for a block's registers (drift 3: most drafts are rejected, so Eq. 2 runs on long
    rows against uniform, copied and predicted drafts)."""
    case = make_verify_case(batch, window=6, vocab=100000, top_k=2000, seed=12, mixed_kinds=True, drift=3.0)
    _check_case(case, max_flag_frac=0.06)


def test_verify_streamed_rows_in_a_grid_of_several_waves():
    """160 streamed rows on 148 SMs: the rejected rows leave Eq. 2 to their sequence's last block, which streams
    the two rows again."""
    case = make_verify_case(10, window=16, vocab=70000, top_k=2000, seed=13, drift=2.0)
    _check_case(case, max_flag_frac=0.06)


@pytest.mark.parametrize("batch", [3, 20])
def test_verify_temperature_and_ties(batch):
    case = make_verify_case(batch, window=8, vocab=8192, top_k=500, temperature=0.7, seed=5)
    _check_case(case)
    # coarse logits: many exact ties at the top-k threshold (all must be kept)
    case = make_verify_case(batch, window=8, vocab=8192, top_k=500, seed=6)
    case.logits_cur = round_bf16(np.round(case.logits_cur * 2) / 2)
    case.logits_prev = round_bf16(np.round(case.logits_prev * 2) / 2)
    _check_case(case)


@pytest.mark.parametrize("batch", [2, 26])
@pytest.mark.parametrize("shift,top_k", [
    (-9.0, 2000),    # positive maximum, negative threshold: more than 4095 bf16 codes apart
    (-30.0, 2000),   # every logit negative: maximum and threshold within a few binades
    (0.0, 8000),     # half the row kept: threshold around zero
    (0.0, 16384),    # top_k == V: no filtering
])
def test_verify_threshold_far_from_the_maximum(shift, top_k, batch):
    """Entries are counted by their distance below the row maximum.  Where the threshold is out of the histogram's reach, a
    cluster counts on in further windows and a block per row takes its general route."""
    case = make_verify_case(batch, window=6, vocab=16384, top_k=top_k, seed=31)
    case.logits_cur = round_bf16(case.logits_cur + np.float32(shift))
    case.logits_prev = round_bf16(case.logits_prev + np.float32(shift))
    _check_case(case, max_flag_frac=0.06)


@pytest.mark.parametrize("batch", [2, 38])
def test_verify_zeros_at_the_threshold(batch):
    """Exact zeros of both signs around the top-k threshold (bf16 comparison cannot order +0 and -0, the
    order-preserving keys can): with a block per row such rows take the general route."""
    case = make_verify_case(batch, window=4, vocab=8192, top_k=3000, seed=33)
    for arr in (case.logits_cur, case.logits_prev):
        small = np.abs(arr) < 0.35
        arr[small] = np.where(arr[small] < 0, np.float32(-0.0), np.float32(0.0))
    _check_case(case, max_flag_frac=0.06)


def test_verify_identical_rows_accept_everything():
    """p == q bit for bit: every ratio is 1 and every draft is accepted for any uniform."""
    case = make_verify_case(2, window=12, vocab=4096, top_k=100, seed=3)
    case.logits_prev = case.logits_cur.copy()
    got = _run_gpu(case)
    assert list(got["n_accepted"]) == [12, 12] and list(got["n_committed"]) == [12, 12]
    assert np.array_equal(got["committed"], case.draft)
    assert np.all(got["draft"] == -1)


@pytest.mark.parametrize("batch", [2, 38])
def test_verify_nonfinite_rows_are_flagged(batch):
    case = make_verify_case(batch, window=4, vocab=2048, top_k=50, seed=9)
    case.logits_cur[0, 1, 5] = np.nan
    case.logits_cur[0, 1, 9] = np.inf
    got = _check_and_flags(case)
    assert got["flags"][0] & B.SJD_FLAG_NONFINITE
    assert not (got["flags"][1] & B.SJD_FLAG_NONFINITE)


def _check_and_flags(case):
    _check_case(case)
    return _run_gpu(case)


def test_verify_is_deterministic():
    case = make_verify_case(4, window=16, vocab=16384, seed=21)
    a, b = _run_gpu(case), _run_gpu(case)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("rows,dtype", [((4096, 16000), "f32"), ((12001, 30001), "bf16")])   # a cluster, a block per row
def test_verify_threads_with_different_rows(rows, dtype):
    """Two threads whose rows need different amounts of shared memory in the same kernel."""
    def calls(vocab):
        case = make_verify_case(20, window=8, vocab=vocab, dtype=dtype, top_k=100, seed=4)
        dt = torch.bfloat16 if dtype == "bf16" else torch.float32
        args = [torch.from_numpy(a).cuda() for a in (case.logits_cur, case.logits_prev, case.draft, case.q_kind.astype(np.int32),
                                                     case.base_pos)]
        args[:2] = [a.to(dt) for a in args[:2]]
        sample = B.make_sample_cfg(temperature=case.temperature, top_k=case.top_k, seed=case.seed, window=case.window)
        outs = [B.StepOut(case.batch, case.window) for _ in range(2)]
        ws = torch.empty(B.sjd_verify_workspace_bytes(case.batch, case.window), dtype=torch.uint8, device="cuda")
        stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        call = [(case.batch, case.window, vocab, B.SJD_BF16 if dtype == "bf16" else B.SJD_F32,
                 *(C.c_void_p(a.data_ptr()) for a in args), C.byref(sample), case.step, C.byref(o.c), C.c_void_p(ws.data_ptr()),
                 ws.numel(), stream) for o in outs]
        verify = B.lib().sjd_verify
        assert all(verify(*call[i > 0]) == B.SJD_OK for i in range(5000))
        a, b = outs[0].host(), outs[1].host()
        assert all(np.array_equal(a[k], b[k]) for k in a)

    run_in_threads(*[lambda v=v: calls(v) for v in rows * 2])


def test_verify_argument_errors():
    out = B.StepOut(1, 4)
    s = B.make_sample_cfg(top_k=10, window=4)
    cur = torch.zeros(1, 4, 128, device="cuda")
    d = torch.zeros(1, 4, dtype=torch.int32, device="cuda")
    ws = torch.empty(B.sjd_verify_workspace_bytes(1, 4), dtype=torch.uint8, device="cuda")
    L = B.lib()
    import ctypes as C
    args = lambda **kw: [kw.get("b", 1), kw.get("w", 4), 128, kw.get("dt", 0), C.c_void_p(cur.data_ptr()),
                         C.c_void_p(cur.data_ptr()), C.c_void_p(d.data_ptr()), None, None, C.byref(kw.get("s", s)), 0,
                         C.byref(out.c), C.c_void_p(ws.data_ptr()), kw.get("n", ws.numel()), None]
    assert L.sjd_verify(*args()) == B.SJD_OK
    assert L.sjd_verify(*args(b=0)) == B.SJD_ERR_BAD_ARG
    assert L.sjd_verify(*args(dt=5)) == B.SJD_ERR_UNSUPPORTED
    assert L.sjd_verify(*args(n=16)) == B.SJD_ERR_CAPACITY
    assert L.sjd_verify(*args(s=B.make_sample_cfg(temperature=0.0, top_k=10))) == B.SJD_ERR_BAD_ARG
    assert L.sjd_verify(*args(s=B.make_sample_cfg(top_k=0))) == B.SJD_ERR_BAD_ARG
    torch.cuda.synchronize()
