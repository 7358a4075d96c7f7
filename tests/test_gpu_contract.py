"""What the header promises of every call, checked where a size decides which kernel serves it."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import parity
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu


def select(lens, keeps, scores, protect=None, q_idx=None, cu_qlens=None, total_q=0, flags=0):
    """fastav_select on host arrays: (keep_idx, cu_keep, status)."""
    dev = lambda a, dt: None if a is None else torch.as_tensor(np.asarray(a), dtype=dt).cuda()
    n, kept = sum(lens), sum(keeps)
    params = fastav.make_params(batch=len(lens), total_tokens=n, max_seqlen=max(lens), total_q=total_q, max_qlen=total_q, total_keep=kept,
                                max_keep=max(keeps), num_q_heads=4, num_kv_heads=2, head_dim=64, hidden=64, flags=flags)
    ws = torch.empty(max(256, fastav.fastav_workspace_bytes(params)), dtype=torch.uint8, device="cuda")
    idx = torch.full((kept + 1,), -7, dtype=torch.int32, device="cuda")
    cu_keep, status = torch.empty(len(lens) + 1, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    fastav.fastav_select(params, dev(scores, torch.float32), dev(np.concatenate([[0], np.cumsum(lens)]), torch.int32), dev(keeps, torch.int32),
                         dev(protect, torch.uint8), dev(q_idx, torch.int32), dev(cu_qlens, torch.int32), idx, cu_keep, ws, status)
    torch.cuda.synchronize()
    return idx.cpu().numpy()[:kept], cu_keep.cpu().numpy(), int(status)


@pytest.mark.parametrize("longest", [2048, 2049])
def test_select_reads_the_scored_rows_only_under_their_flag(longest):
    """Without FASTAV_PROTECT_QUERY_ROWS the arrays may say anything, here rows that total_q = 0 denies."""
    lens, keeps = [longest, 100], [700, 33]
    scores = np.random.default_rng(longest).random(sum(lens)).astype(np.float32)
    idx, cu_keep, status = select(lens, keeps, scores, q_idx=[5, 6, 7], cu_qlens=[0, 2, 3])
    want_idx, want_cu = oracle.select(scores, np.concatenate([[0], np.cumsum(lens)]), np.asarray(keeps))
    assert status == 0
    assert np.array_equal(idx, want_idx) and np.array_equal(cu_keep, want_cu)


@pytest.mark.parametrize("longest", [2048, 2049])
@pytest.mark.parametrize("keep", [0, 1, 2, 3])
@pytest.mark.parametrize("by_rows", [False, True])
def test_more_protected_tokens_than_are_kept_is_reported(longest, keep, by_rows):
    """Two protected tokens in the first sequence: the bit is set exactly when fewer are kept, none included."""
    lens, keeps = [longest, 64], [keep, 10]
    scores = np.random.default_rng(7).random(sum(lens)).astype(np.float32)
    protect = np.zeros(sum(lens), dtype=np.uint8)
    rows = dict(q_idx=[40, longest - 1], cu_qlens=[0, 2, 2], total_q=2, flags=fastav.FASTAV_PROTECT_QUERY_ROWS)
    if not by_rows:
        protect[[40, longest - 1]] = 1
        rows = {}
    idx, cu_keep, status = select(lens, keeps, scores, protect, **rows)
    assert status == (fastav.FASTAV_DEV_PROTECT_OVERFLOW if keep < 2 else 0)
    assert cu_keep.tolist() == [0, keep, keep + 10] and {40, longest - 1} & set(idx[:keep]) == ({40, longest - 1} if keep >= 2 else {40} if keep else set())


def mask_call(mask, cu, total_keep):
    params = fastav.make_params(batch=len(cu) - 1, total_tokens=len(mask), max_seqlen=len(mask), total_q=0, max_qlen=0, total_keep=total_keep,
                                max_keep=total_keep, num_q_heads=4, num_kv_heads=2, head_dim=64, hidden=64)
    idx = torch.full((total_keep,), -7, dtype=torch.int32, device="cuda")
    cu_keep, status = torch.empty(len(cu), dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(max(256, 4 * len(cu) + 256), dtype=torch.uint8, device="cuda")
    fastav.fastav_select_mask(params, torch.as_tensor(mask).cuda(), torch.as_tensor(np.asarray(cu), dtype=torch.int32).cuda(), idx, cu_keep, ws, status)
    torch.cuda.synchronize()
    return idx.cpu().numpy(), cu_keep.cpu().numpy(), int(status)


@pytest.mark.parametrize("total", [5000, (1 << 17) + 77])
def test_mask_counts_the_tokens_of_the_sequences_only(total):
    """Marked tokens before the first sequence belong to none."""
    mask = (np.random.default_rng(total).random(total) < 0.5).astype(np.uint8)
    mask[:900] = 1
    cu = np.array([900, 900, 1700, total - 3], dtype=np.int32)
    want_idx, want_cu = oracle.select_mask(mask, cu)
    idx, cu_keep, status = mask_call(mask, cu, int(want_cu[-1]))
    assert status == 0 and np.array_equal(cu_keep, want_cu) and np.array_equal(idx, want_idx)


@pytest.mark.parametrize("total", [5000, (1 << 17) + 77])
def test_mask_cuts_impossible_spans_down(total):
    """Bounds beyond the batch are cut down and reported; the survivors' prefix sums never fall back."""
    mask = np.ones(total, dtype=np.uint8)
    cu = [0, 100, total + 50, total + 60, 40, 300]  # 100 tokens; the rest of the batch; none; none (backwards); 260 tokens
    idx, cu_keep, status = mask_call(mask, cu, total)
    assert status == fastav.FASTAV_DEV_SHAPE_MISMATCH | fastav.FASTAV_DEV_K_CLAMPED
    assert cu_keep.tolist() == [0, 100, total, total, total, total]
    assert np.array_equal(idx, np.concatenate([np.arange(100), np.arange(total - 100)]))


@pytest.mark.parametrize("first", [2, 6])
def test_a_rollout_may_start_at_any_even_layer_number(first):
    """`layer_index` chooses which copy of the state is read; nothing else depends on where the
    count starts (begin leaves the identity where an even layer reads)."""
    from test_gpu_rollout import _layers, _params

    n, hq, hkv, d, layers = 300, 4, 2, 64, 3
    qk = [(q.cuda(), k.cuda()) for q, k in _layers(3, n, hq, hkv, d, layers)]
    p = _params(n, hq, hkv, d, *qk[0], d**-0.5, True)
    ws = torch.empty(fastav.fastav_rollout_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    got = []
    for start in (0, first):
        state = torch.full((fastav.fastav_rollout_state_bytes(n),), 255, dtype=torch.uint8, device="cuda")
        fastav.fastav_rollout_begin(n, state)
        for i, (q, k) in enumerate(qk):
            fastav.fastav_rollout_layer(p, q, k, 0.5, start + i, state, ws)
        imp, r = torch.empty(n, device="cuda"), torch.empty(n, n, device="cuda")
        fastav.fastav_rollout_read(n, start + layers, state, imp, r)
        got.append((imp, r))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("longest,rows", [(6, 5), (600, 1)])
def test_batches_of_thousands(longest, rows):
    """More (sequence, KV head) pairs than the tensor-core kernels' blocks, one per SM, can list: on its sweeps (forced, the one-pass
    score would take them) and on its logits for few rows."""
    lens = [longest] + [6] * 3599
    p = W.random_problem(3, lens, [rows] * 3600, [2] * 3600, 4, 2, 64, 16)
    buf = parity.to_device(p, extra_flags=fastav.FASTAV_SCORE_PATH_WIDE if rows > 4 else 0)
    buf.prune()
    torch.cuda.synchronize()
    stats = parity.check_fused_against_oracle(p, buf, parity.oracle_prune(p))
    assert stats["device_status"] & ~fastav.FASTAV_DEV_PROTECT_OVERFLOW == 0


def test_rows_are_right_where_max_keep_says_too_little():
    """2,048 survivors of 1,458 pieces each in one block, where max_keep promises one: rows are found by a division that is a
    multiplication only for what max_keep allows."""
    lens = [2048] + [1] * 74
    p = W.random_problem(8, lens, [1] * 75, lens, 2, 1, 64, 11536)
    buf = parity.to_device(p)
    buf.params.max_keep = 1
    buf.prune()
    torch.cuda.synchronize()
    for name, source in (("hidden_out", p.hidden), ("pos_out", p.pos), ("k_out", p.k), ("v_out", p.v)):
        parity.assert_bits_equal(getattr(buf, name), source, name)


@pytest.mark.parametrize("rows", [1, 9])
def test_calls_work_in_a_second_context_of_the_same_device(rows):
    """Kernel attributes belong to a context: what was set in torch's does not count in another one."""
    buf = parity.to_device(W.random_problem(5, [700, 300], [rows, rows], [350, 100], 8, 2, 64, 128))
    buf.prune()
    torch.cuda.synchronize()
    names = ("q", "q_idx", "cu_qlens", "k", "v", "cu_seqlens", None, "keep_counts", None, "hidden", "pos", "scores", "keep_idx", "cu_keep",
             "hidden_out", "pos_out", "k_out", "v_out")
    host = {n: getattr(buf, n).cpu().contiguous() for n in names if n}
    cuda = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        assert getattr(cuda, name)(*args) == 0, name

    def allocated(size):
        at = ctypes.c_uint64()
        call("cuMemAlloc_v2", ctypes.byref(at), ctypes.c_size_t(size))
        return at

    before, context = ctypes.c_void_p(), ctypes.c_void_p()
    call("cuCtxGetCurrent", ctypes.byref(before))
    call("cuCtxCreate_v2", ctypes.byref(context), 0, torch.cuda.current_device())
    try:
        where = {n: allocated(t.nbytes) for n, t in host.items()}
        for n, t in host.items():
            call("cuMemcpyHtoD_v2", where[n], ctypes.c_void_p(t.data_ptr()), ctypes.c_size_t(t.nbytes))
        outputs = names[names.index("scores"):]
        for n in outputs:
            call("cuMemsetD8_v2", where[n], ctypes.c_ubyte(0xEE), ctypes.c_size_t(host[n].nbytes))
        workspace = allocated(buf.workspace.nbytes)
        rc = fastav.library().fastav_prune(ctypes.byref(buf.params), *(ctypes.c_void_p(where[n].value) if n else None for n in names),
                                           ctypes.c_void_p(workspace.value), buf.workspace.nbytes, None, None)
        assert rc == 0, fastav.library().fastav_last_cuda_error()
        call("cuCtxSynchronize")
        for n in outputs:
            got = torch.empty_like(host[n])
            call("cuMemcpyDtoH_v2", ctypes.c_void_p(got.data_ptr()), where[n], ctypes.c_size_t(got.nbytes))
            parity.assert_bits_equal(got, host[n], n)
    finally:
        call("cuCtxDestroy_v2", context)
        call("cuCtxSetCurrent", before)


@pytest.mark.parametrize("batch", [31, 32, 33, 64, 65, 1024, 1025, 1057])
def test_statistics_find_their_sequence_in_any_batch(batch):
    """The merge of the two sweeps' statistics looks a row's sequence up, 32 at a time; empty sequences and ones without rows among
    them."""
    lens = [(37 * i) % 23 + 6 if i % 7 else 0 for i in range(batch)]
    p = W.random_problem(batch, lens, [0 if n == 0 or n % 5 == 0 else 5 for n in lens], [n // 2 for n in lens], 4, 2, 64, 16)
    buf = parity.to_device(p, extra_flags=fastav.FASTAV_SCORE_PATH_WIDE)
    buf.score()
    torch.cuda.synchronize()
    parity.assert_scores_close(buf.scores, parity.oracle_scores(p))
    assert int(buf.device_status) == 0


def test_a_key_that_is_not_a_number_shows_in_the_attention_map():
    """Whatever column it stands in: every row that sees the key has NaN there."""
    from test_gpu_rollout import _layers, _params

    n, hq, hkv, d = 160, 2, 1, 64
    (q, k), = [(q.cuda(), k.cuda()) for q, k in _layers(5, n, hq, hkv, d, 1)]
    p = _params(n, hq, hkv, d, q, k, d**-0.5, True)
    ws = torch.empty(fastav.fastav_rollout_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    state = torch.empty(fastav.fastav_rollout_state_bytes(n), dtype=torch.uint8, device="cuda")
    for j in range(32, 49):
        bad = k.clone()
        bad[j] = float("nan")
        out = torch.zeros(n, n, device="cuda")
        fastav.fastav_rollout_begin(n, state)
        fastav.fastav_rollout_layer(p, q, bad, 0.5, 0, state, ws, map_out_opt=out)
        assert out[j:, j].isnan().all(), j


# More survivors than total_keep says, on every path that writes a keep list: from the keys by counting and by digits, from partial
# sums of short and of long sequences, after the sweeps of more sequences than clusters run at once, from scores (three layouts).
@pytest.mark.parametrize("lens,rows", [([500, 40], 1), ([2048, 40], 1), ([1000, 40], 8), ([2600, 40], 9), ([40000, 40], 9), ([2600, 40], 1), ([40000, 40], 1),
                                       ([60000, 40], 1)])
@pytest.mark.parametrize("short", [1, 15, 60])  # of the second sequence's 30 survivors one, half, or all of them and some of the first's
def test_survivors_beyond_the_capacity_are_left_out(lens, rows, short):
    """The buffers hold all survivors, the parameters promise fewer: what lies beyond stays as it was, and the bit says so."""
    p = W.random_problem(sum(lens) + rows, lens, [rows] * len(lens), [lens[0] // 2, 30], 4, 2, 64, 16)
    buf = parity.to_device(p)
    kept = sum(p.keep_counts.tolist())
    buf.params.total_keep, buf.params.max_keep = kept - short, min(lens[0] // 2, kept - short)
    outputs = ("keep_idx", "hidden_out", "pos_out", "k_out", "v_out")
    for name in outputs:
        getattr(buf, name).fill_(-7)
    buf.prune()
    torch.cuda.synchronize()
    assert int(buf.device_status) == fastav.FASTAV_DEV_SHAPE_MISMATCH
    idx, cu = oracle.select(buf.scores.cpu().numpy(), p.cu_seqlens.numpy(), p.keep_counts.numpy())
    assert buf.cu_keep.cpu().tolist() == cu.tolist()
    assert np.array_equal(buf.keep_idx.cpu().numpy()[:kept - short], idx[:kept - short])
    rows_of = parity.gather_rows(p, idx, cu)
    for name in outputs[1:]:
        parity.assert_bits_equal(getattr(buf, name)[:kept - short], rows_of[name.removesuffix("_out")][:kept - short], name)
    for name in outputs:
        assert bool((getattr(buf, name)[kept - short:kept] == -7).all()), name
