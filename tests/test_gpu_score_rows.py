"""Few scored rows on sequences beyond 2,048 tokens (score_rows.cu, and the selection from its logits in select_long.cu): ends of tiles of
64 tokens and of a block's slice, up to 32 sequences and more (the padded list of tiles), 1 to 128 query rows per KV head, empty
sequences and ones without scored rows, head-major and packed keys.  Against the oracle, and the separate calls against the fused one."""
import pytest
import torch

import parity
import test_gpu_equal_keys as equal_keys
import timing
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu


def _problem(lens, rows, hq, hkv, d, **more):
    rows = [min(rows, n) if i % 5 != 3 else 0 for i, n in enumerate(lens)]
    return W.random_problem(seed=sum(lens) + hq, lens=lens, rows=rows, keeps=[(i % 3 + 1) * n // 4 for i, n in enumerate(lens)], num_q_heads=hq,
                            num_kv_heads=hkv, head_dim=d, hidden=64, duplicate_keys=2, **more)


@pytest.mark.parametrize("lens,rows,hq,hkv,d", [
    ([2049], 1, 28, 4, 128), ([2111, 64, 63, 65, 0, 1], 4, 8, 2, 64), ([4096, 4097], 2, 16, 16, 64), ([8257, 2050, 128], 3, 32, 4, 128), ([33000], 1, 8, 2, 64),
    ([2500] * 3 + [300] * 5, 4, 32, 1, 64), ([2060] * 32, 1, 4, 2, 64), ([2060, 31, 0] * 11, 2, 4, 2, 128), ([2049] * 75, 1, 4, 2, 64), ([640] * 150, 1, 4, 1, 128),
])
@pytest.mark.parametrize("trailing", [True, False])
def test_few_rows_of_long_sequences(lens, rows, hq, hkv, d, trailing):
    p = _problem(lens, rows, hq, hkv, d, trailing_rows=trailing)
    buf = parity.to_device(p)
    buf.prune()
    torch.cuda.synchronize()
    stats = parity.check_fused_against_oracle(p, buf, parity.oracle_prune(p), what=f"{lens[0]} x {len(lens)}")
    assert stats["device_status"] & ~fastav.FASTAV_DEV_PROTECT_OVERFLOW == 0
    fused = buf.scores.clone()
    buf.scores.fill_(-1.0)
    buf.score()
    torch.cuda.synchronize()
    assert torch.equal(buf.scores.view(torch.int32), fused.view(torch.int32))
    # The statistics by themselves: fp32 sums of up to 33,000 terms in a tree, and the logits' fp32 rounding (2^-24 of at most 128 products).
    if p.q_idx.numel():
        lse = torch.empty(p.q.shape[0], hq, device="cuda")
        fastav.fastav_lse(buf.params, buf.q, buf.q_idx, buf.cu_qlens, buf.k, buf.cu_seqlens, lse, buf.workspace, buf.device_status)
        torch.testing.assert_close(lse.cpu().double(), parity.log_sum_exp(p).double(), rtol=0, atol=2e-5)


@pytest.mark.parametrize("layout", ["packed", "head_major"])
def test_strided_keys(layout):
    p = _problem([2300, 2100], 2, 8, 4, 64)
    n, heads, d = p.k.shape
    if layout == "packed":  # a view into a projection output that holds more than the keys
        held = torch.zeros(n, heads + 3, d, dtype=p.k.dtype, device="cuda")
        k = held[:, 2:2 + heads]
    else:
        held = torch.zeros(heads, n, d, dtype=p.k.dtype, device="cuda")
        k = held.transpose(0, 1)
    k.copy_(p.k)
    plain = parity.to_device(p)
    plain.prune()
    buf = fastav.make_buffers(q=plain.q, q_idx=plain.q_idx, cu_qlens=plain.cu_qlens, k=k, v=plain.v, cu_seqlens=plain.cu_seqlens, keep_counts=plain.keep_counts,
                              hidden=plain.hidden, pos=plain.pos, softmax_scale=p.softmax_scale, flags=parity.flags_of(p))
    buf.prune()
    torch.cuda.synchronize()
    assert int(buf.device_status) == int(plain.device_status)
    for name in ("scores", "keep_idx", "cu_keep", "hidden_out", "pos_out", "k_out", "v_out"):
        assert torch.equal(getattr(buf, name), getattr(plain, name)), name


@pytest.mark.parametrize("lens", [
    [2050] + [70] * 32, [64] * 40 + [0] * 3 + [2113, 1, 0, 65], [3, 130] * 500 + [2049] + [64] * 22, [2049] + [40] * 1024, [65, 0, 1] * 700 + [2300, 0, 0],
    [5] * 33000 + [2049, 7],
], ids=len)
@pytest.mark.parametrize("rows", [1, 3])
def test_many_sequences(lens, rows):
    """The table of a block: 33 sequences, one entry per thread and several, its last entry, two and three sequences per entry, more than a warp."""
    p = _problem(lens, rows, 2, 1, 64)
    buf = parity.to_device(p)
    buf.prune()
    torch.cuda.synchronize()
    parity.check_fused_against_oracle(p, buf, parity.oracle_prune(p), what=f"{len(lens)} sequences")


def test_a_cut_sequence_among_many_is_reported():
    p = _problem([2100] + [50] * 40, 1, 2, 1, 64)
    buf = parity.to_device(p)
    buf.params.max_seqlen = 2080
    buf.prune()
    torch.cuda.synchronize()
    assert int(buf.device_status) & fastav.FASTAV_DEV_SHAPE_MISMATCH


def _score_us(lens, rows):
    """A score call, heads as in the benchmark's larger decoder."""
    total, cu = sum(lens), lambda v: torch.tensor([0] + v, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    k = torch.randn(total, 8, 128, dtype=torch.bfloat16, device="cuda")
    buf = fastav.make_buffers(q=torch.randn(sum(rows), 32, 128, dtype=torch.bfloat16, device="cuda"), q_idx=torch.tensor([n - 1 for n, r in zip(lens, rows) if r], dtype=torch.int32).cuda(),
                              cu_qlens=cu(rows), k=k, v=None, cu_seqlens=cu(lens), keep_counts=torch.ones(len(lens), dtype=torch.int32).cuda(), lens=lens, rows=rows,
                              keeps=[1] * len(lens))
    return timing.us_per_call(buf.score)


def test_a_long_sequence_among_many_is_shared_out():
    """64 sequences against 32 with as many tokens and the same longest one: every block's share is as large.  Twice the time leaves room for
    finding the sequences; two or three blocks with the long one to themselves took ten times as long."""
    assert _score_us([20000] + [500] * 63, [1] * 64) < 2 * _score_us([20000] + [1016] * 30 + [1020], [1] * 32)


def test_keys_of_sequences_without_scored_rows_are_not_read():
    """Half of the sequences without: the keys are what the call's time goes on, so it should take well below what it takes with all of them."""
    assert _score_us([3000] * 40, [0, 1] * 20) < 0.8 * _score_us([3000] * 40, [1] * 40)


@pytest.mark.parametrize("lens,rows,hq,hkv,d", [([2049], 1, 28, 4, 128), ([5000, 2100, 70], 3, 8, 2, 64)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_an_infinite_key_leaves_the_others_alone(lens, rows, hq, hkv, d, value):
    """By the separate kernels and by the selection from the logits: +infinity for the even heads, -infinity for the odd ones, in two keys of each sequence."""
    p, _ = equal_keys._problem(lens, rows, hq, hkv, d, 0.5)
    p.q[:, ::2, 0], p.q[:, 1::2, 0] = 1, -1
    for a, n in zip(p.cu_seqlens.tolist(), lens):
        p.k[[a + n // 3, a + n // 2], :, 0] = value
    want = equal_keys._reference(p)
    there = ~want.isnan()
    buf = parity.to_device(p)
    for call in (buf.score, buf.prune):
        buf.scores.fill_(-1.0)
        call()
        got = buf.scores.cpu().double()
        assert torch.equal(got.isnan(), want.isnan()), f"{int(got.isnan().sum())} scores are NaN, {int(want.isnan().sum())} should be"
        err = (got - want).abs()[there]
        assert bool((err <= parity.SCORE_RTOL * want[there].abs() + parity.SCORE_ATOL).all()), float(err.max())


@pytest.mark.parametrize("hq,hkv,rows", [(28, 4, 4), (32, 8, 4), (32, 8, 2)])
def test_a_prune_call_takes_no_longer_than_its_parts(hq, hkv, rows):
    """1 x 2,500 tokens: the selection from the logits against score, select and compact one after the other."""
    p = W.random_problem(seed=4, lens=[2500], rows=[rows], keeps=[1750], num_q_heads=hq, num_kv_heads=hkv, head_dim=128, hidden=3584)
    buf = parity.to_device(p)

    def parts(stream):
        buf.score(stream)
        buf.select(stream)
        buf.compact(stream)

    assert timing.us_per_call(buf.prune) < 1.05 * timing.us_per_call(parts)
