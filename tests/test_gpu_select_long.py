"""Scores and selection of sequences beyond 2,048 tokens from the sweeps' partial sums by clusters (select_long.cu), against the
oracle: ends of the range and of a block's slice, clusters of 16 to 2 and the paths next to them (too many sequences, too
long), keys that share one bin of every pass, more protected tokens than are kept, empty and short sequences beside long ones."""
import pytest
import torch

import parity
import timing
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu

LENS = [[2049], [2050, 1, 0, 2111], [4097], [8191, 8193], [16384], [32768], [32769], [2600] * 7, [2600] * 8, [2051] * 15, [2051] * 16, [2500, 0, 1] * 11,
        [2100] * 34, [4097] * 34, [2049] * 75]


@pytest.mark.parametrize("lens", LENS, ids=lambda v: f"{len(v)}x{max(v)}")
@pytest.mark.parametrize("equal", [False, True])
def test_select_from_sums(lens, equal):
    rows = [min(9, n) for n in lens]
    shares = [0.4, 0.0, 1.0, 0.01, 0.9]
    p = W.random_problem(seed=sum(lens), lens=lens, rows=rows, keeps=[min(n, int(round(shares[i % 5] * n))) for i, n in enumerate(lens)], num_q_heads=4,
                         num_kv_heads=2, head_dim=64, hidden=64, duplicate_keys=2)
    if equal:  # every token of a sequence that all its rows see has the same score
        p.q.zero_()
    protect = (torch.arange(p.total_tokens) % 31 == 5).to(torch.uint8) if len(lens) % 2 else None
    buf = parity.to_device(p, protect=protect)
    buf.prune()
    torch.cuda.synchronize()
    stats = parity.check_fused_against_oracle(p, buf, parity.oracle_prune(p, protect=protect), protect=protect, what=f"{lens} equal {equal}")
    assert stats["device_status"] & ~fastav.FASTAV_DEV_PROTECT_OVERFLOW == 0


@pytest.mark.parametrize("lens", [[2049], [8191, 8193], [2600] * 8, [2051, 40] * 8, [2100] * 34, [4097] * 46], ids=lambda v: f"{len(v)}x{max(v)}")
@pytest.mark.parametrize("lowest,global_idx,by_rows,lse", [(True, False, False, False), (False, True, False, True), (False, False, True, False), (True, True, True, True)])
def test_flags_of_the_selection(lens, lowest, global_idx, by_rows, lse):
    """Scored rows lie on both sides of the borders that a block's slice has in clusters of 16, 8, 4 and 2."""
    rows = [sorted({j for blocks in (16, 8, 4, 2) for j in ((n + blocks - 1) // blocks + 31 & ~31, ((n + blocks - 1) // blocks + 31 & ~31) - 1) if j < n} | {n - 1})
            for n in lens]
    p = W.random_problem(seed=sum(lens) + 1, lens=lens, rows=[len(r) for r in rows], keeps=[(i + 1) * n // (len(lens) + 1) for i, n in enumerate(lens)],
                         num_q_heads=4, num_kv_heads=2, head_dim=64, hidden=64, duplicate_keys=2)
    p.q_idx = torch.tensor([j for r in rows for j in r], dtype=torch.int32)
    protect = (torch.arange(p.total_tokens) % 37 == 5).to(torch.uint8) if len(lens) % 4 else None
    parity.check_prune_under_flags(p, lowest, global_idx, by_rows, lse, protect, f"{lens[0]} x {len(lens)}")


# The first pass looks at scores from 2^-63 to 2 in bins of 1/32 octave (one scored row and up to 2,048 tokens, in the few-rows kernel: 1/64).  `crowd`: a hundred different scores within one or two bins and one
# block's slice, the k-th largest among them (more than a block sends; some 40 per block where the bin has more); `small`: all scores but one
# below 2^-63; `hidden`: most tokens behind the scored rows (score 0) and k beyond the others; `above`: the k-th largest is protected.
@pytest.mark.parametrize("kind", ["crowd", "wide_crowd", "small", "hidden", "above"])
@pytest.mark.parametrize("lens", [[1500], [2000, 900], [2049], [5000, 2100], [17000]], ids=lambda v: f"{len(v)}x{max(v)}")
@pytest.mark.parametrize("rows", [1, 9])
@pytest.mark.parametrize("lowest", [False, True])
def test_window_of_the_first_pass(kind, lens, rows, lowest):
    p = W.random_problem(seed=sum(lens) + rows, lens=lens, rows=[rows] * len(lens), keeps=[n // 2 for n in lens], num_q_heads=2, num_kv_heads=1, head_dim=64,
                         hidden=64)
    gen = torch.Generator().manual_seed(rows)
    p.softmax_scale = 1.0
    p.q.zero_()
    p.k.zero_()
    p.q[..., 0], p.q[..., 1] = 8.0, 2.0 ** -13
    protect, keeps, start = None, [], 0
    for b, n in enumerate(lens):
        z = (torch.rand(n, generator=gen) * 2 - 1).bfloat16()
        tail = torch.zeros(n)
        if kind == "crowd" or kind == "wide_crowd":
            crowd = torch.arange(300, 400) if kind == "crowd" else torch.arange(100, n, 7)[:400]
            z[crowd], tail[crowd] = 0.0, torch.arange(len(crowd)).float() % 128
            above = int((z < 0).sum() if lowest else (z > 0).sum())
            keeps.append(above + len(crowd) // 2)
        elif kind == "small":
            z[5] = 7.5
            keeps.append(n // 3)
        else:
            keeps.append(n // 3)
        if kind == "hidden":
            p.q_idx[b * rows:(b + 1) * rows] = torch.arange(n // 5, n // 5 + rows)
        p.k[start:start + n, 0, 0], p.k[start:start + n, 0, 1] = z, tail.bfloat16()
        start += n
    if kind == "above":
        protect = (torch.arange(p.total_tokens) % 2).to(torch.uint8)
    p.keep_counts = torch.tensor(keeps, dtype=torch.int32)
    parity.check_prune_under_flags(p, lowest, False, True, False, protect, f"{kind} {lens[0]} x {len(lens)}")


def test_scores_close_together_take_no_longer():
    """1 x 3,633 tokens with scores from far apart to within a few percent: the threshold's first bin holds from some 60 keys to more than a
    thousand.  Ranking them by counting up to 512 of them made one of these calls 1.3 times as long as another; another pass is a tenth."""
    medians = []
    for spread in (0.5, 1.0, 1.15, 1.3, 1.5, 1.75):
        gen = torch.Generator(device="cuda").manual_seed(3)
        normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
        one = lambda *v: torch.tensor(v, dtype=torch.int32, device="cuda")
        k = normal(3633, 4, 128)
        buf = fastav.make_buffers(q=normal(23, 32, 128) * spread, q_idx=torch.arange(3610, 3633, dtype=torch.int32, device="cuda"), cu_qlens=one(0, 23), k=k, v=None,
                                  cu_seqlens=one(0, 3633), keep_counts=one(1453), lens=[3633], rows=[23], keeps=[1453])
        medians.append(timing.us_per_call(buf.prune))
    assert max(medians) < 1.12 * min(medians), medians
