"""The prune call's paths for short sequences and their borders: the few-rows cluster kernel (up to 4 scored rows, 2,048 tokens),
the one-pass score in tensor memory (up to 4,096 tokens; one round of clusters or several), the cluster selection from partial
sums and from finished scores, rows gathered by the selecting blocks or by the compaction, the mask's emission with one kernel
or two.  Against the oracle; keep sets as parity.py judges them (scores within its bound, equal keys bit-equal)."""
import numpy as np
import pytest
import torch

import oracle
import parity
import timing
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu


def _check(lens, rows, hq, hkv, d, hid=64, keep=0.5, **more):
    p = W.random_problem(seed=sum(lens) + hq + rows, lens=lens, rows=[min(rows, n) for n in lens], keeps=[max(min(1, n), int(n * keep)) for n in lens],
                         num_q_heads=hq, num_kv_heads=hkv, head_dim=d, hidden=hid, duplicate_keys=2, **more)
    p.protect_rows = rows % 2 == 1
    protect = (torch.arange(p.total_tokens) % 29 == 3).to(torch.uint8) if hq % 8 == 0 else None
    buf = parity.to_device(p, protect=protect)
    buf.prune()
    torch.cuda.synchronize()
    stats = parity.check_fused_against_oracle(p, buf, parity.oracle_prune(p, protect=protect), protect=protect, what=f"{lens} x {rows}")
    assert stats["device_status"] & ~fastav.FASTAV_DEV_PROTECT_OVERFLOW == 0  # (that bit is checked with the rest)


# Few rows: ends of fragments (8, 16), segments (32) and of the token range; 1-4 rows; groups of 1, 2, 4, 7; clusters of 16 down to 1
# (more sequences than clusters that run at once), and batches beyond the number of SMs on either side of 512 tokens.
@pytest.mark.parametrize("lens,rows,hq,hkv,d", [
    ([1], 1, 2, 1, 64), ([15, 33, 8], 2, 4, 4, 64), ([511, 512, 513], 3, 8, 2, 128), ([2047], 4, 28, 4, 128), ([2048], 1, 28, 4, 128),
    ([2049], 1, 28, 4, 128), ([1025, 0, 31] * 4, 1, 8, 4, 64), ([200, 64] * 20, 2, 4, 2, 64), ([70] * 149, 1, 4, 1, 64), ([512] * 2 + [9] * 150, 1, 4, 2, 64),
    ([513] + [9] * 150, 1, 4, 2, 64),
])
def test_few_rows(lens, rows, hq, hkv, d):
    _check(lens, rows, hq, hkv, d)


# Many rows, one pass: ends of key tiles (128) and of the range, row tiles that are not full, groups of 1 to 16, one round of
# clusters and several, and the two-sweep path next to it (4,097 tokens; a group of 17).
@pytest.mark.parametrize("lens,rows,hq,hkv,d", [
    ([5], 5, 2, 2, 64), ([127, 128, 129], 9, 8, 8, 64), ([1000, 3], 33, 28, 4, 128), ([4095], 8, 8, 2, 128), ([4096], 17, 16, 1, 64), ([4097], 8, 8, 2, 128),
    ([2048, 100], 130, 4, 2, 64), ([300], 12, 17, 1, 64), ([512] * 40, 32, 28, 4, 128), ([1024, 640, 999] * 5, 32, 8, 8, 64), ([256] * 24, 128, 16, 4, 64),
    ([4200, 4097, 4150], 40, 32, 4, 64), ([5000, 4600], 9, 8, 2, 64), ([5000, 4900], 9, 8, 2, 64),  # chunks for about one length, and for ragged ones
])
@pytest.mark.parametrize("trailing", [True, False])
def test_many_rows(lens, rows, hq, hkv, d, trailing):
    _check(lens, rows, hq, hkv, d, trailing_rows=trailing)


# Rows gathered by the selecting blocks (little per block) or by the compaction (more), and rows per warp around the ring's depth.
@pytest.mark.parametrize("n,keep,hid", [(64, 1.0, 8), (512, 0.9, 512), (1500, 0.7, 64), (1500, 0.9, 2048), (2048, 0.1, 3584), (2048, 1.0, 1024)])
@pytest.mark.parametrize("rows", [1, 8])
def test_gather_by_either_kernel(n, keep, hid, rows):
    _check([n, n // 3], rows, 8, 2, 64, hid=hid, keep=keep)


@pytest.mark.parametrize("total,batch", [(1, 1), (4095, 3), (4097, 1), ((1 << 18), 7), ((1 << 18) + 1, 7), ((1 << 17), 7), ((1 << 17) + 1, 7), (3000, 148), (3000, 149), (300_000, 513)])
@pytest.mark.parametrize("offset", [0, 1])  # masks that are not 16-byte aligned
def test_mask_emission(total, batch, offset):
    rng = np.random.default_rng(total + offset)
    cu = np.concatenate([[0], np.sort(rng.integers(0, total + 1, batch - 1)), [total]]).astype(np.int32)
    mask = (rng.random(total) < 0.6).astype(np.uint8)
    ref_idx, ref_cu = oracle.select_mask(mask, cu)
    kept = int(ref_cu[-1])
    params = fastav.make_params(batch=batch, total_tokens=total, max_seqlen=int(np.diff(cu).max()), total_q=0, max_qlen=0, total_keep=kept,
                                max_keep=kept, num_q_heads=4, num_kv_heads=2, head_dim=64, hidden=64)
    held = torch.zeros(total + 16, dtype=torch.uint8, device="cuda")
    held[offset:offset + total] = torch.from_numpy(mask).cuda()
    idx = torch.full((kept + 8,), -7, dtype=torch.int32, device="cuda")
    cu_keep, status = torch.empty(batch + 1, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(max(256, fastav.fastav_workspace_bytes(params)), dtype=torch.uint8, device="cuda")
    fastav.fastav_select_mask(params, held[offset:offset + total], torch.from_numpy(cu).cuda(), idx, cu_keep, ws, status)
    torch.cuda.synchronize()
    assert int(status) == 0 and cu_keep.cpu().tolist() == ref_cu.tolist()
    assert np.array_equal(idx.cpu().numpy(), np.concatenate([ref_idx, np.full(8, -7)]))


# Who gathers also depends on how many sequences there are, and on what one block's slice of the tokens can hold.
@pytest.mark.parametrize("batch,n,keep", [(7, 1000, 0.05), (8, 1000, 0.05), (8, 1000, 0.3), (15, 400, 0.3), (16, 400, 0.3), (150, 120, 0.5)])
@pytest.mark.parametrize("rows", [1, 8])
def test_gather_of_batches(batch, n, keep, rows):
    _check([n] * batch, rows, 8, 2, 64, hid=64, keep=keep)


# The few-rows kernel ranks a slice's keys by counting while (tokens x tokens of a slice) is small: both sides of that border for
# clusters of 16, 8, 4 and 2, lengths that are no multiple of 4, one token, all scores equal (the lower index wins) and not.
@pytest.mark.parametrize("lens", [[1], [2, 3, 5], [513], [767], [768], [769], [511] * 8, [577] * 8, [288] * 16, [289, 7] * 8, [143] * 34, [145, 0] * 17])
@pytest.mark.parametrize("equal", [False, True])
def test_selection_by_counting(lens, equal):
    p = W.random_problem(seed=sum(lens), lens=lens, rows=[min(1, n) for n in lens], keeps=[(2 * n + 2) // 3 for n in lens], num_q_heads=8, num_kv_heads=2,
                         head_dim=64, hidden=64, duplicate_keys=2)
    if equal:
        p.q.zero_()
    protect = (torch.arange(p.total_tokens) % 3 != 1).to(torch.uint8) if len(lens) % 3 == 1 else None  # now and then more than are kept
    buf = parity.to_device(p, protect=protect)
    buf.prune()
    torch.cuda.synchronize()
    stats = parity.check_fused_against_oracle(p, buf, parity.oracle_prune(p, protect=protect), protect=protect, what=f"{lens} equal {equal}")
    assert stats["device_status"] & ~fastav.FASTAV_DEV_PROTECT_OVERFLOW == 0


# The compaction keeps the bounds of up to 31 sequences in a warp's lanes; warps with one row, a few, and more than 32.
@pytest.mark.parametrize("batch,n", [(1, 40), (1, 592), (30, 50), (31, 50), (32, 50), (31, 1000), (33, 1000)])
def test_gather_bounds_by_lane(batch, n):
    _check([n if b % 5 else 0 for b in range(1, batch)] + [n], 1, 4, 2, 64, hid=3584, keep=0.8)


# The flags that the selection reads, from the keys (by counting and by digits) and from partial sums; scored rows around the borders of
# a block's tokens.
@pytest.mark.parametrize("lens", [[63], [512], [767], [2047], [300, 5] * 4, [1000] * 9, [140] * 35], ids=lambda v: f"{len(v)}x{max(v)}")
@pytest.mark.parametrize("rows", [2, 9])
@pytest.mark.parametrize("lowest,global_idx,by_rows,lse", [(True, False, False, False), (False, True, False, True), (False, False, True, False), (True, True, True, True)])
def test_flags_of_the_selection(lens, rows, lowest, global_idx, by_rows, lse):
    p = W.random_problem(seed=sum(lens) + rows, lens=lens, rows=[min(rows, n) for n in lens], keeps=[(i + 1) * n // (len(lens) + 1) for i, n in enumerate(lens)],
                         num_q_heads=8, num_kv_heads=2, head_dim=64, hidden=64, duplicate_keys=2, trailing_rows=False)
    cuq = p.cu_qlens.tolist()
    for b, n in enumerate(lens):
        edges = sorted({j for j in (31, 32, 47, 48, 255, 256) if j < n - 1})[-(cuq[b + 1] - cuq[b]) + 1:] + [n - 1]
        p.q_idx[cuq[b + 1] - len(edges):cuq[b + 1]] = torch.tensor(edges, dtype=torch.int32)
        p.q_idx[cuq[b]:cuq[b + 1]] = p.q_idx[cuq[b]:cuq[b + 1]].sort().values
    protect = (torch.arange(p.total_tokens) % 29 == 3).to(torch.uint8) if len(lens) % 2 else None
    parity.check_prune_under_flags(p, lowest, global_idx, by_rows, lse, protect, f"{lens[0]} x {len(lens)}, {rows} rows")


def test_the_scores_of_a_short_sequence_alone():
    """300 tokens of a small model: without a selection and a gather behind, by far less than with them (the next call's launch is hidden)."""
    buf = parity.to_device(W.random_problem(seed=2, lens=[300], rows=[1], keeps=[150], num_q_heads=8, num_kv_heads=2, head_dim=64, hidden=512))
    assert timing.us_per_call(buf.score) < 0.6 * timing.us_per_call(buf.prune)
