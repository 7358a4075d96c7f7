"""Many scored rows in one pass over K (score_once.cu): equal keys get bit-equal scores whatever stands around them, and a key
that is infinite or not a number changes no other key's score but through the rows it takes out."""
import numpy as np
import pytest
import torch

import parity
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [([2048], 64, 28, 4, 128), ([1500, 700, 333], 40, 8, 2, 64), ([900, 4096], 9, 4, 4, 128)]


def _problem(lens, rows, hq, hkv, d, sharp):
    """Keys of very different lengths, so that the maxima of neighbouring groups of keys differ; logits `sharp` times as large."""
    p = W.random_problem(seed=sum(lens), lens=lens, rows=[rows] * len(lens), keeps=[n // 2 for n in lens], num_q_heads=hq, num_kv_heads=hkv, head_dim=d,
                         hidden=64, trailing_rows=False)
    gen = torch.Generator().manual_seed(rows)
    p.k.mul_(torch.randn(p.total_tokens, 1, 1, generator=gen).mul(0.5).exp().to(torch.bfloat16))
    p.q.mul_(sharp)
    return p, gen


# From logits that stay within 2^±100 as they are, over rows in which some groups do, to ones far beyond.
@pytest.mark.parametrize("lens,rows,hq,hkv,d", SHAPES)
@pytest.mark.parametrize("sharp", [0.3, 2.0, 8.0, 30.0, 3e4, 1e9])
def test_equal_keys_have_one_score_and_the_first_is_kept(lens, rows, hq, hkv, d, sharp):
    p, gen = _problem(lens, rows, hq, hkv, d, sharp)
    p.causal = False
    cu = p.cu_seqlens.tolist()
    twins = []  # [groups, 3] ascending token indices of the batch, scattered over all of a sequence
    for a, n in zip(cu, lens):
        twins.append(a + torch.randperm(n, generator=gen)[:n // 4 // 3 * 3].view(-1, 3).sort(dim=1).values)
        p.k[twins[-1]] = p.k[twins[-1][:, :1]]
    buf = parity.to_device(p)
    buf.score()
    scores = buf.scores.cpu()
    bits = scores.view(torch.int32)
    for t in twins:
        assert torch.equal(bits[t], bits[t[:, :1]].expand(-1, 3)), f"{int((bits[t] != bits[t[:, :1]]).sum())} of {t.numel()} differ"
    if sharp < 100:
        parity.assert_scores_close(buf.scores, parity.oracle_scores(p))
    for a, n in zip(cu, lens):
        assert abs(float(scores[a:a + n].double().sum()) - 1) < 1e-5
    # As many survivors as put the border inside a group of three.
    keeps = []
    for t, a, n in zip(twins, cu, lens):
        own = scores[a:a + n]
        middle = own[t[:, 0] - a].sort().values[len(t) // 2]
        keeps.append(int((own > middle).sum()) + 2)
    p.keep_counts = torch.tensor(keeps, dtype=torch.int32)
    buf = parity.to_device(p)
    buf.prune()
    torch.cuda.synchronize()
    assert int(buf.device_status) == 0 and torch.equal(buf.scores.cpu().view(torch.int32), bits)
    kept = torch.zeros(p.total_tokens, dtype=torch.bool)
    cu_keep = buf.cu_keep.tolist()
    for b, a in enumerate(cu[:-1]):
        kept[a + buf.keep_idx[cu_keep[b]:cu_keep[b + 1]].cpu()] = True
    for t in twins:
        assert bool((kept[t].int().diff(dim=1) <= 0).all())


def _reference(p):
    """Eq. 4 in 64 bits; a row and head with an infinite or undefined logit has no softmax: NaN at that key, 0 elsewhere."""
    cu, cuq = p.cu_seqlens.tolist(), p.cu_qlens.tolist()
    hq, hkv = p.q.shape[1], p.k.shape[1]
    out = torch.zeros(p.total_tokens, dtype=torch.float64)
    for b, a in enumerate(cu[:-1]):
        n, r0, r1 = cu[b + 1] - a, cuq[b], cuq[b + 1]
        k = p.k[a:a + n].double().repeat_interleave(hq // hkv, dim=1)
        z = torch.einsum("rhd,nhd->rhn", p.q[r0:r1].double(), k) * p.softmax_scale
        hidden = torch.arange(n)[None, :] > p.q_idx[r0:r1, None]
        z = z.masked_fill(hidden[:, None, :], -np.inf)
        bad = z.isnan() | (z == np.inf)
        lost = bad.any(dim=2, keepdim=True)
        w = torch.softmax(torch.where(lost, torch.zeros_like(z), z), dim=2)
        w = torch.where(lost, torch.zeros_like(w), w).masked_fill(bad, np.nan)
        out[a:a + n] = w.sum(dim=(0, 1)) / (hq * (r1 - r0))
    return out


@pytest.mark.parametrize("lens,rows,hq,hkv,d", SHAPES)
@pytest.mark.parametrize("value,path", [(np.inf, 0), (np.nan, 0), (np.inf, fastav.FASTAV_SCORE_PATH_WIDE)])  # one pass, and the two sweeps beside it
def test_an_infinite_key_leaves_the_others_alone(lens, rows, hq, hkv, d, value, path):
    p, _ = _problem(lens, rows, hq, hkv, d, 0.5)
    p.q[:, ::2, 0] = 1    # +infinity for the even heads of every row that sees the key,
    p.q[:, 1::2, 0] = -1  # -infinity for the odd ones: a key without weight
    cu = p.cu_seqlens.tolist()
    for a, n in zip(cu, lens):
        p.k[[a + n // 3, a + n // 2], :, 0] = value
    buf = parity.to_device(p, extra_flags=path)
    buf.score()
    got, want = buf.scores.cpu().double(), _reference(p)
    assert torch.equal(got.isnan(), want.isnan()), f"{int(got.isnan().sum())} scores are NaN, {int(want.isnan().sum())} should be"
    there = ~want.isnan()
    err = (got - want).abs()[there]
    assert bool((err <= parity.SCORE_RTOL * want[there].abs() + parity.SCORE_ATOL).all()), float(err.max())
