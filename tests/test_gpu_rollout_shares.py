"""The rollout's work is shared out by size: statistics in equal runs (a row block split over up to four blocks), the map in
strips of 1 to 5 units of 32 columns (which are not tile-aligned), the product's long K loops in parts.  The sizes below take
every strip width under either mask, one, several and cut row blocks, and KV groups of 1, 2, 3 and 7 (the K slots' reuse).

Reference: the definition in double precision (PyTorch).  Map: the logits are fp32 sums of 64 or 128 exact products of bf16
values, |error| <= 128 * 2^-24 * sum |q k| * scale, some 1e-4 in the exponent for unit normals, and the exponentials add
3e-7: 2e-3 relative.  Product: each factor carries 16 mantissa bits, a few 1e-5 per layer, 1e-3 allowed (as in
test_gpu_rollout.py)."""
import pytest
import torch

from paper_2601_13143_b200 import fastav
from test_gpu_rollout import _layers, _params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,hq,hkv,d,causal", [
    (31, 3, 1, 128, True), (1024, 4, 4, 64, True), (1097, 6, 3, 128, True), (1473, 9, 3, 64, True), (1921, 2, 1, 128, True),
    (2177, 7, 1, 128, True), (2304, 5, 5, 128, True), (2305, 4, 4, 64, True), (769, 8, 8, 128, False), (1100, 40, 40, 64, False),
    (1536, 3, 1, 128, False), (1601, 4, 2, 128, False),
])
def test_every_share_of_the_work(n, hq, hkv, d, causal):
    alpha, scale, layers = 0.7, d**-0.5, 2
    qk = [(q.cuda(), k.cuda()) for q, k in _layers(n + hq, n, hq, hkv, d, layers)]
    state = torch.empty(fastav.fastav_rollout_state_bytes(n), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    p = _params(n, hq, hkv, d, *qk[0], scale, causal)
    ws = torch.full((fastav.fastav_rollout_workspace_bytes(p),), 255, dtype=torch.uint8, device="cuda")  # all NaN
    fastav.fastav_rollout_begin(n, state)
    ref = torch.eye(n, dtype=torch.float64, device="cuda")
    for l, (q, k) in enumerate(qk):
        out = torch.full((n, n), float("nan"), device="cuda")
        fastav.fastav_rollout_layer(p, q, k, alpha, l, state, ws, map_out_opt=out, device_status=status)
        a = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        hidden = torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1)
        for h in range(hq):
            z = q[:, h].double() @ k[:, h // (hq // hkv)].double().T * scale
            a += torch.softmax(z.masked_fill(hidden, float("-inf")) if causal else z, dim=1) / hq
        assert ((out.double() - a).abs() <= 2e-3 * a + 1e-12).all()
        ref = (alpha * a + (1 - alpha) * torch.eye(n, dtype=torch.float64, device="cuda")) @ ref
    imp, r = torch.empty(n, device="cuda"), torch.full((n, n), float("nan"), device="cuda")
    fastav.fastav_rollout_read(n, layers, state, imp, r)
    assert int(status) == 0
    assert ((r.double() - ref).abs() <= 1e-3 * ref + 1e-12).all()
    assert ((imp.double() - ref.mean(0)).abs() <= 1e-3 * ref.mean(0)).all()
