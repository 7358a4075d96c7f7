"""Rows read ahead of the selection (compact_placed_kernel, behind the few-rows kernel): against the oracle, and bit for bit against the
gather that starts from the keep list.  One token up to what shared memory holds, up to 31 sequences and 32, empty ones, nothing and
everything kept, more protected tokens than are kept, selection by counting and by digits, keys and values packed and head-major, a call
without values or positions, tokens ahead of the first sequence, and index arrays that promise less than they hold."""
import pytest
import torch

import parity
import timing
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu

OUT = ("keep_idx", "cu_keep", "hidden_out", "pos_out", "k_out", "v_out")


def _problem(lens, keeps, hid=1024, hq=4, hkv=2, d=128, rows=1):
    return W.random_problem(seed=sum(lens) + hid, lens=lens, rows=[min(rows, n) for n in lens], keeps=keeps, num_q_heads=hq, num_kv_heads=hkv, head_dim=d,
                            hidden=hid, duplicate_keys=2)


def _both(buf):
    """The call as it is, and with the gather by loads and stores, which starts from the list."""
    got = []
    for flag in (0, fastav.FASTAV_COMPACT_PATH_LOADSTORE):
        buf.params.flags = buf.params.flags & ~fastav.FASTAV_COMPACT_PATH_LOADSTORE | flag
        for name in OUT:
            if getattr(buf, name) is not None:
                getattr(buf, name).view(torch.uint8).fill_(0x55)
        buf.device_status.zero_()
        buf.prune()
        torch.cuda.synchronize()
        got.append({name: getattr(buf, name).clone() for name in OUT if getattr(buf, name) is not None} | {"status": buf.device_status.clone()})
    for name in got[0]:
        assert torch.equal(got[0][name].view(torch.uint8), got[1][name].view(torch.uint8)), name
    return got[0]


@pytest.mark.parametrize("lens,keep,hid,hkv,d", [
    ([1], 1.0, 1024, 2, 128), ([147, 1], 0.7, 3584, 4, 128), ([149], 0.8, 3584, 4, 128), ([744], 0.8, 3584, 4, 128), ([2048], 0.9, 4096, 8, 128),
    ([2048, 300], 0.8, 2048, 2, 128), ([100] * 31, 0.8, 1024, 4, 64), ([100] * 32, 0.8, 1024, 4, 64), ([300, 0, 5] * 5, 0.9, 1024, 2, 128), ([1500], 0.9, 512, 2, 128),
    ([1500], 0.9, 504, 2, 128),
])
def test_against_the_oracle(lens, keep, hid, hkv, d):
    p = _problem(lens, [int(keep * n) if i % 4 else n * int(keep * 10) // 10 for i, n in enumerate(lens)], hid, 2 * hkv, hkv, d)
    protect = (torch.arange(p.total_tokens) % 3 != 1).to(torch.uint8) if len(lens) % 3 == 0 else None
    buf = parity.to_device(p, protect=protect)
    buf.prune()
    torch.cuda.synchronize()
    parity.check_fused_against_oracle(p, buf, parity.oracle_prune(p, protect=protect), protect=protect, what=f"{lens}")
    _both(buf)


@pytest.mark.parametrize("keeps", [[0, 500], [700, 0], [700, 500], [1, 1]])
@pytest.mark.parametrize("protected", [False, True])
def test_nothing_and_everything_kept(keeps, protected):
    p = _problem([700, 500], keeps)
    _both(parity.to_device(p, protect=(torch.arange(1200) % 2).to(torch.uint8) if protected else None))


@pytest.mark.parametrize("layout", ["head_major", "no_values", "no_positions", "no_hidden"])
def test_layouts(layout):
    p = _problem([600, 333], [500, 200], hkv=4, hq=4)
    buf = parity.to_device(p)
    if layout == "head_major":
        k, v = (torch.empty(4, 933, 128, dtype=torch.bfloat16, device="cuda").transpose(0, 1) for _ in range(2))
        k.copy_(buf.k), v.copy_(buf.v)
        buf = fastav.make_buffers(q=buf.q, q_idx=buf.q_idx, cu_qlens=buf.cu_qlens, k=k, v=v, cu_seqlens=buf.cu_seqlens, keep_counts=buf.keep_counts, hidden=buf.hidden,
                                  pos=buf.pos, softmax_scale=p.softmax_scale, flags=parity.flags_of(p))
    elif layout == "no_values":
        buf.v = buf.v_out = None
    elif layout == "no_positions":
        buf.pos = buf.pos_out = None
    else:
        buf.hidden = buf.hidden_out = None
    _both(buf)


def test_tokens_ahead_of_the_first_sequence():
    p = _problem([400, 350], [300, 250])
    buf = parity.to_device(p)
    buf.cu_seqlens += torch.tensor([37, 0, 0], dtype=torch.int32, device="cuda")
    _both(buf)


def test_a_sequence_longer_than_promised_stays_inside_the_buffers():
    """The excess is left out and reported; whatever the workspace held for those tokens moves no row."""
    p = _problem([400, 350], [300, 250])
    buf = parity.to_device(p)
    buf.params.max_seqlen = 380
    buf.workspace.fill_(1)  # a valid place for every token, were it read
    assert int(_both(buf)["status"]) & fastav.FASTAV_DEV_SHAPE_MISMATCH


@pytest.mark.parametrize("layout", ["packed", "head_major", "no_values", "no_positions", "no_hidden"])
@pytest.mark.parametrize("lens,rows", [([333, 0, 90], 1), ([700], 2), ([60] * 9, 9)])
def test_rows_read_ahead_by_the_blocks_that_select(layout, lens, rows):
    """Little per block: the slice's rows lie in shared memory before the selection is known (from the keys, and from partial sums)."""
    p = W.random_problem(seed=sum(lens), lens=lens, rows=[min(rows, n) for n in lens], keeps=[n // 3 if i % 3 else n * 4 // 5 for i, n in enumerate(lens)],
                         num_q_heads=4, num_kv_heads=2, head_dim=64, hidden=128)
    buf = parity.to_device(p)
    if layout == "head_major":
        k, v = (torch.empty(2, p.total_tokens, 64, dtype=torch.bfloat16, device="cuda").transpose(0, 1) for _ in range(2))
        k.copy_(buf.k), v.copy_(buf.v)
        buf = fastav.make_buffers(q=buf.q, q_idx=buf.q_idx, cu_qlens=buf.cu_qlens, k=k, v=v, cu_seqlens=buf.cu_seqlens, keep_counts=buf.keep_counts, hidden=buf.hidden,
                                  pos=buf.pos, softmax_scale=p.softmax_scale, flags=parity.flags_of(p))
    for name in {"no_values": ("v",), "no_positions": ("pos",), "no_hidden": ("hidden",)}.get(layout, ()):
        setattr(buf, name, None)
        setattr(buf, name + "_out", None)
    before = fastav.fastav_kernel_launches()
    buf.prune()
    torch.cuda.synchronize()
    if rows <= 4 or len(lens) >= 8:
        assert fastav.fastav_kernel_launches() - before == (1 if rows <= 4 else 2)  # no gather of its own
    keep, cu = buf.keep_idx.cpu().numpy(), buf.cu_keep.cpu().numpy()
    mine = parity.gather_rows(p, keep[:cu[-1]], cu)
    assert int(buf.device_status) & ~fastav.FASTAV_DEV_PROTECT_OVERFLOW == 0
    for name in ("hidden", "pos", "k", "v"):
        if getattr(buf, name + "_out") is not None:
            parity.assert_bits_equal(getattr(buf, name + "_out"), mine[name], f"{layout} {name}")


@pytest.mark.parametrize("lens,keep,hid,hkv,d,ahead", [
    ([744], 0.8, 3584, 4, 128, True), ([330], 0.1, 3584, 4, 128, True), ([2000], 0.8, 3584, 4, 128, True), ([2000], 0.3, 3584, 4, 128, False),
    ([2000], 0.1, 4096, 8, 128, False), ([250] * 4, 0.8, 3584, 4, 128, True), ([250] * 4, 0.3, 3584, 4, 128, False), ([480] * 4, 0.8, 3584, 4, 128, True),
    ([480] * 4, 0.6, 3584, 4, 128, False), ([120] * 8, 0.75, 3584, 4, 128, True), ([120] * 8, 0.5, 3584, 4, 128, False), ([230] * 8, 0.9, 3584, 4, 128, False),
    ([120, 0, 90, 33] * 2, 0.8, 1024, 16, 64, True), ([60] * 16, 0.8, 3584, 4, 128, True), ([60, 0, 7, 90] * 4, 0.9, 1024, 16, 64, True),
    ([60] * 16, 0.5, 3584, 4, 128, False), ([60] * 17, 0.9, 3584, 4, 128, False), ([170] * 10, 0.8, 3584, 4, 128, False), ([1500], 0.9, 504, 2, 128, False),
])
def test_rows_are_read_ahead_where_most_of_them_stay(lens, keep, hid, hkv, d, ahead):
    """The kernel that selects leaves every token's place in the workspace's last part for the gather that reads ahead, and nothing there for the other."""
    p = _problem(lens, [int(keep * n) for n in lens], hid, 2 * hkv, hkv, d)
    buf = parity.to_device(p)
    size = -(-4 * p.total_tokens // 256) * 256
    places = buf.workspace[fastav.fastav_workspace_bytes(buf.params) - size:].view(torch.int32)[:p.total_tokens]
    places.fill_(0x77777777)
    buf.prune()
    torch.cuda.synchronize()
    left = places != 0x77777777
    assert bool(left.all()) if ahead else not bool(left.any())
    _both(buf)


def test_few_survivors_take_no_longer_behind_partial_sums():
    """8 x 300 tokens, 24 scored rows: 10 % kept against 60 %."""
    medians = []
    for keep in (0.1, 0.6):
        p = W.random_problem(seed=9, lens=[300] * 8, rows=[24] * 8, keeps=[int(300 * keep)] * 8, num_q_heads=4, num_kv_heads=1, head_dim=64, hidden=256)
        buf = parity.to_device(p)
        medians.append(timing.us_per_call(buf.prune))
    assert medians[0] < 1.05 * medians[1]


def test_what_the_workspace_held_moves_no_row():
    """Tokens cut off a sequence that is longer than promised have no place: were the stale one read, it would name an output row that no survivor has."""
    p = _problem([400, 350], [300, 250])
    buf = parity.to_device(p)
    buf.params.max_seqlen = 380
    buf.keep_counts -= 10
    spare = buf.params.total_keep - 1
    buf.workspace.view(torch.int32).fill_(spare)
    for name in ("hidden_out", "pos_out", "k_out", "v_out"):
        getattr(buf, name).view(torch.uint8).fill_(0x55)
    buf.prune()
    torch.cuda.synchronize()
    assert int(buf.cu_keep[-1]) == spare - 19 and int(buf.device_status) & fastav.FASTAV_DEV_SHAPE_MISMATCH
    for name in ("hidden_out", "pos_out", "k_out", "v_out"):
        assert bool((getattr(buf, name)[spare - 19:].contiguous().view(torch.uint8) == 0x55).all()), name
