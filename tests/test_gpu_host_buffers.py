"""fastav_prune_host reaches page-locked buffers from its kernels and copies the others: both ways give what fastav_prune gives
on the device, whatever the sizes, alignments and mixture."""
import pytest
import torch

import parity
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu
NAMES = ("q", "q_idx", "cu_qlens", "k", "v", "cu_seqlens", "keep_counts", "hidden", "pos")
OUTS = ("scores", "keep_idx", "cu_keep", "hidden_out", "pos_out", "k_out", "v_out")


def off_by(t, elements):
    """A page-locked copy of t that starts `elements` after a 16-byte boundary."""
    room = torch.empty(t.numel() + 64, dtype=t.dtype).pin_memory()
    out = room[elements:elements + t.numel()].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("how", ["pinned", "pageable", "one pageable input", "one pageable output", "odd index arrays", "odd rows", "in place"])
@pytest.mark.parametrize("lens,rows,keeps", [([512], [4], [200]), ([300, 1, 900], [16, 1, 16], [100, 1, 333]), ([2500], [1], [2500]),
                                             ([4000, 33], [40, 2], [1, 33]), ([7, 5], [1, 1], [0, 2])])
def test_host_buffers_give_what_the_device_call_gives(how, lens, rows, keeps):
    p = W.random_problem(11 + len(lens) + sum(lens), lens, rows, keeps, 8, 2, 64, 136)
    protect = torch.zeros(sum(lens), dtype=torch.uint8)
    protect[::37] = 1
    flags = fastav.FASTAV_CAUSAL | fastav.FASTAV_KEEP_IDX_GLOBAL
    buf = parity.to_device(p, protect=protect, flags=flags)
    buf.prune()
    pin = lambda t: t if how == "pageable" else t.pin_memory()
    host = {n: pin(getattr(p, n)) for n in NAMES}
    out = {n: pin(torch.full_like(getattr(buf, n), 3, device="cpu")) for n in OUTS}
    status = pin(torch.full((1,), 77, dtype=torch.int32))
    if how == "one pageable input":
        host["v"] = p.v
    if how == "one pageable output":
        out["hidden_out"] = torch.full_like(buf.hidden_out, 3, device="cpu")
    if how == "odd index arrays":
        host = {n: off_by(t, 1) if t.dtype == torch.int32 else t for n, t in host.items()}
        out["scores"], out["pos_out"] = off_by(out["scores"], 3), off_by(out["pos_out"], 1)
    if how == "odd rows":
        host["hidden"] = off_by(host["hidden"], 4)
        out["k_out"] = off_by(out["k_out"], 1)
    if how == "in place" and out["hidden_out"].numel():
        out["hidden_out"] = host["hidden"].view(-1)[:out["hidden_out"].numel()].view(out["hidden_out"].shape)
    arena = torch.empty(fastav.fastav_host_arena_bytes(buf.params), dtype=torch.uint8, device="cuda")
    fastav.fastav_prune_host(buf.params, host["q"], host["q_idx"], host["cu_qlens"], host["k"], host["v"], host["cu_seqlens"],
                             host["keep_counts"], pin(protect), host["hidden"], host["pos"], *(out[n] for n in OUTS), status, arena)
    torch.cuda.synchronize()
    kept = int(buf.cu_keep[-1])
    assert int(status) == int(buf.device_status)
    for n in OUTS:
        want = getattr(buf, n).cpu()
        if n == "keep_idx":
            want, out[n] = want[:kept], out[n][:kept]
        parity.assert_bits_equal(out[n], want, f"{how}: {n}")


class At:
    """A host array at any byte address, as far as fastav_prune_host looks at it."""
    is_cuda = False

    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address

    def is_contiguous(self):
        return True


@pytest.mark.parametrize("shift", [1, 2, 3])
def test_small_arrays_may_start_at_any_byte(shift):
    """The small arrays are copied as bytes; positions, which a kernel would store as words, then take the copies too."""
    p = W.random_problem(4, [300, 90], [1, 1], [120, 40], 8, 2, 64, 136)
    buf = parity.to_device(p)
    buf.prune()
    torch.cuda.synchronize()
    host = {n: getattr(p, n).pin_memory() for n in NAMES}
    out = {n: torch.zeros_like(getattr(buf, n), device="cpu").pin_memory() for n in OUTS}
    small = {n: torch.zeros(out[n].nbytes + 8, dtype=torch.uint8).pin_memory() for n in ("scores", "keep_idx", "cu_keep", "pos_out")}
    arena = torch.empty(fastav.fastav_host_arena_bytes(buf.params), dtype=torch.uint8, device="cuda")
    fastav.fastav_prune_host(buf.params, *(host[n] for n in NAMES[:7]), None, host["hidden"], host["pos"],
                             *(At(small[n].data_ptr() + shift) if n in small else out[n] for n in OUTS), None, arena)
    torch.cuda.synchronize()
    for n in OUTS:
        got = small[n][shift:shift + out[n].nbytes].clone().view(out[n].dtype) if n in small else out[n]
        parity.assert_bits_equal(got, getattr(buf, n).cpu(), n)
        assert n not in small or (small[n][:shift].eq(0).all() and small[n][shift + out[n].nbytes:].eq(0).all())
