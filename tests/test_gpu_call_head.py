"""The first kernel of a call is launched while earlier work on the stream may still be running and waits for it: the index
arrays of a call may be what a copy, a torch kernel or an earlier call wrote right before it, eagerly or from a graph."""
import numpy as np
import pytest
import torch

import parity
from paper_2601_13143_b200 import fastav, workloads as W

pytestmark = pytest.mark.gpu


def check(buf, ref):
    assert np.array_equal(buf.keep_idx.cpu().numpy(), ref["keep_idx"])
    parity.assert_bits_equal(buf.hidden_out, ref["hidden"], "hidden")
    parity.assert_bits_equal(buf.pos_out, ref["pos"], "pos")
    parity.assert_scores_close(buf.scores, ref["scores"])


@pytest.mark.parametrize("rows", [1, 16])
@pytest.mark.parametrize("writer", ["copy", "kernel", "call"])
def test_index_arrays_written_right_before_the_call(writer, rows):
    """Two problems of the same shapes but other boundaries take turns in ONE set of buffers; the arrays of the next one are
    written on the stream with nothing in between.  Stale values would be the other problem's."""
    lens = [[700, 900, 300], [300, 1100, 500]]
    keeps = [[350, 450, 150], [150, 550, 250]]
    problems = [W.random_problem(40 + i, lens[i], [rows] * 3, keeps[i], 8, 2, 64, 128) for i in range(2)]
    refs = [parity.oracle_prune(p) for p in problems]
    buf = parity.to_device(problems[0])
    buf.params.max_seqlen, buf.params.max_keep = 1100, 550
    buf.workspace = torch.empty(fastav.fastav_workspace_bytes(buf.params), dtype=torch.uint8, device="cuda")
    names = ("q", "q_idx", "cu_qlens", "k", "v", "cu_seqlens", "keep_counts", "hidden", "pos")
    sources = [{n: getattr(p, n).cuda() for n in names} for p in problems]
    pinned = [{n: getattr(p, n).pin_memory() for n in names} for p in problems]
    cu_as_keep = [torch.cat([torch.arange(a, dtype=torch.int32) for a in l]).cuda() for l in lens]
    masks = [torch.ones(1900, dtype=torch.uint8, device="cuda")] * 2
    small = torch.empty(256, dtype=torch.uint8, device="cuda")
    idx = torch.empty(1900, dtype=torch.int32, device="cuda")
    for rep in range(12):
        i = rep % 2
        for n in names:
            if n != "cu_seqlens" or writer != "call":
                getattr(buf, n).copy_((pinned if writer == "copy" else sources)[i][n], non_blocking=True)
        if writer == "call":  # the boundaries are the survivor counts another call leaves
            buf.params.total_keep = 1900
            fastav.fastav_select_mask(buf.params, masks[i], sources[i]["cu_seqlens"], idx, buf.cu_seqlens, small)
            buf.params.total_keep = 950
        buf.prune()
        torch.cuda.synchronize()
        check(buf, refs[i])
        if writer == "call":
            assert torch.equal(idx, cu_as_keep[i])


def test_a_call_captured_after_copies_replays_with_new_arrays():
    problems = [W.random_problem(50 + i, [600 + 100 * i, 500 - 100 * i], [8, 8], [200, 180], 8, 2, 64, 128) for i in range(2)]
    refs = [parity.oracle_prune(p) for p in problems]
    buf = parity.to_device(problems[0])
    buf.params.max_seqlen = 700
    buf.workspace = torch.empty(fastav.fastav_workspace_bytes(buf.params), dtype=torch.uint8, device="cuda")
    names = ("q", "q_idx", "cu_qlens", "k", "v", "cu_seqlens", "keep_counts", "hidden", "pos")
    staged = {n: getattr(problems[0], n).cuda() for n in names}
    buf.prune()  # attribute set-up does not belong in a capture
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        for n in names:
            getattr(buf, n).copy_(staged[n], non_blocking=True)
        buf.prune(side)
    for rep in range(6):
        for n in names:
            staged[n].copy_(getattr(problems[rep % 2], n))
        graph.replay()
        torch.cuda.synchronize()
        check(buf, refs[rep % 2])
