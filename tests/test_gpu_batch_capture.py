"""Batches on a stream that is being captured: generated and corner batches are
captured and replay right after many other batches have come and gone; edge
and Gaussian batches are refused, seen before or not, and leave the capture as
it is."""
import numpy as np
import pytest
import torch

from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [(129, 121), (640, 480)]


@pytest.fixture
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


def build(ctx, op, w, h, src, dst):
    if op == "corner":
        return PG.harris_graph(ctx, src, dst)
    if op == "edge":
        return PG.edge_graph(ctx, src, dst)
    g = H.hvxCreateGraph(ctx)
    if op == "gaussian":
        H.hvxGaussian3x3Node(g, src, dst)
    else:
        v = H.hvxCreateVirtualImage(g)
        H.hvxDilate3x3Node(g, src, v)
        H.hvxAbsDiffNode(g, v, src, dst)
    H.hvxVerifyGraph(g)
    return g


def batch(ctx, op, seed):
    graphs, ins, outs = [], [], []
    for i, (w, h) in enumerate(SIZES):
        ins.append(PG.upload(ctx, synth.rects_noise(w, h, seed + i), H.HVX_DF_U8))
        outs.append(PG.empty(ctx, w, h, H.HVX_DF_U8))
        graphs.append(build(ctx, op, w, h, ins[-1], outs[-1]))
    return graphs, ins, outs


def write(im, a):
    H.hvxCopyImage(im, a.ctypes.data, a.strides[0], H.HVX_WRITE)


@pytest.mark.parametrize("seen", [False, True], ids=["first", "seen"])
@pytest.mark.parametrize("op", ["generated", "corner"])
def test_captured_batch_outlives_the_cache(ctx, op, seen):
    graphs, ins, outs = batch(ctx, op, 1)
    if seen:
        H.hvxProcessGraphBatch(graphs)
        H.hvxWaitBatch(ctx)
    s, cap = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        cap.capture_begin()
        H.hvxProcessGraphBatch(graphs, s.cuda_stream)
        cap.capture_end()
    for k in range(20):
        H.hvxProcessGraphBatch(batch(ctx, ["generated", "corner", "gaussian"][k % 3], 10 * k + 5)[0])
    H.hvxWaitBatch(ctx)
    for k in range(2):
        for i, (w, h) in enumerate(SIZES):
            write(ins[i], synth.rects_noise(w, h, 300 + 10 * k + i))
        cap.replay()
        torch.cuda.synchronize()
        got = [PG.download(o) for o in outs]
        for i, g in enumerate(graphs):
            write(outs[i], np.full_like(got[i], 7))
            H.hvxProcessGraph(g)
            np.testing.assert_array_equal(got[i], PG.download(outs[i]))


@pytest.mark.parametrize("seen", [False, True], ids=["first", "seen"])
@pytest.mark.parametrize("op", ["edge", "gaussian"])
def test_refused_batch_leaves_the_capture(ctx, op, seen):
    graphs, _, outs = batch(ctx, op, 1)
    want = []
    if seen:
        H.hvxProcessGraphBatch(graphs)
        H.hvxWaitBatch(ctx)
        want = [PG.download(o) for o in outs]
    s, cap = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    x = torch.zeros(4, device="cuda")
    with torch.cuda.stream(s):
        cap.capture_begin()
        x += 1
        with pytest.raises(H.HvxError):
            H.hvxProcessGraphBatch(graphs, s.cuda_stream)
        x += 1
        cap.capture_end()
    cap.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 4
    H.hvxProcessGraphBatch(graphs)
    H.hvxWaitBatch(ctx)
    for o, r in zip(outs, want):
        np.testing.assert_array_equal(PG.download(o), r)
