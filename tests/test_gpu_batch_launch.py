"""Batches launched back to back on one stream, where a launch may begin while
the one before it ends: a batch that reads what the previous one wrote, and one
that overwrites what the previous one read.  Bit-exact against the same graphs
run one by one with a wait after each."""
import numpy as np
import pytest
import torch

from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

# one tile, fewer tiles than CTAs, several tiles per CTA (ragged)
SIZES = [[(1, 1)], [(128, 120), (129, 121), (640, 480)], [(2043, 1361)] * 9]
B5 = [a * b for a in (1, 4, 6, 4, 1) for b in (1, 4, 6, 4, 1)]


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


def node_graph(ctx, op, a, b):
    g = H.hvxCreateGraph(ctx)
    if op == "gaussian":
        n = H.hvxGaussian3x3Node(g, a, b)
    else:
        n = H.hvxConvolveNode(g, a, B5, 5, 5, 8, b)
    H.hvxSetNodeBorder(n, H.HVX_BORDER_REPLICATE, 0)
    H.hvxVerifyGraph(g)
    return g


def ring(ctx, op, sizes):
    """Three images per size and the graphs a -> b, b -> c, c -> a."""
    sets, images = [[], [], []], []
    for i, (w, h) in enumerate(sizes):
        ims = [PG.upload(ctx, synth.rects_noise(w, h, 70 + i), H.HVX_DF_U8)]
        ims += [PG.empty(ctx, w, h, H.HVX_DF_U8) for _ in range(2)]
        images.append(ims)
        for k in range(3):
            if op == "edge":
                g = PG.edge_graph(ctx, ims[k], ims[(k + 1) % 3], PG.empty(ctx, w, h, H.HVX_DF_U8),
                                  border=H.HVX_BORDER_REPLICATE, cval=0)
            else:
                g = node_graph(ctx, op, ims[k], ims[(k + 1) % 3])
            sets[k].append(g)
    return sets, images


@pytest.mark.parametrize("sizes", SIZES, ids=["one", "edges", "waves"])
@pytest.mark.parametrize("op", ["gaussian", "binomial", "edge"])
def test_dependent_batches(ctx, op, sizes):
    sets, got = ring(ctx, op, sizes)
    one_by_one, want = ring(ctx, op, sizes)
    for gs in sets:  # (the first call of each also runs the tuner's trials)
        H.hvxProcessGraphBatch(gs)
    H.hvxWaitBatch(ctx)
    for ims, ref in zip(got, want):
        for im, r in zip(ims, ref):
            a = PG.download(im)
            H.hvxCopyImage(r, a.ctypes.data, a.strides[0], H.HVX_WRITE)
    for _ in range(4):
        for gs in sets:
            H.hvxProcessGraphBatch(gs)
    H.hvxWaitBatch(ctx)
    for _ in range(4):
        for gs in one_by_one:
            for g in gs:
                H.hvxProcessGraph(g)
    for ims, ref in zip(got, want):
        for im, r in zip(ims, ref):
            np.testing.assert_array_equal(PG.download(im), PG.download(r))


def test_batch_is_refused_under_capture(ctx):
    sets, _ = ring(ctx, "gaussian", SIZES[1])
    H.hvxProcessGraphBatch(sets[0])
    H.hvxWaitBatch(ctx)
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        graph.capture_begin()
        with pytest.raises(H.HvxError):
            H.hvxProcessGraphBatch(sets[0], s.cuda_stream)
        graph.capture_end()
    H.hvxProcessGraphBatch(sets[0])
    H.hvxWaitBatch(ctx)
