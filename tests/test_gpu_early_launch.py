"""Launches back to back on one stream, where a kernel may begin while the one
before it ends, for the kernels that tests/test_gpu_batch_launch.py leaves out:
generated strip kernels (their inputs from memory and from boxes), EqualizeHist
and the corner kernels.  Every launch reads what the previous one wrote, and
overwrites what the one before that read.  Bit-exact against the same graphs run
one by one with a wait after each."""
import numpy as np
import pytest

from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

# one tile, fewer tiles than CTAs, several waves (ragged)
SIZES = [[(1, 1)], [(128, 120), (129, 121), (640, 480)], [(2043, 1361)] * 6]


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


def node_graph(ctx, op, a, b, key):
    """Graph a -> b; `key` is an image that no launch writes."""
    if op.startswith("corner"):
        border = H.HVX_BORDER_UNDEFINED if op == "corner" else H.HVX_BORDER_REPLICATE
        return PG.harris_graph(ctx, a, b, border=border)
    g = H.hvxCreateGraph(ctx)
    v = H.hvxCreateVirtualImage(g)
    if op == "point":  # input rows straight from memory
        H.hvxNotNode(g, a, v)
        H.hvxXorNode(g, v, key, b)
    elif op == "strips":  # a box, and `key` from memory
        H.hvxDilate3x3Node(g, a, v)
        H.hvxXorNode(g, v, key, b)
    else:
        H.hvxEqualizeHistNode(g, a, v)
        H.hvxXorNode(g, v, key, b)
    H.hvxVerifyGraph(g)
    return g


def ring(ctx, op, sizes):
    """Three images per size and the graphs a -> b, b -> c, c -> a."""
    sets, images = [[], [], []], []
    for i, (w, h) in enumerate(sizes):
        key = PG.upload(ctx, synth.uniform_u8(w, h, 90 + i), H.HVX_DF_U8)
        ims = [PG.upload(ctx, synth.rects_noise(w, h, 70 + i), H.HVX_DF_U8)]
        ims += [PG.empty(ctx, w, h, H.HVX_DF_U8) for _ in range(2)]
        images.append(ims)
        for k in range(3):
            sets[k].append(node_graph(ctx, op, ims[k], ims[(k + 1) % 3], key))
    return sets, images


@pytest.mark.parametrize("batch", [False, True], ids=["frames", "batch"])
@pytest.mark.parametrize("sizes", SIZES, ids=["one", "edges", "waves"])
@pytest.mark.parametrize("op", ["point", "strips", "equalize", "corner", "corner replicate"])
def test_dependent_launches(ctx, op, sizes, batch):
    sets, got = ring(ctx, op, sizes)
    one_by_one, want = ring(ctx, op, sizes)
    for _ in range(4):
        for gs in sets:
            if batch:
                H.hvxProcessGraphBatch(gs)
            else:
                for g in gs:
                    H.hvxScheduleGraph(g)
    H.hvxWaitBatch(ctx)
    for _ in range(4):
        for gs in one_by_one:
            for g in gs:
                H.hvxProcessGraph(g)
    for ims, ref in zip(got, want):
        for im, r in zip(ims, ref):
            np.testing.assert_array_equal(PG.download(im), PG.download(r))
