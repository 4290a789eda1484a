"""The tile form with its TMA boxes behind a histogram's bins, and with two
boxes: against the interpreter, bit-exact."""
import numpy as np
import pytest

from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

W, HT = 450, 170  # interior and border tiles


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


@pytest.mark.parametrize("bins", [1, 7, 33])
def test_box_after_bins(ctx, bins, monkeypatch):
    monkeypatch.setenv("HVX_STRIP_ROWS", "0")
    img = synth.rects_noise(W, HT, bins)
    res = []
    for codegen in (H.HVX_CODEGEN_OFF, H.HVX_CODEGEN_ONLY):
        out = PG.empty(ctx, W, HT, H.HVX_DF_S16)
        g = H.hvxCreateGraph(ctx)
        src, d = PG.upload(ctx, img, H.HVX_DF_U8), H.hvxCreateVirtualImage(g)
        H.hvxConvolveNode(g, src, np.full(25, 30), 5, 5, 1, out)
        H.hvxCopyNode(g, src, d)
        hist = H.hvxHistogramNode(g, d, bins, 20, 200)
        H.hvxSetGraphCodegen(g, codegen)
        H.hvxVerifyGraph(g)
        for batch in (False, True):
            if batch:
                H.hvxProcessGraphBatch([g])
                H.hvxWaitBatch(ctx)
            else:
                H.hvxProcessGraph(g)
            res.append((PG.download(out), H.hvxGetNodeResult(hist, np.zeros(bins, np.uint32))))
    for out, hist in res[1:]:
        np.testing.assert_array_equal(out, res[0][0])
        np.testing.assert_array_equal(hist, res[0][1])


@pytest.mark.parametrize("halo", [2, 3, 4, 5])
def test_two_boxes(ctx, halo, monkeypatch):
    monkeypatch.setenv("HVX_STRIP_ROWS", "0")
    imgs = [synth.rects_noise(W, HT, 5), synth.uniform_u8(W, HT, 6)]
    res = []
    for codegen in (H.HVX_CODEGEN_OFF, H.HVX_CODEGEN_ONLY):
        a, b = (PG.upload(ctx, i, H.HVX_DF_U8) for i in imgs)
        g = H.hvxCreateGraph(ctx)
        e, d, f, x, o = (H.hvxCreateVirtualImage(g) for _ in range(5))
        H.hvxAbsDiffNode(g, a, b, e)
        H.hvxDilate3x3Node(g, a, d)
        H.hvxErode3x3Node(g, b, f)
        H.hvxXorNode(g, d, f, x)
        H.hvxAndNode(g, x, e, o)
        for _ in range(halo - 1):
            v, o = o, H.hvxCreateVirtualImage(g)
            H.hvxMedian3x3Node(g, v, o)
        out = PG.empty(ctx, W, HT, H.HVX_DF_U8)
        H.hvxNotNode(g, o, out)
        H.hvxSetGraphCodegen(g, codegen)
        H.hvxVerifyGraph(g)
        assert H.hvxQueryGraph(g, H.HVX_GRAPH_NUM_LAUNCHES) == 1
        for batch in (False, True):
            if batch:
                H.hvxProcessGraphBatch([g])
                H.hvxWaitBatch(ctx)
            else:
                H.hvxProcessGraph(g)
            res.append(PG.download(out))
    for r in res[1:]:
        np.testing.assert_array_equal(r, res[0])
