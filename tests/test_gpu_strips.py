"""The strip form of generated kernels (pixel pairs in 16-bit lanes, a sliding
window per thread) at the sizes where it can go wrong: around its 128-column
tiles and its 8-column strips, around the rows of a row group, and with every
number of rows per thread, single and batched (images of one size and of
several).  Reference: the staged-tile interpreter and the CPU oracle.
Bit-exact."""
import numpy as np
import pytest

import oracle as O
from paper_2008_11476_gb300 import apps as A
from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (7, 26), (8, 3), (127, 24), (128, 25), (129, 73), (136, 49), (257, 200)]
ROWS = ["", "3", "9", "24"]  # "": chosen by the library


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


def chain(ctx, src, w, h, border):
    """Local operators of every kind in one group, S16 and U8 outputs."""
    g = H.hvxCreateGraph(ctx)
    a, b, c, d, e = (H.hvxCreateVirtualImage(g) for _ in range(5))
    s = H.hvxCreateVirtualImage(g, 0, 0, H.HVX_DF_S16)
    out, o16 = PG.empty(ctx, w, h, H.HVX_DF_U8), PG.empty(ctx, w, h, H.HVX_DF_S16)
    sharpen = np.array([0, -1, 0, -1, 9, -1, 0, -1, 0])
    for n in (H.hvxBox3x3Node(g, src, a), H.hvxMedian3x3Node(g, a, b),
              H.hvxConvolveNode(g, b, sharpen, 3, 3, 1, s), H.hvxDilate3x3Node(g, src, d)):
        H.hvxSetNodeBorder(n, border, 77)
    H.hvxConvertDepthNode(g, s, c, H.HVX_POLICY_SATURATE, 2)
    H.hvxAbsDiffNode(g, c, d, e)
    H.hvxThresholdNode(g, e, H.HVX_THRESHOLD_BINARY, 40, 0, 201, 3, out)
    H.hvxSubtractNode(g, s, d, H.HVX_POLICY_WRAP, o16)
    return g, [out, o16]


def verified(g, codegen):
    H.hvxSetGraphCodegen(g, codegen)
    H.hvxVerifyGraph(g)
    return g


@pytest.mark.parametrize("rows", ROWS)
@pytest.mark.parametrize("border", [H.HVX_BORDER_REPLICATE, H.HVX_BORDER_CONSTANT,
                                    H.HVX_BORDER_UNDEFINED])
def test_strips_match_the_interpreter(ctx, border, rows, monkeypatch):
    if rows:
        monkeypatch.setenv("HVX_STRIP_ROWS", rows)
    graphs, outs, refs = [], [], []
    for i, (w, h) in enumerate(SIZES):
        src = PG.upload(ctx, synth.rects_noise(w, h, seed=i + 1), H.HVX_DF_U8)
        g, got = chain(ctx, src, w, h, border)
        verified(g, H.HVX_CODEGEN_REQUIRE)
        assert "hvx_generated_strips" in H.hvxGetGraphKernelSource(g, 0)
        g2, want = chain(ctx, src, w, h, border)
        verified(g2, H.HVX_CODEGEN_OFF)
        H.hvxProcessGraph(g)
        H.hvxProcessGraph(g2)
        refs.append([PG.download(im) for im in want])
        for im, r in zip(got, refs[-1]):
            np.testing.assert_array_equal(PG.download(im), r, err_msg=f"{w}x{h}")
        graphs.append(g)
        outs.append(got)
    # one launch over images of several sizes, then of one size
    for pick in (range(len(SIZES)), [3, len(SIZES)]):
        if max(pick) >= len(graphs):
            w, h = SIZES[3]
            src = PG.upload(ctx, synth.rects_noise(w, h, seed=4), H.HVX_DF_U8)
            g, got = chain(ctx, src, w, h, border)
            graphs.append(verified(g, H.HVX_CODEGEN_REQUIRE))
            outs.append(got)
            refs.append(refs[3])
        for i in pick:
            for im in outs[i]:
                stale = np.full_like(PG.download(im), 7)
                H.hvxCopyImage(im, stale.ctypes.data, stale.strides[0], H.HVX_WRITE)
        H.hvxProcessGraphBatch([graphs[i] for i in pick])
        H.hvxWaitBatch(ctx)
        for i in pick:
            for im, r in zip(outs[i], refs[i]):
                np.testing.assert_array_equal(PG.download(im), r)


@pytest.mark.parametrize("w,h", [(2, 1), (130, 25), (256, 97)])
def test_camera_chain_with_16_bit_inputs(ctx, w, h):
    """A UYVY input read with a halo (its luma is filtered) and an S16 input:
    out = saturate(luma - Gaussian3x3(luma) + s16)."""
    raw = synth.uyvy(w, h, seed=w)
    s16 = (np.arange(w * h, dtype=np.int64).reshape(h, w) * 7919 % 65536 - 32768).astype(np.int16)
    g = H.hvxCreateGraph(ctx)
    y, b = H.hvxCreateVirtualImage(g), H.hvxCreateVirtualImage(g)
    d = H.hvxCreateVirtualImage(g, 0, 0, H.HVX_DF_S16)
    out = PG.empty(ctx, w, h, H.HVX_DF_S16)
    H.hvxChannelExtractNode(g, PG.upload(ctx, raw, H.HVX_DF_UYVY), H.HVX_CHANNEL_Y, y)
    H.hvxGaussian3x3Node(g, y, b)
    H.hvxSubtractNode(g, y, b, H.HVX_POLICY_SATURATE, d)
    H.hvxAddNode(g, d, PG.upload(ctx, s16, H.HVX_DF_S16), H.HVX_POLICY_SATURATE, out)
    verified(g, H.HVX_CODEGEN_REQUIRE)
    assert H.hvxQueryGraph(g, H.HVX_GRAPH_NUM_LAUNCHES) == 1
    assert "hvx_generated_strips" in H.hvxGetGraphKernelSource(g, 0)
    H.hvxProcessGraph(g)
    luma = np.ascontiguousarray(raw[:, 1::2])
    diff = luma.astype(int) - O.gaussian3x3(luma, O.BORDER_REPLICATE).data
    want = np.clip(diff + s16.astype(int), -32768, 32767)
    np.testing.assert_array_equal(PG.download(out), want)


@pytest.mark.parametrize("name", ["FChain", "Unsharp", "Laplacian"])
def test_strip_and_tile_forms_agree(ctx, name, monkeypatch):
    w, h = 1000, 311
    img = synth.rects_noise(w, h, seed=3)
    got = []
    for rows in ("", "0"):  # "0": the tile form
        if rows:
            monkeypatch.setenv("HVX_STRIP_ROWS", rows)
        g, res = dict(A.APPS)[name](ctx, PG.upload(ctx, img, H.HVX_DF_U8), w, h, True)
        H.hvxProcessGraph(g)
        got.append(PG.download(res[0][1]))
    np.testing.assert_array_equal(got[0], got[1])


@pytest.mark.parametrize("w,h", [(1, 1), (130, 40), (1031, 517)])
@pytest.mark.parametrize("border", [H.HVX_BORDER_REPLICATE, H.HVX_BORDER_UNDEFINED])
def test_global_operators_of_strips(ctx, w, h, border):
    """MeanStdDev, MinMaxLoc and Histogram of images computed in the group (a
    Gaussian, and its S16 difference from the input), run twice: the scratch of
    the partial results is left clean.  Saturated areas, so that extrema are
    taken by many pixels."""
    img = synth.rects_noise(w, h, seed=h, sigma=40.0)
    src = PG.upload(ctx, img, H.HVX_DF_U8)
    g = H.hvxCreateGraph(ctx)
    b, d = H.hvxCreateVirtualImage(g), H.hvxCreateVirtualImage(g, 0, 0, H.HVX_DF_S16)
    H.hvxSetNodeBorder(H.hvxGaussian3x3Node(g, src, b), border, 0)
    H.hvxSubtractNode(g, src, b, H.HVX_POLICY_SATURATE, d)
    nodes = [H.hvxMeanStdDevNode(g, d), H.hvxMinMaxLocNode(g, b), H.hvxHistogramNode(g, b, 7, 20, 200),
             H.hvxMinMaxLocNode(g, d)]
    verified(g, H.HVX_CODEGEN_REQUIRE)
    assert "hvx_generated_strips" in H.hvxGetGraphKernelSource(g, 0)
    ob = O.BORDER_REPLICATE if border == H.HVX_BORDER_REPLICATE else O.BORDER_UNDEFINED
    blur = O.gaussian3x3(img, ob)
    x0, y0, x1, y1 = blur.rect
    part = blur.data[y0:y1, x0:x1]
    diff = img[y0:y1, x0:x1].astype(int) - part
    for _ in range(2):
        H.hvxProcessGraph(g)
        m = H.hvxGetNodeResult(nodes[0], H.HvxMeanStdDev())
        assert (m.sum, m.sum_squares, m.count) == (diff.sum(), (diff * diff).sum(), diff.size)
        hist = H.hvxGetNodeResult(nodes[2], np.zeros(7, np.uint32))
        v = part.astype(int)
        want = np.bincount(((v - 20) * 7 // 200)[(v >= 20) & (v < 220)], minlength=7)
        np.testing.assert_array_equal(hist, want)
        for node, a in ((nodes[1], part.astype(int)), (nodes[3], diff)):
            r = H.hvxGetNodeResult(node, H.HvxMinMaxLoc())
            if a.size == 0:
                assert (r.min_count, r.max_count, r.min_x) == (0, 0, -1)
                continue
            assert (r.min, r.max) == (a.min(), a.max())
            assert (r.min_count, r.max_count) == ((a == a.min()).sum(), (a == a.max()).sum())
            for at, (x, y) in ((a.argmin(), (r.min_x, r.min_y)), (a.argmax(), (r.max_x, r.max_y))):
                assert (x, y) == (x0 + at % a.shape[1], y0 + at // a.shape[1])
    H.hvxReleaseGraph(g)
