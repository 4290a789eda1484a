"""The corner strip kernel under border modes (its border tiles): every pair of
Sobel and window-sum borders it takes, around its 112-column tiles, its
8-column strips and its row groups, mask alone and with the response, single
and batched.  Reference: the plain one-launch-per-node form.  Bit-exact."""
import numpy as np
import pytest

from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

U, R, C = H.HVX_BORDER_UNDEFINED, H.HVX_BORDER_REPLICATE, H.HVX_BORDER_CONSTANT
# (Sobel border, its constant, window sums' border, its constant)
BORDERS = [(R, 0, R, 0), (C, 200, R, 0), (C, 31, C, 0), (R, 0, C, 0), (R, 0, U, 0), (U, 0, R, 0),
           (U, 0, C, 0), (R, 0, C, 9)]
SIZES = [(1, 1), (2, 7), (8, 3), (111, 25), (112, 24), (113, 49), (225, 130)]


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


def corner_graph(ctx, src, w, h, borders, tomasi, want_resp, fusion=True):
    bs, cs, bb, cb = borders
    g = H.hvxCreateGraph(ctx)
    gx, gy = H.hvxCreateVirtualImage(g), H.hvxCreateVirtualImage(g)
    H.hvxSetNodeBorder(H.hvxSobel3x3Node(g, src, gx, gy), bs, cs)
    sums = []
    for a, b in ((gx, gx), (gy, gy), (gx, gy)):
        p, s = H.hvxCreateVirtualImage(g), H.hvxCreateVirtualImage(g)
        H.hvxPointNode(g, H.HVX_POINT_MUL, [a, b], p)
        H.hvxSetNodeBorder(H.hvxLocalNode(g, H.HVX_LOCAL_SUM, 5, 5, p, s), bb, cb)
        sums.append(s)
    outs = [PG.empty(ctx, w, h, H.HVX_DF_U8)]
    if want_resp:
        outs.append(PG.empty(ctx, w, h, H.HVX_DF_F32))
        r = outs[1]
    else:
        r = H.hvxCreateVirtualImage(g)
    if tomasi:
        H.hvxPointNode(g, H.HVX_POINT_TOMASI_RESPONSE, sums, r)
    else:
        H.hvxPointNode(g, H.HVX_POINT_HARRIS_RESPONSE, sums, r, (1, 25))
    H.hvxThresholdNode(g, r, H.HVX_THRESHOLD_BINARY, 20000.0 if tomasi else 1e6, 0, 255, 0, outs[0])
    H.hvxSetGraphFusion(g, fusion)
    H.hvxVerifyGraph(g)
    return g, outs


@pytest.mark.parametrize("borders", BORDERS)
@pytest.mark.parametrize("tomasi", [False, True])
def test_corner_kernel_borders(ctx, borders, tomasi):
    for want_resp in (False, True):
        graphs, outs, refs = [], [], []
        for i, (w, h) in enumerate(SIZES):
            src = PG.upload(ctx, synth.rects_noise(w, h, seed=11 + i), H.HVX_DF_U8)
            g, got = corner_graph(ctx, src, w, h, borders, tomasi, want_resp)
            assert PG.kernel_kinds(g) == ["fused_harris_tma"]
            g2, want = corner_graph(ctx, src, w, h, borders, tomasi, want_resp, fusion=False)
            H.hvxProcessGraph(g)
            H.hvxProcessGraph(g2)
            refs.append([PG.download(im) for im in want])
            for im, ref in zip(got, refs[-1]):
                np.testing.assert_array_equal(PG.download(im), ref, err_msg=f"{w}x{h}")
            graphs.append(g)
            outs.append(got)
        for got in outs:
            for im in got:
                stale = np.full_like(PG.download(im), 7)
                H.hvxCopyImage(im, stale.ctypes.data, stale.strides[0], H.HVX_WRITE)
        H.hvxProcessGraphBatch(graphs)
        H.hvxWaitBatch(ctx)
        for got, ref in zip(outs, refs):
            for im, r in zip(got, ref):
                np.testing.assert_array_equal(PG.download(im), r)


@pytest.mark.parametrize("tomasi", [False, True])
def test_wide_and_narrow_strip_rows_agree(ctx, tomasi):
    """Mask alone (240-column tiles where they suit the width, 112 otherwise)
    against the mask of the same graph exporting its response (112 columns
    always); widths and heights around both tiles, single and batched."""
    sizes = [(1920, 1080), (1913, 1079), (480, 4000), (479, 3997), (473, 4003), (2409, 611)]
    graphs, masks, refs = [], [], []
    for i, (w, h) in enumerate(sizes):
        src = PG.upload(ctx, synth.rects_noise(w, h, seed=50 + i), H.HVX_DF_U8)
        g, (mask,) = corner_graph(ctx, src, w, h, (U, 0, U, 0), tomasi, False)
        g2, (want, _) = corner_graph(ctx, src, w, h, (U, 0, U, 0), tomasi, True)
        H.hvxProcessGraph(g)
        H.hvxProcessGraph(g2)
        refs.append(PG.download(want))
        np.testing.assert_array_equal(PG.download(mask), refs[-1], err_msg=f"{w}x{h}")
        graphs.append(g)
        masks.append(mask)
    for m, r in zip(masks, refs):
        stale = np.full_like(r, 7)
        H.hvxCopyImage(m, stale.ctypes.data, stale.strides[0], H.HVX_WRITE)
    H.hvxProcessGraphBatch(graphs)
    H.hvxWaitBatch(ctx)
    for m, r in zip(masks, refs):
        np.testing.assert_array_equal(PG.download(m), r)
