"""Groups that the hand-written kernels run, on a stored input whose valid region
is smaller than the image: pixels outside the output's valid region are 0
(hvx.h), whatever the border mode and wherever tiles end.  Reference: the oracle
operator by operator."""
import numpy as np
import pytest

import oracle as O
from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [(227, 100), (257, 130), (258, 131), (512, 72), (640, 480)]
BORDERS = [(H.HVX_BORDER_UNDEFINED, O.BORDER_UNDEFINED), (H.HVX_BORDER_REPLICATE, O.BORDER_REPLICATE),
           (H.HVX_BORDER_CONSTANT, O.BORDER_CONSTANT)]
B5 = [a * b for a in (1, 4, 6, 4, 1) for b in (1, 4, 6, 4, 1)]


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


def border(n, mode, cval=90):
    H.hvxSetNodeBorder(n, mode, cval)


def shrink(ctx, img, g):
    """EqualizeHist of Gaussian3x3 UNDEFINED, three times: a virtual image that
    another group stores, valid from 3 pixels inside the image on."""
    v = PG.upload(ctx, img, H.HVX_DF_U8)
    ref = img
    for _ in range(3):
        b, e = H.hvxCreateVirtualImage(g), H.hvxCreateVirtualImage(g)
        border(H.hvxGaussian3x3Node(g, v, b), H.HVX_BORDER_UNDEFINED, 0)
        H.hvxEqualizeHistNode(g, b, e)
        v, ref = e, O.equalize_hist(O.gaussian3x3(ref, O.BORDER_UNDEFINED))
    assert ref.rect == (3, 3, img.shape[1] - 3, img.shape[0] - 3)
    return v, ref


def gaussian(g, v, ref, mode, om, w, h, ctx):
    out = PG.empty(ctx, w, h, H.HVX_DF_U8)
    border(H.hvxGaussian3x3Node(g, v, out), mode)
    return [(out, O.gaussian3x3(ref, om, 90))]


def binomial(g, v, ref, mode, om, w, h, ctx):
    out = PG.empty(ctx, w, h, H.HVX_DF_U8)
    border(H.hvxConvolveNode(g, v, B5, 5, 5, 8, out), mode)
    return [(out, O.convolve(ref, np.array(B5, np.int32).reshape(5, 5), 8, om, 90, np.uint8))]


def sobel_x(g, v, ref, mode, om, w, h, ctx):
    out = PG.empty(ctx, w, h, H.HVX_DF_S16)
    border(H.hvxSobel3x3Node(g, v, out, None), mode)
    return [(out, O.sobel3x3(ref, om, 90)[0])]


def sobel_mask(g, v, ref, mode, om, w, h, ctx):
    out = PG.empty(ctx, w, h, H.HVX_DF_U8)
    x, y, m = (H.hvxCreateVirtualImage(g) for _ in range(3))
    border(H.hvxSobel3x3Node(g, v, x, y), mode)
    H.hvxMagnitudeNode(g, x, y, m)
    H.hvxThresholdNode(g, m, H.HVX_THRESHOLD_BINARY, 100, 0, 255, 1, out)
    return [(out, O.threshold(O.magnitude(*O.sobel3x3(ref, om, 90)), 100, 255, 1))]


def edge(g, v, ref, mode, om, w, h, ctx):
    ph, mk = PG.empty(ctx, w, h, H.HVX_DF_U8), PG.empty(ctx, w, h, H.HVX_DF_U8)
    b, x, y, m = (H.hvxCreateVirtualImage(g) for _ in range(4))
    border(H.hvxGaussian3x3Node(g, v, b), mode)
    border(H.hvxSobel3x3Node(g, b, x, y), mode)
    H.hvxMagnitudeNode(g, x, y, m)
    H.hvxThresholdNode(g, m, H.HVX_THRESHOLD_BINARY, 100, 0, 255, 0, mk)
    H.hvxPhaseNode(g, x, y, ph)
    gx, gy = O.sobel3x3(O.gaussian3x3(ref, om, 90), om, 90)
    return [(ph, O.phase(gx, gy)), (mk, O.threshold(O.magnitude(gx, gy), 100))]


def harris(g, v, ref, mode, om, w, h, ctx):
    out = PG.empty(ctx, w, h, H.HVX_DF_U8)
    x, y = H.hvxCreateVirtualImage(g), H.hvxCreateVirtualImage(g)
    cval = 0  # of products
    border(H.hvxSobel3x3Node(g, v, x, y), mode, cval)
    gx, gy = O.sobel3x3(ref, om, cval)
    sums, want = [], []
    for a, b, ra, rb in ((x, x, gx, gx), (y, y, gy, gy), (x, y, gx, gy)):
        p, s = H.hvxCreateVirtualImage(g), H.hvxCreateVirtualImage(g)
        H.hvxPointNode(g, H.HVX_POINT_MUL, [a, b], p)
        border(H.hvxLocalNode(g, H.HVX_LOCAL_SUM, 5, 5, p, s), mode, cval)
        sums.append(s)
        want.append(O.window_sum(O.mul_s32(ra, rb), 5, 5, om, cval))
    r = H.hvxCreateVirtualImage(g)
    H.hvxPointNode(g, H.HVX_POINT_HARRIS_RESPONSE, sums, r, (1, 25))
    H.hvxThresholdNode(g, r, H.HVX_THRESHOLD_BINARY, 1e6, 0, 255, 7, out)
    return [(out, O.threshold(O.harris_response(*want), 1e6, 255, 7))]


@pytest.mark.parametrize("codegen", [H.HVX_CODEGEN_OFF, H.HVX_CODEGEN_AUTO])
@pytest.mark.parametrize("mode", range(3), ids=["undefined", "replicate", "constant"])
@pytest.mark.parametrize("w,h", SIZES)
@pytest.mark.parametrize("op", [gaussian, binomial, sobel_x, sobel_mask, edge, harris],
                         ids=lambda f: f.__name__)
def test_zero_outside_the_valid_region(ctx, op, w, h, mode, codegen):
    img = synth.rects_noise(w, h, seed=w)
    g = H.hvxCreateGraph(ctx)
    v, ref = shrink(ctx, img, g)
    outs = op(g, v, ref, *BORDERS[mode], w, h, ctx)
    H.hvxSetGraphCodegen(g, codegen)
    H.hvxVerifyGraph(g)
    H.hvxProcessGraph(g)
    for im, want in outs:
        assert H.hvxGetValidRegion(im) == want.rect
        np.testing.assert_array_equal(PG.download(im), want.data)
    H.hvxReleaseGraph(g)
