"""Strip kernels on images that have interior tiles (three tiles of the largest
height down, three across), with every kind of input: their unchecked code,
beside the border tiles that tests/test_gpu_strips.py runs.  Also results with
the page-locked block of their host copies full, and corner batches whose
images mix border modes.  Bit-exact."""
import numpy as np
import pytest

import oracle as O
from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth
from test_gpu_strips import chain, verified

pytestmark = pytest.mark.gpu

SIZES = [(400, 600), (389, 577)]
ROWS = ["", "3", "6", "9", "12", "15", "18", "21", "24"]  # "": chosen by the library


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


@pytest.mark.parametrize("rows", ROWS)
@pytest.mark.parametrize("border", [H.HVX_BORDER_REPLICATE, H.HVX_BORDER_CONSTANT,
                                    H.HVX_BORDER_UNDEFINED])
def test_local_chain(ctx, border, rows, monkeypatch):
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
            stale = np.full_like(r, 7)
            H.hvxCopyImage(im, stale.ctypes.data, stale.strides[0], H.HVX_WRITE)
        graphs.append(g)
        outs.append(got)
    H.hvxProcessGraphBatch(graphs)
    H.hvxWaitBatch(ctx)
    for got, ref in zip(outs, refs):
        for im, r in zip(got, ref):
            np.testing.assert_array_equal(PG.download(im), r)


@pytest.mark.parametrize("rows", ["", "3", "24"])
@pytest.mark.parametrize("w,h", SIZES[:1] + [(390, 577)])
def test_camera_chain(ctx, w, h, rows, monkeypatch):
    """A UYVY box (luma filtered), an S16 input from memory and its statistics:
    out = saturate(luma - Gaussian3x3(luma) + s16)."""
    if rows:
        monkeypatch.setenv("HVX_STRIP_ROWS", rows)
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
    ms, mm = H.hvxMeanStdDevNode(g, out), H.hvxMinMaxLocNode(g, out)
    verified(g, H.HVX_CODEGEN_REQUIRE)
    assert "hvx_generated_strips" in H.hvxGetGraphKernelSource(g, 0)
    H.hvxProcessGraph(g)
    luma = np.ascontiguousarray(raw[:, 1::2])
    diff = luma.astype(int) - O.gaussian3x3(luma, O.BORDER_REPLICATE).data
    want = np.clip(diff + s16.astype(int), -32768, 32767)
    np.testing.assert_array_equal(PG.download(out), want)
    m = H.hvxGetNodeResult(ms, H.HvxMeanStdDev())
    assert (m.sum, m.sum_squares, m.count) == (want.sum(), (want * want).sum(), want.size)
    r = H.hvxGetNodeResult(mm, H.HvxMinMaxLoc())
    assert (r.min, r.max, r.min_count, r.max_count) == (
        want.min(), want.max(), (want == want.min()).sum(), (want == want.max()).sum())


def test_results_without_a_host_copy():
    """256 bins take 1 KB of the context's 64 KB of page-locked memory: later
    graphs have none left, and read their results from the device."""
    c = H.hvxCreateContext()
    try:
        img = synth.uniform_u8(300, 70, 3)
        want = np.bincount(img.ravel(), minlength=256)
        for _ in range(2):  # (released blocks are used again)
            graphs = []
            for _ in range(70):
                g = H.hvxCreateGraph(c)
                n = H.hvxHistogramNode(g, PG.upload(c, img, H.HVX_DF_U8), 256, 0, 256)
                H.hvxVerifyGraph(g)
                graphs.append((g, n))
            H.hvxProcessGraphBatch([g for g, _ in graphs])
            H.hvxWaitBatch(c)
            for g, n in graphs:
                np.testing.assert_array_equal(H.hvxGetNodeResult(n, np.zeros(256, np.uint32)), want)
            for g, n in graphs:
                H.hvxProcessGraph(g)
                np.testing.assert_array_equal(H.hvxGetNodeResult(n, np.zeros(256, np.uint32)), want)
                H.hvxReleaseGraph(g)
    finally:
        H.hvxReleaseContext(c)


@pytest.mark.parametrize("tomasi", [False, True])
def test_corner_batch_of_mixed_borders(ctx, tomasi):
    """Rows of 32 strips suit the first batch; border modes, an exported
    response and small images among them keep the batch at 16."""
    U, R, C = H.HVX_BORDER_UNDEFINED, H.HVX_BORDER_REPLICATE, H.HVX_BORDER_CONSTANT
    plain = [(1920, 1080, U, False)] * 3
    mixed = [(1920, 1080, U, False), (1920, 1080, R, False), (240, 33, C, False),
             (241, 100, U, True), (7, 5, R, True), (1920, 1080, U, False)]
    thr = 40.0 if tomasi else 1e6
    for images in (plain, mixed, mixed[:2], mixed[3:4] + plain[:1]):
        graphs, outs, refs = [], [], []
        for i, (w, h, border, resp) in enumerate(images):
            src = PG.upload(ctx, synth.rects_noise(w, h, 40 + i), H.HVX_DF_U8)
            for fusion in (True, False):
                mask = PG.empty(ctx, w, h, H.HVX_DF_U8)
                r = PG.empty(ctx, w, h, H.HVX_DF_F32) if resp else None
                g = PG.harris_graph(ctx, src, mask, r, border=border, thr=thr, fusion=fusion,
                                    tomasi=tomasi)
                if fusion:
                    assert PG.kernel_kinds(g) == ["fused_harris_tma"]
                    graphs.append(g)
                    outs.append((mask, r))
                else:
                    H.hvxProcessGraph(g)
                    refs.append((PG.download(mask), PG.download(r) if resp else None))
        H.hvxProcessGraphBatch(graphs)
        H.hvxWaitBatch(ctx)
        for (mask, r), (want, want_r) in zip(outs, refs):
            np.testing.assert_array_equal(PG.download(mask), want)
            if r is not None:
                np.testing.assert_array_equal(PG.download(r), want_r)
