"""The state that global operators and EqualizeHist keep between launches
(partial sums, bins, counters of finished CTAs): cleared before a graph's first
launch on any stream."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


class Statistics:
    """Dilate3x3, its MeanStdDev, MinMaxLoc and Histogram, and EqualizeHist of
    the input."""

    def __init__(self, ctx, w, h, seed):
        img = synth.rects_noise(w, h, seed)
        self.src = PG.upload(ctx, img, H.HVX_DF_U8)
        self.out = PG.empty(ctx, w, h, H.HVX_DF_U8)
        self.g = g = H.hvxCreateGraph(ctx)
        d = H.hvxCreateVirtualImage(g)
        H.hvxDilate3x3Node(g, self.src, d)
        self.ms = H.hvxMeanStdDevNode(g, d)
        self.mm = H.hvxMinMaxLocNode(g, d)
        self.hs = H.hvxHistogramNode(g, d, 256, 0, 256)
        H.hvxEqualizeHistNode(g, self.src, self.out)
        ref = O.morph3x3(img, O.MORPH_DILATE)
        self.sums = O.mean_stddev(ref)[2]
        self.minmax = O.minmaxloc(ref)
        self.hist = O.histogram(ref, 256, 0, 256)
        self.equalized = O.equalize_hist(img).data

    def check(self):
        m = H.hvxGetNodeResult(self.ms, H.HvxMeanStdDev())
        assert (m.sum, m.sum_squares, m.count) == self.sums
        r, want = H.hvxGetNodeResult(self.mm, H.HvxMinMaxLoc()), self.minmax
        assert (r.min, r.max, r.min_count, r.max_count) == (want["min"], want["max"],
                                                            want["min_count"], want["max_count"])
        assert ((r.min_x, r.min_y), (r.max_x, r.max_y)) == (want["min_loc"], want["max_loc"])
        np.testing.assert_array_equal(H.hvxGetNodeResult(self.hs, np.zeros(256, np.uint32)), self.hist)
        np.testing.assert_array_equal(PG.download(self.out), self.equalized)


@pytest.mark.parametrize("w,h", [(7, 5), (640, 480)])
def test_first_launch_on_a_stream_that_does_not_wait(ctx, w, h):
    """Verified while the default stream is busy, run on a non-blocking one at
    once, then again."""
    s = Statistics(ctx, w, h, seed=w)
    side = torch.cuda.Stream()
    a = torch.ones(1 << 28, dtype=torch.uint8, device="cuda")
    b = torch.empty_like(a)
    for _ in range(300):  # some 25 ms of copies
        b.copy_(a)
    H.hvxVerifyGraph(s.g)
    for _ in range(3):
        H.hvxScheduleGraph(s.g, side.cuda_stream)
        H.hvxWaitGraph(s.g)
        s.check()
    torch.cuda.synchronize()
    H.hvxScheduleGraph(s.g, side.cuda_stream)
    H.hvxWaitGraph(s.g)
    s.check()


def single_group(ctx, w, h, seed, codegen=H.HVX_CODEGEN_AUTO):
    """MeanStdDev, MinMaxLoc and Histogram of a Dilate3x3 in one launch."""
    img = synth.rects_noise(w, h, seed)
    g = H.hvxCreateGraph(ctx)
    d = H.hvxCreateVirtualImage(g)
    H.hvxDilate3x3Node(g, PG.upload(ctx, img, H.HVX_DF_U8), d)
    nodes = (H.hvxMeanStdDevNode(g, d), H.hvxMinMaxLocNode(g, d),
             H.hvxHistogramNode(g, d, 256, 0, 256))
    H.hvxSetGraphCodegen(g, codegen)
    H.hvxVerifyGraph(g)
    assert H.hvxQueryGraph(g, H.HVX_GRAPH_NUM_LAUNCHES) == 1
    return g, nodes, O.morph3x3(img, O.MORPH_DILATE)


def check_group(nodes, ref):
    m = H.hvxGetNodeResult(nodes[0], H.HvxMeanStdDev())
    assert (m.sum, m.sum_squares, m.count) == O.mean_stddev(ref)[2]
    r, want = H.hvxGetNodeResult(nodes[1], H.HvxMinMaxLoc()), O.minmaxloc(ref)
    assert (r.min, r.max, r.min_count, r.max_count) == (want["min"], want["max"],
                                                        want["min_count"], want["max_count"])
    np.testing.assert_array_equal(H.hvxGetNodeResult(nodes[2], np.zeros(256, np.uint32)),
                                  O.histogram(ref, 256, 0, 256))


@pytest.mark.parametrize("codegen", [H.HVX_CODEGEN_OFF, H.HVX_CODEGEN_REQUIRE])
def test_graph_that_occurs_twice_in_a_batch(ctx, codegen):
    graphs = [single_group(ctx, w, h, w, codegen) for w, h in [(640, 480), (7, 5), (1920, 1080)]]
    for order in ([0, 2, 0, 1, 2, 2], [0, 1, 2], [2, 2], [1]):
        for _ in range(2):
            H.hvxProcessGraphBatch([graphs[i][0] for i in order])
            H.hvxWaitBatch(ctx)
            for i in order:
                check_group(*graphs[i][1:])


def test_graph_on_several_streams_without_waits(ctx):
    s = Statistics(ctx, 1920, 1080, seed=8)
    H.hvxVerifyGraph(s.g)
    g, nodes, ref = single_group(ctx, 1921, 1081, 9)
    streams = [torch.cuda.Stream() for _ in range(3)]
    for k in range(30):
        H.hvxScheduleGraph(s.g, streams[k % 3].cuda_stream)
        # alone and as a batch in turn
        if k % 2:
            H.hvxProcessGraphBatch([g], streams[(k + 1) % 3].cuda_stream)
        else:
            H.hvxScheduleGraph(g, streams[(k + 2) % 3].cuda_stream)
    torch.cuda.synchronize()
    s.check()
    check_group(nodes, ref)
    # a server between two runs on a stream
    server = H.hvxCreateServer(ctx, 0, 4, 4)
    for _ in range(5):
        H.hvxScheduleGraph(s.g, streams[0].cuda_stream)
        ticket = H.hvxServerSubmit(server, s.g)
        H.hvxServerWait(server, ticket)
        s.check()
    H.hvxReleaseServer(server)


def test_blocks_of_a_released_graph_are_idle(ctx):
    """A graph released right after its launch: its blocks go to a new graph of
    the same shape, whose first run must find them clear."""
    side = torch.cuda.Stream()
    for k in range(10):
        g, _, _ = single_group(ctx, 1920, 1080, k)
        H.hvxProcessGraphBatch([g], side.cuda_stream)
        H.hvxReleaseGraph(g)
        g, nodes, ref = single_group(ctx, 640, 480, 20 + k)
        H.hvxProcessGraph(g)
        check_group(nodes, ref)
        H.hvxReleaseGraph(g)


@pytest.mark.parametrize("w,h", [(7, 5), (1920, 1080)])
def test_only_results_count_against_the_budget(w, h):
    """256 bytes (the pool's step) for MeanStdDev and MinMaxLoc, 1024 for 256
    bins, whatever the image's size: a budget of just that verifies."""
    c = H.hvxCreateContext()
    try:
        src = PG.upload(c, synth.rects_noise(w, h, 1), H.HVX_DF_U8)
        used = H.hvxGetContextMemoryUsage(c)
        g = H.hvxCreateGraph(c)
        H.hvxMeanStdDevNode(g, src)
        mm = H.hvxMinMaxLocNode(g, src)
        H.hvxHistogramNode(g, src, 256, 0, 256)
        H.hvxSetContextMemoryBudget(c, used + 256 + 256 + 1024)
        H.hvxVerifyGraph(g)
        assert H.hvxGetContextMemoryUsage(c) == used + 256 + 256 + 1024
        H.hvxProcessGraph(g)
        img = PG.download(src)
        assert H.hvxGetNodeResult(mm, H.HvxMinMaxLoc()).max_count == (img == img.max()).sum()
    finally:
        H.hvxReleaseContext(c)


def test_minmax_of_every_tile_count():
    """The extrema's scratch holds one entry per CTA: sizes around the limits of
    one tile, of tiles per CTA and of 1024 CTAs, alone and batched."""
    c = H.hvxCreateContext()
    try:
        graphs = []
        for w, h in [(1, 1), (128, 24), (129, 25), (1, 32768), (32768, 1), (4096, 2160)]:
            img = synth.uniform_u8(w, h, w + h)
            g = H.hvxCreateGraph(c)
            mm = H.hvxMinMaxLocNode(g, PG.upload(c, img, H.HVX_DF_U8))
            H.hvxVerifyGraph(g)
            graphs.append((g, mm, img))
        for batch in (False, True):
            if batch:
                H.hvxProcessGraphBatch([g for g, _, _ in graphs])
            else:
                for g, _, _ in graphs:
                    H.hvxScheduleGraph(g)
            H.hvxWaitBatch(c)
            for _, mm, img in graphs:
                r = H.hvxGetNodeResult(mm, H.HvxMinMaxLoc())
                assert (r.min, r.max, r.min_count, r.max_count) == (
                    img.min(), img.max(), (img == img.min()).sum(), (img == img.max()).sum())
                assert img.argmin() == r.min_y * img.shape[1] + r.min_x
    finally:
        H.hvxReleaseContext(c)
