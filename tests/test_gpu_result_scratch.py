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
