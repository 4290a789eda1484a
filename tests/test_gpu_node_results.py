"""hvxGetNodeResult returns the last run's results, whichever form of the graph
wrote them (strip kernels also write a host copy, the others do not), and waits
for a run that was launched after the one waited for."""
import numpy as np
import pytest
import torch

from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

pytestmark = pytest.mark.gpu

W, HT = 640, 480


@pytest.fixture(scope="module")
def ctx():
    c = H.hvxCreateContext()
    yield c
    H.hvxReleaseContext(c)


def write(im, a):
    H.hvxCopyImage(im, a.ctypes.data, a.strides[0], H.HVX_WRITE)


def statistics(ctx, src):
    g = H.hvxCreateGraph(ctx)
    v = H.hvxCreateVirtualImage(g)
    H.hvxNotNode(g, src, v)
    return g, (H.hvxMeanStdDevNode(g, v), H.hvxMinMaxLocNode(g, v),
               H.hvxHistogramNode(g, v, 256, 0, 256))


def check(nodes, img):
    v = 255 - img.astype(np.int64)
    m = H.hvxGetNodeResult(nodes[0], H.HvxMeanStdDev())
    assert (m.sum, m.sum_squares, m.count) == (v.sum(), (v * v).sum(), v.size)
    r = H.hvxGetNodeResult(nodes[1], H.HvxMinMaxLoc())
    assert (r.min, r.max) == (v.min(), v.max())
    np.testing.assert_array_equal(H.hvxGetNodeResult(nodes[2], np.zeros(256, np.uint32)),
                                  np.bincount(v.ravel(), minlength=256))


@pytest.mark.parametrize("batch", [False, True], ids=["alone", "batch"])
def test_one_graph_through_every_form(ctx, batch, monkeypatch):
    src = PG.empty(ctx, W, HT, H.HVX_DF_U8)
    g, nodes = statistics(ctx, src)
    # strip form, interpreter, strip form, tile form, strip form
    forms = [(H.HVX_CODEGEN_REQUIRE, ""), (H.HVX_CODEGEN_OFF, ""), (H.HVX_CODEGEN_REQUIRE, ""),
             (H.HVX_CODEGEN_REQUIRE, "0"), (H.HVX_CODEGEN_REQUIRE, "")]
    last = None
    for k, (mode, rows) in enumerate(forms):
        img = synth.rects_noise(W, HT, seed=k)
        write(src, img)
        if rows:
            monkeypatch.setenv("HVX_STRIP_ROWS", rows)
        else:
            monkeypatch.delenv("HVX_STRIP_ROWS", raising=False)
        H.hvxSetGraphCodegen(g, mode)
        H.hvxVerifyGraph(g)
        if last is not None:
            check(nodes, last)  # not run in its new form yet
        if batch:
            H.hvxProcessGraphBatch([g])
            H.hvxWaitBatch(ctx)
        else:
            H.hvxProcessGraph(g)
        check(nodes, img)
        last = img
    H.hvxReleaseGraph(g)


@pytest.mark.parametrize("captured", [False, True])
def test_run_after_the_one_waited_for(ctx, captured):
    """A run on a side stream, then one on the default stream behind long copies
    (a batch, or the replay of a capture); the wait covers the first alone."""
    x = torch.empty((HT, W), dtype=torch.uint8, device="cuda")
    src = H.hvxCreateImageFromHandle(ctx, W, HT, H.HVX_DF_U8, x.data_ptr(), W)
    g, nodes = statistics(ctx, src)
    H.hvxVerifyGraph(g)
    side, cap = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    if captured:
        with torch.cuda.stream(side):
            cap.capture_begin()
            H.hvxProcessGraphBatch([g], side.cuda_stream)
            cap.capture_end()
    a = torch.ones(1 << 28, dtype=torch.uint8, device="cuda")
    b = torch.empty_like(a)
    imgs = [synth.rects_noise(W, HT, seed=s) for s in (50, 51)]
    dev = [torch.from_numpy(i).cuda() for i in imgs]
    x.copy_(dev[0])
    torch.cuda.synchronize()
    H.hvxScheduleGraph(g, side.cuda_stream)
    side.synchronize()
    for _ in range(300):  # some 25 ms
        b.copy_(a)
    x.copy_(dev[1])
    if captured:
        cap.replay()
    else:
        H.hvxProcessGraphBatch([g])
    H.hvxWaitGraph(g)
    check(nodes, imgs[1])
    H.hvxReleaseGraph(g)
