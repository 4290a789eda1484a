"""Global operators read only the valid region of a stored image (hvx.h), also
where a kernel's interior tiles reach its rim: with fusion off, Gaussian3x3
UNDEFINED is stored with a zero rim and reduced by a second launch.  Widths and
heights that tiles divide, and ragged ones.  Reference: numpy on the oracle's
valid region."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("rows", ["", "3", "24", "0"])  # "0": the tile form
@pytest.mark.parametrize("codegen", [H.HVX_CODEGEN_OFF, H.HVX_CODEGEN_REQUIRE])
@pytest.mark.parametrize("w,h", [(128, 24), (256, 192), (384, 576), (260, 200), (2, 2), (1920, 1080)])
def test_reductions_of_a_stored_image(ctx, w, h, codegen, rows, monkeypatch):
    if rows:
        monkeypatch.setenv("HVX_STRIP_ROWS", rows)
    img = 1 + synth.uniform_u8(w, h, seed=w) // 2  # no zeros but the rim's
    src = PG.upload(ctx, img, H.HVX_DF_U8)
    g = H.hvxCreateGraph(ctx)
    b = H.hvxCreateVirtualImage(g)
    H.hvxSetNodeBorder(H.hvxGaussian3x3Node(g, src, b), H.HVX_BORDER_UNDEFINED, 0)
    nodes = (H.hvxMeanStdDevNode(g, b), H.hvxMinMaxLocNode(g, b),
             H.hvxHistogramNode(g, b, 256, 0, 256))
    H.hvxSetGraphFusion(g, False)
    H.hvxSetGraphCodegen(g, codegen)
    H.hvxVerifyGraph(g)
    assert H.hvxQueryGraph(g, H.HVX_GRAPH_NUM_LAUNCHES) == 4
    H.hvxProcessGraphBatch([g])
    H.hvxWaitBatch(ctx)
    ref = O.gaussian3x3(img, O.BORDER_UNDEFINED)
    x0, y0, x1, y1 = ref.rect
    v = ref.data[y0:y1, x0:x1].astype(np.int64)
    m = H.hvxGetNodeResult(nodes[0], H.HvxMeanStdDev())
    assert (m.sum, m.sum_squares, m.count) == (v.sum(), (v * v).sum(), v.size)
    r = H.hvxGetNodeResult(nodes[1], H.HvxMinMaxLoc())
    if v.size:
        assert (r.min, r.max, r.min_count, r.max_count) == (
            v.min(), v.max(), (v == v.min()).sum(), (v == v.max()).sum())
    else:
        assert (r.min_count, r.max_count, r.min_x) == (0, 0, -1)
    np.testing.assert_array_equal(H.hvxGetNodeResult(nodes[2], np.zeros(256, np.uint32)),
                                  np.bincount(v.ravel(), minlength=256))
    H.hvxReleaseGraph(g)


@pytest.mark.parametrize("w,h", [(256, 192), (260, 200)])
def test_batched_reductions_of_stored_images(ctx, w, h):
    """Images stored by one graph's launches and reduced in a batch: the batch's
    graphs read them as whole images, rim included."""
    outs, graphs, nodes = [], [], []
    for k in range(3):
        img = synth.uniform_u8(w, h, seed=k)
        g = H.hvxCreateGraph(ctx)
        outs.append(PG.empty(ctx, w, h, H.HVX_DF_U8))
        H.hvxSetNodeBorder(H.hvxGaussian3x3Node(g, PG.upload(ctx, img, H.HVX_DF_U8), outs[-1]),
                           H.HVX_BORDER_UNDEFINED, 0)
        H.hvxVerifyGraph(g)
        H.hvxProcessGraph(g)
        g = H.hvxCreateGraph(ctx)
        nodes.append(H.hvxMeanStdDevNode(g, outs[-1]))
        H.hvxVerifyGraph(g)
        graphs.append(g)
    H.hvxProcessGraphBatch(graphs)
    H.hvxWaitBatch(ctx)
    for o, n in zip(outs, nodes):
        v = PG.download(o).astype(np.int64)
        m = H.hvxGetNodeResult(n, H.HvxMeanStdDev())
        assert (m.sum, m.sum_squares, m.count) == (v.sum(), (v * v).sum(), v.size)
