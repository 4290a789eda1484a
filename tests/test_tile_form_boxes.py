"""Destinations of the tile form's TMA boxes: a 128-byte boundary of shared
memory, whatever lies before them (bins of a histogram, another box)."""
import re

import numpy as np
import pytest

from paper_2008_11476_gb300 import hvx as H


@pytest.fixture
def pctx():
    c = H.hvxCreateContextEx(H.HVX_CONTEXT_PLAN_ONLY)
    yield c
    H.hvxReleaseContext(c)


def boxes(g):
    """Word offsets in shared memory of the group's box destinations."""
    H.hvxSetGraphCodegen(g, H.HVX_CODEGEN_ONLY)
    H.hvxVerifyGraph(g)
    assert H.hvxQueryGraph(g, H.HVX_GRAPH_NUM_LAUNCHES) == 1
    s = H.hvxGetGraphKernelSource(g, 0).split("#ifndef HVX_STRIPS")[1].split("#endif")[0]
    assert re.findall(r"extern __shared__ __align__\((\d+)\) int smem", s) == ["128", "128"]
    at = dict(re.findall(r"unsigned char\* const (B\d+) = \(unsigned char\*\)\(smem \+ (\d+)\)", s))
    return [int(at[b]) for b in re.findall(r"hvx_tma_2d\((B\d+),", s)]


def test_box_after_bins(pctx):
    w, h = 300, 200
    src = H.hvxCreateImage(pctx, w, h, H.HVX_DF_U8)
    g = H.hvxCreateGraph(pctx)
    d = H.hvxCreateVirtualImage(g)
    # sums beyond 16 bits: the tile form
    H.hvxConvolveNode(g, src, np.full(25, 30), 5, 5, 1, H.hvxCreateImage(pctx, w, h, H.HVX_DF_S16))
    H.hvxCopyNode(g, src, d)
    H.hvxHistogramNode(g, d, 7, 20, 200)
    assert [b % 32 for b in boxes(g)] == [0]
    assert "hvx_generated_strips" not in H.hvxGetGraphKernelSource(g, 0)


@pytest.mark.parametrize("halo", [2, 3, 4, 5])
def test_two_boxes(pctx, monkeypatch, halo):
    """|a - b| & (Dilate3x3(a) ^ Erode3x3(b)), then medians: both inputs are staged."""
    monkeypatch.setenv("HVX_STRIP_ROWS", "0")
    w, h = 300, 200
    a, b = (H.hvxCreateImage(pctx, w, h, H.HVX_DF_U8) for _ in range(2))
    g = H.hvxCreateGraph(pctx)
    e, d, f, x, o = (H.hvxCreateVirtualImage(g) for _ in range(5))
    H.hvxAbsDiffNode(g, a, b, e)
    H.hvxDilate3x3Node(g, a, d)
    H.hvxErode3x3Node(g, b, f)
    H.hvxXorNode(g, d, f, x)
    H.hvxAndNode(g, x, e, o)
    for _ in range(halo - 1):
        v, o = o, H.hvxCreateVirtualImage(g)
        H.hvxMedian3x3Node(g, v, o)
    H.hvxNotNode(g, o, H.hvxCreateImage(pctx, w, h, H.HVX_DF_U8))
    at = boxes(g)
    assert len(at) == 2 and all(b % 32 == 0 for b in at)
