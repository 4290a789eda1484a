"""Kernels launched with programmatic serialisation run while the kernel ahead of
them may still write their input images, so they must not read images by
read-only (__ldg) loads; those stay for tables that were uploaded before the
launch, and for kernels that are launched in the ordinary way (the tile form's
batch kernel)."""
import pathlib
import re

import pytest

from paper_2008_11476_gb300 import apps as A
from paper_2008_11476_gb300 import hvx as H

CSRC = pathlib.Path(H.__file__).parent / "csrc"
# first operand of the read-only loads of tables
TABLES = re.compile(r"__ldg\((d\.tile_start|d\.tiles_x|tile_start|tiles_x|cta_start)\b|"
                    r"__ldg\(reinterpret_cast<const uint32_t\*>\(ps \+ i\)")


@pytest.fixture
def pctx():
    c = H.hvxCreateContextEx(H.HVX_CONTEXT_PLAN_ONLY)
    yield c
    H.hvxReleaseContext(c)


def image_reads(source):
    # hvx_ld's read-only branch is taken with GMAP alone, in the batch kernel
    source = re.sub(r"  if \(RO\) \{.*?\n  \}\n", "", source, flags=re.S)
    assert not re.search(r"hvx_ld<\d+, true>", source)
    single = source.split("hvx_generated_batch")[0]
    assert not re.search(r"hvx_tile<\w+, true>\(p", single)
    return [source[m.start():m.start() + 60] for m in re.finditer(r"__ldg\(", source)
            if not TABLES.match(source, m.start())]


def point_group(ctx):
    g = H.hvxCreateGraph(ctx)
    a = H.hvxCreateImage(ctx, 300, 200, H.HVX_DF_U8)
    v = H.hvxCreateVirtualImage(g)
    H.hvxNotNode(g, a, v)
    H.hvxXorNode(g, v, a, H.hvxCreateImage(ctx, 300, 200, H.HVX_DF_U8))
    return g


def statistics_group(ctx):
    g = H.hvxCreateGraph(ctx)
    y = H.hvxCreateVirtualImage(g)
    H.hvxChannelExtractNode(g, H.hvxCreateImage(ctx, 300, 200, H.HVX_DF_UYVY), H.HVX_CHANNEL_Y, y)
    H.hvxMeanStdDevNode(g, y)
    H.hvxMinMaxLocNode(g, y)
    return g


def s32_group(ctx):
    """S32 images keep the tile form."""
    g = H.hvxCreateGraph(ctx)
    a, b = (H.hvxCreateImage(ctx, 300, 200, H.HVX_DF_S16) for _ in range(2))
    v = H.hvxCreateVirtualImage(g)
    H.hvxPointNode(g, H.HVX_POINT_MUL, [a, b], v)
    H.hvxLocalNode(g, H.HVX_LOCAL_SUM, 5, 5, v, H.hvxCreateImage(ctx, 300, 200, H.HVX_DF_S32))
    return g


@pytest.mark.parametrize("build", [point_group, statistics_group, s32_group])
def test_generated_groups_read_images_by_ordinary_loads(pctx, build):
    g = build(pctx)
    H.hvxSetGraphCodegen(g, H.HVX_CODEGEN_REQUIRE)
    H.hvxVerifyGraph(g)
    assert image_reads(H.hvxGetGraphKernelSource(g, 0)) == []


@pytest.mark.parametrize("name", [a for a, _ in A.APPS])
def test_generated_applications_read_images_by_ordinary_loads(pctx, name):
    src = H.hvxCreateImage(pctx, 1920, 1080, H.HVX_DF_U8)
    g, _ = dict(A.APPS)[name](pctx, src, 1920, 1080, True)
    H.hvxSetGraphCodegen(g, H.HVX_CODEGEN_ONLY)
    H.hvxVerifyGraph(g)
    assert image_reads(H.hvxGetGraphKernelSource(g, 0)) == []


def test_hand_written_kernels_read_images_by_ordinary_loads():
    files = [*CSRC.glob("*.cu"), *CSRC.glob("*.cuh")]
    assert len(files) > 5
    for f in files:
        assert image_reads(f.read_text()) == [], f.name
