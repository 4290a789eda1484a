// The strip form of a generated kernel (codegen_strip.cpp): source emission for
// a fused group whose images all fit 16-bit lanes.
#pragma once

#include <string>
#include <vector>

#include "kernel_params.h"

namespace hvx {

constexpr int STRIP_TW = 128;       // tile width: 16 strips of 8 pixels
constexpr int STRIP_THREADS = 128;  // 16 strips x 8 row groups
constexpr int STRIP_BOX_W = 160;    // TMA box width in pixels: 16 to each side of the tile

// An external input read with a halo: one TMA box per tile.
struct StripBox {
    int ext;   // external input
    int elem;  // bytes per pixel (1 or 2)
    int halo;
};

struct StripPlan {
    int unroll = 0;  // rows per thread are a multiple of this
    std::vector<StripBox> boxes;
    bool reduces = false;  // has global operators: p.ctas CTAs per image over its tiles
};

// Bytes of shared memory of a strip tile with `rows` rows per thread: the
// mbarrier's 128 bytes, then the boxes, each 128-byte aligned.
inline int strip_smem_bytes(const StripPlan& s, int rows) {
    int n = 128;
    for (const StripBox& b : s.boxes)
        n += (STRIP_BOX_W * b.elem * (8 * rows + 2 * b.halo) + 127) & ~127;
    return n;
}

// Emits the strip kernels of a group, or returns false when some image or
// operator of the group does not fit the form.
bool emit_strips(const GenericDesc& d, std::string* source, StripPlan* plan);

}  // namespace hvx
