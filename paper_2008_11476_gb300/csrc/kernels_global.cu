// EqualizeHist (Table 2: histogram + point).  The mapping of every pixel
// needs the histogram of the whole image, so it takes two launches: a
// histogram of the input's valid rectangle, whose last CTA to finish forms the
// 256-entry table from the cumulative histogram, then the mapping.
//
// Both kernels take 16 pixels per thread step (one 16-byte access; rows start
// 16-byte aligned) and spread the steps of all rows evenly over the threads.
// The histogram is bound by shared-memory atomics: 8 copies of the bins, one
// per lane modulo 8, halve the bank conflicts of one copy.  The mapping is
// bound by the latency of its loads and the byte look-ups in shared memory.
// 3840x2160 (cold L2, one launch each): count 16.0 -> 11.5 us, mapping 23.4 ->
// 7.4 us against one pixel per thread step (12.7 and 9.6 without the loads one
// step ahead).
#include "device_common.cuh"
#include "launchers.h"

namespace hvx {
namespace {

using namespace dev;

constexpr int kThreads = 256;
constexpr int kCopies = 8;

__device__ __forceinline__ uint32_t byte_of(const uint4& v, int j) {
    const uint32_t w = j < 8 ? (j < 4 ? v.x : v.y) : (j < 12 ? v.z : v.w);
    return (w >> (8 * (j & 3))) & 0xFFu;
}

// Step i of an image's rows (per_row steps of 16 pixels each from column a0 on),
// with its pixels where all 16 lie in columns v0 .. v2 - 1.  An ordinary load:
// the kernel before this one may write the image while this one already runs
// (programmatic dependent launches), which the read-only path does not allow.
struct Step {
    unsigned r;
    int x;
    bool full;
    uint4 v;
};
__device__ __forceinline__ Step load_step(const uint8_t* base, uint64_t pitch, unsigned i,
                                          unsigned per_row, int a0, int v0, int v2) {
    Step s;
    s.r = i / per_row;
    s.x = a0 + 16 * (int)(i - s.r * per_row);
    s.full = s.x >= v0 && s.x + 16 <= v2;
    s.v = make_uint4(0u, 0u, 0u, 0u);
    if (s.full) s.v = *reinterpret_cast<const uint4*>(base + (size_t)s.r * pitch + s.x);
    return s;
}

__global__ void __launch_bounds__(kThreads) eqhist_count_kernel(const EqHistParams p) {
    __shared__ uint32_t bins[256 * kCopies];
    __shared__ uint32_t c[256];
    __shared__ uint32_t cmin;
    __shared__ bool last;
    pdl_launch_dependents();  // launched by launch_pdl
    for (int i = threadIdx.x; i < 256 * kCopies; i += kThreads) bins[i] = 0;
    __syncthreads();
    pdl_wait();
    const int v0 = p.valid[0], v2 = p.valid[2], h = p.valid[3] - p.valid[1];
    const int a0 = v0 & ~15, per_row = (v2 - a0 + 15) / 16;
    const unsigned copy = threadIdx.x & (kCopies - 1);
    const unsigned steps = v2 > v0 && h > 0 ? (unsigned)h * (unsigned)per_row : 0u;
    const uint8_t* base = p.in + (size_t)p.valid[1] * p.in_pitch;
    const unsigned stride = gridDim.x * kThreads;
    unsigned i = blockIdx.x * kThreads + threadIdx.x;
    Step s = {};
    if (i < steps) s = load_step(base, p.in_pitch, i, (unsigned)per_row, a0, v0, v2);
    while (i < steps) {
        // the next step's load ahead of this one's atomics
        Step n = {};
        if (i + stride < steps)
            n = load_step(base, p.in_pitch, i + stride, (unsigned)per_row, a0, v0, v2);
        if (s.full) {
#pragma unroll
            for (int j = 0; j < 16; ++j) atomicAdd(&bins[byte_of(s.v, j) * kCopies + copy], 1u);
        } else {
            const uint8_t* row = base + (size_t)s.r * p.in_pitch;
            for (int j = max(s.x, v0); j < min(s.x + 16, v2); ++j)
                atomicAdd(&bins[row[j] * kCopies + copy], 1u);
        }
        s = n;
        i += stride;
    }
    __syncthreads();
    const unsigned t = threadIdx.x;
    uint32_t sum = 0;
    for (int k = 0; k < kCopies; ++k) sum += bins[t * kCopies + k];
    if (sum) atomicAdd(&p.hist[t], sum);
    // (the barrier orders the CTA's additions before thread 0's cumulative fence)
    __syncthreads();
    if (t == 0) {
        __threadfence();
        last = atomicAdd(p.done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the last CTA: the table, and bins and counter back to zero
    c[t] = atomicExch(&p.hist[t], 0u);
    if (t == 0) {
        *p.done = 0u;
        cmin = 0xFFFFFFFFu;
    }
    __syncthreads();
    // inclusive prefix sum of the 256 bins (Hillis-Steele, 8 steps)
    for (int o = 1; o < 256; o <<= 1) {
        const uint32_t v = t >= (unsigned)o ? c[t - o] : 0u;
        __syncthreads();
        c[t] += v;
        __syncthreads();
    }
    const unsigned long long n = c[255];
    // cmin: the cumulative count at the smallest value present = the
    // smallest nonzero prefix
    if (c[t]) atomicMin(&cmin, c[t]);
    __syncthreads();
    const unsigned long long den = n - cmin;
    if (n == 0 || den == 0) {
        p.lut[t] = (uint8_t)t;  // constant image: unchanged
    } else {
        const unsigned long long cv = c[t] > cmin ? c[t] - cmin : 0ull;
        p.lut[t] = (uint8_t)((2ull * cv * 255ull + den) / (2ull * den));  // halves rounded up
    }
}

__global__ void __launch_bounds__(kThreads) eqhist_map_kernel(const EqHistParams p) {
    __shared__ uint8_t lut[256];
    pdl_launch_dependents();  // launched by launch_pdl
    pdl_wait();
    lut[threadIdx.x] = p.lut[threadIdx.x];
    __syncthreads();
    const int W = (int)p.W, v0 = p.valid[0], v2 = p.valid[2];
    const unsigned per_row = (unsigned)(W + 15) / 16, steps = per_row * p.H;
    const unsigned stride = gridDim.x * kThreads;
    for (unsigned i = blockIdx.x * kThreads + threadIdx.x; i < steps; i += 2 * stride) {
        Step s[2];  // both loads ahead of the first store
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (i + u * stride < steps)
                s[u] = load_step(p.in, p.in_pitch, i + u * stride, per_row, 0, v0, v2);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (i + u * stride >= steps) break;
            const int x = s[u].x, y = (int)s[u].r;
            uint8_t* out = p.out + (size_t)y * p.out_pitch;
            const bool yin = y >= p.valid[1] && y < p.valid[3];
            if (yin && s[u].full) {
                uint32_t o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t lo = lut[byte_of(s[u].v, 4 * k)] |
                                        (uint32_t)lut[byte_of(s[u].v, 4 * k + 1)] << 8;
                    const uint32_t hi = lut[byte_of(s[u].v, 4 * k + 2)] |
                                        (uint32_t)lut[byte_of(s[u].v, 4 * k + 3)] << 8;
                    o[k] = lo | hi << 16;
                }
                *reinterpret_cast<uint4*>(out + x) = make_uint4(o[0], o[1], o[2], o[3]);
            } else {
                const uint8_t* in = p.in + (size_t)y * p.in_pitch;
                for (int j = x; j < min(x + 16, W); ++j)
                    out[j] = yin && j >= v0 && j < v2 ? lut[in[j]] : 0;
            }
        }
    }
}

// CTAs for `steps` thread steps: at most 8 per SM.
int grid_for(unsigned long long steps, int num_sms) {
    const unsigned long long n = (steps + kThreads - 1) / kThreads;
    const unsigned long long most = 8ull * (unsigned long long)num_sms;
    return (int)(n < 1 ? 1 : n < most ? n : most);
}

}  // namespace

cudaError_t launch_eqhist(const EqHistParams& p, cudaStream_t s) {
    const unsigned long long steps = (unsigned long long)((p.W + 15) / 16) * p.H;
    // (about 4 steps per thread share the count's 8 KB of bins and its commit)
    cudaError_t e = launch_pdl(eqhist_count_kernel, dim3(grid_for((steps + 3) / 4, p.num_sms)),
                               dim3(kThreads), 0, s, p);
    if (e != cudaSuccess) return e;
    return launch_pdl(eqhist_map_kernel, dim3(grid_for(steps, p.num_sms)), dim3(kThreads), 0, s, p);
}

}  // namespace hvx
