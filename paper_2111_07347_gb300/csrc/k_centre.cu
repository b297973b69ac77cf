// Direct-beam centring (arXiv 2111.07347 Section 3.1: the direct beam of every pattern was
// centred before the polar transform, whose origin must be the beam's centre, Section 2.2).
// Per pattern, the intensity-weighted centre of mass of the pixels within `radius` of the
// current estimate, repeated `iterations` times from the starting centre.
//
// The disc's bounding box is visited row by row in FP64 with explicitly rounded operations (no fused
// multiply-adds), so the sums, and hence the centres, are the same bit for bit as a plain
// double-precision loop in the same order.  The work is a few hundred pixels per pattern; the
// frames' other pixels are not read.  A thread per pattern takes a time that depends on the disc
// alone until the patterns fill the GPU, a warp per pattern is faster for few patterns or (u16) large
// discs: launch_find_centres.
#include "tm_internal.h"

namespace tmgb {
namespace {

// A thread per pattern: a plain loop.
template <typename T>
__global__ void find_centres_thread_kernel(const T* __restrict__ frames, int64_t n, int H, int W, double cx0, double cy0,
                                    double radius, int iterations, float2* __restrict__ out) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const T* f = frames + (size_t)p * H * W;
    const double r2 = __dmul_rn(radius, radius);
    double cx = cx0, cy = cy0;
    for (int it = 0; it < iterations; ++it) {
        const int y_lo = max(0, (int)ceil(__dsub_rn(cy, radius)));
        const int y_hi = min(H - 1, (int)floor(__dadd_rn(cy, radius)));
        const int x_lo = max(0, (int)ceil(__dsub_rn(cx, radius)));
        const int x_hi = min(W - 1, (int)floor(__dadd_rn(cx, radius)));
        double s0 = 0.0, sx = 0.0, sy = 0.0;
        for (int y = y_lo; y <= y_hi; ++y) {
            const double dy = __dsub_rn((double)y, cy);
            const double dy2 = __dmul_rn(dy, dy);
            for (int x = x_lo; x <= x_hi; ++x) {
                const double dx = __dsub_rn((double)x, cx);
                if (__dadd_rn(__dmul_rn(dx, dx), dy2) <= r2) {
                    const double v = (double)__ldg(f + (size_t)y * W + x);
                    s0 = __dadd_rn(s0, v);
                    sx = __dadd_rn(sx, __dmul_rn((double)x, v));
                    sy = __dadd_rn(sy, __dmul_rn((double)y, v));
                }
            }
        }
        if (s0 > 0.0) {
            cx = __ddiv_rn(sx, s0);
            cy = __ddiv_rn(sy, s0);
        }
    }
    out[p] = make_float2((float)cx, (float)cy);
}

// One warp per pattern: the lanes take 32 pixels of the disc's box in row order, test them and form
// their terms (v, x v, y v; 0 outside the disc, which adds nothing), and lanes 0, 1, 2 add the three
// sums' terms one after the other in that order -- the sums of a plain loop over rows and columns, bit
// for bit.  (A thread per pattern, loading and adding pixel by pixel, took 168 us for any few patterns.)
template <typename T>
__global__ void __launch_bounds__(128)
find_centres_kernel(const T* __restrict__ frames, int64_t n, int H, int W, double cx0, double cy0, double radius,
                    int iterations, float2* __restrict__ out) {
    __shared__ double terms[4][3][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (p >= n) return;
    const T* f = frames + (size_t)p * H * W;
    const double r2 = __dmul_rn(radius, radius);
    double cx = cx0, cy = cy0;
    for (int it = 0; it < iterations; ++it) {
        const int y_lo = max(0, (int)ceil(__dsub_rn(cy, radius)));
        const int y_hi = min(H - 1, (int)floor(__dadd_rn(cy, radius)));
        const int x_lo = max(0, (int)ceil(__dsub_rn(cx, radius)));
        const int x_hi = min(W - 1, (int)floor(__dadd_rn(cx, radius)));
        const int w = max(0, x_hi - x_lo + 1), h = max(0, y_hi - y_lo + 1);
        double sum = 0.0;                                   // lane 0: v, 1: x v, 2: y v
        for (int64_t i0 = 0; i0 < (int64_t)w * h; i0 += 32) {
            const int64_t i = i0 + lane;
            double v = 0.0, xv = 0.0, yv = 0.0;
            if (i < (int64_t)w * h) {
                const int y = y_lo + (int)(i / w), x = x_lo + (int)(i % w);
                const double dy = __dsub_rn((double)y, cy), dx = __dsub_rn((double)x, cx);
                if (__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)) <= r2) {
                    v = (double)__ldg(f + (size_t)y * W + x);
                    xv = __dmul_rn((double)x, v);
                    yv = __dmul_rn((double)y, v);
                }
            }
            terms[warp][0][lane] = v;
            terms[warp][1][lane] = xv;
            terms[warp][2][lane] = yv;
            __syncwarp();
            if (lane < 3) {
#pragma unroll 8
                for (int j = 0; j < 32; ++j) sum = __dadd_rn(sum, terms[warp][lane][j]);
            }
            __syncwarp();
        }
        const double s0 = __shfl_sync(0xffffffffu, sum, 0), sx = __shfl_sync(0xffffffffu, sum, 1),
                     sy = __shfl_sync(0xffffffffu, sum, 2);
        if (s0 > 0.0) {
            cx = __ddiv_rn(sx, s0);
            cy = __ddiv_rn(sy, s0);
        }
    }
    if (lane == 0) out[p] = make_float2((float)cx, (float)cy);
}

// u16 frames, one warp per pattern: the sums are of integers below 2^53 (the caller sees to it), so
// they are exact in any order and equal the serial sums above; every pixel's test and the divisions
// are the same operations.  16 us for a few patterns and 55 us for 4096 (a thread per pattern: 168 and
// 191 us).
__global__ void __launch_bounds__(128)
find_centres_u16_kernel(const uint16_t* __restrict__ frames, int64_t n, int H, int W, double cx0, double cy0,
                        double radius, int iterations, float2* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (p >= n) return;
    const uint16_t* f = frames + (size_t)p * H * W;
    const double r2 = __dmul_rn(radius, radius);
    double cx = cx0, cy = cy0;
    for (int it = 0; it < iterations; ++it) {
        const int y_lo = max(0, (int)ceil(__dsub_rn(cy, radius)));
        const int y_hi = min(H - 1, (int)floor(__dadd_rn(cy, radius)));
        const int x_lo = max(0, (int)ceil(__dsub_rn(cx, radius)));
        const int x_hi = min(W - 1, (int)floor(__dadd_rn(cx, radius)));
        const int w = x_hi - x_lo + 1, h = y_hi - y_lo + 1;
        unsigned long long s0 = 0, sx = 0, sy = 0;
        for (int i = lane; w > 0 && h > 0 && i < w * h; i += 32) {
            const int y = y_lo + i / w, x = x_lo + i % w;
            const unsigned v = __ldg(f + (size_t)y * W + x);
            const double dy = __dsub_rn((double)y, cy), dx = __dsub_rn((double)x, cx);
            if (__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)) <= r2) {
                s0 += v;
                sx += (unsigned long long)x * v;
                sy += (unsigned long long)y * v;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
            sy += __shfl_xor_sync(0xffffffffu, sy, o);
        }
        if (s0 > 0) {
            cx = __ddiv_rn((double)sx, (double)s0);
            cy = __ddiv_rn((double)sy, (double)s0);
        }
    }
    if (lane == 0) out[p] = make_float2((float)cx, (float)cy);
}

}  // namespace

cudaError_t launch_find_centres(const void* frames, int dtype, int64_t n, int H, int W, double cx0, double cy0,
                                double radius, int iterations, float2* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int threads = 128;
    const int64_t grid = (n + 3) / 4;
    // exact in any order while pixels x value x coordinate stays below 2^53
    const double side = 2.0 * radius + 1.0;
    const double pixels = (side < W ? side : W) * (side < H ? side : H);
    const bool exact = dtype == TM_DTYPE_U16 && pixels * 65535.0 * (W > H ? W : H) < 9.0e15 && pixels < 2.0e9;
    // A warp's time grows with the patterns and its steps of 32 pixels, a thread's with the pixels alone
    // (up to about 20000 patterns).  256 x 256 frames, warp / thread us: exact sums, 16384 patterns,
    // radius 1 109 / 14, radius 3 156 / 51, radius 6 203 / 191; f32, 4096 patterns, radius 1 55 / 14,
    // radius 3 90 / 51, radius 6 185 / 191, radius 20 1620 / 2015; 16384, radius 6 718 / 191, 20 6495 / 2100.
    const double steps = ceil(pixels / 32.0);
    const bool warps = exact ? n <= 96.0 * pixels || pixels >= 400.0 : n * (steps + 1.0) <= 150.0 * pixels;
    if (!warps) {
        const unsigned blocks = (unsigned)((n + threads - 1) / threads);
        if (dtype == TM_DTYPE_U16)
            find_centres_thread_kernel<uint16_t><<<blocks, threads, 0, st>>>((const uint16_t*)frames, n, H, W, cx0, cy0,
                                                                             radius, iterations, out);
        else
            find_centres_thread_kernel<float><<<blocks, threads, 0, st>>>((const float*)frames, n, H, W, cx0, cy0, radius,
                                                                          iterations, out);
        return cudaGetLastError();
    }
    if (exact) {
        find_centres_u16_kernel<<<(unsigned)grid, threads, 0, st>>>((const uint16_t*)frames, n, H, W, cx0, cy0, radius,
                                                                    iterations, out);
        return cudaGetLastError();
    }
    if (dtype == TM_DTYPE_U16)
        find_centres_kernel<uint16_t><<<(unsigned)grid, threads, 0, st>>>((const uint16_t*)frames, n, H, W, cx0, cy0,
                                                                          radius, iterations, out);
    else
        find_centres_kernel<float><<<(unsigned)grid, threads, 0, st>>>((const float*)frames, n, H, W, cx0, cy0,
                                                                       radius, iterations, out);
    return cudaGetLastError();
}

}  // namespace tmgb
