// Background removal and smoothing before the polar transform (arXiv 2111.07347, Section 3.1:
// the diffuse background of each pattern was removed with a difference of Gaussians and the
// result smoothed by a Gaussian blur).  Separable Gaussian filters with the edge pixel
// repeated outside the frame: a row pass, then a column pass, each output a sum over the
// 2R + 1 offsets in ascending order (FP32 multiply-adds), weights computed in double
// precision on the host and zero-padded to a multiple of four taps.
//
// Each thread computes eight consecutive outputs.  Taps go four at a time: the four inputs
// that enter the thread's window and the four weights are read once from shared memory and
// feed 32 multiply-adds (the window's other inputs stay in registers), so shared memory
// serves a quarter of an operand per multiply-add.
// gauss_rows_kernel: one warp per image row (256 outputs per pass over the row); the row and
//   a clamped halo are staged in shared memory with one padding word every eight, so the
//   lanes' stride-8 reads fall in distinct banks; up to two filters per pass (the two
//   Gaussians of the difference share the row).
// gauss_cols_kernel: one CTA per 32-column strip of a frame; the strip of one or two inputs
//   is staged in shared memory (rows clamped on reading), lanes are columns, each thread takes
//   eight consecutive rows; the difference of Gaussians (clipped at 0) is formed in the same
//   pass.
//
// gauss_stream_kernel: all of it in one pass over memory, for frames whose rolling rows fit in shared
//   memory.  A CTA streams down a band of rows of one frame, eight rows a step: (0) the row filters of
//   the eight newest rows into rings of the last 2 r + 8 (and fewer) rows; (1) the column filters
//   from the rings, eight rows a thread, and their clipped difference; (2) the blur's row filter of
//   these into a third ring; (3) the blur's column filter, written out.  Each thread's eight outputs
//   take the taps in two groups of eight per loop turn, so the window's registers need no moves; odd
//   row pitches keep the row filters' lanes (eight rows x four runs of columns) in distinct banks.  The
//   next step's pixels are loaded while a step is computed.  Sums run in the same order as in the
//   kernels above: the same bits.  4096 frames of 256 x 256 u16, sigma 1 / 4 and blur 1: 2.79 ms, the
//   four passes 5.79 ms (1 frame: 30 and 51 us; 64 frames: 103 and 115).  Bound by issue (70 % of
//   the slots, a third of them the 102 multiply-adds a pixel).  A frame is one band while there are two frames per SM; fewer
//   frames are cut into more bands, each repeating the filters' reach at its ends.
#include <algorithm>
#include <type_traits>

#include "tm_internal.h"

namespace tmgb {
namespace {

constexpr int kRowWarps = 8;
constexpr int kStrip = 32;
constexpr int kOut = 8;                                     // outputs per thread
constexpr int kTap = 4;                                     // taps per step (weights padded to it)

template <typename T>
__device__ __forceinline__ float as_float(T v) {
    return (float)v;
}

__host__ __device__ inline int padded_taps(int r) { return ((2 * r + 1 + kTap - 1) / kTap) * kTap; }

// Shared-memory index of row element e with one padding word every eight.
__device__ __forceinline__ int skew(int e) { return e + (e >> 3); }

// acc[j] += sum_t w[t] x[base + j + t] over t < nt (nt a multiple of kTap); x(e) reads
// element e.  The window of kOut + kTap inputs slides by kTap per step.
template <typename F>
__device__ __forceinline__ void conv8(float (&acc)[kOut], const float* __restrict__ w, int nt, int base, F x) {
    float a[kOut];
#pragma unroll
    for (int j = 0; j < kOut; ++j) a[j] = x(base + j);
    for (int t0 = 0; t0 < nt; t0 += kTap) {
        float b[kTap], wt[kTap];
#pragma unroll
        for (int u = 0; u < kTap; ++u) {
            b[u] = x(base + kOut + t0 + u);
            wt[u] = w[t0 + u];
        }
#pragma unroll
        for (int u = 0; u < kTap; ++u) {
#pragma unroll
            for (int j = 0; j < kOut; ++j) acc[j] = fmaf(wt[u], j + u < kOut ? a[j + u] : b[j + u - kOut], acc[j]);
        }
#pragma unroll
        for (int j = 0; j < kOut; ++j) a[j] = j + kTap < kOut ? a[j + kTap] : b[j + kTap - kOut];
    }
}

template <typename T>
__global__ void __launch_bounds__(32 * kRowWarps)
gauss_rows_kernel(const T* __restrict__ in, int64_t rows, int W, const float* __restrict__ w1, int r1,
                  const float* __restrict__ w2, int r2, float* __restrict__ out1, float* __restrict__ out2) {
    extern __shared__ float sm[];
    const int R = max(r1, w2 ? r2 : 0);
    const int nt1 = padded_taps(r1), nt2 = w2 ? padded_taps(r2) : 0;
    float* sw1 = sm;                                         // [nt1]
    float* sw2 = sw1 + nt1;                                  // [nt2]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int span = 32 * kOut;                              // outputs per pass over the row
    const int chunks = (W + span - 1) / span;
    const int ne = chunks * span + 2 * R + kOut + kTap;      // staged elements (pixel e - R, clamped)
    float* row_s = sw2 + nt2 + warp * skew(ne);
    for (int i = threadIdx.x; i < nt1; i += blockDim.x) sw1[i] = w1[i];
    for (int i = threadIdx.x; i < nt2; i += blockDim.x) sw2[i] = w2[i];
    __syncthreads();
    for (int64_t r = (int64_t)blockIdx.x * kRowWarps + warp; r < rows; r += (int64_t)gridDim.x * kRowWarps) {
        const T* src = in + (size_t)r * W;
        for (int e = lane; e < ne; e += 32) row_s[skew(e)] = as_float(__ldg(src + min(max(e - R, 0), W - 1)));
        __syncwarp();
        for (int c = 0; c < chunks; ++c) {
            const int x0 = c * span + kOut * lane;           // the thread's first output
            float acc[kOut];
#pragma unroll
            for (int j = 0; j < kOut; ++j) acc[j] = 0.0f;
            conv8(acc, sw1, nt1, x0 + (R - r1), [&](int e) { return row_s[skew(e)]; });
#pragma unroll
            for (int j = 0; j < kOut; ++j)
                if (x0 + j < W) out1[(size_t)r * W + x0 + j] = acc[j];
            if (w2) {
#pragma unroll
                for (int j = 0; j < kOut; ++j) acc[j] = 0.0f;
                conv8(acc, sw2, nt2, x0 + (R - r2), [&](int e) { return row_s[skew(e)]; });
#pragma unroll
                for (int j = 0; j < kOut; ++j)
                    if (x0 + j < W) out2[(size_t)r * W + x0 + j] = acc[j];
            }
        }
        __syncwarp();
    }
}

// dog: out = max(a - b, 0) with a the column filter of in1 by w1 and b that of in2 by w2;
// else out = a.
__global__ void __launch_bounds__(256)
gauss_cols_kernel(const float* __restrict__ in1, const float* __restrict__ in2, int64_t n, int H, int W,
                  const float* __restrict__ w1, int r1, const float* __restrict__ w2, int r2, int dog,
                  float* __restrict__ out) {
    extern __shared__ float sm[];
    const int nt1 = padded_taps(r1), nt2 = dog ? padded_taps(r2) : 0;
    float* sw1 = sm;
    float* sw2 = sw1 + nt1;
    float* s1 = sw2 + nt2;                                   // [H][kStrip]
    float* s2 = s1 + (size_t)H * kStrip;                     // [H][kStrip] (dog)
    for (int i = threadIdx.x; i < nt1; i += blockDim.x) sw1[i] = w1[i];
    for (int i = threadIdx.x; i < nt2; i += blockDim.x) sw2[i] = w2[i];
    const int strips = (W + kStrip - 1) / kStrip;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int64_t t = blockIdx.x; t < n * strips; t += gridDim.x) {
        const int64_t p = t / strips;
        const int x0 = (int)(t - p * strips) * kStrip;
        const int x = x0 + lane;
        const bool col = x < W;
        const size_t base = (size_t)p * H * W;
        __syncthreads();                                     // previous strip's reads are done
        for (int y = warp; y < H; y += nwarps) {
            s1[y * kStrip + lane] = col ? __ldg(in1 + base + (size_t)y * W + x) : 0.0f;
            if (dog) s2[y * kStrip + lane] = col ? __ldg(in2 + base + (size_t)y * W + x) : 0.0f;
        }
        __syncthreads();
        if (!col) continue;
        for (int y0 = kOut * warp; y0 < H; y0 += kOut * nwarps) {
            float a[kOut];
#pragma unroll
            for (int j = 0; j < kOut; ++j) a[j] = 0.0f;
            conv8(a, sw1, nt1, y0 - r1, [&](int e) { return s1[min(max(e, 0), H - 1) * kStrip + lane]; });
            if (dog) {
                float b[kOut];
#pragma unroll
                for (int j = 0; j < kOut; ++j) b[j] = 0.0f;
                conv8(b, sw2, nt2, y0 - r2, [&](int e) { return s2[min(max(e, 0), H - 1) * kStrip + lane]; });
#pragma unroll
                for (int j = 0; j < kOut; ++j) a[j] = fmaxf(a[j] - b[j], 0.0f);
            }
#pragma unroll
            for (int j = 0; j < kOut; ++j)
                if (y0 + j < H) out[base + (size_t)(y0 + j) * W + x] = a[j];
        }
    }
}

// ---------------------------------------------------------------- one pass
constexpr int kB = 8;                                       // rows per step
constexpr int kStreamThreads = 256;

// acc[j] += sum_{u < 8} w[u] x[j + u], x the 16 elements lo, hi (w 16-byte aligned).
__device__ __forceinline__ void taps8(float (&acc)[8], const float (&lo)[8], const float (&hi)[8], const float* w) {
    const float4 w0 = *reinterpret_cast<const float4*>(w), w1 = *reinterpret_cast<const float4*>(w + 4);
    const float wt[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = fmaf(wt[u], j + u < 8 ? lo[j + u] : hi[j + u - 8], acc[j]);
}
// acc[j] = sum_t w[t] x[j + t], t < nt ascending, for eight outputs.  group(g, v) gives the elements
// x[8 g .. 8 g + 7]; at most groups 0 .. nt / 8 + 1 are asked for, in order.
template <typename G>
__device__ __forceinline__ void filter8(float (&acc)[8], const float* w, int nt, G group) {
    float a[8], b[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.0f;
    group(0, a);
    int g = 1;
#pragma unroll 1
    for (; 8 * g <= nt; ++g) {
        group(g, b);
        taps8(acc, a, b, w + 8 * g - 8);
#pragma unroll
        for (int j = 0; j < 8; ++j) a[j] = b[j];
    }
    const int rem = nt - 8 * g + 8;                         // 0 .. 7 taps left; uniform
    if (rem > 1) group(g, b);
#pragma unroll 1
    for (int u = 0; u < rem;) {
        const float wt = w[8 * g - 8 + u];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = fmaf(wt, a[j], acc[j]);
        if (++u == rem) break;
#pragma unroll
        for (int j = 0; j < 7; ++j) a[j] = a[j + 1];
        a[7] = b[0];
#pragma unroll
        for (int j = 0; j < 7; ++j) b[j] = b[j + 1];
    }
}

struct StreamShape {                                        // shared memory, in floats
    int dog, blur;                                          // which filters run
    int r1, r2, rb, R;                                      // radii; R: of the first stage
    int in_p, d_p;                                          // row pitches (odd): staged rows, difference
    int n1, n2, nb;                                         // rows of the rings (multiples of 8)
    int o_w1, o_w2, o_wb, o_in, o_1, o_2, o_d, o_b, total;
};

// Ring row pitches built: the smallest that holds a row (odd: no bank conflicts).
constexpr int kPitches[3] = {129, 257, 513};

// dog: filters 1 and 2 and their difference, then the blur when there is one; else the blur alone.
// A ring holds what its column filter reads, 2 r + 8 rows, and the rows the first stage is ahead.
bool stream_shape(int W, int r1, int r2, int rb, bool dog, bool blur, StreamShape* out, int* pitch) {
    StreamShape s;
    s.dog = dog;
    s.blur = blur;
    s.r1 = dog ? r1 : 0;
    s.r2 = dog ? r2 : 0;
    s.rb = blur ? rb : 0;
    s.R = std::max(s.r1, s.r2);
    const int halo = dog ? s.R : s.rb, segs = (W + 7) / 8 * 8;
    *pitch = 0;
    for (int q : kPitches)
        if (!*pitch && segs <= q) *pitch = q;
    if (!*pitch) return false;
    auto up8 = [](int x) { return (x + 7) & ~7; };
    s.in_p = (segs + 2 * halo + 8) | 1;
    s.d_p = (segs + 2 * s.rb + 8) | 1;
    // (a filter's last group may reach past its rows: round the ring, into rows it does not use)
    s.n1 = dog ? up8(s.R + s.r1 + kB) : 0;
    s.n2 = dog ? up8(s.R + s.r2 + kB) : 0;
    // (blur alone: a step's rows are written while the rows before are still read)
    s.nb = blur ? up8(2 * s.rb + kB) + (dog ? 0 : 2 * kB) : 0;
    int o = 0;
    auto take = [&](int floats) {
        const int at = o;
        o += (floats + 3) & ~3;
        return at;
    };
    s.o_w1 = take(dog ? 2 * s.r1 + 1 : 0);
    s.o_w2 = take(dog ? 2 * s.r2 + 1 : 0);
    s.o_wb = take(blur ? 2 * s.rb + 1 : 0);
    s.o_in = take(kB * s.in_p);
    s.o_1 = take(s.n1 * *pitch);
    s.o_2 = take(s.n2 * *pitch);
    s.o_d = take(dog && blur ? kB * s.d_p : 0);
    s.o_b = take(s.nb * *pitch);
    s.total = o;
    *out = s;
    return (size_t)s.total * 4 <= 200 * 1024;
}

__device__ __forceinline__ void unpack8(const uint4 (&v)[1], float (&f)[8]) {
    const uint32_t u[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
#pragma unroll
    for (int j = 0; j < 8; ++j) f[j] = (float)(j & 1 ? u[j >> 1] >> 16 : u[j >> 1] & 0xffffu);
}
__device__ __forceinline__ void unpack8(const uint4 (&v)[2], float (&f)[8]) {
    const uint32_t u[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
    for (int j = 0; j < 8; ++j) f[j] = __uint_as_float(u[j]);
}

template <typename T, int PITCH>
__global__ void __launch_bounds__(kStreamThreads, 2)
gauss_stream_kernel(const T* __restrict__ in, int64_t n, int H, int W, const float* __restrict__ w1,
                    const float* __restrict__ w2, const float* __restrict__ wb, const StreamShape s, int bands,
                    int band_rows, float* __restrict__ out) {
    extern __shared__ __align__(16) float sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int nwarps = kStreamThreads / 32, kVec = sizeof(T) / 2;   // 16-byte vectors per 8 pixels
    for (int i = threadIdx.x; i < 2 * s.r1 + 1 && s.dog; i += kStreamThreads) sm[s.o_w1 + i] = w1[i];
    for (int i = threadIdx.x; i < 2 * s.r2 + 1 && s.dog; i += kStreamThreads) sm[s.o_w2 + i] = w2[i];
    for (int i = threadIdx.x; i < 2 * s.rb + 1 && s.blur; i += kStreamThreads) sm[s.o_wb + i] = wb[i];
    float* s_in = sm + s.o_in;
    const int halo = s.dog ? s.R : s.rb;
    // row passes: a warp takes 8 rows x 4 runs of 8 columns
    const int row8 = lane & 7, sub = lane >> 3, segs = (W + 7) >> 3;
    const bool vec = W % 8 == 0 && ((uintptr_t)in & 15) == 0;
    // Rings: row y (counted from the band's first input row) lives at slot (y + off) mod rows, with off
    // such that every column filter starts at a multiple of 8 (a run of 8 rows never wraps).
    const int off1 = (s.R + s.r1) & 7, off2 = (s.R + s.r2) & 7, offb = (2 * s.rb) & 7;
    // slots of the step's column filters behind the step's first slot (all modulo the ring)
    auto behind = [](int back, int rows) { return rows ? ((-back) % rows + rows) % rows : 0; };
    const int back1 = behind(s.R + s.r1 - off1, s.n1), back2 = behind(s.R + s.r2 - off2, s.n2);
    auto wrap = [](int q, int rows) { return q >= rows ? q - rows : q; };

    for (int64_t item = blockIdx.x; item < n * bands; item += gridDim.x) {
        const int64_t p = item / bands;
        const int y0 = (int)(item - p * bands) * band_rows, y1 = min(H, y0 + band_rows);
        const T* src = in + (size_t)p * H * W;
        float* dst = out + (size_t)p * H * W;
        // rows of the first stage's result that the band needs, and the first input row
        const int d0 = max(0, y0 - s.rb), d1 = min(H, y1 + s.rb);
        const int yb0 = d0 - s.R;
        const int steps = (d1 - 1 + s.R - yb0) / kB + 1;
        int base1 = 0, base2 = 0;                           // the step's first slot of the rings

        // the thread's run of 8 pixels of the rows yb .. yb + 7, loaded a step ahead
        uint4 ahead[kVec];
        auto row_ptr = [&](int yb) { return src + (size_t)min(max(yb + row8, 0), H - 1) * W; };
        auto load = [&](int yb) {
            const int seg = 4 * warp + sub;
            if (vec && seg < segs) {
                const uint4* r = reinterpret_cast<const uint4*>(row_ptr(yb) + 8 * seg);
#pragma unroll
                for (int i = 0; i < kVec; ++i) ahead[i] = __ldg(r + i);
            }
        };
        auto stage = [&](int yb) {
            const T* r = row_ptr(yb);
            float* d = s_in + row8 * s.in_p + halo;
            for (int sg = warp; 4 * sg < segs; sg += nwarps) {
                const int seg = 4 * sg + sub;
                if (seg >= segs) continue;
                float f[8];
                if (vec) {
                    if (sg != warp) {
#pragma unroll
                        for (int i = 0; i < kVec; ++i) ahead[i] = __ldg(reinterpret_cast<const uint4*>(r + 8 * seg) + i);
                    }
                    unpack8(ahead, f);
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) f[j] = as_float(__ldg(r + min(8 * seg + j, W - 1)));
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) d[8 * seg + j] = f[j];   // (past the row: its edge pixel)
                // the edge pixels repeated outside the frame
                if (seg == 0)
                    for (int i = 1; i <= halo; ++i) d[-i] = f[0];
                if (seg == segs - 1) {
                    const float e = as_float(__ldg(r + W - 1));
                    for (int i = 8 * segs; i < W + halo; ++i) d[i] = e;
                }
            }
        };
        __syncthreads();                                    // the weights; the item before is done
        load(yb0);
        stage(yb0);
        __syncthreads();
#pragma unroll 1
        for (int st = 0; st < steps; ++st) {
            const int yb = yb0 + st * kB;                   // the newest rows: yb .. yb + 7
            if (st + 1 < steps) load(yb + kB);
            // ---- (0) row filters of the newest rows
            for (int sg = warp; 4 * sg < segs; sg += nwarps) {
                const int seg = 4 * sg + sub;
                if (seg < segs) {
                    const float* x = s_in + row8 * s.in_p + 8 * seg;
                    auto run = [&](const float* q) {
                        return [q](int g, float (&v)[8]) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[j] = q[8 * g + j];
                        };
                    };
                    auto store = [&](float* o, const float (&acc)[8]) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) o[j] = acc[j];
                    };
                    float acc[8];
                    if (s.dog) {
                        filter8(acc, sm + s.o_w1, 2 * s.r1 + 1, run(x + s.R - s.r1));
                        store(sm + s.o_1 + wrap(base1 + row8 + off1, s.n1) * PITCH + 8 * seg, acc);
                        filter8(acc, sm + s.o_w2, 2 * s.r2 + 1, run(x + s.R - s.r2));
                        store(sm + s.o_2 + wrap(base2 + row8 + off2, s.n2) * PITCH + 8 * seg, acc);
                    } else if (yb + row8 < d1) {
                        filter8(acc, sm + s.o_wb, 2 * s.rb + 1, run(x));
                        store(sm + s.o_b + ((yb + row8 - yb0 + s.R + offb) % s.nb) * PITCH + 8 * seg, acc);
                    }
                }
            }
            __syncthreads();
            // runs of 8 rows of column x of a ring from slot `at` (a multiple of 8) on
            auto column = [&](int o, int at, int rows, int x) {
                const float* base = sm + o + x;
                return [base, at, rows](int g, float (&v)[8]) {
                    int q = at + 8 * g;
                    if (q >= rows) q -= rows;
                    const float* c = base + q * PITCH;
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = c[j * PITCH];
                };
            };
            // ---- (1) column filters and their clipped difference, rows yd .. yd + 7
            const int yd = yb - s.R;                        // (dog: R rows behind; else the newest rows)
            if (s.dog && yd + kB > d0) {
                // (runs before the band's first row enter no row of [d0, d1))
                const int at1 = wrap(base1 + back1, s.n1), at2 = wrap(base2 + back2, s.n2);
                for (int x = threadIdx.x; x < W; x += kStreamThreads) {
                    float a[8], b[8];
                    filter8(a, sm + s.o_w1, 2 * s.r1 + 1, column(s.o_1, at1, s.n1, x));
                    filter8(b, sm + s.o_w2, 2 * s.r2 + 1, column(s.o_2, at2, s.n2, x));
#pragma unroll
                    for (int j = 0; j < 8; ++j) a[j] = fmaxf(a[j] - b[j], 0.0f);
                    if (!s.blur) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (yd + j >= y0 && yd + j < y1) dst[(size_t)(yd + j) * W + x] = a[j];
                    } else {
                        float* d = sm + s.o_d + s.rb + x;
#pragma unroll
                        for (int j = 0; j < 8; ++j) d[j * s.d_p] = a[j];
                        // the edge pixel repeated outside the frame
                        if (x == 0 || x == W - 1) {
                            const int step = x == 0 ? -1 : 1;
                            for (int i = 1; i <= s.rb; ++i) {
#pragma unroll
                                for (int j = 0; j < 8; ++j) d[j * s.d_p + i * step] = a[j];
                            }
                            if (W == 1)
                                for (int i = 1; i <= s.rb; ++i) {
#pragma unroll
                                    for (int j = 0; j < 8; ++j) d[j * s.d_p + i] = a[j];
                                }
                        }
                    }
                }
            }
            if (s.dog && s.blur && yd + kB > d0) {
                __syncthreads();
                // ---- (2) the blur's row filter
                for (int sg = warp; 4 * sg < segs; sg += nwarps) {
                    const int seg = 4 * sg + sub, y = yd + row8;
                    if (seg < segs && y >= d0 && y < d1) {
                        const float* x = sm + s.o_d + row8 * s.d_p + 8 * seg;
                        float acc[8];
                        filter8(acc, sm + s.o_wb, 2 * s.rb + 1, [x](int g, float (&v)[8]) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[j] = x[8 * g + j];
                        });
                        float* ob = sm + s.o_b + ((y - yb0 + s.R + offb) % s.nb) * PITCH + 8 * seg;
#pragma unroll
                        for (int j = 0; j < 8; ++j) ob[j] = acc[j];
                    }
                }
            }
            base1 = wrap(base1 + kB, s.n1);
            base2 = wrap(base2 + kB, s.n2);
            if (st + 1 < steps) stage(yb + kB);             // (the staged rows were read before a barrier)
            __syncthreads();
            // ---- (3) the blur's column filter: the rows whose reach is complete (all that are left in
            // the last step; a row past the frame's edge is its edge row)
            const int newest = min(yd + kB, d1) - 1;        // last row in the blur's ring
            const int lo = max(y0, yd - s.rb), hi = newest == d1 - 1 ? y1 : min(y1, newest + 1 - s.rb);
            if (s.blur && lo < hi) {
                // (in steps of 8 from yd - rb, so that the runs stay aligned)
                int yo0 = yd - s.rb;
                while (yo0 + kB <= lo) yo0 += kB;
#pragma unroll 1
                for (int yo = yo0; yo < hi; yo += kB) {
                    const bool inside = yo - s.rb >= d0 && yo + 7 + s.rb <= newest;
                    int at = (yo - s.rb - yb0 + s.R + offb) % s.nb;
                    if (at < 0) at += s.nb;
                    for (int x = threadIdx.x; x < W; x += kStreamThreads) {
                        float acc[8];
                        if (inside) {
                            filter8(acc, sm + s.o_wb, 2 * s.rb + 1, column(s.o_b, at, s.nb, x));
                        } else {
                            const float* base = sm + s.o_b + x;
                            filter8(acc, sm + s.o_wb, 2 * s.rb + 1, [&](int g, float (&v)[8]) {
#pragma unroll 1
                                for (int j = 0; j < 8; ++j) {
                                    const int y = min(max(yo - s.rb + 8 * g + j, d0), newest);
                                    const float e = base[((y - yb0 + s.R + offb) % s.nb) * PITCH];
#pragma unroll
                                    for (int i = 0; i < 8; ++i)
                                        if (i == j) v[i] = e;
                                }
                            });
                        }
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (yo + j >= lo && yo + j < hi) dst[(size_t)(yo + j) * W + x] = acc[j];
                    }
                }
            }
        }
    }
}

int grid_of(int64_t items, int per_block) {
    const int64_t g = (items + per_block - 1) / per_block;
    const int64_t cap = (int64_t)device_sms() * 16;
    return (int)(g < 1 ? 1 : (g < cap ? g : cap));
}

}  // namespace

size_t gauss_cols_smem(int H, int r1, int r2, int dog) {
    return ((size_t)padded_taps(r1) + (dog ? padded_taps(r2) : 0) + (size_t)H * kStrip * (dog ? 2 : 1)) * sizeof(float);
}

int gauss_padded_taps(int r) { return padded_taps(r); }

// Whether the whole of it takes one pass: where the frames' rolling rows fit shared memory and the frames
// are large enough.  A band repeats the filters' reach at its ends, and a narrow or short frame leaves
// warps of the row filters and bands idle.  One pass against the separate ones, us, u16:
//   sigma 1 / 4, blur 1 (reach 20): 100 x 100, 1 / 4096 frames 30 / 974 against 31 / 1281;
//     256 x 256 29 / 2780 against 51 / 5783; 512 x 64 24 / 3630 against 84 / 7557;
//     32 x 32 25 / 355 against 21 / 247; without blur, 1 frame, 100 x 100 20 against 19, 64 x 512 29
//     against 19.
//   sigma 2 / 10, blur 2 (reach 48): 256 x 256 54 / 5970 against 56 / 7280; 144 x 200 52 / 3659
//     against 41 / 3394.
//   a blur alone: sigma 1 (reach 4) 256 x 256 15 / 1130 against 21 / 1615, 100 x 100 15 / 471 against
//     14 / 407; sigma 3 (reach 12) 256 x 256, 16 frames 31 against 27, 300 x 500, 128 frames 225
//     against 156.
bool gauss_stream_supported(int H, int W, int r1, int r2, int rb, bool dog, bool blur) {
    StreamShape s;
    int pitch;
    if (!(dog || blur) || !stream_shape(W, r1, r2, rb, dog, blur, &s, &pitch)) return false;
    if (!dog) return rb <= 4 && H >= 144 && W >= 144;
    const int rows = std::max(blur ? 96 : 112, 5 * (s.R + s.rb));
    return H >= rows && W >= 64 && (int64_t)H * W >= (int64_t)rows * 96;
}

namespace {
template <typename T, int PITCH>
cudaError_t launch_stream(const T* in, int64_t n, int H, int W, const float* w1, const float* w2, const float* wb,
                          const StreamShape& s, float* out, int num_sms, cudaStream_t st) {
    const size_t smem = (size_t)s.total * sizeof(float);
    int per_sm = 1;
    const cudaError_t e = kernel_occupancy((const void*)gauss_stream_kernel<T, PITCH>, kStreamThreads, smem, &per_sm);
    if (e != cudaSuccess) return e;
    const int64_t slots = (int64_t)num_sms * std::max(1, per_sm);
    // one band a frame while the frames fill the GPU; else the number of bands (of at least 16 rows)
    // with the fewest row steps, counting the reach that each band repeats at its ends and the waves
    const int reach = 2 * (s.R + s.rb);
    int bands = 1;
    int64_t least = INT64_MAX;
    for (int b = 1; b <= std::max(1, H / 16) && (b == 1 || n < slots); ++b) {
        const int64_t cost = ((n * b + slots - 1) / slots) * ((H + b - 1) / b + kB - 1 + reach);
        if (cost < least) {
            least = cost;
            bands = b;
        }
    }
    const int band_rows = ((H + bands - 1) / bands + kB - 1) / kB * kB;
    bands = (H + band_rows - 1) / band_rows;
    const int grid = (int)std::min<int64_t>(n * bands, slots);
    gauss_stream_kernel<T, PITCH><<<grid, kStreamThreads, smem, st>>>(in, n, H, W, w1, w2, wb, s, bands, band_rows, out);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_gauss_stream(const void* in, int dtype, int64_t n, int H, int W, const float* w1, int r1,
                                const float* w2, int r2, const float* wb, int rb, bool dog, bool blur, float* out,
                                int num_sms, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    StreamShape s;
    int pitch;
    if (!stream_shape(W, r1, r2, rb, dog, blur, &s, &pitch)) return cudaErrorInvalidValue;
    auto run = [&](auto* f) {
        return pitch == kPitches[0]   ? launch_stream<std::decay_t<decltype(*f)>, kPitches[0]>(f, n, H, W, w1, w2, wb, s, out, num_sms, st)
               : pitch == kPitches[1] ? launch_stream<std::decay_t<decltype(*f)>, kPitches[1]>(f, n, H, W, w1, w2, wb, s, out, num_sms, st)
                                      : launch_stream<std::decay_t<decltype(*f)>, kPitches[2]>(f, n, H, W, w1, w2, wb, s, out, num_sms, st);
    };
    return dtype == TM_DTYPE_U16 ? run((const uint16_t*)in) : run((const float*)in);
}

cudaError_t launch_gauss_rows(const void* in, int dtype, int64_t rows, int W, const float* w1, int r1, const float* w2,
                              int r2, float* out1, float* out2, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    const int R = w2 ? (r1 > r2 ? r1 : r2) : r1;
    const int span = 32 * kOut, ne = ((W + span - 1) / span) * span + 2 * R + kOut + kTap;
    const size_t smem = ((size_t)padded_taps(r1) + (w2 ? padded_taps(r2) : 0) + (size_t)kRowWarps * (ne + (ne >> 3))) *
                        sizeof(float);
    const int grid = grid_of(rows, kRowWarps);
    cudaError_t e;
    if (dtype == TM_DTYPE_U16) {
        e = kernel_occupancy((const void*)gauss_rows_kernel<uint16_t>, 32 * kRowWarps, smem, nullptr);
        if (e != cudaSuccess) return e;
        gauss_rows_kernel<uint16_t><<<grid, 32 * kRowWarps, smem, st>>>((const uint16_t*)in, rows, W, w1, r1, w2, r2,
                                                                        out1, out2);
    } else {
        e = kernel_occupancy((const void*)gauss_rows_kernel<float>, 32 * kRowWarps, smem, nullptr);
        if (e != cudaSuccess) return e;
        gauss_rows_kernel<float><<<grid, 32 * kRowWarps, smem, st>>>((const float*)in, rows, W, w1, r1, w2, r2, out1,
                                                                     out2);
    }
    return cudaGetLastError();
}

cudaError_t launch_gauss_cols(const float* in1, const float* in2, int64_t n, int H, int W, const float* w1, int r1,
                              const float* w2, int r2, int dog, float* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const size_t smem = gauss_cols_smem(H, r1, r2, dog);
    const cudaError_t e = kernel_occupancy((const void*)gauss_cols_kernel, 256, smem, nullptr);
    if (e != cudaSuccess) return e;
    const int64_t strips = (int64_t)n * ((W + kStrip - 1) / kStrip);
    gauss_cols_kernel<<<grid_of(strips, 1), 256, smem, st>>>(in1, in2, n, H, W, w1, r1, w2, r2, dog, out);
    return cudaGetLastError();
}

}  // namespace tmgb
