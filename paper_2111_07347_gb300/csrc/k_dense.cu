// BF16 tensor-core pre-score, stage B: the inverse angular DFT on tcgen05 with the maximum
// over shifts fused into the epilogue.
//
// The correlation of Eq. 1 along the azimuth is evaluated through the correlation theorem
// (the FFT cross-correlation alternative the paper names in Section 2.2's complexity
// paragraph):
//   C[k, s] = sum_{m=0}^{H} (w_m / n) Re( G[k, m] e^{2 pi i m s / n} ),  H = n / 2,
//   G[k, m] = sum_r conj(T^_k[r, m]) P^[r, m],
// with T^ and P^ the angular DFTs of the template (divided by |T_k|) and of the polar pattern
// (divided by |P|), so C is Q directly.  Stage A (G, a GEMM per frequency over the radii) runs
// before this kernel and leaves G in global memory as BF16, frequency-major:
//   G[j][p][c][k]  (slot j, pattern p of the batch, c = 0 real / 1 imaginary, template k),
// slot j < 96 holding m = 2 j and slot j >= 96 holding m = 2 (j - 96) + 1.  Slots with m > H add
// nothing: their rows of the basis are zero, and where the even and odd slots have a tensor map each
// they lie outside it and are not read (zero fill); small batches compute and read all slots through
// one map, their spectra being zero.  Two radix-2 splits quarter
// the work of the full sum.  With E[s] the even-m part and O[s] the odd-m part of the sum, C[s] = E[s] + O[s]
// and C[s + H] = E[s] - O[s], so max(C[s], C[s + H]) = E[s] + |O[s]| for s < H.  And with the cosine (real)
// and sine (imaginary) parts of each, E = Ec + Es, O = Oc + Os, their symmetry about H / 2 gives
//   E[H - s] = Ec[s] - Es[s],  |O[H - s]| = |Os[s] - Oc[s]|,
// so s <= H / 2 is enough: per (pattern, tile of 128 templates) four products [128 x 96] x [96 x 96]
// give Ec, Es, Oc, Os.
//
// Operands: A = G read by TMA as MN-major tiles (template index contiguous; per ring slot one of the
// four parts, 96 K-rows of 2 x 64 templates, 24 KB, 128-byte swizzle); B = the inverse-DFT basis
// (w_m / n) cos / -sin, K-major, resident in shared memory (72 KB).  CTA (persistent over
// (pattern, tile) units, 640 threads):
//   warp 0 lane 0  TMA producer into a 6-slot ring (one and a half units);
//   warp 1 lane 0  MMA issuer (tcgen05.mma.cta_group::1.kind::f16, BF16 x BF16 -> FP32 in TMEM);
//   warp 2         TMEM allocation;
//   warps 4-19     epilogue: four warps per TMEM lane quadrant (32 templates), each a quarter of the
//                  shift columns of the four parts (tcgen05.ld) and their maximum; the quarters are
//                  combined in shared memory and one pre-score per (pattern, template) is written to
//                  global memory (masked-out templates: -NaN).
// The parts go round five TMEM blocks, so a unit's first part is multiplied beside the epilogue of
// the unit before.
// 512 patterns against the 13986-template HCP library: 1.13 ms (with the even / odd split alone and
// twice the MMA work 1.18 ms), 4.9 TB/s of G, 72 % of the copy rate.  The loads alone take 1.13
// ms and everything else alone 1.00 ms.  The arrivals that free the accumulator are one per warp.
// Every mbarrier wait is bounded by the global timer (1 s); on timeout the CTA records an error
// in a device word, stops its roles, lets the copies and MMAs it issued finish, releases TMEM
// and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <float.h>
#include <math.h>

#include "tm_internal.h"
#include "tm_tcgen05.h"

namespace tmgb {
namespace {

constexpr int kRows = 128;                 // templates per tile (MMA M)
constexpr int kN = 96;                     // shifts of a part (MMA N), >= n_theta / 4 + 1
constexpr int kK = 96;                     // slots of a part (contraction), >= n_theta / 4 + 1
constexpr int kParts = 4;                  // Ec, Es, Oc, Os
constexpr int kBlocks = 5;                 // TMEM blocks of kN columns the units' parts go round
constexpr int kBoxBytes = 64 * kK * 2;     // 12 KB: 64 templates x 96 slots
constexpr int kSlotBytes = 2 * kBoxBytes;  // 24 KB
constexpr int kStages = 6;
constexpr int kBasisChunks = 3;            // of 64 K elements: 96 cosines and 96 sines of an even or odd part
constexpr int kBasisChunkBytes = kN * 128; // 12 KB
constexpr int kEpiWarp0 = 4;
constexpr int kEpiWarps = 16;              // four per TMEM lane quadrant, each a quarter of the shift columns
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kThreads = (kEpiWarp0 + kEpiWarps) * 32;

// Instruction descriptor: kind::f16, A = B = BF16, D = F32, A MN-major (bit 15), B K-major.
__host__ __device__ constexpr uint32_t idesc_bf16_amn(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

// 8 columns of each of the four parts (at the TMEM addresses t) of the warp's 32 lanes into
// registers, and the wait for them.
__device__ __forceinline__ void tmem_ld4x8(const uint32_t (&t)[kParts], uint32_t col, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%33];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%34];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%35];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        :
          "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
          "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
          "=r"(r[30]), "=r"(r[31])
        : "r"(t[0] + col), "r"(t[1] + col), "r"(t[2] + col), "r"(t[3] + col)
        : "memory");
}

// A CTA's (pattern, tile) units blockIdx.x, blockIdx.x + gridDim.x, ..., counted on without divisions.
struct Unit {
    int p, t, dp, dt, tiles;
    __device__ __forceinline__ explicit Unit(int n_tiles) : tiles(n_tiles) {
        p = blockIdx.x / tiles;
        t = blockIdx.x - p * tiles;
        dp = gridDim.x / tiles;
        dt = gridDim.x - dp * tiles;
    }
    __device__ __forceinline__ void next() {
        p += dp;
        t += dt;
        if (t >= tiles) {
            t -= tiles;
            ++p;
        }
    }
};

__global__ void __launch_bounds__(kThreads, 1) dense_kernel(const __grid_constant__ CUtensorMap emap,
                                                                   const __grid_constant__ CUtensorMap omap,
                                                                   const DenseCall c) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* s_basis = base;                                   // 2 x kBasisChunks x [kN rows x 128 B]
    uint8_t* s_ring = s_basis + 2 * kBasisChunks * kBasisChunkBytes;   // kStages x 24 KB
    uint64_t* bar = (uint64_t*)(s_ring + kStages * kSlotBytes);  // full[S], empty[S], acc_full, acc_empty
    uint32_t* s_tmem = (uint32_t*)(bar + 2 * kStages + 2);
    int* s_abort = (int*)(s_tmem + 1);
    int* s_epi_stop = s_abort + 1;                             // [2], by unit parity
    float* s_part = (float*)(s_epi_stop + 2);                  // [4 quarters][kRows] partial maxima
    volatile int* abort_flag = s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int H = c.n_theta / 2;
    const int tiles = (c.K + kRows - 1) / kRows;
    const uint32_t bar_full0 = smem_u32(&bar[0]), bar_empty0 = smem_u32(&bar[kStages]);
    const uint32_t bar_accf = smem_u32(&bar[2 * kStages]), bar_acce = smem_u32(&bar[2 * kStages + 1]);

    // ---- one-time setup: the basis, swizzled (16-byte chunk q of row r at (q ^ (r & 7)))
    for (int i = threadIdx.x; i < 2 * kBasisChunks * kN * 8; i += blockDim.x) {
        const int ch = i / (kN * 8), rem = i - ch * kN * 8, n = rem >> 3, q = rem & 7;
        const int part = ch / kBasisChunks, c3 = ch - part * kBasisChunks;
        const uint4 v = *(const uint4*)((const __nv_bfloat16*)c.basis + ((size_t)part * kN + n) * 2 * kK + c3 * 64 + q * 8);
        *(uint4*)(s_basis + ch * kBasisChunkBytes + n * 128 + ((q ^ (n & 7)) << 4)) = v;
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(smem_u32(&bar[i]), 1);
            mbar_init(smem_u32(&bar[kStages + i]), 1);
        }
        mbar_init(bar_accf, 1);
        mbar_init(bar_acce, kEpiWarps);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&emap) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&omap) : "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_proxy_async();           // basis stores -> visible to the tensor-core (async) proxy
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;

    if (warp == 0) {
        // ================================================================ TMA producer
        if (lane == 0) {
            uint32_t g = 0;
            bool stop = false;
            for (Unit w(tiles); w.p < c.n && !stop; w.next()) {
                const int p = w.p, t = w.t;
                for (int ch = 0; ch < kParts; ++ch, ++g) {
                    const uint32_t slot = g % kStages, use = g / kStages;
                    if (!mbar_wait(bar_empty0 + 8 * slot, (use & 1u) ^ 1u, abort_flag)) {
                        *abort_flag = 1;
                        stop = true;
                        break;
                    }
                    const uint32_t full = bar_full0 + 8 * slot;
                    const uint32_t box = (uint32_t)c.box_rows * 128;
                    mbar_expect_tx(full, 2 * box);
                    const uint32_t dst = smem_u32(s_ring + slot * kSlotBytes);
                    const CUtensorMap* map = ch < 2 ? &emap : &omap;
                    const int j0 = ch < 2 ? 0 : c.odd_slot;
                    tma_load_4d(dst, map, t * kRows, ch & 1, p, j0, full);
                    tma_load_4d(dst + kBoxBytes, map, t * kRows + 64, ch & 1, p, j0, full);
                }
            }
            // the copies issued last must land before the CTA exits (they complete on their own)
            volatile int never = 0;
            const uint32_t n_issued = g;
            for (uint32_t i = 0; i < kStages && i < n_issued; ++i) {
                const uint32_t gg = n_issued - 1 - i, slot = gg % kStages, use = gg / kStages;
                mbar_wait(bar_full0 + 8 * slot, use & 1u, &never);
            }
        }
    } else if (warp == 1) {
        // ================================================================ MMA issuer
        if (lane == 0 && !c.stall) {
            const uint32_t idesc = idesc_bf16_amn(kRows, kN);
            const uint64_t a_desc = sdesc_mnmajor(smem_u32(s_ring), kBoxBytes), b_desc = sdesc_kmajor(smem_u32(s_basis));
            uint32_t g = 0, tt = 0;
            bool stop = false, issued = false;
            uint32_t last_bar = 0, last_par = 0;
            for (Unit w(tiles); w.p < c.n && !stop; w.next(), ++tt) {
                // kept rolled: fully unrolled by nvcc 13.0 it gave wrong sums, and reading the phases, the
                // blocks' rotation and the descriptors shows no reason (test_gpu_tensor.py compares every
                // pre-score with the oracle's)
#pragma unroll 1
                for (int ch = 0; ch < kParts; ++ch, ++g) {
                    const uint32_t slot = g % kStages, use = g / kStages;
                    if (!mbar_wait(bar_full0 + 8 * slot, use & 1u, abort_flag)) {
                        *abort_flag = 1;
                        stop = true;
                        break;
                    }
                    // the first part goes to the block that the unit before does not use
                    if (ch == 1 && !mbar_wait(bar_acce, (tt & 1u) ^ 1u, abort_flag)) {
                        *abort_flag = 1;
                        stop = true;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + (kParts * tt + ch) % kBlocks * kN;
                    // K step ks of the part: 2 KB on in A; in the basis (cosines, then sines) step
                    // 6 (ch & 1) + ks, four of 32 bytes to a chunk
                    const uint64_t da = a_desc + (uint64_t)(slot * (kSlotBytes >> 4));
                    const uint64_t db = b_desc + (uint64_t)((ch >> 1) * kBasisChunks * (kBasisChunkBytes >> 4));
                    const int ks_n = c.box_rows / 16;
#pragma unroll
                    for (int ks = 0; ks < kK / 16; ++ks) {
                        const int kb = 6 * (ch & 1) + ks;
                        if (ks < ks_n)
                            mma_f16(d, da + ks * (2048 >> 4), db + (kb >> 2) * (kBasisChunkBytes >> 4) + (kb & 3) * 2, idesc,
                                    ks == 0 ? 0u : 1u);
                    }
                    mma_commit(bar_empty0 + 8 * slot);
                    last_bar = bar_empty0 + 8 * slot;
                    last_par = use & 1u;
                    issued = true;
                }
                if (stop) break;
                mma_commit(bar_accf);
            }
            if (stop && issued) {
                // let the MMAs already issued finish before TMEM is released
                volatile int never = 0;
                mbar_wait(last_bar, last_par, &never);
            }
        }
    } else if (warp >= kEpiWarp0) {
        // ================================================================ epilogue (warps 4-19)
        const int ew = warp - kEpiWarp0;
        const int quad = warp & 3, quarter = ew >> 2;         // TMEM lanes 32 quad.., shift columns by quarter
        const int row = quad * 32 + lane;
        const int et = ew * 32 + lane;                         // epilogue thread index
        const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16);
        const int s_max = H / 2;                               // shifts 0 .. H / 2 and their mirrors
        constexpr int kCols = kN / 4;
        uint32_t tt = 0;
        for (Unit w(tiles); w.p < c.n; w.next(), ++tt) {
            const int p = w.p, t = w.t;
            // one thread waits and publishes one decision (a word per unit parity, so the next
            // unit's write cannot overtake a slow reader of this one)
            if (et == 0) {
                const bool ok = mbar_wait(bar_accf, tt & 1u, abort_flag);
                if (!ok) *abort_flag = 1;
                s_epi_stop[tt & 1u] = (!ok || *abort_flag) ? 1 : 0;
            }
            named_bar(1, kEpiThreads);
            if (*(volatile int*)&s_epi_stop[tt & 1u]) break;
            tc_fence_after();
            uint32_t tp[kParts];
#pragma unroll
            for (int ch = 0; ch < kParts; ++ch) tp[ch] = tbase + (kParts * tt + ch) % kBlocks * kN + quarter * kCols;
            float m[4] = {-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
#pragma unroll
            for (int b = 0; b < kCols / 8; ++b) {
                // (the basis repeats its last shift past s_max; blocks that hold nothing else are left out)
                const bool in = quarter * kCols + 8 * b <= s_max;
                uint32_t r[32];                                // Ec, Es, Oc, Os
                if (in) tmem_ld4x8(tp, 8 * b, r);
                if (b == kCols / 8 - 1) {                      // the accumulator is in registers
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_acce);
                }
                if (in) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float ec = __uint_as_float(r[j]), es = __uint_as_float(r[8 + j]);
                        const float oc = __uint_as_float(r[16 + j]), os = __uint_as_float(r[24 + j]);
                        m[j & 3] = fmaxf(m[j & 3], fmaxf((ec + es) + fabsf(oc + os), (ec - es) + fabsf(os - oc)));
                    }
                }
            }
            float best = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
            s_part[quarter * kRows + row] = best;
            named_bar(2 + quad, 128);
            const int k = t * kRows + row;
            if (quarter == 0 && k < c.K) {
                best = fmaxf(fmaxf(best, s_part[kRows + row]), fmaxf(s_part[2 * kRows + row], s_part[3 * kRows + row]));
                const int64_t p_glob = c.p0 + p;
                bool keep = true;
                if (c.mask) keep = (c.mask[p_glob * c.words + (k >> 5)] >> (k & 31)) & 1u;
                c.pre[p_glob * c.K + k] = keep ? best : __int_as_float(0xFFFFFFFF);
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*abort_flag && threadIdx.x == 0) atomicOr(c.error, 1u);
    if (warp == 2) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

}  // namespace

size_t dense_smem_bytes() {
    return 1024 + (size_t)2 * kBasisChunks * kBasisChunkBytes + (size_t)kStages * kSlotBytes + (2 * kStages + 2) * 8 + 16 +
           4 * kRows * 4;
}

bool dense_supported(int n_theta) { return n_theta % 2 == 0 && n_theta >= 4 && (n_theta / 2) / 2 + 1 <= kN; }

int dense_basis_rows() { return 2 * kN; }
int dense_basis_cols() { return 2 * kK; }
int dense_slots() { return 2 * kK; }

cudaError_t launch_dense(const void* emap, const void* omap, const DenseCall& c, int num_sms, cudaStream_t st) {
    if (c.n <= 0 || c.K <= 0) return cudaSuccess;
    const size_t smem = dense_smem_bytes();
    const cudaError_t e = kernel_occupancy((const void*)dense_kernel, kThreads, smem, nullptr);
    if (e != cudaSuccess) return e;
    const int64_t units = c.n * (int64_t)((c.K + kRows - 1) / kRows);
    int64_t grid = num_sms;
    if (grid > units) grid = units;
    dense_kernel<<<(int)grid, kThreads, smem, st>>>(*(const CUtensorMap*)emap, *(const CUtensorMap*)omap, c);
    return cudaGetLastError();
}

}  // namespace tmgb
