// Upper bounds of Eq. 1's correlation index for every template, on the tensor cores (arXiv
// 2111.07347, Section 2.2: only the best N templates of a pattern are kept, so templates that
// provably cannot be among them need no exact score).
//
// With intensities I >= 0 the numerator of Eq. 1 at shift s is sum_i I_i P'[r_i, t_i + s].  The
// azimuth is cut into P pieces; nch = P / (pieces per chunk) chunks of columns and nw windows of
// shifts are runs of pieces.  A spot at (row a, column t in chunk j) visits, over the shifts of
// window h, only columns of a run of pieces that depends on (j, h) alone, so
//     max over the shifts of window h of C(s)  <=  sum_i I_i W[a_i, j_i; h],
// W[a, j; h] the maximum of row a over that run.  For a library of n_rad rows this is a contraction
// over kd = n_rad nch + 1 entries (a, j): the templates' rows B[k, (a, j)] -- the sum of their
// intensities there, divided by |T_k| -- are made once per library, each pattern gives nw columns
// W[(a, j); h] / |P|, and U[k, p] = max_h (B W)[k, (p, h)].
//
// Why U is a bound of Q as the exact kernels compute it: W is FP16 rounded up and I >= 0.  B is FP16
// rounded to nearest, which changes an entry by at most 2^-11 of itself or, below 2^-14 (subnormal),
// by 2^-25, so the sum by at most (2^-11 sum|I| / |T| + 2^-25 entries) max|P'| / |P|; the products
// are exact in FP32 and their sum is off by less than 512 * 2^-22 of sum|I| / |T| max|P'| / |P|; the
// exact sum by at most (2 spots + 40) 2^-24 of that.  The last entry of the contraction adds all of it
// (factors rounded up); the result is raised by 2^-18 of itself for the rounding of Q's division, and
// rounded up to FP16.  So a template with U below the N-th best Q found so far can be left out
// without changing the result.
//
// window_kernel: one CTA per pattern; piece maxima of the library's rows, then the W columns.
// bound_templates_kernel: B, one warp per template (once per library).
// bound_kernel: the contraction (32768 patterns against the 13986-template HCP library, six windows:
//   2.3 ms; 2.55 ms before the issuing threads were freed of divisions and descriptor arithmetic; its
//   loads alone, its MMAs alone and its epilogue alone take within a fifth of each other).
//   D[128 templates x 240 columns] per unit = 240 / nw patterns; a persistent CTA keeps its 128
//   templates' B (kd <= 512: at most 128 KB) in shared memory and streams W through a ring, in plain
//   loads of its own.  Two accumulators in TMEM (columns 0 and 256), so the epilogue of one
//   unit runs beside the MMAs of the next.  Units are ordered in blocks of kSuper column tiles
//   (W of one block: 15 MB, kept in L2 while every template tile passes over it).  Warps: 0 TMA
//   producer, 1 MMA issuer, 2 TMEM allocation, 4-11 epilogue (TMEM lane quadrant x column half):
//   maximum over the windows, U [p][K] as order-preserving 16-bit keys of FP16, and the maximum of
//   each 32-template word [p][words].
#include <cuda.h>
#include <cuda_fp16.h>
#include <float.h>

#include <algorithm>
#include <numeric>

#include "tm_internal.h"
#include "tm_tcgen05.h"

namespace tmgb {
namespace {

constexpr int kM = 128;                    // templates per unit (MMA M)
constexpr int kN = 240;                    // columns (pattern, window) per unit (MMA N)
constexpr int kHalf = kN / 2;              // columns per epilogue warp
constexpr int kChunkK = 64;                // contraction entries per ring slot (one swizzle row)
constexpr int kAChunk = kM * kChunkK * 2;  // 16 KB
constexpr int kBChunk = kN * kChunkK * 2;  // 30 KB
constexpr int kMaxStages = 5;
constexpr int kAccStride = 256;            // TMEM columns between the two accumulators
constexpr int kSuper = 64;                 // column tiles per block of units
constexpr int kEpi0 = 4, kEpiThreads = 256;
constexpr int kBoundThreads = kEpi0 * 32 + kEpiThreads;
constexpr float kRaise = 3.814697265625e-6f;   // 2^-18
constexpr float kMarginScale = 1024.0f;    // keeps the margin's two factors in FP16's normal range

// kind::f16, A = B = FP16, D = F32, both K-major.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// 120 consecutive TMEM columns of the warp's 32 lanes into registers, and the wait for them.
__device__ __forceinline__ void tmem_ld120(uint32_t t, uint32_t (&r)[120]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {"
        "%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,"
        "%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,"
        "%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%120];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
        "%64,%65,%66,%67,%68,%69,%70,%71,%72,%73,%74,%75,%76,%77,%78,%79,"
        "%80,%81,%82,%83,%84,%85,%86,%87,%88,%89,%90,%91,%92,%93,%94,%95}, [%121];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {"
        "%96,%97,%98,%99,%100,%101,%102,%103,%104,%105,%106,%107,%108,%109,%110,%111}, [%122];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {"
        "%112,%113,%114,%115,%116,%117,%118,%119}, [%123];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        :
          "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
          "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
          "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]),
          "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]),
          "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]),
          "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]),
          "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]), "=r"(r[64]),
          "=r"(r[65]), "=r"(r[66]), "=r"(r[67]), "=r"(r[68]), "=r"(r[69]), "=r"(r[70]), "=r"(r[71]),
          "=r"(r[72]), "=r"(r[73]), "=r"(r[74]), "=r"(r[75]), "=r"(r[76]), "=r"(r[77]), "=r"(r[78]),
          "=r"(r[79]), "=r"(r[80]), "=r"(r[81]), "=r"(r[82]), "=r"(r[83]), "=r"(r[84]), "=r"(r[85]),
          "=r"(r[86]), "=r"(r[87]), "=r"(r[88]), "=r"(r[89]), "=r"(r[90]), "=r"(r[91]), "=r"(r[92]),
          "=r"(r[93]), "=r"(r[94]), "=r"(r[95]), "=r"(r[96]), "=r"(r[97]), "=r"(r[98]), "=r"(r[99]),
          "=r"(r[100]), "=r"(r[101]), "=r"(r[102]), "=r"(r[103]), "=r"(r[104]), "=r"(r[105]), "=r"(r[106]),
          "=r"(r[107]), "=r"(r[108]), "=r"(r[109]), "=r"(r[110]), "=r"(r[111]), "=r"(r[112]), "=r"(r[113]),
          "=r"(r[114]), "=r"(r[115]), "=r"(r[116]), "=r"(r[117]), "=r"(r[118]), "=r"(r[119])
        : "r"(t), "r"(t + 64), "r"(t + 96), "r"(t + 112)
        : "memory");
}

// FP16 bits as an integer of the same order.
__device__ __forceinline__ uint32_t bound_key(__half h) {
    const uint32_t b = __half_as_ushort(h);
    return b & 0x8000u ? ~b & 0xffffu : b | 0x8000u;
}

// First column of piece i of P.
__host__ __device__ inline int piece_start(int i, int P, int n_theta) { return (int)((int64_t)i * n_theta / P); }

// Windows of one pattern: W[(p nw + h)][(a, j)] FP16, rows `pitch` halves apart.
__global__ void __launch_bounds__(256)
window_kernel(const float* __restrict__ polar, const float* __restrict__ pnorm, int64_t n, int n_r, int n_theta,
              const int32_t* __restrict__ radii, int n_rad, BoundShape s, __half* __restrict__ w,
              int* __restrict__ counter) {
    extern __shared__ float pm[];                          // [n_rad][P] piece maxima
    __shared__ float s_abs[8];
    const int P = s.pieces, cl = P / s.nch, wl = P / s.nw;
    // pieces a (chunk, window) pair covers: columns t + s with t in pieces [a, a + cl) and s in pieces
    // [b, b + wl) lie in pieces [a + b, a + b + cl + wl); with uneven pieces (starts floor(i Nθ / P))
    // the lowest may be the last column of the piece before
    const int before = n_theta % P ? 1 : 0, run = cl + wl + before;
    if (blockIdx.x == 0 && threadIdx.x == 0 && counter) *counter = 0;
    for (int64_t p = blockIdx.x; p < n; p += gridDim.x) {
        const float* img = polar + (size_t)p * n_r * n_theta;
        const float pn = __ldg(pnorm + p);
        float ma = 0.0f;
        for (int it = threadIdx.x; it < n_rad * P; it += blockDim.x) {
            const int a = it / P, i = it - a * P;
            const float* row = img + (size_t)__ldg(radii + a) * n_theta;
            float m = -INFINITY;
            const int c1 = piece_start(i + 1, P, n_theta);
            for (int c = piece_start(i, P, n_theta); c < c1; ++c) {
                const float v = __ldg(row + c);
                m = fmaxf(m, v);
                ma = fmaxf(ma, fabsf(v));
            }
            pm[it] = m;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
        if ((threadIdx.x & 31) == 0) s_abs[threadIdx.x >> 5] = ma;
        __syncthreads();
        // (a norm that is zero or NaN: every Q is 0, and so is every bound; an infinite norm: every finite
        // correlation gives 0 and an infinite one a Q that is not a number, which ranks below them)
        const bool usable = pn > 0.0f && pn <= FLT_MAX;
        const float inv = usable ? __fdiv_ru(1.0f, pn) : 0.0f, inv_dn = usable ? __fdiv_rd(1.0f, pn) : 0.0f;
        float mabs = 0.0f;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) mabs = fmaxf(mabs, s_abs[i]);
        const int kd1 = n_rad * s.nch;                      // the margin's entry
        const int pairs = s.pitch / 2;
        for (int it = threadIdx.x; it < pairs * s.nw; it += blockDim.x) {
            const int h = it / pairs, e0 = 2 * (it - h * pairs);
            __half v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int e = e0 + u;
                float x = 0.0f;
                if (e < kd1 && usable) {
                    x = -INFINITY;
                    const int a = e / s.nch, j = e - a * s.nch;
                    int q = j * cl + h * wl - before;
                    if (q < 0) q += P;
                    if (q >= P) q -= P;
                    for (int i = 0; i < run; ++i) {
                        x = fmaxf(x, pm[a * P + q]);
                        if (++q == P) q = 0;
                    }
                    x = __fmul_ru(x, x > 0.0f ? inv : inv_dn);
                } else if (e == kd1 && usable) {
                    x = __fmul_ru(__fmul_ru(mabs, inv), 1.0f / kMarginScale);
                }
                v[u] = __float2half_ru(x);
            }
            *reinterpret_cast<__half2*>(w + ((size_t)p * s.nw + h) * s.pitch + e0) = __halves2half2(v[0], v[1]);
        }
        __syncthreads();
    }
}

// B[k][(a, j)] FP16: one warp per template, its row summed in shared memory.
__global__ void __launch_bounds__(128)
bound_templates_kernel(const int4* __restrict__ meta, const int4* __restrict__ order, const int2* __restrict__ spot,
                       int K, int n_theta, int n_rad, BoundShape s, __half* __restrict__ out) {
    extern __shared__ float rows[];                        // [4][pitch]
    const int lane = threadIdx.x & 31;
    float* row = rows + (threadIdx.x >> 5) * s.pitch;
    const int k = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (k >= K) return;
    for (int i = lane; i < s.pitch; i += 32) row[i] = 0.0f;
    __syncwarp();
    const int4 m = __ldg(meta + __ldg(&order[k].w));
    const int cnt = m.y & 0xffff;
    const float tn = __int_as_float(m.z);
    if (lane == 0 && tn > 0.0f) {
        for (int i = 0; i < cnt; ++i) {
            const int2 sp = __ldg(spot + m.x + i);
            const int t = sp.x & 0x7ff, a = (sp.x >> 11) & 0x1fff;
            int j = (int)((int64_t)t * s.nch / n_theta);   // the chunk that holds column t
            const int cl = s.pieces / s.nch;
            while (j + 1 < s.nch && t >= piece_start((j + 1) * cl, s.pieces, n_theta)) ++j;
            while (j > 0 && t < piece_start(j * cl, s.pieces, n_theta)) --j;
            float* e = row + a * s.nch + j;
            *e += __fdiv_rn(__int_as_float(sp.y), tn);
        }
        // the margins' factor: ((2 spots + 40) 2^-24 + 2^-11 + 2^-13) sum|I| / |T| (2^-22 more for the
        // FP32 sums of B), and 2^-25 for every entry that holds a spot
        const float rel = (2.0f * (float)cnt + 40.0f) * 5.9604645e-8f + 6.1059e-4f;
        const float tiny = (float)min(cnt, n_rad * s.nch) * 2.9802322e-8f;
        row[n_rad * s.nch] =
            __fmul_ru(kMarginScale, __fadd_ru(__fdiv_ru(__fmul_ru(rel, __int_as_float(m.w)), tn), tiny));
    }
    __syncwarp();
    for (int i = lane; i < s.pitch; i += 32) out[(size_t)k * s.pitch + i] = i == n_rad * s.nch ? __float2half_ru(row[i]) : __float2half_rn(row[i]);
}

struct Units {                                             // the order of a CTA's units
    int mt, nt;                                            // template tiles, column tiles
    int cta, ctas;                                         // this CTA of how many
    __device__ __forceinline__ int super(int s) const { return min(kSuper, nt - s * kSuper); }
};

// Calls f(template tile, column tile, first unit of the tile, last unit of it) for the CTA's units;
// stops when f returns false.
template <typename F>
__device__ __forceinline__ void for_units(const Units& g, F f) {
    const int supers = (g.nt + kSuper - 1) / kSuper;
    int prev = -1;
    for (int s = 0; s < supers; ++s) {
        const int sb = g.super(s);
        const int64_t total = (int64_t)g.mt * sb;
        const int64_t lo = total * g.cta / g.ctas, hi = total * (g.cta + 1) / g.ctas;
        // whether the units of the next block (if the CTA has any) go on with the same template tile
        int next_mt = -1;
        for (int s2 = s + 1; s2 < supers && next_mt < 0; ++s2) {
            const int sb2 = g.super(s2);
            const int64_t t2 = (int64_t)g.mt * sb2;
            const int64_t l2 = t2 * g.cta / g.ctas, h2 = t2 * (g.cta + 1) / g.ctas;
            if (l2 < h2) next_mt = (int)(l2 / sb2);
        }
        // (counted on, not divided: a 64-bit division a unit in every role had been a quarter of the time)
        const int count = (int)(hi - lo);
        int m = (int)(lo / sb), c = (int)(lo - (int64_t)m * sb);
        for (int i = 0; i < count; ++i) {
            const bool row_ends = c + 1 == sb;
            const int after = i + 1 < count ? (row_ends ? m + 1 : m) : next_mt;
            if (!f(m, s * kSuper + c, m != prev, after != m)) return;
            prev = m;
            c = row_ends ? 0 : c + 1;
            m += row_ends;
        }
    }
}

template <int NW>
__global__ void __launch_bounds__(kBoundThreads, 1)
bound_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap, const BoundCall c) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int chunks = (c.kd + kChunkK - 1) / kChunkK, steps = (c.kd + 15) / 16;
    const int stages = c.stages;
    uint8_t* s_a = base;                                    // chunks x 16 KB
    uint8_t* s_b = s_a + chunks * kAChunk;                  // stages x 30 KB
    __shared__ uint64_t bar[2 * kMaxStages + 7];            // full[S], empty[S], a_full, a_empty, acc_full[2], acc_empty[2], done
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ int s_stop[2];
    volatile int* abort_flag = &s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t full0 = smem_u32(&bar[0]), empty0 = smem_u32(&bar[kMaxStages]);
    const uint32_t a_full = smem_u32(&bar[2 * kMaxStages]), a_empty = smem_u32(&bar[2 * kMaxStages + 1]);
    const uint32_t accf0 = smem_u32(&bar[2 * kMaxStages + 2]), acce0 = smem_u32(&bar[2 * kMaxStages + 4]);
    const uint32_t done = smem_u32(&bar[2 * kMaxStages + 6]);   // MMAs finished, when stopping
    constexpr int kPat = kN / NW;                           // patterns per unit
    Units g;
    g.mt = (c.K + kM - 1) / kM;
    g.cta = blockIdx.x;
    g.ctas = gridDim.x;
    g.nt = (int)((c.n + kPat - 1) / kPat);

    if (threadIdx.x == 0) {
        for (int i = 0; i < kMaxStages; ++i) {
            mbar_init(full0 + 8 * i, 1);
            mbar_init(empty0 + 8 * i, 1);
        }
        mbar_init(a_full, 1);
        mbar_init(a_empty, 1);
        mbar_init(done, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(accf0 + 8 * i, 1);
            mbar_init(acce0 + 8 * i, kEpiThreads / 32);
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&amap) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&bmap) : "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        // ================================================================ TMA producer
        if (lane == 0) {
            uint32_t q = 0, na = 0;                         // ring chunks and template tiles loaded
            uint32_t slot = 0, phase = 0;                   // of the next chunk (counted on, not divided)
            for_units(g, [&](int m, int ct, bool first, bool) {
                if (first) {
                    if (!mbar_wait(a_empty, (na & 1u) ^ 1u, abort_flag)) { *abort_flag = 1; return false; }
                    mbar_expect_tx(a_full, (uint32_t)(chunks * kAChunk));
                    for (int ch = 0; ch < chunks; ++ch)
                        tma_load_2d(smem_u32(s_a + ch * kAChunk), &amap, ch * kChunkK, m * kM, a_full);
                    ++na;
                }
                for (int ch = 0; ch < chunks; ++ch, ++q) {
                    if (!mbar_wait(empty0 + 8 * slot, phase ^ 1u, abort_flag)) { *abort_flag = 1; return false; }
                    mbar_expect_tx(full0 + 8 * slot, kBChunk);
                    tma_load_2d(smem_u32(s_b + slot * kBChunk), &bmap, ch * kChunkK, ct * kN, full0 + 8 * slot);
                    if (++slot == (uint32_t)stages) { slot = 0; phase ^= 1u; }
                }
                return true;
            });
            // the copies issued last must land before the CTA exits (they complete on their own)
            volatile int never = 0;
            for (uint32_t i = 0; i < (uint32_t)stages && i < q; ++i) {
                const uint32_t qq = q - 1 - i, last = qq % stages;
                mbar_wait(full0 + 8 * last, (qq / stages) & 1u, &never);
            }
            if (na) mbar_wait(a_full, (na - 1) & 1u, &never);
        }
    } else if (warp == 1) {
        // ================================================================ MMA issuer
        if (lane == 0 && !c.stall) {
            const uint32_t idesc = idesc_f16(kM, kN);
            const uint64_t a_desc = sdesc_kmajor(smem_u32(s_a)), b_desc = sdesc_kmajor(smem_u32(s_b));
            uint32_t na = 0, tt = 0, slot = 0, phase = 0;
            bool stop = false, issued = false;
            for_units(g, [&](int, int, bool first, bool last) {
                if (first) {
                    if (!mbar_wait(a_full, na & 1u, abort_flag)) { stop = true; return false; }
                    ++na;
                }
                const uint32_t buf = tt & 1u;
                if (!mbar_wait(acce0 + 8 * buf, ((tt >> 1) & 1u) ^ 1u, abort_flag)) { stop = true; return false; }
                tc_fence_after();
                const uint32_t d = tmem + buf * kAccStride;
                for (int ch = 0; ch < chunks; ++ch) {
                    if (!mbar_wait(full0 + 8 * slot, phase, abort_flag)) { stop = true; return false; }
                    tc_fence_after();
                    // (descriptors counted on from the chunk's: an MMA takes 127 clocks, and building
                    // both from scratch for each had taken the issuing thread longer than that)
                    const uint64_t da = a_desc + (uint64_t)(ch * (kAChunk >> 4));
                    const uint64_t db = b_desc + (uint64_t)(slot * (kBChunk >> 4));
                    const int ks_n = steps - ch * (kChunkK / 16);
#pragma unroll
                    for (int ks = 0; ks < kChunkK / 16; ++ks)
                        if (ks < ks_n) mma_f16(d, da + 2 * ks, db + 2 * ks, idesc, (ch | ks) ? 1u : 0u);
                    mma_commit(empty0 + 8 * slot);
                    issued = true;
                    if (++slot == (uint32_t)stages) { slot = 0; phase ^= 1u; }
                }
                if (last) mma_commit(a_empty);
                mma_commit(accf0 + 8 * buf);
                ++tt;
                return true;
            });
            if (stop) {
                *abort_flag = 1;
                if (issued) {                               // let the MMAs already issued finish
                    volatile int never = 0;
                    mma_commit(done);
                    mbar_wait(done, 0, &never);
                }
            }
        }
    } else if (warp >= kEpi0) {
        // ================================================================ epilogue (warps 4-11)
        const int ew = warp - kEpi0, quad = warp & 3, half = ew >> 2;
        const int et = threadIdx.x - kEpi0 * 32;
        const uint32_t tb = tmem + ((uint32_t)(quad * 32) << 16) + half * kHalf;
        constexpr int kMine = kHalf / NW;                   // patterns of this warp's columns
        uint32_t tt = 0;
        for_units(g, [&](int m, int ct, bool, bool) {
            const uint32_t buf = tt & 1u;
            // one thread waits and publishes one decision (a word per unit parity, so the next unit's
            // write cannot overtake a slow reader of this one)
            if (et == 0) {
                const bool ok = mbar_wait(accf0 + 8 * buf, (tt >> 1) & 1u, abort_flag);
                if (!ok) *abort_flag = 1;
                s_stop[buf] = (!ok || *abort_flag) ? 1 : 0;
            }
            named_bar(1, kEpiThreads);
            if (*(volatile int*)&s_stop[buf]) return false;
            tc_fence_after();
            uint32_t r[kHalf];
            tmem_ld120(tb + buf * kAccStride, r);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce0 + 8 * buf);    // the accumulator is in registers
            const int k = m * kM + quad * 32 + lane, word = m * (kM / 32) + quad;
            const int64_t p0 = (int64_t)ct * kPat + half * kMine;
            uint32_t wm = 0;                                // lane i: the word's maximum for pattern i
#pragma unroll
            for (int i = 0; i < kMine; ++i) {
                float v = __uint_as_float(r[i * NW]);
#pragma unroll
                for (int h = 1; h < NW; ++h) v = fmaxf(v, __uint_as_float(r[i * NW + h]));
                const uint32_t u = k < c.K ? bound_key(__float2half_ru(fmaf(fabsf(v), kRaise, v))) : 0u;
                if (k < c.K && p0 + i < c.n) c.u[(size_t)(p0 + i) * c.words * 32 + k] = (unsigned short)u;
                const uint32_t x = __reduce_max_sync(0xffffffffu, u);
                if (lane == i) wm = x;
            }
            if (lane < kMine && p0 + lane < c.n && word < c.words)
                c.wmax[(size_t)(p0 + lane) * c.words + word] = (unsigned short)wm;
            ++tt;
            return true;
        });
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*abort_flag && threadIdx.x == 0) atomicOr(c.error, 8u);
    if (warp == 2) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

int bound_stages(int kd) {
    const int chunks = (kd + kChunkK - 1) / kChunkK;
    return std::min(kMaxStages, (int)((226 * 1024 - 1024 - chunks * kAChunk) / kBChunk));
}

}  // namespace

// Six windows, twelve where templates of like weights compete (`fine`: unit intensities, or 20 and
// more spots a template).  Twelve cost more to make and leave fewer scores.  The whole call, us, six /
// twelve, 1024 patterns without pre-filter: 3 spots 567 / 548, with unit intensities 693 / 667; 7 spots
// 406 / 482, unit 545 / 505; 12 spots (20896 templates) 616 / 672, (5292) 569 / 475; 24 spots 2433 / 2265;
// 33 spots (6990) 1873 / 1114, (1780) 1449 / 941.  8192 patterns: 3 spots 2415 / 2561, 7 spots 2561 /
// 3166, unit 2986 / 3261, 33 spots (1780) 8837 / 5275.  64 patterns: 7 spots 100 / 109, unit 159 / 119,
// 33 spots 354 / 204.  Unit intensities over a subtracted background (two-stage scan, bounds and scores,
// 8192 patterns): 6040 / 3480.  Between 8 and 20 spots either side wins by up to a sixth.
bool bound_shape(int n_rad, int n_theta, bool fine, BoundShape* out) {
    if (n_rad < 1 || n_theta < 64) return false;
    BoundShape s;
    s.nw = fine ? 12 : 6;
    s.nch = 0;
    for (int nch : {24, 18, 12, 9})
        if (n_rad * nch + 1 <= 512) {
            s.nch = nch;
            break;
        }
    if (!s.nch) return false;
    s.pieces = std::lcm(s.nch, s.nw);
    if (s.pieces > n_theta) return false;
    s.kd = n_rad * s.nch + 1;
    s.pitch = (s.kd + 7) & ~7;
    *out = s;
    return true;
}

cudaError_t launch_bound_templates(const int4* meta, const int4* order, const int2* spot, int K, int n_theta, int n_rad,
                                   const BoundShape& s, void* out, cudaStream_t st) {
    if (K <= 0) return cudaSuccess;
    bound_templates_kernel<<<(K + 3) / 4, 128, (size_t)4 * s.pitch * sizeof(float), st>>>(
        meta, order, spot, K, n_theta, n_rad, s, (__half*)out);
    return cudaGetLastError();
}

cudaError_t launch_bound_windows(const float* polar, const float* pnorm, int64_t n, int n_r, int n_theta,
                                 const int32_t* radii, int n_rad, const BoundShape& s, void* w, int* counter,
                                 cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int64_t cap = (int64_t)device_sms() * 8;
    const size_t smem = (size_t)n_rad * s.pieces * sizeof(float);
    window_kernel<<<(int)std::min<int64_t>(n, cap), 256, smem, st>>>(polar, pnorm, n, n_r, n_theta, radii, n_rad, s,
                                                                     (__half*)w, counter);
    return cudaGetLastError();
}

int bound_box_rows(bool templates) { return templates ? kM : kN; }

cudaError_t launch_bound(const void* amap, const void* bmap, const BoundCall& call, int nw, int num_sms,
                         cudaStream_t st) {
    if (call.n <= 0 || call.K <= 0) return cudaSuccess;
    BoundCall c = call;
    c.stages = bound_stages(c.kd);
    const int chunks = (c.kd + kChunkK - 1) / kChunkK;
    const size_t smem = 1024 + (size_t)chunks * kAChunk + (size_t)c.stages * kBChunk;
    const void* fn = nw == 12 ? (const void*)bound_kernel<12> : (const void*)bound_kernel<6>;
    const cudaError_t e = kernel_occupancy(fn, kBoundThreads, smem, nullptr);
    if (e != cudaSuccess) return e;
    const int pat = kN / nw;
    const int64_t units = (int64_t)((c.K + kM - 1) / kM) * ((c.n + pat - 1) / pat);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms, units));
    if (nw == 12)
        bound_kernel<12><<<grid, kBoundThreads, smem, st>>>(*(const CUtensorMap*)amap, *(const CUtensorMap*)bmap, c);
    else
        bound_kernel<6><<<grid, kBoundThreads, smem, st>>>(*(const CUtensorMap*)amap, *(const CUtensorMap*)bmap, c);
    return cudaGetLastError();
}

}  // namespace tmgb
