// Exact scores of the few templates that can enter a pattern's top N, and the top N (arXiv
// 2111.07347, Eq. 1 and Section 2.2), for one library.
//
// With upper bounds U[p][j] of the correlation index (k_bound.cu; position j is template order[j].w,
// fewest spots first): a CTA takes a pattern, stages its polar rows (k_sparse.cu's layouts), scores
// first the templates of highest bound (the seeds: the best of a few words of 32 positions per
// warp), and then, word by word, every template whose bound reaches the threshold.  The words'
// maxima say which words hold one at all, so most of a library's bounds are never read.
// The threshold is the N-th best of the scores so far under the order of the results, (Q desc,
// template asc), as one 64-bit key: a pool of N keys in shared memory holds the N best; an arriving
// score replaces the smallest (compare-and-swap; every key is another template's, and keys only
// grow, so the smallest is at any time a lower bound of the final N-th best).  A template whose
// (bound, index) is below it cannot be among the final N, ties included (patterns on which every
// template ties, such as blank ones, are decided by index after a few dozen scores).
// Without bounds (u null) the templates of the mask are scored, all of them, by words or
// quarters of words: the rescoring of a few candidates per pattern, or a small library.
//
// 32768 patterns against the 13986-template HCP library: bounds and scores 5.8 ms (windows 0.57, the
// contraction 2.3, this kernel 2.9), where bounding and scoring in one kernel on the CUDA cores took
// 18.9 ms.  Bound by latency and issue: 0.59 warp instructions a cycle per scheduler, most other
// cycles at the barriers between a pattern's phases.
// One warp scores one template (score_template: all its shifts in registers, spots in CSR order, as
// every other kernel does, so scores are the same bits).  Results do not depend on scheduling.
#include <cuda_fp16.h>

#include <algorithm>

#include "tm_device.h"
#include "tm_internal.h"
#include "tm_score.h"

namespace tmgb {
namespace {

constexpr int kMaxWarps = 32;
constexpr int kSeeds = 64;                 // templates scored first, over all warps, at most
constexpr int kQueue = 512;                // items (words or parts of them) taken per round

// The bound of a key (k_bound.cu): FP16 from its order-preserving 16 bits.
__device__ __forceinline__ float bound_of(uint32_t key) {
    return __half2float(__ushort_as_half((unsigned short)(key & 0x8000u ? key & 0x7fffu : ~key)));
}

// Results' order as integers: larger is better; none is below every template's.  A score that is not a
// number (an infinite correlation over an infinite norm) ranks below every number: it is -inf here and
// in the warps' lists, and written out as NaN.
__device__ __forceinline__ unsigned long long rank_key(float q, int k) {
    return ((unsigned long long)score_key(q + 0.0f) << 32) | (0xffffffffu - (unsigned)k);   // (-0 ties with 0)
}
constexpr unsigned long long kNoKey = 0x007fffffull << 32;              // score -inf, no template
__device__ __forceinline__ float rank_score(unsigned long long key) { return key_score((unsigned)(key >> 32)); }
__device__ __forceinline__ unsigned long long warp_min(unsigned long long v) {
    const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(v >> 32));
    const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)(v >> 32) == hi ? (unsigned)v : 0xffffffffu);
    return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
    return ((unsigned long long)hi << 32) | lo;
}

// Largest block: 64 registers a thread hold up to 12 accumulators a lane, else 128.
constexpr int max_threads(int nb_max) { return nb_max <= 12 ? 1024 : 512; }

// BOUNDS: behind bounds (c.u), or the templates of the mask.  At compile time: together in one kernel,
// the registers of each cost the other up to 7 %.
template <int NBMAX, int LAYOUT, bool BOUNDS>
__global__ void __launch_bounds__(max_threads(NBMAX), 1)
score_kernel(const ScoreCall c) {
    extern __shared__ __align__(16) float smem[];
    const SparseLib& L = c.lib;
    const int n_theta = c.n_theta, pitch = c.pitch, N = c.top_n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    float* sP = smem;                                       // [n_rad][pitch]
    // [N] keys of the N best scores so far, 8-byte aligned
    unsigned long long* s_pool = (unsigned long long*)(sP + (((size_t)L.n_rad * pitch + 1) & ~(size_t)1));
    float* lq = (float*)(s_pool + N);                       // [nwarps][N] scores, templates, shifts
    int* lk = (int*)(lq + nwarps * N);
    int* ls = lk + nwarps * N;
    __shared__ int lcnt[kMaxWarps];
    __shared__ int s_seed[kSeeds];                          // seeded positions (-1: none)
    __shared__ unsigned long long s_seedkey[kSeeds];        // and their scores' keys
    __shared__ unsigned short s_queue[kQueue];              // words of a round, from its first word
    __shared__ int s_pattern, s_push, s_pop;
    __shared__ unsigned long long s_thr;                    // their smallest
    __shared__ __align__(8) uint64_t s_bar;
    const bool bulk = c.bulk && (pitch & 3) == 0 && (n_theta & 3) == 0;
    uint32_t n_bulk = 0;
    if (bulk && threadIdx.x == 0) mbar_init1(&s_bar);
    const int2* spots = LAYOUT == TM_LAYOUT_WRAP ? L.spot : L.spot2;
    float* wq = lq + warp * N;
    int* wk = lk + warp * N;
    int* ws = ls + warp * N;
    unsigned long long work = 0;                            // multiply-adds of this warp (lane 0)
    const int wseeds = max(1, c.seeds / nwarps);            // seeds per warp
    // items of 8 templates while the words alone would not occupy the warps (with bounds, which leave
    // few templates of most words, only in the large blocks of few patterns or long rows and up to 2048
    // templates: 64 patterns against 600 templates that the bounds cannot tell apart 279 us, by words
    // 328; 1024 against 1000 of them 2064 and 2282)
    const int part = (BOUNDS ? nwarps >= 16 && L.words < 64 : L.words < 8 * nwarps) ? 2 : 0;
    auto part_mask = [&](int w) -> uint32_t { return part ? 0xffu << (8 * (w & 3)) : 0xffffffffu; };

    for (;;) {
        __syncthreads();                                    // previous pattern fully done
        if (threadIdx.x == 0) {
            s_pattern = atomicAdd(c.counter, 1);
            s_push = 0;
            s_pop = 0;
            s_thr = kNoKey;
        }
        if (threadIdx.x < nwarps) lcnt[threadIdx.x] = 0;
        for (int i = threadIdx.x; i < N; i += blockDim.x) s_pool[i] = kNoKey;
        __syncthreads();
        const int64_t p = s_pattern;
        if (p >= c.n) break;
        const float* src = c.polar + (size_t)p * c.n_r * n_theta;
        const float pn = __ldg(c.pnorm + p);
        const uint32_t* mrow = c.mask ? c.mask + (size_t)p * L.words : nullptr;
        const unsigned short* urow = BOUNDS ? c.u + (size_t)p * L.words * 32 : nullptr;
        const unsigned short* wrow = BOUNDS ? c.wmax + (size_t)p * L.words : nullptr;

        // ---- the library's polar rows
        if (bulk) {
            const int nseg = (pitch + n_theta - 1) / n_theta;
            fence_proxy_async_smem();                       // earlier reads of sP before the copies
            if (threadIdx.x == 0)
                mbar_arrive_expect_tx(&s_bar, (uint32_t)(L.n_rad * pitch * 4) + (c.test_stall ? 16u : 0u));
            for (int it = threadIdx.x; it < L.n_rad * nseg; it += blockDim.x) {
                const int rr = it / nseg, c0 = (it - rr * nseg) * n_theta;
                bulk_g2s(sP + (size_t)rr * pitch + c0, src + (size_t)__ldg(L.radii + rr) * n_theta,
                         (uint32_t)(min(n_theta, pitch - c0) * 4), &s_bar);
            }
        } else {
            for (int rr = warp; rr < L.n_rad; rr += nwarps) {
                const float* row = src + (size_t)__ldg(L.radii + rr) * n_theta;
                float* dst = sP + (size_t)rr * pitch;
#pragma unroll 4
                for (int col = lane; col < pitch; col += 32) {
                    int sc = col;
                    while (sc >= n_theta) sc -= n_theta;
                    dst[col] = __ldg(row + sc);
                }
            }
        }
        // bring into L2 the same rows, and the word maxima, of pattern p + gridDim.x: patterns are taken
        // in order, so some CTA takes it soon (one 128-byte line per thread)
        if (p + gridDim.x < c.n) {
            const int lines = (n_theta * (int)sizeof(float) + 127) >> 7;
            const float* nsrc = src + (size_t)gridDim.x * c.n_r * n_theta;
            for (int i = threadIdx.x; i < L.n_rad * lines; i += blockDim.x) {
                const int r0 = i / lines, l = i - r0 * lines;
                const char* a = reinterpret_cast<const char*>(nsrc + (size_t)__ldg(L.radii + r0) * n_theta) + 128 * l;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
            }
            if (BOUNDS && threadIdx.x * 64 < L.words)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(wrow + (size_t)gridDim.x * L.words + threadIdx.x * 64));
        }
        // whether the template at a position takes part (bounds: positions are in `order`)
        auto word_mask = [&](int w) -> uint32_t {
            uint32_t m = mrow ? __ldg(mrow + w) : 0xffffffffu;
            const int rem = L.K - w * 32;
            return rem < 32 ? m & ((1u << rem) - 1u) : m;
        };
        auto takes_part = [&](int k) -> bool {
            return k >= 0 && (!mrow || ((__ldg(mrow + (k >> 5)) >> (k & 31)) & 1u));
        };
        // ---- seeds: of the warp's words (w = warp mod nwarps), those of highest maximum
        int seed_l = -1;                                    // lane i < wseeds: position of the warp's i-th seed
        if (BOUNDS) {
            uint32_t best = 0;                              // lane's best word: maximum << 16 | local index
            for (int i = lane; warp + i * nwarps < L.words; i += 32) {
                const uint32_t m = __ldg(wrow + warp + i * nwarps);
                const uint32_t key = (m << 16) | (uint32_t)(0xffff - min(i, 0xffff));
                best = max(best, key);
            }
            for (int i = 0; i < wseeds; ++i) {
                const uint32_t top = __reduce_max_sync(0xffffffffu, best);
                if (top == 0) break;                        // fewer words than seeds
                if (best == top) best = 0;                  // (the local index makes keys distinct)
                const int w = warp + (int)(0xffffu - (top & 0xffffu)) * nwarps;
                const bool in = takes_part(__ldg(&c.order[w * 32 + lane].w));
                const uint32_t u = in ? (uint32_t)__ldg(urow + w * 32 + lane) + 1u : 0u;
                const uint32_t um = __reduce_max_sync(0xffffffffu, u);
                if (um == 0) continue;                      // every template of the word is masked out
                const int b = __ffs(__ballot_sync(0xffffffffu, u == um)) - 1;
                if (lane == i) seed_l = w * 32 + b;
            }
            if (lane < wseeds) {
                s_seed[warp * wseeds + lane] = seed_l;
                s_seedkey[warp * wseeds + lane] = kNoKey;
            }
        }
        if (bulk) {
            // one warp polls, the others wait at the barrier without taking issue slots
            const bool ok = warp != 0 || mbar_wait_bounded(&s_bar, n_bulk & 1u);
            if (__syncthreads_or(!ok)) {
                // the copies did not land in time: report it, let them finish (bounded), stop
                if (threadIdx.x == 0) {
                    atomicOr(c.error, 4u);
                    mbar_wait_bounded(&s_bar, n_bulk & 1u);
                }
                __syncthreads();
                return;
            }
            ++n_bulk;
        } else {
            __syncthreads();
        }

        // score template k (warp-collective; `mine`: its first spots) and keep it in the warp's top-N
        // when it enters; returns its key (kNoKey when it cannot enter the result)
        auto score_one = [&](int k, const int4& meta, int2 mine) -> unsigned long long {
            const int cnt = meta.y & 0xffff, S = (int)((unsigned)meta.y >> 16);
            const float d = pn * __int_as_float(meta.z);
            const float thr = rank_score(*(volatile unsigned long long*)&s_thr);
            // a template whose correlation stays below the threshold (in correlation units, with a
            // margin for the division's rounding) cannot enter the top-N: its shift is not resolved
            float thr_c = -FLT_MAX;
            if (thr > -INFINITY && d > 0.0f) {
                const float t = thr * d;
                thr_c = fmaxf(t - fabsf(t) * 1e-6f, -FLT_MAX);   // (an infinite norm, NaN: every template is resolved)
            }
            int s = 0;
            bool resolved = false;
            const float best = score_dispatch<NBMAX, LAYOUT>(sP, spots, meta.x, cnt, mine, S, n_theta, pitch, lane,
                                                             thr_c, s, resolved);
            if (c.work) work += (unsigned long long)cnt * (unsigned long long)S;
            if (!resolved) return kNoKey;
            float q;
            if (d > 0.0f) q = __fdiv_rn(best, d);
            else { q = 0.0f; s = 0; }
            if (q != q) q = -INFINITY;
            if (lane == 0) {
                const int cnt_w = lcnt[warp];
                if (cnt_w < N || better(q, k, wq[N - 1], wk[N - 1])) {
                    int i = cnt_w < N ? cnt_w : N - 1;
                    while (i > 0 && better(q, k, wq[i - 1], wk[i - 1])) {
                        wq[i] = wq[i - 1]; wk[i] = wk[i - 1]; ws[i] = ws[i - 1];
                        --i;
                    }
                    wq[i] = q; wk[i] = k; ws[i] = s;
                    if (cnt_w < N) lcnt[warp] = cnt_w + 1;
                }
            }
            __syncwarp();
            return rank_key(q, k);
        };
        // a key into the pool: in place of the smallest while it is larger (warp-collective)
        auto pool_add = [&](unsigned long long key) {
            for (;;) {
                unsigned long long lo = ~0ull;
                int at = 0;
                for (int i = lane; i < N; i += 32) {
                    const unsigned long long v = *(volatile unsigned long long*)&s_pool[i];
                    if (v < lo) { lo = v; at = i; }
                }
                const unsigned long long m = warp_min(lo);
                if (m >= key) break;
                const int from = __ffs(__ballot_sync(0xffffffffu, lo == m)) - 1;
                unsigned long long old = 0;
                if (lane == from) old = atomicCAS(&s_pool[at], m, key);
                if (__shfl_sync(0xffffffffu, old, from) != m) continue;
                lo = ~0ull;                                 // taken: the smallest of the pool now
                for (int i = lane; i < N; i += 32) lo = min(lo, *(volatile unsigned long long*)&s_pool[i]);
                lo = warp_min(lo);
                if (lane == 0) atomicMax(&s_thr, lo);
                break;
            }
        };

        unsigned long long thr0 = kNoKey;                   // the N-th best of the seeds
        if (BOUNDS) {
            // the seeds, each one's metadata and spots on their way before the one before is scored
            int4 meta_l = make_int4(0, 0, 0, -1);
            if (seed_l >= 0) meta_l = __ldg(c.order + seed_l);
            int4 m;
            int2 mine;
            auto fetch = [&](int i) {
                m.x = __shfl_sync(0xffffffffu, meta_l.x, i);
                m.y = __shfl_sync(0xffffffffu, meta_l.y, i);
                m.z = __shfl_sync(0xffffffffu, meta_l.z, i);
                m.w = __shfl_sync(0xffffffffu, meta_l.w, i);
                mine = lane_spot(spots, m.x, m.y & 0xffff, lane);
            };
            fetch(0);
            for (int i = 0; i < wseeds; ++i) {
                const int4 m_i = m;
                const int2 mine_i = mine;
                if (i + 1 < wseeds) fetch(i + 1);
                if (m_i.w < 0) continue;
                const unsigned long long key = score_one(m_i.w, m_i, mine_i);
                if (lane == 0) s_seedkey[warp * wseeds + i] = key;
            }
            __syncthreads();
            // every warp ranks the seeds' keys; the last one puts the N best into the pool, which is
            // read after the next barrier
            const int total = nwarps * wseeds;              // at most 64: two per lane
            unsigned long long key[kSeeds / 32];
#pragma unroll
            for (int i = 0; i < kSeeds / 32; ++i) key[i] = lane + 32 * i < total ? s_seedkey[lane + 32 * i] : kNoKey;
            for (int j = 0; j < N; ++j) {
                unsigned long long top = key[0];
#pragma unroll
                for (int i = 1; i < kSeeds / 32; ++i) top = max(top, key[i]);
                top = warp_max(top);
                if (top == kNoKey) break;                   // (thr0 stays: fewer than N)
                if (warp == nwarps - 1 && lane == 0) s_pool[j] = top;
#pragma unroll
                for (int i = 0; i < kSeeds / 32; ++i)
                    if (key[i] == top) key[i] = kNoKey;
                if (j == N - 1) {
                    thr0 = top;
                    if (warp == nwarps - 1 && lane == 0) s_thr = top;
                }
            }
        }
        // ---- the other templates, in rounds of kQueue items: the words that hold a template whose
        // bound reaches the threshold (or the parts of words that hold a template of the mask) go to
        // a queue, the warps take them from it and score their templates
        const int items = L.words << part;
        for (int w0 = 0; w0 < items; w0 += kQueue) {
            if (w0) {
                __syncthreads();                            // the round before is done
                if (threadIdx.x == 0) { s_push = 0; s_pop = 0; }
                __syncthreads();
            }
            const float cut0 = rank_score(w0 ? *(volatile unsigned long long*)&s_thr : thr0);
            for (int b = w0 + warp * 32; b < min(w0 + kQueue, items); b += blockDim.x) {
                const int w = b + lane;
                bool in = w < items;
                if (in)
                    in = BOUNDS ? !(bound_of(__ldg(wrow + (w >> part))) < cut0)
                                : (word_mask(w >> part) & part_mask(w)) != 0u;
                const unsigned bal = __ballot_sync(0xffffffffu, in);
                int at = 0;
                if (lane == 0 && bal) at = atomicAdd(&s_push, __popc(bal));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
                if (in) s_queue[at] = (unsigned short)(w - w0);
            }
            __syncthreads();
            const int n_q = s_push;
            for (;;) {
                int i = 0;
                if (lane == 0) i = atomicAdd(&s_pop, 1);
                i = __shfl_sync(0xffffffffu, i, 0);
                if (i >= n_q) break;
                const int w = w0 + s_queue[i], k0 = (w >> part) * 32;
                uint32_t m;
                int4 meta_l = make_int4(0, 0, 0, 0);
                float u_l = INFINITY;
                if (BOUNDS) {
                    // the word's templates that take part, not the seeds, that the threshold as it is
                    // now leaves
                    u_l = bound_of(__ldg(urow + k0 + lane));
                    const unsigned long long thr = *(volatile unsigned long long*)&s_thr;
                    bool in = !(u_l < rank_score(thr));
                    if (in) meta_l = __ldg(c.order + k0 + lane);
                    in = in && takes_part(meta_l.w) && rank_key(u_l, meta_l.w) > thr;
                    uint32_t seeded = 0;
                    for (int i = lane; i < nwarps * wseeds; i += 32) {
                        const int sd = s_seed[i];
                        if ((sd >> 5) == (w >> part)) seeded |= 1u << (sd & 31);
                    }
                    m = __ballot_sync(0xffffffffu, in) & ~__reduce_or_sync(0xffffffffu, seeded) & part_mask(w);
                } else {
                    m = word_mask(w >> part) & part_mask(w);
                    if ((m >> lane) & 1u) {
                        meta_l = __ldg(L.meta + k0 + lane);
                        meta_l.w = k0 + lane;
                    }
                }
                if (!m) continue;
                // each template's spots are on their way while the one before is scored
                int4 next;
                int2 mine;
                int bit = __ffs(m) - 1;
                auto fetch = [&]() {
                    next.x = __shfl_sync(0xffffffffu, meta_l.x, bit);
                    next.y = __shfl_sync(0xffffffffu, meta_l.y, bit);
                    next.z = __shfl_sync(0xffffffffu, meta_l.z, bit);
                    next.w = __shfl_sync(0xffffffffu, meta_l.w, bit);
                    mine = lane_spot(spots, next.x, next.y & 0xffff, lane);
                };
                fetch();
                while (m) {
                    const int4 cur = next;
                    const int2 mine_c = mine;
                    const float u_c = __shfl_sync(0xffffffffu, u_l, bit);
                    m &= m - 1;
                    if (m) {
                        bit = __ffs(m) - 1;
                        fetch();
                    }
                    if (BOUNDS && rank_key(u_c, cur.w) < *(volatile unsigned long long*)&s_thr) continue;
                    const unsigned long long key = score_one(cur.w, cur, mine_c);
                    if (key > *(volatile unsigned long long*)&s_thr) pool_add(key);
                }
            }
        }
        __syncthreads();
        // ---- the results: the pool holds the N best keys; an entry of the warps' lists that is one of
        // them goes to its rank
        tm_hit* out = c.hits + (size_t)p * N;
        for (int i = threadIdx.x; i < nwarps * N; i += blockDim.x) {
            const int w = i / N;
            if (i - w * N >= lcnt[w]) continue;
            const float q = lq[i];
            const int k = lk[i];
            const unsigned long long key = rank_key(q, k);
            if (key < s_thr) continue;
            int rank = 0;
            for (int j = 0; j < N; ++j) rank += s_pool[j] > key;
            if (rank >= N) continue;
            tm_hit h;
            h.template_index = k;
            h.shift = ls[i] < n_theta ? ls[i] : 0;          // (no shift's sum is a number)
            h.score = q == -INFINITY ? nanf("") : q;
            h.angle_deg = (float)h.shift * (360.0f / (float)n_theta);
            h.mirror = (L.mirror && k >= L.K0) ? 1 : 0;
            out[rank] = h;
        }
        // fewer than N templates took part: the last rows are empty
        for (int j = threadIdx.x; j < N; j += blockDim.x) {
            if (s_thr != kNoKey) break;
            int filled = 0;
            for (int i = 0; i < N; ++i) filled += s_pool[i] != kNoKey;
            if (j >= filled) {
                tm_hit h;
                h.template_index = -1; h.shift = -1; h.score = -INFINITY;
                h.angle_deg = 0.0f; h.mirror = 0;
                out[j] = h;
            }
        }
    }
    if (c.work && lane == 0 && work) atomicAdd(c.work, work);
}

// Accumulators a lane for n_theta shifts: the instantiation that serves them.
int nb_max(int n_theta) {
    const int nb = (n_theta + 31) / 32;
    return nb <= 6 ? 6 : nb <= 12 ? 12 : nb <= 24 ? 24 : 32;
}

// Shared memory of the rows (row pitch `pitch`), the pool and the lists of `warps` warps.
size_t score_smem(int n_rad, int pitch, int top_n, int warps) {
    return (size_t)n_rad * pitch * 4 + 8 + (size_t)top_n * 8 + (size_t)warps * top_n * 12;
}
constexpr size_t kMaxSmem = 227 * 1024 - 2560;             // (the rest: the kernel's static arrays)

// The row layout (wrap-free while two CTAs fit an SM, else wrapped) and its pitch; false where the
// largest block's lists do not fit beside the rows.  Chosen once per call, for the largest block of
// the instantiation, so every smaller block fits as well.  Not the dual layout: its halved loads gain
// less than its shared memory costs in resident warps (FCC library, 16384 patterns with pre-filter:
// bounds and scores 2.94 ms, wrap-free 2.60 ms).
bool score_layout(int n_rad, int n_theta, int top_n, int* layout, int* pitch) {
    if (n_theta < 1 || n_theta > 1024 || top_n < 1 || top_n > TM_MAX_TOPN || n_rad < 1) return false;
    const int warps = max_threads(nb_max(n_theta)) / 32;
    const int order[2] = {TM_LAYOUT_WF, TM_LAYOUT_WRAP};
    const size_t limit[2] = {113 * 1024 - 2560, kMaxSmem};
    for (int i = 0; i < 2; ++i) {
        const int pch = sparse_pitch(n_theta, order[i]);
        if (order[i] == TM_LAYOUT_WF && (size_t)n_rad * pch > 65535) continue;   // 16-bit offsets
        if (score_smem(n_rad, pch, top_n, warps) <= limit[i]) {
            *layout = order[i];
            *pitch = pch;
            return true;
        }
    }
    return false;
}

int block_sizes(int n_rad, int n_theta, int pitch, int top_n, int threads[3]) {
    int n = 0;
    for (int t : {256, 512, 1024})
        if (t <= max_threads(nb_max(n_theta)) && score_smem(n_rad, pitch, top_n, t / 32) <= kMaxSmem)
            threads[n++] = t;
    return n;
}

template <int NBMAX, int LAYOUT, bool BOUNDS>
cudaError_t launch_sizes(const ScoreCall& c, int num_sms, cudaStream_t st) {
    // Block size: with at most two patterns per SM, as many warps on each as fit; else the smallest
    // block that fills the SM's registers (blocks run their phases out of step).
    int threads = 0, per_sm = 0;
    size_t smem = 0;
    const int64_t share = (c.n + num_sms - 1) / num_sms;
    int sizes[3];
    const int n_sizes = block_sizes(c.lib.n_rad, c.n_theta, c.pitch, c.top_n, sizes);
    for (int i = 0; i < n_sizes; ++i) {
        const int t = sizes[i];
        int b = 0;
        const size_t sm = score_smem(c.lib.n_rad, c.pitch, c.top_n, t / 32);
        const cudaError_t e = kernel_occupancy((const void*)score_kernel<NBMAX, LAYOUT, BOUNDS>, t, sm, &b);
        if (e != cudaSuccess) return e;
        const int64_t used = std::min<int64_t>(b, share);
        if (b > 0 && used * t > (int64_t)threads * std::min<int64_t>(per_sm, share)) {
            threads = t;
            per_sm = b;
            smem = sm;
        }
    }
    if (!threads) return cudaErrorInvalidConfiguration;
    int64_t grid = (int64_t)num_sms * per_sm;
    if (grid > c.n) grid = c.n;
    score_kernel<NBMAX, LAYOUT, BOUNDS><<<(int)grid, threads, smem, st>>>(c);
    return cudaGetLastError();
}

template <int NBMAX, int LAYOUT>
cudaError_t launch_nb(const ScoreCall& c, int num_sms, cudaStream_t st) {
    return c.u ? launch_sizes<NBMAX, LAYOUT, true>(c, num_sms, st) : launch_sizes<NBMAX, LAYOUT, false>(c, num_sms, st);
}

}  // namespace

// Block sizes that can take the call (0: the sparse kernel serves it).
int score_shapes(int n_rad, int n_theta, int top_n, int threads[3]) {
    int layout, pitch;
    return score_layout(n_rad, n_theta, top_n, &layout, &pitch) ? block_sizes(n_rad, n_theta, pitch, top_n, threads) : 0;
}

bool score_supported(int n_rad, int n_theta, int top_n) {
    int layout, pitch;
    return score_layout(n_rad, n_theta, top_n, &layout, &pitch);
}

cudaError_t launch_score(const ScoreCall& call, int num_sms, cudaStream_t st) {
    if (call.n <= 0) return cudaSuccess;
    ScoreCall c = call;
    int layout = TM_LAYOUT_WRAP;
    if (!score_layout(c.lib.n_rad, c.n_theta, c.top_n, &layout, &c.pitch)) return cudaErrorInvalidValue;
    const int nb = nb_max(c.n_theta);
    if (layout == TM_LAYOUT_WF) {
        if (nb == 6) return launch_nb<6, TM_LAYOUT_WF>(c, num_sms, st);
        if (nb == 12) return launch_nb<12, TM_LAYOUT_WF>(c, num_sms, st);
        if (nb == 24) return launch_nb<24, TM_LAYOUT_WF>(c, num_sms, st);
        return launch_nb<32, TM_LAYOUT_WF>(c, num_sms, st);
    }
    if (nb == 6) return launch_nb<6, TM_LAYOUT_WRAP>(c, num_sms, st);
    if (nb == 12) return launch_nb<12, TM_LAYOUT_WRAP>(c, num_sms, st);
    if (nb == 24) return launch_nb<24, TM_LAYOUT_WRAP>(c, num_sms, st);
    return launch_nb<32, TM_LAYOUT_WRAP>(c, num_sms, st);
}

}  // namespace tmgb
