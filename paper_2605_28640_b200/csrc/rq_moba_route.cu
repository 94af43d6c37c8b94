// MoBA routing for bf16 caches (Sec. 2.2, Eq. 3; App. A.1, MoBA paragraph) on the tensor cores: block
// representatives, the scores of every query against the representatives of the blocks before it, and the
// budget's best blocks of every query as a bit mask.
//
//   moba_means_bf16_kernel   per (head, block): the mean of the block's stored keys, fp32
//   moba_route_mma_kernel    per (head, 128 consecutive queries): the representatives cut into three bf16 terms (hi + mid
//                            + lo: 24 significand bits, nothing of the fp32 mean is lost), scores = Q (hi + mid + lo)^T in
//                            tensor memory, then per query the threshold of the budget by value buckets, the mask and,
//                            if asked for, the ascending list
#include <limits.h>
#include <math_constants.h>

#include "rq_async.cuh"
#include "rq_device.cuh"
#include "rq_internal.h"
#include "rq_tmap.h"
#include "rq_umma.cuh"

namespace rq {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kRouteQueries = 128;             // queries of a CTA: the lanes of the accumulator
constexpr int kRouteThreads = 512;             // four threads per query, each a quarter of the score words
constexpr int kRouteGroup = 64;                // blocks of one product (N)
constexpr int kPanelGroups = 8;                // groups whose scores fit in tensor memory at once (512 columns)
constexpr int kRouteBins = 64;                 // value buckets of the threshold search
constexpr int kRouteCap = 16;                  // blocks of the threshold's bucket that are ranked directly

// ---------------------------------------------------------------- block representatives
// Grid (ceil(blocks / R), heads), R = 256 / (D / 2) blocks per CTA, a thread per two channels of a block.  The sum
// runs over the block's valid positions in order.
__global__ void __launch_bounds__(256) moba_means_bf16_kernel(const bf16 *kv, int64_t page_cap, int S, int D, int64_t len, int block,
                                                             float *means, int nb)
{
    const int per = D / 2, r = threadIdx.x / per, c = 2 * (threadIdx.x % per);
    const int j = blockIdx.x * (256 / per) + r, bh = blockIdx.y;
    grid_launch_dependents();
    if (j >= nb) return;
    const int64_t lo = (int64_t)j * block, hi = min(lo + block, len);
    float s0 = 0.0f, s1 = 0.0f;
    int64_t p = lo;
    // sixteen loads in flight at a time (a page holds a multiple of 16 positions and lo is a multiple of 64, so a run
    // of 16 stays inside one page); the additions keep the order of the positions
    for (; p + 16 <= hi; p += 16) {
        const bf16 *src = kv + ((((int64_t)bh * page_cap + p / S) * 2) * S + p % S) * D + c;
        uint32_t x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = __ldg(reinterpret_cast<const uint32_t *>(src + (int64_t)i * D));
#pragma unroll
        for (int i = 0; i < 16; ++i) { s0 += bf16lo(x[i]); s1 += bf16hi(x[i]); }
    }
    for (; p < hi; ++p) {
        const uint32_t x = *reinterpret_cast<const uint32_t *>(kv + ((((int64_t)bh * page_cap + p / S) * 2) * S + p % S) * D + c);
        s0 += bf16lo(x);
        s1 += bf16hi(x);
    }
    const float n = (float)(hi - lo), m0 = s0 / n, m1 = s1 / n;
    *reinterpret_cast<float2 *>(means + ((int64_t)bh * nb + j) * D + c) = make_float2(m0, m1);
}

// ---------------------------------------------------------------- routing
template <int D> struct RouteGeom {
    static constexpr int HALVES = D / 64;
    static constexpr int Q_BYTES = HALVES * kRouteQueries * 128;
    static constexpr int PLANE_BYTES = HALVES * kRouteGroup * 128;
    static constexpr int GROUP_BYTES = 3 * PLANE_BYTES;
    static constexpr int WORK_BYTES = kRouteBins * kRouteQueries * 4 + kRouteCap * kRouteQueries * 6;   // buckets, ranked blocks
    static constexpr int SMALL_BYTES = (12 + 6) * kRouteQueries * 4;
    // a prompt of one panel is done with queries and representatives when the buckets are needed, so these share the space
    static __host__ __device__ int front_bytes(bool one_panel)
    {
        const int qb = Q_BYTES + GROUP_BYTES;
        return one_panel ? (qb > WORK_BYTES ? qb : WORK_BYTES) : qb + WORK_BYTES;
    }
    static int smem_bytes(bool one_panel, int words)
    {
        return 1024 + front_bytes(one_panel) + 2 * words * kRouteQueries * 4 + SMALL_BYTES;
    }
};

// order-preserving image of a score; -0 counts as +0
__device__ __forceinline__ uint32_t score_key(float v)
{
    const uint32_t b = __float_as_uint(v + 0.0f);
    return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
// Value bucket of a score between the query's smallest and largest: monotone in v, 0 .. kRouteBins - 1.
__device__ __forceinline__ uint32_t score_bin(float v, float lo, float inv)
{
    return min(__float_as_uint(fmaf(v - lo, inv, 8388609.0f)) - 0x4B000000u, (uint32_t)(kRouteBins - 1));
}

// Grid (heads, tiles of 128 queries; the tiles of the last queries first: their work is the largest).  Bound by the
// instructions of the three passes over the scores (smallest and largest, buckets, mask; about a dozen per score and
// 32 queries), which is why a pass that ranks every candidate, or one that takes one block per round, is so much
// slower.  Per query:
//   1. smallest and largest score of its candidates (the complete blocks between the first and the query's own);
//   2. 64 value buckets between them: the bucket that holds the last block taken, and how many of it are wanted;
//   3. blocks of higher buckets into the mask; those of the threshold's bucket are ranked against each other by
//      (score, lower block first).
// A threshold bucket of more than 16 blocks is cut further by buckets on the scores' integer images until at most 16
// are left or all left are equal (equal scores: the lowest blocks).  More than 512 blocks are taken in panels of 512,
// whose scores are computed again for each pass (the tensor cores have nothing else to do here).
// Measured, 32 heads x 128 channels: 4096 queries, 16 of 64 blocks each, 158 -> 42 us; 30011 queries, 30 of 469 blocks
// each, 28.9 -> 1.0 ms.  (Before: fp32 FMA scores, a lane per block, then a bit-wise vote search up to 128 blocks and one
// round per taken block beyond.  Of the former: queries by tensor map and four product steps per election 58 -> 52 us,
// candidates noted by one atomic per word instead of one each 52 -> 47 us, half words for up to 64 blocks 47 -> 42 us.)
// HALF: prompts of at most 64 blocks, whose two words of scores are taken by half words, so that all four threads of a query
// have some.
template <int D, bool HALF>
__global__ void __launch_bounds__(kRouteThreads, 2) moba_route_mma_kernel(const __grid_constant__ CUtensorMap qmap, const float *means, int64_t len, int H,
                                                                      int block, int nb, int K, int words, uint32_t *masks,
                                                                      int32_t *list, int32_t *status)
{
    using G = RouteGeom<D>;
    constexpr int NQ = kRouteQueries, NB = kRouteBins, CAP = kRouteCap;
    extern __shared__ __align__(1024) unsigned char rsm_raw[];
    __shared__ __align__(8) uint64_t full_q, done;                                    // a product is complete
    __shared__ uint32_t tbase;
    unsigned char *sm = rsm_raw + ((1024u - (smem_addr(rsm_raw) & 1023u)) & 1023u);
    const int groups_all = (nb + kRouteGroup - 1) / kRouteGroup;
    const bool one_panel_launch = groups_all <= kPanelGroups;
    unsigned char *qs = sm, *bs = sm + G::Q_BYTES;
    uint32_t *hist = reinterpret_cast<uint32_t *>(one_panel_launch ? sm : sm + G::Q_BYTES + G::GROUP_BYTES);   // [NB][NQ]
    uint32_t *ckey = hist + NB * NQ;                                           // [CAP][NQ]
    uint16_t *cidx = reinterpret_cast<uint16_t *>(ckey + CAP * NQ);            // [CAP][NQ]
    uint32_t *mk = reinterpret_cast<uint32_t *>(sm + G::front_bytes(one_panel_launch));   // [words][NQ] chosen blocks
    uint32_t *tie = mk + words * NQ;                                           // [words][NQ] equal scores at the threshold
    uint32_t *part_a = tie + words * NQ, *part_b = part_a + 4 * NQ, *part_c = part_b + 4 * NQ;    // [4][NQ] each
    int32_t *s_tb = reinterpret_cast<int32_t *>(part_c + 4 * NQ), *s_need = s_tb + NQ, *s_cnt = s_need + NQ;
    uint32_t *s_klo = reinterpret_cast<uint32_t *>(s_cnt + NQ), *s_khi = s_klo + NQ, *s_n = s_khi + NQ;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ql = (warp & 3) * 32 + lane, part = warp >> 2;                   // this thread's query and quarter of the words
    const int bh = blockIdx.x, b = bh / H, h = bh % H;
    const int64_t t0 = (int64_t)(gridDim.y - 1 - blockIdx.y) * NQ, t = t0 + ql;
    const int own = (int)(t / block), own_last = (int)((min(t0 + NQ, len) - 1) / block), own_first = (int)(t0 / block);
    const int want = K - 2;                                                    // beside the first block and the query's own
    const bool active = t < len && K < own + 1;                                // otherwise everything up to the query is taken
    const int c_hi = active ? own : 0;                                         // candidates: blocks 1 .. c_hi - 1
    const bool any = K < own_last + 1;                                         // some query of the CTA has to choose
    const int groups = any ? (own_last + kRouteGroup - 1) / kRouteGroup : 0;   // groups that hold blocks 0 .. own_last - 1
    const int panels = (groups + kPanelGroups - 1) / kPanelGroups;
    const int words_cta = any ? (own_last + 31) / 32 : 0;
    uint32_t tcols = kRouteGroup;
    while ((int)tcols < min(groups, kPanelGroups) * kRouteGroup) tcols *= 2;

    for (int i = tid; i < 2 * words * NQ; i += kRouteThreads) mk[i] = 0u;      // mk and tie
    if (part == 0) {
        s_tb[ql] = NB; s_need[ql] = 0; s_cnt[ql] = 0;
        s_klo[ql] = 0u; s_khi[ql] = 0xffffffffu; s_n[ql] = 0u;
    }
    bool ok = true;
    if (any) {
        if (tid == 0) {
            mbar_init(&done, 1);
            mbar_init(&full_q, 1);
            mbar_init_fence();
        }
        if (warp == 0) tmem_alloc(&tbase, tcols);
        tcgen05_before_sync();
        __syncthreads();
        tcgen05_after_sync();
        if (warp == 0) {                                                       // the queries; rows past the prompt come as zeros
            mbar_expect_warp(&full_q, G::Q_BYTES);
#pragma unroll
            for (int hf = 0; hf < G::HALVES; ++hf) tma_load_4d(qs + hf * (NQ * 128), &qmap, hf * 64, h, (int)t0, b, &full_q);
        }
        grid_dependency_wait();                                                // the representatives come from the kernel before
        const uint32_t tb = __shfl_sync(FULL, tbase, 0), tl = tb + ((uint32_t)((warp & 3) * 32) << 16);
        int used = 0;                                                          // products started

        // the scores of panel p into tensor memory, 64 blocks at a time: all threads cut representatives into terms, the
        // first warp starts the products (the whole warp, see rq_umma.cuh)
        constexpr int PER = kRouteGroup * D / 4 / kRouteThreads;               // float4 of a thread
        auto rest = [](float x, float term) { return fabsf(term) == CUDART_INF_F ? 0.0f : x - term; };     // of an infinite mean: nothing
        auto panel = [&](int p) {
            const int g0 = p * kPanelGroups, gn = min(kPanelGroups, groups - g0);
            float4 f[PER];
            auto load = [&](int g) {
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    const int e = tid + i * kRouteThreads, j = g * kRouteGroup + e / (D / 4);
                    f[i] = j < nb ? __ldcg(reinterpret_cast<const float4 *>(means + ((int64_t)bh * nb + j) * D) + e % (D / 4))
                                  : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
            };
            load(g0);
#pragma unroll 1
            for (int g = 0; g < gn; ++g) {
                if (used > 0) ok = ok && mbar_wait(&done, (uint32_t)((used - 1) & 1));     // the product before has read its terms
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    const int e = tid + i * kRouteThreads, r = e / (D / 4), c = 4 * (e % (D / 4));
                    unsigned char *dst = bs + (c >> 6) * (kRouteGroup * 128) + umma_sw128_offset(r, (c & 63) >> 3) + (c & 7) * 2;
                    float4 x = f[i];
#pragma unroll
                    for (int t = 0; t < 3; ++t) {                              // the remainders are exact: each term takes the next 8 bits
                        const uint2 w = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
                        *reinterpret_cast<uint2 *>(dst + t * G::PLANE_BYTES) = w;
                        x = make_float4(rest(x.x, bf16lo(w.x)), rest(x.y, bf16hi(w.x)), rest(x.z, bf16lo(w.y)), rest(x.w, bf16hi(w.y)));
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // ordinary stores, read by the tensor core
                if (g + 1 < gn) load(g0 + g + 1);
                ok = __syncthreads_and(ok);
                if (!ok) break;
                if (warp == 0) {
                    constexpr uint32_t idesc = umma_idesc_bf16(NQ, kRouteGroup);
                    const uint64_t qd = umma_desc_sw128(smem_addr(qs)), bd = umma_desc_sw128(smem_addr(bs));
                    if (used == 0) ok = __all_sync(FULL, mbar_wait(&full_q, 0u) || mbar_wait(&full_q, 0u));
                    tcgen05_after_sync();
#pragma unroll
                    for (int pl = 2; pl >= 0; --pl)                            // the smallest terms first
#pragma unroll
                        for (int hf = 0; hf < G::HALVES; ++hf)
                            umma_bf16_x4<2, 2>(tb + (uint32_t)g * kRouteGroup, qd + (uint64_t)((hf * (NQ * 128)) >> 4),
                                               bd + (uint64_t)((pl * G::PLANE_BYTES + hf * (kRouteGroup * 128)) >> 4), idesc, !(pl == 2 && hf == 0));
                    umma_commit(&done);
                }
                ++used;
            }
            ok = ok && mbar_wait(&done, (uint32_t)((used - 1) & 1));
            ok = __syncthreads_and(ok);
            tcgen05_after_sync();
        };
        // body(word, its first column taken, scores, candidates among them as bits) for this thread's words of every panel
        auto for_scores = [&](bool first, auto body) {
            for (int p = 0; p < panels && ok; ++p) {
                if (first || panels > 1) panel(p);
                if (!ok) break;
                if constexpr (HALF) {
                    if ((part >> 1) < words_cta) {
                        uint32_t x[16];
                        float v[16];
                        tmem_ld16(tl + (uint32_t)part * 16u, x);
#pragma unroll
                        for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(x[c]);
                        const int hi = c_hi - 16 * part;
                        uint32_t cand = hi >= 16 ? 0xffffu : hi <= 0 ? 0u : (1u << hi) - 1u;
                        if (part == 0) cand &= ~1u;
                        body(part >> 1, (part & 1) * 16, v, cand);
                    }
                } else
#pragma unroll 1
                for (int wl = part; wl < 2 * kPanelGroups; wl += 4) {
                    const int w = p * 2 * kPanelGroups + wl;
                    if (w >= words_cta) break;
                    float v[32];
                    __syncwarp();
                    tmem_ld32(tl + (uint32_t)wl * 32u, v);
                    const int hi = c_hi - 32 * w;
                    uint32_t cand = hi >= 32 ? 0xffffffffu : hi <= 0 ? 0u : (1u << hi) - 1u;
                    if (w == 0) cand &= ~1u;
                    body(w, 0, v, cand);
                }
                tcgen05_before_sync();
                if (panels > 1) __syncthreads();                               // the scores may be overwritten
            }
        };
        // the bucket that holds the want-th largest of a query's counted scores: thread `part` of the query adds up a
        // quarter of the buckets, the one whose quarter holds the threshold walks it
        auto find_bin = [&](bool mine, int wanted, int &bin, int &need, int &cnt) -> bool {
            uint32_t s = 0u;
#pragma unroll
            for (int i = 0; i < NB / 4; ++i) s += hist[(part * (NB / 4) + i) * NQ + ql];
            part_c[part * NQ + ql] = s;
            __syncthreads();
            int cum = 0, pt = 3;
            for (; pt > 0; --pt) {
                const int c = (int)part_c[pt * NQ + ql];
                if (cum + c >= wanted) break;
                cum += c;
            }
            if (!mine || part != pt) return false;
            int i = NB / 4 - 1;
            for (; i > 0; --i) {
                const int c = (int)hist[(pt * (NB / 4) + i) * NQ + ql];
                if (cum + c >= wanted) break;
                cum += c;
            }
            bin = pt * (NB / 4) + i;
            cnt = (int)hist[bin * NQ + ql];
            need = wanted - cum;
            return true;
        };

        // ---- 1. smallest and largest
        float mn = CUDART_INF_F, mx = -CUDART_INF_F;
        constexpr int N = HALF ? 16 : 32;                                      // scores taken at a time
        for_scores(true, [&](int w, int c0, float (&v)[N], uint32_t cand) {
            if (w + c0 > 0 && 32 * w + c0 + N <= own_first && own_first >= K) {         // every score is a candidate of every query
#pragma unroll
                for (int c = 0; c < N; ++c) { mn = fminf(mn, v[c]); mx = fmaxf(mx, v[c]); }
            } else {
#pragma unroll
                for (int c = 0; c < N; ++c)
                    if ((cand >> c) & 1u) { mn = fminf(mn, v[c]); mx = fmaxf(mx, v[c]); }
            }
        });
        if (ok) {
            part_a[part * NQ + ql] = __float_as_uint(mn);
            part_b[part * NQ + ql] = __float_as_uint(mx);
            for (int i = tid; i < NB * NQ; i += kRouteThreads) hist[i] = 0u;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                mn = fminf(mn, __uint_as_float(part_a[i * NQ + ql]));
                mx = fmaxf(mx, __uint_as_float(part_b[i * NQ + ql]));
            }
        }
        const float range = mx - mn;
        const float inv = range > 0.0f ? fminf((float)(NB - 3) / range, 3.0e38f) : 0.0f;

        // ---- 2. buckets
        for_scores(false, [&](int, int, float (&v)[N], uint32_t cand) {
#pragma unroll
            for (int c = 0; c < N; ++c)
                if ((cand >> c) & 1u) atomicAdd(&hist[score_bin(v[c], mn, inv) * NQ + ql], 1u);
        });
        if (ok) {
            __syncthreads();
            int bin, need, cnt;
            if (find_bin(active, want, bin, need, cnt)) {
                if (need == cnt) { bin -= 1; need = 0; }                       // the whole bucket
                s_tb[ql] = bin; s_need[ql] = need; s_cnt[ql] = cnt;
            }
            __syncthreads();
        }
        // ---- 2b. (rare) a threshold bucket with too many blocks: buckets on the integer images of its scores
        bool tied = false;
        while (ok) {
            const int tbin = s_tb[ql];
            const uint32_t klo = s_klo[ql], khi = s_khi[ql];
            bool over = active && s_need[ql] > 0 && s_cnt[ql] > CAP && !tied;
            if (over && klo == khi) { tied = true; over = false; }             // all equal: the lowest blocks are taken below
            if (!__syncthreads_or(over)) break;
            uint32_t kmin = 0xffffffffu, kmax = 0u;
            for_scores(false, [&](int, int, float (&v)[N], uint32_t cand) {
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    const uint32_t k = score_key(v[c]);
                    if (over && ((cand >> c) & 1u) && (int)score_bin(v[c], mn, inv) == tbin && k >= klo && k <= khi) {
                        kmin = min(kmin, k);
                        kmax = max(kmax, k);
                    }
                }
            });
            if (!ok) break;
            part_a[part * NQ + ql] = kmin;
            part_b[part * NQ + ql] = kmax;
            for (int i = tid; i < NB * NQ; i += kRouteThreads) hist[i] = 0u;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                kmin = min(kmin, part_a[i * NQ + ql]);
                kmax = max(kmax, part_b[i * NQ + ql]);
            }
            const uint32_t span = over ? kmax - kmin : 0u;
            const int sh = max(0, 26 - __clz((int)span));                      // (span >> sh) < 64
            for_scores(false, [&](int, int, float (&v)[N], uint32_t cand) {
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    const uint32_t k = score_key(v[c]);
                    if (over && ((cand >> c) & 1u) && (int)score_bin(v[c], mn, inv) == tbin && k >= kmin && k <= kmax)
                        atomicAdd(&hist[((k - kmin) >> sh) * NQ + ql], 1u);
                }
            });
            if (!ok) break;
            __syncthreads();
            int bin, need, cnt;
            const bool got = find_bin(over, over ? s_need[ql] : 1, bin, need, cnt);
            __syncthreads();
            if (got) {
                const uint32_t lo = kmin + ((uint32_t)bin << sh), hi = lo + min(kmax - lo, (1u << sh) - 1u);
                if (need == cnt) { s_khi[ql] = lo - 1u; need = 0; }            // everything from lo upwards
                else { s_klo[ql] = lo; s_khi[ql] = hi; }
                s_need[ql] = need; s_cnt[ql] = cnt;
            }
            __syncthreads();
        }
        // ---- 3. the mask
        if (ok) {
            const int tbin = s_tb[ql], need = s_need[ql];
            const uint32_t klo = s_klo[ql], khi = s_khi[ql];
            const bool refined = klo != 0u || khi != 0xffffffffu || tied;
            auto put = [&](uint32_t *words_of, int w, int c0, uint32_t x) {
                if constexpr (HALF) reinterpret_cast<uint16_t *>(words_of)[(w * NQ + ql) * 2 + (c0 >> 4)] = (uint16_t)x;
                else words_of[w * NQ + ql] = x;
            };
            for_scores(false, [&](int w, int c0, float (&v)[N], uint32_t cand) {
                uint32_t bits = 0u, eq = 0u;
                if (!__any_sync(FULL, refined)) {
                    // one atomic per thread and word: one per candidate, each waited for while most lanes had none, took
                    // half of a CTA's time
#pragma unroll
                    for (int c = 0; c < N; ++c) {
                        const int bin = (int)score_bin(v[c], mn, inv);
                        if (bin > tbin) bits |= 1u << c;
                        if (bin == tbin) eq |= 1u << c;
                    }
                    put(mk, w, c0, bits & cand);
                    eq = need > 0 ? eq & cand : 0u;
                    if (!__any_sync(FULL, eq != 0u)) return;
                    uint32_t at = eq ? atomicAdd(&s_n[ql], (uint32_t)__popc(eq)) : (uint32_t)CAP;
#pragma unroll
                    for (int c = 0; c < N; ++c)
                        if (((eq >> c) & 1u) && at < (uint32_t)CAP) {
                            ckey[at * NQ + ql] = score_key(v[c]);
                            cidx[at * NQ + ql] = (uint16_t)(32 * w + c0 + c);
                            ++at;
                        }
                    return;
                }
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    const int bin = (int)score_bin(v[c], mn, inv);
                    if (bin > tbin) bits |= 1u << c;
                    if (bin == tbin && ((cand >> c) & 1u)) {
                        const uint32_t k = score_key(v[c]);
                        if (k > khi) {
                            bits |= 1u << c;
                        } else if (k >= klo && need > 0) {
                            if (tied) {
                                eq |= 1u << c;
                            } else {
                                const uint32_t at = atomicAdd(&s_n[ql], 1u);
                                if (at < (uint32_t)CAP) {
                                    ckey[at * NQ + ql] = k;
                                    cidx[at * NQ + ql] = (uint16_t)(32 * w + c0 + c);
                                }
                            }
                        }
                    }
                }
                put(mk, w, c0, bits & cand);
                if (tied) put(tie, w, c0, eq);
            });
            __syncthreads();
            if (active && need > 0) {
                if (tied) {
                    if (part == 0) {
                        int left = need;
                        for (int w = 0; w < words_cta && left > 0; ++w) {
                            uint32_t e = tie[w * NQ + ql], take = 0u;
                            while (e && left > 0) { take |= e & (0u - e); e &= e - 1u; --left; }
                            mk[w * NQ + ql] |= take;
                        }
                    }
                } else {
                    const int n = min((int)s_n[ql], CAP);
                    for (int i = part; i < n; i += 4) {
                        const uint32_t k = ckey[i * NQ + ql];
                        const int j = cidx[i * NQ + ql];
                        int rank = 0;
                        for (int u = 0; u < n; ++u) {
                            const uint32_t ku = ckey[u * NQ + ql];
                            rank += (ku > k || (ku == k && (int)cidx[u * NQ + ql] < j)) ? 1 : 0;
                        }
                        if (rank < need) atomicOr(&mk[(j >> 5) * NQ + ql], 1u << (j & 31));
                    }
                }
            }
        }
        tcgen05_before_sync();
        __syncthreads();
        if (warp == 0) tmem_dealloc(tbase, tcols);
    }
    if (!ok && tid == 0) atomicCAS(status, RQ_OK, RQ_ERR_TIMEOUT);
    grid_dependency_wait();
    grid_launch_dependents();
    __syncthreads();
    // the masks go out, with the first block and the query's own
    for (int i = tid; i < NQ * words; i += kRouteThreads) {
        const int r = i / words, w = i % words;
        const int64_t tq = t0 + r;
        if (tq >= len) continue;
        const int o = (int)(tq / block), hi = o + 1 - 32 * w;
        uint32_t m;
        if (K >= o + 1) m = hi >= 32 ? 0xffffffffu : hi <= 0 ? 0u : (1u << hi) - 1u;
        else m = mk[w * NQ + r] | (w == 0 ? 1u : 0u) | (w == (o >> 5) ? 1u << (o & 31) : 0u);
        if (masks) masks[((int64_t)bh * len + t0) * words + i] = m;
        if (list) mk[w * NQ + r] = m;
    }
    if (!list) return;
    __syncthreads();
    // the ascending lists for the caller, a warp per query
    for (int r = warp; r < NQ && t0 + r < len; r += kRouteThreads / 32) {
        int32_t *out = list + ((int64_t)bh * len + t0 + r) * K;
        int base = 0;
        for (int w0 = 0; w0 < words; w0 += 32) {
            const uint32_t m = w0 + lane < words ? mk[(w0 + lane) * NQ + r] : 0u;
            const int cnt = __popc(m);
            int inc = cnt;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(FULL, inc, off);
                if (lane >= off) inc += o;
            }
            int pos = base + inc - cnt;
            for (uint32_t bits = m; bits; bits &= bits - 1u, ++pos)
                if (pos < K) out[pos] = (w0 + lane) * 32 + __ffs(bits) - 1;
            base += __shfl_sync(FULL, inc, 31);
        }
        for (int i = base + lane; i < K; i += 32) out[i] = -1;
    }
}

template <int D> cudaError_t route_run(const MobaArgs &a, cudaStream_t s)
{
    using G = RouteGeom<D>;
    const int BH = a.B * a.H, nb = (int)((a.len + a.block - 1) / a.block), words = (nb + 31) / 32;
    const int groups = (nb + kRouteGroup - 1) / kRouteGroup;
    const bool one_panel = groups <= kPanelGroups;
    const bool half = words <= 2;
    static bool ready[2][64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const auto kernel = half ? moba_route_mma_kernel<D, true> : moba_route_mma_kernel<D, false>;
    if (!ready[half][dev]) {
        const int one = G::smem_bytes(true, kPanelGroups * kRouteGroup / 32), more = G::smem_bytes(false, kMobaMaxBlocks / 32);
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, half ? G::smem_bytes(true, 2) : one > more ? one : more);
        if (e != cudaSuccess) return e;
        ready[half][dev] = true;
    }
    const int per = 256 / (D / 2);
    moba_means_bf16_kernel<<<dim3((unsigned)((nb + per - 1) / per), (unsigned)BH), 256, 0, s>>>(
        (const bf16 *)a.kv, a.page_cap, a.S, D, a.len, a.block, a.means, nb);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    alignas(64) CUtensorMap qmap;
    e = query_tensor_map(&qmap, a.q, D, a.H, a.len, a.B, kRouteQueries);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)BH, (unsigned)((a.len + kRouteQueries - 1) / kRouteQueries));
    cfg.blockDim = dim3(kRouteThreads);
    cfg.dynamicSmemBytes = (size_t)G::smem_bytes(one_panel, words);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, qmap, (const float *)a.means, a.len, a.H, a.block, nb, a.K, words, a.masks,
                              a.list, a.status);
}

}  // namespace

cudaError_t launch_moba_route_bf16(const MobaArgs &a, cudaStream_t s)
{
    return a.D == 128 ? route_run<128>(a, s) : a.D == 64 ? route_run<64>(a, s) : cudaErrorInvalidValue;
}

}  // namespace rq
