// MoBA attention for bf16 caches (Sec. 2.2, Eq. 4; App. A.1, MoBA paragraph): softmax attention of every prompt
// position over the positions up to its own of the blocks it chose, both contractions on the tensor cores (tcgen05).
#include <math_constants.h>

#include <algorithm>

#include "rq_async.cuh"
#include "rq_device.cuh"
#include "rq_internal.h"
#include "rq_tmap.h"
#include "rq_umma.cuh"

namespace rq {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kChunk = 64;                     // positions of a step
constexpr int kTile = 128;                     // queries of an accumulator (its lanes)
constexpr int kTiles = 2;                      // accumulators of a CTA: 256 consecutive queries share the keys and values
constexpr int kStages = 4;                     // chunks of keys, and of values, in shared memory
constexpr int kReadWarps = 4 * kTiles;         // warps that turn scores into weights: a thread per query
constexpr int kThreads = (kReadWarps + kTiles + 2) * 32;   // and one for the copies, two for the score products, one for the output products
// Heads are worked on in sets of up to kSetBytes of keys and values, which stay in L2 while the set's CTAs walk over them; the set
// that is not full comes first, so that no few heads' longest walks are left for the end.  Call, us, one set / sets, 128 channels:
// 32 heads x 30011 positions (492 MB) 7457 / 7027, 33 heads 7628 / 7251 (the smaller set last 7689), 27 x 20000 (276 MB) 2768 / 2711,
// 17 x 30011 (261 MB) 3800 / 3703, 320 x 9486 (1.55 GB) 10266 / 9212, 320 x 3001 (492 MB) 1335 / 1275, 20 x 20000 (205 MB) 2052 / 1997,
// 30 x 9001 (138 MB) 682 / 678; just above one set 14 x 14500 709 / 717, 7 x 30000 1498 / 1497, 50 x 4096 336 / 334.  Of 64
// channels, whose walks the readers bound, within 1 % of each other from 102 to 737 MB.  Sets of 32 MB win less (33 heads 7224 when
// sets of 64 and of 96 MB take 7198 and 7176; 16 x 14001 827, 764, 770).
constexpr int64_t kSetBytes = 96 << 20;
constexpr float kRaise = 8.0f;                 // powers of two a query's maximum may grow before its output is rescaled

template <int D> struct AttGeom {
    static constexpr int HALVES = D / 64;
    static constexpr int Q_BYTES = HALVES * kTile * 128;           // the queries of one accumulator
    static constexpr int C_BYTES = HALVES * kChunk * 128;          // the keys (or the values) of a chunk
    static constexpr int OFF_K = kTiles * Q_BYTES;
    static constexpr int OFF_V = OFF_K + kStages * C_BYTES;
    static constexpr int OFF_LIST = OFF_V + kStages * C_BYTES;     // blocks to walk
    static constexpr int SMEM_BYTES = OFF_LIST + kMobaMaxBlocks * 2 + 1024;   // + room to align the base to 1024 bytes
};

__device__ __forceinline__ uint64_t desc_sw128_mn(uint32_t saddr, uint32_t lbo_bytes)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}
__device__ __forceinline__ float exp2_fast(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// the larger one; NaN if one is NaN
__device__ __forceinline__ float max_nan(float a, float b)
{
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}

// two bf16 added to a sum each (their values are exact in fp32)
__device__ __forceinline__ void add_bf16(float2 &sum, uint32_t pair)
{
    asm("{\n\t.reg .b16 lo, hi;\n\t"
        "mov.b32 {lo, hi}, %2;\n\t"
        "add.rn.f32.bf16 %0, lo, %0;\n\t"
        "add.rn.f32.bf16 %1, hi, %1;\n\t}"
        : "+f"(sum.x), "+f"(sum.y)
        : "r"(pair));
}

// The walk over the chunks of the listed blocks: (entry of the list, chunk inside the block).
struct Walk {
    int bi = 0, r = 0;
    __device__ __forceinline__ void next(int cpb)
    {
        if (++r == cpb) { r = 0; ++bi; }
    }
};

// Grid: tiles of 256 queries of all heads, the last queries of a head first (their work is the largest).  A CTA owns 256
// consecutive queries as two accumulators of 128 lanes; everything per query (choice of blocks, causal cut, what its weights
// are relative to, their sum, the weights) belongs to one thread.  The 64-position chunks of the blocks that any of the 256
// queries chose are walked once:
//   S = Q K^T        128 x 64 per accumulator, fp32 in tensor memory, two score buffers per accumulator, so that the
//                    product of the next chunk runs while the weights of this one are computed
//   weights          2^(s - m) for the chosen blocks' positions up to the query's own, rounded to bf16, written over
//                    the first half of their scores as the A operand of the second product; the rounded weights are
//                    summed in fp32
//   O += P V         accumulated in tensor memory over all chunks
// m is the query's largest score so far, but it is raised (and the query's row of O multiplied down) only when a score
// exceeds it by more than 8 powers of two: weights of up to 256 lose nothing in bf16 and fp32, and the output is divided
// by their sum at the end.  The sum is that of the rounded weights: relative to a lagging maximum the largest weight is not 1
// exactly, and its rounding would be an error of the whole output; so it cancels.  Error against fp64 (2-norm; 4096 positions,
// 16 of 64 blocks, plain keys, logits of 1.5 / 5 / 15): 2.142e-3 / 1.799e-3 / 1.509e-3.  The more queries end with an m that is not
// their maximum, the larger it is: with the first chunk's maximum kept until a chunk's weights add up to more than 2^32, 0 / 1.4 /
// 0.8 % more, and values above 2^92 overflow.  The first keys of a prompt have hardly been accumulated and score low, so that a fifth
// to a half of a warp's chunks raise one of its queries; the row of O is therefore multiplied down after the chunk's weights have
// been written, when the product before is mostly over, 32 columns at a time with the next 32 on their way.
// Warps 0..7 read scores, warp 8 starts the tensor-map copies, warps 9 and 10 the score products of an accumulator each,
// warp 11 the output products; they meet through mbarriers only, every wait bounded.  256 queries per CTA because keys and
// values come from L2 for every CTA.  A CTA's queries come by tensor map, and it may start before the routing kernel has ended.
// Measured, call, 32 heads x 128 channels, 4096 positions (16 of 64 blocks) at logits of 1.4 / 5 / 11: rows multiplied down before
// the weights, 16 columns at a time, 223.5 / 238 / 243 us; after them 217 / 227 / 231 (without ever doing it 214).  Bound: the
// readers' chain per chunk (about 1850 cycles at 4096 positions, of which ex2 alone takes 1024, against 1280 for the products, whose
// operands take shared memory's bandwidth); at 30011 positions the power limit as well.  Slower: weights taken before the maximum is known and again where it
// was too far off (251 us; by halves of a chunk 240); the next chunk's scores loaded while the weights are handed over; queries as
// columns, so that weights are taken only for eights or sixteens of queries some of which chose the chunk (236 us / 7.1 ms at 30011);
// and only the queries that chose a chunk gathered for it (377 us / 9.6 ms: lists, gathers and scattered weights cost more than
// the products they save).
template <int D>
__global__ void __launch_bounds__(kThreads, 1) moba_mma_kernel(const __grid_constant__ CUtensorMap tmap,
                                                               const __grid_constant__ CUtensorMap qmap,
                                                               const __grid_constant__ CUtensorMap omap, int64_t page_cap, int S,
                                                               int64_t len, int H, int BH, int set, int tiles, int block, int nb,
                                                               const uint32_t *masks, const int32_t *lists, int K, float scale_log2, int32_t *status)
{
    using G = AttGeom<D>;
    constexpr int NST = kStages;
    // tensor memory of accumulator s: columns s * 256: two score buffers of 64 columns (their first 32 hold the weights
    // afterwards), then the output
    constexpr uint32_t ACC = 256, OFF_O = 128;
    extern __shared__ __align__(1024) unsigned char asm_raw[];
    __shared__ __align__(8) uint64_t full_k[NST], full_v[NST], free_k[NST], free_v[NST], full_q;
    __shared__ __align__(8) uint64_t s_ready[kTiles][2], p_ready[kTiles][2], pv_done[kTiles][2];
    __shared__ uint32_t um[kTiles][kMobaMaxBlocks / 32];         // blocks chosen by any query of an accumulator
    __shared__ uint32_t tbase;
    __shared__ int n_list;
    unsigned char *sm = asm_raw + ((1024u - (smem_addr(asm_raw) & 1023u)) & 1023u);
    unsigned char *qs = sm, *kst = sm + G::OFF_K, *vst = sm + G::OFF_V;
    uint16_t *list = reinterpret_cast<uint16_t *>(sm + G::OFF_LIST);   // block | 0x4000 (first accumulator) | 0x8000 (second)
    const int words = (nb + 31) / 32;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int part = BH % set;                                   // heads of the first set, if it is not full
    const int at_tile = (int)blockIdx.x - part * tiles;
    const int first = at_tile < 0 ? 0 : part + at_tile / (set * tiles) * set, in_set = at_tile < 0 ? part : set;
    const int rest = at_tile < 0 ? (int)blockIdx.x : at_tile % (set * tiles);
    const int bh = first + rest % in_set, b = bh / H, h = bh % H;
    const int64_t t0 = (int64_t)(tiles - 1 - rest / in_set) * (kTile * kTiles);
    const int n_chunks_all = (int)((min(t0 + kTile * kTiles, len) + kChunk - 1) / kChunk);
    const int cpb = block / kChunk;                              // chunks of a block
    const int ppc = kChunk / S;                                  // pages of a chunk

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            mbar_init(&full_k[i], 1); mbar_init(&full_v[i], 1);
            mbar_init(&free_k[i], kTiles); mbar_init(&free_v[i], 1);
        }
        mbar_init(&full_q, 1);
        for (int s = 0; s < kTiles; ++s)
            for (int i = 0; i < 2; ++i) {
                mbar_init(&s_ready[s][i], 1);
                mbar_init(&p_ready[s][i], kTile);
                mbar_init(&pv_done[s][i], 1);
            }
        mbar_init_fence();
    }
    if (warp == kReadWarps) tmem_alloc(&tbase, 512);
    for (int i = tid; i < kTiles * words; i += kThreads) um[i / words][i % words] = 0u;
    __syncthreads();
    if (warp == kReadWarps) {                                    // the queries; rows past the prompt come as zeros
        mbar_expect_warp(&full_q, kTiles * G::Q_BYTES);
#pragma unroll
        for (int s = 0; s < kTiles; ++s)
#pragma unroll
            for (int hf = 0; hf < G::HALVES; ++hf)
                tma_load_4d(qs + s * G::Q_BYTES + hf * (kTile * 128), &qmap, hf * 64, h, (int)t0 + s * kTile, b, &full_q);
    }
    grid_dependency_wait();                                      // the choices of blocks come from the kernel before
    if (warp < kReadWarps) {
        const bool in = t0 + tid < len;
        if (masks) {
            const uint32_t *row = masks + ((int64_t)bh * len + (in ? t0 + tid : 0)) * words;
            for (int w0 = 0; w0 < words; w0 += 8) {              // eight loads in flight
                uint32_t m[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) m[u] = in && w0 + u < words ? __ldcg(row + w0 + u) : 0u;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    m[u] = __reduce_or_sync(FULL, m[u]);
                    if (lane == 0 && m[u]) atomicOr(&um[warp >> 2][w0 + u], m[u]);
                }
            }
        } else if (in) {
            const int32_t *mine = lists + ((int64_t)bh * len + t0 + tid) * K;
            for (int i = 0; i < K; ++i) {
                const int j = __ldcg(mine + i);
                if (j >= 0) atomicOr(&um[warp >> 2][j >> 5], 1u << (j & 31));
            }
        }
    }
    __syncthreads();
    if (warp == 0) {                                             // the list of blocks, ascending
        int base = 0;
#pragma unroll 4
        for (int w = 0; w < words; ++w) {                        // a lane per block
            const uint32_t m0 = um[0][w], m1 = um[1][w], m = m0 | m1;
            if ((m >> lane) & 1u)
                list[base + __popc(m & ((1u << lane) - 1u))] =
                    (uint16_t)((w * 32 + lane) | (((m0 >> lane) & 1u) << 14) | (((m1 >> lane) & 1u) << 15));
            base += __popc(m);
        }
        if (lane == 0) n_list = base;
    }
    tcgen05_before_sync();
    __syncthreads();
    tcgen05_after_sync();
    const uint32_t tb = __shfl_sync(FULL, tbase, 0);             // (the shuffle tells the compiler that it is uniform)
    // steps of the walk: whole blocks, the last one (the last query's own) up to the CTA's last chunk
    const int nl = n_list, n = (nl - 1) * cpb + min(cpb, n_chunks_all - (list[nl - 1] & 0x3fff) * cpb);
    bool ok = true;

    if (warp == kReadWarps) {
        // ---- copies (the whole warp, like the products below: see rq_umma.cuh)
        {
            Walk w;
            int issued = 0;
#pragma unroll 1
            for (int i = 0; i < n; ++i, w.next(cpb)) {
                const int st = i % NST;
                if (i >= NST) {
                    const uint32_t ph = (uint32_t)((i / NST - 1) & 1);
                    ok = mbar_wait(&free_k[st], ph) && mbar_wait(&free_v[st], ph);
                    ok = __all_sync(FULL, ok);
                    if (!ok) break;
                }
                const int page = (int)((int64_t)bh * page_cap + (int64_t)(__shfl_sync(FULL, list[w.bi] & 0x3fff, 0) * cpb + w.r) * ppc);
                mbar_expect_warp(&full_k[st], G::C_BYTES);
#pragma unroll
                for (int hf = 0; hf < G::HALVES; ++hf)
                    tma_load_4d(kst + (size_t)st * G::C_BYTES + hf * (kChunk * 128), &tmap, hf * 64, 0, 0, page, &full_k[st]);
                mbar_expect_warp(&full_v[st], G::C_BYTES);
#pragma unroll
                for (int hf = 0; hf < G::HALVES; ++hf)
                    tma_load_4d(vst + (size_t)st * G::C_BYTES + hf * (kChunk * 128), &tmap, hf * 64, 0, 1, page, &full_v[st]);
                issued = i + 1;
            }
            // no copy may still be on its way into this CTA's shared memory when it exits, after a wait that ran out either
            ok = mbar_wait(&full_q, 0u) && ok;
            if (!ok)
                for (int k = max(0, issued - NST); k < issued; ++k) {
                    mbar_wait(&full_k[k % NST], (uint32_t)((k / NST) & 1));
                    mbar_wait(&full_v[k % NST], (uint32_t)((k / NST) & 1));
                }
        }
    } else if (warp > kReadWarps && warp <= kReadWarps + kTiles) {
        // ---- score products, a warp per accumulator
        const int s = warp - kReadWarps - 1;
        constexpr uint32_t idesc_s = umma_idesc_bf16(kTile, kChunk);
        const uint64_t qd = umma_desc_sw128(smem_addr(qs) + s * G::Q_BYTES), kd = umma_desc_sw128(smem_addr(kst));
        const uint32_t ts = tb + s * ACC;
        int u = 0;                                               // products started
        Walk w;
        ok = __all_sync(FULL, mbar_wait(&full_q, 0u));
#pragma unroll 1
        for (int i = 0; i < n && ok; ++i, w.next(cpb)) {
            const int st = i % NST;
            // (waited for even if not used: the stage's release counts one arrival of each of the two warps per filling)
            ok = __all_sync(FULL, mbar_wait(&full_k[st], (uint32_t)((i / NST) & 1)));
            if (!ok) break;
            if ((__shfl_sync(FULL, (uint32_t)list[w.bi], 0) >> (14 + s)) & 1u) {
                if (u >= 2) ok = mbar_wait(&pv_done[s][u & 1], (uint32_t)(((u >> 1) - 1) & 1));   // the buffer's weights were used
                ok = __all_sync(FULL, ok);
                if (!ok) break;
                tcgen05_after_sync();
#pragma unroll
                for (int hf = 0; hf < G::HALVES; ++hf)
                    umma_bf16_x4<2, 2>(ts + (uint32_t)(u & 1) * kChunk, qd + (uint64_t)((hf * (kTile * 128)) >> 4),
                                       kd + (uint64_t)((st * G::C_BYTES + hf * (kChunk * 128)) >> 4), idesc_s, hf > 0);
                umma_commit(&s_ready[s][u & 1]);
                ++u;
            }
            umma_commit(&free_k[st]);
        }
    } else if (warp == kReadWarps + kTiles + 1) {
        // ---- output products
        constexpr uint32_t idesc_o = umma_idesc_bf16(kTile, D) | (1u << 16);       // the values are MN-major
        const uint64_t vd = desc_sw128_mn(smem_addr(vst), kChunk * 128);
        int up[kTiles] = {0, 0};                                 // products started
        Walk w;
#pragma unroll 1
        for (int i = 0; i < n && ok; ++i, w.next(cpb)) {
            const int st = i % NST;
            const uint32_t e = __shfl_sync(FULL, (uint32_t)list[w.bi], 0);
            ok = __all_sync(FULL, mbar_wait(&full_v[st], (uint32_t)((i / NST) & 1)));
#pragma unroll
            for (int s = 0; s < kTiles; ++s) {
                if (!ok || !((e >> (14 + s)) & 1u)) continue;
                const int u = up[s]++;
                ok = __all_sync(FULL, mbar_wait(&p_ready[s][u & 1], (uint32_t)((u >> 1) & 1)));
                if (!ok) continue;
                tcgen05_after_sync();
                umma_bf16_ta_x4<8, 128>(tb + s * ACC + OFF_O, tb + s * ACC + (uint32_t)(u & 1) * kChunk, vd + (uint64_t)((st * G::C_BYTES) >> 4),
                                        idesc_o, u > 0);
                umma_commit(&pv_done[s][u & 1]);
            }
            if (ok) umma_commit(&free_v[st]);
        }
    } else {
        // ---- weights: a thread per query
        const int s = warp >> 2, lq = (warp & 3) * 32 + lane;
        const int64_t tq = t0 + s * kTile + lq;
        const bool in = tq < len;
        const uint32_t tl = tb + s * ACC + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t *row = masks + ((int64_t)bh * len + (in ? tq : 0)) * words;
        uint32_t w_cur = 0u, w_next = 0u;                        // the query's choice of the 32 blocks around the walk, and of the next 32
        int w_at = -1;
        const int32_t *mine = lists + ((int64_t)bh * len + (in ? tq : 0)) * K;
        int at = 0;                                              // without masks: the query's first list entry that is not behind the walk
        float m = -CUDART_INF_F;                                 // what the weights are relative to (scaled, log2)
        float2 l2 = make_float2(0.0f, 0.0f);                     // sums of the weights (even and odd positions)
        const float2 sc2 = make_float2(scale_log2, scale_log2);
        int u = 0;
        Walk wk;
#pragma unroll 1
        for (int i = 0; i < n; ++i, wk.next(cpb)) {
            const uint32_t e = list[wk.bi];
            if (!((e >> (14 + s)) & 1u)) continue;
            const int j = e & 0x3fff;
            bool chosen;
            if (masks) {
                if ((j >> 5) != w_at) {
                    const int w = j >> 5;
                    w_cur = w_at >= 0 && w == w_at + 1 ? w_next : in ? __ldcg(row + w) : 0u;
                    w_next = in && w + 1 < words ? __ldcg(row + w + 1) : 0u;
                    w_at = w;
                }
                chosen = (w_cur >> (j & 31)) & 1u;
            } else {
                while (in && at < K && (uint32_t)__ldcg(mine + at) < (uint32_t)j) ++at;    // (-1: beyond every block)
                chosen = in && at < K && __ldcg(mine + at) == j;
            }
            const int c = j * cpb + wk.r;
            const int64_t p0 = (int64_t)c * kChunk;
            // positions this query attends among the chunk's: none if it did not choose the block, else those up to its own
            int nv = 0;
            if (in && chosen) nv = (int)max((int64_t)0, min((int64_t)kChunk, tq - p0 + 1));
            ok = mbar_wait(&s_ready[s][u & 1], (uint32_t)((u >> 1) & 1));
            if (!__all_sync(FULL, ok)) break;
            tcgen05_after_sync();
            const uint32_t ts = tl + (uint32_t)(u & 1) * kChunk;
            if (__any_sync(FULL, nv > 0)) {
                float v[kChunk];
                tmem_ld64(ts, v);
                const bool cut = __any_sync(FULL, nv > 0 && nv < kChunk);
                if (cut) {
#pragma unroll
                    for (int k = 0; k < kChunk; ++k) v[k] = k < nv ? v[k] : -CUDART_INF_F;
                }
                float tm[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                for (int k = 4; k < kChunk; ++k) tm[k & 3] = max_nan(tm[k & 3], v[k]);
                const float top = max_nan(max_nan(tm[0], tm[1]), max_nan(tm[2], tm[3])) * scale_log2;
                const bool raise = nv > 0 && top > m + kRaise;
                const bool stray = nv == 0 && !(top < CUDART_INF_F);       // infinite or NaN scores of a block the query did not choose
                bool touch = false;
                float f = 1.0f;                                            // what the sum and the query's row of O are multiplied by
                if (__any_sync(FULL, raise || stray)) {
#pragma unroll
                    for (int k = 0; k < kChunk; ++k) v[k] = stray ? -CUDART_INF_F : v[k];
                    touch = raise && m > -CUDART_INF_F;                    // (otherwise the query's row of O is still zero)
                    f = touch ? exp2_fast(m - top) : 1.0f;
                    if (raise) m = top;
                    l2.x *= f;
                    l2.y *= f;
                }
                // a block the query did not choose: 2^-3e38 = 0; nor do scores of -inf weigh anything while there is no other
                const float nm = nv > 0 ? fminf(-m, 3.0e38f) : -3.0e38f;
                const float2 nm2 = make_float2(nm, nm);
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    uint32_t w[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const float2 x = fma2(make_float2(v[hf * 32 + 2 * k], v[hf * 32 + 2 * k + 1]), sc2, nm2);
                        const float2 p = make_float2(exp2_fast(x.x), exp2_fast(x.y));
                        w[k] = pack_bf16(p.x, p.y);
                        add_bf16(l2, w[k]);
                    }
                    tmem_st16(ts + hf * 16, w);
                }
                if (__any_sync(FULL, touch)) {
                    ok = mbar_wait(&pv_done[s][(u - 1) & 1], (uint32_t)(((u - 1) >> 1) & 1));   // nothing is being added to O
                    if (!__all_sync(FULL, ok)) break;
                    tcgen05_after_sync();
                    float x[2][32];
                    tmem_ld32_start(tl + OFF_O, x[0]);
#pragma unroll
                    for (int cb = 0; cb < D / 32; ++cb) {
                        float (&y)[32] = x[cb & 1];
                        tmem_ld32_wait(y);
                        if (cb + 1 < D / 32) tmem_ld32_start(tl + OFF_O + (cb + 1) * 32, x[(cb + 1) & 1]);
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            uint32_t w[16];
#pragma unroll
                            for (int k = 0; k < 16; ++k) w[k] = __float_as_uint(y[hf * 16 + k] * f);
                            tmem_st16(tl + OFF_O + cb * 32 + hf * 16, w);
                        }
                    }
                }
            } else {                                             // none of the warp's queries chose the block
                const uint32_t z[16] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
                tmem_st16(ts, z);
                tmem_st16(ts + 16, z);
            }
            if (p0 + kChunk > len) {
                // the prompt ends inside this chunk: the value rows past its end hold whatever the cache's memory held; a
                // weight of zero would not stop a NaN there, so those rows are cleared once they have landed
                ok = mbar_wait(&full_v[i % NST], (uint32_t)((i / NST) & 1));
                if (!__all_sync(FULL, ok)) break;
                const int r = lq & (kChunk - 1), hf = lq >> 6;
                if (hf < G::HALVES && p0 + r >= len) {
                    uint4 *vrow = reinterpret_cast<uint4 *>(vst + (size_t)(i % NST) * G::C_BYTES + hf * (kChunk * 128) + (r >> 3) * 1024 +
                                                            (r & 7) * 128);
#pragma unroll
                    for (int k = 0; k < 8; ++k) vrow[k] = make_uint4(0u, 0u, 0u, 0u);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // ordinary stores, read by the tensor core
            }
            tmem_st_wait();                                      // the weights are in tensor memory
            tcgen05_before_sync();
            mbar_arrive(&p_ready[s][u & 1]);
            ++u;
        }
        // the output once the last product is complete, divided by the sum of the query's weights
        if (__all_sync(FULL, ok) && u > 0) {
            ok = mbar_wait(&pv_done[s][(u - 1) & 1], (uint32_t)(((u - 1) >> 1) & 1));
            if (__all_sync(FULL, ok)) {
                tcgen05_after_sync();
                const float inv = 1.0f / (l2.x + l2.y);          // (nothing but scores of -inf: NaN; rows past the prompt are not stored)
                // (the accumulator's queries are not read any more: its rows go out through their room, a store per warp and
                // 64 channels; rows past the prompt are cut off by the map)
                unsigned char *os = qs + s * G::Q_BYTES + (warp & 3) * 32 * 128;
#pragma unroll 1
                for (int cb = 0; cb < D; cb += 32) {
                    float v[32];
                    tmem_ld32(tl + OFF_O + cb, v);
#pragma unroll
                    for (int k = 0; k < 32; k += 8)
                        *reinterpret_cast<uint4 *>(os + (cb >> 6) * (kTile * 128) + umma_sw128_offset(lane, ((cb & 63) + k) >> 3)) =
                            make_uint4(pack_bf16(v[k] * inv, v[k + 1] * inv), pack_bf16(v[k + 2] * inv, v[k + 3] * inv),
                                       pack_bf16(v[k + 4] * inv, v[k + 5] * inv), pack_bf16(v[k + 6] * inv, v[k + 7] * inv));
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (tq - lane < len) {
#pragma unroll
                    for (int hf = 0; hf < G::HALVES; ++hf)
                        tma_store_4d(os + hf * (kTile * 128), &omap, hf * 64, h, (int)(tq - lane), b);
                    tma_store_commit();
                    tma_store_wait_read();
                }
            }
        }
    }
    if (__any_sync(FULL, !ok) && lane == 0) atomicCAS(status, RQ_OK, RQ_ERR_TIMEOUT);
    tcgen05_before_sync();
    __syncthreads();
    if (warp == kReadWarps) tmem_dealloc(tbase, 512);
}

template <int D> cudaError_t attend_run(const MobaArgs &a, cudaStream_t s)
{
    using G = AttGeom<D>;
    const int BH = a.B * a.H, nb = (int)((a.len + a.block - 1) / a.block);
    static bool ready[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!ready[dev]) {
        e = cudaFuncSetAttribute(moba_mma_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM_BYTES);
        if (e != cudaSuccess) return e;
        ready[dev] = true;
    }
    alignas(64) CUtensorMap tmap, qmap, omap;
    e = cache_tensor_map(&tmap, a.kv, D, a.S, (int64_t)BH * a.page_cap, kChunk);
    if (e != cudaSuccess) return e;
    e = query_tensor_map(&qmap, a.q, D, a.H, a.len, a.B, kTile);
    if (e != cudaSuccess) return e;
    e = query_tensor_map(&omap, a.o, D, a.H, a.len, a.B, 32);
    if (e != cudaSuccess) return e;
    const int tiles = (int)((a.len + kTile * kTiles - 1) / (kTile * kTiles));
    const int64_t head_bytes = a.len * D * 4;
    const int set = (int)std::max<int64_t>(1, std::min<int64_t>(BH, kSetBytes / head_bytes));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)BH * (unsigned)tiles);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = G::SMEM_BYTES;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, moba_mma_kernel<D>, tmap, qmap, omap, a.page_cap, a.S, a.len, a.H, BH, set, tiles, a.block, nb, (const uint32_t *)a.masks,
                              (const int32_t *)a.list, a.K, a.scale * 1.4426950408889634f, a.status);
}

}  // namespace

cudaError_t launch_moba_attend_bf16(const MobaArgs &a, cudaStream_t s)
{
    return a.D == 128 ? attend_run<128>(a, s) : a.D == 64 ? attend_run<64>(a, s) : cudaErrorInvalidValue;
}

}  // namespace rq
