// MoBA-style block-sparse prefill attention on the cache of decayed keys and values (Sec. 2.2, Eq. 3
// and Eq. 4, Table 1 row MoBA; App. A.1, "Sparse inference settings", MoBA paragraph): every prompt
// position routes its query to a few of the KV blocks before it, scored with mean-pooled block
// representatives, and attends over the chosen blocks only; the first block and the query's own
// block (cut at the query's position) are always among them and count inside the budget.
//
//   rq_moba_route.cu     bf16 caches: the blocks' mean keys and every query's choice of blocks (a bit mask)
//   moba_means_kernel    fp32 caches.  Per (head, block): the mean of the block's stored keys
//   moba_route_kernel    fp32 caches.  Per (head, 16 consecutive queries), a warp per query: scores q . mean of the
//                        complete blocks before the query's own (a lane per block; the head's
//                        representatives staged in shared memory once per CTA when they fit), then the
//                        budget's best (equal scores to the lower block) by a bit-wise search for the
//                        threshold score, or by repeated arg-max when the budget is small or the candidates many;
//                        the list written ascending
//   rq_moba_attend.cu    bf16 caches: the attention on the tensor cores
//   moba_attend_kernel   fp32 caches.  Per (head, 16 consecutive queries), a warp per query: the blocks
//                        any of the 16 queries chose pass through shared memory once, 64 positions at a
//                        time (cp.async, two buffers); a warp folds a chunk into its online softmax
//                        only if its own query chose the block (plain fp32 FMA work; the arithmetic is
//                        the decode path's tile routine)
#include <limits.h>
#include <math_constants.h>

#include "rq_async.cuh"
#include "rq_device.cuh"
#include "rq_internal.h"
#include "rq_stream.cuh"

namespace rq {

namespace {

constexpr int kMobaChunk = 64;                 // positions that pass through shared memory at a time
constexpr int kMobaQueries = 16;               // queries (warps) of one attention CTA
constexpr int kMobaRouteWarps = 16;            // warps of one routing CTA
constexpr int kMobaRouteQ = 2;                 // consecutive queries of one routing warp when the representatives are staged (they share the reads)
constexpr unsigned FULLMASK = 0xffffffffu;

// floats of shared memory one routing warp needs: query, scores, mask words; a multiple of 4 so that
// every warp's query starts on a 16-byte boundary
__host__ __device__ inline int moba_route_floats(int D, int nb) { return (D + nb + (nb + 31) / 32 + 3) & ~3; }

__device__ __forceinline__ void cp_async16(void *dst_smem, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---------------------------------------------------------------- block representatives
// Grid (blocks, heads), a thread per channel; the sum runs over the block's valid positions in order.
template <typename T>
__global__ void moba_means_kernel(const T *kv, int64_t page_cap, int S, int D, int64_t len, int block, float *means, int nb)
{
    const int j = blockIdx.x, bh = blockIdx.y, c = threadIdx.x;
    const int64_t lo = (int64_t)j * block, hi = min(lo + block, len);
    float s = 0.0f;
    int64_t p = lo;
    // sixteen loads in flight at a time (a page holds a multiple of 16 positions and lo is a multiple of 64, so
    // a run of 16 stays inside one page); the additions keep the order of the positions
    for (; p + 16 <= hi; p += 16) {
        const T *src = kv + ((((int64_t)bh * page_cap + p / S) * 2) * S + p % S) * D + c;
        float x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = load1<T>(src + (int64_t)i * D);
#pragma unroll
        for (int i = 0; i < 16; ++i) s += x[i];
    }
    for (; p < hi; ++p) s += load1<T>(kv + ((((int64_t)bh * page_cap + p / S) * 2) * S + p % S) * D + c);
    means[((int64_t)bh * nb + j) * D + c] = s / (float)(hi - lo);
}

// The `want` best of the candidate blocks c_lo .. c_hi - 1 with scores sc[], for one warp; lane l owns the
// candidates c_lo + l + 32 r, r < R.  A candidate beats another with a higher score, or the same score and a lower
// block.  The score of the want-th best is found bit by bit on the order-preserving integer image of the scores
// (32 rounds of one comparison and one vote per owned candidate: far fewer operations than ranking every candidate
// against every other); the candidates above it are taken, and of those equal to it the lowest blocks.  Sets their
// mask bits.
template <int R>
__device__ __forceinline__ void moba_rank_take(const float *sc, uint32_t *mask, int c_lo, int c_hi, int want, int lane)
{
    uint32_t key[R];
    bool valid[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = c_lo + lane + 32 * r;
        valid[r] = j < c_hi;
        const uint32_t b = __float_as_uint((valid[r] ? sc[j] : 0.0f) + 0.0f);     // -0 becomes +0
        key[r] = b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
    }
    // the largest t with at least `want` keys >= t: the want-th largest key (want <= number of candidates)
    uint32_t t = 0u;
#pragma unroll 4
    for (int bit = 31; bit >= 0; --bit) {
        const uint32_t trial = t | (1u << bit);
        int cnt = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) cnt += __popc(__ballot_sync(0xffffffffu, valid[r] && key[r] >= trial));
        if (cnt >= want) t = trial;
    }
    int above = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) above += __popc(__ballot_sync(0xffffffffu, valid[r] && key[r] > t));
    int need = want - above;                         // of the candidates equal to the threshold, in block order
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t eq = __ballot_sync(0xffffffffu, valid[r] && key[r] == t);
        const bool mine = valid[r] && (key[r] > t || (key[r] == t && __popc(eq & lt) < need));
        need = max(0, need - __popc(eq));
        const unsigned take = __ballot_sync(0xffffffffu, mine);          // blocks c_lo + 32 r + bit
        if (lane == 0 && take) {
            const int p = c_lo + 32 * r;
            mask[p >> 5] |= take << (p & 31);
            if (p & 31) mask[(p >> 5) + 1] |= take >> (32 - (p & 31));
        }
    }
}

// ---------------------------------------------------------------- routing
// Grid (ceil(T / queries of a CTA), heads); a warp per query, or per two consecutive queries when the
// representatives are staged (a lane reads a representative once for both).  Shared memory per query: the
// query (D floats), the scores of the candidate blocks (nb floats), the chosen blocks as a bit mask
// (nb / 32 words); and, when they fit (STAGED), the head's representatives for the whole CTA, rows padded
// by four floats so that the lanes of a quarter-warp, each reading its own row, hit different banks.
// q: [B][T][H][D].  sel: [BH][T][K], ascending, -1 beyond the chosen blocks.
constexpr int kMobaStagedBlocks = 128;         // representatives of up to this many blocks are staged in shared memory

// The selection of one query once the scores of its candidate blocks c_lo .. c_hi - 1 are in sc[]: the `want` best
// into the mask, the first block(s) and the own block(s) added, the chosen blocks written ascending.  One warp.
__device__ __forceinline__ void moba_route_finish(const float *sc, uint32_t *mask, int32_t *out, int words, int K, int P, int ns,
                                                  int nl, int c_lo, int c_hi, int want, int lane)
{
    if (c_hi - c_lo <= 4 * 32 && want >= 8) {
        // few candidates and more than a handful to take (a round per taken block is cheaper otherwise): the
        // threshold score by bit-wise search, a lane holding one, two or four candidates
        const int ncand = c_hi - c_lo;
        if (ncand <= 32) moba_rank_take<1>(sc, mask, c_lo, c_hi, want, lane);
        else if (ncand <= 64) moba_rank_take<2>(sc, mask, c_lo, c_hi, want, lane);
        else moba_rank_take<4>(sc, mask, c_lo, c_hi, want, lane);
        __syncwarp();
    } else {
    // the `want` best candidates, one per round: every lane's best of its blocks, then the warp's best;
    // equal scores go to the lower block
    for (int r = 0; r < want; ++r) {
        float bv = -CUDART_INF_F;
        int bj = INT_MAX;
        for (int j = c_lo + lane; j < c_hi; j += 32) {
            const float v = sc[j];
            const bool taken = (mask[j >> 5] >> (j & 31)) & 1u;
            if (!taken && (bj == INT_MAX || v > bv)) { bv = v; bj = j; }   // ascending j: '>' keeps the lower block
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float ov = __shfl_xor_sync(FULLMASK, bv, off);
            const int oj = __shfl_xor_sync(FULLMASK, bj, off);
            if (oj != INT_MAX && (bj == INT_MAX || ov > bv || (ov == bv && oj < bj))) { bv = ov; bj = oj; }
        }
        if (lane == 0 && bj != INT_MAX) mask[bj >> 5] |= 1u << (bj & 31);
        __syncwarp();
    }
    }
    if (lane == 0) {
        for (int j = 0; j < ns; ++j) mask[j >> 5] |= 1u << (j & 31);
        for (int j = P - nl; j < P; ++j) mask[j >> 5] |= 1u << (j & 31);
    }
    __syncwarp();
    // ascending list from the mask
    int base = 0;
    if (words <= 4) {
        // few blocks: a lane looks at its own bit of every word; a chosen block's place in the list is the
        // number of chosen blocks below it
        const uint32_t lt = (1u << lane) - 1u;
        for (int r = 0; r < words; ++r) {
            const uint32_t w = mask[r];
            if ((w >> lane) & 1u) {
                const int pos = base + __popc(w & lt);
                if (pos < K) out[pos] = r * 32 + lane;
            }
            base += __popc(w);
        }
        for (int i = base + lane; i < K; i += 32) out[i] = -1;
        return;
    }
    for (int w0 = 0; w0 < words; w0 += 32) {
        const uint32_t w = w0 + lane < words ? mask[w0 + lane] : 0u;
        const int cnt = __popc(w);
        int inc = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(FULLMASK, inc, off);
            if (lane >= off) inc += o;
        }
        int pos = base + inc - cnt;
        uint32_t bits = w;
        while (bits) {
            const int bit = __ffs(bits) - 1;
            bits &= bits - 1;
            if (pos < K) out[pos] = (w0 + lane) * 32 + bit;
            ++pos;
        }
        base += __shfl_sync(FULLMASK, inc, 31);
    }
    for (int i = base + lane; i < K; i += 32) out[i] = -1;
}

template <typename T, int D, bool STAGED>
__global__ void __launch_bounds__(kMobaRouteWarps * 32) moba_route_kernel(const T *q, const float *means, int64_t len, int H,
                                                                         int block, int nb, int K, int32_t *sel)
{
    extern __shared__ __align__(16) float rsm[];
    constexpr int LDM = STAGED ? D + 4 : D;            // floats from one representative to the next
    constexpr int QW = STAGED ? kMobaRouteQ : 1, QC = kMobaRouteWarps * QW;   // queries of a warp, of the CTA
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int words = (nb + 31) / 32;
    const int per = moba_route_floats(D, nb);
    float *wsm = rsm + (size_t)warp * QW * per;        // this warp's queries, scores and masks
    const int bh = blockIdx.y;
    const float *mh = means + (int64_t)bh * nb * D;
    if (STAGED) {
        // the representatives the CTA's queries can need: blocks before the last query's own
        float *ms = rsm + (size_t)kMobaRouteWarps * QW * per;
        const int64_t t_last = min((int64_t)blockIdx.x * QC + QC - 1, len - 1);
        const int need = (int)(t_last / block);
        for (int i = threadIdx.x; i < need * (D / 4); i += kMobaRouteWarps * 32) {
            const int j = i / (D / 4), c = i % (D / 4);
            *reinterpret_cast<float4 *>(ms + j * LDM + 4 * c) = __ldg(reinterpret_cast<const float4 *>(mh + (int64_t)j * D) + c);
        }
        __syncthreads();
        mh = ms;
    }
    const int b = bh / H, h = bh % H;
    // the first block and the own block inside the budget (K >= 2), as the first and the newest page of a decode step
    const int ns = min(1, K), nl = min(1, K - ns), want = K - ns - nl;
    const int c_lo = ns;
    int P[QW], c_hi[QW];                               // blocks a query may attend; its candidates end before c_hi
    bool active[QW];
    int c_hi_max = 0;
#pragma unroll
    for (int u = 0; u < QW; ++u) {
        const int64_t t = (int64_t)blockIdx.x * QC + warp * QW + u;
        active[u] = false;
        P[u] = c_hi[u] = 0;
        if (t >= len) continue;                        // (no CTA-wide barrier below)
        int32_t *out = sel + ((int64_t)bh * len + t) * K;
        P[u] = (int)(t / block) + 1;
        if (K >= P[u]) {                               // everything before the query
            for (int i = lane; i < K; i += 32) out[i] = i < P[u] ? i : -1;
            continue;
        }
        active[u] = true;
        c_hi[u] = P[u] - nl;                           // candidates: blocks c_lo .. c_hi - 1 (all complete)
        c_hi_max = max(c_hi_max, c_hi[u]);
        float *qs = wsm + u * per;
        uint32_t *mask = reinterpret_cast<uint32_t *>(qs + D + nb);
        for (int i = lane; i < D; i += 32) qs[i] = load1<T>(q + (((int64_t)b * len + t) * H + h) * D + i);
        for (int i = lane; i < words; i += 32) mask[i] = 0u;
    }
    if (c_hi_max == 0) return;
    __syncwarp();
    // scores: a lane per block, the block's representative read as 16-byte pieces once for the warp's queries
    for (int j0 = c_lo; j0 < c_hi_max; j0 += 32) {
        const int j = j0 + lane;
        if (j < c_hi_max) {
            const float4 *row = reinterpret_cast<const float4 *>(mh + (int64_t)j * LDM);
            // packed pairs: the even and the odd channels are summed apart and added at the end
            float2 s2[QW];
#pragma unroll
            for (int u = 0; u < QW; ++u) s2[u] = make_float2(0.0f, 0.0f);
#pragma unroll 8
            for (int i = 0; i < D / 4; ++i) {
                const float4 m4 = STAGED ? row[i] : __ldg(row + i);
#pragma unroll
                for (int u = 0; u < QW; ++u) {
                    if (!active[u]) continue;          // (the same for the whole warp)
                    const float4 q4 = *reinterpret_cast<const float4 *>(wsm + u * per + 4 * i);
                    s2[u] = fma2(make_float2(q4.x, q4.y), make_float2(m4.x, m4.y), s2[u]);
                    s2[u] = fma2(make_float2(q4.z, q4.w), make_float2(m4.z, m4.w), s2[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < QW; ++u)
                if (active[u] && j < c_hi[u]) (wsm + u * per + D)[j] = s2[u].x + s2[u].y;
        }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < QW; ++u) {
        if (!active[u]) continue;
        const int64_t t = (int64_t)blockIdx.x * QC + warp * QW + u;
        float *sc = wsm + u * per + D;
        moba_route_finish(sc, reinterpret_cast<uint32_t *>(sc + nb), sel + ((int64_t)bh * len + t) * K, words, K, P[u], ns, nl, c_lo,
                          c_hi[u], want, lane);
    }
}

// ---------------------------------------------------------------- attention
// Grid (ceil(T / 16), heads), 16 warps, a warp per query.  Shared memory: two chunk buffers (64 key
// rows then 64 value rows each), the blocks chosen by any of the CTA's queries (bit mask) and by each
// query (16 bit masks).
template <typename T, int D>
__global__ void __launch_bounds__(kMobaQueries * 32) moba_attend_kernel(const T *kv, int64_t page_cap, int S, int64_t len,
                                                                       const T *q, int H, int block, int nb, int K,
                                                                       const int32_t *sel, float scale_log2, T *o)
{
    constexpr int CH = VecOf<T>::N, LPR = D / CH;
    constexpr int ROW_BYTES = D * (int)sizeof(T), PPR = ROW_BYTES / 16;      // 16-byte pieces of a row
    constexpr int CHUNK_BYTES = 2 * kMobaChunk * ROW_BYTES;
    constexpr int NT = kMobaQueries * 32;
    extern __shared__ __align__(16) unsigned char asmem[];
    unsigned char *buf = asmem;                                              // [2][CHUNK_BYTES]
    uint32_t *umask = reinterpret_cast<uint32_t *>(asmem + 2 * CHUNK_BYTES); // [words]
    const int words = (nb + 31) / 32;
    uint32_t *qmask = umask + words;                                         // [16][words]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bh = blockIdx.y, b = bh / H, h = bh % H;
    const int64_t t = (int64_t)blockIdx.x * kMobaQueries + warp;
    const bool active = t < len;

    for (int i = tid; i < words * (kMobaQueries + 1); i += NT) umask[i] = 0u;
    __syncthreads();
    if (active) {
        const int32_t *list = sel + ((int64_t)bh * len + t) * K;
        for (int i = lane; i < K; i += 32) {
            const int j = list[i];
            if (j >= 0 && j < nb) {
                atomicOr(&qmask[warp * words + (j >> 5)], 1u << (j & 31));
                atomicOr(&umask[j >> 5], 1u << (j & 31));
            }
        }
    }
    __syncthreads();

    AttendState<T> st;
    attend_begin_head<T, D>(st, q + (((int64_t)b * len + (active ? t : 0)) * H + h) * D, 0, scale_log2, lane);

    const T *head = kv + (int64_t)bh * page_cap * 2 * S * D;
    // copies of chunk `ci` of block j (positions j * block + ci * 64 ...) into buffer `bi`
    auto issue = [&](int j, int ci, int bi) {
        const int64_t p0 = (int64_t)j * block + (int64_t)ci * kMobaChunk;
        unsigned char *dst = buf + (size_t)bi * CHUNK_BYTES;
        for (int i = tid; i < kMobaChunk * PPR; i += NT) {
            const int r = i / PPR, c = i % PPR;
            const int64_t p = p0 + r;
            if (p < len) {
                const unsigned char *src =
                    reinterpret_cast<const unsigned char *>(head + (((p / S) * 2) * S + p % S) * D) + c * 16;
                cp_async16(dst + r * ROW_BYTES + c * 16, src);
                cp_async16(dst + (kMobaChunk + r) * ROW_BYTES + c * 16, src + (int64_t)S * ROW_BYTES);
            } else {                                         // rows past the prompt: defined (a masked row still multiplies its values by 0)
                *reinterpret_cast<uint4 *>(dst + r * ROW_BYTES + c * 16) = make_uint4(0u, 0u, 0u, 0u);
                *reinterpret_cast<uint4 *>(dst + (kMobaChunk + r) * ROW_BYTES + c * 16) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    };
    // the chunks of the chosen blocks in ascending order: (block, chunk) -> next
    const int cpb = block / kMobaChunk;
    auto next_chunk = [&](int &j, int &ci) -> bool {     // from (j, ci) to the following chunk; false at the end
        if (j >= 0 && ci + 1 < cpb && ((int64_t)j * block + (int64_t)(ci + 1) * kMobaChunk) < len) { ++ci; return true; }
        for (int jj = j + 1; jj < nb; ++jj)
            if ((umask[jj >> 5] >> (jj & 31)) & 1u) { j = jj; ci = 0; return true; }
        return false;
    };
    int j = -1, ci = 0, bi = 0;
    bool have = next_chunk(j, ci);
    if (have) issue(j, ci, 0);
    cp_async_commit();
    while (have) {
        int jn = j, cn = ci;
        const bool have_next = next_chunk(jn, cn);
        if (have_next) issue(jn, cn, bi ^ 1);           // the other buffer was released by the barrier below
        cp_async_commit();
        cp_async_wait<1>();                              // this thread's pieces of the current chunk
        __syncthreads();                                 // everybody's
        if (active && ((qmask[warp * words + (j >> 5)] >> (j & 31)) & 1u)) {
            const T *ks = reinterpret_cast<const T *>(buf + (size_t)bi * CHUNK_BYTES);
            const T *vs = ks + kMobaChunk * D;
            const int64_t p0 = (int64_t)j * block + (int64_t)ci * kMobaChunk;
#pragma unroll 1
            for (int i = 0; i < kMobaChunk / kTileRows; ++i) {
                const int64_t pt = p0 + (int64_t)i * kTileRows;
                const int valid = (int)min((int64_t)kTileRows, t - pt + 1);   // the query sees positions up to its own
                if (valid > 0) attend_tile<T, D, kTileRows>(st, ks + i * kTileRows * D, vs + i * kTileRows * D, valid, lane);
            }
        }
        __syncthreads();                                 // the buffer may be refilled
        j = jn; ci = cn; have = have_next; bi ^= 1;
    }
    cp_async_wait<0>();
    if (active) {
        attend_merge_rows<T, D, kTileRows>(st);
        if (lane < LPR) {
            const float inv = 1.0f / st.l;               // the own block always holds the query's own position
            T *orow = o + (((int64_t)b * len + t) * H + h) * D + lane * CH;
#pragma unroll
            for (int c = 0; c < CH; ++c) store1<T>(orow + c, st.acc[c] * inv);
        }
    }
}

size_t round256(size_t x) { return (x + 255) & ~(size_t)255; }

// fp32 caches: everything on plain fp32 FMAs (tf32 products would round the operands).
template <int D>
cudaError_t moba_run_f32(const MobaArgs &a, cudaStream_t s)
{
    const int BH = a.B * a.H;
    const int nb = (int)((a.len + a.block - 1) / a.block);
    const int words = (nb + 31) / 32;
    const bool staged = nb <= kMobaStagedBlocks;
    const int rq = staged ? kMobaRouteQ : 1;         // queries of a routing warp
    const size_t rs = (size_t)kMobaRouteWarps * rq * moba_route_floats(D, nb) * sizeof(float) + (staged ? (size_t)nb * (D + 4) * sizeof(float) : 0);
    constexpr int CHUNK_BYTES = 2 * kMobaChunk * D * (int)sizeof(float);
    const size_t as = 2 * (size_t)CHUNK_BYTES + (size_t)words * (kMobaQueries + 1) * sizeof(uint32_t);
    static bool ready[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!ready[dev]) {
        e = cudaFuncSetAttribute(moba_route_kernel<float, D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)((size_t)kMobaRouteWarps * moba_route_floats(D, kMobaMaxBlocks) * sizeof(float)));
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(moba_route_kernel<float, D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)((size_t)kMobaRouteWarps * kMobaRouteQ * moba_route_floats(D, kMobaStagedBlocks) * sizeof(float) +
                                       (size_t)kMobaStagedBlocks * (D + 4) * sizeof(float)));
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(moba_attend_kernel<float, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(2 * (size_t)CHUNK_BYTES + (size_t)(kMobaMaxBlocks / 32) * (kMobaQueries + 1) * sizeof(uint32_t)));
        if (e != cudaSuccess) return e;
        ready[dev] = true;
    }
    moba_means_kernel<float><<<dim3((unsigned)nb, (unsigned)BH), D, 0, s>>>((const float *)a.kv, a.page_cap, a.S, D, a.len, a.block,
                                                                          a.means, nb);
    const dim3 rgrid((unsigned)((a.len + kMobaRouteWarps * rq - 1) / (kMobaRouteWarps * rq)), (unsigned)BH);
    if (staged)
        moba_route_kernel<float, D, true><<<rgrid, kMobaRouteWarps * 32, rs, s>>>((const float *)a.q, a.means, a.len, a.H, a.block, nb, a.K, a.list);
    else
        moba_route_kernel<float, D, false><<<rgrid, kMobaRouteWarps * 32, rs, s>>>((const float *)a.q, a.means, a.len, a.H, a.block, nb, a.K, a.list);
    moba_attend_kernel<float, D><<<dim3((unsigned)((a.len + kMobaQueries - 1) / kMobaQueries), (unsigned)BH), kMobaQueries * 32, as, s>>>(
        (const float *)a.kv, a.page_cap, a.S, a.len, (const float *)a.q, a.H, a.block, nb, a.K, a.list, a.scale * 1.4426950408889634f,
        (float *)a.o);
    return cudaGetLastError();
}

}  // namespace

size_t moba_scratch_bytes(int BH, int64_t len, int D, int block, int K)
{
    const size_t nb = (size_t)((len + block - 1) / block);
    return round256((size_t)BH * nb * D * sizeof(float)) + round256((size_t)BH * (size_t)len * K * sizeof(int32_t));
}

void moba_carve(void *scratch, int32_t *blocks_out, MobaArgs &a)
{
    const size_t nb = (size_t)((a.len + a.block - 1) / a.block);
    a.means = (float *)scratch;
    void *rest = (char *)scratch + round256((size_t)a.B * a.H * nb * a.D * sizeof(float));     // room for the lists
    a.masks = a.dtype == RQ_BF16 && (nb + 31) / 32 <= (size_t)a.K ? (uint32_t *)rest : nullptr;
    a.list = blocks_out ? blocks_out : a.masks ? nullptr : (int32_t *)rest;
    // what the lists would take, where they are not in it, holds more behind the masks, but for the smallest budgets of short prompts
    const size_t BH = (size_t)a.B * a.H, words = (nb + 31) / 32, room = a.list == (int32_t *)rest ? 0 : round256(BH * (size_t)a.len * a.K * sizeof(int32_t));
    size_t used = a.masks ? round256(BH * (size_t)a.len * words * sizeof(uint32_t)) : 0;
    auto take = [&](size_t bytes) -> void * {
        if (a.dtype != RQ_BF16 || used + round256(bytes) > room) return nullptr;
        void *p = (char *)rest + used;
        used += round256(bytes);
        return p;
    };
    a.unions = (uint32_t *)take(BH * (((size_t)a.len + 127) / 128) * words * sizeof(uint32_t));
    a.terms = take(BH * ((nb + 63) / 64) * 64 * a.D * 6);      // 64 blocks' terms: 6 bytes a channel
}

cudaError_t launch_moba(const MobaArgs &a, cudaStream_t s)
{
    if (a.block < kMobaChunk || a.block % kMobaChunk != 0 || a.block % a.S != 0 || a.K < 2 || a.len < 1) return cudaErrorInvalidValue;
    if ((a.len + a.block - 1) / a.block > kMobaMaxBlocks || a.B * a.H > 65535 || (a.len + 127) / 128 > 65535)
        return cudaErrorInvalidValue;
    if (a.dtype == RQ_BF16) {
        const cudaError_t e = launch_moba_route_bf16(a, s);
        return e != cudaSuccess ? e : launch_moba_attend_bf16(a, s);
    } else {
        if (a.D == 128) return moba_run_f32<128>(a, s);
        if (a.D == 64) return moba_run_f32<64>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace rq
