// Prefill: the gated decay recurrence (Eq. 1) over a whole sequence, fused with
// the paged cache write and the per-page min/max of the stored keys
// (Appendix A.1, "Sparse inference settings").  One launch, every input byte
// read once, every output byte written once, no scratch in global memory, but for very long
// prompts of a few heads, which are cut into time chunks (three launches, the inputs of all
// chunks but the last read twice, the chunks' maps and entry states in the workspace).
//
// The recurrence x~_t = g_t x~_{t-1} + (1-g_t) x_t runs along time and is
// independent per (batch, head, channel).  Work decomposition: a unit is one
// (batch, head) pair and 32 neighbouring channels; it belongs to one CTA, or, when
// there are few units and many positions, to a cluster of up to four CTAs that take
// its tiles in turn.
//
// Time is cut into tiles of 256 positions that move through a ring of shared-memory
// stages, filled by tiled bulk-tensor copies several tiles ahead of the arithmetic.
// A lane owns two neighbouring channels (one 4-byte access for a bf16 pair) and a
// half-warp owns a run of 8 consecutive positions of the tile.  A run of tokens acts on
// the incoming state as the affine map s -> A s + B with A = prod g and B = the
// run's own state from zero, and maps compose as (A2,B2)o(A1,B1) = (A2 A1,
// A2 B1 + B2).  Per tile: every thread reduces its run to a map (pass 1), its gates and
// gated inputs staying in registers, and the two runs of a warp are composed by shuffles;
// after a barrier (the stage may be refilled) the 16 warp maps of every channel are scanned
// by 16 lanes (warp w takes channels 2w and 2w+1), which, with the state entering the tile,
// gives the state entering every warp and the state entering the next tile; after a second
// barrier every thread applies the recurrence token by token (pass 2), rounds to the storage
// type and its rows go out to the cache, 64 or 128 bytes of a row per half-warp.  Page
// bounds are taken before rounding (rounding is monotone: the rounded minimum is the minimum
// of the rounded).
//
// In a cluster the state entering a tile comes from the CTA that has the tile before, as 256
// bytes written into this CTA's shared memory (st.async, counted on a barrier); the maps of
// the tile are ready by then, so that a hop costs one multiplication and one message.  The
// arithmetic is the same whatever the size of the cluster.
//
// The order of all floating-point operations is fixed: the same bits on every run.
//
// Bound: the phases of a tile between its two barriers, with DRAM close behind (131072 tokens of 32 heads x 128, bf16: 5.5
// GB in 0.90 to 0.99 ms, 5.6 to 6.1 TB/s; the copies alone run at 5.8 TB/s).  Before (copies started and rows stored in
// 16-byte pieces by all threads, one CTA per unit, three barriers, the inputs read twice for few heads) / now, us: 32 heads,
// 131072 tokens 1120 / 900; 4001 tokens and the clearing before them 50 / 40; 8 heads, 50003 tokens, fp32 gates 195 / 111; 8
// heads, 8000 tokens 76 / 33; 4 heads, 8000 tokens 75 / 31; 256 heads, 16 tokens 22 / 18; fp32, 12 heads, 20000 tokens 176 /
// 120; fp32, 32 heads, 8000 tokens, pages of 16, 120 / 121.
#include "rq_async.cuh"
#include "rq_device.cuh"
#include "rq_internal.h"
#include "rq_tmap.h"
#include "rq_umma.cuh"

#include <cooperative_groups.h>

namespace rq {

namespace {

namespace cg = cooperative_groups;

constexpr int NT = kScanThreads;
constexpr int NW = NT / 32;
constexpr int CG = kScanChannels;               // channels of one unit: two per lane of a half-warp
constexpr int RT = kScanRunTokens;              // consecutive positions of one half-warp in a tile
constexpr int TT = 2 * NW * RT;                 // positions of one tile
constexpr int kMapStride = 3 * CG + 2;          // floats between two warps' maps: an even count, and lanes that read
                                                // the same channel of 16 consecutive maps hit 16 different banks
constexpr int kInStride = 2 * CG + 2;           // likewise for the states entering the warps
constexpr int LPC = NW;                         // lanes that scan the warp maps of one channel
constexpr int kMaxCluster = 4;
static_assert(CG == 32 && NW == 16 && RT == 8, "the layouts below");

// two neighbouring elements as floats
__device__ __forceinline__ float2 unpack2(uint32_t w) { return make_float2(bf16lo(w), bf16hi(w)); }
__device__ __forceinline__ float2 load2(const bf16 *p) { return unpack2(*reinterpret_cast<const uint32_t *>(p)); }
__device__ __forceinline__ float2 load2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
// round two floats to the storage type and store them side by side
__device__ __forceinline__ void store2(bf16 *p, float x, float y) { *reinterpret_cast<uint32_t *>(p) = pack_bf16(x, y); }
__device__ __forceinline__ void store2(float *p, float x, float y) { *reinterpret_cast<float2 *>(p) = make_float2(x, y); }
// the same for data that nobody reads soon
__device__ __forceinline__ void store2_cs(bf16 *p, float2 x) { __stcs(reinterpret_cast<uint32_t *>(p), pack_bf16(x.x, x.y)); }
__device__ __forceinline__ void store2_cs(float *p, float2 x) { __stcs(reinterpret_cast<float2 *>(p), x); }

template <bool B> struct BoolTag { static constexpr bool value = B; };

// bytes of one ring stage: the k, v and g segments of a tile
template <typename T, typename G> __host__ __device__ constexpr int scan_stage_bytes()
{
    return TT * CG * (2 * (int)sizeof(T) + (int)sizeof(G));
}
// stages of the ring: as many as fit in 192 KiB, at most four
template <typename T, typename G> __host__ __device__ constexpr int scan_stages()
{
    return 192 * 1024 / scan_stage_bytes<T, G>() < 4 ? 192 * 1024 / scan_stage_bytes<T, G>() : 4;
}

// wait for data that other CTAs of the cluster have written
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity)
{
    const uint32_t addr = smem_addr(bar);
    for (int it = 0; it < kMbarPollLimit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(addr), "r"(parity), "r"(kMbarSuspendNs)
            : "memory");
        if (ok) return true;
    }
    return false;
}
// the address of `p` in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t peer_smem(const void *p, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}
// one float into a peer's shared memory, its four bytes counted on the peer's barrier
__device__ __forceinline__ void send_float(uint32_t dst, float x, uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst), "r"(__float_as_uint(x)), "r"(bar)
                 : "memory");
}

struct ScanMaps {
    CUtensorMap k, v, g, cache;
};
struct ScanPlan {
    int64_t tile0;          // first tile (of 256 cache positions) that the call touches
    int ntiles, units;
    int tma;                // full tiles come through the tensor maps (otherwise with plain loads)
    int chunks, chunk_tiles;
};

// MODE 0: the scan proper.  MODE 1: the affine map of a time chunk only (no output), for the time-chunked form.
// MODE 2: MODE 0 with one CTA per unit and the CTAs of a head as a cluster that keeps them within a tile of each other.
// MODE 4: MODE 0 where heads or batch items may share their numbers.
// MODE 3: MODE 0 for a call inside one tile, with plain loads and without the ring, so that two CTAs share an SM.
// Time chunks (chunks > 1; so few units that not even clusters fill the chip, and a long prompt): CTA x works on unit
// x % units and the chunk_tiles tiles of chunk x / units.  First every chunk but the last is reduced to its map s -> A s + B
// (MODE 1), a small kernel chains the maps into the state that enters every chunk, then every chunk runs the scan proper
// from its own entry state.  The inputs of all chunks but the last are read twice.  (Chunks and clusters exclude each other.)
//   maps   [units][chunks][3][CG]   A, B of the keys, B of the values
//   entry  [units][chunks][2][CG]   state entering a chunk (not chunk 0), and the state before the call
template <typename T, typename G, int D, int S, int MODE, bool STAGED>
__global__ void __launch_bounds__(NT, MODE == 3 ? 2 : 1) scan_kernel(ScanArgs a, const __grid_constant__ ScanMaps tm, ScanPlan plan, float *maps, const float *entry)
{
    constexpr int NST = scan_stages<T, G>();
    constexpr int STAGE = scan_stage_bytes<T, G>();
    constexpr int OFF_V = TT * CG * (int)sizeof(T), OFF_G = 2 * OFF_V;
    // a warp's rows go back into their stage and out with tensor-map stores, or out straight from registers (rule in run())
    constexpr bool BY_STAGE = STAGED;
    constexpr int WPP = S / (2 * RT);                                          // warps that share a page
    constexpr unsigned FULLMASK = 0xffffffffu;
    static_assert(D % CG == 0, "a head is a whole number of channel groups");
    static_assert(S % (2 * RT) == 0 && TT % S == 0 && NW % WPP == 0, "a page is a whole number of warps inside one tile");
    static_assert(NST >= 2, "the ring needs two stages");

    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) float wmap[NW * kMapStride];    // the warps' maps of the current tile: [warp][A, Bk, Bv][channel]
    __shared__ __align__(8) float sin_[NW * kInStride];     // state entering every warp: [warp][k, v][channel]
    __shared__ float carry[2][2][CG];                       // state entering this CTA's tile (by parity): k, v
    __shared__ float carry_a[2][CG];                        // MODE 1: product of the gates since the chunk began
    __shared__ float mm[2][NW][2][CG];                      // min / max of the warps (pages wider than a warp's 16 positions), by tile parity
    __shared__ __align__(8) uint64_t full[NST], carried[2]; // a stage has landed; the state entering a tile has arrived

    cg::cluster_group cl = cg::this_cluster();
    const int CL = MODE == 2 || MODE == 3 ? 1 : (int)cl.num_blocks(), cr = MODE == 2 || MODE == 3 ? 0 : (int)cl.block_rank();
    const int unit = blockIdx.x / CL % plan.units, chunk = blockIdx.x / CL / plan.units, chunks = plan.chunks;
    const int64_t tile0 = plan.tile0 + (int64_t)chunk * plan.chunk_tiles;
    const int ntiles = min(plan.chunk_tiles, plan.ntiles - chunk * plan.chunk_tiles);
    const int mine = cr < ntiles ? (ntiles - cr + CL - 1) / CL : 0;            // tiles of this CTA: cr, cr + CL, ...
    if (MODE == 1 && chunk == chunks - 1) return;           // the last chunk's map is not needed

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int hl = lane & 15, half = lane >> 4;  // channel pair of this lane; which of the warp's two runs
    const int ch2 = 2 * hl;                      // first of this lane's two channels inside the group
    constexpr int GPH = D / CG;                  // channel groups per head
    const int bh = unit / GPH, c0 = (unit % GPH) * CG;
    // coordinates in the inputs' tensor maps.  (Chosen only where numbers may be shared: the choice leaves the uniform
    // registers, and each copy is started later: 32 heads x 128, 50000 tokens 348 -> 365 us)
    constexpr bool SHARED = MODE == 1 || MODE == 4;
    const int b = SHARED && a.sb == 0 ? 0 : bh / a.H, h = SHARED && a.sh == 0 ? 0 : bh % a.H;
    const int64_t end = a.len0 + a.T;
    const int64_t tail_end = (end + S - 1) / S * S;   // end of the last touched page
    const int64_t in_base = (int64_t)b * a.sb + (int64_t)h * a.sh + c0 + ch2;
    const T *kp = static_cast<const T *>(a.k) + in_base;
    const T *vp = static_cast<const T *>(a.v) + in_base;
    const G *gp = static_cast<const G *>(a.g) + in_base;
    const int row0 = (2 * warp + half) * RT;     // first row of this thread's run

    // tile i of the unit (chunk): does it come through the tensor maps (rows past the prompt's end as zeros), and is it full?
    auto by_map = [&](int i) { return MODE != 3 && plan.tma && (tile0 + i) * TT >= a.len0; };
    auto full_tile = [&](int i) { return by_map(i) && (tile0 + i + 1) * TT <= end; };
    const uint64_t once = l2_evict_first_policy();
    // start the copies of this CTA's j-th tile.  The whole first warp.
    auto issue = [&](int j) {
        const int i = cr + j * CL, st = j % NST;
        if (by_map(i)) {
            unsigned char *dst = dsm + (size_t)st * STAGE;
            const int tok = (int)((tile0 + i) * TT - a.len0);
            mbar_expect_warp(&full[st], STAGE);
            // (rows of 128 bytes are whole lines that nobody else reads; of 64 bytes, half a line whose other half another CTA
            // reads at about the same time.  fp32 rows that go out by their stage do better without: 32 heads x 128, 131072
            // tokens 1861 -> 1780 us)
            constexpr bool HINT_KV = sizeof(T) == 4 && !STAGED, HINT_G = sizeof(G) == 4 && (sizeof(T) == 2 || !STAGED);
            if (HINT_KV) {
                tma_load_4d_hint(dst, &tm.k, c0, h, tok, b, &full[st], once);
                tma_load_4d_hint(dst + OFF_V, &tm.v, c0, h, tok, b, &full[st], once);
            } else {
                tma_load_4d(dst, &tm.k, c0, h, tok, b, &full[st]);
                tma_load_4d(dst + OFF_V, &tm.v, c0, h, tok, b, &full[st]);
            }
            if (HINT_G) tma_load_4d_hint(dst + OFF_G, &tm.g, c0, h, tok, b, &full[st], once);
            else tma_load_4d(dst + OFF_G, &tm.g, c0, h, tok, b, &full[st]);
        } else if (lane == 0) {
            mbar_arrive(&full[st]);
        }
        __syncwarp();
    };
    bool ok = true;
    if (MODE != 3 && tid == 0) {
        for (int s = 0; s < NST; ++s) mbar_init(&full[s], 1);
        mbar_init(&carried[0], 1);
        mbar_init(&carried[1], 1);
        mbar_init_fence();
    }
    grid_dependency_wait();                      // earlier kernels may still write what is read here, or read what is written
    grid_launch_dependents();
    if (MODE != 3) __syncthreads();
    if (MODE != 3 && warp == 0) {
        for (int j = 0; j < NST && j < mine; ++j) issue(j);
        if (CL > 1 && lane == 0) {
            // the first tile's state is the cache's, every other one comes as 2 * CG floats from the CTA before
            if (cr == 0) mbar_arrive(&carried[0]);
            else mbar_arrive_expect_tx(&carried[0], 2 * CG * sizeof(float));
            mbar_arrive_expect_tx(&carried[1], 2 * CG * sizeof(float));
        }
    }
    float first_k = 0.0f, first_v = 0.0f;        // MODE 3: the state, on its way while the tile is
    if (tid < CG && cr == 0) {                   // the state the (chunk of the) sequence starts from
        if (MODE == 1) {
            carry[0][0][tid] = 0.0f;
            carry[0][1][tid] = 0.0f;
            carry_a[0][tid] = 1.0f;
        } else if (MODE == 3) {
            first_k = a.state[(int64_t)bh * 2 * D + c0 + tid];
            first_v = a.state[(int64_t)bh * 2 * D + D + c0 + tid];
        } else if (MODE == 2 && chunks == 1) {   // (of its own: read like below, the copies start later, 32 heads x 128, 50000 tokens 361 -> 391 us)
            carry[0][0][tid] = a.state[(int64_t)bh * 2 * D + c0 + tid];
            carry[0][1][tid] = a.state[(int64_t)bh * 2 * D + D + c0 + tid];
        } else if (MODE != 2 && chunk == 0) {
            // (with several chunks a copy behind the entry states: the CTA of the last chunk overwrites the cache's state meanwhile)
            const float *from = chunks == 1 ? a.state : entry + (int64_t)plan.units * chunks * 2 * CG;
            carry[0][0][tid] = from[(int64_t)bh * 2 * D + c0 + tid];
            carry[0][1][tid] = from[(int64_t)bh * 2 * D + D + c0 + tid];
        } else {
            const float *e = entry + ((int64_t)unit * chunks + chunk) * 2 * CG;
            carry[0][0][tid] = e[tid];
            carry[0][1][tid] = e[CG + tid];
        }
    }
    if (CL > 1) cl.sync();                       // the barriers of all CTAs are ready
    T *kv = static_cast<T *>(a.kv) + (int64_t)bh * a.page_cap * 2 * S * D + c0 + ch2;
    T *meta = static_cast<T *>(a.meta) + (int64_t)bh * a.page_cap * 2 * D + c0 + ch2;
    const int next = cr + 1 < CL ? cr + 1 : 0;
    float amax = 0.0f;                           // largest |key| this thread has written, before rounding

    // bounds of the page that begins at position `pstart` (merged with what the page held before)
    auto put_bounds = [&](int64_t pstart, float mn0, float mn1, float mx0, float mx1) {
        T *mrow = meta + pstart / S * 2 * D;
        if (pstart < a.len0) {
            const float2 o = load2(mrow), p = load2(mrow + D);
            mn0 = fminf(mn0, o.x); mn1 = fminf(mn1, o.y);
            mx0 = fmaxf(mx0, p.x); mx1 = fmaxf(mx1, p.y);
        }
        store2(mrow, mn0, mn1);
        store2(mrow + D, mx0, mx1);
    };
    // pages wider than a warp's rows: the bounds of this CTA's j-th tile, once all its warps have left theirs in mm
    auto wide_bounds = [&](int j) {
        const int64_t pstart = (tile0 + cr + (int64_t)j * CL) * TT + 2 * warp * RT;   // a multiple of S for the page's first warp
        if (warp % WPP == 0 && half == 0 && pstart < end && pstart + S > a.len0) {
            const float (*m)[2][CG] = mm[j & 1];
            float2 lo = *reinterpret_cast<const float2 *>(&m[warp][0][ch2]), hi = *reinterpret_cast<const float2 *>(&m[warp][1][ch2]);
#pragma unroll
            for (int w = 1; w < WPP; ++w) {
                const float2 l2 = *reinterpret_cast<const float2 *>(&m[warp + w][0][ch2]);
                const float2 h2 = *reinterpret_cast<const float2 *>(&m[warp + w][1][ch2]);
                lo.x = fminf(lo.x, l2.x); lo.y = fminf(lo.y, l2.y);
                hi.x = fmaxf(hi.x, h2.x); hi.y = fmaxf(hi.y, h2.y);
            }
            put_bounds(pstart, lo.x, lo.y, hi.x, hi.y);
        }
    };

    // this CTA's j-th tile; MAP: it lands in its stage and every row of it is a new token
    auto tile = [&](auto map_tag, int j) {
        constexpr bool MAP = decltype(map_tag)::value;
        const int i = cr + j * CL;
        const int64_t tile_start = (tile0 + i) * TT;
        // rows of the tile that hold new tokens: [lo, hi); rows up to fill_hi pad the last page
        const int lo = MAP ? 0 : (int)max((int64_t)0, a.len0 - tile_start), hi = MAP ? TT : (int)min((int64_t)TT, end - tile_start);
        const int fill_hi = (int)min((int64_t)TT, tail_end - tile_start);
        const int64_t tok0 = tile_start - a.len0 + row0;                     // input token of this thread's first row

        // ---- pass 1: this thread's run as a map from a zero state (identity outside the new range)
        float2 g2[RT], k2[RT], v2[RT];                           // g, (1-g) k, (1-g) v of the two channels
        float2 A2 = make_float2(1.0f, 1.0f), Bk2 = make_float2(0.0f, 0.0f), Bv2 = make_float2(0.0f, 0.0f);
        // (a warp without new rows leaves its part of a short prompt out; elsewhere the branches cost more than they save)
        const bool idle = MODE == 3 && (2 * warp * RT >= hi || 2 * (warp + 1) * RT <= lo);
        if (!idle) {
        if (MAP || by_map(i)) {
            ok = ok && mbar_wait(&full[j % NST], (uint32_t)((j / NST) & 1));
            // (2-byte elements: the two halves of a warp, eight rows of 64 bytes apart, share banks: two reads instead of one)
            const unsigned char *st = dsm + (size_t)(j % NST) * STAGE;
            const T *kt = reinterpret_cast<const T *>(st) + row0 * CG + ch2, *vt = reinterpret_cast<const T *>(st + OFF_V) + row0 * CG + ch2;
            const G *gt = reinterpret_cast<const G *>(st + OFF_G) + row0 * CG + ch2;
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                g2[r] = load2(gt + r * CG);
                k2[r] = load2(kt + r * CG);
                v2[r] = load2(vt + r * CG);
                if (!MAP && row0 + r >= hi) g2[r] = make_float2(1.0f, 1.0f);     // (k and v are zero there)
            }
        } else {
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const bool in = row0 + r >= lo && row0 + r < hi;
                const int64_t src = (tok0 + r) * a.st;
                g2[r] = in ? load2(gp + src) : make_float2(1.0f, 1.0f);
                k2[r] = in ? load2(kp + src) : make_float2(0.0f, 0.0f);
                v2[r] = in ? load2(vp + src) : make_float2(0.0f, 0.0f);
            }
        }
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const float2 o2 = fma2(g2[r], make_float2(-1.0f, -1.0f), make_float2(1.0f, 1.0f));   // 1 - g
            k2[r] = mul2(o2, k2[r]);
            v2[r] = mul2(o2, v2[r]);
            A2 = mul2(A2, g2[r]);
            Bk2 = fma2(g2[r], Bk2, k2[r]);
            Bv2 = fma2(g2[r], Bv2, v2[r]);
        }
        }
        if (MODE == 3 && tid < CG) {
            carry[0][0][tid] = first_k;
            carry[0][1][tid] = first_v;
        }
        // the map of the warp's first run, for the second run; the second run's lanes publish the warp's map
        const float2 LA = make_float2(__shfl_sync(FULLMASK, A2.x, hl), __shfl_sync(FULLMASK, A2.y, hl));
        const float2 LBk = make_float2(__shfl_sync(FULLMASK, Bk2.x, hl), __shfl_sync(FULLMASK, Bk2.y, hl));
        const float2 LBv = make_float2(__shfl_sync(FULLMASK, Bv2.x, hl), __shfl_sync(FULLMASK, Bv2.y, hl));
        if (half == 1) {
            float *wm = wmap + warp * kMapStride + ch2;
            *reinterpret_cast<float2 *>(wm) = mul2(A2, LA);
            *reinterpret_cast<float2 *>(wm + CG) = fma2(A2, LBk, Bk2);
            *reinterpret_cast<float2 *>(wm + 2 * CG) = fma2(A2, LBv, Bv2);
        }
        if (BY_STAGE) tma_store_wait_read();                     // the warp's rows of the tile before have left their stage
        __syncthreads();                                         // the maps are there
        // the stage of the tile before (of this tile, if nothing goes back into it) is free
        if (MODE != 3 && warp == 0 && (!BY_STAGE || j >= 1) && j - BY_STAGE + NST < mine) issue(j - BY_STAGE + NST);
        if (WPP > 1 && MODE != 1 && j > 0) wide_bounds(j - 1);

        // ---- scan of the 16 warp maps of channels 2 warp and 2 warp + 1 (one per half-warp) by 16 lanes
        {
            const int ci = warp * (32 / LPC) + lane / LPC, m = lane % LPC;   // channel inside the group, map (= warp) index
            const float *wm = wmap + m * kMapStride + ci;
            float sa = wm[0], sbk = wm[CG], sbv = wm[2 * CG];
#pragma unroll
            for (int off = 1; off < LPC; off <<= 1) {
                const float pa = __shfl_up_sync(FULLMASK, sa, off, LPC);
                const float pbk = __shfl_up_sync(FULLMASK, sbk, off, LPC);
                const float pbv = __shfl_up_sync(FULLMASK, sbv, off, LPC);
                if (m >= off) {
                    sbk = fmaf(sa, pbk, sbk);
                    sbv = fmaf(sa, pbv, sbv);
                    sa *= pa;
                }
            }
            float ea = __shfl_up_sync(FULLMASK, sa, 1, LPC);  // maps of the warps before this one
            float ebk = __shfl_up_sync(FULLMASK, sbk, 1, LPC);
            float ebv = __shfl_up_sync(FULLMASK, sbv, 1, LPC);
            if (m == 0) { ea = 1.0f; ebk = 0.0f; ebv = 0.0f; }
            if (CL > 1) ok = ok && mbar_wait_cluster(&carried[j & 1], (uint32_t)((j >> 1) & 1));
            const float ck = carry[j & 1][0][ci], cv = carry[j & 1][1][ci];
            if (m == LPC - 1) {                              // the state after the tile: to the next tile, or the end
                const float nk = fmaf(sa, ck, sbk), nv = fmaf(sa, cv, sbv);
                if (MODE != 1 && i == ntiles - 1 && chunk == chunks - 1) {
                    a.state[(int64_t)bh * 2 * D + c0 + ci] = nk;
                    a.state[(int64_t)bh * 2 * D + D + c0 + ci] = nv;
                } else if (CL > 1) {
                    if (i + 1 < ntiles) {
                        const int nb = ((i + 1) / CL) & 1;
                        const uint32_t bar = peer_smem(&carried[nb], next);
                        send_float(peer_smem(&carry[nb][0][ci], next), nk, bar);
                        send_float(peer_smem(&carry[nb][1][ci], next), nv, bar);
                    }
                } else {
                    carry[(j + 1) & 1][0][ci] = nk;
                    carry[(j + 1) & 1][1][ci] = nv;
                    if (MODE == 1) carry_a[(j + 1) & 1][ci] = sa * carry_a[j & 1][ci];
                }
            }
            sin_[m * kInStride + ci] = fmaf(ea, ck, ebk);
            sin_[m * kInStride + CG + ci] = fmaf(ea, cv, ebv);
        }
        __syncthreads();
        if (MODE == 1) return;                                   // the map needs no more of the tile
        // (everybody has seen the state that entered; the barrier is armed for the CTA's tile after the next)
        if (CL > 1 && tid == 0 && j + 2 < mine) mbar_arrive_expect_tx(&carried[j & 1], 2 * CG * sizeof(float));

        // ---- pass 2: token by token, the rounded rows to their page, bounds of the keys
        float2 sk2 = *reinterpret_cast<const float2 *>(sin_ + warp * kInStride + ch2);
        float2 sv2 = *reinterpret_cast<const float2 *>(sin_ + warp * kInStride + CG + ch2);
        if (half == 1) {                                         // through the warp's first run
            sk2 = fma2(LA, sk2, LBk);
            sv2 = fma2(LA, sv2, LBv);
        }
        const int64_t pos = tile_start + row0;                   // a run lies inside one page
        T *dst = kv + (pos / S * 2 * S + pos % S) * D;
        float mn0 = INFINITY, mn1 = INFINITY, mx0 = -INFINITY, mx1 = -INFINITY;
        if (!idle || (2 * warp * RT >= hi && 2 * warp * RT < fill_hi)) {
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            if (MAP || (row0 + r >= lo && row0 + r < hi)) {
                sk2 = fma2(g2[r], sk2, k2[r]);
                sv2 = fma2(g2[r], sv2, v2[r]);
                if constexpr (MAP && BY_STAGE) {
                    T *kt = reinterpret_cast<T *>(dsm + (size_t)(j % NST) * STAGE) + (row0 + r) * CG + ch2;
                    store2(kt, sk2.x, sk2.y);
                    store2(kt + TT * CG, sv2.x, sv2.y);
                } else {
                    store2_cs(dst + r * D, sk2);
                    store2_cs(dst + (S + r) * D, sv2);
                }
                mn0 = fminf(mn0, sk2.x); mx0 = fmaxf(mx0, sk2.x);
                mn1 = fminf(mn1, sk2.y); mx1 = fmaxf(mx1, sk2.y);
            } else if (row0 + r >= hi && row0 + r < fill_hi) {   // unused slots of the last page
                store2_cs(dst + r * D, make_float2(0.0f, 0.0f));
                store2_cs(dst + (S + r) * D, make_float2(0.0f, 0.0f));
            }
        }
        }
        if constexpr (MAP && BY_STAGE) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            const T *kt = reinterpret_cast<const T *>(dsm + (size_t)(j % NST) * STAGE) + warp * 2 * RT * CG;
            const int64_t wpos = tile_start + 2 * warp * RT;
            const int page = (int)(bh * a.page_cap + wpos / S), slot = (int)(wpos % S);
            tma_store_4d(kt, &tm.cache, c0, slot, 0, page);
            tma_store_4d(kt + TT * CG, &tm.cache, c0, slot, 1, page);
            tma_store_commit();
        }
        if (mn0 <= mx0) amax = fmaxf(amax, fmaxf(fmaxf(-mn0, mx0), fmaxf(-mn1, mx1)));   // this run held new tokens
        // the warp's two runs together (16 positions)
        mn0 = fminf(mn0, __shfl_xor_sync(FULLMASK, mn0, 16)); mn1 = fminf(mn1, __shfl_xor_sync(FULLMASK, mn1, 16));
        mx0 = fmaxf(mx0, __shfl_xor_sync(FULLMASK, mx0, 16)); mx1 = fmaxf(mx1, __shfl_xor_sync(FULLMASK, mx1, 16));
        if (WPP > 1) {
            if (half == 0) {
                *reinterpret_cast<float2 *>(&mm[j & 1][warp][0][ch2]) = make_float2(mn0, mn1);
                *reinterpret_cast<float2 *>(&mm[j & 1][warp][1][ch2]) = make_float2(mx0, mx1);
            }
        } else if (half == 0) {
            const int64_t pstart = tile_start + 2 * warp * RT;
            if (pstart < end && pstart + S > a.len0) put_bounds(pstart, mn0, mn1, mx0, mx1);
        }
    };

    // (full tiles in a loop of their own: 42.2 -> 41.0 us for 4001 tokens)
    const int64_t full_from = plan.tma ? (a.len0 + TT - 1) / TT - tile0 : (int64_t)ntiles, full_to = plan.tma ? end / TT - tile0 : (int64_t)0;
    int j = 0;
#pragma unroll 1
    while (j < mine) {
#pragma unroll 1
        for (; MODE != 3 && j < mine && cr + j * CL >= full_from && cr + j * CL < full_to; ++j) {
            if (MODE == 2) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
            tile(BoolTag<true>(), j);
            if (MODE == 2) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        }
        if (j < mine) {
            tile(BoolTag<false>(), j);
            ++j;
        }
    }
    if (BY_STAGE) tma_store_wait_read();
    __syncthreads();
    if (MODE == 1) {
        if (tid < CG) {                          // the chunk's map
            float *mp = maps + ((int64_t)unit * chunks + chunk) * 3 * CG;
            mp[tid] = carry_a[ntiles & 1][tid];
            mp[CG + tid] = carry[ntiles & 1][0][tid];
            mp[2 * CG + tid] = carry[ntiles & 1][1][tid];
        }
    } else {
        if (WPP > 1 && mine > 0) wide_bounds(mine - 1);
        if (a.absmax) {
            // the head's largest |stored key| (both copies): non-negative floats order like their bit patterns
            const unsigned m = __reduce_max_sync(FULLMASK, __float_as_uint(round_storage<T>(amax)));
            if (lane == 0 && m != 0u) {
                atomicMax(reinterpret_cast<unsigned *>(a.absmax) + bh, m);
                atomicMax(reinterpret_cast<unsigned *>(a.absmax) + (int64_t)a.B * a.H + bh, m);
            }
        }
    }
    if (!ok) {                                   // a wait ran out: no copy may still be on its way when the CTA exits
        atomicCAS(a.status, RQ_OK, RQ_ERR_TIMEOUT);
        if (MODE != 3 && tid == 0)
            for (int j = max(0, mine - NST); j < mine; ++j) mbar_wait(&full[j % NST], (uint32_t)((j / NST) & 1));
        __syncwarp();
    }
    if (CL > 1) cl.sync();                       // nobody's shared memory is written any more
}

// The state entering every chunk from the chunks' maps, in order.  Grid: channel groups; a thread per (k or v, channel).
__global__ void scan_chain_kernel(const float *state, int D, int gph, int chunks, const float *maps, float *entry, float *state_copy)
{
    const int unit = blockIdx.x, kv = threadIdx.x / CG, ch = threadIdx.x % CG;
    const int bh = unit / gph, c0 = (unit % gph) * CG;
    float s = state[(int64_t)bh * 2 * D + kv * D + c0 + ch];
    state_copy[(int64_t)bh * 2 * D + kv * D + c0 + ch] = s;
    for (int c = 0; c + 1 < chunks; ++c) {
        const float *mp = maps + ((int64_t)unit * chunks + c) * 3 * CG;
        s = fmaf(mp[ch], s, mp[(1 + kv) * CG + ch]);
        entry[(((int64_t)unit * chunks + c + 1) * 2 + kv) * CG + ch] = s;
    }
}

template <typename T, typename G, int D, int S, int MODE, bool STAGED>
cudaError_t start(const ScanArgs &a, const ScanMaps &tm, const ScanPlan &p, int cl, float *maps, const float *entry, int smem, cudaStream_t s)
{
    static bool ready[64];                                       // (set up form by form: the first use of a kernel loads it)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!ready[dev]) {
        e = cudaFuncSetAttribute(scan_kernel<T, G, D, S, MODE, STAGED>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        ready[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)(MODE == 2 ? D / CG : cl);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(p.units * p.chunks * cl));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    // (CTAs that are no cluster are launched as none: as clusters of one, 64 heads x 128 of 50000 tokens took 950 us, so 752)
    const bool clusters = MODE == 2 || cl > 1;
    cfg.attrs = clusters ? at : at + 1;
    cfg.numAttrs = clusters ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, scan_kernel<T, G, D, S, MODE, STAGED>, a, tm, p, maps, entry);
}

template <typename T, typename G, int D, int S>
cudaError_t run(const ScanArgs &a, cudaStream_t s)
{
    const int64_t end = a.len0 + a.T;
    const int64_t t0 = a.len0 / TT;
    const int64_t t1 = (end + TT - 1) / TT;
    if (t1 <= t0) return cudaSuccess;
    if (t1 - t0 >= (int64_t)1 << 31) return cudaErrorInvalidValue;
    const int64_t units = (int64_t)a.B * a.H * (D / CG);
    if (units >= (int64_t)1 << 28) return cudaErrorInvalidValue;
    constexpr int DSM = scan_stages<T, G>() * scan_stage_bytes<T, G>();
    cudaError_t e;
    ScanPlan p;
    p.tile0 = t0;
    p.ntiles = (int)(t1 - t0);
    p.units = (int)units;
    alignas(64) ScanMaps tm;
    const int sms = sm_count();
    // A call inside one tile with more units than SMs: its CTAs follow one another, and what counts is how soon a CTA is done.
    // 256 heads x 128, bf16, 16 / 100 / 255 tokens: one CTA per SM and tensor maps 25.3 / 26.6 / 30.8 us, two CTAs and plain
    // loads 17.8 / 21.4 / 30.1 (copies of 16 bytes by all threads, before there were tensor maps, 22.0 / 23.9 / 31.9).  With
    // fewer units the tensor maps win: 32 heads, 16 / 255 tokens 4.4 / 6.2 against 4.8 / 7.5.
    const bool brief = p.ntiles == 1 && units > sms;
    const bool shared = !brief && ((a.H > 1 && a.sh == 0) || (a.B > 1 && a.sb == 0));
    // tensor maps where the strides can be described (positions that are all the same, a stride of zero, cannot)
    p.tma = !brief && a.T < ((int64_t)1 << 31) &&
            prompt_tensor_map(&tm.k, a.k, sizeof(T), D, a.H, a.T, a.B, a.sh, a.st, a.sb, CG, TT) == cudaSuccess &&
            prompt_tensor_map(&tm.v, a.v, sizeof(T), D, a.H, a.T, a.B, a.sh, a.st, a.sb, CG, TT) == cudaSuccess &&
            prompt_tensor_map(&tm.g, a.g, sizeof(G), D, a.H, a.T, a.B, a.sh, a.st, a.sb, CG, TT) == cudaSuccess &&
            page_tensor_map(&tm.cache, a.kv, sizeof(T), D, S, (int64_t)a.B * a.H * a.page_cap, CG, 2 * RT) == cudaSuccess;
    // Time chunks: as many as give every SM a CTA, of at least 16 tiles and within the scratch.  They read the inputs
    // twice, so they only pay where they are at least seven (4 heads x 128, 131072 tokens: 223 us; a cluster of four, bound
    // by its hops of about 0.55 us, 290).  Otherwise as many CTAs per unit as leave every SM at most one, with at least four
    // tiles each (8 heads, 131072 tokens: 469 -> 283 us; 16 heads: 913 -> 543; clusters of eight find too little room: 386 for
    // the 4 heads).
    int cl = 1, chunks = 1;
    if (a.chunk_scratch && 2 * units <= sms) {
        chunks = sms / p.units;
        if (chunks > p.ntiles / 16) chunks = p.ntiles / 16;
        while (chunks > 1 && (size_t)p.units * (chunks * 5 + 2) * CG * sizeof(float) > kScanScratchBytes) --chunks;
    }
    if (chunks < 7) {
        chunks = 1;
        while (cl < kMaxCluster && 2 * cl * units <= sms && p.ntiles >= 8 * cl) cl *= 2;
    }
    // Long prompts of nearly as many units as SMs are bound by DRAM, and it likes a head's units, neighbours in every row,
    // together: 32 heads, 131072 tokens 923 -> 900 us.  Short ones lose by the barriers (4001 tokens 41.0 -> 42.1), and so
    // would more units than the clusters find room for at once.
    const bool abreast = cl == 1 && chunks == 1 && p.ntiles >= 64 && 9 * units <= 8 * sms;
    p.chunk_tiles = (p.ntiles + chunks - 1) / chunks;
    p.chunks = (p.ntiles + p.chunk_tiles - 1) / p.chunk_tiles;
    // Rows of 2-byte elements go out by their stage (32 heads x 128, 131072 tokens: 973 -> 956 us).  Rows of 4 bytes, in stages of
    // which only two find room, do so where enough CTAs with enough tiles wait for DRAM, which then has whole pages written
    // side by side; elsewhere the refill would wait for them.  us, straight from registers / by their stage: fp32 gates, 32
    // heads x 128, 50000 tokens 777 / 670 (by 16-byte pieces through shared memory, before, 675), 8 heads 201 / 172, 24 heads
    // 537 / 578, 32 heads of 2000 tokens 31 / 33; bf16 gates, 32 heads, 60000 tokens 0.86 / 0.93 of the speed before, 64 heads
    // of 64 pages 1.02 / 0.98.
    const int64_t ctas = units * cl * p.chunks;
    const bool staged = p.ntiles >= 12 * cl * p.chunks && 5 * ctas >= 4 * sms && (sizeof(G) == 4 || ctas <= sms);
    float *maps = a.chunk_scratch, *entry = a.chunk_scratch ? a.chunk_scratch + (size_t)units * p.chunks * 3 * CG : nullptr;
    if (p.chunks > 1) {
        e = start<T, G, D, S, 1, sizeof(T) == 2>(a, tm, p, 1, maps, entry, DSM, s);
        if (e != cudaSuccess) return e;
        scan_chain_kernel<<<(unsigned)units, 2 * CG, 0, s>>>(a.state, D, D / CG, p.chunks, maps, entry, entry + (size_t)units * p.chunks * 2 * CG);
    }
    auto go = [&](auto staged) {
        constexpr bool ST = decltype(staged)::value;
        return abreast ? start<T, G, D, S, 2, ST>(a, tm, p, 1, maps, entry, DSM, s) : start<T, G, D, S, 0, ST>(a, tm, p, cl, maps, entry, DSM, s);
    };
    if (brief) e = start<T, G, D, S, 3, false>(a, tm, p, 1, maps, entry, 0, s);
    else if (shared) e = start<T, G, D, S, 4, sizeof(T) == 2>(a, tm, p, cl, maps, entry, DSM, s);
    else if constexpr (sizeof(T) == 2) e = go(BoolTag<true>());
    else e = staged ? go(BoolTag<true>()) : go(BoolTag<false>());
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T, typename G>
cudaError_t dispatch_shape(const ScanArgs &a, cudaStream_t s)
{
    if (a.D == 128 && a.S == 16) return run<T, G, 128, 16>(a, s);
    if (a.D == 128 && a.S == 64) return run<T, G, 128, 64>(a, s);
    if (a.D == 64 && a.S == 16) return run<T, G, 64, 16>(a, s);
    if (a.D == 64 && a.S == 64) return run<T, G, 64, 64>(a, s);
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_scan(const ScanArgs &a, cudaStream_t s)
{
    if (a.dtype == RQ_BF16) {
        return a.gate_dtype == RQ_BF16 ? dispatch_shape<bf16, bf16>(a, s) : dispatch_shape<bf16, float>(a, s);
    }
    return a.gate_dtype == RQ_BF16 ? dispatch_shape<float, bf16>(a, s) : dispatch_shape<float, float>(a, s);
}

}  // namespace rq
