// tiles.cu -- bin construction for EXACT mode (Sec. 3.3; supplement Alg. 3),
// arranged for GB300.  With the monotone split map every entry of a Gaussian
// falls in the same bin b(z_g), so:
//
//   1. count[t, b]: each Gaussian adds its tile rect to layer b of a stack of
//      K 2D difference arrays over the tile grid (four atomics per Gaussian
//      instead of one per entry); per-layer 2D prefix sums give the counts;
//   2. exclusive scan of count in tile-major, bin-minor order -> bin offsets
//      (the same array Alg. 3's global count/scan produces);
//   3. scatter: each entry takes a slot in its (t, b) segment from an atomic
//      cursor -- straight from the Gaussians' rects (warp-cooperative
//      expansion, the emission-order entries are never written) or from
//      materialised entries.
//
// The order inside a segment is left to the repair (Alg. 4): an eager sort of
// every segment, or the raster's in-shared-memory sort of each segment it
// reaches (segments too long for its buffer are sorted here, eagerly).
#include "device.cuh"
#include "offsets.cuh"
#include "rows.cuh"
#include "scan.cuh"

namespace gs {

// ------------------------------------------------------------------ counts
// Per visible Gaussian: its bin (kept in gbin) and its rect added to layer b.
__global__ void __launch_bounds__(256)
k_bin_diff(const uint2* __restrict__ rect, const float4* __restrict__ c_o_z, int64_t n, int tiles_x, int tiles_y,
           const BinParams* __restrict__ bp, int K, int32_t* __restrict__ D, uint8_t* __restrict__ gbin)
{
    __shared__ float s_split[GS_MAX_K];
    for (int k = threadIdx.x; k < K - 1; k += blockDim.x) s_split[k] = bp->splits[k];
    __syncthreads();
    const int W1 = tiles_x + 1;
    const int64_t layer = (int64_t)(tiles_y + 1) * W1;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += stride) {
        const uint2 r = rect[g];
        const int tx0 = r.x & 0xffff, ty0 = r.x >> 16, tx1 = r.y & 0xffff, ty1 = r.y >> 16;
        if (tx0 >= tx1 || ty0 >= ty1) continue;
        const int b = bin_split(c_o_z[g].z, s_split, K);
        gbin[g] = (uint8_t)b;
        int32_t* L = D + b * layer;
        atomicAdd(&L[ty0 * W1 + tx0], 1);
        atomicAdd(&L[ty0 * W1 + tx1], -1);
        atomicAdd(&L[ty1 * W1 + tx0], -1);
        atomicAdd(&L[ty1 * W1 + tx1], 1);
    }
}

// One block per layer: 2D inclusive prefix (columns, then rows) in place.
__global__ void __launch_bounds__(1024)
k_layer_prefix(int32_t* __restrict__ D, int tiles_x, int tiles_y)
{
    const int W1 = tiles_x + 1;
    int32_t* L = D + (int64_t)blockIdx.x * (tiles_y + 1) * W1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int x = threadIdx.x; x < tiles_x; x += blockDim.x) {
        int32_t run = 0;
        for (int y = 0; y < tiles_y; ++y) {
            run += L[y * W1 + x];
            L[y * W1 + x] = run;
        }
    }
    __syncthreads();
    for (int y = warp; y < tiles_y; y += blockDim.x / 32) {
        int32_t carry = 0;
        for (int x0 = 0; x0 < tiles_x; x0 += 32) {
            const int x = x0 + lane;
            int32_t v = x < tiles_x ? L[y * W1 + x] : 0;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int32_t u = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += u;
            }
            if (x < tiles_x) L[y * W1 + x] = carry + v;
            carry += __shfl_sync(0xffffffffu, v, 31);
        }
    }
}

// ------------------------------------------------------------------ row spans (tile cull): rows.cuh

struct LoadRectRows {
    const uint2* rect;
    __device__ int64_t operator()(int64_t i) const
    {
        const uint2 r = rect[i];
        const int64_t w = (int64_t)(r.y & 0xffffu) - (int64_t)(r.x & 0xffffu);
        const int64_t h = (int64_t)(r.y >> 16) - (int64_t)(r.x >> 16);
        return (w > 0 && h > 0) ? h : 0;
    }
};

// Warp-cooperative over (Gaussian, row) pairs (warp_row_spans): a warp owns 32
// consecutive Gaussians, whose rows are consecutive records [roff[g0], roff[g0
// + 32)).  Per record the row's culled span, the record (gid, row | start,
// width), and +1 / -1 at the span ends of layer b's row (a per-row difference
// array).
__global__ void __launch_bounds__(256, kRowBlocks)
k_row_spans(const uint2* __restrict__ rect, int64_t n, const int32_t* __restrict__ roff, CullArgs ca, int tiles_x,
            const BinParams* __restrict__ bp, int K, const int64_t* __restrict__ m_dev, int64_t m_cap,
            int32_t* __restrict__ Drow, int64_t layer, uint8_t* __restrict__ gbin, RowRecords rs)
{
    grid_dependency_sync();
    __shared__ float s_split[GS_MAX_K];
    __shared__ RowOwners s_own[8];
    for (int k = threadIdx.x; k < K - 1; k += blockDim.x) s_split[k] = bp->splits[k];
    __syncthreads();
    if (*m_dev > m_cap) return;
    const int64_t g0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 32;
    if (g0 >= n) return;
    const int64_t gl = g0 + (threadIdx.x & 31);
    const int32_t off = roff[gl < n ? gl : n], next = roff[gl + 1 < n ? gl + 1 : n];
    uint2 r = make_uint2(0u, 0u);
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f), q = p;
    float margin = 0.0f;
    uint32_t bin = 0u;
    if (next > off) {
        r = rect[gl];
        p = __ldg(ca.xy_ab + gl);
        q = __ldg(ca.c_o_z + gl);
        margin = __ldg(&ca.rgb[gl].w);
        bin = (uint32_t)bin_split(q.z, s_split, K);
        gbin[gl] = (uint8_t)bin;
    }
    const int W1 = tiles_x + 1;
    warp_row_spans(s_own[threadIdx.x >> 5], g0, off, next, __shfl_sync(0xffffffffu, off, 0),
                   __shfl_sync(0xffffffffu, next, 31), r, p, q, margin, bin, 0, ca.tile, rs,
                   [&](uint32_t b, uint32_t, int ty) { return Drow + b * layer + ty * W1; });
}

// One block per layer: inclusive prefix along each row.
__global__ void __launch_bounds__(1024)
k_layer_rows_prefix(int32_t* __restrict__ D, int tiles_x, int tiles_y, int64_t layer)
{
    grid_dependency_sync();
    const int W1 = tiles_x + 1;
    int32_t* L = D + (int64_t)blockIdx.x * layer;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int y = warp; y < tiles_y; y += blockDim.x / 32) {
        int32_t carry = 0;
        for (int x0 = 0; x0 < tiles_x; x0 += 32) {
            const int x = x0 + lane;
            int32_t v = x < tiles_x ? L[y * W1 + x] : 0;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int32_t u = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += u;
            }
            if (x < tiles_x) L[y * W1 + x] = carry + v;
            carry += __shfl_sync(0xffffffffu, v, 31);
        }
    }
}

// What a planned frame's pass can tell of a record from its tile row, bin and
// span alone, by the block, so that most records it drops are dropped on their
// first word: a first pass the bins below the row's largest plan, a completing
// pass the bins from the row's smallest plan of a flagged tile on, and there
// the spans that meet a flagged tile (one bit a tile, for frames of up to
// kMaskWords * 32 tiles).
constexpr int kMaxRows = 4096;  // row records hold 12 bits of tile row
constexpr int kMaskWords = 4096;
constexpr int kNoRow = 256;     // above every bin

// s_row[y] of every tile row; with mask, the flagged tiles (flagged = {count,
// tiles...}, a completing pass's).  Ends with a block barrier.
__device__ __forceinline__ void plan_rows(const ScatterPass& sp, int tiles_x, int tiles_y,
                                          const int32_t* __restrict__ flagged, int32_t* s_row, uint32_t* mask)
{
    const int words = (tiles_x + 31) / 32;
    if (sp.pass == 1) {  // a warp a row (32 atomics on one row's word before)
        const int lane = threadIdx.x & 31;
        for (int y = threadIdx.x >> 5; y < tiles_y; y += blockDim.x >> 5) {
            int m = 0;
#pragma unroll 8
            for (int x = lane; x < tiles_x; x += 32) m = max(m, (int)__ldg(sp.plan + (int64_t)y * tiles_x + x));
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) s_row[y] = m;
        }
        __syncthreads();
        return;
    }
    for (int y = threadIdx.x; y < tiles_y; y += blockDim.x) s_row[y] = kNoRow;
    if (mask)
        for (int q = threadIdx.x; q < tiles_y * words; q += blockDim.x) mask[q] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < flagged[0]; i += blockDim.x) {
        const int t = flagged[1 + i], y = t / tiles_x, x = t - y * tiles_x;
        atomicMin(&s_row[y], (int)__ldg(sp.plan + t));
        if (mask) atomicOr(&mask[y * words + (x >> 5)], 1u << (x & 31));
    }
    __syncthreads();
}

__device__ __forceinline__ bool plan_row_live(const ScatterPass& sp, const int32_t* s_row, uint32_t ya)
{
    const int b = (int)(ya >> 24), r = s_row[ya & 0xfffu];
    return sp.pass == 1 ? b < r : b >= r;
}

// whether tiles [x0, x0 + w) of row y (1 <= w) meet the mask
__device__ __forceinline__ bool mask_meets(const uint32_t* mask, int words, int y, int x0, int w)
{
    const int x1 = x0 + w - 1, q0 = x0 >> 5, q1 = x1 >> 5;
    for (int q = q0; q <= q1; ++q) {
        uint32_t m = mask[y * words + q];
        if (q == q0) m &= 0xffffffffu << (x0 & 31);
        if (q == q1) m &= 0xffffffffu >> (31 - (x1 & 31));
        if (m) return true;
    }
    return false;
}

// The tile a pass keeps of a record (ScatterPass::keep), from the lane that
// holds it in the warp's shared copy of the row words.
struct KeepPlanned {
    const ScatterPass& sp;
    const uint32_t* ya;
    int tiles_x;
    __device__ __forceinline__ bool operator()(int o, uint32_t d) const
    {
        const uint32_t r = ya[o];
        return sp.keep((int64_t)(r & 0xfffu) * tiles_x + ((r >> 12) & 0xfffu) + d, (int)(r >> 24));
    }
};

// The scatter of a frame's row records (rows.cuh).  PLANNED: one pass of a
// planned frame, which drops the records and entries it does not take.
template <bool PLANNED>
__global__ void __launch_bounds__(256)
k_bin_scatter_rows(const uint32_t* __restrict__ rs_g, const uint32_t* __restrict__ rs_ya, const uint32_t* __restrict__ rs_w,
                   const uint32_t* __restrict__ rs_z, const int32_t* __restrict__ roff, int64_t n, int tiles_x, int tiles_y,
                   const int64_t* __restrict__ m_dev, int64_t m_cap, const Cursors cur,
                   uint64_t* __restrict__ words, const ScatterPass sp, const int32_t* __restrict__ flagged)
{
    grid_dependency_sync();
    __shared__ ScatterShared s_sc[8];
    __shared__ uint32_t s_ya[PLANNED ? 8 : 1][32], s_queue[PLANNED ? 8 : 1][160];
    __shared__ int32_t s_row[PLANNED ? kMaxRows : 1];
    __shared__ uint32_t s_mask[PLANNED ? kMaskWords : 1];
    if (*m_dev > m_cap) return;
    if (PLANNED && sp.pass == 2 && flagged[0] == 0) return;  // no tile to complete
    const int mwords = (tiles_x + 31) / 32;
    const bool masked = PLANNED && sp.pass == 2 && tiles_y * mwords <= kMaskWords;
    if constexpr (PLANNED) plan_rows(sp, tiles_x, tiles_y, flagged, s_row, masked ? s_mask : nullptr);
    const int64_t R = roff[n];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nchunks = (R + 31) / 32;
    const int64_t w0 = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp, wstride = (int64_t)gridDim.x * (blockDim.x >> 5);
    // records read once: streamed past L2
    auto first_slot = [&](uint32_t ya) {
        return (uint32_t)(((int64_t)(ya & 0xfffu) * tiles_x + ((ya >> 12) & 0xfffu)) * cur.tile +
                          (int64_t)(ya >> 24) * cur.bin);
    };
    if constexpr (PLANNED) {
        // Few records are taken (138 us with each warp placing its
        // chunks of 32 as they came, 84 now, 4M Gaussians): a warp looks at
        // the row words of 128 at a time, the next ones' on their way, queues
        // those their row, bin and span do not drop, and places them 32 by 32.
        uint32_t* queue = s_queue[warp];
        int queued = 0;
        auto place = [&](int first, int count) {
            uint32_t w = 0, g = 0, ya = 0, z = 0;
            if (lane < count) {
                const uint32_t k = queue[first + lane];
                ya = rs_ya[k];
                w = rs_w[k];
                sp.trim(ya, w, tiles_x);
                if (w != 0u) {
                    g = rs_g[k];
                    z = rs_z[k];
                }
            }
            if (!__any_sync(0xffffffffu, w != 0u)) return;
            s_ya[warp][lane] = ya;  // read after the warp barriers of the scatter
            scatter_row_records(w, g, z, first_slot(ya), (uint32_t)cur.tile, cur.p, words, s_sc[warp],
                                KeepPlanned{sp, s_ya[warp], tiles_x});
        };
        auto load = [&](const uint32_t* words, int64_t c) {
            const int64_t k = c * 128 + 4 * lane;  // the words past R are allocated and not looked at
            return k < R ? *reinterpret_cast<const uint4*>(words + k) : make_uint4(0u, 0u, 0u, 0u);
        };
        uint4 next = load(rs_ya, w0), next_w = masked ? load(rs_w, w0) : next;
        for (int64_t c = w0; c * 128 < R; c += wstride) {
            const int64_t k0 = c * 128 + 4 * lane;
            const uint32_t rows[4] = {next.x, next.y, next.z, next.w};
            const uint32_t wide[4] = {next_w.x, next_w.y, next_w.z, next_w.w};
            next = load(rs_ya, c + wstride);
            if (masked) next_w = load(rs_w, c + wstride);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                bool live = k0 + u < R && plan_row_live(sp, s_row, rows[u]);
                if (live && masked)
                    live = wide[u] != 0u && mask_meets(s_mask, mwords, (int)(rows[u] & 0xfffu),
                                                       (int)((rows[u] >> 12) & 0xfffu), (int)wide[u]);
                const unsigned m = __ballot_sync(0xffffffffu, live);
                if (live) queue[queued + __popc(m & ((1u << lane) - 1u))] = (uint32_t)(k0 + u);
                queued += __popc(m);
            }
            __syncwarp();
            while (queued >= 32) {
                queued -= 32;
                place(queued, 32);
            }
            __syncwarp();  // the queue is read before it is written again
        }
        place(0, queued);
    } else {
        for (int64_t c = w0; c < nchunks; c += wstride) {
            uint32_t w = 0, g = 0, ya = 0, z = 0;
            const int64_t k = c * 32 + lane;
            if (k < R) {
                ya = __ldcs(rs_ya + k);
                w = __ldcs(rs_w + k);
                g = __ldcs(rs_g + k);
                z = __ldcs(rs_z + k);
            }
            scatter_row_records(w, g, z, first_slot(ya), (uint32_t)cur.tile, cur.p, words, s_sc[warp], KeepAll());
        }
    }
}

// The completing pass's cursors: those of every flagged tile start at its
// segment offsets (the first pass placed none of the bins it leaves).
__global__ void k_flagged_cursors(const int32_t* __restrict__ list, const int32_t* __restrict__ offsets, int K,
                                  const Cursors cur)
{
    grid_dependency_sync();
    const int32_t nl = list[0];
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nl * K; i += gridDim.x * blockDim.x) {
        const int32_t t = list[1 + i / K];
        *cur.at(t, i % K) = offsets[(int64_t)t * K + i % K];
    }
}

// ------------------------------------------------------------------ scatter by (row, bin) groups
// For deep frames the per-entry cursor atomics in global memory are the
// bin construction's limit.  Here the row records are first grouped by
// (tile row, bin) -- a counting pass and a writing pass over C slices of the
// records with block histograms in shared memory, one scan in between -- and
// then one block per group holds the cursors of that row's tiles for that bin
// (tiles_x words) and takes every slot with a shared-memory atomic.
constexpr int kGroupThreads = 1024;
template <bool PLANNED>
constexpr int kGroupIF = PLANNED ? 2 : 8;  // records a thread has in flight
constexpr int kMaxGroupKeys = 12288;  // (tile row, bin) keys in 48 KB of shared memory
// reserved entries per tile from which the grouped scatter is used: measured
// slower at ~3k (1M Gaussians, 1080p: bin stage 0.228 vs 0.210 ms), faster at
// ~19k (3M, 1080p: 0.60 vs 0.83 ms) and ~43k (6M, 4K: 3.74 vs 7.6 ms)
constexpr int64_t kGroupedMinPerTile = 8192;

__host__ __device__ inline int group_slices(int num_sms) { return 2 * num_sms; }

// the record slice [r0, r1) of slice c out of C
__device__ __forceinline__ void record_slice(int64_t R, int C, int c, int64_t* r0, int64_t* r1)
{
    *r0 = R * c / C;
    *r1 = R * (c + 1) / C;
}

// key of a row record: (tile row, bin)
__device__ __forceinline__ int group_key(uint32_t ya, int K) { return (int)(ya & 0xfffu) * K + (int)(ya >> 24); }

// The record words and widths of records k0 + u kGroupThreads, the width 0 when
// the pass drops one or it lies past r1.  Several in flight: both passes wait
// on their loads (one a thread and round: count 31 us and
// write 124, eight 26 and 104; planned passes, whose records mostly drop on the
// row word, 66 and 66, two 52 and 54).
template <bool PLANNED>
__device__ __forceinline__ void group_records(const uint32_t* __restrict__ rs_ya, const uint32_t* __restrict__ rs_w,
                                              int64_t k0, int64_t r1, const ScatterPass& sp, const int32_t* s_row,
                                              int tiles_x, uint32_t (&ya)[kGroupIF<PLANNED>], uint32_t (&w)[kGroupIF<PLANNED>])
{
#pragma unroll
    for (int u = 0; u < kGroupIF<PLANNED>; ++u) {
        const int64_t k = k0 + u * kGroupThreads;
        ya[u] = k < r1 ? rs_ya[k] : 0u;
        w[u] = !PLANNED && k < r1 ? rs_w[k] : 0u;
    }
    if constexpr (PLANNED) {
        // most records are dropped on their row word
#pragma unroll
        for (int u = 0; u < kGroupIF<PLANNED>; ++u) {
            const int64_t k = k0 + u * kGroupThreads;
            if (k < r1 && plan_row_live(sp, s_row, ya[u])) w[u] = rs_w[k];
        }
#pragma unroll
        for (int u = 0; u < kGroupIF<PLANNED>; ++u)
            if (w[u] != 0u) sp.trim(ya[u], w[u], tiles_x);
    }
}

// pass 1: H[key * C + c] = non-empty records of slice c with that key
template <bool PLANNED>
__global__ void __launch_bounds__(kGroupThreads)
k_group_count(const uint32_t* __restrict__ rs_ya, const uint32_t* __restrict__ rs_w, const int32_t* __restrict__ roff,
              int64_t n, int K, int nkeys, const int64_t* __restrict__ m_dev, int64_t m_cap, int32_t* __restrict__ H,
              const ScatterPass sp, int tiles_x)
{
    grid_dependency_sync();
    extern __shared__ int32_t s_h[];
    __shared__ int32_t s_row[PLANNED ? kMaxRows : 1];
    const int C = gridDim.x, c = blockIdx.x;
    for (int i = threadIdx.x; i < nkeys; i += blockDim.x) s_h[i] = 0;
    if (PLANNED) plan_rows(sp, tiles_x, nkeys / K, nullptr, s_row, nullptr);
    __syncthreads();
    if (*m_dev <= m_cap) {
        int64_t r0, r1;
        record_slice(roff[n], C, c, &r0, &r1);
        for (int64_t k0 = r0 + threadIdx.x; k0 < r1; k0 += kGroupIF<PLANNED> * kGroupThreads) {
            uint32_t ya[kGroupIF<PLANNED>], w[kGroupIF<PLANNED>];
            group_records<PLANNED>(rs_ya, rs_w, k0, r1, sp, s_row, tiles_x, ya, w);
#pragma unroll
            for (int u = 0; u < kGroupIF<PLANNED>; ++u)
                if (w[u] != 0u) atomicAdd(&s_h[group_key(ya[u], K)], 1);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nkeys; i += blockDim.x) H[(int64_t)i * C + c] = s_h[i];
}

// pass 2: list[Hs[key * C + c] + rank] = the record {gid, row word, width,
// depth bits} (any order within a key), so the scatter reads its group
// contiguously
template <bool PLANNED>
__global__ void __launch_bounds__(kGroupThreads)
k_group_write(const uint32_t* __restrict__ rs_g, const uint32_t* __restrict__ rs_ya,
              const uint32_t* __restrict__ rs_w, const uint32_t* __restrict__ rs_z, const int32_t* __restrict__ roff,
              int64_t n, int K, int nkeys, const int64_t* __restrict__ m_dev, int64_t m_cap,
              const int32_t* __restrict__ Hs, uint4* __restrict__ list, const ScatterPass sp, int tiles_x)
{
    grid_dependency_sync();
    extern __shared__ int32_t s_h[];  // [nkeys] next slot, from the slice's base
    __shared__ int32_t s_row[PLANNED ? kMaxRows : 1];
    const int C = gridDim.x, c = blockIdx.x;
    if (*m_dev > m_cap) return;
    for (int i = threadIdx.x; i < nkeys; i += blockDim.x) s_h[i] = Hs[(int64_t)i * C + c];
    if (PLANNED) plan_rows(sp, tiles_x, nkeys / K, nullptr, s_row, nullptr);
    __syncthreads();
    int64_t r0, r1;
    record_slice(roff[n], C, c, &r0, &r1);
    for (int64_t k0 = r0 + threadIdx.x; k0 < r1; k0 += kGroupIF<PLANNED> * kGroupThreads) {
        uint32_t ya[kGroupIF<PLANNED>], w[kGroupIF<PLANNED>], g[kGroupIF<PLANNED>], z[kGroupIF<PLANNED>];
        group_records<PLANNED>(rs_ya, rs_w, k0, r1, sp, s_row, tiles_x, ya, w);
#pragma unroll
        for (int u = 0; u < kGroupIF<PLANNED>; ++u) {
            if (w[u] == 0u) continue;
            g[u] = __ldcs(rs_g + k0 + u * kGroupThreads);
            z[u] = __ldcs(rs_z + k0 + u * kGroupThreads);
        }
#pragma unroll
        for (int u = 0; u < kGroupIF<PLANNED>; ++u)
            if (w[u] != 0u) list[atomicAdd(&s_h[group_key(ya[u], K)], 1)] = make_uint4(g[u], ya[u], w[u], z[u]);
    }
}

// one block per (tile row, bin): that bin's cursor of every tile of the row
// (NT = 1024 threads: the groups' sizes vary widely, and the largest bound the
// kernel's tail: 217 us, with 512 threads 277, for 3M Gaussians seen from
// inside a cluster; 512 in a planned first pass, most of whose groups are
// empty: 45 us against 97 at 2560 x 1440); a thread takes a record and walks
// its span of tiles (two records at a time in flight: 302 us)

template <int NT>
__global__ void __launch_bounds__(NT)
k_scatter_groups(const uint4* __restrict__ list, const int32_t* __restrict__ Hs, int C,
                 const int32_t* __restrict__ offsets, int tiles_x, int K, const int64_t* __restrict__ m_dev,
                 int64_t m_cap, uint64_t* __restrict__ words, const ScatterPass sp,
                 const int32_t* __restrict__ flagged)
{
    grid_dependency_sync();
    extern __shared__ int32_t s_cur[];  // [tiles_x]
    const int key = blockIdx.x;
    if (*m_dev > m_cap) return;
    if (sp.pass == 2 && flagged[0] == 0) return;  // no tile to complete
    const int ty = key / K, b = key - ty * K;
    const int32_t L0 = Hs[(int64_t)key * C], L1 = Hs[(int64_t)(key + 1) * C];
    if (L1 <= L0) return;
    // the first records are on their way while the cursors are
    int32_t i = L0 + (int32_t)threadIdx.x;
    uint4 next = i < L1 ? __ldcs(list + i) : make_uint4(0u, 0u, 0u, 0u);
    int any = 0;
    for (int x = threadIdx.x; x < tiles_x; x += blockDim.x) {
        const int64_t t = (int64_t)ty * tiles_x + x;
        s_cur[x] = offsets[t * K + b];
        any |= sp.keep(t, b) ? 1 : 0;
    }
    // a planned pass skips the groups no tile of the row takes in this pass
    if (!__syncthreads_or(any)) return;
    while (i < L1) {
        const uint4 rec = next;
        i += NT;
        if (i < L1) next = __ldcs(list + i);
        const uint64_t word = ((uint64_t)rec.w << 32) | rec.x;
        const int a = (int)((rec.y >> 12) & 0xfffu);
        for (int j = 0; j < (int)rec.z; ++j) {
            if (!sp.keep((int64_t)ty * tiles_x + a + j, b)) continue;
            const int32_t slot = atomicAdd(&s_cur[a + j], 1);
            words[slot] = word;
        }
    }
}

// ------------------------------------------------------------------ scatter
// Without the tile cull: straight from the rects with the warp-cooperative
// expansion, four entries per lane in flight so the returning atomics overlap.
__global__ void __launch_bounds__(256)
k_bin_scatter_rects(const uint2* __restrict__ rect, const float4* __restrict__ c_o_z,
                    const int32_t* __restrict__ goff, const uint8_t* __restrict__ gbin, int64_t n, int tiles_x,
                    int K, const int64_t* __restrict__ m_dev, int64_t m_cap, const int32_t* __restrict__ off,
                    int32_t* __restrict__ cur, uint64_t* __restrict__ words)
{
    if (*m_dev > m_cap) return;  // capacity error raised by the caller's check
    const int64_t g0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32;
    if (g0 >= n) return;
    const WarpExpand wx(rect, c_o_z, goff, n, g0);
    const int lane = threadIdx.x & 31;
    const int64_t gl = g0 + lane;
    const uint32_t mybin = (gl < n && ((wx.r1 & 0xffffu) > (wx.r0 & 0xffffu))) ? gbin[gl] : 0u;
    for (int32_t e0 = wx.base; e0 < wx.end; e0 += 128) {
        uint32_t g[4], t[4], z[4], b[4];
        int32_t p[4];
        bool live[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            wx.entry(e0 + 32 * u + lane, tiles_x, &g[u], &t[u], &z[u]);
            b[u] = __shfl_sync(0xffffffffu, mybin, (int)(g[u] - (uint32_t)g0) & 31);
            live[u] = e0 + 32 * u + lane < wx.end;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (live[u]) {
                const int64_t q = (int64_t)t[u] * K + b[u];
                p[u] = atomicAdd(&cur[q], 1);
            }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (live[u]) words[p[u]] = ((uint64_t)z[u] << 32) | g[u];
    }
}

// Count of segment q = t*K + b from the prefixed layers (tile-major order).
// count[t, b] from the layer-major row prefix D [b][y][x] into C [t][b]
// (t = y * tiles_x + x): 32 x 32 (x, b) blocks through shared memory, so both
// the reads (along x) and the writes (along b) are coalesced.
__global__ void __launch_bounds__(256)
k_transpose_counts(const int32_t* __restrict__ D, int tiles_x, int tiles_y, int K, int64_t layer,
                   int32_t* __restrict__ C)
{
    grid_dependency_sync();
    __shared__ int32_t s[32][33];
    const int y = blockIdx.z;
    const int x0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
    const int W1 = tiles_x + 1;
    const int lx = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < 32; r += blockDim.x >> 5) {
        const int b = b0 + r, x = x0 + lx;
        s[r][lx] = (b < K && x < tiles_x) ? D[b * layer + (int64_t)y * W1 + x] : 0;
    }
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < 32; r += blockDim.x >> 5) {
        const int x = x0 + r, b = b0 + lx;
        if (x < tiles_x && b < K) C[((int64_t)y * tiles_x + x) * K + b] = s[lx][r];
    }
}

// The tile rows of one frame (offsets.cuh).
struct FrameRows {
    const int32_t* D;
    int tiles_x, tiles_y, K;
    int64_t layer;
    __device__ __forceinline__ OffsetRow operator()(int y) const
    {
        return OffsetRow{D + (int64_t)y * (tiles_x + 1), layer, tiles_x, K, (int64_t)y * tiles_x * K,
                         (int64_t)y * tiles_x, (int64_t)tiles_x * tiles_y, y * tiles_x};
    }
};

struct LoadPlainCount {
    const int32_t* C;
    __device__ int64_t operator()(int64_t q) const { return C[q]; }
};

struct LoadLayerCount {
    const int32_t* D;
    int K, tiles_x, W1;
    int64_t layer;
    __device__ int64_t operator()(int64_t q) const
    {
        const int64_t t = q / K;
        const int b = (int)(q - t * K);
        const int y = (int)(t / tiles_x), x = (int)(t - (int64_t)y * tiles_x);
        return D[b * layer + (int64_t)y * W1 + x];
    }
};

__global__ void k_zero_if_over(const int64_t* __restrict__ m_dev, int64_t m_cap, int32_t* __restrict__ off, int64_t nq,
                               int* err)
{
    grid_dependency_sync();
    if (*m_dev <= m_cap) return;  // over capacity: empty stream, nothing out of bounds downstream
    if (blockIdx.x == 0 && threadIdx.x == 0) raise_error(err, GS_ERR_CAPACITY);
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += (int64_t)gridDim.x * blockDim.x)
        off[q] = 0;
}

// The grouped scatter pays off once the frame is deep: decided on the host
// from the reserved entry capacity per tile (the entry count itself lives on
// the device).
static bool grouped_scatter(int64_t m_cap, int64_t T)
{
    return T > 0 && m_cap / T >= kGroupedMinPerTile;
}

struct ExactScratch {
    int32_t* D;      // K layers of (tiles_y + 1) x (tiles_x + 1) difference counts
    int32_t* cur;    // T*K scatter cursors
    uint8_t* gbin;   // n per-Gaussian bins
    int32_t* roff;   // n + 1 row-record offsets
    uint32_t *rs_g, *rs_ya, *rs_w, *rs_z;  // row records (<= m_cap)
    int64_t* total;  // scratch count
    int32_t *H, *Hs; // per ((tile row, bin) key, slice) record counts and their exclusive scan
    uint4* list;     // the records grouped by key (<= m_cap)
};

static size_t exact_scratch(gs_ctx* ctx, int64_t n, int64_t m_cap, int32_t tiles_x, int32_t tiles_y, int K,
                            ExactScratch* v)
{
    const size_t layer = (size_t)(tiles_x + 1) * (tiles_y + 1);
    const size_t T = (size_t)tiles_x * tiles_y;
    const size_t mc = (size_t)(m_cap > 0 ? m_cap : 1), nn = (size_t)(n > 0 ? n : 1);
    const size_t nh = (size_t)tiles_y * K * group_slices(ctx->num_sms);
    const size_t sizes[] = {layer * K * 4, T * K * 4, nn, (nn + 1) * 4, mc * 4, mc * 4, mc * 4, mc * 4, 8,
                            nh * 4, (nh + 1) * 4, grouped_scatter(m_cap, (int64_t)T) ? mc * 16 : 16};
    size_t total = 0;
    for (size_t s : sizes) total += align256(s);
    if (v) {
        char* b = (char*)ctx->d_tiles;
        void** dst[] = {(void**)&v->D, (void**)&v->cur, (void**)&v->gbin, (void**)&v->roff, (void**)&v->rs_g,
                        (void**)&v->rs_ya, (void**)&v->rs_w, (void**)&v->rs_z, (void**)&v->total,
                        (void**)&v->H, (void**)&v->Hs, (void**)&v->list};
        for (int k = 0; k < 12; ++k) {
            *dst[k] = b;
            b += align256(sizes[k]);
        }
    }
    return total;
}

// items of the grouped scatter's count scan (for reserving the scan's sums)
int64_t group_scan_items(gs_ctx* ctx, int32_t tiles_y, int K)
{
    return (int64_t)tiles_y * K * group_slices(ctx->num_sms);
}

int exact_bins_reserve(gs_ctx* ctx, int64_t n, int64_t m_cap, int32_t tiles_x, int32_t tiles_y, int K)
{
    void* p = ctx->d_tiles;
    int r = ensure(&p, &ctx->tiles_cap, exact_scratch(ctx, n, m_cap, tiles_x, tiles_y, K, nullptr));
    ctx->d_tiles = (int32_t*)p;
    return r;
}

// The scatter's cursors: bin by bin where the one-pass offsets kernel writes
// them, tile by tile where the wide rows' scan does.
static Cursors cursors(const ExactScratch& v, int32_t tiles_x, int32_t tiles_y, int K)
{
    if (bin_offsets_smem(tiles_x, K) <= kOffMaxSmem) return Cursors{v.cur, 1, (int64_t)tiles_x * tiles_y};
    return Cursors{v.cur, K, 1};
}

// Whether a first-pass scatter takes the grouped path (records grouped by
// (tile row, bin), cursors in shared memory) rather than per-entry global
// cursors.
static bool grouped_path(int64_t m_cap, int32_t tiles_x, int32_t tiles_y, int K)
{
    return grouped_scatter(m_cap, (int64_t)tiles_x * tiles_y) && tiles_y * K <= kMaxGroupKeys;
}

// The record scatter of the tile-cull path, for one pass (grouped by (tile
// row, bin) on deep frames, else per-entry global cursors, which the offsets'
// kernels have set to the segment offsets before a first pass).
static int exact_scatter(gs_ctx* ctx, const ExactScratch& v, int64_t n, int32_t tiles_x, int32_t tiles_y, int K,
                         int64_t m_cap, const int64_t* m_dev, uint64_t* words, const int32_t* offsets,
                         const ScatterPass& sp, cudaStream_t st)
{
    const int nkeys = tiles_y * K;
    const unsigned g_sm = (unsigned)ctx->num_sms * 8;
    const int32_t* flagged = sp.pass ? ctx->d_plist : nullptr;
    if (n <= 0) return GS_OK;
    if (sp.pass != 2 && grouped_path(m_cap, tiles_x, tiles_y, K)) {
        // records grouped by (tile row, bin), then cursors in shared memory
        // (a planned first pass groups only the records it keeps)
        const int C = group_slices(ctx->num_sms);
        const size_t hsm = (size_t)nkeys * 4;
        GS_CUDA_TRY(launch_k(ctx, sp.pass ? k_group_count<true> : k_group_count<false>, (unsigned)C, kGroupThreads, hsm, st, v.rs_ya, v.rs_w, v.roff, n, K, nkeys, m_dev, m_cap,
                                                                v.H, sp, tiles_x));
        ctx->launches += 1;
        int r;
        if ((r = scan_impl(ctx, LoadI32{v.H}, (int64_t)nkeys * C, v.Hs, nullptr, st)) != GS_OK) return r;
        GS_CUDA_TRY(launch_k(ctx, sp.pass ? k_group_write<true> : k_group_write<false>, (unsigned)C, kGroupThreads, hsm, st, v.rs_g, v.rs_ya, v.rs_w, v.rs_z, v.roff, n, K, nkeys,
                                                                m_dev, m_cap, v.Hs, v.list, sp, tiles_x));
        GS_CUDA_TRY(launch_k(ctx, sp.pass ? k_scatter_groups<512> : k_scatter_groups<1024>, (unsigned)nkeys, sp.pass ? 512 : 1024, (size_t)tiles_x * 4, st, 
            v.list, v.Hs, C, offsets, tiles_x, K, m_dev, m_cap, words, sp, flagged));
        ctx->launches += 2;
    } else {
        // per-entry cursors in global memory: all of them from the offsets
        // before a first pass, those of the flagged tiles before the
        // completing pass (few entries: no grouping)
        const Cursors cur = cursors(v, tiles_x, tiles_y, K);
        if (sp.pass == 2) {
            GS_CUDA_TRY(launch_k(ctx, k_flagged_cursors, (unsigned)ctx->num_sms * 2, 256, 0, st, flagged, offsets, K, cur));
            ctx->launches += 1;
        }
        GS_CUDA_TRY(launch_k(ctx, sp.pass ? k_bin_scatter_rows<true> : k_bin_scatter_rows<false>, sp.pass ? g_sm : g_sm * 2, 256, 0, st, v.rs_g, v.rs_ya, v.rs_w, v.rs_z, v.roff, n, tiles_x, tiles_y,
                                                     m_dev, m_cap, cur, words, sp, flagged));
        ctx->launches += 1;
    }
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

// The regions a frame of the tile-cull EXACT path needs zeroed, so that no
// memset sits between its kernels: the frame's scan-flag arena (the row-count
// scan, the offsets scan and, on deep frames, the grouped scatter's count
// scan), the bin stage's difference counts, the counters of d_tail.  The projection (*fz) clears the row-count scan's flags, the
// depth-range sampling (ctx->late_*) the rest.  Reserves the scratch they
// live in.
int exact_frame_zero(gs_ctx* ctx, int64_t n, const gs_camera* cam, int64_t m_cap, FrameZero* fz)
{
    const int tile = ctx->cfg.tile_size, K = ctx->cfg.K;
    const int32_t tiles_x = (cam->width + tile - 1) / tile, tiles_y = (cam->height + tile - 1) / tile;
    const int64_t T = (int64_t)tiles_x * tiles_y, nseg = T * K;
    int r;
    if ((r = exact_bins_reserve(ctx, n, m_cap, tiles_x, tiles_y, K)) != GS_OK) return r;
    if ((r = bins_reserve(ctx, 1, nseg)) != GS_OK) return r;
    if (!ctx->capturing && !raster_resident(ctx, tile, T) && (r = tile_order_reserve(ctx, T)) != GS_OK) return r;
    ExactScratch v;
    exact_scratch(ctx, n, m_cap, tiles_x, tiles_y, K, &v);
    auto blocks = [](int64_t items) { return items > 0 ? (items + kScanTile - 1) / kScanTile : 1; };
    int64_t words = 2 * blocks(n) + (blocks(nseg) > tiles_y ? blocks(nseg) : tiles_y);
    if (grouped_path(m_cap, tiles_x, tiles_y, K))
        words += blocks((int64_t)tiles_y * K * group_slices(ctx->num_sms));
    if ((size_t)(words + 2) * sizeof(uint64_t) > ctx->scan_bytes) {
        if (ctx->capturing) return GS_OK;  // no allocation inside a capture: the scans clear their own flags
        if ((r = ensure(&ctx->d_scan, &ctx->scan_bytes, (size_t)(words + 2) * sizeof(uint64_t))) != GS_OK) return r;
    }
    const int64_t w2 = 2 * blocks(n);  // the row-count scan's flags: cleared by the projection
    fz->p[0] = static_cast<int32_t*>(ctx->d_scan);
    fz->n[0] = 2 * w2;
    ctx->late_p[0] = v.D;
    ctx->late_n[0] = (int64_t)(tiles_x + 1) * (tiles_y + 1) * K;
    ctx->late_p[1] = static_cast<int32_t*>(ctx->d_scan) + 2 * w2;
    ctx->late_n[1] = 2 * (words - w2);
    ctx->late_p[2] = ctx->d_tail;
    ctx->late_n[2] = kTailHead;
    ctx->scan_arena = words;
    ctx->scan_used = 0;
    ctx->scan_arena_bytes = ctx->scan_bytes;
    ctx->zeroed_D = v.D;
    ctx->zeroed_D_bytes = ctx->tiles_cap;
    ctx->zeroed_tail = ctx->d_tail;
    ctx->zeroed_tail_bytes = ctx->tail_cap;
    return GS_OK;
}

// The one-pass offsets kernel takes up to kOffMaxSmem of dynamic shared
// memory (tile rows of up to kOffMaxSmem / 4 / (K + 1) tiles): set once per
// context, on its device.
int bin_offsets_prepare()
{
    GS_CUDA_TRY(cudaFuncSetAttribute(k_bin_offsets<FrameRows>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kOffMaxSmem));
    // the planned grouping's keys and row table together pass 48 KB
    GS_CUDA_TRY(cudaFuncSetAttribute(k_group_count<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxGroupKeys * 4));
    GS_CUDA_TRY(cudaFuncSetAttribute(k_group_write<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxGroupKeys * 4));
    return group_offsets_prepare();
}

int exact_scatter_rest(gs_ctx* ctx, int64_t n, const gs_camera* cam, int64_t m_cap, const int64_t* m_dev,
                       uint64_t* words, const int32_t* offsets, cudaStream_t st)
{
    const int tile = ctx->cfg.tile_size, K = ctx->cfg.K;
    const int32_t tiles_x = (cam->width + tile - 1) / tile, tiles_y = (cam->height + tile - 1) / tile;
    ExactScratch v;
    exact_scratch(ctx, n, m_cap, tiles_x, tiles_y, K, &v);
    v.roff = ctx->exact_roff;  // the first pass's row records (the fused scan's offsets on the render path)
    ScatterPass sp;
    sp.plan = ctx->d_plan;
    sp.T = tiles_x * tiles_y;
    sp.pass = 2;
    return exact_scatter(ctx, v, n, tiles_x, tiles_y, K, m_cap, m_dev, words, offsets, sp, st);
}

// The frame's long segments and tile order go to d_tail and d_tiles_order.
TileOrder frame_tile_order(const gs_ctx* ctx, int64_t T)
{
    TileOrder o;
    if (raster_resident(ctx, ctx->cfg.tile_size, T) || ctx->order_cap < (size_t)T * kTileLists * 4) return o;
    o.count = ctx->d_tail;
    o.lists = ctx->d_tiles_order;
    o.stride = T;
    return o;
}

int tile_order_reserve(gs_ctx* ctx, int64_t T)
{
    void* p = ctx->d_tiles_order;
    const int r = ensure(&p, &ctx->order_cap, (size_t)T * kTileLists * 4);
    ctx->d_tiles_order = (int32_t*)p;
    return r;
}

int exact_bins(gs_ctx* ctx, const ProjView& pv, int64_t n, const gs_camera* cam, bool goff_ready, int64_t m_cap,
               const int64_t* m_dev, uint64_t* words, int32_t* offsets, cudaStream_t st, int32_t long_min,
               bool* long_listed, bool rows_ready, bool planned)
{
    *long_listed = false;
    ctx->tile_ordered = 0;
    const int tile = ctx->cfg.tile_size, K = ctx->cfg.K;
    const int32_t tiles_x = (cam->width + tile - 1) / tile, tiles_y = (cam->height + tile - 1) / tile;
    const int64_t T = (int64_t)tiles_x * tiles_y, nseg = T * K;
    int r;
    if ((r = exact_bins_reserve(ctx, n, m_cap, tiles_x, tiles_y, K)) != GS_OK) return r;
    ExactScratch v;
    exact_scratch(ctx, n, m_cap, tiles_x, tiles_y, K, &v);
    const size_t layer = (size_t)(tiles_x + 1) * (tiles_y + 1);
    if (tiles_x > 4096 || tiles_y > 4096) return GS_ERR_INVALID_ARG;  // row-record packing
    if (!(ctx->zeroed_D == v.D && ctx->zeroed_D_bytes == ctx->tiles_cap))
        GS_CUDA_TRY(cudaMemsetAsync(v.D, 0, layer * K * 4, st));
    ctx->zeroed_D = nullptr;  // zeroed by the frame's first kernel once, for this call
    const unsigned g_sm = (unsigned)ctx->num_sms * 8;
    if (ctx->cfg.tile_cull) {
        // rows of every rect, each row's culled span, per-row difference counts
        const int64_t rlayer = (int64_t)tiles_y * (tiles_x + 1);
        if (rows_ready && goff_ready) {
            v.roff = rows_offsets(ctx, n);
            v.total = rows_total(ctx, n);
        } else if ((r = scan_impl(ctx, LoadRectRows{pv.rect}, n, v.roff, v.total, st)) != GS_OK) {
            return r;
        }
        CullArgs ca{pv.xy_ab, pv.c_o_z, pv.rgb, tile};
        const int64_t warps = (n + 31) / 32;
        if (warps > 0)
            GS_CUDA_TRY(launch_k(ctx, k_row_spans, (unsigned)((warps + 7) / 8), 256, 0, st, pv.rect, n, v.roff, ca, tiles_x, ctx->d_bp, K,
                                                                     m_dev, m_cap, v.D, rlayer, v.gbin,
                                                                     RowRecords{v.rs_g, v.rs_ya, v.rs_w, v.rs_z}));
        ctx->launches += 1;
        // the per-entry scatter starts its cursors at the offsets
        const bool want_cur = n > 0 && !grouped_path(m_cap, tiles_x, tiles_y, K);
        const size_t osm = bin_offsets_smem(tiles_x, K);
        if (osm <= kOffMaxSmem) {
            // one pass: counts, tile-major scan, look-back over tile rows
            uint64_t* flags;
            if ((r = scan_flags(ctx, tiles_y, &flags, st)) != GS_OK) return r;
            if ((r = bins_reserve(ctx, 1, nseg)) != GS_OK) return r;
            if (!(ctx->zeroed_tail == ctx->d_tail && ctx->zeroed_tail_bytes == ctx->tail_cap))
                GS_CUDA_TRY(cudaMemsetAsync(ctx->d_tail, 0, kTailHead * 4, st));
            ctx->zeroed_tail = nullptr;  // zeroed by the frame's first kernel once, for this call
            OffsetsExtra ex;
            ex.long_list = ctx->d_tail + kTailLong;
            ex.min_len = long_min;
            *long_listed = true;
            const TileOrder to = frame_tile_order(ctx, T);
            // A whole frame: the raster follows.  Not a deep one, whose tiles are
            // all long and stop early, so that their lengths do not tell their
            // work and taking neighbours apart only costs L2 hits (3M Gaussians
            // seen from inside a cluster: raster 162 us in image order, 166
            // longest first; 1M at 1080p 229 and 219, 437k at 1237x823 133 and
            // 121).
            ctx->tile_ordered = rows_ready && to.lists && !grouped_path(m_cap, tiles_x, tiles_y, K);
            if (ctx->tile_ordered) {
                ex.count = ctx->d_tail;
                ex.order = ctx->d_tiles_order;
                ex.stride = T;
            }
            GS_CUDA_TRY(launch_k(ctx, k_bin_offsets<FrameRows>, (unsigned)tiles_y, kOffThreads, osm, st,
                                 FrameRows{v.D, tiles_x, tiles_y, K, rlayer}, (int)tiles_y, m_dev, m_cap, flags,
                                 ctx->d_scan_done, offsets, want_cur ? v.cur : nullptr, ctx->d_err, ex));
            ctx->launches += 1;
        } else {
            // rows too wide for one block's shared memory: per-layer prefix,
            // the counts tile-major (the cursor array serves as the staging
            // copy; the scan rewrites it with the offsets when the per-entry
            // scatter will start its cursors there), a coalesced scan
            GS_CUDA_TRY(launch_k(ctx, k_layer_rows_prefix, (unsigned)K, 1024, 0, st, v.D, tiles_x, tiles_y, rlayer));
            GS_CUDA_TRY(launch_k(ctx, k_transpose_counts,
                                 dim3((unsigned)((tiles_x + 31) / 32), (unsigned)((K + 31) / 32), (unsigned)tiles_y),
                                 256, 0, st, v.D, tiles_x, tiles_y, K, rlayer, v.cur));
            ctx->launches += 2;
            if ((r = scan_impl(ctx, LoadPlainCount{v.cur}, nseg, offsets, nullptr, st, want_cur ? v.cur : nullptr)) !=
                GS_OK)
                return r;
            GS_CUDA_TRY(launch_k(ctx, k_zero_if_over, g_sm, 256, 0, st, m_dev, m_cap, offsets, nseg + 1, ctx->d_err));
            ctx->launches += 1;
        }
        ScatterPass sp;
        if (planned) {
            ctx->exact_roff = v.roff;
            // the bin planner sets each tile's first-pass bins from the counts
            if ((r = plan_frame(ctx, offsets, K, (int32_t)T, ctx->d_plan, nullptr, st)) != GS_OK) return r;
            sp.plan = ctx->d_plan;
            sp.T = (int32_t)T;
            sp.pass = 1;
        }
        if ((r = exact_scatter(ctx, v, n, tiles_x, tiles_y, K, m_cap, m_dev, words, offsets, sp, st)) !=
            GS_OK)
            return r;
    } else {
        // whole rects per bin layer: four atomics per Gaussian, 2D prefix sums
        if (!goff_ready && (r = count_scan(ctx, pv, n, v.total, st)) != GS_OK) return r;
        if (n > 0) k_bin_diff<<<g_sm, 256, 0, st>>>(pv.rect, pv.c_o_z, n, tiles_x, tiles_y, ctx->d_bp, K, v.D, v.gbin);
        k_layer_prefix<<<(unsigned)K, 1024, 0, st>>>(v.D, tiles_x, tiles_y);
        ctx->launches += 2;
        if ((r = scan_impl(ctx, LoadLayerCount{v.D, K, tiles_x, tiles_x + 1, (int64_t)layer}, nseg, offsets, nullptr,
                           st)) != GS_OK)
            return r;
        GS_CUDA_TRY(launch_k(ctx, k_zero_if_over, g_sm, 256, 0, st, m_dev, m_cap, offsets, nseg + 1, ctx->d_err));
        GS_CUDA_TRY(cudaMemcpyAsync(v.cur, offsets, (size_t)nseg * 4, cudaMemcpyDeviceToDevice, st));
        const int64_t warps = (n + 31) / 32;
        if (warps > 0)
            k_bin_scatter_rects<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(pv.rect, pv.c_o_z, ctx->d_goff, v.gbin, n,
                                                                             tiles_x, K, m_dev, m_cap, offsets, v.cur,
                                                                             words);
        ctx->launches += 2;
    }
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

}  // namespace gs
