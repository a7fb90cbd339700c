// offsets.cuh -- the one-pass (tile, bin) segment offsets of EXACT bin
// construction with the tile cull, for one frame (tiles.cu) or the views of a
// batch (batch_bins.cu).
#pragma once
#include "scan.cuh"

namespace gs {

// The (tile, bin) segment offsets from the layered row differences
// D[b][ty][x] in one pass, tile-major (t = ty tiles_x + x, bins inside; the
// views of a batch one after the other): one block per tile row (taken in
// ticket order) forms its counts by a prefix
// along x per bin, scans them in tile-major order, finds the rows before it
// by decoupled look-back over the rows' published totals (bounded waits),
// and writes offsets and, when given, the scatter cursors.  Over capacity
// (or past INT32_MAX) every offset is written 0 and GS_ERR_CAPACITY raised,
// so nothing downstream reads out of bounds.  On the way it lists the long
// segments and orders the tiles by span (OffsetsExtra): a pass over all the
// offsets and its launch less each (5 us at 1080p; the batch's three ordering
// kernels took 43 us).  Replaces a per-layer prefix,
// a transposition, a device-wide scan and the over-capacity pass.
constexpr int kOffThreads = 1024;
constexpr size_t kOffMaxSmem = 160 * 1024;
__host__ __device__ inline size_t bin_offsets_smem(int tiles_x, int K) { return (size_t)tiles_x * (K + 1) * 4; }

// One tile row: its difference counts (bin b's at D + b layer), its tiles and
// bins, its first segment, its first cursor and the cursors' stride from one
// bin to the next (neighbouring tiles lie side by side).
struct OffsetRow {
    const int32_t* D;
    int64_t layer;
    int tiles_x, K;
    int64_t seg, cur, cur_bin;
    int32_t tile;  // its first tile
};

// Rows: OffsetRow of row y (0 <= y < n_rows, in segment order).
template <class Rows>
__global__ void __launch_bounds__(kOffThreads)
k_bin_offsets(const __grid_constant__ Rows rows, int n_rows, const int64_t* __restrict__ m_dev, int64_t m_cap,
              uint64_t* flags, unsigned int* ticket, int32_t* __restrict__ off, int32_t* __restrict__ cur, int* err, const OffsetsExtra ex)
{
    grid_dependency_sync();
    extern __shared__ int32_t s_c[];  // [tiles_x][K + 1]: counts, then exclusive offsets in the row
    __shared__ int32_t s_warp[kOffThreads / 32];
    __shared__ int64_t s_pre;
    __shared__ int s_row;
    if (threadIdx.x == 0) {
        const unsigned t = atomicAdd(ticket, 1u);
        s_row = (int)t;
        if ((int)t == n_rows - 1) *ticket = 0u;  // every ticket is out: ready for the next scan
    }
    __syncthreads();
    const int ty = s_row;
    const OffsetRow rw = rows(ty);
    const int tiles_x = rw.tiles_x, K = rw.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KP = K + 1;
    // counts: per bin, the inclusive prefix of the row's differences
    for (int b = warp; b < K; b += kOffThreads / 32) {
        const int32_t* row = rw.D + (int64_t)b * rw.layer;
        int32_t carry = 0;
        for (int x0 = 0; x0 < tiles_x; x0 += 32) {
            const int x = x0 + lane;
            int32_t v = x < tiles_x ? row[x] : 0;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int32_t u = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += u;
            }
            if (x < tiles_x) s_c[x * KP + b] = carry + v;
            carry += __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    // the row's exclusive scan in tile-major order: a run of items a thread
    const int items = tiles_x * K;
    const int per = (items + kOffThreads - 1) / kOffThreads;
    const int j0 = threadIdx.x * per;
    int32_t run = 0;
    {
        int x = j0 / K, b = j0 - (j0 / K) * K;
        for (int k = 0; k < per && j0 + k < items; ++k) {
            run += s_c[x * KP + b];
            if (++b == K) { b = 0; ++x; }
        }
    }
    int32_t incl = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        constexpr int NW = kOffThreads / 32;
        int32_t w = lane < NW ? s_warp[lane] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += u;
        }
        if (lane < NW) s_warp[lane] = w;  // inclusive warp totals
    }
    __syncthreads();
    const int64_t total = s_warp[kOffThreads / 32 - 1];
    int32_t e = (warp > 0 ? s_warp[warp - 1] : 0) + incl - run;
    {
        int x = j0 / K, b = j0 - (j0 / K) * K;
        for (int k = 0; k < per && j0 + k < items; ++k) {
            const int32_t c = s_c[x * KP + b];
            s_c[x * KP + b] = e;
            e += c;
            if (++b == K) { b = 0; ++x; }
        }
    }
    // the rows before: publish this row's total, look back over theirs
    volatile uint64_t* vf = flags;
    if (threadIdx.x == 0) vf[ty] = (ty == 0 ? kScanFlagP : kScanFlagA) | (uint64_t)total;
    if (warp == 0) {
        const int64_t pre = ty > 0 ? scan_lookback(vf, ty, err) : 0;
        if (lane == 0) {
            if (ty > 0) vf[ty] = kScanFlagP | (uint64_t)(pre + total);
            s_pre = pre;
        }
    }
    __syncthreads();
    const int64_t pre = s_pre;
    const bool over = *m_dev > m_cap || pre + total > (int64_t)INT32_MAX - 1;
    if (over && threadIdx.x == 0) raise_error(err, GS_ERR_CAPACITY);
    for (int j = threadIdx.x; j < items; j += kOffThreads) {
        const int x = j / K, b = j - x * K;
        const int32_t v = over ? 0 : (int32_t)(pre + s_c[x * KP + b]);
        off[rw.seg + j] = v;
        if (ex.min_len > 0 && !over) {
            const int32_t end = b + 1 < K ? s_c[x * KP + b + 1] : (x + 1 < tiles_x ? s_c[(x + 1) * KP] : (int32_t)total);
            if (end - s_c[x * KP + b] >= ex.min_len)
                ex.long_list[1 + atomicAdd(ex.long_list, 1)] = (int32_t)(rw.seg + j);
        }
    }
    if (ex.order)
        for (int x = threadIdx.x; x < tiles_x; x += kOffThreads) {
            const int32_t n = over ? 0 : (x + 1 < tiles_x ? s_c[(x + 1) * KP] : (int32_t)total) - s_c[x * KP];
            const int q = 31 - __clz(n + 1);
            ex.order[q * ex.stride + atomicAdd(ex.count + q, 1)] = rw.tile + x;
        }
    if (cur) {  // bin by bin, tiles inside
        for (int j = threadIdx.x; j < items; j += kOffThreads) {
            const int b = j / tiles_x, x = j - b * tiles_x;
            cur[rw.cur + b * rw.cur_bin + x] = over ? 0 : (int32_t)(pre + s_c[x * KP + b]);
        }
    }
    if (ty == n_rows - 1 && threadIdx.x == 0) off[rw.seg + items] = over ? 0 : (int32_t)(pre + total);
}

}  // namespace gs
