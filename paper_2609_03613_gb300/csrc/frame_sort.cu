// frame_sort.cu -- the global-sort ordering of a whole frame (Sec. 3.1: the
// stream grouped by tile and ordered by depth inside), from the projected
// Gaussians.  Every entry of a Gaussian has its depth, so the Gaussians are put
// in depth order first and emit their entries in that order; a stable radix
// sort of the entries by tile alone then leaves each tile in (depth, gid)
// order:
//   n Gaussians by (depth bits, gid)       four 8-bit passes over 8 n bytes
//   entry counts in that order, one scan   (M)
//   emission of (tile, place in the order)
//   M entries by tile                      one pass per 8 tile bits over 8 M bytes
// where a sort of the entries by (tile, depth) takes four more passes over 12 M
// bytes (sort.cu, which serves the callers' own entries).  500k Gaussians at
// 1280x720, 6 M entries: intersect and sort stages 584 -> 266 us.
//
// A pass is one kernel: blocks take chunks of 4096 words in ticket order, rank
// them by digit, and find where their digits' words go from the digit totals
// and their predecessors' published counts (decoupled look-back: D. Merrill and
// M. Garland, 2016; its use for radix passes: A. Adinets and D. Merrill,
// "Onesweep", 2022), with bounded waits.
#include "device.cuh"
#include "scan.cuh"

namespace gs {

constexpr int kSwThreads = 256, kSwItems = 16, kSwChunk = kSwThreads * kSwItems, kSwWarps = kSwThreads / 32;
constexpr int kGaussPasses = 4;    // 8 bits of depth each
constexpr int kMaxTilePasses = 4;  // up to 8 bits of tile each

// Words of the depth sort: (depth bits << 32) | gid, and the four passes'
// digit totals.
__global__ void __launch_bounds__(256)
k_depth_words(const float4* __restrict__ c_o_z, int64_t n, uint64_t* __restrict__ out, uint32_t* __restrict__ hist)
{
    grid_dependency_sync();
    __shared__ uint32_t s_h[kGaussPasses * 256];
    for (int k = threadIdx.x; k < kGaussPasses * 256; k += blockDim.x) s_h[k] = 0u;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t z = __float_as_uint(__ldg(&c_o_z[i].z));
        out[i] = ((uint64_t)z << 32) | (uint32_t)i;
#pragma unroll
        for (int p = 0; p < kGaussPasses; ++p) atomicAdd(&s_h[p * 256 + ((z >> (8 * p)) & 255u)], 1u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kGaussPasses * 256; k += blockDim.x)
        if (s_h[k]) atomicAdd(&hist[k], s_h[k]);
}

// Exclusive scan of one value a thread over the block (kSwThreads).
__device__ __forceinline__ uint32_t sweep_scan(uint32_t v, uint32_t* s_w)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < kSwWarps; ++w)
        if (w < warp) before += s_w[w];
    __syncthreads();
    return before + incl - v;
}

// The words of block bid's predecessors with digit d, summed back to the
// nearest published prefix; four are in flight at once.  ok turns false when
// a wait runs out.
__device__ __forceinline__ uint64_t sweep_lookback(const volatile uint64_t* status, int64_t bid, int nd, int d, bool& ok)
{
    uint64_t pre = 0;
    for (int64_t j = bid - 1; j >= 0;) {
        uint64_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = j - u >= 0 ? status[(j - u) * nd + d] : 0ull;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j < 0) return pre;
            int it = 0;
            while ((w[u] & kScanFlagMask) == 0 && ++it < kLookbackPolls) w[u] = status[j * nd + d];
            if ((w[u] & kScanFlagMask) == 0) {
                ok = false;
                return pre;
            }
            pre += w[u] & ~kScanFlagMask;
            if ((w[u] & kScanFlagMask) == kScanFlagP) return pre;
            --j;
        }
    }
    return pre;
}

// One stable pass over the words by digit (word >> shift) & (2^bits - 1).  The
// count is n when m_dev is null, else the live entry count.  FINAL (the
// entries' last pass): the word (tile << 32) | place leaves as the stream word
// order[place] and its tile.
template <bool FINAL>
__global__ void __launch_bounds__(kSwThreads)
k_sweep(const uint64_t* __restrict__ in, int64_t n, const int64_t* __restrict__ m_dev, int shift, int bits,
        const uint32_t* __restrict__ hist, uint64_t* status, unsigned int* ticket, uint64_t* __restrict__ out,
        const uint64_t* __restrict__ order, uint32_t* __restrict__ tiles, int* err)
{
    grid_dependency_sync();
    __shared__ uint64_t s_key[kSwChunk];
    __shared__ uint32_t s_cnt[kSwWarps][256];
    __shared__ uint32_t s_start[256];  // first place of the digit in the chunk
    __shared__ uint32_t s_dst[256];    // its output position, less that
    __shared__ uint32_t s_w[kSwWarps];
    __shared__ int64_t s_bid;
    if (threadIdx.x == 0) {
        const unsigned t = atomicAdd(ticket, 1u);
        s_bid = t;
        if (t == gridDim.x - 1) *ticket = 0u;  // every ticket is out: ready for the next pass
    }
#pragma unroll
    for (int w = 0; w < kSwWarps; ++w) s_cnt[w][threadIdx.x] = 0u;
    __syncthreads();
    const int64_t M = m_dev ? live_count(m_dev, n) : n, bid = s_bid, base = bid * kSwChunk;
    if (base >= M) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nd = 1 << bits;
    const uint32_t lt = (1u << lane) - 1u, dmask = (uint32_t)nd - 1u;
    uint64_t key[kSwItems];
    uint16_t rank[kSwItems];
#pragma unroll
    for (int k = 0; k < kSwItems; ++k) {
        const int64_t i = base + warp * (32 * kSwItems) + k * 32 + lane;
        key[k] = i < M ? __ldcs(reinterpret_cast<const unsigned long long*>(in) + i) : 0ull;
    }
#pragma unroll
    for (int k = 0; k < kSwItems; ++k) {
        const bool ok = base + warp * (32 * kSwItems) + k * 32 + lane < M;
        const uint32_t d = (uint32_t)(key[k] >> shift) & dmask;
        uint32_t peers = __ballot_sync(0xffffffffu, ok);
        for (int b = 0; b < bits; ++b) {
            const bool one = (d >> b) & 1u;
            const uint32_t m = __ballot_sync(0xffffffffu, one);
            peers &= one ? m : ~m;
        }
        const int before = __popc(peers & lt);
        if (ok) rank[k] = (uint16_t)(s_cnt[warp][d] + before);
        __syncwarp();
        if (ok && before == 0) s_cnt[warp][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // per digit: prefix over the warps and the chunk's count, published
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < kSwWarps; ++w) {
        const uint32_t x = s_cnt[w][threadIdx.x];
        s_cnt[w][threadIdx.x] = run;
        run += x;
    }
    const int d = threadIdx.x;
    volatile uint64_t* vs = status;
    if (d < nd) vs[bid * nd + d] = (bid == 0 ? kScanFlagP : kScanFlagA) | (uint64_t)run;
    const uint32_t start = sweep_scan(run, s_w);
    const uint32_t first = sweep_scan(d < nd ? hist[d] : 0u, s_w);
    bool ok = true;
    if (d < nd) {
        const uint64_t pre = bid > 0 ? sweep_lookback(vs, bid, nd, d, ok) : 0;
        if (bid > 0) vs[bid * nd + d] = kScanFlagP | (pre + run);
        s_start[d] = start;
        s_dst[d] = first + (uint32_t)pre - start;
    }
    if (!ok) raise_error(err, GS_ERR_TIMEOUT);
    if (!__syncthreads_and(ok)) return;  // nothing is written at a wrong place
#pragma unroll
    for (int k = 0; k < kSwItems; ++k)
        if (base + warp * (32 * kSwItems) + k * 32 + lane < M) {
            const uint32_t q = (uint32_t)(key[k] >> shift) & dmask;
            s_key[s_start[q] + s_cnt[warp][q] + rank[k]] = key[k];
        }
    __syncthreads();
    const int cnt = (int)(M - base < kSwChunk ? M - base : kSwChunk);
    for (int j = threadIdx.x; j < cnt; j += kSwThreads) {
        const uint64_t w = s_key[j];
        const uint32_t dst = s_dst[(uint32_t)(w >> shift) & dmask] + (uint32_t)j;
        if (FINAL) {
            out[dst] = __ldg(order + (uint32_t)w);
            tiles[dst] = (uint32_t)(w >> 32);
        } else {
            out[dst] = w;
        }
    }
}

// Entry count of the Gaussian at place i of the depth order.
struct LoadOrderedCount {
    const uint64_t* order;
    const uint2* rect;
    __device__ int64_t operator()(int64_t i) const { return LoadRectCount{rect}((int64_t)(uint32_t)order[i]); }
};

// The entries in depth order: a warp owns 32 consecutive places, whose entries
// are consecutive (warp-cooperative expansion, device.cuh); the tile digits are
// counted on the way.  Nothing is written when the total exceeds the capacity.
struct TileDigits {
    int passes, bits;
};

__global__ void __launch_bounds__(256)
k_emit_ordered(const uint64_t* __restrict__ order, const uint2* __restrict__ rect, const int32_t* __restrict__ goff,
               int64_t n, int tiles_x, const int64_t* __restrict__ m_dev, int64_t m_cap, TileDigits td,
               uint64_t* __restrict__ out, uint32_t* __restrict__ hist, int* err)
{
    grid_dependency_sync();
    __shared__ uint32_t s_h[kMaxTilePasses * 256];
    for (int k = threadIdx.x; k < kMaxTilePasses * 256; k += blockDim.x) s_h[k] = 0u;
    __syncthreads();
    const int64_t M = *m_dev;
    if (M > m_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) raise_error(err, GS_ERR_CAPACITY);
        return;
    }
    const int lane = threadIdx.x & 31;
    const uint32_t dmask = (1u << td.bits) - 1u;
    const int64_t groups = (n + 31) / 32, wstride = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t gq = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); gq < groups; gq += wstride) {
        const int64_t g0 = gq * 32, gl = g0 + lane;
        const bool ok = gl < n;
        const int32_t my = goff[ok ? gl : n];
        const uint2 r = ok ? rect[(uint32_t)order[gl]] : make_uint2(0u, 0u);
        const int32_t base = __shfl_sync(0xffffffffu, my, 0), end = goff[g0 + 32 < n ? g0 + 32 : n];
        for (int32_t e0 = base; e0 < end; e0 += 32) {
            const int32_t e = e0 + lane;
            int k = 0;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                const int32_t v = __shfl_sync(0xffffffffu, my, (k + s) & 31);
                if (k + s < 32 && v <= e) k += s;
            }
            const uint32_t a = __shfl_sync(0xffffffffu, r.x, k), b = __shfl_sync(0xffffffffu, r.y, k);
            const int32_t o = __shfl_sync(0xffffffffu, my, k);
            if (e < end) {
                const uint32_t w = (b & 0xffffu) - (a & 0xffffu), l = (uint32_t)(e - o), dy = l / w;
                const uint32_t tile = ((a >> 16) + dy) * (uint32_t)tiles_x + (a & 0xffffu) + (l - dy * w);
                out[e] = ((uint64_t)tile << 32) | (uint32_t)(g0 + k);
                for (int p = 0; p < td.passes; ++p) atomicAdd(&s_h[p * 256 + ((tile >> (p * td.bits)) & dmask)], 1u);
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < td.passes * 256; k += blockDim.x)
        if (s_h[k]) atomicAdd(&hist[k], s_h[k]);
}

// offsets[t] = first sorted position whose tile is >= t (t = 0..n_tiles)
__global__ void __launch_bounds__(256)
k_tile_bounds(const uint32_t* __restrict__ tiles, const int64_t* __restrict__ m_dev, int64_t m_cap, int32_t n_tiles,
              int32_t* __restrict__ offsets)
{
    grid_dependency_sync();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t > n_tiles) return;
    int64_t lo = 0, hi = live_count(m_dev, m_cap);
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(tiles + mid) < (uint32_t)t) lo = mid + 1;
        else hi = mid;
    }
    offsets[t] = (int32_t)lo;
}

// ------------------------------------------------------------------ host
static TileDigits tile_digits(int32_t n_tiles)
{
    int tb = 1;
    while (tb < 31 && (1ll << tb) < (long long)n_tiles) ++tb;
    TileDigits d;
    d.passes = (tb + 7) / 8;
    d.bits = (tb + d.passes - 1) / d.passes;
    return d;
}

static int64_t chunks(int64_t n) { return n > 0 ? (n + kSwChunk - 1) / kSwChunk : 1; }

// ctx->d_gsort: the two buffers of Gaussian words, then (zeroed per frame)
// the digit totals of all passes and the depth passes' status words.
// ctx->d_hist: the tile passes' status words; d_keys: the entries' two
// buffers; d_vals[0]: the sorted entries' tiles.
struct FrameSort {
    uint64_t *g[2], *status_g, *status_m;
    uint32_t* hist;
    size_t zero_bytes, bytes, status_m_bytes;
};

static FrameSort frame_sort_view(gs_ctx* c, int64_t n, int64_t m_cap, TileDigits td)
{
    FrameSort f;
    const size_t gb = align256((size_t)(n > 0 ? n : 1) * 8), hb = align256((kGaussPasses + kMaxTilePasses) * 256 * 4);
    const size_t sb = (size_t)kGaussPasses * chunks(n) * 256 * 8;
    char* b = static_cast<char*>(c->d_gsort);
    f.g[0] = reinterpret_cast<uint64_t*>(b);
    f.g[1] = reinterpret_cast<uint64_t*>(b + gb);
    f.hist = reinterpret_cast<uint32_t*>(b + 2 * gb);
    f.status_g = reinterpret_cast<uint64_t*>(b + 2 * gb + hb);
    f.zero_bytes = hb + sb;
    f.bytes = 2 * gb + hb + sb;
    f.status_m = reinterpret_cast<uint64_t*>(c->d_hist);
    f.status_m_bytes = (size_t)td.passes * chunks(m_cap) * ((size_t)1 << td.bits) * 8;
    return f;
}

int frame_sort_reserve(gs_ctx* c, int64_t n, int64_t m_cap, int32_t n_tiles)
{
    int r = sort_reserve(c, m_cap);
    if (r != GS_OK) return r;
    const FrameSort f = frame_sort_view(c, n, m_cap, tile_digits(n_tiles));
    void* p = c->d_gsort;
    r = ensure(&p, &c->gsort_cap, f.bytes);
    c->d_gsort = p;
    if (r != GS_OK) return r;
    p = c->d_hist;
    r = ensure(&p, &c->hist_cap, f.status_m_bytes);
    c->d_hist = static_cast<uint32_t*>(p);
    if (r != GS_OK) return r;
    return goff_reserve(c, n);
}

static int sweep(gs_ctx* c, bool final_pass, const uint64_t* in, int64_t n, const int64_t* m_dev, int shift, int bits,
                 const uint32_t* hist, uint64_t* status, uint64_t* out, const uint64_t* order, uint32_t* tiles,
                 cudaStream_t st)
{
    GS_CUDA_TRY(launch_k(c, final_pass ? k_sweep<true> : k_sweep<false>, (unsigned)chunks(n), kSwThreads, 0, st, in, n,
                         m_dev, shift, bits, hist, status, c->d_scan_done, out, order, tiles, c->d_err));
    c->launches += 1;
    return GS_OK;
}

// The Gaussians in depth order, their entry offsets (ctx->d_goff) and M.
int frame_sort_gaussians(gs_ctx* c, const ProjView& pv, int64_t n, int64_t m_cap, int32_t n_tiles, int64_t* m_dev,
                         cudaStream_t st)
{
    int r = frame_sort_reserve(c, n, m_cap > 0 ? m_cap : 1, n_tiles);
    if (r != GS_OK) return r;
    if (n == 0) {
        GS_CUDA_TRY(cudaMemsetAsync(m_dev, 0, sizeof(int64_t), st));
        return GS_OK;
    }
    const FrameSort f = frame_sort_view(c, n, m_cap, tile_digits(n_tiles));
    GS_CUDA_TRY(cudaMemsetAsync(f.hist, 0, f.zero_bytes, st));
    const int64_t want = (n + 1023) / 1024, most = (int64_t)c->num_sms * 8;
    GS_CUDA_TRY(launch_k(c, k_depth_words, (unsigned)(want < most ? want : most), 256, 0, st, pv.c_o_z, n, f.g[0], f.hist));
    c->launches += 1;
    for (int p = 0; p < kGaussPasses; ++p)
        if ((r = sweep(c, false, f.g[p & 1], n, nullptr, 32 + 8 * p, 8, f.hist + p * 256,
                       f.status_g + (size_t)p * chunks(n) * 256, f.g[(p & 1) ^ 1], nullptr, nullptr, st)) != GS_OK)
            return r;
    static_assert(kGaussPasses % 2 == 0, "the order ends in the first buffer");
    return scan_impl(c, LoadOrderedCount{f.g[0], pv.rect}, n, c->d_goff, m_dev, st);
}

// The stream and its tile offsets, after frame_sort_gaussians (m_cap may have
// grown since: n and n_tiles may not).
int frame_sort_entries(gs_ctx* c, const ProjView& pv, int64_t n, int64_t m_cap, int32_t tiles_x, int32_t n_tiles,
                       const int64_t* m_dev, uint64_t* words, int32_t* offsets, cudaStream_t st)
{
    int r = frame_sort_reserve(c, n, m_cap, n_tiles);
    if (r != GS_OK) return r;
    if (n == 0) {
        GS_CUDA_TRY(cudaMemsetAsync(offsets, 0, ((size_t)n_tiles + 1) * 4, st));
        return GS_OK;
    }
    const TileDigits td = tile_digits(n_tiles);
    const FrameSort f = frame_sort_view(c, n, m_cap, td);
    uint32_t* hist = f.hist + kGaussPasses * 256;
    GS_CUDA_TRY(cudaMemsetAsync(f.status_m, 0, f.status_m_bytes, st));
    const int64_t want = (n + 255) / 256, most = (int64_t)c->num_sms * 8;
    GS_CUDA_TRY(launch_k(c, k_emit_ordered, (unsigned)(want < most ? want : most), 256, 0, st, f.g[0], pv.rect, c->d_goff,
                         n, tiles_x, m_dev, m_cap, td, c->d_keys[0], hist, c->d_err));
    c->launches += 1;
    for (int p = 0; p < td.passes; ++p) {
        const bool last = p == td.passes - 1;
        if ((r = sweep(c, last, c->d_keys[p & 1], m_cap, m_dev, 32 + p * td.bits, td.bits, hist + p * 256,
                       f.status_m + (size_t)p * chunks(m_cap) * ((size_t)1 << td.bits),
                       last ? words : c->d_keys[(p & 1) ^ 1], f.g[0], c->d_vals[0], st)) != GS_OK)
            return r;
    }
    GS_CUDA_TRY(launch_k(c, k_tile_bounds, (unsigned)(n_tiles / 256 + 1), 256, 0, st, c->d_vals[0], m_dev, m_cap, n_tiles,
                         offsets));
    c->launches += 1;
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

}  // namespace gs
