// batch_bins.cu -- the EXACT binning of several views of one scene in one
// launch per stage (the batched render of gs_render_batch; the paper renders
// single views only).
//
// The views that can share it (EXACT, repair in the raster, 16x16 tiles, the
// tile cull, no planner) form one group: their projected records sit side by
// side in one buffer, so Gaussian g of view v is item G = v n + g of a single
// frame of V n items, and their tiles and (tile, bin) segments are
// concatenated.  Every stage then runs once over all views:
//   counts and row counts of every item, one scan     (as a single frame)
//   per-view entry counts, samples and depth range    (Alg. 2, a block a view)
//   row spans, per-row difference counts per view     (Alg. 3's histogram)
//   one pass over every view's tile rows              (bin offsets)
//   the scatter of every view's row records           (one cursor per segment)
//   the eager sort of segments over 2048 entries
// and the persistent multi-view raster composites every view's tiles from
// the group's stream, view v's offsets starting at its first segment.  Stream
// words carry G, so the raster gathers from the shared records; the last-id
// output subtracts the view's first item (v n).
#include <string.h>

#include "depth_range.cuh"
#include "offsets.cuh"
#include "rows.cuh"
#include "scan.cuh"

namespace gs {

// Per-view geometry of a group (a kernel parameter).
struct GroupViews {
    int nv;
    int64_t n;                                  // Gaussians per view
    int32_t K[kMaxBatchViews];                  // bins per tile
    int32_t tiles_x[kMaxBatchViews], tiles_y[kMaxBatchViews];
    int32_t tile_base[kMaxBatchViews + 1];      // first tile of view v in the group
    int64_t seg_base[kMaxBatchViews + 1];       // first (tile, bin) segment of view v
    int32_t row_base[kMaxBatchViews + 1];       // first tile row of view v
    int32_t layer_base[kMaxBatchViews + 1];     // first bin layer of view v
    int64_t d_base[kMaxBatchViews + 1];         // first difference count of view v (K layers of ty x (tx + 1))
    float near_plane[kMaxBatchViews], far_plane[kMaxBatchViews];
    __device__ __forceinline__ int view_of(int64_t G) const { return (int)((uint32_t)G / (uint32_t)n); }
};

// Entries of each view: view v owns the entries [base, base + M) of the
// group, and takes S' = min(S, M) depth samples of them.
struct ViewCount {
    int64_t base, M, ns;
};

__global__ void k_group_counts(const int32_t* __restrict__ goff, int64_t n, int nv, int S,
                               ViewCount* __restrict__ vc, int64_t* __restrict__ m_out)
{
    const int v = threadIdx.x;
    if (v >= nv) return;
    const int64_t b = goff[(int64_t)v * n], e = goff[(int64_t)(v + 1) * n];
    ViewCount c;
    c.base = b;
    c.M = e - b;
    c.ns = c.M < (int64_t)S ? c.M : (int64_t)S;
    vc[v] = c;
    m_out[v] = c.M;
}

// Sample i of view v's S' is its entry j = floor(i M / S') (Alg. 2's
// sampling, as for a single frame); its item is the G of the view with
// goff[G] - base <= j < goff[G + 1] - base, found by binary search over the
// view's items (one thread per sample, grid.y = the view).
__global__ void __launch_bounds__(256)
k_group_sample_keys(const int32_t* __restrict__ goff, const float4* __restrict__ c_o_z, const GroupViews gv,
                    const ViewCount* __restrict__ vc, int S, uint32_t* __restrict__ out)
{
    const int v = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const ViewCount c = vc[v];
    if (i >= c.ns) return;
    const int64_t j = c.base + ((int64_t)i * c.M) / c.ns;
    // the last item G in [v n, (v+1) n) with goff[G] <= j
    int64_t lo = (int64_t)v * gv.n, hi = lo + gv.n - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (goff[mid] <= j) lo = mid;
        else hi = mid - 1;
    }
    out[(int64_t)v * S + i] = __float_as_uint(c_o_z[lo].z);
}

// One block per view: Alg. 2 over the view's samples, its bin parameters.
__global__ void __launch_bounds__(kDrThreads)
k_group_depth_range(const float4* __restrict__ c_o_z, const GroupViews gv, const ViewCount* __restrict__ vc,
                    const uint32_t* __restrict__ samples, DrArgs a, BinParams* __restrict__ bp)
{
    const int v = blockIdx.x;
    a.near_plane = gv.near_plane[v];
    a.far_plane = gv.far_plane[v];
    a.K = gv.K[v];
    depth_range_block(c_o_z, nullptr, KeyFromSamples{samples + (int64_t)v * a.S}, vc[v].M, a, bp + v);
}

// The row spans of k_row_spans (tiles.cu) for the group's items: each lane's
// item and each record's owner look up their view (tile grid, bin splits,
// difference counts); records carry the item G.
__global__ void __launch_bounds__(256, kRowBlocks)
k_group_row_spans(const uint2* __restrict__ rect, const int32_t* __restrict__ roff, CullArgs ca,
                  const __grid_constant__ GroupViews gv, const BinParams* __restrict__ bp,
                  const int64_t* __restrict__ m_dev, int64_t m_cap, int32_t* __restrict__ D, RowRecords rs)
{
    __shared__ RowOwners s_own[8];
    if (*m_dev > m_cap) return;
    const int64_t n = gv.n * gv.nv;
    const int64_t g0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 32;
    if (g0 >= n) return;
    const int64_t gl = g0 + (threadIdx.x & 31);
    const int32_t off = roff[gl < n ? gl : n], next = roff[gl + 1 < n ? gl + 1 : n];
    uint2 r = make_uint2(0u, 0u);
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f), q = p;
    float margin = 0.0f;
    uint32_t bin = 0u;
    int view = 0;
    if (next > off) {
        r = rect[gl];
        p = __ldg(ca.xy_ab + gl);
        q = __ldg(ca.c_o_z + gl);
        margin = __ldg(&ca.rgb[gl].w);
        view = gv.view_of(gl);
        bin = (uint32_t)bin_split(q.z, bp[view].splits, gv.K[view]);
    }
    warp_row_spans(s_own[threadIdx.x >> 5], g0, off, next, __shfl_sync(0xffffffffu, off, 0),
                   __shfl_sync(0xffffffffu, next, 31), r, p, q, margin, bin, view, ca.tile, rs,
                   [&](uint32_t b, uint32_t v, int ty) {
                       return D + gv.d_base[v] + ((int64_t)b * gv.tiles_y[v] + ty) * (gv.tiles_x[v] + 1);
                   });
}

// One block per (view, bin layer): inclusive prefix along each tile row.
__global__ void __launch_bounds__(1024) k_group_layer_prefix(int32_t* __restrict__ D, const GroupViews gv)
{
    int v = 0;
    while (v + 1 < gv.nv && gv.layer_base[v + 1] <= (int)blockIdx.x) ++v;
    const int b = (int)blockIdx.x - gv.layer_base[v];
    const int tiles_x = gv.tiles_x[v], tiles_y = gv.tiles_y[v], W1 = tiles_x + 1;
    int32_t* L = D + gv.d_base[v] + (int64_t)b * tiles_y * W1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int y = warp; y < tiles_y; y += blockDim.x / 32) {
        int32_t carry = 0;
        for (int x0 = 0; x0 < tiles_x; x0 += 32) {
            const int x = x0 + lane;
            int32_t val = x < tiles_x ? L[y * W1 + x] : 0;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int32_t u = __shfl_up_sync(0xffffffffu, val, d);
                if (lane >= d) val += u;
            }
            if (x < tiles_x) L[y * W1 + x] = carry + val;
            carry += __shfl_sync(0xffffffffu, val, 31);
        }
    }
}

// count[t, b] of every view into the group's segment order (view v's tile t,
// bin b at seg_base[v] + t K_v + b), through 32 x 32 shared-memory blocks;
// blockIdx.z is the group's tile row.
__global__ void __launch_bounds__(256)
k_group_transpose(const int32_t* __restrict__ D, const GroupViews gv, int32_t* __restrict__ C)
{
    __shared__ int32_t s[32][33];
    int v = 0;
    while (v + 1 < gv.nv && gv.row_base[v + 1] <= (int)blockIdx.z) ++v;
    const int y = (int)blockIdx.z - gv.row_base[v];
    const int tiles_x = gv.tiles_x[v], K = gv.K[v], W1 = tiles_x + 1;
    const int x0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
    if (x0 >= tiles_x || b0 >= K) return;  // block-uniform
    const int64_t layer = (int64_t)gv.tiles_y[v] * W1;
    const int32_t* Dv = D + gv.d_base[v];
    const int lx = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < 32; r += blockDim.x >> 5) {
        const int b = b0 + r, x = x0 + lx;
        s[r][lx] = (b < K && x < tiles_x) ? Dv[b * layer + (int64_t)y * W1 + x] : 0;
    }
    __syncthreads();
    int32_t* Cv = C + gv.seg_base[v];
    for (int r = threadIdx.x >> 5; r < 32; r += blockDim.x >> 5) {
        const int x = x0 + r, b = b0 + lx;
        if (x < tiles_x && b < K) Cv[((int64_t)y * tiles_x + x) * K + b] = s[lx][r];
    }
}

// The group's tile rows (offsets.cuh): view by view.
struct GroupRows {
    const int32_t* D;
    GroupViews gv;
    __device__ __forceinline__ OffsetRow operator()(int row) const
    {
        int v = 0;
        while (v + 1 < gv.nv && gv.row_base[v + 1] <= row) ++v;
        const int y = row - gv.row_base[v], tx = gv.tiles_x[v], K = gv.K[v];
        return OffsetRow{D + gv.d_base[v] + (int64_t)y * (tx + 1), (int64_t)gv.tiles_y[v] * (tx + 1), tx, K,
                         gv.seg_base[v] + (int64_t)y * tx * K, gv.seg_base[v] + (int64_t)y * tx,
                         (int64_t)tx * gv.tiles_y[v], gv.tile_base[v] + y * tx};
    }
};

int group_offsets_prepare()
{
    GS_CUDA_TRY(cudaFuncSetAttribute(k_bin_offsets<GroupRows>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kOffMaxSmem));
    return GS_OK;
}

// The cursors from the segment offsets, where the scan wrote those alone.
__global__ void __launch_bounds__(256)
k_group_cursors(const int32_t* __restrict__ off, const __grid_constant__ GroupViews gv, int32_t* __restrict__ cur)
{
    const int64_t n = gv.seg_base[gv.nv];
    int v = 0;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        while (v + 1 < gv.nv && gv.seg_base[v + 1] <= q) ++v;
        const int64_t l = q - gv.seg_base[v], t = l / gv.K[v], b = l - t * gv.K[v];
        cur[gv.seg_base[v] + b * gv.tiles_x[v] * gv.tiles_y[v] + t] = off[q];
    }
}

// The tile order (OffsetsExtra), where no offsets pass wrote it.
__global__ void __launch_bounds__(256)
k_group_order(const int32_t* __restrict__ off, const __grid_constant__ GroupViews gv, int32_t* __restrict__ count,
              int32_t* __restrict__ order)
{
    const int n = gv.tile_base[gv.nv];
    int v = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        while (v + 1 < gv.nv && gv.tile_base[v + 1] <= i) ++v;
        const int64_t q = gv.seg_base[v] + (int64_t)(i - gv.tile_base[v]) * gv.K[v];
        const int b = 31 - __clz(off[q + gv.K[v]] - off[q] + 1);
        order[(int64_t)b * n + atomicAdd(count + b, 1)] = i;
    }
}

// The scatter of k_bin_scatter_rows (tiles.cu) for the group: a record's
// item gives its view, whose tile grid and first segment place its entries
// (cursors bin by bin inside their view).
__global__ void __launch_bounds__(256)
k_group_scatter(const uint32_t* __restrict__ rs_g, const uint32_t* __restrict__ rs_ya, const uint32_t* __restrict__ rs_w,
                const uint32_t* __restrict__ rs_z, const int32_t* __restrict__ roff, const __grid_constant__ GroupViews gv,
                const int64_t* __restrict__ m_dev, int64_t m_cap, int32_t* __restrict__ cur,
                uint64_t* __restrict__ words)
{
    __shared__ ScatterShared s_sc[8];
    if (*m_dev > m_cap) return;
    const int64_t R = roff[gv.n * gv.nv];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nchunks = (R + 31) / 32;
    const int64_t wstride = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; c < nchunks; c += wstride) {
        const int64_t k = c * 32 + lane;
        uint32_t w = 0, g = 0, z = 0, slot = 0;
        if (k < R) {  // read once: streamed past L2
            const uint32_t ya = __ldcs(rs_ya + k);
            w = __ldcs(rs_w + k);
            g = __ldcs(rs_g + k);
            z = __ldcs(rs_z + k);
            const int v = gv.view_of(g), tx = gv.tiles_x[v];
            slot = (uint32_t)(gv.seg_base[v] + (int64_t)(ya >> 24) * tx * gv.tiles_y[v] +
                              (int)(ya & 0xfffu) * tx + (int)((ya >> 12) & 0xfffu));
        }
        scatter_row_records(w, g, z, slot, 1u, cur, words, s_sc[warp], KeepAll());
    }
}

// ------------------------------------------------------------------ host

// zero offsets when the entries overflow the capacity (tiles.cu)
__global__ void k_zero_if_over(const int64_t* __restrict__ m_dev, int64_t m_cap, int32_t* __restrict__ off, int64_t nq,
                               int* err);

GroupViews* group_views_new() { return new GroupViews(); }
void group_views_free(GroupViews* gv) { delete gv; }
int64_t group_seg_base(const GroupViews* gv, int v) { return gv->seg_base[v]; }

int64_t group_views_set(GroupViews* gv, int64_t n, int nv, const gs_camera* cams, const int32_t* K)
{
    memset(gv, 0, sizeof(*gv));
    gv->nv = nv;
    gv->n = n;
    for (int v = 0; v < nv; ++v) {
        const int tx = (cams[v].width + 15) / 16, ty = (cams[v].height + 15) / 16;
        gv->K[v] = K[v];
        gv->tiles_x[v] = tx;
        gv->tiles_y[v] = ty;
        gv->tile_base[v + 1] = gv->tile_base[v] + tx * ty;
        gv->seg_base[v + 1] = gv->seg_base[v] + (int64_t)tx * ty * K[v];
        gv->row_base[v + 1] = gv->row_base[v] + ty;
        gv->layer_base[v + 1] = gv->layer_base[v] + K[v];
        gv->d_base[v + 1] = gv->d_base[v] + (int64_t)K[v] * ty * (tx + 1);
        gv->near_plane[v] = cams[v].near_plane;
        gv->far_plane[v] = cams[v].far_plane;
    }
    return gv->seg_base[nv];
}

// The group's scratch in gc->d_tiles: difference counts, cursors (also the
// staging copy of the transposed counts), row records, samples, per-view bin
// parameters and entry counts.
struct GroupScratch {
    int32_t* D;
    int32_t* cur;
    uint32_t *rs_g, *rs_ya, *rs_w, *rs_z;
    uint32_t* samples;
    BinParams* bp;
    ViewCount* vc;
    int64_t* m_views;
};

static size_t group_scratch(const GroupViews& gv, int64_t m_cap, int S, char* base, GroupScratch* s)
{
    const size_t mc = (size_t)(m_cap > 0 ? m_cap : 1);
    const size_t sizes[] = {(size_t)gv.d_base[gv.nv] * 4, (size_t)gv.seg_base[gv.nv] * 4, mc * 4, mc * 4, mc * 4,
                            mc * 4, (size_t)gv.nv * S * 4, (size_t)gv.nv * sizeof(BinParams),
                            (size_t)gv.nv * sizeof(ViewCount), (size_t)gv.nv * 8};
    size_t total = 0;
    for (size_t z : sizes) total += align256(z > 0 ? z : 4);
    if (s) {
        char* p = base;
        void** dst[] = {(void**)&s->D, (void**)&s->cur, (void**)&s->rs_g, (void**)&s->rs_ya, (void**)&s->rs_w,
                        (void**)&s->rs_z, (void**)&s->samples, (void**)&s->bp, (void**)&s->vc, (void**)&s->m_views};
        for (int k = 0; k < 10; ++k) {
            *dst[k] = p;
            p += align256(sizes[k] > 0 ? sizes[k] : 4);
        }
    }
    return total;
}

int group_reserve(gs_ctx* gc, const GroupViews* gvp, int64_t m_cap)
{
    const GroupViews& gv = *gvp;
    const int64_t N = gv.n * gv.nv, NS = gv.seg_base[gv.nv];
    int r;
    if ((r = ensure(&gc->r_proj, &gc->r_proj_cap, gs_projected_bytes(N))) != GS_OK) return r;
    if (m_cap > gc->r_m_cap) {
        if (gc->r_stream) cudaFree(gc->r_stream);
        gc->r_stream = nullptr;
        gc->r_m_cap = 0;
        size_t sb = 0;
        void* sp = nullptr;
        if ((r = ensure(&sp, &sb, (size_t)m_cap * 8)) != GS_OK) return r;
        gc->r_stream = (uint64_t*)sp;
        gc->r_m_cap = m_cap;
    }
    void* op = gc->r_off;
    if ((r = ensure(&op, &gc->r_off_cap, ((size_t)NS + 1) * 4)) != GS_OK) return r;
    gc->r_off = (int32_t*)op;
    void* tp = gc->d_tiles;
    if ((r = ensure(&tp, &gc->tiles_cap, group_scratch(gv, gc->r_m_cap, gc->cfg.sample_count, nullptr, nullptr))) !=
        GS_OK)
        return r;
    gc->d_tiles = (int32_t*)tp;
    if ((r = goff_reserve(gc, N)) != GS_OK) return r;
    if ((r = scan_reserve(gc, N > NS ? N : NS)) != GS_OK) return r;
    // ... and one flag word a tile row (the offsets' pass), its lists
    if ((r = bins_reserve(gc, 1, NS)) != GS_OK) return r;
    if ((r = tile_order_reserve(gc, gv.tile_base[gv.nv])) != GS_OK) return r;
    return ensure(&gc->d_scan, &gc->scan_bytes, ((size_t)gv.row_base[gv.nv] + 2) * sizeof(uint64_t));
}

int group_binning(gs_ctx* gc, const GroupViews* gvp, int32_t flags, int64_t* h_m_views, TileOrder* order,
                  cudaStream_t st)
{
    const GroupViews& gv = *gvp;
    const int64_t N = gv.n * gv.nv, NS = gv.seg_base[gv.nv];
    const int S = gc->cfg.sample_count;
    int r;
    if ((r = group_reserve(gc, gvp, gc->r_m_cap > 0 ? gc->r_m_cap : 1)) != GS_OK) return r;
    const ProjView pv = proj_view(gc->r_proj, N);
    // tile counts and row counts of every item, one scan (as a single frame)
    if ((r = count_rows_scan(gc, pv, N, gc->r_m, st)) != GS_OK) return r;
    if (!(flags & GS_RENDER_NO_SYNC)) {
        GS_CUDA_TRY(cudaMemcpyAsync(gc->h_m, gc->r_m, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        GS_CUDA_TRY(cudaStreamSynchronize(st));
        if (gc->h_m[0] > gc->r_m_cap && (r = group_reserve(gc, gvp, gc->h_m[0])) != GS_OK) return r;
    }
    GroupScratch s;
    group_scratch(gv, gc->r_m_cap, S, reinterpret_cast<char*>(gc->d_tiles), &s);
    const int32_t* roff = rows_offsets(gc, N);
    // per-view entry counts, samples and depth range (Alg. 2)
    k_group_counts<<<1, 32, 0, st>>>(gc->d_goff, gv.n, gv.nv, S, s.vc, s.m_views);
    if (h_m_views)
        GS_CUDA_TRY(cudaMemcpyAsync(h_m_views, s.m_views, (size_t)gv.nv * 8, cudaMemcpyDeviceToHost, st));
    if (N > 0) k_group_sample_keys<<<dim3((unsigned)((S + 255) / 256), (unsigned)gv.nv), 256, 0, st>>>(gc->d_goff, pv.c_o_z, gv, s.vc, S, s.samples);
    const DrArgs a = dr_args(gc->cfg, 0, 0.0f, 0.0f, 0);  // EXACT mode; planes and K are set per view
    k_group_depth_range<<<(unsigned)gv.nv, kDrThreads, 0, st>>>(pv.c_o_z, gv, s.vc, s.samples, a, s.bp);
    gc->launches += N > 0 ? 3 : 2;
    // row spans and per-row difference counts, then the offsets
    GS_CUDA_TRY(cudaMemsetAsync(s.D, 0, (size_t)gv.d_base[gv.nv] * 4, st));
    const CullArgs ca{pv.xy_ab, pv.c_o_z, pv.rgb, 16};
    const int64_t warps = (N + 31) / 32;
    if (warps > 0)
        k_group_row_spans<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(pv.rect, roff, ca, gv, s.bp, gc->r_m,
                                                                       gc->r_m_cap, s.D, RowRecords{s.rs_g, s.rs_ya, s.rs_w, s.rs_z});
    int max_tx = 1, max_k = 1;
    size_t osm = 0;
    for (int v = 0; v < gv.nv; ++v) {
        max_tx = gv.tiles_x[v] > max_tx ? gv.tiles_x[v] : max_tx;
        max_k = gv.K[v] > max_k ? gv.K[v] : max_k;
        const size_t need = bin_offsets_smem(gv.tiles_x[v], gv.K[v]);
        osm = need > osm ? need : osm;
    }
    const unsigned g_sm = (unsigned)gc->num_sms * 8;
    const int n_rows = gv.row_base[gv.nv];
    gc->launches += 1;
    GS_CUDA_TRY(cudaMemsetAsync(gc->d_tail, 0, kTailHead * 4, st));
    const bool one_pass = osm <= kOffMaxSmem;
    const int32_t min_len = raster_sort_cap(16) + 1;
    if (one_pass) {
        // one pass over every view's tile rows, cursors included (prefixes, a
        // transposition, a scan, the over-capacity pass and a copy before:
        // 57 us of kernels for 16 views of 1M Gaussians; the scatter with its
        // cursors in segment order and four entries in flight 947 us)
        uint64_t* flags;
        if ((r = scan_flags(gc, n_rows, &flags, st)) != GS_OK) return r;
        OffsetsExtra ex;
        ex.long_list = gc->d_tail + kTailLong;
        ex.min_len = min_len;
        ex.count = gc->d_tail;
        ex.order = gc->d_tiles_order;
        ex.stride = gv.tile_base[gv.nv];
        GS_CUDA_TRY(launch_k(gc, k_bin_offsets<GroupRows>, (unsigned)n_rows, kOffThreads, osm, st, GroupRows{s.D, gv},
                             n_rows, gc->r_m, gc->r_m_cap, flags, gc->d_scan_done, gc->r_off, s.cur, gc->d_err, ex));
        gc->launches += 1;
    } else {
        // a view's tile rows too wide for one block's shared memory
        k_group_layer_prefix<<<(unsigned)gv.layer_base[gv.nv], 1024, 0, st>>>(s.D, gv);
        k_group_transpose<<<dim3((unsigned)((max_tx + 31) / 32), (unsigned)((max_k + 31) / 32), (unsigned)n_rows), 256, 0,
                            st>>>(s.D, gv, s.cur);
        if ((r = scan_impl(gc, LoadI32{s.cur}, NS, gc->r_off, nullptr, st)) != GS_OK) return r;
        k_zero_if_over<<<g_sm, 256, 0, st>>>(gc->r_m, gc->r_m_cap, gc->r_off, NS + 1, gc->d_err);
        k_group_cursors<<<g_sm, 256, 0, st>>>(gc->r_off, gv, s.cur);
        k_group_order<<<g_sm, 256, 0, st>>>(gc->r_off, gv, gc->d_tail, gc->d_tiles_order);
        gc->launches += 5;
    }
    order->count = gc->d_tail;
    order->lists = gc->d_tiles_order;
    order->stride = gv.tile_base[gv.nv];
    // the scatter: every entry a slot in its view's (tile, bin) segment
    if (N > 0)
        k_group_scatter<<<g_sm * 2, 256, 0, st>>>(s.rs_g, s.rs_ya, s.rs_w, s.rs_z, roff, gv, gc->r_m, gc->r_m_cap,
                                                  s.cur, gc->r_stream);
    gc->launches += 1;
    GS_CUDA_TRY(cudaGetLastError());
    // segments longer than the raster sorts in shared memory
    return sort_long_segments(gc, NS, gc->r_off, gc->r_stream, min_len, one_pass, st);
}

}  // namespace gs
