// rows.cuh -- the per-(Gaussian, tile row) span geometry of EXACT bin
// construction with the tile cull (tiles.cu, and its multi-view form in
// batch_bins.cu): which tiles of a row of the Gaussian's rect can hold a pixel
// with alpha >= 1/255, and the row record that carries the span.
#pragma once
#include "internal.cuh"

namespace gs {

// ------------------------------------------------------------------ row spans (tile cull)
struct CullArgs {
    const float4* xy_ab;
    const float4* c_o_z;
    const float4* rgb;
    int tile;
};

// Tiles [*a, *b) of row ty (inside [tx0, tx1)) whose pixel-centre boxes can
// hold a pixel with alpha >= 1/255.  A contributing pixel p has
// Q(m - p) <= tau / margin (the tile cull's bound), so it lies in that
// ellipse; the ellipse meets the row's band of pixel centres in a convex set
// whose x-projection is one interval, found from the band ends and the
// ellipse's leftmost/rightmost points.  Every box is widened (5e-3 relative +
// 0.05 px) to cover float32 rounding; margin 0 (ill-conditioned conic) keeps
// the whole row.  The per-Gaussian part (RowGeom) is computed once by the
// lane that owns the Gaussian; the widening also covers the reciprocals it
// multiplies by in place of divisions.
struct RowGeom {
    float my, hb, inv2ha, a4tp, D, dymax, ext, dyl;  // dymax < 0: keep the whole row
};

__device__ __forceinline__ RowGeom row_geom(float ha, float hb, float hc, float tau, float margin, float my)
{
    RowGeom g;
    g.my = my;
    g.hb = hb;
    g.inv2ha = 0.0f;
    g.a4tp = g.D = g.ext = g.dyl = 0.0f;
    g.dymax = -1.0f;
    if (!(margin > 0.0f)) return g;
    const float tp = tau / margin;
    const float D = 4.0f * ha * hc - hb * hb;
    if (!(D > 0.0f) || !(tp > 0.0f)) return g;
    g.D = D;
    g.a4tp = 4.0f * ha * tp;
    g.dymax = sqrtf(g.a4tp / D) * (1.0f + 5e-3f) + 0.05f;
    g.ext = sqrtf(4.0f * hc * tp / D);
    g.dyl = hb * g.ext / (2.0f * hc);  // dy of the leftmost point (dx = -ext)
    g.inv2ha = 1.0f / (2.0f * ha);
    return g;
}

__device__ __forceinline__ void row_span(float mx, const RowGeom& g, int ty, int tile, float inv_tile, int tx0,
                                         int tx1, int* a, int* b)
{
    *a = tx0;
    *b = tx1;
    if (g.dymax < 0.0f) return;
    const float y0 = (float)(ty * tile);
    float yl = g.my - (y0 + (float)tile - 0.5f), yh = g.my - (y0 + 0.5f);
    yl = yl - (0.05f + 5e-3f * fabsf(yl));
    yh = yh + (0.05f + 5e-3f * fabsf(yh));
    const float ya = fmaxf(yl, -g.dymax), yb = fminf(yh, g.dymax);
    if (ya > yb) {
        *b = *a;  // the band misses the ellipse
        return;
    }
    // the hardware's approximate square root (relative error below 2^-22):
    // the widening below is 5e-3 relative + 0.05 px
    float s_a, s_b;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s_a) : "f"(fmaxf(0.0f, g.a4tp - g.D * ya * ya)));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s_b) : "f"(fmaxf(0.0f, g.a4tp - g.D * yb * yb)));
    const float La = (-g.hb * ya - s_a) * g.inv2ha, Lb = (-g.hb * yb - s_b) * g.inv2ha;
    const float Ra = (-g.hb * ya + s_a) * g.inv2ha, Rb = (-g.hb * yb + s_b) * g.inv2ha;
    float dxmin = (g.dyl >= ya && g.dyl <= yb) ? -g.ext : fminf(La, Lb);
    float dxmax = (-g.dyl >= ya && -g.dyl <= yb) ? g.ext : fmaxf(Ra, Rb);
    dxmin = dxmin - (0.05f + 5e-3f * fabsf(dxmin));
    dxmax = dxmax + (0.05f + 5e-3f * fabsf(dxmax));
    const float ft = (float)tile;
    float fa = ceilf((mx - dxmax - (ft - 0.5f)) * inv_tile), fb = floorf((mx - dxmin - 0.5f) * inv_tile) + 1.0f;
    fa = fminf(fmaxf(fa, (float)tx0), (float)tx1);
    fb = fminf(fmaxf(fb, (float)tx0), (float)tx1);
    *a = (int)fa;
    *b = fb > fa ? (int)fb : (int)fa;
}

// Row record word: tile row (12 bits) | first tile of the span (12 bits) |
// bin (8 bits); exact_bins checks tiles_x, tiles_y <= 4096 (K <= 128 < 256).
__device__ __forceinline__ uint32_t row_record(int ty, int a, uint32_t bin)
{
    return (uint32_t)ty | ((uint32_t)a << 12) | (bin << 24);
}

// ------------------------------------------------------------------ scatter
// The cursors of one bin lie tile by tile (Cursors): the entries of a record,
// which neighbouring lanes hold, take their slots from neighbouring words, so
// that a warp's atomic instruction reaches the L2 as a few sectors instead of
// one a lane (bin stage at 1080p, 1M Gaussians, with two records a lane: 203 -> 182 us).
struct Cursors {
    int32_t* p;
    int64_t tile, bin;  // strides
    __device__ __forceinline__ int32_t* at(int64_t t, int b) const { return p + t * tile + b * bin; }
};

constexpr int kScatIF = 8;                 // entries a lane has in flight
constexpr int kScatWin = 32 * kScatIF;     // entries a warp places a round

// Per warp: its 32 records {gid, depth bits, first entry, first cursor}, and
// for a round's window of entries the record of each.
struct ScatterShared {
    uint4 rec[32];
    uint8_t own[kScatWin];
};

struct KeepAll {
    __device__ __forceinline__ bool operator()(int, uint32_t) const { return true; }
};

// Warp-cooperative over the entries of 32 consecutive row records, one a
// lane: a warp scans the records' widths and keeps its records (gid, tile row
// | first tile | bin, depth bits, first entry) in shared memory; then, a
// window of 256 entries at a time, each record marks the window's entries that
// are its own in a per-warp owner map, and each lane takes every 32nd entry,
// reads its record through the map and takes a slot in the entry's (tile, bin)
// segment -- the cursors start at the segment offsets, so the atomic returns
// the slot itself.  Up to eight entries per lane are in flight: the kernel
// waits on its atomics' returns.  Measured at 1080p (bin stage): two records a
// lane with 12 in flight 182-184 us, one with 16 / 12 / 8 / 6 / 4 in flight
// 182 / 172 / 170 / 172 / 176 us (a warp's 32 records hold about 70 entries);
// more resident blocks at fewer registers no faster.  Against the owner map,
// a binary search over the warp's prefix with the fields shuffled from the
// owning lane was slower by 7 us.  The records carry the Gaussian's bin and
// depth bits, so nothing is gathered.
// The calling lane's record: w entries of item g with depth bits z, the first
// one's cursor at cur[slot], the next ones' `stride` words apart.  keep(o, d):
// whether entry d of lane o's record is placed.  Whole warp.
template <class Keep>
__device__ __forceinline__ void scatter_row_records(uint32_t w, uint32_t g, uint32_t z, uint32_t slot, uint32_t stride,
                                                    int32_t* __restrict__ cur, uint64_t* __restrict__ words,
                                                    ScatterShared& sm, const Keep keep)
{
    const int lane = threadIdx.x & 31;
    uint32_t incl = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t st = incl - w;
    sm.rec[lane] = make_uint4(g, z, st, slot);
    for (uint32_t e0 = 0; e0 < total; e0 += kScatWin) {
        // each record marks the entries of this window that are its own
        const uint32_t lo = st > e0 ? st : e0, wend = e0 + kScatWin;
        const uint32_t hi = incl < wend ? incl : wend;
        for (uint32_t x = lo; x < hi; ++x) sm.own[x - e0] = (uint8_t)lane;
        __syncwarp();
        int32_t p[kScatIF];
        uint64_t word[kScatIF];
        bool live[kScatIF];
#pragma unroll
        for (int u = 0; u < kScatIF; ++u) {
            const uint32_t e = e0 + 32 * u + lane;
            live[u] = e < total;
            if (live[u]) {
                const int o = sm.own[e - e0];
                const uint4 r = sm.rec[o];
                live[u] = keep(o, e - r.z);
                if (live[u]) {
                    p[u] = atomicAdd(cur + r.w + (e - r.z) * stride, 1);
                    word[u] = ((uint64_t)r.y << 32) | r.x;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kScatIF; ++u)
            if (live[u]) words[p[u]] = word[u];
        __syncwarp();  // the window's owner map is read before the next one is written
    }
    __syncwarp();  // the records are read before the next ones are written
}

}  // namespace gs
