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

// The row records of one warp's 32 consecutive Gaussians (a frame's or a
// batch's items), which are the consecutive records [base, end).  The owners'
// geometry goes to shared memory, the ones with rows close together; a window
// of 32 records finds its owners from the mask of the records that start one,
// and every record is computed by one lane from its owner's fields.
//
// What bounds it: the L2 sectors that the count atomics touch, two ends a
// record.  Both ends of a span in one atomic instruction (they mostly share a
// sector): 1M Gaussians at 1080p 49 -> 37 us, 3M seen from inside 135 -> 102,
// a batch of 16 views 661 -> 478.  The owners through shared memory instead of
// 18 shuffles a window gave 163 -> 135 of the second and nothing of the others;
// five, six, seven blocks an SM 39.7, 38.6, 40.8 us.
constexpr int kRowBlocks = 6;  // blocks of 256 threads an SM
struct RowOwners {
    float4 a[32];  // mx, my, b, 1 / a
    float4 b[32];  // a4tp, D, dymax, ext
    uint4 c[32];   // first tile | first row << 16, past the last tile | bin << 16, depth bits, first record
    uint2 d[32];   // dyl, lane | view << 8
};

struct RowRecords {
    uint32_t *g, *ya, *w, *z;  // (Gaussian, row record, width, depth bits)
};

// Of the lane's Gaussian g0 + lane: records [off, next), rect r, fields p =
// xy_ab, q = c_o_z, margin, bin and view.  +1 and -1 are added at the ends of
// each record's span in row(bin, view, row), a row of difference counts.
template <class Row>
__device__ __forceinline__ void warp_row_spans(RowOwners& own, int64_t g0, int32_t off, int32_t next, int32_t base,
                                               int32_t end, const uint2& r, const float4& p, const float4& q,
                                               float margin, uint32_t bin, int view, int tile, const RowRecords& rs,
                                               Row row)
{
    const int lane = threadIdx.x & 31;
    const bool has = next > off;
    const unsigned owners = __ballot_sync(0xffffffffu, has);
    if (has) {
        const RowGeom g = row_geom(0.5f * p.z, p.w, 0.5f * q.x, q.w, margin, p.y);
        const int i = __popc(owners & ((1u << lane) - 1u));
        own.a[i] = make_float4(p.x, g.my, g.hb, g.inv2ha);
        own.b[i] = make_float4(g.a4tp, g.D, g.dymax, g.ext);
        own.c[i] = make_uint4(r.x, (r.y & 0xffffu) | (bin << 16), __float_as_uint(q.z), (uint32_t)off);
        own.d[i] = make_uint2(__float_as_uint(g.dyl), (uint32_t)lane | ((uint32_t)view << 8));
    }
    __syncwarp();
    const float inv_tile = 1.0f / (float)tile;  // exact: tiles are 8, 16 or 32
    int before = -1;  // the last owner that starts before the window
    for (int32_t e0 = base; e0 < end; e0 += 32) {
        const uint32_t at = (uint32_t)(off - e0);
        const uint32_t starts = __reduce_or_sync(0xffffffffu, has && at < 32u ? 1u << at : 0u);
        const int k = before + __popc(starts & (0xffffffffu >> (31 - lane)));
        before += __popc(starts);
        const int32_t e = e0 + lane;
        uint32_t ya = 0u, wv = 0u;  // the record and its width | view << 16 (0: nothing to count)
        if (e < end) {
            const float4 A = own.a[k], B = own.b[k];
            const uint4 C = own.c[k];
            const uint2 D = own.d[k];
            const RowGeom g{A.y, A.z, A.w, B.x, B.y, B.z, B.w, __uint_as_float(D.x)};
            const int ty = (int)(C.x >> 16) + (e - (int32_t)C.w);
            int a, x1;
            row_span(A.x, g, ty, tile, inv_tile, (int)(C.x & 0xffffu), (int)(C.y & 0xffffu), &a, &x1);
            ya = row_record(ty, a, C.y >> 16);
            wv = (uint32_t)(x1 - a);
            rs.g[e] = (uint32_t)g0 + (D.y & 31u);
            rs.ya[e] = ya;
            rs.w[e] = wv;
            rs.z[e] = C.z;
            wv |= (D.y >> 8) << 16;
        }
        // the two ends of a span lie close together, mostly in one sector:
        // two lanes take them in one atomic instruction, sixteen records each
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t y = __shfl_sync(0xffffffffu, ya, 16 * h + (lane >> 1));
            const uint32_t w = __shfl_sync(0xffffffffu, wv, 16 * h + (lane >> 1));
            if ((w & 0xffffu) == 0u) continue;
            const int at = (int)((y >> 12) & 0xfffu) + (lane & 1 ? (int)(w & 0xffffu) : 0);
            atomicAdd(row(y >> 24, w >> 16, (int)(y & 0xfffu)) + at, lane & 1 ? -1 : 1);
        }
    }
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
