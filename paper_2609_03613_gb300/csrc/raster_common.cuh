// raster_common.cuh -- what the forward raster (raster.cu) and its backward
// (raster_bwd.cu) share: the batch staging of a tile's entries into shared
// memory (with the conservative tile-alpha cull and the per-warp strip mask)
// and the walk over a tile's span -- either the whole span at once, or, for
// EXACT streams whose repair runs in the raster, chunk by chunk with each
// segment of 2..raster_sort_cap(TILE) entries sorted in shared memory by (depth bits,
// gid) right before it is composited (Sec. 3.5 selective repair; supplement,
// binned raster traversal after repair).  A forward that saves its state for
// the backward stores the sorted chunks back, so the backward walks the same
// order in place.
#pragma once
#include "device.cuh"

namespace gs {

// ------------------------------------------------------------------ packed float32 pairs
__device__ __forceinline__ uint64_t pk2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t same2(float v) { return pk2(v, v); }

// exp(-q) of two q by spec_exp_core's steps (internal.cuh), bit for bit where
// its value is used (0 <= q <= 87).  The reduced argument is carried negated
// (s = -r), which mirrors every rounding: the odd Horner stages come out
// negated and the last one does not.  2^n is applied to the normal result by
// adding n to its exponent field: the low 9 bits of the shifter's bits are
// zero, so bits(k) << 23 is n << 23.
__device__ __forceinline__ void spec_exp_neg2(float q0, float q1, float& e0, float& e1)
{
    const uint64_t q = pk2(q0, q1);
    const uint64_t k = fma2(q, same2(-1.44269504088896341f), same2(12582912.0f));
    const uint64_t n = add2(k, same2(-12582912.0f));
    uint64_t s = fma2(n, same2(0.693145751953125f), q);
    s = fma2(n, same2(1.42860682030941723e-6f), s);
    uint64_t p = fma2(same2(-1.0f / 5040.0f), s, same2(1.0f / 720.0f));
    p = fma2(p, s, same2(-1.0f / 120.0f));
    p = fma2(p, s, same2(1.0f / 24.0f));
    p = fma2(p, s, same2(-1.0f / 6.0f));
    p = fma2(p, s, same2(0.5f));
    p = fma2(p, s, same2(-1.0f));
    p = fma2(p, s, same2(1.0f));
    float p0, p1, k0, k1;
    upk2(p, p0, p1);
    upk2(k, k0, k1);
    e0 = __uint_as_float(__float_as_uint(p0) + (__float_as_uint(k0) << 23));
    e1 = __uint_as_float(__float_as_uint(p1) + (__float_as_uint(k1) << 23));
}

// One staged entry at two pixels of a row (centres x0, x1; y): q of each.
__device__ __forceinline__ void entry_q(const float4& ga, const float4& gb, float x0, float x1, float y, float& q0,
                                        float& q1)
{
    const float dy = ga.y - y;
    const uint64_t dx = pk2(ga.x - x0, ga.x - x1);
    upk2(fma2(dx, fma2(same2(ga.z), dx, same2(ga.w * dy)), same2((gb.x * dy) * dy)), q0, q1);
}

// Values at a lane's P pixels.  Two, of a row of the warp's 8 x 8 block: they
// share dy and the entry's shared-memory reads, and what is done to both runs on
// packed float32 pairs (each half rounded as the scalar operation).  One: a
// pixel of the warp's 8 x 4 block, scalar.
template <int P>
struct Lane;
template <>
struct Lane<2> {
    using V = uint64_t;  // pixel 0 in the low half
    static __device__ __forceinline__ V same(float v) { return same2(v); }
    static __device__ __forceinline__ V put(const float (&v)[2]) { return pk2(v[0], v[1]); }
    static __device__ __forceinline__ void get(V v, float (&o)[2]) { upk2(v, o[0], o[1]); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return fma2(a, b, c); }
    static __device__ __forceinline__ V mul(V a, V b) { return mul2(a, b); }
    static __device__ __forceinline__ void exp_neg(const float (&q)[2], float (&e)[2])
    {
        spec_exp_neg2(q[0], q[1], e[0], e[1]);
    }
    static __device__ __forceinline__ float least(const float (&v)[2]) { return fminf(v[0], v[1]); }
};
template <>
struct Lane<1> {
    using V = float;
    static __device__ __forceinline__ V same(float v) { return v; }
    static __device__ __forceinline__ V put(const float (&v)[1]) { return v[0]; }
    static __device__ __forceinline__ void get(V v, float (&o)[1]) { o[0] = v; }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return fmaf(a, b, c); }
    static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
    static __device__ __forceinline__ void exp_neg(const float (&q)[1], float (&e)[1]) { e[0] = spec_exp_core(-q[0]); }
    static __device__ __forceinline__ float least(const float (&v)[1]) { return v[0]; }
};

// q of one staged entry at the lane's pixels (centres x[h], y).
template <int P>
__device__ __forceinline__ void entry_dist(const float4& ga, const float4& gb, const float (&x)[P], float y, float (&q)[P])
{
    if constexpr (P == 2) {
        entry_q(ga, gb, x[0], x[1], y, q[0], q[1]);
    } else {
        const float dx = ga.x - x[0], dy = ga.y - y;
        q[0] = fmaf(dx, fmaf(ga.z, dx, ga.w * dy), (gb.x * dy) * dy);
    }
}

struct RasterArgs {
    int width, height, tiles_x, n_tiles, stride;
    float bg0, bg1, bg2;
    int32_t gid_base = 0;  // stream words hold gid_base + gid (the last-id output subtracts it)
};

// A warp owns a block of 8 x 4P pixels of the tile, P a lane.  Blocks are laid
// out TILE/8 wide and TILE/4P tall, warps row-major over them; the block of
// the tile has one warp for each.
template <int TILE, int P = 2>
struct TileBlocks {
    static constexpr int BH = 4 * P;                     // rows of a block
    static constexpr int COLS = TILE / 8, ROWS = TILE / BH;
    static constexpr int NW = COLS * ROWS;               // warps of the tile
    static constexpr int NT = 32 * NW;                   // threads of the tile
    __device__ static int x0() { return ((threadIdx.x >> 5) % COLS) * 8; }
    __device__ static int y0() { return ((threadIdx.x >> 5) / COLS) * BH; }
};

// Entries staged per batch.
template <int TILE>
constexpr int raster_batch() { return TILE == 8 ? 128 : 256; }

template <int TILE, int P = 2>
struct RasterShared {
    using TB = TileBlocks<TILE, P>;
    static constexpr int BATCH = raster_batch<TILE>();
    float4 a[BATCH + 1];  // {mx, my, a/2, b}; the last slot of each array is a
    float4 b[BATCH + 1];  // {c/2, o, tau, gid bits}        zero record, which no
    float4 c[BATCH + 1];  // colour, warp mask              pixel ever passes
    // per warp: the slots its mask admits, as byte offsets into a, b, c; read
    // two at a time
    alignas(8) uint16_t list[TB::NW][BATCH + 4];

    // The zero record (before the first block barrier of the kernel).
    __device__ __forceinline__ void init_pad()
    {
        if (threadIdx.x == 0) a[BATCH] = b[BATCH] = c[BATCH] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
};

// The staged entries (of cnt) whose warp mask admits the calling warp, in
// stage order, into sh.list[warp], followed by three references to the zero
// record (a whole round of two or four); returns their count.  Whole warp.
template <int TILE, int P>
__device__ __forceinline__ int warp_strip_list(RasterShared<TILE, P>& sh, int cnt)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int nw = 0;
    for (int j0 = 0; j0 < cnt; j0 += 32) {
        const int j = j0 + lane;
        const bool mine = j < cnt && ((__float_as_uint(sh.c[j].w) >> warp) & 1u);
        const unsigned bal = __ballot_sync(0xffffffffu, mine);
        if (mine) sh.list[warp][nw + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(16 * j);
        nw += __popc(bal);
    }
    if (lane < 3) sh.list[warp][nw + lane] = (uint16_t)(16 * RasterShared<TILE, P>::BATCH);
    __syncwarp();
    return nw;
}

// Warp mask of an entry: bit w is set when the entry's alpha >= 1/255
// ellipse (the tile cull's bound Q(d) <= tau / margin, d = mean - pixel
// centre, widened as there) reaches a pixel centre of warp w's block of the
// tile (origin x0, y0).  Per band of a block's pixel rows the ellipse's
// x-extent over the band's centre rows (the row-span geometry of the bin
// stage: band ends and the ellipse's leftmost / rightmost points) is widened
// by 5e-3 relative + 0.05 px and tested against each block's centre columns,
// so a warp never skips a pixel the entry can reach.  The geometry takes the
// hardware's approximate division and square root (relative errors near
// 2^-22, far inside the widening).
template <int TILE, int P>
__device__ __forceinline__ uint32_t strip_mask(float mx, float my, float ha, float hb, float hc, float tau,
                                               float margin, float x0, float y0)
{
    using WB = TileBlocks<TILE, P>;
    constexpr int NWT = WB::NW;
    const uint32_t all = NWT >= 32 ? 0xffffffffu : ((1u << NWT) - 1u);
    if (!(margin > 0.0f)) return all;
    const float D = 4.0f * ha * hc - hb * hb;
    const float tp = __fdividef(tau, margin);
    if (!(D > 0.0f) || !(tp > 0.0f)) return all;
    const float a4tp = 4.0f * ha * tp;
    const float iD = __fdividef(1.0f, D);
    float dymax, ext;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(dymax) : "f"(a4tp * iD));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(ext) : "f"(4.0f * hc * tp * iD));
    dymax = dymax * (1.0f + 5e-3f) + 0.05f;
    const float dyl = hb * ext * __fdividef(1.0f, 2.0f * hc);  // dy of the leftmost point (dx = -ext)
    const float inv2ha = __fdividef(1.0f, 2.0f * ha);
    uint32_t m = 0u;
#pragma unroll
    for (int by = 0; by < WB::ROWS; ++by) {
        float yl = my - (y0 + (float)(WB::BH * (by + 1)) - 0.5f), yh = my - (y0 + (float)(WB::BH * by) + 0.5f);
        yl = yl - (0.05f + 5e-3f * fabsf(yl));
        yh = yh + (0.05f + 5e-3f * fabsf(yh));
        const float ya = fmaxf(yl, -dymax), yb = fminf(yh, dymax);
        if (ya > yb) continue;  // the band misses the ellipse
        float s_a, s_b;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s_a) : "f"(fmaxf(0.0f, a4tp - D * ya * ya)));
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s_b) : "f"(fmaxf(0.0f, a4tp - D * yb * yb)));
        const float La = (-hb * ya - s_a) * inv2ha, Lb = (-hb * yb - s_b) * inv2ha;
        const float Ra = (-hb * ya + s_a) * inv2ha, Rb = (-hb * yb + s_b) * inv2ha;
        float dxmin = (dyl >= ya && dyl <= yb) ? -ext : fminf(La, Lb);
        float dxmax = (-dyl >= ya && -dyl <= yb) ? ext : fmaxf(Ra, Rb);
        dxmin = dxmin - (0.05f + 5e-3f * fabsf(dxmin));
        dxmax = dxmax + (0.05f + 5e-3f * fabsf(dxmax));
        // pixel centres x with mx - x in [dxmin, dxmax]
        const float xlo = mx - dxmax - x0, xhi = mx - dxmin - x0;
#pragma unroll
        for (int bx = 0; bx < WB::COLS; ++bx)
            if (xlo <= (float)(8 * bx) + 7.5f && xhi >= (float)(8 * bx) + 0.5f) m |= 1u << (by * WB::COLS + bx);
    }
    return m & all;
}

// How a stream's entries are staged (bits of cullmode).
constexpr int kCullTile = 1;   // the tile-alpha cull
constexpr int kCullWarp = 2;   // per-warp masks
constexpr int kPlain = 4;      // neither: the plain raster

// The staged record of entry g from its projected fields p = xy_ab[g],
// q = c_o_z[g] and colour c = rgbv[g]: {mx, my, a/2, b}, {c/2, o, tau, gid
// bits} and the colour with the warp mask in .w (zero when the tile cull
// drops the entry: no warp's list admits it).
template <int TILE, int P>
__device__ __forceinline__ void stage_record(uint32_t g, const float4& p, const float4& q, float4 c, int cullmode,
                                             int tx, int ty, float4& A, float4& B, float4& C)
{
    A = make_float4(p.x, p.y, 0.5f * p.z, p.w);
    // the plain raster takes nothing from the record's cull fields: its
    // early-out bound comes from the opacity itself, within the exp's range
    const float tau = (cullmode & kPlain) ? fminf(fmaxf(logf(255.0f * q.y) + 2e-4f, 0.0f), 87.0f) : q.w;
    B = make_float4(0.5f * q.x, q.y, tau, __uint_as_float(g));
    bool keep = true;
    if (cullmode & kCullTile)
        keep = !tile_culled(A.x, A.y, A.z, A.w, B.x, q.w, c.w, (float)(tx * TILE), (float)(ty * TILE), (float)TILE);
    const uint32_t m = (cullmode & kCullWarp) ? strip_mask<TILE, P>(A.x, A.y, A.z, A.w, B.x, q.w, c.w,
                                                                        (float)(tx * TILE), (float)(ty * TILE))
                                              : 0xffffffffu;
    c.w = __uint_as_float(keep ? m : 0u);
    C = c;
}

// Stage the batch [b0, b0 + BATCH) of n_entries stream words from src (global
// or shared memory): per entry {mx, my, a/2, b}, {c/2, o, tau, gid bits} and
// the colour with the warp mask in .w (zero for an entry the tile cull
// drops).  Returns the number staged (block-uniform); the caller
// synchronises the block before reading sh.
template <int TILE, int P>
__device__ __forceinline__ int stage_batch(const uint64_t* src, int32_t b0, int32_t n_entries,
                                           RasterShared<TILE, P>& sh, const float4* __restrict__ xy_ab,
                                           const float4* __restrict__ c_o_z, const float4* __restrict__ rgbv,
                                           int cullmode, int tx, int ty)
{
    using SH = RasterShared<TILE, P>;
    const int cnt = min(SH::BATCH, n_entries - b0);
    // entry i of the batch goes to slot i: the tile cull and the warp mask
    // leave a zero mask, which no warp's list admits (stream order is kept
    // without a compaction pass)
    auto put = [&](int i) {
        const uint32_t g = (uint32_t)(src[b0 + i] & 0xffffffffull);
        float4 A, B, C;
        stage_record<TILE, P>(g, __ldg(xy_ab + g), __ldg(c_o_z + g), __ldg(rgbv + g), cullmode, tx, ty, A, B, C);
        sh.a[i] = A;
        sh.b[i] = B;
        sh.c[i] = C;
    };
    if constexpr (SH::TB::NT >= SH::BATCH) {
        if ((int)threadIdx.x < cnt) put(threadIdx.x);
    } else {
        for (int i = threadIdx.x; i < cnt; i += SH::TB::NT) put(i);
    }
    return cnt;
}

// Shared memory of the tile walk.
template <int TILE, bool LAZY>
struct WalkShared {
    static constexpr int LOG = TILE == 8 ? 7 : 8;  // buckets of a long segment
    uint64_t sort[LAZY ? raster_sort_cap(TILE) : 1];
    int32_t off[LAZY ? GS_MAX_K + 1 : 1];
    uint16_t boff[LAZY ? (1 << LOG) + 1 : 1];
};

// The sorted position of word `key`, entry i of the chunk held in ws.sort
// (bins bfirst..e-1 from stream position c0): the start of its segment plus
// the number of smaller words in the segment (the words are distinct, their
// low half being the gid).
template <class WS>
__device__ __forceinline__ int chunk_rank(const WS& ws, int i, uint64_t key, int32_t c0, int bfirst, int e)
{
    int lo = bfirst, hi = e - 1;  // the last bin starting at or before i
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (ws.off[mid] - c0 <= i) lo = mid;
        else hi = mid - 1;
    }
    const int s0 = ws.off[lo] - c0, s1 = ws.off[lo + 1] - c0;
    int r = s0;
    for (int j = s0; j < s1; ++j) r += ws.sort[j] < key ? 1 : 0;
    return r;
}

// Walk tile t's span of the stream front to back by NT threads, handing runs
// of entries to span(src, n, checked, base) (src[0] is stream position base;
// returns -1 after consuming all n, or, block-uniformly, the offset within the
// run at which every pixel of the tile had terminated; span.done() is true
// when the calling thread's pixels have terminated; span.stage_at(slot, gid)
// stages one entry of a run of at most kBatch, which span.composite_staged(n,
// base) then composites).  Only bins [kbegin, kend) of the tile's K are walked
// (a planned frame's passes; 0, K: the whole span).
// Not LAZY: one run, [off[t*K], off[t*K + kend]).  LAZY: chunks of
// consecutive segments of at most `cap` entries (and at most one batch), whose
// words are loaded into shared memory, ranked within their segments and
// staged straight at their sorted slots; a single longer segment of up to
// raster_sort_cap(TILE) entries is put in bucket order there and staged batch
// by batch, one beyond that was sorted before the raster and is handed over
// in place.  The chunks are the tile's repair bins.  ws.off holds all K + 1
// bin offsets of the tile on return (LAZY).
// Returns the stream index at which the walk ended: the end of the walked
// bins, or the position (in the composited order) where every pixel had
// terminated.  With writeback (the stream itself), every sorted chunk is also
// stored back in place, so the tile's composited prefix is left in (depth,
// gid) order.
template <int TILE, bool LAZY, int NT, class Span>
__device__ __forceinline__ int32_t walk_tile(const uint64_t* words, const int32_t* __restrict__ off, int t, int K,
                                             int kbegin, int kend, int cap, WalkShared<TILE, LAZY>& ws, Span& span,
                                             uint64_t* writeback = nullptr)
{
    if constexpr (!LAZY) {
        const int32_t s0 = off[(int64_t)t * K + kbegin], s1 = off[(int64_t)t * K + kend];
        const int32_t r = span(words + s0, s1 - s0, false, s0);
        return r < 0 ? s1 : s0 + r;
    } else {
        const unsigned long long* wl = reinterpret_cast<const unsigned long long*>(words);
        cap = min(cap, Span::kBatch);
        for (int b = threadIdx.x; b <= K; b += NT) ws.off[b] = off[(int64_t)t * K + b];
        __syncthreads();
        constexpr int PER = (Span::kBatch + NT - 1) / NT;
        // the chunk that starts with bin b: it ends before the first bin j > b
        // whose end passes the start + cap (bin ends are nondecreasing, so the
        // bins that fit are a prefix): counted 32 bins a ballot by every warp,
        // in place of a serial walk.  Bins without entries are passed over.
        // Its words, when they fit a batch, are loaded at once (the stream is
        // read once: streamed past L2): the next chunk's while this one is
        // staged and composited.
        int b = kbegin, e;
        int32_t c0, len;
        uint64_t key[PER];
        auto find = [&]() {
            len = 0;
            while (b < kend && len == 0) {
                c0 = ws.off[b];
                e = b + 1;
                if (ws.off[b + 1] - c0 <= cap) {
                    const int lane = threadIdx.x & 31;
                    for (int j0 = b + 1; j0 < kend; j0 += 32) {
                        const int j = j0 + lane;
                        const int fit = __popc(__ballot_sync(0xffffffffu, j < kend && ws.off[j + 1] - c0 <= cap));
                        e += fit;
                        if (fit < 32) break;
                    }
                }
                len = ws.off[e] - c0;
                if (len == 0) b = e;
            }
            if (len <= Span::kBatch) {
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int i = threadIdx.x + u * NT;
                    if (i < len) key[u] = __ldcs(wl + c0 + i);
                }
            }
        };
        find();
        while (len > 0) {
            const int32_t at = c0, n = len;
            const int bfirst = b, bend = e;
            b = e;
            if (__syncthreads_count(span.done()) == NT) return at;
            if (n <= Span::kBatch) {
                // each thread finds its words' ranks in their segments and
                // stages each entry straight at its sorted slot: no sorted
                // copy of the chunk (raster 0.264 -> 0.259 ms at 1080p;
                // gathering the entry's fields before the rank count instead
                // held them across it and spilled: 0.291 ms)
                uint64_t mine[PER];
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int i = threadIdx.x + u * NT;
                    mine[u] = key[u];
                    if (i < n) ws.sort[i] = mine[u];
                }
                __syncthreads();
                find();
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int i = threadIdx.x + u * NT;
                    if (i < n) {
                        const int r = chunk_rank(ws, i, mine[u], at, bfirst, bend);
                        if (writeback) writeback[at + r] = mine[u];
                        span.stage_at(r, (uint32_t)mine[u]);
                    }
                }
                __syncthreads();
                span.composite_staged(n, at);  // termination just counted above
                continue;
            }
            if (n > raster_sort_cap(TILE)) {  // sorted before the raster
                const int32_t r = span(words + at, n, true, at);
                if (r >= 0) return at + r;
                find();
                continue;
            }
            // one long segment, into shared memory in order of depth buckets
            // (or sorted by the network): its batches are then staged one by
            // one, each thread ranking the words of the buckets a batch meets,
            // so that batches past the tile's termination are never ranked
            // (119 x 657 pixels of a few deep tiles: raster 303 -> 252 us with
            // four warps a tile; 3M Gaussians seen from inside 162 -> 164)
            using WS = WalkShared<TILE, LAZY>;
            BucketMap map;
            const bool ranked = block_buckets<NT, WS::LOG>(words + at, n, ws.sort, span.scratch(),
                                                           span.scratch() + (1 << WS::LOG), ws.boff, map);
            if (!ranked) bitonic_mem(ws.sort, n, threadIdx.x, NT, SyncBlock{});
            if (writeback)
                for (int i = threadIdx.x; i < n; i += NT) {
                    const uint64_t w = ws.sort[i];
                    writeback[at + (ranked ? bucket_rank(ws.sort, ws.boff, map, w) : i)] = w;
                }
            for (int b0 = 0; b0 < n; b0 += Span::kBatch) {
                if (b0 > 0 && __syncthreads_count(span.done()) == NT) return at + b0;
                const int b1 = min(b0 + Span::kBatch, n);
                const int i0 = ranked ? ws.boff[map.of(ws.sort[b0])] : b0;
                const int i1 = ranked ? ws.boff[map.of(ws.sort[b1 - 1]) + 1] : b1;
                for (int i = i0 + (int)threadIdx.x; i < i1; i += NT) {
                    const uint64_t w = ws.sort[i];
                    const int r = ranked ? bucket_rank(ws.sort, ws.boff, map, w) : i;
                    if (r >= b0 && r < b1) span.stage_at(r - b0, (uint32_t)w);
                }
                __syncthreads();
                span.composite_staged(b1 - b0, at + b0);
            }
            find();
        }
        return ws.off[kend];
    }
}

// The walk of walk_tile in reverse over the entries before stream index
// `end` (a walk_tile result), for a stream sorted throughout or one whose
// composited prefixes the forward wrote back sorted: the span
// [off[t*K], min(end, off[(t+1)*K])) handed to span(src, n) in place.
template <class Span>
__device__ __forceinline__ void walk_tile_rev(const uint64_t* __restrict__ words, const int32_t* __restrict__ off,
                                              int t, int K, int32_t end, Span& span)
{
    const int32_t s0 = off[(int64_t)t * K], s1 = off[(int64_t)(t + 1) * K];
    const int32_t e = end < s1 ? end : s1;
    if (e > s0) span(words + s0, e - s0);
}

}  // namespace gs
