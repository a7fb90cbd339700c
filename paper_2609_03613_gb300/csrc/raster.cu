// raster.cu -- K6 / K16: front-to-back compositing over each tile's span of
// the tile-major stream (Sec. 3.4; supplement "Binned raster traversal after
// repair").  One CTA per tile, one or two pixels a thread, the span consumed in
// batches staged through shared memory, and a block-wide vote ends the tile
// once every pixel has terminated.
//
// Per pixel centre (x + 0.5, y + 0.5) and entry in stream order, in this exact
// float32 order (the same as the compositing definition of the library):
//   dx = mx - px; dy = my - py;
//   q  = fmaf(dx, fmaf(a/2, dx, b*dy), ((c/2)*dy)*dy)
//   skip unless q >= 0;  e = exp(-q) (Cody-Waite/Taylor, internal.cuh)
//   alpha = min(0.99, o*e); skip if alpha < 1/255
//   Tn = T*(1 - alpha); stop before applying if Tn < 1e-4
//   C = fmaf(col, alpha*T, C); T = Tn; last = gid
//
// One kernel for every stream.  Binned streams take the paper's default raster
// additions: a conservative tile-level alpha cull at staging (entries that
// cannot reach alpha >= 1/255 anywhere in the tile are dropped, order kept;
// EXACT streams were culled when built) and per-warp masks.  The plain raster
// of the global-sort path takes neither: every warp visits every entry.  In
// both an entry's exp is evaluated only where q <= tau matters, tau >= ln(255
// o), past which alpha < 1/255 is certain.  The images are identical.
#include <string.h>

#include "raster_common.cuh"

namespace gs {

// The lane's pixel h in its warp's block: (x, y) and (x + 4, y), or (x, y).
template <int P>
__device__ __forceinline__ int lane_x(int lane, int h) { return P == 2 ? (lane & 3) + 4 * h : lane & 7; }
template <int P>
__device__ __forceinline__ int lane_y(int lane) { return P == 2 ? lane >> 2 : lane >> 3; }

// Per-thread compositing state.  A pixel that has stopped (or lies outside the
// image) has a NaN centre, so that no entry passes it again.
template <int P>
struct PixelState {
    using V = typename Lane<P>::V;
    float x[P], y;  // pixel centres
    V T, C0, C1, C2;
    int32_t last[P], ntests[P];
    int32_t stop;   // stream position of the entry that stopped a pixel last
    int live;       // bit h: pixel h is still compositing
    unsigned long long ops;
};

// alpha of one entry where the pixel takes it (pass), else 0.  0 <= q <= tau
// as one unsigned compare of the float bits (negative q and NaN compare above
// any positive tau).
template <int P>
struct EntryAlpha {
    float a[P];
    bool pass[P];
};
template <int P>
__device__ __forceinline__ EntryAlpha<P> entry_alpha(const float (&q)[P], const float4& gb)
{
    using L = Lane<P>;
    float e[P];
    L::exp_neg(q, e);
    L::get(L::mul(L::same(gb.y), L::put(e)), e);
    const uint32_t tau = __float_as_uint(gb.z);
    EntryAlpha<P> r;
#pragma unroll
    for (int h = 0; h < P; ++h) {
        const float f = fminf(0.99f, e[h]);
        r.pass[h] = __float_as_uint(q[h]) <= tau && f >= 1.0f / 255.0f;
        r.a[h] = r.pass[h] ? f : 0.0f;
    }
    return r;
}

// C = fma(colour, w, C) at the lane's pixels.
template <int P>
__device__ __forceinline__ void add_colour(const float4& c, typename Lane<P>::V w, PixelState<P>& st)
{
    using L = Lane<P>;
    st.C0 = L::fma(L::same(c.x), w, st.C0);
    st.C1 = L::fma(L::same(c.y), w, st.C1);
    st.C2 = L::fma(L::same(c.z), w, st.C2);
}

// T (1 - alpha) at the lane's pixels, 1 - alpha rounded once.
template <int P>
__device__ __forceinline__ typename Lane<P>::V transmit(typename Lane<P>::V T, typename Lane<P>::V a)
{
    using L = Lane<P>;
    return L::mul(T, L::fma(a, L::same(-1.0f), L::same(1.0f)));
}

// One entry (id g, stream position pos) with its stops: a pixel whose
// transmittance would fall below 1e-4 stops before it is applied.
template <int P>
__device__ __forceinline__ void apply_with_stops(const EntryAlpha<P>& e, const float4& c, int32_t g, int32_t pos,
                                                 PixelState<P>& st)
{
    using L = Lane<P>;
    float T[P], t[P], a[P];
#pragma unroll
    for (int h = 0; h < P; ++h) a[h] = e.a[h];
    L::get(st.T, T);
    L::get(transmit<P>(st.T, L::put(a)), t);
#pragma unroll
    for (int h = 0; h < P; ++h) {
        if (((st.live >> h) & 1) && t[h] < 1e-4f) {
            st.live &= ~(1 << h);
            st.x[h] = __uint_as_float(0x7fc00000u);
            st.stop = pos;
        }
        if (!((st.live >> h) & 1)) {
            a[h] = 0.0f;
            t[h] = T[h];
        }
        if (a[h] > 0.0f) st.last[h] = g;
    }
    add_colour<P>(c, L::mul(L::put(a), st.T), st);
    st.T = L::put(t);
}

// Composite the cnt staged entries of a batch into the calling thread's
// pixels (slot k is stream position base + k); the warp visits the entries
// its mask admits.  The whole warp stays in the loop until all its pixels have
// stopped (a stopped one passes nothing), so no branch in it diverges.  R
// entries (2 or 4) go a round: a pixel's transmittance after all of them tells
// whether any stopped it (it never grows), so one vote a round looks for
// stops; a round without one (five in six of two at 1080p) is one straight
// run, the others go entry by entry.
//
// What bounds it: register reads and issue together.  A packed multiply-add
// reads three register pairs and takes 2.3 to 3 cycles of a scheduler where
// two scalar ones take 2 to 3 (measured), so packing buys issue slots, not
// arithmetic; a round of two takes about 110 instructions for 2 x 64 tests.  Measured
// raster times, 1M Gaussians at 1080p / 3M inside a cluster at 1080p / 500k
// global at 720p: one pixel a lane, scalar, 8 x 4 blocks 254 / 207 / 560 us;
// this loop with lanes leaving at their stops 250 / 180 / 481 us; with the
// stops in their own path 235 / 168 / 457 us; with q, opacity and colour
// packed too 229 / 164 / 446 us, the last 276 with SKIP.  Scalar exps 254 / 178 / 496 us; one pixel a
// lane with two entries packed 248 / 203 / 516 us.
//
// SKIP (the plain raster, whose warps visit entries far from their pixels):
// a round no pixel of which has q <= tau ends there.
template <int TILE, int P, bool SKIP, int R>
__device__ __forceinline__ void composite_batch(int cnt, RasterShared<TILE, P>& sh, PixelState<P>& st, int32_t base)
{
    using L = Lane<P>;
    const int warp = threadIdx.x >> 5;
    if (__all_sync(0xffffffffu, st.live == 0)) return;
    const int nk = warp_strip_list(sh, cnt);
    const char* pa = reinterpret_cast<const char*>(sh.a);
    const char* pb = reinterpret_cast<const char*>(sh.b);
    const char* pc = reinterpret_cast<const char*>(sh.c);
    for (int i = 0; i < nk; i += R) {
        uint32_t k[R];
#pragma unroll
        for (int j = 0; j < R; j += 2) {
            const uint32_t pair = *reinterpret_cast<const uint32_t*>(&sh.list[warp][i + j]);
            k[j] = pair & 0xffffu;
            k[j + 1] = pair >> 16;
        }
        float4 gb[R];
        float q[R][P];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            gb[j] = *reinterpret_cast<const float4*>(pb + k[j]);
            entry_dist(*reinterpret_cast<const float4*>(pa + k[j]), gb[j], st.x, st.y, q[j]);
        }
        if constexpr (SKIP) {
            bool any = false;
#pragma unroll
            for (int j = 0; j < R; ++j)
#pragma unroll
                for (int h = 0; h < P; ++h) any |= __float_as_uint(q[j][h]) <= __float_as_uint(gb[j].z);
            if (!__any_sync(0xffffffffu, any)) continue;
        }
        EntryAlpha<P> e[R];
        typename L::V A[R], T[R + 1];
        T[0] = st.T;
#pragma unroll
        for (int j = 0; j < R; ++j) e[j] = entry_alpha<P>(q[j], gb[j]);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            A[j] = L::put(e[j].a);
            T[j + 1] = transmit<P>(T[j], A[j]);
        }
        float t[P];
        L::get(T[R], t);
        if (__any_sync(0xffffffffu, L::least(t) < 1e-4f)) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                apply_with_stops<P>(e[j], *reinterpret_cast<const float4*>(pc + k[j]), __float_as_int(gb[j].w),
                                    base + (int32_t)(k[j] >> 4), st);
            if (__all_sync(0xffffffffu, st.live == 0)) break;
        } else {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                add_colour<P>(*reinterpret_cast<const float4*>(pc + k[j]), L::mul(A[j], T[j]), st);
                const int32_t g = __float_as_int(gb[j].w);
#pragma unroll
                for (int h = 0; h < P; ++h) st.last[h] = e[j].pass[h] ? g : st.last[h];
            }
            st.T = T[R];
        }
    }
}

// The counting twin: one pixel and one entry at a time, the same values.
template <int TILE>
__device__ __forceinline__ void composite_batch_count(int cnt, RasterShared<TILE, 2>& sh, PixelState<2>& st,
                                                      int32_t base)
{
    const int warp = threadIdx.x >> 5;
    const int nk = warp_strip_list(sh, cnt);
    float T[2], C0[2], C1[2], C2[2];
    upk2(st.T, T[0], T[1]);
    upk2(st.C0, C0[0], C0[1]);
    upk2(st.C1, C1[0], C1[1]);
    upk2(st.C2, C2[0], C2[1]);
    for (int i = 0; i < nk && st.live; ++i) {
        const int k = sh.list[warp][i] >> 4;
        const float4 ga = sh.a[k], gb = sh.b[k], col = sh.c[k];
        const float dy = ga.y - st.y;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!((st.live >> h) & 1)) continue;
            const float dx = ga.x - st.x[h];
            const float q = fmaf(dx, fmaf(ga.z, dx, ga.w * dy), (gb.x * dy) * dy);
            const bool inq = __float_as_uint(q) <= __float_as_uint(gb.z);
            const float alpha = inq ? fminf(0.99f, gb.y * spec_exp_core(-q)) : 0.0f;
            const bool pass = alpha >= 1.0f / 255.0f;
            ++st.ntests[h];
            st.ops += 8 + (inq ? 17 : 0) + (pass ? 3 : 0);
            if (!pass) continue;
            const float Tn = T[h] * (1.0f - alpha);
            if (Tn < 1e-4f) {
                st.live &= ~(1 << h);
                st.x[h] = __uint_as_float(0x7fc00000u);
                st.stop = base + k;
                continue;
            }
            st.ops += 4;
            const float w = alpha * T[h];
            C0[h] = fmaf(col.x, w, C0[h]);
            C1[h] = fmaf(col.y, w, C1[h]);
            C2[h] = fmaf(col.z, w, C2[h]);
            T[h] = Tn;
            st.last[h] = __float_as_int(gb.w);
        }
    }
    st.T = pk2(T[0], T[1]);
    st.C0 = pk2(C0[0], C0[1]);
    st.C1 = pk2(C1[0], C1[1]);
    st.C2 = pk2(C2[0], C2[1]);
}

// A run of entries composited into the tile's pixels: what the walk hands its
// runs and staged chunks to (raster_common.cuh).
template <int TILE, int P, bool COUNT, bool LAZY, int R>
struct FwdSpan {
    using SH = RasterShared<TILE, P>;
    static constexpr int kBatch = SH::BATCH;
    SH& sh;
    const float4* __restrict__ xy_ab;
    const float4* __restrict__ c_o_z;
    const float4* __restrict__ rgbv;
    int cullmode, tx, ty;
    PixelState<P>& st;
    // n entries from src (global or shared memory) in batches: -1 after the
    // last, or the offset of the first batch left once every pixel of the
    // tile has terminated
    __device__ __forceinline__ int32_t operator()(const uint64_t* src, int32_t n, bool checked, int32_t base)
    {
        for (int32_t b0 = 0; b0 < n; b0 += kBatch) {
            // checked: the caller has just counted the terminated pixels (block
            // barrier included) with nothing composited since
            if (!(checked && b0 == 0) && __syncthreads_count(done()) == SH::TB::NT) return b0;
            const int cnt = stage_batch(src, b0, n, sh, xy_ab, c_o_z, rgbv, cullmode, tx, ty);
            __syncthreads();
            composite_staged(cnt, base + b0);
        }
        return -1;
    }
    __device__ __forceinline__ bool done() const { return st.live == 0; }
    // shared memory free between the batches (the staging arrays')
    __device__ __forceinline__ uint32_t* scratch() const { return reinterpret_cast<uint32_t*>(sh.a); }
    __device__ __forceinline__ void stage_at(int slot, uint32_t g)
    {
        float4 A, B, C;
        stage_record<TILE, P>(g, __ldg(xy_ab + g), __ldg(c_o_z + g), __ldg(rgbv + g), cullmode, tx, ty, A, B, C);
        sh.a[slot] = A;
        sh.b[slot] = B;
        sh.c[slot] = C;
    }
    __device__ __forceinline__ void composite_staged(int cnt, int32_t base)
    {
        if constexpr (COUNT) {
            composite_batch_count<TILE>(cnt, sh, st, base);
        } else {
            if constexpr (!LAZY)
                if (cullmode & kPlain) return composite_batch<TILE, P, true, R>(cnt, sh, st, base);
            composite_batch<TILE, P, false, R>(cnt, sh, st, base);
        }
    }
};

// LAZY (EXACT mode with the repair in the raster): the tile's segments are
// walked front to back; each segment of 2..raster_sort_cap(TILE) entries is
// loaded into shared memory and sorted by (depth bits, gid) right before it is
// composited (longer ones were sorted eagerly), so segments after every
// pixel's termination are never sorted.
// One tile t by the whole block (the body of the raster kernels below).
template <int TILE, int P, bool COUNT, bool LAZY, int R>
__device__ __forceinline__ void raster_tile(
    int t, RasterShared<TILE, P>& sh, WalkShared<TILE, LAZY>& ws, const float4* __restrict__ xy_ab,
    const float4* __restrict__ c_o_z, const float4* __restrict__ rgbv, uint64_t* words,
    const int32_t* __restrict__ off, const RasterArgs& a, int cullmode, float* __restrict__ out_rgb,
    float* __restrict__ out_alpha, int32_t* __restrict__ out_last, int32_t* __restrict__ out_ntests,
    unsigned long long* __restrict__ ops_total, float* __restrict__ out_T, int32_t* __restrict__ out_end,
    const PlanView& pl, int cap, int32_t* __restrict__ out_wend = nullptr)
{
    using TB = TileBlocks<TILE, P>;
    using L = Lane<P>;
    const int tx = t % a.tiles_x, ty = t / a.tiles_x;
    const int lane = threadIdx.x & 31;
    const int px0 = tx * TILE + TB::x0(), py0 = ty * TILE + TB::y0();  // the warp's block
    const int py = py0 + lane_y<P>(lane);
    int inside = 0;
#pragma unroll
    for (int h = 0; h < P; ++h) inside |= (py < a.height && px0 + lane_x<P>(lane, h) < a.width ? 1 : 0) << h;

    // float32 operations of the compositing definition each pixel executes
    // (COUNT builds): 8 per visit (offsets, q, sign test), 17 more when exp is
    // evaluated (exp, o*e, clamp, threshold), 3 when alpha passes (1-alpha,
    // T*, stop test), 4 when applied (alpha*T and three colour fmas)
    PixelState<P> st;
    st.y = (float)py + 0.5f;
    st.T = L::same(1.0f);
    st.C0 = st.C1 = st.C2 = L::same(0.0f);
#pragma unroll
    for (int h = 0; h < P; ++h) {
        st.last[h] = -1;
        st.ntests[h] = 0;
    }
    st.stop = -1;
    st.ops = 0;
    st.live = inside;

    const int K = a.stride;
    int kbegin = 0, kend = K;
    if (pl.bins) {
        const int B = min((int)pl.bins[t], K);
        if (pl.resume) kbegin = B;
        else kend = B;
    }
    if (pl.resume) {
        float T[P], C[3][P];
#pragma unroll
        for (int h = 0; h < P; ++h) {
            T[h] = 1.0f;
            C[0][h] = C[1][h] = C[2][h] = 0.0f;
            if ((inside >> h) & 1) {
                const int64_t p = (int64_t)py * a.width + px0 + lane_x<P>(lane, h);
                // the first pass's state: C in rgb, T in alpha (negative once the
                // pixel stopped), last
                const float Ts = out_alpha[p];
                T[h] = fabsf(Ts);
                if (signbit(Ts)) st.live &= ~(1 << h);
                C[0][h] = out_rgb[3 * p];
                C[1][h] = out_rgb[3 * p + 1];
                C[2][h] = out_rgb[3 * p + 2];
                st.last[h] = out_last[p];
            }
        }
        st.T = L::put(T);
        st.C0 = L::put(C[0]);
        st.C1 = L::put(C[1]);
        st.C2 = L::put(C[2]);
    }
#pragma unroll
    for (int h = 0; h < P; ++h)
        st.x[h] = (st.live >> h) & 1 ? (float)(px0 + lane_x<P>(lane, h)) + 0.5f : __uint_as_float(0x7fc00000u);
    sh.init_pad();
    FwdSpan<TILE, P, COUNT, LAZY, R> span{sh, xy_ab, c_o_z, rgbv, cullmode, tx, ty, st};
    // saving for the backward: the sorted chunks go back into the stream
    const int32_t end =
        walk_tile<TILE, LAZY, TB::NT>(words, off, t, K, kbegin, kend, cap, ws, span, out_end ? words : nullptr);
    if (out_end && threadIdx.x == 0) out_end[t] = end;
    if (out_wend) {
        // per 8 x 8 block (a warp of the backward), the stream position past the
        // entry that stopped its last pixel (the tile's end when one of its
        // pixels never stopped): the backward has nothing to do for the block
        // at or beyond it
        const int32_t m = __reduce_max_sync(0xffffffffu, !inside ? 0 : (st.live ? end : min(st.stop + 1, end)));
        constexpr int NB = TileBlocks<TILE, 2>::NW;
        const int blk = TB::y0() / 8 * TB::COLS + TB::x0() / 8;
        if constexpr (P == 2) {
            if (lane == 0) out_wend[(int64_t)t * NB + blk] = m;
        } else {
            __shared__ int32_t s_wend[NB];
            if (threadIdx.x < NB) s_wend[threadIdx.x] = 0;
            __syncthreads();
            if (lane == 0) atomicMax(&s_wend[blk], m);
            __syncthreads();
            if (threadIdx.x < NB) out_wend[(int64_t)t * NB + threadIdx.x] = s_wend[threadIdx.x];
        }
    }
    bool unfinished = false;
    if (pl.flag && kend < K) {
        // a planned first pass: a tile with a pixel still compositing when its
        // bins ran out, and entries in later bins, is left to the completing
        // pass with its pixels' state in the outputs
        const bool all_done = __syncthreads_count(st.live == 0) == TB::NT;
        unfinished = !all_done && off[(int64_t)t * K + K] > off[(int64_t)t * K + kend];
        if (unfinished && threadIdx.x == 0) {
            pl.flag[t] = 1;
            pl.flag[a.n_tiles + ty] = 1;
            pl.list[1 + atomicAdd(&pl.list[0], 1)] = t;
        }
    }
    if (COUNT && pl.needed) {
        // the bins the tile needs: through the one holding the last entry any
        // pixel visits (a pixel that never stops visits the whole span)
        __shared__ int32_t s_end;
        const int32_t s0 = off[(int64_t)t * K], s1 = off[(int64_t)t * K + K];
        if (threadIdx.x == 0) s_end = s0;
        __syncthreads();
        if (inside) atomicMax(&s_end, st.live ? s1 : st.stop + 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            int need = 0;
            if (s_end > s0) {
                int lo = 0, hi = K - 1;  // the last bin starting at or before s_end - 1
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (off[(int64_t)t * K + mid] <= s_end - 1) lo = mid;
                    else hi = mid - 1;
                }
                need = lo + 1;
            }
            pl.needed[t] = need;
        }
    }
    float T[P], C0[P], C1[P], C2[P];
    L::get(st.T, T);
    L::get(st.C0, C0);
    L::get(st.C1, C1);
    L::get(st.C2, C2);
    if (unfinished) {  // the transmittance signed by termination
#pragma unroll
        for (int h = 0; h < P; ++h) T[h] = (st.live >> h) & 1 ? T[h] : -T[h];
    }
    const bool odd = (lane & 4) != 0;
    if constexpr (P == 2) {
        // The lanes of two neighbouring rows exchange one pixel each, so that
        // eight lanes hold eight neighbouring pixels of one row (96 bytes of
        // rgb) in each of the two store rounds: a lane of an even row then
        // holds its pixel x of that row and of the next, one of an odd row its
        // pixel x + 4 of the row before and of its own.
        auto pair_rows = [&](auto& v) {
            const auto mine = odd ? v[0] : v[1];
            const auto other = __shfl_xor_sync(0xffffffffu, mine, 4);
            if (odd) v[0] = other;
            else v[1] = other;
        };
        pair_rows(T);
        pair_rows(C0);
        pair_rows(C1);
        pair_rows(C2);
        pair_rows(st.last);
        if (COUNT) pair_rows(st.ntests);
    }
    const int ox = px0 + (P == 2 ? (lane & 3) + (odd ? 4 : 0) : lane_x<P>(lane, 0));
#pragma unroll
    for (int h = 0; h < P; ++h) {
        const int oy = P == 2 ? py0 + ((lane >> 2) & ~1) + h : py;
        if (ox >= a.width || oy >= a.height) continue;
        const int64_t p = (int64_t)oy * a.width + ox;
        if (unfinished) {
            out_rgb[3 * p] = C0[h];
            out_rgb[3 * p + 1] = C1[h];
            out_rgb[3 * p + 2] = C2[h];
            out_alpha[p] = T[h];
            out_last[p] = st.last[h];
        } else {
            // the image is not read again on the device: streaming stores
            __stcs(out_rgb + 3 * p, fmaf(T[h], a.bg0, C0[h]));
            __stcs(out_rgb + 3 * p + 1, fmaf(T[h], a.bg1, C1[h]));
            __stcs(out_rgb + 3 * p + 2, fmaf(T[h], a.bg2, C2[h]));
            __stcs(out_alpha + p, 1.0f - T[h]);
            __stcs(out_last + p, st.last[h] >= 0 ? st.last[h] - a.gid_base : st.last[h]);
            if (out_T) out_T[p] = T[h];
            if (COUNT && out_ntests) out_ntests[p] = st.ntests[h];
        }
    }
    if (COUNT) {
        // block reduction of the op count, one atomic per block
        __shared__ unsigned long long s_ops;
        if (threadIdx.x == 0) s_ops = 0;
        __syncthreads();
        atomicAdd(&s_ops, st.ops);
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(ops_total, s_ops);
    }
}

// The k-th tile of the order (warp-uniform k; -1: there is none).  Whole warp.
__device__ __forceinline__ int ordered_tile(const TileOrder& o, int32_t k)
{
    const int q = kTileLists - 1 - (int)(threadIdx.x & 31);  // longest first
    const int32_t c = o.count[q];
    int32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, incl, d);
        if ((int)(threadIdx.x & 31) >= d) incl += u;
    }
    const unsigned past = __ballot_sync(0xffffffffu, incl > k);
    if (past == 0u) return -1;
    const int l = __ffs(past) - 1;
    const int32_t at = k - __shfl_sync(0xffffffffu, incl - c, l);
    return o.lists[(kTileLists - 1 - l) * o.stride + at];
}

// Threads of a tile's block and the blocks an SM holds: 16 x 16 tiles' seven
// blocks of 128 threads fill the shared memory (32.9 KB each).
template <int TILE, int P = 2>
constexpr int raster_threads() { return TileBlocks<TILE, P>::NT; }
template <int TILE, int P = 2>
constexpr int raster_min_blocks()
{
    return P == 2 ? (TILE == 16 ? 7 : TILE == 8 ? 16 : 2) : (TILE == 16 ? 3 : 12);
}
// Entries a round of composite_batch: four where a warp's registers allow it.
template <int TILE, int P = 2>
constexpr int raster_round() { return P == 1 || TILE == 8 ? 4 : 2; }

template <int TILE, int P, bool COUNT, bool LAZY>
__global__ void __launch_bounds__(raster_threads<TILE, P>(), COUNT ? 1 : raster_min_blocks<TILE, P>())
k_raster(const float4* __restrict__ xy_ab, const float4* __restrict__ c_o_z, const float4* __restrict__ rgbv,
         uint64_t* words, const int32_t* __restrict__ off, RasterArgs a, int cullmode,
         float* __restrict__ out_rgb, float* __restrict__ out_alpha, int32_t* __restrict__ out_last,
         int32_t* __restrict__ out_ntests, unsigned long long* __restrict__ ops_total, float* __restrict__ out_T,
         int32_t* __restrict__ out_end, const PlanView pl, int cap, int32_t* __restrict__ out_wend, const TileOrder ord)
{
    grid_dependency_sync();
    __shared__ RasterShared<TILE, P> sh;
    __shared__ WalkShared<TILE, LAZY> ws;
    const int t = ord.lists ? ordered_tile(ord, (int32_t)blockIdx.x) : (int)blockIdx.x;
    if (t < 0) return;
    raster_tile<TILE, P, COUNT, LAZY, raster_round<TILE, P>()>(t, sh, ws, xy_ab, c_o_z, rgbv, words, off, a, cullmode,
                                                               out_rgb, out_alpha, out_last, out_ntests, ops_total,
                                                               out_T, out_end, pl, cap, out_wend);
}

// The completing pass of a planned frame: persistent blocks take the listed
// tiles ({count, tiles...}) one at a time and composite each on from the bin
// where its first pass stopped, from the pixel state that pass left.
template <int TILE>
__global__ void __launch_bounds__(raster_threads<TILE>(), raster_min_blocks<TILE>())
k_raster_listed(const float4* __restrict__ xy_ab, const float4* __restrict__ c_o_z, const float4* __restrict__ rgbv,
                uint64_t* words, const int32_t* __restrict__ off, RasterArgs a, int cullmode,
                float* __restrict__ out_rgb, float* __restrict__ out_alpha, int32_t* __restrict__ out_last,
                float* __restrict__ out_T, int32_t* __restrict__ out_end, const uint8_t* __restrict__ plan,
                const int32_t* __restrict__ list, int cap)
{
    grid_dependency_sync();
    __shared__ RasterShared<TILE, 2> sh;
    __shared__ WalkShared<TILE, true> ws;
    PlanView pl;
    pl.bins = plan;
    pl.resume = 1;
    const int32_t nl = list[0];
    for (int32_t k = blockIdx.x; k < nl; k += gridDim.x) {
        const int t = list[1 + k];
        raster_tile<TILE, 2, false, true, raster_round<TILE>()>(t, sh, ws, xy_ab, c_o_z, rgbv, words, off, a, cullmode, out_rgb,
                                              out_alpha, out_last, nullptr, nullptr, out_T, out_end, pl, cap);
        __syncthreads();  // the next tile reuses the shared memory
    }
}

// Several views in one persistent launch: blocks take (view, tile) work items
// from a counter, longest tiles first, until all views' tiles are composited.
struct ViewRasterSet {
    struct View {
        const float4* xy_ab;
        const float4* c_o_z;
        const float4* rgbv;
        uint64_t* words;
        const int32_t* off;
        RasterArgs a;
        int cullmode, cap;
        float* rgb;
        float* alpha;
        int32_t* last;
        int32_t item0;  // first work item of the view
    } v[kMaxBatchViews];
    int nviews;
    int32_t total;
};

__device__ __forceinline__ int view_of(const ViewRasterSet& vs, int32_t item)
{
    int v = 0;
    while (v + 1 < vs.nviews && vs.v[v + 1].item0 <= item) ++v;
    return v;
}

template <int TILE, bool LAZY>
__global__ void __launch_bounds__(raster_threads<TILE>(), raster_min_blocks<TILE>())
k_raster_views(const __grid_constant__ ViewRasterSet vs, const TileOrder order, int32_t* __restrict__ counter)
{
    __shared__ RasterShared<TILE, 2> sh;
    __shared__ WalkShared<TILE, LAZY> ws;
    __shared__ int32_t s_item;
    for (;;) {
        if (threadIdx.x < 32) {
            int32_t k = 0;
            if (threadIdx.x == 0) k = atomicAdd(counter, 1);
            const int t = ordered_tile(order, __shfl_sync(0xffffffffu, k, 0));
            if (threadIdx.x == 0) s_item = t;
        }
        __syncthreads();  // also: every thread is done with the previous tile's shared memory
        const int32_t item = s_item;
        __syncthreads();
        if (item < 0) break;
        const ViewRasterSet::View& V = vs.v[view_of(vs, item)];
        raster_tile<TILE, 2, false, LAZY, raster_round<TILE>()>(item - V.item0, sh, ws, V.xy_ab, V.c_o_z, V.rgbv, V.words, V.off, V.a,
                                              V.cullmode, V.rgb, V.alpha, V.last, nullptr, nullptr, nullptr, nullptr,
                                              PlanView(), V.cap);
    }
}

// Whether a frame of T tiles goes by one pixel a lane.  A frame of few tiles
// lasts as long as its deepest tile, whose warps wait for their own results:
// twice the warps of one pixel a lane, each with rounds of four and the
// registers of twelve (8 x 8) or three (16 x 16) blocks an SM, take it down
// faster.  Past some tiles an SM the frame is bound by issue, where two pixels
// a lane need fewer instructions.  Measured, two pixels a lane / one, us:
// 16 x 16 tiles, Gaussians in clusters, 336 tiles 291 / 182, 475 tiles 168 /
// 102, 1200 tiles 65 / 47, 2040 tiles 90 / 88; spread evenly, 475 tiles 49 /
// 41, 1200 tiles 61 / 63, 1900 tiles 93 / 98; seen from inside, 1900 tiles 72 /
// 86.  The plain raster, whose warps visit every entry of a tile: 300 tiles
// 180 / 135, 475 tiles 158 / 145 and, even, 76 / 80, 1200 tiles 147 / 156 and
// 102 / 135.  8 x 8 tiles: 840 tiles 178 / 115, 2646 tiles 63 / 47, 8160 tiles
// 94 / 88 (even, 7500 tiles 102 / 100; plain, 4800 tiles 96 / 95).  32 x 32
// tiles' 32 warps have to share one block's registers: 80 tiles 233 / 223,
// plain 489 / 561, 300 tiles 80 / 94.
static bool one_pixel(const gs_ctx* ctx, int tile, bool plain, int64_t T)
{
    const int64_t per_sm = tile == 8 ? 48 : tile == 16 ? (plain ? 3 : 10) : 0;
    return T <= per_sm * ctx->num_sms;
}

// Whether a frame's tiles are all resident at once (their order is then of no use).
bool raster_resident(const gs_ctx* ctx, int tile, int64_t T)
{
    return T <= (int64_t)ctx->num_sms *
                    (tile == 8 ? raster_min_blocks<8, 1>() : tile == 16 ? raster_min_blocks<16, 1>() : raster_min_blocks<32>());
}

template <int TILE>
static cudaError_t launch_tile(const gs_ctx* ctx, bool count, bool lazy, unsigned grid, cudaStream_t st,
                               const ProjView& pv, uint64_t* words, const int32_t* off, const RasterArgs& a, int cull,
                               float* rgb, float* alpha, int32_t* last, int32_t* ntests, unsigned long long* ops,
                               float* final_T, int32_t* tile_end, const PlanView& pl, int cap, int32_t* warp_end,
                               const TileOrder& order)
{
    constexpr int ONE = TILE == 32 ? 2 : 1;
    const bool one = !count && one_pixel(ctx, TILE, (cull & kPlain) != 0, grid);
    const auto kern = count ? (lazy ? k_raster<TILE, 2, true, true> : k_raster<TILE, 2, true, false>)
                      : one ? (lazy ? k_raster<TILE, ONE, false, true> : k_raster<TILE, ONE, false, false>)
                            : (lazy ? k_raster<TILE, 2, false, true> : k_raster<TILE, 2, false, false>);
    return launch_k(ctx, kern, grid, one ? raster_threads<TILE, ONE>() : raster_threads<TILE>(), 0, st, pv.xy_ab, pv.c_o_z, pv.rgb, words, off, a, cull,
                    rgb, alpha, last, ntests, ops, final_T, tile_end, pl, cap, warp_end, order);
}

int raster_fwd(gs_ctx* ctx, const ProjView& pv, const gs_camera* cam, uint64_t* words,
               const int32_t* offsets, int32_t stride, const float* bg, float* rgb, float* alpha,
               int32_t* last, int32_t* ntests, cudaStream_t st, float* final_T, int32_t* tile_end,
               const PlanView& pl, int32_t* warp_end, const TileOrder& order)
{
    const int tile = ctx->cfg.tile_size;
    RasterArgs a;
    a.width = cam->width;
    a.height = cam->height;
    a.tiles_x = (cam->width + tile - 1) / tile;
    a.n_tiles = gs_num_tiles(cam->width, cam->height, tile);
    a.stride = stride;
    a.bg0 = bg[0];
    a.bg1 = bg[1];
    a.bg2 = bg[2];
    const bool count = ntests != nullptr || pl.needed != nullptr;
    const bool lazy = ctx->cfg.mode == GS_MODE_BINNED_EXACT && ctx->cfg.repair_in_raster;
    // EXACT streams are culled when they are built: no second tile test at
    // staging, only the per-warp mask.  GLOBAL without the cull is the plain
    // raster.
    const bool exact = ctx->cfg.mode == GS_MODE_BINNED_EXACT;
    const int cull_here = ctx->cfg.tile_cull ? (exact ? kCullWarp : kCullTile | kCullWarp)
                                             : (ctx->cfg.mode == GS_MODE_GLOBAL_SORT ? kPlain : 0);
    const int cap = chunk_cap(ctx->cfg);
    const unsigned grid = (unsigned)a.n_tiles;
    if (grid == 0) return GS_OK;
    unsigned long long* ops = reinterpret_cast<unsigned long long*>(ctx->d_ops);
    if (count) GS_CUDA_TRY(cudaMemsetAsync(ops, 0, sizeof(unsigned long long), st));
    cudaError_t e;
    switch (tile) {
        case 8: e = launch_tile<8>(ctx, count, lazy, grid, st, pv, words, offsets, a, cull_here, rgb, alpha, last, ntests, ops, final_T, tile_end, pl, cap, warp_end, order); break;
        case 32: e = launch_tile<32>(ctx, count, lazy, grid, st, pv, words, offsets, a, cull_here, rgb, alpha, last, ntests, ops, final_T, tile_end, pl, cap, warp_end, order); break;
        default: e = launch_tile<16>(ctx, count, lazy, grid, st, pv, words, offsets, a, cull_here, rgb, alpha, last, ntests, ops, final_T, tile_end, pl, cap, warp_end, order); break;
    }
    GS_CUDA_TRY(e);
    ctx->launches += 1;
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

int raster_listed(gs_ctx* ctx, const ProjView& pv, const gs_camera* cam, uint64_t* words, const int32_t* offsets,
                  int32_t stride, const float* bg, float* rgb, float* alpha, int32_t* last, const uint8_t* plan,
                  const int32_t* list, cudaStream_t st, float* final_T, int32_t* tile_end)
{
    const int tile = ctx->cfg.tile_size;
    RasterArgs a;
    a.width = cam->width;
    a.height = cam->height;
    a.tiles_x = (cam->width + tile - 1) / tile;
    a.n_tiles = gs_num_tiles(cam->width, cam->height, tile);
    a.stride = stride;
    a.bg0 = bg[0];
    a.bg1 = bg[1];
    a.bg2 = bg[2];
    if (a.n_tiles == 0) return GS_OK;
    // EXACT streams are culled when built: the strip mask only
    const int cull = ctx->cfg.tile_cull ? kCullWarp : 0;
    const int cap = chunk_cap(ctx->cfg);
    switch (tile) {
        case 8: GS_CUDA_TRY(launch_k(ctx, k_raster_listed<8>, (unsigned)ctx->num_sms * 8, raster_threads<8>(), 0, st, pv.xy_ab, pv.c_o_z, pv.rgb, words, offsets, a, cull, rgb, alpha, last, final_T, tile_end, plan, list, cap)); break;
        case 32: GS_CUDA_TRY(launch_k(ctx, k_raster_listed<32>, (unsigned)ctx->num_sms, raster_threads<32>(), 0, st, pv.xy_ab, pv.c_o_z, pv.rgb, words, offsets, a, cull, rgb, alpha, last, final_T, tile_end, plan, list, cap)); break;
        default: GS_CUDA_TRY(launch_k(ctx, k_raster_listed<16>, (unsigned)ctx->num_sms * raster_min_blocks<16>(), raster_threads<16>(), 0, st, pv.xy_ab, pv.c_o_z, pv.rgb, words, offsets, a, cull, rgb, alpha, last, final_T, tile_end, plan, list, cap)); break;
    }
    ctx->launches += 1;
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

int raster_views(gs_ctx* ctx, const RasterView* views, int nv, const TileOrder& order, int32_t* work, cudaStream_t st)
{
    if (nv < 1 || nv > kMaxBatchViews) return GS_ERR_INVALID_ARG;
    ViewRasterSet vs;
    memset(&vs, 0, sizeof(vs));
    int32_t total = 0;
    for (int i = 0; i < nv; ++i) {
        const RasterView& r = views[i];
        ViewRasterSet::View& V = vs.v[i];
        const int tile = 16;
        V.xy_ab = r.pv.xy_ab;
        V.c_o_z = r.pv.c_o_z;
        V.rgbv = r.pv.rgb;
        V.words = r.words;
        V.off = r.offsets;
        V.a.width = r.cam.width;
        V.a.height = r.cam.height;
        V.a.tiles_x = (r.cam.width + tile - 1) / tile;
        V.a.n_tiles = gs_num_tiles(r.cam.width, r.cam.height, tile);
        V.a.stride = r.stride;
        V.a.bg0 = r.bg[0];
        V.a.bg1 = r.bg[1];
        V.a.bg2 = r.bg[2];
        V.cullmode = r.cull ? kCullWarp : 0;
        V.cap = r.cap;
        V.rgb = r.rgb;
        V.alpha = r.alpha;
        V.last = r.last;
        V.a.gid_base = r.gid_base;
        V.item0 = total;
        total += V.a.n_tiles;
    }
    vs.nviews = nv;
    vs.total = total;
    if (total == 0) return GS_OK;
    const int held = ctx->num_sms * raster_min_blocks<16>();
    const unsigned grid = (unsigned)(held < total ? held : total);
    k_raster_views<16, true><<<grid, raster_threads<16>(), 0, st>>>(vs, order, work);
    ctx->launches += 1;
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

}  // namespace gs
