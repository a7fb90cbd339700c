// depth_range.cuh -- the robust depth-range estimate (supplement, "Robust
// depth-range estimation", Alg. 2) as the body of one block, and the bin
// parameters it feeds (the log-depth-bin formula; monotone split depths for
// EXACT mode).  Used per frame by bins.cu and per view by batch_bins.cu.
#pragma once
#include "device.cuh"

namespace gs {

// ------------------------------------------------------------------ depth range
constexpr int kDrThreads = 1024;
constexpr int kDrMaxS = 8192;

constexpr int kDrBits = 11;            // bits of a radix pass
constexpr int kDrBins = 1 << kDrBits;  // 64 a warp of the block

struct DrArgs {
    float near_plane, far_plane;
    int S;
    int near_shift;
    float near_alpha, near_gamma;
    float pad, eps;
    double lo, hi;  // the percentiles as fractions of 1
    int K;
};

// Of a context's settings; near_shift only where the mode shifts the keys.
inline DrArgs dr_args(const gs_config& c, int near_shift, float near_plane, float far_plane, int K)
{
    DrArgs a;
    a.near_plane = near_plane;
    a.far_plane = far_plane;
    a.S = c.sample_count;
    a.near_shift = near_shift;
    a.near_alpha = c.near_alpha;
    a.near_gamma = c.near_gamma;
    a.pad = c.pad;
    a.eps = c.eps;
    a.lo = (double)c.p_lo / 100.0;
    a.hi = (double)c.p_hi / 100.0;
    a.K = K;
    return a;
}

__device__ __forceinline__ float zkey_of(float z, const float* __restrict__ scales, uint32_t g, float a, float gm)
{
    const float s0 = __ldg(scales + 3 * (size_t)g), s1 = __ldg(scales + 3 * (size_t)g + 1),
                s2 = __ldg(scales + 3 * (size_t)g + 2);
    const float smax = fmaxf(fmaxf(s0, s1), s2);
    return z - fminf(a * smax, gm * z);
}

__device__ __forceinline__ int rank_of(double p, int n)
{
    const double k = ceil(p * (double)n);
    return k < 1.0 ? 1 : k > (double)n ? n : (int)k;
}

// Bin parameters from [zmin, zmax]: z'min = max(zmin, eps),
// z'max = max(zmax, z'min + 1e-6), lmin/lmax their logs, and K-1 log-spaced
// split depths exp(lmin + (lmax - lmin) k/K), kept non-decreasing (a running
// maximum).  By the block's first warp.
__device__ __forceinline__ void write_bin_params(BinParams* bp, float zmin, float zmax, int K, float eps, int nsamples)
{
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    const float zmn = fmaxf(zmin, eps);
    const float zmx = fmaxf(zmax, zmn + 1e-6f);
    const float l = spec_log(lane == 0 ? zmn : zmx);
    const float lmin = __shfl_sync(0xffffffffu, l, 0), lmax = __shfl_sync(0xffffffffu, l, 1);
    if (lane == 0) {
        bp->zmin = zmin;
        bp->zmax = zmax;
        bp->lmin = lmin;
        bp->lmax = lmax;
        bp->K = K;
        bp->nsamples = nsamples;
    }
    float carry = -INFINITY;
    for (int k0 = 1; k0 < K; k0 += 32) {
        const float t = (float)(k0 + lane) / (float)K;
        float s = spec_exp(lmin + (lmax - lmin) * t);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float u = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= d && s < u) s = u;
        }
        if (s < carry) s = carry;
        carry = __shfl_sync(0xffffffffu, s, 31);
        if (k0 + lane < K) bp->splits[k0 + lane - 1] = s;
    }
}

// The samples' keys themselves (depth, or the near-shifted key, as float
// bits), gathered by a wide sampling kernel.
struct KeyFromSamples {
    static constexpr bool kKeys = true;
    const uint32_t* key;  // indexed by sample number
    __device__ uint32_t operator()(int64_t i, int64_t) const { return key[i]; }
};

// The key of Gaussian g's depth sample: its depth, or the near-shifted key.
__device__ __forceinline__ float sample_key(const float4* __restrict__ c_o_z, const float* __restrict__ scales,
                                            uint32_t g, const DrArgs& a)
{
    float z = c_o_z[g].z;
    if (a.near_shift) z = zkey_of(z, scales, g, a.near_alpha, a.near_gamma);
    return z;
}

// The bin of h[0..64 * 32) whose cumulative count first reaches k (k >= 1),
// by one warp: lane l's group is the 64 bins from 64 l on, group its count.
// k is left less the counts before the bin.
__device__ __forceinline__ uint32_t warp_bin_select(const uint32_t* __restrict__ h, uint32_t group, int& k)
{
    const int lane = threadIdx.x & 31;
    auto scan = [&](uint32_t v) {
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v += u;
        }
        return v;
    };
    const uint32_t gi = scan(group);
    const int L = __ffs(__ballot_sync(0xffffffffu, (int)gi >= k)) - 1;
    k -= (int)__shfl_sync(0xffffffffu, gi - group, L);
    const uint2 c = *reinterpret_cast<const uint2*>(h + 64 * L + 2 * lane);
    const uint32_t bi = scan(c.x + c.y);
    const int l = __ffs(__ballot_sync(0xffffffffu, (int)bi >= k)) - 1;
    k -= (int)__shfl_sync(0xffffffffu, bi - c.x - c.y, l);
    const int cx = (int)__shfl_sync(0xffffffffu, c.x, l);
    const uint32_t bin = 64u * L + 2u * l + (k > cx ? 1u : 0u);
    if (k > cx) k -= cx;
    return bin;
}

// Alg. 2 by one block of kDrThreads threads over the first S' = min(S, M)
// samples gid_of(i, floor(i M / S')) of M entries: the positive depths (or
// near-shifted keys) clamped to [max(near, eps), far], their exact p_lo / p_hi
// order statistics by radix select on the float bits (positive floats: bit
// order = value order) above the least, padded by pad of the span; the bin
// parameters of [zmin, zmax] are written to bp.
//
// One block and a chain of barriers: what it costs is latency, so each thread
// keeps its samples in registers, a pass takes 11 bits (two or three passes),
// the first counts once for both ranks, and every warp sums its 64 bins for
// the two that select.  (Samples compacted in shared memory, passes of 8 bits,
// splits kept monotone by one thread: 13.7 us a frame, now 7.5.)
template <class GidOf>
__device__ __forceinline__ void depth_range_block(const float4* __restrict__ c_o_z, const float* __restrict__ scales,
                                                  GidOf gid_of, int64_t M, const DrArgs& a, BinParams* bp)
{
    static_assert(kDrBins == 64 * (kDrThreads / 32), "64 bins a warp");
    __shared__ __align__(8) uint32_t s_h[2][kDrBins];
    __shared__ uint32_t s_red[3][kDrThreads / 32];
    __shared__ uint32_t s_pref[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ns = (int)(M < (int64_t)a.S ? M : (int64_t)a.S);
    const float lo_clamp = fmaxf(a.near_plane, a.eps);
    // every sample's key: read (the sampling kernel gathered them), or its
    // gid then its depth (and scale) gathered at once, so the dependent loads
    // cost two round trips rather than two per round
    constexpr int kPer = kDrMaxS / kDrThreads;
    float zk[kPer];
    if constexpr (GidOf::kKeys) {
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            const int i = r * kDrThreads + (int)threadIdx.x;
            zk[r] = i < ns ? __uint_as_float(gid_of(i, 0)) : 0.0f;
        }
    } else {
        // floor(x / ns) by a multiply (the product's high word is it or one
        // less): a 64-bit division a sample was a quarter of the kernel
        const uint64_t inv = ns > 0 ? ~0ull / (uint64_t)ns : 0ull;
        uint32_t gk[kPer];
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            const int i = r * kDrThreads + (int)threadIdx.x;
            const uint64_t x = (uint64_t)i * (uint64_t)M;
            uint64_t j = __umul64hi(x, inv);
            if ((j + 1) * (uint64_t)ns <= x) ++j;
            gk[r] = i < ns ? gid_of(i, (int64_t)j) : 0u;
        }
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            const int i = r * kDrThreads + (int)threadIdx.x;
            zk[r] = i < ns ? sample_key(c_o_z, scales, gk[r], a) : 0.0f;
        }
    }
    // the positive keys, clamped (dropped: all bits set); their count, minimum
    // and maximum
    uint32_t v[kPer], lo_v = 0xffffffffu, hi_v = 0u, cnt = 0u;
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const bool keep = zk[r] > 0.0f;
        v[r] = keep ? __float_as_uint(fminf(fmaxf(zk[r], lo_clamp), a.far_plane)) : 0xffffffffu;
        if (keep) {
            lo_v = min(lo_v, v[r]);
            hi_v = max(hi_v, v[r]);
            ++cnt;
        }
    }
    lo_v = __reduce_min_sync(0xffffffffu, lo_v);
    hi_v = __reduce_max_sync(0xffffffffu, hi_v);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) {
        s_red[0][warp] = lo_v;
        s_red[1][warp] = hi_v;
        s_red[2][warp] = cnt;
    }
    reinterpret_cast<uint2*>(s_h[0])[threadIdx.x] = make_uint2(0u, 0u);
    __syncthreads();
    lo_v = __reduce_min_sync(0xffffffffu, s_red[0][lane]);
    hi_v = __reduce_max_sync(0xffffffffu, s_red[1][lane]);
    const int n = (int)__reduce_add_sync(0xffffffffu, s_red[2][lane]);
    float zmin, zmax;
    if (n == 0) {
        zmin = lo_clamp;
        zmax = a.far_plane;
    } else {
        int k = 0;  // warps 0 and 1: the rank left to find, lower and upper
        if (warp < 2) k = rank_of(warp == 0 ? a.lo : a.hi, n);
        uint32_t p0 = 0u, p1 = 0u;  // the bits found, of key - lo_v
        for (int left = 32 - __clz(hi_v - lo_v); left > 0;) {
            const int w = left < kDrBits ? left : kDrBits;
            const int shift = left - w;
            const bool both = p0 == p1;  // one count serves both ranks
#pragma unroll
            for (int r = 0; r < kPer; ++r) {
                const uint32_t u = v[r] - lo_v;
                const uint32_t top = u >> left;  // left <= 31: both are positive floats' bits
                const uint32_t dg = (u >> shift) & ((1u << w) - 1u);
                if (v[r] == 0xffffffffu) continue;
                if (top == p0) atomicAdd(&s_h[0][dg], 1u);
                if (!both && top == p1) atomicAdd(&s_h[1][dg], 1u);
            }
            __syncthreads();
            const uint2 c0 = *reinterpret_cast<const uint2*>(&s_h[0][64 * warp + 2 * lane]);
            const uint2 c1 = *reinterpret_cast<const uint2*>(&s_h[1][64 * warp + 2 * lane]);
            const uint32_t g0 = __reduce_add_sync(0xffffffffu, c0.x + c0.y);
            const uint32_t g1 = __reduce_add_sync(0xffffffffu, c1.x + c1.y);
            if (lane == 0) {
                s_red[0][warp] = g0;
                s_red[1][warp] = both ? g0 : g1;
            }
            __syncthreads();
            if (warp < 2) {
                const uint32_t bin = warp_bin_select(s_h[both ? 0 : warp], s_red[warp][lane], k);
                if (lane == 0) s_pref[warp] = ((warp == 0 ? p0 : p1) << w) | bin;
            }
            __syncthreads();
            p0 = s_pref[0];
            p1 = s_pref[1];
            left = shift;
            if (left > 0) {
                reinterpret_cast<uint2*>(s_h[0])[threadIdx.x] = make_uint2(0u, 0u);
                reinterpret_cast<uint2*>(s_h[1])[threadIdx.x] = make_uint2(0u, 0u);
                __syncthreads();
            }
        }
        const float zlo = __uint_as_float(p0 + lo_v);
        const float zhi = __uint_as_float(p1 + lo_v);
        const float span = fmaxf(zhi - zlo, 1e-6f);
        zmin = fmaxf(a.near_plane, zlo - a.pad * span);
        zmax = fminf(a.far_plane, zhi + a.pad * span);
    }
    write_bin_params(bp, zmin, zmax, a.K, a.eps, n);
}

}  // namespace gs
