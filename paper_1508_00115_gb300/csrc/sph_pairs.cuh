// sph_pairs.cuh -- what the pair kernels share: the stencil orders, the source stream of
// a leaf list, tile reductions and the pair terms.
#pragma once

#include "sph_internal.cuh"

namespace sph {

constexpr int kPairThreads = 256;
// Padding sources sit at -kFar and target-less lanes at +kFar: the squared distance
// between either and anything else overflows to +inf, so no test can pass.
constexpr float kFar = 1e30f;
// an h bracket end at or above this is open (the bytes 0x7f7f7f7f read 3.39e38)
constexpr float kHUnbounded = 3e38f;
// relative width of an h bracket at which the iteration stops refining (2^-21: 4 to 8
// FP32 ulps of h); near the root the FP32 neighbour sums are noisy at about this level
// of h, so that for particles whose N_w is very sensitive to h a tolerance far below
// 1e-5 may have no FP32 h that meets it
constexpr float kHResolution = 4.76837158e-7f;
// a little less: the nudge of an h whose Newton step is below its last bit
constexpr float kHNudge = 4.3e-7f;

// Neighbour cells in visiting order: the own cell, then each of the 13 directions
// of a half stencil followed by its opposite, so that every staged batch mixes
// cells on both sides of the tile and the lanes' hit counts stay balanced.
static __constant__ signed char kOrder[27][3] = {
    {0, 0, 0},   {1, 0, 0},   {-1, 0, 0},  {0, 1, 0},   {0, -1, 0},   {0, 0, 1},  {0, 0, -1},
    {1, 1, 0},   {-1, -1, 0}, {1, -1, 0},  {-1, 1, 0},  {1, 0, 1},    {-1, 0, -1}, {1, 0, -1},
    {-1, 0, 1},  {0, 1, 1},   {0, -1, -1}, {0, 1, -1},  {0, -1, 1},   {1, 1, 1},  {-1, -1, -1},
    {1, 1, -1},  {-1, -1, 1}, {1, -1, 1},  {-1, 1, -1}, {-1, 1, 1},   {1, -1, -1}};

// Radius-2 stencils visit the 27 cells above, in that order, then the 98 cells at
// distance two (z, y, x lexicographic), so a tile's summation order never depends
// on which stencil its warp runs.
static __constant__ signed char kOuter[98][3] = {
    {-2, -2, -2}, {-1, -2, -2}, {0, -2, -2}, {1, -2, -2}, {2, -2, -2}, {-2, -1, -2}, {-1, -1, -2},
    {0, -1, -2}, {1, -1, -2}, {2, -1, -2}, {-2, 0, -2}, {-1, 0, -2}, {0, 0, -2}, {1, 0, -2},
    {2, 0, -2}, {-2, 1, -2}, {-1, 1, -2}, {0, 1, -2}, {1, 1, -2}, {2, 1, -2}, {-2, 2, -2},
    {-1, 2, -2}, {0, 2, -2}, {1, 2, -2}, {2, 2, -2}, {-2, -2, -1}, {-1, -2, -1}, {0, -2, -1},
    {1, -2, -1}, {2, -2, -1}, {-2, -1, -1}, {2, -1, -1}, {-2, 0, -1}, {2, 0, -1}, {-2, 1, -1},
    {2, 1, -1}, {-2, 2, -1}, {-1, 2, -1}, {0, 2, -1}, {1, 2, -1}, {2, 2, -1}, {-2, -2, 0},
    {-1, -2, 0}, {0, -2, 0}, {1, -2, 0}, {2, -2, 0}, {-2, -1, 0}, {2, -1, 0}, {-2, 0, 0},
    {2, 0, 0}, {-2, 1, 0}, {2, 1, 0}, {-2, 2, 0}, {-1, 2, 0}, {0, 2, 0}, {1, 2, 0},
    {2, 2, 0}, {-2, -2, 1}, {-1, -2, 1}, {0, -2, 1}, {1, -2, 1}, {2, -2, 1}, {-2, -1, 1},
    {2, -1, 1}, {-2, 0, 1}, {2, 0, 1}, {-2, 1, 1}, {2, 1, 1}, {-2, 2, 1}, {-1, 2, 1},
    {0, 2, 1}, {1, 2, 1}, {2, 2, 1}, {-2, -2, 2}, {-1, -2, 2}, {0, -2, 2}, {1, -2, 2},
    {2, -2, 2}, {-2, -1, 2}, {-1, -1, 2}, {0, -1, 2}, {1, -1, 2}, {2, -1, 2}, {-2, 0, 2},
    {-1, 0, 2}, {0, 0, 2}, {1, 0, 2}, {2, 0, 2}, {-2, 1, 2}, {-1, 1, 2}, {0, 1, 2},
    {1, 1, 2}, {2, 1, 2}, {-2, 2, 2}, {-1, 2, 2}, {0, 2, 2}, {1, 2, 2}, {2, 2, 2},};

// The sources of a tile's leaf list as one stream (adaptive cells).  The TW entries
// of a window are fetched at once (lane tl: entry wb + tl), their particle counts are
// prefix-summed across the TW lanes, and chunk ch of the window covers stream
// positions [ch TW, ch TW + TW): leaves much smaller than TW share a chunk instead of
// each leaving lanes idle.  The stream order -- entries in list order, particles in
// slot order -- is that of the entries taken one by one.
template <int TW>
struct ListStream {
    int wb = -TW;  // first entry of the window (warp-uniform)
    int incl = 0;  // prefix count of the window's entries up to this lane's, inclusive
    int st = 0;    // stream position of this lane's entry (its first particle)
    int sb = 0;    // first slot of this lane's entry minus its stream position
    int tot = 0;   // particles in this tile's window
    float px = 0.f, py = 0.f, pz = 0.f;  // offset of this lane's entry

    // next window (warp-uniform); false once the longest list of the warp is done;
    // *nchunk = the warp's largest chunk count of the window.  An entry whose leaf box
    // (moved by the entry's offset) lies beyond reach of the tile's box contributes no
    // sources: the staging would reject every one of them.  Reach: sqrt(reach2) for the
    // density (targets' h); for the force (FORCE) the larger of the targets' h and the
    // leaf's largest current h (set before the force pass).
    template <bool FORCE>
    __device__ __forceinline__ bool next(const float4 *__restrict__ list, const int2 *__restrict__ rng,
                                         const float4 *__restrict__ blo, const float4 *__restrict__ bhi, uint32_t e0,
                                         int ne, int ncell, int tl, int &nchunk, float lox, float hix, float loy,
                                         float hiy, float loz, float hiz, float reach2, float H, float L)
    {
        wb += TW;
        if (wb >= ncell) return false;
        int c = 0, b = 0;
        px = py = pz = 0.f;
        if (wb + tl < ne) {
            const float4 en = list[e0 + (uint32_t)(wb + tl)];
            const int lf = __float_as_int(en.w);
            const int2 r = rng[lf];
            b = r.x;
            c = r.y - r.x;
            px = en.x;
            py = en.y;
            pz = en.z;
            const float4 lo = blo[lf], hi = bhi[lf];
            const float gx = fmaxf(fmaxf(lo.x + px - hix, lox - (hi.x + px)), 0.f);
            const float gy = fmaxf(fmaxf(lo.y + py - hiy, loy - (hi.y + py)), 0.f);
            const float gz = fmaxf(fmaxf(lo.z + pz - hiz, loz - (hi.z + pz)), 0.f);
            float r2 = reach2;
            if (FORCE) {
                const float m = fmaxf(H, lo.w);
                r2 = m * m * (1.f + kPruneMargin) + 2.f * kBandK * m * (m + L);
            }
            if (fmaf(gx, gx, fmaf(gy, gy, gz * gz)) > r2 * 1.00001f) c = 0;
        }
        // the window's non-empty entries moved to the front (list order kept), so that
        // the lookup below meets no empty entry before the last non-empty one
        {
            const int g = TW == 32 ? 0 : (int)(threadIdx.x & 31) / TW;
            const unsigned gm = TW == 32 ? kFull : (((1u << TW) - 1u) << (TW * g));
            const unsigned mine = __ballot_sync(kFull, c > 0) & gm;
            const unsigned src = __fns(mine, (unsigned)(TW * g), tl + 1);
            const bool has = src < 32u;
            const int sl = has ? (int)src : (int)(threadIdx.x & 31);
            c = __shfl_sync(kFull, c, sl);
            b = __shfl_sync(kFull, b, sl);
            px = __shfl_sync(kFull, px, sl);
            py = __shfl_sync(kFull, py, sl);
            pz = __shfl_sync(kFull, pz, sl);
            if (!has) c = 0;
        }
        incl = c;
#pragma unroll
        for (int d = 1; d < TW; d <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, d, TW);
            if (tl >= d) incl += v;
        }
        st = incl - c;
        sb = b - st;
        tot = __shfl_sync(kFull, incl, TW - 1, TW);
        nchunk = (int)__reduce_max_sync(kFull, (unsigned)((tot + TW - 1) / TW));
        return true;
    }

    // slot j, validity and entry offset of the stream position base + tl of chunk
    // base (every lane calls it): the entry holding position base is the number of
    // entries that end at or before it; each entry that starts inside the chunk, at
    // or before the lane's position, adds one
    __device__ __forceinline__ void slot(int base, int tl, int &j, bool &v, float &sx, float &sy, float &sz) const
    {
        const int g = TW == 32 ? 0 : (int)(threadIdx.x & 31) / TW;  // tile of the lane within the warp
        const unsigned gm = TW == 32 ? kFull : (((1u << TW) - 1u) << (TW * g));
        const bool inside = st > base && st < base + TW && st < incl;
        const unsigned starts = __reduce_or_sync(kFull, inside ? 1u << (TW * g + st - base) : 0u) >> (TW * g);
        const int eb = __popc(__ballot_sync(kFull, incl <= base) & gm);
        const int e = min(eb + __popc(starts & ((2u << tl) - 2u)), TW - 1);
        const int q = base + tl;
        j = __shfl_sync(kFull, sb, e, TW) + q;
        sx = __shfl_sync(kFull, px, e, TW);
        sy = __shfl_sync(kFull, py, e, TW);
        sz = __shfl_sync(kFull, pz, e, TW);
        v = q < tot;
    }
};

// reductions over the TW lanes of a tile (xor offsets < TW stay inside the tile)
template <int TW>
__device__ __forceinline__ float tile_min(float v)
{
#pragma unroll
    for (int o = TW / 2; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
template <int TW>
__device__ __forceinline__ float tile_max(float v)
{
#pragma unroll
    for (int o = TW / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum_ull(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// The next iterate of N_w(h) = N_ngb from h, where N_w misses it by g and lo, up bracket the
// root: Newton's step, at most a factor 2 either way; a step that leaves a two-sided bracket is
// replaced by its geometric middle.  Where N_w is so steep that the step rounds to
// nothing (a kernel whose edge is in a halo: two neighbouring floats miss h_tol on either side
// of the root), h goes past the root, so that the bracket closes; it would stay for ever.
__device__ __forceinline__ float next_h(float h, float g, float dnw_dh, float lo, float up)
{
    float hn = dnw_dh > 0.f ? h - g / dnw_dh : (g < 0.f ? 2.f * h : 0.5f * h);
    hn = fminf(fmaxf(hn, 0.5f * h), 2.f * h);
    if (hn == h) hn = g < 0.f ? h * (1.f + kHNudge) : h * (1.f - kHNudge);
    if (lo > 0.f && up < kHUnbounded && !(hn > lo && hn < up)) hn = sqrtf(lo) * sqrtf(up);
    return hn;
}

__device__ __forceinline__ int wrapc(int j, int nc) { return j < 0 ? j + nc : (j >= nc ? j - nc : j); }

// Cubic spline of support 1 without its normalisation sigma, in truncated-power form:
// w/sigma = 2(1-q)^3_+ - 8(1/2-q)^3_+,  (dw/dq)/sigma = -6(1-q)^2_+ + 24(1/2-q)^2_+
// (identical to the piecewise polynomial; branch-free).
__device__ __forceinline__ void spline_u(float q, float &w, float &dw)
{
    const float a = fmaxf(1.f - q, 0.f), b = fmaxf(0.5f - q, 0.f);
    const float a2 = a * a, b2 = b * b;
    w = fmaf(-8.f * b2, b, 2.f * a2 * a);
    dw = fmaf(24.f, b2, -6.f * a2);
}
__device__ __forceinline__ float spline_dw_u(float q)
{
    const float a = fmaxf(1.f - q, 0.f), b = fmaxf(0.5f - q, 0.f);
    return fmaf(24.f * b, b, -6.f * a * a);
}

// Partial force sums of one target: a, du/dt and the largest v_sig.
struct ForceSum {
    float x = 0.f, y = 0.f, z = 0.f, u = 0.f, v = 0.f;
    // store into slot idx (sums into the float4, v_sig beside) and start again
    __device__ __forceinline__ void put(float4 *s4, float *sv, int idx)
    {
        s4[idx] = make_float4(x, y, z, u);
        sv[idx] = v;
        x = y = z = u = v = 0.f;
    }
};

// The pair term of the force pass (Sec. 2: the grad-h pressure force with the
// Monaghan viscosity and its Balsara switch, and du/dt) of target i (1/h_i, 1/h_i^4,
// v_i, thermo_i = {rho, f P / rho^2, c, B}) and source j (h_j, {v_j, m_j}, thermo_j)
// at d = p_i - p_j, r2 = |d|^2 > 0; in_i, in_j: r < h_i, r < h_j.
__device__ __forceinline__ void force_term(float dx, float dy, float dz, float r2, bool in_i, bool in_j, float hinv,
                                           float hinv4, const float4 vi, const float4 ti, float hj, const float4 vj,
                                           const float4 tj, float alpha, ForceSum &f)
{
    const float rinv = rsqrtf(r2);
    const float r = r2 * rinv;
    const float hjinv = __fdividef(1.f, hj);
    const float hj2inv = hjinv * hjinv;
    const float dWi = in_i ? kSigma * spline_dw_u(r * hinv) * hinv4 : 0.f;
    const float dWj = in_j ? kSigma * spline_dw_u(r * hjinv) * (hj2inv * hj2inv) : 0.f;
    const float vx = vi.x - vj.x, vy = vi.y - vj.y, vz = vi.z - vj.z;
    const float mu = fmaf(vx, dx, fmaf(vy, dy, vz * dz)) * rinv;
    // viscosity only on approach (mu < 0): branch-free, Pi = 0 otherwise
    const float muc = fminf(mu, 0.f);
    const float vsig_ij = ti.z + tj.z - 3.f * muc;
    const float Pi = -alpha * vsig_ij * muc * (0.5f * (ti.w + tj.w)) * __fdividef(1.f, ti.x + tj.x);
    const float dWbar = 0.5f * (dWi + dWj);
    const float mj = vj.w;
    const float sc = mj * fmaf(ti.y, dWi, fmaf(tj.y, dWj, Pi * dWbar)) * rinv;
    f.x = fmaf(-sc, dx, f.x);
    f.y = fmaf(-sc, dy, f.y);
    f.z = fmaf(-sc, dz, f.z);
    f.u = fmaf(mj * mu, fmaf(ti.y, dWi, 0.5f * Pi * dWbar), f.u);
    f.v = fmaxf(f.v, vsig_ij);
}

}  // namespace sph
