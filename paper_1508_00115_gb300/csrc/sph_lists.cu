// sph_lists.cu -- the neighbour sums over per-particle neighbour lists.
//
// The search for neighbours and the sums over them are separate kernels:
//   k_search    finds, for every target, the particles within a list radius a little
//               beyond max(h_i, h_j) and writes them as a list of 32-bit names;
//   k_density_l iterates h over the list until it converges (Eq. 1 with the
//               smoothing-length criterion) and writes the density sums;
//   k_force_l   sums Eq. 2 over the same list.
// One search then serves every evaluation of the h iteration and the force pass, as
// long as no h grew beyond its list radius (a search at the new h follows where one
// did); searching in every pass, as the kernels of sph_pairs.cu do, spent half to two
// thirds of each pass on reading and testing sources that are no neighbours.
//
// Lists are chains of chunks of consecutive pages of 32 names.  A name is, on the uniform
// grid, the slot and the stencil cell it was met in, with adaptive cells the entry of the
// target's leaf list and the index in that leaf.  Pages come from one pool, handed out by
// an atomic counter; a list's content and order depend on the cells only, so every sum is the
// same on every run.  When the pool runs out, C_STALE tells the kernels of
// sph_pairs.cu to run instead.
#include <cuda_fp16.h>

#include <algorithm>

#include "sph_pairs.cuh"

namespace sph {

constexpr int kCodes = 1024;      // hits of a batch written out at once
constexpr int kListThreads = 128;
// resident blocks per SM the search is compiled for: more warps where there are tiles of similar
// cost for all of them many times over, else more registers for each, which shortens the tiles
// that the others wait for (search_many has the line)
constexpr int kSearchFew = 5, kSearchMany = 7;
// the sums wait for scattered reads: a lane has both names of a step in flight, and five blocks
// of four warps leave it the registers for that (Sedov 2 M, 19 M in 512 boxes, ms per call: one
// name after the other at 24 warps per SM 14.4, 160; both at 24 warps 14.7, 154; at 20 13.4,
// 152; at 16 13.7, 158)
constexpr int kSumThreads = 128;
constexpr int kSumBlocks = 5;
constexpr int kSearchF4 = 352 + 2 * kCodes / 16;  // float4 of shared memory per searching warp
constexpr int kPage = 32;         // names per page
static_assert(kMaxPages * kPage <= (int64_t)1 << 32, "positions in the pool are 32 bits");
constexpr int kSlotBits = 25;     // uniform grid: bits of a name that hold the slot

// ------------------------------------------- candidate search on the tensor cores
// The distance tests of a tile against its staged sources are a contraction: with the
// positions a_i, b_j relative to the centre of the targets' box, in units that make the box and
// its reach about 1, and rounded to FP16,
//   r_ij^2 - T = -2 a_i . b_j + |b_j|^2 + (|a_i|^2 - T)
// is one m16n8k8 product (FP16 operands, FP32 sums) over
//   row i  {-2ax, -2ay, -2az, th, 1, 1, tl, 0},  th + tl = |a_i|^2 - T_i
//   col j  { bx,   by,   bz,  1, nh, nl, 1, 0},  nh + nl = |b_j|^2
// whose sign bit is the answer: 16 x 8 tests per product, and one funnel shift to keep
// each lane's four, in place of about ten FP32 instructions per test.  A second
// product with T_j in the column's norm instead of T_i in the row's gives r < T_j.  The
// norms are those of the rounded positions, so a product is the squared distance of the
// rounded points up to the rounding of its FP32 sum; rounding moves a point by at most
// 2^-11 of its length, so with T = (h + 2^-11 (|a| + |b|))^2 and a slack for the sum every
// pair within h passes.  What passes is decided again, in FP32 with the FP64 band,
// by the sums over the list: the neighbour sets stay exact.
constexpr float kHalfUlp = 4.95e-4f;   // 2^-11 and a little: relative rounding of a coordinate
constexpr float kHalfAbs = 2e-6f;      // FP16 subnormals, FP32 rounding of the scaled coordinates
constexpr float kSumSlack = 1e-5f;     // rounding of the product's FP32 sum (terms up to ~4)
constexpr float kFarSource = 64.f;     // sources beyond this many units are not tested: always hits
constexpr float kAlways = -30000.f;    // in place of a norm: a hit for every target
constexpr unsigned kNeverCol = 0x00007b53u;  // {60000, 0}, in place of a norm: never a hit
constexpr unsigned kHalfOne0 = 0x00003c00u;  // {1, 0}
constexpr unsigned kHalfOne1 = 0x3c003c00u;  // {1, 1}

__device__ __forceinline__ unsigned pack_half2(float lo, float hi)
{
    const __half2 v = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&v);
}
// v as the sum of two halves {high, low}
__device__ __forceinline__ unsigned split_half(float v)
{
    const float h = __half2float(__float2half_rn(v));
    return pack_half2(h, v - h);
}

__device__ __forceinline__ float fast_sqrt(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// frame of the tests: the centre of the targets' box and 1 / (its half diagonal + reach)
struct TestFrame {
    float cx, cy, cz, s;
    __device__ __forceinline__ TestFrame(float x, float y, float z, float scale) : cx(x), cy(y), cz(z), s(scale) {}
    // the point in the frame, rounded to FP16: its rounded coordinates and norm
    __device__ __forceinline__ float round(float x, float y, float z, float &rx, float &ry, float &rz) const
    {
        const float2 q = __half22float2(__floats2half2_rn((x - cx) * s, (y - cy) * s));
        rx = q.x;
        ry = q.y;
        rz = __half2float(__float2half_rn((z - cz) * s));
        return fmaf(rx, rx, fmaf(ry, ry, rz * rz));
    }
    // row of a target: words {-2ax, -2ay}, {-2az, th}, and (the {1, 1} in between left
    // out) {-2az, uh}, {tl, ul}, where u is the norm without the threshold; h2: the squared
    // distance below which a pair has to pass (!act: none does)
    __device__ __forceinline__ uint4 row(bool act, const float4 p, float h2) const
    {
        if (!act) return make_uint4(0u, kNeverCol << 16, kNeverCol << 16, 0u);
        float rx, ry, rz;
        const float n2 = round(p.x, p.y, p.z, rx, ry, rz);
        const float hs = fast_sqrt(h2) * s;
        const float d = hs + kHalfUlp * fmaf(2.f, fast_sqrt(n2), hs) + kHalfAbs;
        const unsigned t = split_half(n2 - fmaf(d * d, 1.f + 1e-5f, kSumSlack)), u = split_half(n2);
        const unsigned z = pack_half2(-2.f * rz, 0.f);
        return make_uint4(pack_half2(-2.f * rx, -2.f * ry), z | (t << 16), z | (u << 16),
                          (t >> 16) | (u & 0xffff0000u));
    }
    // column of a source with reach sqrt(h2) of its own: words {bx, by}, {bz, 1}, {nh, nl}
    // and, for the second product, {mh, ml}, the norm less its threshold
    __device__ __forceinline__ uint4 col(const float4 p, float h2) const
    {
        const float gx = (p.x - cx) * s, gy = (p.y - cy) * s, gz = (p.z - cz) * s;
        if (fmaxf(fabsf(gx), fmaxf(fabsf(gy), fabsf(gz))) > kFarSource)
            return make_uint4(0u, pack_half2(0.f, 1.f), kNeverCol, pack_half2(kAlways, 0.f));
        float rx, ry, rz;
        const float n2 = round(p.x, p.y, p.z, rx, ry, rz);
        const float hs = fast_sqrt(h2) * s;
        const float d = hs + kHalfUlp * (1.002f + 1.001f * fast_sqrt(n2)) + kHalfAbs;
        const float m2 = fmaxf(n2 - fmaf(d * d, 1.f + 1e-5f, kSumSlack), kAlways);
        return make_uint4(pack_half2(rx, ry), pack_half2(rz, 1.f), split_half(n2), split_half(m2));
    }
    static __device__ __forceinline__ uint4 never() { return make_uint4(0u, pack_half2(0.f, 1.f), kNeverCol, kNeverCol); }
};

__device__ __forceinline__ void mma_m16n8k8(float (&d)[4], unsigned a0, unsigned a1, unsigned b)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%7, %7, %7, %7};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(b), "f"(0.f));
}
// append the sign of v or w to a mask
__device__ __forceinline__ void push_sign(unsigned &m, float v, float w)
{
    m = __funnelshift_l(__float_as_uint(v) | __float_as_uint(w), m, 1);
}

// Rows of a warp as product operands: lane (g, q) = (lane / 4, lane % 4) holds word q of rows
// g + 8 t, for the two products.  rows: 32 uint4 in shared memory.
struct RowWords {
    unsigned A[4], A2[4];
    __device__ __forceinline__ void load(const uint4 *rows, int lane)
    {
        const unsigned *r = reinterpret_cast<const unsigned *>(rows);
        const int q = lane & 3;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const unsigned v = r[32 * t + lane];
            A[t] = q == 2 ? kHalfOne1 : (q == 3 ? v & 0xffffu : v);
            A2[t] = q == 1 ? r[32 * t + lane + 1] : (q == 3 ? v >> 16 : A[t]);
        }
    }
};

// Where the k-th of 128 sources stands among the columns: lane q's columns (2 q and 2 q + 1 of
// each product) are sources 32 q .. 32 q + 31, so that the hits of a row come in source order.
__device__ __forceinline__ int column(int k) { return ((k & 31) >> 1) * 8 + 2 * (k >> 5) + (k & 1); }

// Tests of the warp's 32 rows against 128 columns: lane (g, q) gets in M[t] the hits of row
// g + 8 t, bit b the source 32 q + b.
__device__ __forceinline__ void test_batch(const uint4 *op, const RowWords &r, int lane, unsigned (&M)[4])
{
    const unsigned *w = reinterpret_cast<const unsigned *>(op);
    const int q = lane & 3;
    const int lane2 = q == 2 ? lane + 1 : lane;  // the second product takes word 3 in place of word 2
#pragma unroll
    for (int t = 0; t < 4; ++t) M[t] = 0u;
#pragma unroll 4
    for (int blk = 15; blk >= 0; --blk) {
        unsigned b = w[32 * blk + lane], c = w[32 * blk + lane2];
        if (q == 3) b = c = kHalfOne0;
        float d[4], d2[4], e[4], e2[4];
        mma_m16n8k8(d, r.A[0], r.A[1], b);
        mma_m16n8k8(d2, r.A2[0], r.A2[1], c);
        mma_m16n8k8(e, r.A[2], r.A[3], b);
        mma_m16n8k8(e2, r.A2[2], r.A2[3], c);
        push_sign(M[0], d[1], d2[1]);
        push_sign(M[1], d[3], d2[3]);
        push_sign(M[2], e[1], e2[1]);
        push_sign(M[3], e[3], e2[3]);
        push_sign(M[0], d[0], d2[0]);
        push_sign(M[1], d[2], d2[2]);
        push_sign(M[2], e[0], e2[0]);
        push_sign(M[3], e[2], e2[2]);
    }
}

// ------------------------------------------------------------------ the search

// A warp takes a tile (up to 32 targets of one cell or leaf).  The segments around it -- the
// cells of the stencil, or the entries of the leaf's list -- within reach of the targets'
// box form one stream, read 32 sources at a time whatever the segments' lengths; the
// sources within reach of the box are packed into batches of 128, each converted to
// columns and tested at once.  (Measured against this, 19 M particles in 512 clustered boxes
// and 2 M on a lattice: staging once per leaf or per 2 x 2 x 2 cells for all the tiles
// of it, 55 against 23 ms and 1.36 against 0.93 ms: the tiles of a leaf hold targets of
// similar h, and each needs a small part of what the leaf does.)

struct SearchArgs {
    const float4 *__restrict__ pos4;  // .w: the h the sources' reach comes from
    const float *__restrict__ h;      // the targets' current h
    const uint8_t *__restrict__ active;  // targets to search for (null: all)
    const BoxDev *__restrict__ boxes;
    // uniform grid
    const int *__restrict__ cell_start;
    const float *__restrict__ cell_reach;
    int nb;
    const int4 *__restrict__ tiles;
    const int *__restrict__ n_tiles;
    // adaptive cells
    const uint32_t *__restrict__ list_off;
    const float4 *__restrict__ list;
    const int2 *__restrict__ leaf_rng;
    const float *__restrict__ leaf_scale;
    const float4 *__restrict__ leaf_lo, *__restrict__ leaf_hi;
    const float *__restrict__ leaf_hb;
    const int *__restrict__ tord;
    uint32_t *pages;
    int *next;       // chunks: pages, next chunk
    int *head;       // per slot: first page
    int *cnt;        // names
    float *radius;   // list radius of the target
    unsigned long long *counters;
    const unsigned long long *run_if;  // run only if it is above run_above (null: always) ...
    unsigned run_above;
    const unsigned long long *or_if;   // ... or if this is not zero
    unsigned long long *ticket;
    unsigned cap_pages;
    double box;
    float grow;
    int wbits;       // adaptive cells: bits of a name that hold the index in the leaf
    int force;       // the force pass's own search
};

// Where the hits of a warp's rows go: their pages so far, and the codes of one batch.
struct RowPages {
    int fill = 0;                // names of this lane's row so far
    int first = 0, chunk = 0;    // first page of its first and of its last chunk
    int start = 0, end = 0;      // names before the last chunk, and that it ends at
    bool dead = false;           // no page left (warp-uniform)
};

// Pages of the chunk that follows `fill` names (two at least: the first page's word in
// `next` holds the chunk's length, the second's the next chunk).  Lists of thousands of
// names come in long chunks, so that their readers seldom wait for the chain.
__device__ __forceinline__ int chunk_pages(int fill, int need)
{
    const int p = fill < 256 ? 2 : fill < 1024 ? 8 : fill < 4096 ? 32 : 128;
    return max(p, ((need + kPage - 1) / kPage + 1) & ~1);
}

// The hits of a batch (test_batch) to the rows' pages.
__device__ __forceinline__ void emit_batch(const SearchArgs &a, const unsigned (&M)[4], const unsigned *names,
                                           uint16_t *codes, int *off, uint4 *dst, RowPages &R)
{
    const int lane = threadIdx.x & 31;
    const int c01 = __popc(M[0]) | (__popc(M[1]) << 16), c23 = __popc(M[2]) | (__popc(M[3]) << 16);
    int e01 = c01, e23 = c23;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(kFull, e01, d), v = __shfl_up_sync(kFull, e23, d);
        if (lane >= d) {
            e01 += u;
            e23 += v;
        }
    }
    const int T01 = __shfl_sync(kFull, e01, 31), T23 = __shfl_sync(kFull, e23, 31);
    e01 -= c01;
    e23 -= c23;
    const int s1 = T01 & 0xffff, s2 = s1 + (T01 >> 16), s3 = s2 + (T23 & 0xffff), H = s3 + (T23 >> 16);
    if (H == 0 || R.dead) return;
    // flat position of every hit: rows in order, within a row lane by lane
    const int o[4] = {e01 & 0xffff, s1 + (e01 >> 16), s2 + (e23 & 0xffff), s3 + (e23 >> 16)};
    __syncwarp();
    if ((lane & 3) == 0) {
#pragma unroll
        for (int t = 0; t < 4; ++t) off[8 * t + (lane >> 2)] = o[t];
    }
    if (lane == 0) off[32] = H;
    // all rows at once, or (a dense batch) eight at a time: at most 8 x 128 hits
    const bool whole = H <= kCodes;
    for (int part = 0; part < (whole ? 1 : 4); ++part) {
        const int t0 = whole ? 0 : part, t1 = whole ? 4 : part + 1;
        const int p0 = whole ? 0 : (part == 0 ? 0 : part == 1 ? s1 : part == 2 ? s2 : s3);
        const int p1 = whole ? H : (part == 0 ? s1 : part == 1 ? s2 : part == 2 ? s3 : H);
        __syncwarp();
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (t < t0 || t >= t1) continue;
            unsigned m = M[t];
            int p = o[t] - p0;
            const unsigned code = (unsigned)((8 * t + (lane >> 2)) << 7) | (unsigned)((lane & 3) << 5);
            while (m) {
                codes[p++] = (uint16_t)(code + (unsigned)__ffs(m) - 1u);
                m &= m - 1u;
            }
        }
        // pages for the rows' new names
        const bool mine = (lane >> 3) >= t0 && (lane >> 3) < t1;
        const int nh = mine ? off[lane + 1] - off[lane] : 0;
        const int room = R.end - R.fill;  // names the last chunk still takes
        const int np = nh > room ? chunk_pages(R.fill, nh - room) : 0;
        int incl = np;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += v;
        }
        const int total = __shfl_sync(kFull, incl, 31);
        unsigned base = 0u;
        if (total > 0) {
            if (lane == 0) base = atomicAdd(reinterpret_cast<unsigned *>(a.counters + C_PAGES), (unsigned)total);
            base = __shfl_sync(kFull, base, 0);
            if (base > a.cap_pages || (unsigned)total > a.cap_pages - base) R.dead = true;
        }
        if (R.dead) return;  // warp-uniform
        const int fresh = (int)base + incl - np;
        // (positions are 32 bits without a sign: modulo 2^32, as the pool has 2^32 names at most)
        dst[lane] = make_uint4((unsigned)R.chunk * kPage + (unsigned)(R.fill - R.start - off[lane]),
                               (unsigned)fresh * kPage - (unsigned)(room + off[lane]), (unsigned)(off[lane] + room), 0u);
        if (np > 0) {
            if (R.fill == 0) R.first = fresh;
            else a.next[R.chunk + 1] = fresh;
            a.next[fresh] = np;
            R.chunk = fresh;
            R.start = R.end;
            R.end += kPage * np;
        }
        R.fill += nh;
        __syncwarp();
        for (int p = p0 + lane; p < p1; p += 32) {
            const unsigned c = codes[p - p0];
            const uint4 d = dst[c >> 7];
            a.pages[(size_t)((unsigned)p < d.z ? d.x + (unsigned)p : d.y + (unsigned)p)] = names[c & 127u];
        }
    }
    __syncwarp();
}

// MODE: 0 = uniform grid, 1 = adaptive cells
template <int MODE, int BLOCKS>
__global__ void __launch_bounds__(kListThreads, BLOCKS) k_search(SearchArgs a)
{
    if (a.run_if && *a.run_if <= a.run_above && !(a.or_if && (*a.or_if & 3ull))) return;
    constexpr bool LIST = MODE == 1;
    constexpr int W = kListThreads / 32;
    extern __shared__ uint4 search_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint4 *const s_op = search_smem + kSearchF4 * wib;                    // columns
    float4 *const s_pos = reinterpret_cast<float4 *>(s_op + 128);         // sources: position, reach
    uint4 *const s_row = s_op + 256;                                      // rows
    uint4 *const s_dst = s_op + 288;                                      // where the rows' hits go
    unsigned *const s_name = reinterpret_cast<unsigned *>(s_op + 320);    // the sources' names
    uint16_t *const s_code = reinterpret_cast<uint16_t *>(s_op + 352);    // hits of a batch
    int *const s_off = reinterpret_cast<int *>(search_smem + kSearchF4 * W) + 33 * wib;
    const unsigned lt = (1u << lane) - 1u;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const int ntiles = *a.n_tiles;
    const float inf = __int_as_float(0x7f800000);
    unsigned long long acc_cand = 0ull;
    unsigned acc_stream = 0u, acc_staged = 0u;
    bool overflow = false, wide = false;  // warp-uniform
    unsigned *ticket = reinterpret_cast<unsigned *>(a.ticket);
    unsigned tk = 0u;
    if (lane == 0) tk = atomicAdd(ticket, 1u);
    for (int t = gw, t_after = 0; t < ntiles; t = t_after) {
        t_after = nw + (int)__shfl_sync(kFull, tk, 0);
        if (lane == 0 && t_after < ntiles) tk = atomicAdd(ticket, 1u);
        const int4 tile = a.tiles[t];
        const bool valid = lane < tile.z;
        const int i = LIST ? (valid ? a.tord[tile.y + lane] : 0) : tile.y + lane;
        const bool act = valid && (a.active == nullptr || a.active[i]);
        const unsigned amask = __ballot_sync(kFull, act);
        if (!amask) continue;
        float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
        if (act) pi = a.pos4[i];
        const float lox = tile_min<32>(act ? pi.x : inf), hix = tile_max<32>(act ? pi.x : -inf);
        const float loy = tile_min<32>(act ? pi.y : inf), hiy = tile_max<32>(act ? pi.y : -inf);
        const float loz = tile_min<32>(act ? pi.z : inf), hiz = tile_max<32>(act ? pi.z : -inf);
        const BoxDev bx = a.boxes[tile.w];
        const int nc = bx.nc;
        const float L = LIST ? a.leaf_scale[tile.x] : bx.L32;
        // list radius: beyond h by the growth factor, as far as the cells reach
        float ri = 0.f;
        if (act) {
            const float cap = LIST ? fminf(fminf(kTreeReach * a.leaf_hb[tile.x], bx.L32), (float)(0.5 * a.box))
                                   : 2.f * bx.L32 * (1.f - 1e-6f);
            const float hi = a.h[i];
            ri = fmaxf(hi, fminf(hi * a.grow, cap));
        }
        const float H = tile_max<32>(ri);
        const float reach2 = H * H * (1.f + kPruneMargin) + 2.f * kBandK * H * (H + L);
        // uniform grid: largest reach of any source around the cell, and the stencil that holds it
        const float Hs = LIST ? H : fmaxf(H, a.cell_reach[tile.x] * a.grow);
        const int R = !LIST && Hs * (1.f + kPruneMargin) > L ? 2 : 1;
        const int side = 2 * R + 1;
        // frame of the products
        const float ex = 0.5f * (hix - lox), ey = 0.5f * (hiy - loy), ez = 0.5f * (hiz - loz);
        const TestFrame fr(0.5f * (lox + hix), 0.5f * (loy + hiy), 0.5f * (loz + hiz),
                           __fdividef(1.f, sqrtf(fmaf(ex, ex, fmaf(ey, ey, ez * ez))) + H));
        s_row[lane] = fr.row(act, pi, fmaf(ri, ri, kBandK * ri * (ri + L)));  // (a __syncwarp follows in flush)
        const int ca = tile.x - bx.cell_off;
        const int ix = ca % nc, iy = (ca / nc) % nc, iz = ca / (nc * nc);
        uint32_t e0 = 0;
        int nseg = side * side * side;
        if (LIST) {
            e0 = a.list_off[tile.x];
            nseg = (int)(a.list_off[tile.x + 1] - e0);
            wide |= (unsigned)nseg >= (1u << (32 - a.wbits));
        }
        RowPages out;
        out.dead = overflow;
        int nst = 0, staged = 0;

        auto flush = [&]() {
            __syncwarp();
            for (int k = lane; k < 128; k += 32) {
                uint4 c = TestFrame::never();
                if (k < nst) {
                    const float4 p = s_pos[k];
                    c = fr.col(p, fmaf(p.w, p.w, kBandK * p.w * (p.w + L)));
                }
                s_op[column(k)] = c;
            }
            __syncwarp();
            RowWords rows;
            rows.load(s_row, lane);
            unsigned M[4];
            test_batch(s_op, rows, lane, M);
            emit_batch(a, M, s_name, s_code, s_off, s_dst, out);
            staged += nst;
            nst = 0;
            __syncwarp();
        };

        for (int w0 = 0; w0 < nseg && !out.dead; w0 += 32) {
            // a window of segments, one per lane: its length (0 beyond reach), first slot and
            // offset, and the name of its first source
            const int k = w0 + lane;
            int c = 0, b = 0;
            unsigned nm = 0u;
            float sx = 0.f, sy = 0.f, sz = 0.f;
            if (k < nseg) {
                float lx, ly, lz, ux, uy, uz, m = Hs;
                if (LIST) {
                    const float4 en = a.list[e0 + (uint32_t)k];
                    const int lf = __float_as_int(en.w);
                    const int2 r = a.leaf_rng[lf];
                    const float4 lo = a.leaf_lo[lf], hi = a.leaf_hi[lf];
                    b = r.x;
                    c = r.y - r.x;
                    wide |= c > (1 << a.wbits);
                    sx = en.x;
                    sy = en.y;
                    sz = en.z;
                    lx = lo.x;
                    ly = lo.y;
                    lz = lo.z;
                    ux = hi.x;
                    uy = hi.y;
                    uz = hi.z;
                    m = fmaxf(H, lo.w * a.grow);
                    nm = (unsigned)k << a.wbits;
                } else {
                    const int dx = k % side - R, dy = (k / side) % side - R, dz = k / (side * side) - R;
                    const int cb = bx.cell_off + (wrapc(iz + dz, nc) * nc + wrapc(iy + dy, nc)) * nc + wrapc(ix + dx, nc);
                    b = a.cell_start[cb];
                    c = a.cell_start[cb + 1] - b;
                    sx = (float)dx * L;
                    sy = (float)dy * L;
                    sz = (float)dz * L;
                    // (positions are within half a side of the centre up to their rounding)
                    lx = ly = lz = -0.5f * L * (1.f + 1e-5f);
                    ux = uy = uz = 0.5f * L * (1.f + 1e-5f);
                    nm = ((unsigned)(62 + dx + 5 * dy + 25 * dz) << kSlotBits) + (unsigned)b;
                }
                const float gx = fmaxf(fmaxf(lx + sx - hix, lox - (ux + sx)), 0.f);
                const float gy = fmaxf(fmaxf(ly + sy - hiy, loy - (uy + sy)), 0.f);
                const float gz = fmaxf(fmaxf(lz + sz - hiz, loz - (uz + sz)), 0.f);
                if (fmaf(gx, gx, fmaf(gy, gy, gz * gz)) >
                    (m * m * (1.f + kPruneMargin) + 2.f * kBandK * m * (m + L)) * 1.00001f)
                    c = 0;
            }
            // the non-empty segments to the front (in order), and their ends in the stream
            {
                const unsigned mine = __ballot_sync(kFull, c > 0);
                if (mine == 0u) continue;
                const unsigned src = __fns(mine, 0u, lane + 1);
                const bool has = src < 32u;
                const int sl = has ? (int)src : lane;
                c = __shfl_sync(kFull, c, sl);
                b = __shfl_sync(kFull, b, sl);
                nm = __shfl_sync(kFull, nm, sl);
                sx = __shfl_sync(kFull, sx, sl);
                sy = __shfl_sync(kFull, sy, sl);
                sz = __shfl_sync(kFull, sz, sl);
                if (!has) c = 0;
            }
            int incl = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += v;
            }
            const int st = incl - c, total = __shfl_sync(kFull, incl, 31);
            b -= st;             // slot and name less the stream position
            nm -= (unsigned)st;
            // slot, name and offset of stream position base + lane: the segment that holds
            // position base is the number of those that end at or before it; each that
            // starts inside the chunk at or before the lane's position adds one
            auto at = [&](int base, int &j, unsigned &name, float &ox, float &oy, float &oz) -> bool {
                const bool inside = st > base && st < base + 32 && st < incl;
                const unsigned starts = __reduce_or_sync(kFull, inside ? 1u << (st - base) : 0u);
                const int eb = __popc(__ballot_sync(kFull, incl <= base));
                const int e = min(eb + __popc(starts & ((2u << lane) - 2u)), 31);
                const int q = base + lane;
                j = __shfl_sync(kFull, b, e) + q;
                name = __shfl_sync(kFull, nm, e) + (unsigned)q;
                ox = __shfl_sync(kFull, sx, e);
                oy = __shfl_sync(kFull, sy, e);
                oz = __shfl_sync(kFull, sz, e);
                return q < total;
            };
            // software pipeline: the next chunk's positions are loaded before this one's tests
            int j;
            unsigned name;
            float ox, oy, oz;
            bool v = at(0, j, name, ox, oy, oz);
            float4 p = v ? __ldg(a.pos4 + j) : make_float4(kFar, kFar, kFar, 0.f);
            for (int base = 0; base < total && !out.dead; base += 32) {
                int jn = 0;
                unsigned name_n = 0u;
                float nx = 0.f, ny = 0.f, nz = 0.f;
                bool vn = false;
                if (base + 32 < total) vn = at(base + 32, jn, name_n, nx, ny, nz);
                const float4 pn = vn ? __ldg(a.pos4 + jn) : make_float4(kFar, kFar, kFar, 0.f);
                acc_stream += v ? 1u : 0u;
                p.x += ox;
                p.y += oy;
                p.z += oz;
                // reach of the source (uniform grid: two cell sides at most)
                p.w = LIST ? p.w * a.grow : fminf(p.w * a.grow, 2.f * L * (1.f - 1e-6f));
                const float fx = fmaxf(fmaxf(lox - p.x, p.x - hix), 0.f);
                const float fy = fmaxf(fmaxf(loy - p.y, p.y - hiy), 0.f);
                const float fz = fmaxf(fmaxf(loz - p.z, p.z - hiz), 0.f);
                float r2max = reach2;
                if (p.w > H) r2max = p.w * p.w * (1.f + kPruneMargin) + 2.f * kBandK * p.w * (p.w + L);
                const bool keep = fmaf(fx, fx, fmaf(fy, fy, fz * fz)) < r2max;
                const unsigned mine = __ballot_sync(kFull, keep);
                if (keep) {
                    const int at_ = nst + __popc(mine & lt);
                    s_pos[at_] = p;
                    s_name[at_] = name;
                }
                nst += __popc(mine);
                if (nst > 96) flush();
                v = vn;
                p = pn;
                name = name_n;
                ox = nx;
                oy = ny;
                oz = nz;
            }
        }
        if (nst > 0 && !out.dead) flush();
        __syncwarp();
        if (LIST && __any_sync(kFull, wide)) wide = out.dead = true;
        overflow |= out.dead;
        if (lane == 0) {
            acc_cand += (unsigned long long)staged * (unsigned)__popc(amask);
            acc_staged += (unsigned)staged;
        }
        if (act) {
            a.head[i] = out.first;
            a.cnt[i] = out.fill;
            a.radius[i] = ri;
        }
    }
    const unsigned long long tc = warp_sum_ull(acc_cand), ts = warp_sum_ull(acc_stream), tg = warp_sum_ull(acc_staged);
    if (lane == 0) {
        if (tc) atomicAdd(a.counters + (a.force ? C_FCAND : C_DCAND), tc);
        if (LIST && ts) atomicAdd(a.counters + (a.force ? C_FSTREAM : C_DSTREAM), ts);
        if (tg) atomicAdd(a.counters + (a.force ? C_FSTAGED : C_DSTAGED), tg);
        if (overflow) atomicOr(a.counters + (a.force ? C_FOVF : C_STALE), wide ? 5ull : 1ull);
    }
}

// The search for single targets (rows[0 .. *n_rows)), a warp each: the few whose h left
// their list radius, or whose neighbours' did.  The block search would stage the sources of
// every leaf that holds one of them, which with one target in a hundred is every leaf.
struct SearchOneArgs {
    SearchArgs s;
    const int *__restrict__ rows;
    const unsigned long long *__restrict__ n_rows;
    const uint32_t *__restrict__ keys;    // uniform grid: sorted keys (cell << 3 | octant)
    const int *__restrict__ leaf_of;      // adaptive cells
    unsigned run_upto;                    // run only up to so many rows
    const unsigned long long *unless;     // ... and only if this is zero
};

template <int MODE>
__global__ void __launch_bounds__(256) k_search_one(SearchOneArgs b)
{
    const SearchArgs &a = b.s;
    const unsigned long long nr = *b.n_rows;
    if (nr == 0ull || nr > b.run_upto || (*b.unless & 3ull)) return;
    constexpr bool LIST = MODE == 1;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    bool overflow = false;
    for (int u = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); u < (int)nr;
         u += (int)((gridDim.x * blockDim.x) >> 5)) {
        const int i = b.rows[u];
        const float4 pi = a.pos4[i];
        const float hi = a.h[i];
        int lf = 0, bi = 0;
        if (a.nb > 1) {
            int l2 = 0, h2 = a.nb - 1;
            while (l2 < h2) {
                const int mid = (l2 + h2 + 1) >> 1;
                if (a.boxes[mid].p_begin <= i) l2 = mid;
                else h2 = mid - 1;
            }
            bi = l2;
        }
        const BoxDev bx = a.boxes[bi];
        const int nc = bx.nc;
        float L = bx.L32, reach;
        int nseg, R = 1, ix = 0, iy = 0, iz = 0;
        uint32_t e0 = 0;
        float ri;
        if (LIST) {
            lf = b.leaf_of[i];
            L = a.leaf_scale[lf];
            e0 = a.list_off[lf];
            nseg = (int)(a.list_off[lf + 1] - e0);
            ri = fmaxf(hi, fminf(hi * a.grow, fminf(fminf(kTreeReach * a.leaf_hb[lf], bx.L32), (float)(0.5 * a.box))));
            reach = ri;
        } else {
            const int c = (int)(b.keys[i] >> 3), ca = c - bx.cell_off;
            ix = ca % nc;
            iy = (ca / nc) % nc;
            iz = ca / (nc * nc);
            ri = fmaxf(hi, fminf(hi * a.grow, 2.f * L * (1.f - 1e-6f)));
            reach = fmaxf(ri, a.cell_reach[c] * a.grow);
            R = reach * (1.f + kPruneMargin) > L ? 2 : 1;
            nseg = R == 2 ? 125 : 27;
        }
        int fill = 0, first = 0, chunk = 0, start = 0, end = 0;  // as RowPages
        bool dead = overflow;
        const int side = 2 * R + 1;
        for (int w0 = 0; w0 < nseg && !dead; w0 += 32) {
            // segments (leaf entries or cells) within reach of the target
            const int k = w0 + lane;
            float sx = 0.f, sy = 0.f, sz = 0.f;
            int st = 0, c = 0;
            unsigned nm = 0u;
            if (k < nseg) {
                if (LIST) {
                    const float4 en = a.list[e0 + (uint32_t)k];
                    const int l2 = __float_as_int(en.w);
                    const int2 r = a.leaf_rng[l2];
                    const float4 lo = a.leaf_lo[l2], hb = a.leaf_hi[l2];
                    sx = en.x;
                    sy = en.y;
                    sz = en.z;
                    const float ex = fmaxf(fmaxf(lo.x + sx - pi.x, pi.x - (hb.x + sx)), 0.f);
                    const float ey = fmaxf(fmaxf(lo.y + sy - pi.y, pi.y - (hb.y + sy)), 0.f);
                    const float ez = fmaxf(fmaxf(lo.z + sz - pi.z, pi.z - (hb.z + sz)), 0.f);
                    const float m = fmaxf(ri, lo.w * a.grow);
                    st = r.x;
                    if (fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <=
                        (m * m * (1.f + kPruneMargin) + 2.f * kBandK * m * (m + L)) * 1.00001f)
                        c = r.y - r.x;
                    nm = (unsigned)k << a.wbits;
                } else {
                    const int dx = k % side - R, dy = (k / side) % side - R, dz = k / (side * side) - R;
                    const int cb = bx.cell_off + (wrapc(iz + dz, nc) * nc + wrapc(iy + dy, nc)) * nc + wrapc(ix + dx, nc);
                    st = a.cell_start[cb];
                    c = a.cell_start[cb + 1] - st;
                    sx = (float)dx * L;
                    sy = (float)dy * L;
                    sz = (float)dz * L;
                    nm = ((unsigned)(62 + dx + 5 * dy + 25 * dz) << kSlotBits) + (unsigned)st;
                }
            }
            unsigned todo = __ballot_sync(kFull, c > 0);
            while (todo && !dead) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1u;
                const int s0 = __shfl_sync(kFull, st, src), n0 = __shfl_sync(kFull, c, src);
                const float ox = __shfl_sync(kFull, sx, src), oy = __shfl_sync(kFull, sy, src),
                            oz = __shfl_sync(kFull, sz, src);
                const unsigned name0 = __shfl_sync(kFull, nm, src);
                for (int q0 = 0; q0 < n0; q0 += 32) {
                    const int q = q0 + lane;
                    bool in = false;
                    if (q < n0) {
                        const float4 pj = __ldg(a.pos4 + s0 + q);
                        const float dx = pi.x - (pj.x + ox), dy = pi.y - (pj.y + oy), dz = pi.z - (pj.z + oz);
                        const float m = fmaxf(ri, LIST ? pj.w * a.grow : fminf(pj.w * a.grow, 2.f * L * (1.f - 1e-6f)));
                        in = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < fmaf(m, m, kBandK * m * (m + L));
                    }
                    const unsigned hit = __ballot_sync(kFull, in);
                    const int nh = __popc(hit);
                    if (nh == 0) continue;
                    // the names take the rest of the last chunk, then a fresh one
                    const int room = end - fill;
                    int fresh = 0, np = 0;
                    if (nh > room) {
                        np = chunk_pages(fill, nh - room);
                        unsigned base = 0u;
                        if (lane == 0)
                            base = atomicAdd(reinterpret_cast<unsigned *>(a.counters + C_PAGES), (unsigned)np);
                        base = __shfl_sync(kFull, base, 0);
                        if (base > a.cap_pages || (unsigned)np > a.cap_pages - base) {
                            dead = true;
                            break;
                        }
                        fresh = (int)base;
                        if (fill == 0) first = fresh;
                        else if (lane == 0) a.next[chunk + 1] = fresh;
                        if (lane == 0) a.next[fresh] = np;
                    }
                    if (in) {
                        const int x = __popc(hit & lt);
                        const size_t at = x < room ? (size_t)chunk * kPage + (size_t)(fill - start + x)
                                                   : (size_t)fresh * kPage + (size_t)(x - room);
                        a.pages[at] = name0 + (unsigned)q;
                    }
                    if (np > 0) {
                        chunk = fresh;
                        start = end;
                        end += kPage * np;
                    }
                    fill += nh;
                }
            }
        }
        overflow |= dead;
        if (lane == 0) {
            a.head[i] = first;
            a.cnt[i] = fill;
            a.radius[i] = ri;
        }
    }
    if (lane == 0 && overflow) atomicOr(a.counters + (a.force ? C_FOVF : C_STALE), 1ull);
}

// ------------------------------------------------------- sums over the lists
// A warp takes a tile, or (small sets) an equal part of one.  Lists are 50 to 70 names on
// uniform matter, and eight lanes share a target there: the lanes take a list's names in
// turn (one 32-byte sector per round), sum their terms and add them with shuffles, and
// four targets run side by side.  A lane per target would leave the lanes of a warp
// waiting for its longest list, a warp per target two thirds of the last round idle
// and its reductions unshared.  Lists beyond kLongList names (clustered matter: the
// sparse particles whose kernel takes in the edge of a halo have thousands) get the whole
// warp.  The rows of a tile go in order of their lists' lengths, so that the four
// that run side by side end together.

constexpr int kLongList = 128;

struct SumArgs {
    const float4 *__restrict__ pos4;
    const float4 *__restrict__ vel4;
    const float4 *__restrict__ thermo4;
    const int4 *__restrict__ tiles;
    const int *__restrict__ n_tiles;
    const int *__restrict__ tord;
    const BoxDev *__restrict__ boxes;
    const uint32_t *__restrict__ list_off;
    const float4 *__restrict__ list;
    const int *__restrict__ list_slot;
    const float *__restrict__ leaf_scale;
    const float *__restrict__ leaf_hb;
    const uint32_t *__restrict__ pages;
    const int *__restrict__ next;
    const int *__restrict__ head;
    const int *__restrict__ cnt;
    const float *__restrict__ radius;
    const double *__restrict__ x;
    const double *__restrict__ y;
    const double *__restrict__ z;
    unsigned long long *counters;
    double box;
    const unsigned long long *run_if;  // run only if it is not zero (null: always)
    unsigned long long *ticket;
    int wbits;
    int split;  // parts a tile is cut into (1, 2, 4 or 8): a part has 32 / split rows at most
    int first8; // (split 1) one tile in first8, from the first, is cut into eight (0: none)
};

// Part u of the tiles: the tile, and the rows [row0, row0 + per) of it.  The first tiles are the
// costliest (order_tiles): cut, so that a few of them do not outlast the rest of the pass.
__device__ __forceinline__ int tile_parts(const SumArgs &a, int ntiles)
{
    return ntiles * a.split + (a.first8 ? 7 * (ntiles / a.first8) : 0);
}
__device__ __forceinline__ int tile_part(const SumArgs &a, int ntiles, int u, int &row0, int &per)
{
    const int cut = a.first8 ? ntiles / a.first8 : 0;
    if (u < 8 * cut) {
        per = 4;
        row0 = 4 * (u & 7);
        return u >> 3;
    }
    u -= 7 * cut;
    per = 32 / a.split;
    row0 = (u % a.split) * per;
    return u / a.split;
}

struct DensityListArgs {
    SumArgs s;
    const int64_t *__restrict__ ids;
    const float *__restrict__ upred;
    uint8_t *active;
    float *h, *h_lo, *h_hi;
    float *rho, *P, *c, *f, *divv, *curl;
    int32_t *n_ngb;
    float4 *thermo4;
    uint64_t *ngb_hash;
    float n_ngb_target, h_tol, gamma, grow;
    int use_balsara;
    const int *__restrict__ rows;  // targets (null: those of the tiles that are active)
    const unsigned long long *__restrict__ n_rows;
    const int *__restrict__ leaf_of;
    int nb;
    // targets that need another pass ([3], in two halves: most evaluations of one of them, of any)
    unsigned long long *left;
    int *left_rows;            // ... and which
    int *grown_rows;           // targets whose h outgrew the radius their neighbours searched with
    int budget;      // evaluations of a target in this pass
    int last_pass;   // no pass follows: a target that needs one gets results at its last h
    int hold_cells;  // adaptive: the cells cannot be rebuilt during this iteration
};

// slot of a name and the offset of its frame from the target's
template <int MODE>
__device__ __forceinline__ int name_slot(const SumArgs &a, unsigned name, uint32_t e0, float L,
                                         const float4 *__restrict__ shift, float &sx, float &sy, float &sz)
{
    if (MODE == 1) {
        const uint32_t e = e0 + (name >> a.wbits);
        const float4 en = __ldg(a.list + e);
        const int first = __ldg(a.list_slot + e);
        sx = en.x;
        sy = en.y;
        sz = en.z;
        return first + (int)(name & ((1u << a.wbits) - 1u));
    }
    const float4 o = shift[name >> kSlotBits];  // (62 + dx + 5 dy + 25 dz)
    sx = o.x * L;
    sy = o.y * L;
    sz = o.z * L;
    return (int)(name & ((1u << kSlotBits) - 1u));
}

__device__ __forceinline__ void load_shifts(float4 *shift)
{
    for (int o = threadIdx.x; o < 125; o += blockDim.x)
        shift[o] = make_float4((float)(o % 5 - 2), (float)((o / 5) % 5 - 2), (float)(o / 25 - 2), 0.f);
    __syncthreads();
}

// sum over the G lanes of a target
template <int G>
__device__ __forceinline__ float sum_lanes(float v)
{
#pragma unroll
    for (int d = 1; d < G; d <<= 1) v += __shfl_xor_sync(kFull, v, d);
    return v;
}

// Order of a warp's rows by the length of their lists (key: length << 5 | row): lane k
// gets the k-th shortest.
__device__ __forceinline__ unsigned sort_rows(unsigned key)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const unsigned other = __shfl_xor_sync(kFull, key, j);
            const bool low = ((lane & j) == 0) == ((lane & k) == 0);
            key = low ? min(key, other) : max(key, other);
        }
    return key;
}

// 1/sqrt(x), 0 for a separation of zero (a denormal square is one of pairs that are separated:
// three more instructions for its scaling); 1/x as one MUFU instruction
__device__ __forceinline__ float inv_sqrt(float x)
{
    float y;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return x > 0.f ? y : 0.f;
}
__device__ __forceinline__ float inv(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The FP32 band around the cutoff in q = r / h: half the relative band of r^2, and the
// rounding of q itself.  Outside it q < 1 is the FP64 decision.
__device__ __forceinline__ float near_one(float hinv, float L)
{
    return fmaf(0.5f * kBandK * L, hinv, 0.5f * kBandK + 1e-6f);
}

// The names of a list (left of them from page on), taken by G lanes (q: the lane's place
// among them), two each per step: f(names, valid), then end of step g().  Every lane of the
// warp calls it; what a list's lanes add does not depend on the lists beside it.
struct Two {
    unsigned v[2];
    __device__ __forceinline__ unsigned operator[](int k) const { return v[k]; }
};
struct TwoBool {
    bool v[2];
    __device__ __forceinline__ bool operator[](int k) const { return v[k]; }
};
template <int G, class F, class E>
__device__ __forceinline__ void walk_list(const SumArgs &a, int left, int page, int q, F f, E g)
{
    while (__any_sync(kFull, left > 0)) {
        const uint32_t *nm = a.pages + (size_t)page * kPage + q;
        unsigned c0 = q < left ? __ldg(nm) : 0u, c1 = G + q < left ? __ldg(nm + G) : 0u;
        int run = 0, nxt = 0;
        if (left > 0) {
            run = kPage * __ldg(a.next + page);
            nxt = __ldg(a.next + page + 1);
        }
        const int m = min(left, run);
#pragma unroll 1
        for (int x = 0; __any_sync(kFull, x < m); x += 2 * G) {
            const unsigned d0 = x + 2 * G + q < m ? __ldg(nm + x + 2 * G) : 0u;
            const unsigned d1 = x + 3 * G + q < m ? __ldg(nm + x + 3 * G) : 0u;
            f(Two{{c0, c1}}, TwoBool{{x + q < m, x + G + q < m}});
            g();
            c0 = d0;
            c1 = d1;
        }
        // (lists that end their chunk before the longest beside them have been given zeros, which
        // may round a compensated sum again, once: now each of them has been)
        g();
        left -= m;
        page = nxt;
    }
}

struct DensRow {
    int i;           // slot
    int left, page;  // names, first page
    float h, L;
    uint32_t e0;
};

// Sums of one target by G lanes (q: the lane's place among them): to out[0..8].  Every lane
// of the warp calls it (on: the lane's target counts).
template <int MODE, bool HASH, int G>
__device__ __forceinline__ void density_row(const DensityListArgs &a, const float4 *shift, DensRow t, bool on, int q,
                                            float *out, unsigned long long *out_hash)
{
    if (!on) t.left = 0;
    const float4 pi = a.s.pos4[t.i], vi = a.s.vel4[t.i];
    const float hinv = 1.f / t.h;
    const float band = near_one(hinv, t.L);
    float rho_s = 0.f, rho_c = 0.f, sw_s = 0.f, sw_c = 0.f, sqdw = 0.f, drho = 0.f;
    float dv = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
    int hits = 0;
    unsigned long long hh = 0ull;
    float rb = 0.f, wb = 0.f;
    walk_list<G>(
        a.s, t.left, t.page, q,
        [&](Two name, TwoBool ok) {
            // (both sources' reads first, one rare branch for both)
            int j[2];
            float4 pj[2], vj[2];
            float dx[2], dy[2], dz[2], rinv[2], qq[2];
            bool in[2], near = false;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float sx = 0.f, sy = 0.f, sz = 0.f;
                j[e] = ok[e] ? name_slot<MODE>(a.s, name[e], t.e0, t.L, shift, sx, sy, sz) : t.i;
                pj[e] = __ldg(a.s.pos4 + j[e]);
                vj[e] = __ldg(a.s.vel4 + j[e]);
                dx[e] = sx;
                dy[e] = sy;
                dz[e] = sz;
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                dx[e] = pi.x - (pj[e].x + dx[e]);
                dy[e] = pi.y - (pj[e].y + dy[e]);
                dz[e] = pi.z - (pj[e].z + dz[e]);
                const float r2 = fmaf(dx[e], dx[e], fmaf(dy[e], dy[e], dz[e] * dz[e]));
                rinv[e] = inv_sqrt(r2);
                qq[e] = ok[e] ? r2 * rinv[e] * hinv : 2.f;  // (the terms vanish from q = 1 on)
                in[e] = qq[e] < 1.f;
                near |= fabsf(qq[e] - 1.f) < band;
            }
            // inside the FP32 band (rare) the FP64 separation decides
            if (near) {
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (fabsf(qq[e] - 1.f) < band) {
                        in[e] = band_decide(a.s.x, a.s.y, a.s.z, t.i, j[e], a.s.box, t.h, t.h) & 1u;
                        qq[e] = in[e] ? qq[e] : 1.f;
                    }
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float w, dw;
                spline_u(qq[e], w, dw);
                hits += in[e] ? 1 : 0;
                if (HASH && in[e]) hh += mix64((uint64_t)a.ids[j[e]]);
                const float mj = vj[e].w;
                rb = fmaf(mj, w, rb);
                wb += w;
                sqdw = fmaf(qq[e], dw, sqdw);
                drho = fmaf(mj, fmaf(qq[e], dw, 3.f * w), drho);
                const float fr = mj * dw * rinv[e];
                const float vx = vi.x - vj[e].x, vy = vi.y - vj[e].y, vz = vi.z - vj[e].z;
                dv = fmaf(fr, fmaf(vx, dx[e], fmaf(vy, dy[e], vz * dz[e])), dv);
                cx = fmaf(fr, fmaf(vy, dz[e], -vz * dy[e]), cx);
                cy = fmaf(fr, fmaf(vz, dx[e], -vx * dz[e]), cy);
                cz = fmaf(fr, fmaf(vx, dy[e], -vy * dx[e]), cz);
            }
        },
        [&]() {
            kahan_add(rho_s, rho_c, rb);
            kahan_add(sw_s, sw_c, wb);
            rb = wb = 0.f;
        });
    const float r0 = sum_lanes<G>(rho_s - rho_c), r1 = sum_lanes<G>(sw_s - sw_c), r2s = sum_lanes<G>(sqdw),
                r3 = sum_lanes<G>(drho), r4 = sum_lanes<G>(dv), r5 = sum_lanes<G>(cx), r6 = sum_lanes<G>(cy),
                r7 = sum_lanes<G>(cz);
#pragma unroll
    for (int d = 1; d < G; d <<= 1) {
        hits += __shfl_xor_sync(kFull, hits, d);
        if (HASH) hh += __shfl_xor_sync(kFull, hh, d);
    }
    if (on && q == 0) {
        out[0] = r0;
        out[1] = r1;
        out[2] = r2s;
        out[3] = r3;
        out[4] = r4;
        out[5] = r5;
        out[6] = r6;
        out[7] = r7;
        out[8] = __int_as_float(hits);
        if (HASH) *out_hash = hh;
    }
}

template <int MODE, bool HASH>
__global__ void __launch_bounds__(kSumThreads, kSumBlocks) k_density_l(DensityListArgs a)
{
    if (a.s.counters[C_STALE] & 1ull) return;  // no lists: the kernels of sph_pairs.cu run
    if (a.s.run_if && *a.s.run_if == 0ull) return;
    constexpr bool LIST = MODE == 1;
    __shared__ float4 shift[LIST ? 1 : 125];
    __shared__ float s_sum[kSumThreads / 32][32][9];
    __shared__ unsigned long long s_hash[HASH ? kSumThreads / 32 : 1][32];
    __shared__ uint8_t s_ord[kSumThreads / 32][32];
    if (!LIST) load_shifts(shift);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int grp8 = lane >> 3, q = lane & 7;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const int ntiles = *a.s.n_tiles;
    unsigned long long acc_pairs = 0ull;
    unsigned acc_targets = 0u, acc_lost = 0u, acc_flag = 0u, left_ev = 0u, most_ev = 0u;
    unsigned *ticket = reinterpret_cast<unsigned *>(a.s.ticket);
    unsigned tk = 0u;
    if (lane == 0) tk = atomicAdd(ticket, 1u);
    const int nrows = a.rows ? (int)*a.n_rows : 0;
    const int units = a.rows ? (nrows + 3) / 4 : tile_parts(a.s, ntiles);
    for (int u = gw, u_after = 0; u < units; u = u_after) {
        u_after = nw + (int)__shfl_sync(kFull, tk, 0);
        if (lane == 0 && u_after < units) tk = atomicAdd(ticket, 1u);
        // lane = target: its slot, leaf and box, and its state
        int i = 0, leaf = 0, bi = 0;
        bool act;
        if (a.rows) {
            act = lane < 4 && u * 4 + lane < nrows;
            if (act) {
                i = a.rows[u * 4 + lane];
                if (LIST) leaf = a.leaf_of[i];
                int h2 = a.nb - 1;
                while (bi < h2) {
                    const int mid = (bi + h2 + 1) >> 1;
                    if (a.s.boxes[mid].p_begin <= i) bi = mid;
                    else h2 = mid - 1;
                }
            }
        } else {
            int row0, per;
            const int4 tile = a.s.tiles[tile_part(a.s, ntiles, u, row0, per)];
            act = lane < per && row0 + lane < tile.z;
            if (act) i = LIST ? a.s.tord[tile.y + row0 + lane] : tile.y + row0 + lane;
            act = act && a.active[i];
            leaf = tile.x;
            bi = tile.w;
        }
        unsigned todo = __ballot_sync(kFull, act);
        if (!todo) continue;
        const float Lcell = a.s.boxes[bi].L32;
        const float L = LIST ? a.s.leaf_scale[leaf] : Lcell;
        const uint32_t e0 = LIST ? a.s.list_off[leaf] : 0u;
        float hi = 1.f, rad = 0.f, lo = 0.f, up = kHUnbounded;
        int cnt = 0, head = 0;
        if (act) {
            hi = a.h[i];
            rad = a.s.radius[i];
            cnt = a.s.cnt[i];
            head = a.s.head[i];
            lo = a.h_lo[i];
            up = a.h_hi[i];
        }
        const unsigned sorted = sort_rows(((unsigned)min(cnt, (1 << 26) - 1) << 5) | (unsigned)lane);
        bool run = act;
        int ev = 0;
        while (todo) {
            // evaluate the sums of every target in todo: the short lists four at a time,
            // then the long ones one by one
            const bool mine = (todo >> (sorted & 31u)) & 1u;
            const unsigned all = __ballot_sync(kFull, mine);
            const unsigned lng = __ballot_sync(kFull, mine && (sorted >> 5) > (unsigned)kLongList);
            if (mine) s_ord[wib][__popc(all & ((1u << lane) - 1u))] = (uint8_t)(sorted & 31u);
            __syncwarp();
            const int nt = __popc(all), ns = nt - __popc(lng);
            for (int s0 = 0; s0 < ns; s0 += 4) {
                const bool on = s0 + grp8 < ns;
                const int row = on ? s_ord[wib][s0 + grp8] : 0;
                const DensRow r{__shfl_sync(kFull, i, row),  __shfl_sync(kFull, cnt, row), __shfl_sync(kFull, head, row),
                                __shfl_sync(kFull, hi, row), __shfl_sync(kFull, L, row),   __shfl_sync(kFull, e0, row)};
                density_row<MODE, HASH, 8>(a, shift, r, on, q, s_sum[wib][row], s_hash[HASH ? wib : 0] + row);
            }
            for (int s0 = ns; s0 < nt; ++s0) {
                const int row = s_ord[wib][s0];
                const DensRow r{__shfl_sync(kFull, i, row),  __shfl_sync(kFull, cnt, row), __shfl_sync(kFull, head, row),
                                __shfl_sync(kFull, hi, row), __shfl_sync(kFull, L, row),   __shfl_sync(kFull, e0, row)};
                density_row<MODE, HASH, 32>(a, shift, r, true, lane, s_sum[wib][row], s_hash[HASH ? wib : 0] + row);
            }
            __syncwarp();
            // lane = target: Newton's step, or the results
            bool leaves = false, grown = false;
            if (run) {
                const float *o = s_sum[wib][lane];
                const int hits = __float_as_int(o[8]);
                acc_pairs += (unsigned)(hits - 1);  // (the (i, i) pair is not a neighbour)
                ++acc_targets;
                ++ev;
                const float hinv = 1.f / hi;
                const float hinv3 = hinv * hinv * hinv, hinv4 = hinv3 * hinv;
                const float nw_ = kSigma * kFourPi3 * o[1];
                const float dnw_dh = -kSigma * kFourPi3 * o[2] * hinv;
                const float g = nw_ - a.n_ngb_target;
                bool conv = fabsf(g) <= a.h_tol * a.n_ngb_target;
                if (!conv) {
                    // every evaluation narrows a bracket of the root; once it is a few FP32
                    // ulps wide the FP32 sums cannot place the root more finely
                    if (g < 0.f) lo = fmaxf(lo, hi);
                    else up = fminf(up, hi);
                    conv = lo > 0.f && up < kHUnbounded && up - lo <= kHResolution * lo;
                }
                float hn = hi;
                unsigned flag = 0u;
                if (!conv) {
                    hn = next_h(hi, g, dnw_dh, lo, up);
                    if (LIST) {
                        // adaptive cells: h up to just below half the box; beyond what its
                        // leaf's list or the adjacent top cells hold the cells are built
                        // again -- or, where they cannot be (captured steps), the step is cut
                        // back to that limit and reported only once the iterate sits there
                        // with N_w still short
                        const float lim = fminf(fminf(kTreeReach * a.s.leaf_hb[leaf], Lcell), (float)(0.5 * a.s.box));
                        hn = fminf(hn, (float)(0.5 * a.s.box) * (1.f - 1e-5f));
                        if (a.hold_cells) {
                            const float cap = lim * (1.f - 2e-6f);
                            if (hn > cap) {
                                if (g < 0.f && hi >= cap * (1.f - 1e-6f)) flag = 2u;
                                hn = cap;
                            }
                        } else if (hn > lim * (1.f - 1e-6f)) {
                            flag = 2u;
                        }
                    } else if ((double)hn > 2.0 * a.s.boxes[bi].L64 * (1.0 - 1e-6)) {
                        flag = 2u;  // beyond the radius-2 stencil of its cell
                    }
                }
                const bool beyond = flag != 0u || hn > rad;  // beyond the cells, or the list
                if (!conv && ev < a.budget && !(beyond && a.last_pass)) {
                    acc_flag |= flag;
                    if (beyond) {  // another pass
                        run = false;
                        leaves = true;
                        left_ev = max(left_ev, (unsigned)ev);
                        a.h[i] = hn;
                        a.h_lo[i] = lo;
                        a.h_hi[i] = up;
                    }
                    hi = hn;
                } else {
                    run = false;
                    if (!conv) {
                        ++acc_lost;
                        acc_flag |= flag;
                    }
                    // uniform grid: FP32 cell-relative positions resolve h only down to
                    // cell side / SPH_FRAME_RATIO at the density tolerance
                    if (!LIST && Lcell > (float)SPH_FRAME_RATIO * hi) acc_flag |= 4u;
                    // the lists of its neighbours hold it up to this h
                    grown = hi > a.s.pos4[i].w * a.grow * (1.f - 1e-6f);
                    a.active[i] = 0;
                    a.h[i] = hi;
                    // quantities needed before the pressure gradient (EOS, grad-h, Balsara)
                    const float rho = kSigma * hinv3 * o[0];
                    const float drho_dh = -kSigma * hinv4 * o[3];
                    const float divv = -kSigma * hinv4 * o[4] / rho;
                    const float curl = kSigma * hinv4 * sqrtf(o[5] * o[5] + o[6] * o[6] + o[7] * o[7]) / rho;
                    const float u = a.upred[i];
                    const float gam = a.gamma;
                    const float P = (gam - 1.f) * rho * u;
                    const float cs = sqrtf(gam * (gam - 1.f) * u);
                    const float fgh = 1.f / (1.f + hi / (3.f * rho) * drho_dh);
                    float Bq = 1.f;
                    if (a.use_balsara) {
                        const float ad = fabsf(divv);
                        const float den = ad + curl + 1e-4f * cs * hinv;
                        Bq = den > 0.f ? ad / den : 0.f;
                    }
                    a.thermo4[i] = make_float4(rho, fgh * P / (rho * rho), cs, Bq);
                    a.rho[i] = rho;
                    a.P[i] = P;
                    a.c[i] = cs;
                    a.f[i] = fgh;
                    a.divv[i] = divv;
                    a.curl[i] = curl;
                    a.n_ngb[i] = hits - 1;
                    if (HASH) a.ngb_hash[i] = s_hash[wib][lane] - mix64((uint64_t)a.ids[i]);
                }
            }
            const unsigned lv = __ballot_sync(kFull, leaves), gr = __ballot_sync(kFull, grown);
            if (lv) {
                unsigned at = 0u;
                if (lane == 0) at = (unsigned)atomicAdd(a.left, (unsigned long long)__popc(lv));
                at = __shfl_sync(kFull, at, 0);
                if (leaves) a.left_rows[at + __popc(lv & ((1u << lane) - 1u))] = i;
            }
            if (gr) {
                unsigned at = 0u;
                if (lane == 0) at = (unsigned)atomicAdd(a.s.counters + C_GROWN, (unsigned long long)__popc(gr));
                at = __shfl_sync(kFull, at, 0);
                if (grown) a.grown_rows[at + __popc(gr & ((1u << lane) - 1u))] = i;
            }
            todo = __ballot_sync(kFull, run);
        }
        most_ev = max(most_ev, (unsigned)ev);
    }
    const unsigned long long tp = warp_sum_ull(acc_pairs);
    const unsigned tt = __reduce_add_sync(kFull, acc_targets);
    const unsigned tf = __reduce_or_sync(kFull, acc_flag);
    const unsigned tl = __reduce_max_sync(kFull, left_ev), tx = __reduce_add_sync(kFull, acc_lost);
    const unsigned tm = __reduce_max_sync(kFull, most_ev);
    if (lane == 0) {
        unsigned long long *c = a.s.counters;
        if (tp) atomicAdd(c + C_DPAIRS, tp);
        if (tt) atomicAdd(c + C_DTARGETS, (unsigned long long)tt);
        if (tf & 2u) atomicOr(c + C_HFLAG, 1ull);
        if (tf & 4u) atomicOr(c + C_PREC, 1ull);
        if (tl) atomicMax(reinterpret_cast<unsigned *>(a.left + 3), tl);
        if (tm) atomicMax(reinterpret_cast<unsigned *>(a.left + 3) + 1, tm);
        if (tx) atomicAdd(c + C_LOST, (unsigned long long)tx);
    }
}

// The targets that the lists of a few grown particles' neighbours miss: for every j whose h
// outgrew the radius its neighbours searched with, the targets of its own list (searched at
// the new h) beyond that radius, each once (mark: zero from the start of the density call).
// pos4.w still holds the h that the searches used; h the converged one.
struct MarkArgs {
    SumArgs s;
    const float *__restrict__ h;
    const int *__restrict__ grown;
    const int *__restrict__ leaf_of;
    const uint8_t *__restrict__ mask;  // individual time-steps: targets of the force pass (null: all)
    uint8_t *mark;
    int *dirty;
    int nb;
    float grow;
    unsigned run_upto;
};

template <int MODE>
__global__ void __launch_bounds__(256) k_mark_dirty(MarkArgs a)
{
    const unsigned long long ng = a.s.counters[C_GROWN];
    if (ng == 0ull || ng > a.run_upto || (a.s.counters[C_STALE] & 3ull)) return;
    constexpr bool LIST = MODE == 1;
    __shared__ float4 shift[LIST ? 1 : 125];
    if (!LIST) load_shifts(shift);
    const int lane = threadIdx.x & 31;
    for (int u = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); u < (int)ng;
         u += (int)((gridDim.x * blockDim.x) >> 5)) {
        const int i = a.grown[u];
        int bi = 0, h2 = a.nb - 1;
        while (bi < h2) {
            const int mid = (bi + h2 + 1) >> 1;
            if (a.s.boxes[mid].p_begin <= i) bi = mid;
            else h2 = mid - 1;
        }
        const int leaf = LIST ? a.leaf_of[i] : 0;
        const float L = LIST ? a.s.leaf_scale[leaf] : a.s.boxes[bi].L32;
        const uint32_t e0 = LIST ? a.s.list_off[leaf] : 0u;
        const float4 pi = a.s.pos4[i];
        const float hf = a.h[i];
        const float reach = LIST ? pi.w * a.grow : fminf(pi.w * a.grow, 2.f * L * (1.f - 1e-6f));
        const float top = fmaf(hf, hf, 2.f * kBandK * hf * (hf + L));
        walk_list<32>(a.s, a.s.cnt[i], a.s.head[i], lane, [&](Two name, TwoBool ok) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (!ok[e]) continue;
                float sx, sy, sz;
                const int j = name_slot<MODE>(a.s, name[e], e0, L, shift, sx, sy, sz);
                const float4 pj = a.s.pos4[j];
                const float dx = pi.x - (pj.x + sx), dy = pi.y - (pj.y + sy), dz = pi.z - (pj.z + sz);
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                // what j's list holds: pairs within j's own list radius (on adaptive cells as far as
                // its leaf's entries reach, which may end below h_j's growth) or i's reach
                const float held = fmaxf(reach, __ldg(a.s.radius + j)) * (1.f - 1e-5f);
                if (j != i && r2 < top && r2 > held * held && (a.mask == nullptr || a.mask[j])) {
                    // (one writer wins: bytes are marked through their word)
                    const unsigned bit = 1u << (8 * (j & 3));
                    const unsigned old = atomicOr(reinterpret_cast<unsigned *>(a.mark + (j & ~3)), bit);
                    if (!(old & bit)) a.dirty[atomicAdd(reinterpret_cast<unsigned *>(a.s.counters + C_DIRTY), 1u)] = j;
                }
            }
        }, []() {});
    }
}

struct ForceListArgs {
    SumArgs s;
    float *ax, *ay, *az, *dudt, *vsig;
    const uint8_t *__restrict__ fmask;  // individual time-steps: targets to update (null: all)
    float alpha;
};

// Sums of one target by G lanes: to out[0..4]; returns this lane's neighbours.
template <int MODE, int G>
__device__ __forceinline__ int force_row(const ForceListArgs &a, const float4 *shift, int i, int left, int page, float L,
                                         uint32_t e0, bool on, int q, float *out)
{
    if (!on) left = 0;
    const float4 pi = a.s.pos4[i], vi = a.s.vel4[i], ti = a.s.thermo4[i];
    const float hi = pi.w, hinv = 1.f / hi, hinv4 = hinv * hinv * hinv * hinv;
    const float band_i = near_one(hinv, L);
    const float alpha = -0.25f * a.alpha;  // -alpha, the mean of the two Balsara factors and of the two gradients
    float sx_ = 0.f, sxc = 0.f, sy_ = 0.f, syc = 0.f, sz_ = 0.f, szc = 0.f, su = 0.f, suc = 0.f, vs = 0.f;
    int hits = 0;
    ForceSum part;
    walk_list<G>(
        a.s, left, page, q,
        [&](Two name, TwoBool ok) {
            // (both sources' reads first, one rare branch for both)
            int j[2];
            float4 pj[2], vj[2], tj[2];
            float dx[2], dy[2], dz[2], rinv[2], hjinv[2], qi[2], qj[2];
            bool near = false;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float fx = 0.f, fy = 0.f, fz = 0.f;
                j[e] = ok[e] ? name_slot<MODE>(a.s, name[e], e0, L, shift, fx, fy, fz) : i;
                pj[e] = __ldg(a.s.pos4 + j[e]);
                vj[e] = __ldg(a.s.vel4 + j[e]);
                tj[e] = __ldg(a.s.thermo4 + j[e]);
                dx[e] = fx;
                dy[e] = fy;
                dz[e] = fz;
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                dx[e] = pi.x - (pj[e].x + dx[e]);
                dy[e] = pi.y - (pj[e].y + dy[e]);
                dz[e] = pi.z - (pj[e].z + dz[e]);
                const float r2 = fmaf(dx[e], dx[e], fmaf(dy[e], dy[e], dz[e] * dz[e]));
                rinv[e] = inv_sqrt(r2);
                const float r = ok[e] ? r2 * rinv[e] : 1e30f;
                hjinv[e] = inv(pj[e].w);
                qi[e] = r * hinv;  // (a term vanishes from q = 1 on)
                qj[e] = r * hjinv[e];
                near |= fabsf(qi[e] - 1.f) < band_i || fabsf(qj[e] - 1.f) < near_one(hjinv[e], L);
            }
            // inside the FP32 band of either (rare) the FP64 separation decides
            if (near) {
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (fabsf(qi[e] - 1.f) < band_i || fabsf(qj[e] - 1.f) < near_one(hjinv[e], L)) {
                        const unsigned d = band_decide(a.s.x, a.s.y, a.s.z, i, j[e], a.s.box, hi, pj[e].w);
                        qi[e] = (d & 1u) ? fminf(qi[e], 0.99999994f) : fmaxf(qi[e], 1.f);
                        qj[e] = (d & 2u) ? fminf(qj[e], 0.99999994f) : fmaxf(qj[e], 1.f);
                    }
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool in = fminf(qi[e], qj[e]) < 1.f;
                hits += in ? 1 : 0;
                // the pair term (force_term), without sigma; the pair (i, i), and coincident pairs,
                // have no direction: 1/r = 0
                const float hj2inv = hjinv[e] * hjinv[e];
                const float Wi = spline_dw_u(qi[e]) * hinv4, Wj = spline_dw_u(qj[e]) * (hj2inv * hj2inv);
                const float vx = vi.x - vj[e].x, vy = vi.y - vj[e].y, vz = vi.z - vj[e].z;
                const float mu = fmaf(vx, dx[e], fmaf(vy, dy[e], vz * dz[e])) * rinv[e];
                const float muc = fminf(mu, 0.f);
                const float vsig = ti.z + tj[e].z - 3.f * muc;
                const float Pi = alpha * vsig * muc * (ti.w + tj[e].w) * inv(ti.x + tj[e].x) * (Wi + Wj);
                const float mj = vj[e].w;
                const float sc = mj * fmaf(ti.y, Wi, fmaf(tj[e].y, Wj, Pi)) * rinv[e];
                part.x = fmaf(-sc, dx[e], part.x);
                part.y = fmaf(-sc, dy[e], part.y);
                part.z = fmaf(-sc, dz[e], part.z);
                part.u = fmaf(mj * mu, fmaf(ti.y, Wi, 0.5f * Pi), part.u);
                if (in && rinv[e] > 0.f) vs = fmaxf(vs, vsig);
            }
        },
        [&]() {
            kahan_add(sx_, sxc, part.x);
            kahan_add(sy_, syc, part.y);
            kahan_add(sz_, szc, part.z);
            kahan_add(su, suc, part.u);
            part.x = part.y = part.z = part.u = 0.f;
        });
    const float rx = kSigma * sum_lanes<G>(sx_ - sxc), ry = kSigma * sum_lanes<G>(sy_ - syc),
                rz = kSigma * sum_lanes<G>(sz_ - szc), ru = kSigma * sum_lanes<G>(su - suc);
#pragma unroll
    for (int d = 1; d < G; d <<= 1) vs = fmaxf(vs, __shfl_xor_sync(kFull, vs, d));
    if (on && q == 0) {
        out[0] = rx;
        out[1] = ry;
        out[2] = rz;
        out[3] = ru;
        out[4] = vs;
    }
    return hits;
}

template <int MODE>
__global__ void __launch_bounds__(kSumThreads, kSumBlocks) k_force_l(ForceListArgs a)
{
    if (a.s.counters[C_FOVF]) return;
    constexpr bool LIST = MODE == 1;
    __shared__ float4 shift[LIST ? 1 : 125];
    __shared__ float s_sum[kSumThreads / 32][32][5];
    if (!LIST) load_shifts(shift);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int grp8 = lane >> 3, q = lane & 7;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const int ntiles = *a.s.n_tiles;
    unsigned long long acc_pairs = 0ull;
    unsigned *ticket = reinterpret_cast<unsigned *>(a.s.ticket);
    unsigned tk = 0u;
    if (lane == 0) tk = atomicAdd(ticket, 1u);
    const int units = tile_parts(a.s, ntiles);
    for (int u = gw, u_after = 0; u < units; u = u_after) {
        u_after = nw + (int)__shfl_sync(kFull, tk, 0);
        if (lane == 0 && u_after < units) tk = atomicAdd(ticket, 1u);
        int row0, per;
        const int4 tile = a.s.tiles[tile_part(a.s, ntiles, u, row0, per)];
        const bool valid = lane < per && row0 + lane < tile.z;
        const int i = LIST ? (valid ? a.s.tord[tile.y + row0 + lane] : 0) : (valid ? tile.y + row0 + lane : 0);
        const bool act = valid && (a.fmask == nullptr || a.fmask[i]);
        if (!__any_sync(kFull, act)) continue;
        const BoxDev bx = a.s.boxes[tile.w];
        const float L = LIST ? a.s.leaf_scale[tile.x] : bx.L32;
        const uint32_t e0 = LIST ? a.s.list_off[tile.x] : 0u;
        int cnt = 0, head = 0;
        if (act) {
            cnt = a.s.cnt[i];
            head = a.s.head[i];
        }
        // rows without a target sort to the end
        const unsigned sorted = sort_rows((act ? (unsigned)min(cnt, (1 << 26) - 1) << 5 : 0xffffffe0u) | (unsigned)lane);
        const int nt = __popc(__ballot_sync(kFull, act));
        const int ns = __popc(__ballot_sync(kFull, lane < nt && (sorted >> 5) <= (unsigned)kLongList));
        for (int s0 = 0; s0 < ns; s0 += 4) {
            const bool on = s0 + grp8 < ns;
            const int row = (int)(__shfl_sync(kFull, sorted, on ? s0 + grp8 : 0) & 31u);
            acc_pairs += (unsigned)force_row<MODE, 8>(a, shift, __shfl_sync(kFull, i, row), __shfl_sync(kFull, cnt, row),
                                                      __shfl_sync(kFull, head, row), L, e0, on, q, s_sum[wib][row]);
        }
        for (int s0 = ns; s0 < nt; ++s0) {
            const int row = (int)(__shfl_sync(kFull, sorted, s0) & 31u);
            acc_pairs += (unsigned)force_row<MODE, 32>(a, shift, __shfl_sync(kFull, i, row),
                                                       __shfl_sync(kFull, cnt, row), __shfl_sync(kFull, head, row), L, e0,
                                                       true, lane, s_sum[wib][row]);
        }
        __syncwarp();
        if (act) {
            const float *o = s_sum[wib][lane];
            a.ax[i] = o[0];
            a.ay[i] = o[1];
            a.az[i] = o[2];
            a.dudt[i] = o[3];
            a.vsig[i] = o[4];
            acc_pairs -= 1ull;  // the (i, i) pair is not a neighbour
        }
        __syncwarp();
    }
    const unsigned long long tp = warp_sum_ull(acc_pairs);
    if (lane == 0 && tp) atomicAdd(a.s.counters + C_FPAIRS, tp);
}

// ------------------------------------------------------------------ host side

// Targets up to which the search for single targets runs: beyond, staging the sources
// of whole leaves (cells) is cheaper.
unsigned list_few_rows(const sph_ctx *ctx) { return (unsigned)std::max<int64_t>(32, ctx->n / 24); }

// Start of a density call's searches (or of the force pass's own, which starts the pool
// again only where it will run): the pool, the flags, and the tickets and counts of every
// pass, which so need no reset between the passes.
__global__ void k_lists_begin(unsigned long long *c, int force, unsigned few)
{
    const int t = threadIdx.x;
    if (force) {
        if (t == 0) {
            c[C_FOVF] = 0ull;
            if ((c[C_STALE] & 3ull) || c[C_GROWN] > few) c[C_PAGES] = 0ull;  // a search of its own
        }
        if (t < 2) c[C_FTICKET + t] = 0ull;
    } else {
        if (t == 0) c[C_PAGES] = c[C_STALE] = c[C_LOST] = c[C_HFLAG] = c[C_GROWN] = c[C_DIRTY] = 0ull;
        if (t < 4 * kListPasses) c[C_PASS + t] = 0ull;
    }
}

// Whether the names hold the slots (uniform grid: 2^25 of them) and the per-axis sweep, whose
// staging is its own, is off.
bool lists_fit(const sph_ctx *ctx)
{
    if (ctx->n <= 0) return false;
    if (ctx->adaptive) return true;
    return ctx->n <= ((int64_t)1 << kSlotBits) && !(ctx->p.flags & SPH_FLAG_AXIS_SWEEP);
}

// Whether the sums run over lists: as above, and there are arrays for them (ensure_lists).
bool lists_apply(const sph_ctx *ctx)
{
    return lists_fit(ctx) && ctx->lists.pages && ctx->lists.cap >= ctx->cap;
}

// Pages a pool grows to: 512 names a particle on average, 2^32 in all.
int64_t lists_most_pages(const sph_ctx *ctx)
{
    const int64_t most = std::min<int64_t>(16 * std::max<int64_t>(ctx->cap, 64), kMaxPages);
    return ctx->limits.list_pages >= 0 ? std::min(most, ctx->limits.list_pages) : most;
}

void free_lists(sph_ctx *ctx)
{
    ListPool &P = ctx->lists;
    cudaFree(P.pages);
    cudaFree(P.next);
    cudaFree(P.head);
    cudaFree(P.cnt);
    cudaFree(P.radius);
    cudaFree(P.rows);
    cudaFree(P.mark);
    const int64_t made = P.made;
    P = ListPool();
    P.made = made;
}

// Arrays for the lists (never inside a capture): `pages` of them at least, five per particle to
// start with, lists_most_pages at most.  Where they would take more than half of the memory
// that is free once the present ones are given back, and which other allocations of the call
// may need, they are not allocated: the pool at hand stays (false: it is smaller than asked
// for), and a call that needs more than that, or has none, runs the kernels of sph_pairs.cu.
bool ensure_lists(sph_ctx *ctx, int64_t pages)
{
    ListPool &P = ctx->lists;
    const int64_t cap = std::max<int64_t>(ctx->cap, 1), had = P.cap_pages;
    pages = std::min(std::max<int64_t>(pages, 5 * cap + 1024), lists_most_pages(ctx));
    const bool slots = P.cap < cap, more = had < pages;
    if (!slots && !more) return true;
    constexpr size_t kSlotBytes = 29, kPageBytes = 4 * (kPage + 1);
    const size_t need = (slots ? kSlotBytes * (size_t)cap : 0) + (more ? kPageBytes * (size_t)pages : 0);
    const size_t back = (slots ? kSlotBytes * (size_t)P.cap : 0) + (more ? kPageBytes * (size_t)had : 0);
    size_t left = 0, total = 0;
    if (cudaMemGetInfo(&left, &total) != cudaSuccess) {
        cudaGetLastError();
        left = 0;
    }
    if (ctx->limits.free_bytes >= 0) left = (size_t)ctx->limits.free_bytes;
    if (need > (left + back) / 2) {
        if (slots) free_lists(ctx);  // (of a smaller particle count)
        return false;
    }
    auto room = [&](auto **p, size_t bytes) {
        cudaFree(*p);
        *p = nullptr;
        if (cudaMalloc(p, bytes) == cudaSuccess) return true;
        cudaGetLastError();  // (out of memory is not an error here)
        return false;
    };
    auto pool = [&](int64_t n) {
        P.cap_pages = n;
        return room(&P.pages, sizeof(uint32_t) * kPage * (size_t)n) && room(&P.next, sizeof(int) * (size_t)n);
    };
    bool ok = true;
    ++P.made;
    if (slots) {
        ok = room(&P.head, sizeof(int) * cap) && room(&P.cnt, sizeof(int) * cap) &&
             room(&P.radius, sizeof(float) * cap) && room(&P.rows, 4 * sizeof(int) * cap) &&
             room(&P.mark, ((size_t)cap + 3) / 4 * 4);
        P.cap = cap;
    }
    if (ok && more && !pool(pages)) {
        ok = had > 0 && pool(had);  // (another process was quicker)
        if (ok) return false;
    }
    if (!ok) free_lists(ctx);
    return ok;
}

// Whether a density call (or a captured step) searches into lists; `pages` as in ensure_lists.
// Lists that do not fit the largest pool cost a search of no use in every call (adaptive sets of
// more than 40 M particles, whose names would take more than 2^32, and lists beyond 512 names a
// particle): after two such calls in a row the next goes by without, after three the next two,
// then 4, 8, ... up to 64 before one tries again.
bool lists_turn(sph_ctx *ctx, int64_t pages)
{
    ListPool &P = ctx->lists;
    if (!lists_fit(ctx)) return false;
    if (P.misses_n != ctx->n) P.misses = P.skip = 0;
    if (P.skip > 0) {
        --P.skip;
        return false;
    }
    ensure_lists(ctx, pages);
    return lists_apply(ctx);
}

void lists_result(sph_ctx *ctx, bool fitted)
{
    ListPool &P = ctx->lists;
    P.misses = fitted ? 0 : std::min(P.misses + 1, 8);
    P.skip = P.misses < 2 ? 0 : 1 << (P.misses - 2);
    P.misses_n = ctx->n;
}

static int list_grid(sph_ctx *ctx, int threads, int blocks_per_sm, int split = 1)
{
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    if (sms <= 0) sms = 148;
    const int64_t cells = ctx->adaptive ? ctx->tree.n_leaves : ctx->grid.n_cells;
    const int64_t want = ((int64_t)ctx->n / ctx->tile_w + cells) / (threads / 32) + 1;
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * blocks_per_sm, want * split));
}

static int name_bits(const sph_ctx *ctx)
{
    int b = 1;
    while ((1 << b) < std::max(ctx->leaf_max, 2)) ++b;
    return b;
}

int lists_begin(sph_ctx *ctx, bool force)
{
    k_lists_begin<<<1, 32, 0, ctx->stream>>>(ctx->counters, force ? 1 : 0, list_few_rows(ctx));
    SPH_LAUNCH(ctx, "list pool");
    return SPH_OK;
}

// Parts a tile of the sums is cut into: whole tiles where there are several for every
// resident warp, smaller parts down to the four targets that run side by side where
// the tiles would leave warps idle.
static int tile_split(sph_ctx *ctx)
{
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    const int64_t warps = (int64_t)(sms > 0 ? sms : 148) * kSumBlocks * (kSumThreads / 32);
    int split = 1;
    while (split < 8 && ctx->n / 32 * split < 4 * warps) split *= 2;
    return split;
}

static SumArgs sum_args(sph_ctx *ctx, sph_particles *parts)
{
    SumArgs s{};
    const ListPool &P = ctx->lists;
    s.pos4 = ctx->pos4;
    s.vel4 = ctx->vel4;
    s.thermo4 = ctx->thermo4;
    s.tiles = ctx->tiles;
    s.n_tiles = ctx->n_tiles;
    s.tord = ctx->tree.tord;
    s.boxes = ctx->d_boxes;
    s.list_off = ctx->tree.list_off;
    s.list = ctx->tree.list;
    s.list_slot = ctx->tree.list_slot;
    s.leaf_scale = ctx->tree.leaf_scale;
    s.leaf_hb = ctx->tree.leaf_h;
    s.pages = P.pages;
    s.next = P.next;
    s.head = P.head;
    s.cnt = P.cnt;
    s.radius = P.radius;
    s.x = parts->x;
    s.y = parts->y;
    s.z = parts->z;
    s.counters = ctx->counters;
    s.box = ctx->p.box_size;
    s.wbits = name_bits(ctx);
    s.split = tile_split(ctx);
    s.first8 = ctx->adaptive && s.split == 1 ? 64 : 0;
    return s;
}

constexpr size_t kSearchSmem = (kListThreads / 32) * (16 * (size_t)kSearchF4 + 4 * 33);
static_assert(kSearchSmem <= 48 * 1024, "no opt-in needed");

// Uniform matter: ms per call with 5 blocks and with 7, 262,144 particles 3.55, 3.63; 524,288 5.64,
// 5.64; 1 M 9.42, 9.33; 2 M 17.2, 16.9; the point explosion, 512,000 4.21, 4.24; 1 M 6.94, 6.91; 2 M
// 13.3, 13.1.  Adaptive cells: one clustered box has a few tiles with the longest lists and takes
// 5 at every size (500,000 8.8, 9.3; 2 M 17.0, 17.3; 4 M 31.0, 31.8; 8 M 58.5, 60.4); batches of
// 37,000 a box, 16 boxes 9.4, 9.8; 64 22.4, 22.1; 160 52.4, 51.4; 512 152.8, 149.5.
static bool search_many(const sph_ctx *ctx)
{
    if (ctx->adaptive) return ctx->n >= 2000000 && ctx->n_boxes >= 64;
    return ctx->n >= 1000000;
}

// Pass `pass` (below kListPasses) of a density call: lists for the active targets; a pass
// after the first runs only if the one before left targets.  pass < 0: the force pass's own
// search, at the converged h, where the lists of the density passes do not serve.
int run_search(sph_ctx *ctx, sph_particles *parts, int pass, bool all)
{
    const ListPool &P = ctx->lists;
    const bool force = pass < 0;
    SearchArgs a{};
    a.pos4 = ctx->pos4;
    a.h = parts->h;
    a.active = force || all ? (ctx->bin_mode ? ctx->bin_active : nullptr) : ctx->active;
    a.boxes = ctx->d_boxes;
    a.cell_start = ctx->cell_start;
    a.cell_reach = ctx->cell_tmp;
    a.nb = ctx->n_boxes;
    a.tiles = ctx->tiles;
    a.n_tiles = ctx->n_tiles;
    a.list_off = ctx->tree.list_off;
    a.list = ctx->tree.list;
    a.leaf_rng = ctx->tree.leaf_rng;
    a.leaf_scale = ctx->tree.leaf_scale;
    a.leaf_lo = ctx->tree.leaf_lo;
    a.leaf_hi = ctx->tree.leaf_hi;
    a.leaf_hb = ctx->tree.leaf_h;
    a.tord = ctx->tree.tord;
    a.pages = P.pages;
    a.next = P.next;
    a.head = P.head;
    a.cnt = P.cnt;
    a.radius = P.radius;
    a.counters = ctx->counters;
    const unsigned few = list_few_rows(ctx);
    if (force) {
        a.run_if = ctx->counters + C_GROWN;
        a.run_above = few;
        a.or_if = ctx->counters + C_STALE;
    } else if (pass > 0) {
        a.run_if = ctx->counters + C_PASS + 4 * (pass - 1);
        a.run_above = few;
    }
    a.ticket = ctx->counters + (force ? C_FTICKET : C_PASS + 4 * pass + 1);
    a.cap_pages = (unsigned)P.cap_pages;
    a.box = ctx->p.box_size;
    a.grow = force ? 1.f : ctx->lists.grow;
    a.wbits = name_bits(ctx);
    a.force = force ? 1 : 0;
    const bool many = search_many(ctx);
    const int g = list_grid(ctx, kListThreads, many ? kSearchMany : kSearchFew);
    cudaEvent_t end = nullptr;
    timer_begin(ctx, force ? 1 : 0, &end);
    if (ctx->adaptive && many) k_search<1, kSearchMany><<<g, kListThreads, kSearchSmem, ctx->stream>>>(a);
    else if (ctx->adaptive) k_search<1, kSearchFew><<<g, kListThreads, kSearchSmem, ctx->stream>>>(a);
    else if (many) k_search<0, kSearchMany><<<g, kListThreads, kSearchSmem, ctx->stream>>>(a);
    else k_search<0, kSearchFew><<<g, kListThreads, kSearchSmem, ctx->stream>>>(a);
    timer_end(ctx, end);
    SPH_LAUNCH(ctx, "neighbour search");
    if (pass == 0) return SPH_OK;
    // the few targets that the pass before left, or whose neighbours' h grew
    const unsigned blocks = (unsigned)std::min<int64_t>(912, few / 8 + 1);
    const int64_t cap = std::max<int64_t>(ctx->cap, 1);
    SearchOneArgs b{};
    b.s = a;
    b.rows = force ? P.rows + 3 * cap : P.rows + ((pass - 1) & 1) * cap;
    b.n_rows = force ? ctx->counters + C_DIRTY : a.run_if;
    b.run_upto = force ? 0xffffffffu : few;
    b.unless = ctx->counters + C_STALE;
    b.keys = ctx->keys;
    b.leaf_of = ctx->tree.leaf_of;
    if (ctx->adaptive) k_search_one<1><<<blocks, 256, 0, ctx->stream>>>(b);
    else k_search_one<0><<<blocks, 256, 0, ctx->stream>>>(b);
    SPH_LAUNCH(ctx, "search of single targets");
    return SPH_OK;
}

// After the density passes and before pos4 takes the converged h: the targets that miss
// a grown neighbour.
int run_mark(sph_ctx *ctx, sph_particles *parts)
{
    const ListPool &P = ctx->lists;
    const int64_t cap = std::max<int64_t>(ctx->cap, 1);
    MarkArgs m{};
    m.s = sum_args(ctx, parts);
    m.h = parts->h;
    m.grown = P.rows + 2 * cap;
    m.leaf_of = ctx->tree.leaf_of;
    m.mask = ctx->bin_mode ? ctx->bin_active : nullptr;
    m.mark = P.mark;
    m.dirty = P.rows + 3 * cap;
    m.nb = ctx->n_boxes;
    m.grow = ctx->lists.grow;
    m.run_upto = list_few_rows(ctx);
    const unsigned blocks = (unsigned)std::min<int64_t>(912, m.run_upto / 8 + 1);
    if (ctx->adaptive) k_mark_dirty<1><<<blocks, 256, 0, ctx->stream>>>(m);
    else k_mark_dirty<0><<<blocks, 256, 0, ctx->stream>>>(m);
    SPH_LAUNCH(ctx, "neighbours of grown targets");
    return SPH_OK;
}

// budget: evaluations of a target; one that used them up gets results at its last h, in
// the last pass also one that needs another search
int run_density_lists(sph_ctx *ctx, sph_particles *parts, int pass, int budget, bool last_pass)
{
    DensityListArgs a{};
    a.s = sum_args(ctx, parts);
    a.s.run_if = pass > 0 ? ctx->counters + C_PASS + 4 * (pass - 1) : nullptr;
    a.s.ticket = ctx->counters + C_PASS + 4 * pass + 2;
    a.left = ctx->counters + C_PASS + 4 * pass;
    const int64_t cap = std::max<int64_t>(ctx->cap, 1);
    if (pass > 0) {
        a.rows = ctx->lists.rows + ((pass - 1) & 1) * cap;
        a.n_rows = ctx->counters + C_PASS + 4 * (pass - 1);
        a.s.split = 8;
    }
    a.left_rows = ctx->lists.rows + (pass & 1) * cap;
    a.grown_rows = ctx->lists.rows + 2 * cap;
    a.leaf_of = ctx->tree.leaf_of;
    a.nb = ctx->n_boxes;
    a.ids = ctx->ids;
    a.upred = ctx->upred;
    a.active = ctx->active;
    a.h = parts->h;
    a.h_lo = ctx->h_lo;
    a.h_hi = ctx->h_hi;
    a.rho = parts->rho;
    a.P = parts->P;
    a.c = parts->c;
    a.f = parts->f;
    a.divv = parts->divv;
    a.curl = parts->curl;
    a.n_ngb = parts->n_ngb;
    a.thermo4 = ctx->thermo4;
    a.ngb_hash = ctx->ngb_hash;
    a.n_ngb_target = ctx->p.n_ngb;
    a.h_tol = ctx->p.h_tol;
    a.gamma = ctx->p.gamma;
    a.grow = ctx->lists.grow;
    a.use_balsara = ctx->p.use_balsara;
    a.budget = budget;
    a.last_pass = last_pass ? 1 : 0;
    a.hold_cells = ctx->tree.device_sized ? 1 : 0;  // captured steps
    const bool hash = (ctx->p.flags & SPH_FLAG_NGB_HASH) != 0;
    const int g = list_grid(ctx, kSumThreads, kSumBlocks, a.s.split);
    cudaEvent_t end = nullptr;
    timer_begin(ctx, 0, &end);
    if (ctx->adaptive) {
        if (hash) k_density_l<1, true><<<g, kSumThreads, 0, ctx->stream>>>(a);
        else k_density_l<1, false><<<g, kSumThreads, 0, ctx->stream>>>(a);
    } else {
        if (hash) k_density_l<0, true><<<g, kSumThreads, 0, ctx->stream>>>(a);
        else k_density_l<0, false><<<g, kSumThreads, 0, ctx->stream>>>(a);
    }
    timer_end(ctx, end);
    SPH_LAUNCH(ctx, "density sums");
    ctx->st.density_passes++;
    return SPH_OK;
}

int run_force_lists(sph_ctx *ctx, sph_particles *parts)
{
    ForceListArgs a{};
    a.s = sum_args(ctx, parts);
    a.s.ticket = ctx->counters + C_FTICKET + 1;
    a.ax = parts->ax;
    a.ay = parts->ay;
    a.az = parts->az;
    a.dudt = parts->dudt;
    a.vsig = parts->vsig;
    a.fmask = ctx->bin_mode ? ctx->bin_active : nullptr;
    a.alpha = ctx->p.alpha_visc;
    const int g = list_grid(ctx, kSumThreads, kSumBlocks, a.s.split);
    cudaEvent_t end = nullptr;
    timer_begin(ctx, 1, &end);
    if (ctx->adaptive) k_force_l<1><<<g, kSumThreads, 0, ctx->stream>>>(a);
    else k_force_l<0><<<g, kSumThreads, 0, ctx->stream>>>(a);
    timer_end(ctx, end);
    SPH_LAUNCH(ctx, "force sums");
    ctx->st.force_passes++;
    return SPH_OK;
}

}  // namespace sph
