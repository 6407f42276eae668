// sph_gravity.cu -- the near field of the gravity of Theuns et al. 2015, Sec. 3.2
// (Eq. 3): the tree walk of that section ends in tasks in which a node meets the
// multipole of a distant node, and tasks in which all particles of one node
// interact with all particles of a nearby node, "implemented ... using the same
// task-based approach as used for SPH".  This file is the second kind on the SPH
// cell grid: every particle sums the Plummer-softened Eq. 3 over every other
// particle of its own cell and of the 26 adjacent cells (periodic, minimal image).
//
// Work decomposition: the SPH path's tiles (up to 32 targets of one cell), one per warp,
// handed out by the same ticket counter.  The 27 cells' particles form one source stream
// per tile; the lanes copy its positions in turn into shared memory (asynchronously, across
// cell boundaries, so that only the stream's end has pads), a chunk ahead of its use, and
// shift them into the tile's cell frame.  Lane 4 g + q sums, for the targets q, q + 4,
// q + 8, ... of the tile, over the sources g, g + 8, ...: no distance test, no pruning,
// straight-line FP32 arithmetic -- 3 adds, 3 FMAs for r^2, one MUFU reciprocal square
// root, 3 products, 1 add and 3 FMAs per pair, in packed instructions for two targets
// at a time (the last of an odd number by itself).  With the ~23 particles per cell that
// the smoothing length gives, one lane per target left 28 % of the lanes empty and spent a
// shared-memory read on every pair; steps of four targets leave 5 % empty and read a
// source once for all of a lane's targets.  Bound by issue and by the FP32 pipe, on which
// a packed instruction takes two cycles.  2 M particles on a lattice, 627 pairs each: 1.04
// -> 0.91 ms.  (Not kept, same field: two sources packed instead of two targets, 0.96 ms, of
// which every position needs a second register; eight lanes of targets, 0.95 to 1.04 ms; all
// scalar, 0.95 ms; the whole tile instead of the inner loop once per number of targets,
// 1.05 to 1.18 ms, waiting for instructions.)
// Up to 128 terms are summed plainly in each of a target's 8 accumulators, which are
// then added in a fixed order, and the totals with Kahan compensation; the summation
// order of a target never depends on which warp runs its tile.
#include <algorithm>

#include "sph_internal.cuh"

namespace sph {

constexpr int kGravThreads = 128;
constexpr int kGravBlocks = 4;    // resident blocks per SM the kernel is compiled for
constexpr int kGravStage = 128;  // sources staged at a time
constexpr int kGravFlush = 128;  // terms per accumulator that are summed plainly
static_assert(kGravFlush % (kGravStage / 8) == 0, "whole chunks between flushes");
// staging pads: far away (r^2 overflows to +inf, so rsqrt gives 0) and massless
constexpr float kGravFar = 1e30f;
// smallest squared separation (box units) an unsoftened pair contributes at, and the
// smallest eps^2 the softened kernel runs with: FP32 positions relative to a cell
// centre cannot resolve separations near 1e-15 anyway
constexpr float kGravMinR2 = 1e-30f;

struct GravArgs {
    const float4 *__restrict__ pos4;  // {x, y, z} relative to the cell centre, h
    const float4 *__restrict__ vel4;  // {vx, vy, vz, m}
    const int *__restrict__ cell_start;
    const int4 *__restrict__ tiles;
    const int *__restrict__ n_tiles;
    const BoxDev *__restrict__ boxes;
    float *ax, *ay, *az, *phi;  // caller's outputs (phi may be null)
    unsigned long long *counters;
    float G, eps2;
};

__device__ __forceinline__ int wrapg(int j, int nc) { return j < 0 ? j + nc : (j >= nc ? j - nc : j); }

// 1/sqrt(x) as the one MUFU instruction, with denormal inputs and results flushed
// to zero: the squared separations here are at least eps^2 >= kGravMinR2 (softened)
// or, unsoftened, taken only above kGravMinR2 -- never denormal -- so nothing else is
// needed around it; rsqrt(+inf) = 0 keeps the staging pads inert.
__device__ __forceinline__ float rsqrt_mufu(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct GravWarp {  // a warp's shared memory
    float4 xy[kGravStage], zm[kGravStage];  // staged sources, every value twice
    float4 raw[kGravStage];  // copies in flight: positions and masses of the next chunk
    float raw_m[kGravStage];
    float4 cell[32];         // the cells with particles: offset of the frame, slot minus stream position
    int end[32];             // where a cell's particles end in the stream
    float2 sum[4][32];       // compensated sums of the tile's targets {sum, compensation}
};

// stream positions q0 + 32 r + lane (r < 4) on their way to w.raw; returns their cells in
// four bytes.  end: where the lane's cell ends (cells without particles left out)
__device__ __forceinline__ unsigned gravity_fetch(const GravArgs &a, GravWarp &w, int q0, int total, int end)
{
    const int lane = threadIdx.x & 31;
    unsigned cells = 0u;
#pragma unroll
    for (int r = 0; r < kGravStage / 32; ++r) {
        const int base = q0 + 32 * r, k = 32 * r + lane;
        if (base >= total) break;
        // cells that end at or before the position
        const unsigned in = __reduce_or_sync(kFull, end > base && end < base + 32 ? 1u << (end - base) : 0u);
        const int c = __popc(__ballot_sync(kFull, end <= base)) + __popc(in & ((2u << lane) - 1u));
        if (base + lane >= total) continue;
        const int j = __float_as_int(w.cell[c].w) + base + lane;
        cells |= (unsigned)c << (8 * r);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(w.raw + k)),
                     "l"(a.pos4 + j));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(w.raw_m + k)),
                     "l"(&a.vel4[j].w));
    }
    return cells;
}

struct GravSums {  // a lane's 8 targets in 4 pairs: negated positions, terms of the current batch
    float2 px[4], py[4], pz[4];
    float2 x[4], y[4], z[4], p[4];
};

// The staged sources' terms for the first NT targets.  SOFT: eps^2 >= kGravMinR2 --
// every staged source enters the sums, and the target's own term (exactly m_i / eps: its
// separation is exactly 0) is taken out once at the end; otherwise pairs closer than
// sqrt(kGravMinR2) (the target itself, coincident particles) are dropped by their r^2.
template <int NT, bool SOFT>
__device__ __forceinline__ void gravity_terms(GravSums &s, const GravWarp &w, int steps, float eps2)
{
    constexpr int NP = NT / 2, N1 = NP & 3;  // pairs of targets; an odd one by itself
    const int g = (threadIdx.x & 31) >> 2;
    const float2 e2 = make_float2(eps2, eps2);
#pragma unroll 2
    for (int k = 0; k < steps; ++k) {
        const float4 xy = w.xy[8 * k + g], zm = w.zm[8 * k + g];
        const float2 x = make_float2(xy.x, xy.y), y = make_float2(xy.z, xy.w), z = make_float2(zm.x, zm.y),
                     m = make_float2(zm.z, zm.w);
#pragma unroll
        for (int t = 0; t < NP; ++t) {
            const float2 dx = __fadd2_rn(x, s.px[t]), dy = __fadd2_rn(y, s.py[t]), dz = __fadd2_rn(z, s.pz[t]);
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
            float2 inv = make_float2(rsqrt_mufu(r2.x), rsqrt_mufu(r2.y));
            if (!SOFT) {
                inv.x = r2.x > kGravMinR2 ? inv.x : 0.f;
                inv.y = r2.y > kGravMinR2 ? inv.y : 0.f;
            }
            const float2 mi = __fmul2_rn(m, inv), mi3 = __fmul2_rn(__fmul2_rn(mi, inv), inv);
            s.p[t] = __fadd2_rn(s.p[t], mi);
            s.x[t] = __ffma2_rn(mi3, dx, s.x[t]);
            s.y[t] = __ffma2_rn(mi3, dy, s.y[t]);
            s.z[t] = __ffma2_rn(mi3, dz, s.z[t]);
        }
        if (NT & 1) {
            const float dx = x.x + s.px[N1].x, dy = y.x + s.py[N1].x, dz = z.x + s.pz[N1].x;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
            float inv = rsqrt_mufu(r2);
            if (!SOFT) inv = r2 > kGravMinR2 ? inv : 0.f;
            const float mi = m.x * inv, mi3 = mi * inv * inv;
            s.p[N1].x += mi;
            s.x[N1].x = fmaf(mi3, dx, s.x[N1].x);
            s.y[N1].x = fmaf(mi3, dy, s.y[N1].x);
            s.z[N1].x = fmaf(mi3, dz, s.z[N1].x);
        }
    }
}

template <bool SOFT>
__global__ void __launch_bounds__(kGravThreads, kGravBlocks) k_gravity(GravArgs a)
{
    __shared__ GravWarp warps[kGravThreads / 32];
    const int lane = threadIdx.x & 31, tl = lane & 3;
    GravWarp &w = warps[threadIdx.x >> 5];
    const int comp = lane >> 3;  // component this lane totals (x, y, z, phi); see below
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const int ntiles = *a.n_tiles;
    unsigned long long acc_pairs = 0ull;
    unsigned *ticket = reinterpret_cast<unsigned *>(a.counters + C_TICKET);
    unsigned tk = 0u;
    if (lane == 0) tk = atomicAdd(ticket, 1u);
    for (int t = gw, t_after = 0; t < ntiles; t = t_after) {
        t_after = nw + (int)__shfl_sync(kFull, tk, 0);
        if (lane == 0 && t_after < ntiles) tk = atomicAdd(ticket, 1u);
        const int4 tile = a.tiles[t];
        const BoxDev bx = a.boxes[tile.w];
        const int nc = bx.nc;
        const int ca = tile.x - bx.cell_off;
        const int ix = ca % nc, iy = (ca / nc) % nc, iz = ca / (nc * nc);
        // The sources of a tile as one stream: the 27 cells in order o = 0..26 (cell o
        // at offset (o % 3 - 1, (o / 3) % 3 - 1, o / 9 - 1), o = 13 the tile's own),
        // each cell's particles in slot order.
        int first = 0, n = 0;
        if (lane < 27) {
            const int cb = bx.cell_off + (wrapg(iz + lane / 9 - 1, nc) * nc + wrapg(iy + (lane / 3) % 3 - 1, nc)) * nc +
                           wrapg(ix + lane % 3 - 1, nc);
            first = a.cell_start[cb];
            n = a.cell_start[cb + 1] - first;
        }
        int end = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(kFull, end, d);
            if (lane >= d) end += v;
        }
        const int total = __shfl_sync(kFull, end, 31);
        __syncwarp();
        w.end[lane] = total;
        w.sum[0][lane] = w.sum[1][lane] = w.sum[2][lane] = w.sum[3][lane] = make_float2(0.f, 0.f);
        __syncwarp();
        const unsigned some = __ballot_sync(kFull, n > 0);
        if (n > 0) {
            const int k = __popc(some & ((1u << lane) - 1u));
            w.end[k] = end;
            w.cell[k] = make_float4((float)(lane % 3 - 1) * bx.L32, (float)((lane / 3) % 3 - 1) * bx.L32,
                                    (float)(lane / 9 - 1) * bx.L32, __int_as_float(first - (end - n)));
        }
        __syncwarp();
        end = w.end[lane];
        int terms = 0;
        unsigned cells = gravity_fetch(a, w, 0, total, end);
        GravSums s;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int k0 = tl + 8 * k, k1 = k0 + 4;
            const float4 p = k0 < tile.z ? a.pos4[tile.y + k0] : make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 q = k1 < tile.z ? a.pos4[tile.y + k1] : make_float4(0.f, 0.f, 0.f, 0.f);
            s.px[k] = make_float2(-p.x, -q.x);
            s.py[k] = make_float2(-p.y, -q.y);
            s.pz[k] = make_float2(-p.z, -q.z);
            s.x[k] = s.y[k] = s.z[k] = s.p[k] = make_float2(0.f, 0.f);
        }
        for (int q0 = 0; q0 < total; q0 += kGravStage) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();  // the chunk before has been read
#pragma unroll
            for (int r = 0; r < kGravStage / 32; ++r) {
                const int k = 32 * r + lane;
                float4 v = make_float4(kGravFar, kGravFar, kGravFar, 0.f);
                if (q0 + k < total) {  // each lane reads what it copied itself
                    const float4 p = w.raw[k], o = w.cell[(cells >> (8 * r)) & 31u];
                    v = make_float4(p.x + o.x, p.y + o.y, p.z + o.z, w.raw_m[k]);
                }
                w.xy[k] = make_float4(v.x, v.x, v.y, v.y);
                w.zm[k] = make_float4(v.z, v.z, v.w, v.w);
            }
            __syncwarp();
            cells = gravity_fetch(a, w, q0 + kGravStage, total, end);
            const int steps = min((total - q0 + 7) / 8, kGravStage / 8);
            switch ((tile.z + 3) >> 2) {
            case 1: gravity_terms<1, SOFT>(s, w, steps, a.eps2); break;
            case 2: gravity_terms<2, SOFT>(s, w, steps, a.eps2); break;
            case 3: gravity_terms<3, SOFT>(s, w, steps, a.eps2); break;
            case 4: gravity_terms<4, SOFT>(s, w, steps, a.eps2); break;
            case 5: gravity_terms<5, SOFT>(s, w, steps, a.eps2); break;
            case 6: gravity_terms<6, SOFT>(s, w, steps, a.eps2); break;
            case 7: gravity_terms<7, SOFT>(s, w, steps, a.eps2); break;
            default: gravity_terms<8, SOFT>(s, w, steps, a.eps2); break;
            }
            terms += steps;
            if (terms < kGravFlush && q0 + kGravStage < total) continue;
            terms = 0;
            // the 8 lanes' sums of a target: after the exchanges lane bits 4 and 3 select the
            // component it has the total of
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (4 * k >= tile.z) break;
                const float x = k & 1 ? s.x[k / 2].y : s.x[k / 2].x, y = k & 1 ? s.y[k / 2].y : s.y[k / 2].x;
                const float z = k & 1 ? s.z[k / 2].y : s.z[k / 2].x, p = k & 1 ? s.p[k / 2].y : s.p[k / 2].x;
                const bool hi = lane & 16, odd = lane & 8;
                const float u0 = (hi ? z : x) + __shfl_xor_sync(kFull, hi ? x : z, 16);
                const float u1 = (hi ? p : y) + __shfl_xor_sync(kFull, hi ? y : p, 16);
                float v = (odd ? u1 : u0) + __shfl_xor_sync(kFull, odd ? u0 : u1, 8);
                v += __shfl_xor_sync(kFull, v, 4);
                if (!(lane & 4)) {
                    float2 c = w.sum[comp][tl + 4 * k];
                    kahan_add(c.x, c.y, v);
                    w.sum[comp][tl + 4 * k] = c;
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) s.x[k] = s.y[k] = s.z[k] = s.p[k] = make_float2(0.f, 0.f);
        }
        acc_pairs += (unsigned long long)(total - 1) * (unsigned)tile.z;  // warp-uniform
        __syncwarp();
        if (lane >= tile.z) continue;
        const int i = tile.y + lane;
        float2 c = w.sum[3][lane];
        // the target's own term: zero separation, so exactly m_i rsqrt(eps^2) in phi
        // and nothing in a
        if (SOFT) kahan_add(c.x, c.y, -(__ldg(&a.vel4[i].w) * rsqrt_mufu(a.eps2)));
        // a_i = -G sum m_j (r_i - r_j) / (r^2 + eps^2)^(3/2): the sums above run over
        // r_j - r_i, hence +G
        a.ax[i] = a.G * (w.sum[0][lane].x - w.sum[0][lane].y);
        a.ay[i] = a.G * (w.sum[1][lane].x - w.sum[1][lane].y);
        a.az[i] = a.G * (w.sum[2][lane].x - w.sum[2][lane].y);
        if (a.phi) a.phi[i] = -a.G * (c.x - c.y);
    }
    if (lane == 0 && acc_pairs) atomicAdd(a.counters + C_GPAIRS, acc_pairs);
}

template <bool SOFT>
static int launch_gravity(sph_ctx *ctx, const GravArgs &a)
{
    int &blocks_per_sm = ctx->grav_blocks[SOFT];  // occupancy of this instantiation
    if (blocks_per_sm == 0) {
        SPH_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, k_gravity<SOFT>, kGravThreads,
                                                                    0));
        blocks_per_sm = std::max(blocks_per_sm, 1);
    }
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    if (sms <= 0) sms = 148;
    // persistent grid: every resident warp, no more than the tile groups need
    const int64_t want = ((int64_t)ctx->n / ctx->tile_w + ctx->grid.n_cells) / (kGravThreads / 32) + 1;
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * blocks_per_sm, want));
    k_gravity<SOFT><<<g, kGravThreads, 0, ctx->stream>>>(a);
    return SPH_OK;
}

int run_gravity_pass(sph_ctx *ctx, double G, double eps, float *ax, float *ay, float *az, float *phi)
{
    GravArgs a{};
    a.pos4 = ctx->pos4;
    a.vel4 = ctx->vel4;
    a.cell_start = ctx->cell_start;
    a.tiles = ctx->tiles;
    a.n_tiles = ctx->n_tiles;
    a.boxes = ctx->d_boxes;
    a.ax = ax;
    a.ay = ay;
    a.az = az;
    a.phi = phi;
    a.counters = ctx->counters;
    a.G = (float)G;
    a.eps2 = (float)(eps * eps);
    SPH_CUDA(ctx, cudaMemsetAsync(ctx->counters + C_TICKET, 0, sizeof(unsigned long long), ctx->stream));
    cudaEvent_t end = nullptr;
    timer_begin(ctx, 3, &end);
    const bool soft = a.eps2 >= kGravMinR2;
    const int rc = soft ? launch_gravity<true>(ctx, a) : launch_gravity<false>(ctx, a);
    if (rc) return rc;
    timer_end(ctx, end);
    SPH_LAUNCH(ctx, "gravity kernel");
    ctx->st.grav_passes++;
    return SPH_OK;
}

}  // namespace sph
