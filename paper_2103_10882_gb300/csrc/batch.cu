// Batched sweep: many independent uniform periodic simulations of uneven size
// (the paper's (density ratio, Ga) parameter study, Sec. 5) advanced together.
// The coupled step (Algorithm 1) of all simulations is two launches:
//   k_batch_step   stream-collide over a flat list of runs; among its CTAs
//                  those of the cells next to the spheres (CLI links,
//                  momentum exchange), the last of each simulation running
//                  its particle update
//   k_batch_remap  flags, refill and boundary cells
// Two steps are captured in a CUDA graph and replayed.  The stream-collide
// CTA shape is chosen by timing the candidates on the batch itself
// (autotuner).
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "batch.h"
#include "physics.cuh"

namespace lbmp {
namespace {

struct SimDev {
    GridDesc G;
    long long pop_off;   // element offset of the simulation in each population pool
    long long flag_off;  // byte offset in each flag pool
    FastDiv by_edge;     // division by the edge
    int seg_off, nseg;   // segments of the box: boundary cells and their number per 256 box cells
    int bnd_off, bnd_n;  // boundary CTAs of the simulation (and their force partials)
    BoxDesc box;
    CollideParams<double> P;   // FP64: the collision's parameters; else its rates are rounded from here
    long long hist_off;  // records
};

constexpr int BW = 256;   // threads of a CTA
constexpr int BND_SEGS = 2;     // segments per boundary CTA of a large batch (fewer, fuller CTAs: the fixed cost dominates)
constexpr int RECORDS = 32;      // particle records read back at once (a copy of one record takes as long, 12 us)
constexpr int BND_PARTS = 4;    // CTAs that share a segment's cells in a small batch (there the chain of a warp's cells is the step)
// Cell flags: fluid, solid (centre inside the sphere), fluid with a solid
// D3Q19 neighbour (updated by the boundary CTAs instead of the bulk ones).
constexpr uint8_t FLAG_FLUID = 0, FLAG_SOLID = 1, FLAG_BOUNDARY = 2;

template <typename S>
__host__ __device__ __forceinline__ CollideParams<typename Store<S>::A> sim_params(const SimDev& D, typename Store<S>::A scale,
                                               typename Store<S>::A inv) {
    CollideParams<typename Store<S>::A> p;
    if constexpr (sizeof(S) == 8) return D.P;
    p.sp = (typename Store<S>::A)D.P.sp;
    p.sm = (typename Store<S>::A)D.P.sm;
    p.db = (typename Store<S>::A)D.P.db;
    p.F[0] = p.F[1] = p.F[2] = 0;
    p.forced = 0;
    p.scale = scale;
    p.inv_scale = inv;
    return p;
}

// Bulk CTA: its simulation, first item, and what the stream-collide needs of the simulation, so that its pulls wait for
// one load and not for a chain of two (FP64 takes the collision's parameters from SimDev).
struct alignas(16) BulkRun {
    long long pop_off;   // also 19 times the flag offset
    int sim, item, edge;
    FastDiv by_edge;
    float sp, sm, db;
};

// One step of all simulations.
template <typename S>
struct BatchArgs {
    using A = typename Store<S>::A;
    const S* src;
    S* dst;
    const uint8_t* flags;
    const BulkRun* runs;
    const SimDev* sims;
    A scale, inv;
    int* status;
    int bblocks, bshift;   // boundary CTAs: every 2^bshift-th CTA from the first on
    int segs, parts;       // segments of a boundary CTA, CTAs that share them
    const int* seg;
    const int* seg_count;
    const int* bnd_sim;
    ParticleState* ps;
    PFrames* frames;
    int cli, hist_cap;
    double* partials;
    int* done;
    double* history;
};

// ------------------------------------------------------------ stream-collide
// Item i of a simulation: with ZC = 1 cell i, with ZC = 2 the two cells i mod e^2 of the planes 2 (i / e^2) and the
// next, one after the other.  Items are taken in memory order.
template <typename S, int ZC>
__device__ __forceinline__ void batch_bulk(const BatchArgs<S>& T, const BulkRun& R, int item) {
    using A = typename Store<S>::A;
    CollideParams<A> P;
    if constexpr (sizeof(S) == 8) {
        P = T.sims[R.sim].P;
    } else {
        P.sp = R.sp;
        P.sm = R.sm;
        P.db = R.db;
        P.scale = T.scale;
        P.inv_scale = T.inv;
    }
    const int e = R.edge;
    const unsigned row = R.by_edge.div((unsigned)item), plane = R.by_edge.div(row);
    const int x = item - (int)row * e, y = (int)row - (int)plane * e;
    const size_t n = (size_t)e * (size_t)e * (size_t)e;
    const S* s0 = T.src + R.pop_off;
    S* d0 = T.dst + R.pop_off;
    const uint8_t* fl = T.flags + R.pop_off / 19;
    const int xs[3] = {x + 1 < e ? x + 1 : 0, x, x > 0 ? x - 1 : e - 1};
    const int ys[3] = {y + 1 < e ? y + 1 : 0, y, y > 0 ? y - 1 : e - 1};
#pragma unroll
    for (int k = 0; k < ZC; ++k) {
        const int z = (int)plane * ZC + k;
        const int zs[3] = {z + 1 < e ? z + 1 : 0, z, z > 0 ? z - 1 : e - 1};
        const size_t cell = (size_t)(x + e * (y + e * z));
        const uint8_t f = fl[cell];
        A g[19];
#pragma unroll
        for (int q = 0; q < 19; ++q)
            g[q] = Store<S>::fetch(s0 + (size_t)q * n + (size_t)(xs[cx(q) + 1] + e * (ys[cy(q) + 1] + e * zs[cz(q) + 1])),
                                   P.inv_scale);
        if (f != FLAG_FLUID) {   // solid: stored as zero; else a boundary CTA's cell
            if (f == FLAG_SOLID)
#pragma unroll
                for (int q = 0; q < 19; ++q) Store<S>::store(d0 + (size_t)q * n + cell, A(0), P.scale);
            continue;
        }
        trt_collide<A, false>(g, P, T.status);
#pragma unroll
        for (int q = 0; q < 19; ++q) Store<S>::store(d0 + (size_t)q * n + cell, g[q], P.scale);
    }
}

// ----------------------------------------------------------------- boundary
// Boundary cells of every simulation (flag 2), from the segments the remap
// wrote: boundary CTA b belongs to simulation bnd_sim[b] and takes some
// segments of its box, or a part of one's cells, its warps the cells in
// turn, lane q handling population q (CLI links, geometry in the population
// arithmetic, FP64 force partials), with a cooperative collision.  All loads of a link are issued
// at once, its geometry formed meanwhile.  The last of a simulation's CTAs
// to finish runs its particle update (Algorithm 1) and forms the frames of
// the moved sphere, which the next kernels read.
template <typename S>
__device__ __forceinline__ void batch_boundary(const BatchArgs<S>& T, int bid) {
    using A = typename Store<S>::A;
    __shared__ LinkFrame<A> Fr;
    __shared__ double sX[3];
    __shared__ int upto[BND_SEGS];   // cells of the CTA's segments up to and with each
    const int sim = T.bnd_sim[bid];
    const SimDev& D = T.sims[sim];
    const GridDesc& G = D.G;
    const int n3[3] = {G.nx, G.ny, G.nz};
    const int per3[3] = {1, 1, 1};
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int local = bid - D.bnd_off, seg0 = local / T.parts * T.segs, part = local % T.parts;
    if (threadIdx.x == 0) Fr = pframe_link<A>(T.frames[sim]);   // formed by the last particle update
    if (threadIdx.x >= 32 && threadIdx.x < 35) sX[threadIdx.x - 32] = T.ps[sim].x[threadIdx.x - 32];
    if (threadIdx.x == 64) {
        int t = 0;
#pragma unroll
        for (int k = 0; k < BND_SEGS; ++k) {
            t += (k < T.segs && seg0 + k < D.nseg) ? T.seg_count[D.seg_off + seg0 + k] : 0;
            upto[k] = t;
        }
    }
    __syncthreads();
    const CollideParams<A> P = sim_params<S>(D, T.scale, T.inv);
    const S* s0 = T.src + D.pop_off;
    S* d0 = T.dst + D.pop_off;
    const uint8_t* fl = T.flags + D.flag_off;
    const size_t n = (size_t)G.n;
    const int q = lane < 19 ? lane : 0, k = opp(q);
    const int cq[3] = {cx(q), cy(q), cz(q)};
    LinkSums<A> acc;
    // a warp's last cell is stored after the hand-off: the hand-off's release waits for the stores before it
    A kept = A(0);
    S* kept_at = nullptr;
    for (int j = part * (BW / 32) + wib; j < upto[BND_SEGS - 1]; j += T.parts * (BW / 32)) {
        if (kept_at) Store<S>::store(kept_at, kept, P.scale);
        int g = 0;
        while (upto[g] <= j) ++g;
        const int cell = T.seg[(size_t)(D.seg_off + seg0 + g) * SEG + (j - (g > 0 ? upto[g - 1] : 0))];
        const unsigned row = D.by_edge.div((unsigned)cell), plane = D.by_edge.div(row);
        const int xyz[3] = {cell - (int)row * G.nx, (int)row - (int)plane * G.ny, (int)plane};
        A gq = A(0);
        if (lane < 19) {
            int s3[3], f3[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                s3[a] = src_coord(xyz[a], cq[a], n3[a], 1);
                f3[a] = src_coord(xyz[a], -cq[a], n3[a], 1);
            }
            const int sidx = s3[0] + G.nx * (s3[1] + G.ny * s3[2]), far = f3[0] + G.nx * (f3[1] + G.ny * f3[2]);
            const uint8_t fsrc = fl[sidx], ffar = fl[far];
            const A pull = Store<S>::fetch(s0 + (size_t)q * n + sidx, P.inv_scale);
            const A gt_k = Store<S>::fetch(s0 + (size_t)k * n + cell, P.inv_scale);
            const A gt_q = Store<S>::fetch(s0 + (size_t)q * n + cell, P.inv_scale);
            const A vfar = Store<S>::fetch(s0 + (size_t)k * n + far, P.inv_scale);
            A d[3];
            int pu[3];
            Fr.offset(xyz, n3, per3, d, pu);
            CliGeometry<A> L = cli_geometry<A>(q, d, T.cli != 0, Fr);   // as if the far cell were fluid
            gq = pull;
            if (q != 0 && fsrc == FLAG_SOLID) {
                const bool far_ok = ffar != FLAG_SOLID;
                if (T.cli && !far_ok) L = cli_geometry<A>(q, d, false, Fr);
                A flk[3], tl3[3];
                gq = cli_apply<A>(q, L, gt_k, gt_q, far_ok ? vfar : A(0), flk, tl3);
                acc.add(k, pu, flk, tl3);
            }
        }
        kept = warp_trt_collide<A, false>(gq, lane, P, T.status);
        if (lane < 19) kept_at = d0 + (size_t)lane * n + cell;
    }
    block_link_sums<BW>(acc, sX, T.partials + (size_t)D.bnd_off * 6 + local, D.bnd_n);
    const bool last = last_block_done(T.done + sim, D.bnd_n);
    if (kept_at) Store<S>::store(kept_at, kept, P.scale);
    if (last)
        particle_block_update<BW>(
            T.ps + sim, T.partials + (size_t)D.bnd_off * 6, D.bnd_n, G, T.history + (size_t)D.hist_off * 15, T.hist_cap,
            T.status, T.frames[sim].inv,
            [&](const ParticleState& Q, int a, int part) { pframes_axis(T.frames + sim, Q, n3, D.box, a, part); });
}

// One launch, bound by HBM in FP32 and FP16 and by the FP64 pipe in FP64.  As two kernels on two streams the boundary
// CTAs, launched beside the bulk kernel, filled the SMs first and held it back: 566 us a step for the sweep's 64 boxes,
// whose bulk kernel takes 500 alone, now 544 (FP16 467 to 455, 16 boxes in FP64 1643 to 1565).  Spread among the first
// half of the bulk CTAs they take few slots at a time.  A box by itself and four small ones are bound by the chain
// from a boundary CTA's first load to the remap's last store: 49 to 34 and 34 to 23 us, most of it from BND_PARTS and
// from the bulk CTA's one load before its pulls.
// ZC cells per thread along z, CTAS resident CTAs per SM asked of the compiler: the autotuner's choice, timed on the bulk
// CTAs alone (boundary CTAs would advance the spheres).  Neither touches the arithmetic, so the results do not depend on
// it.
template <typename S, int ZC, int CTAS>
__global__ void __launch_bounds__(BW, CTAS) k_batch_step(const __grid_constant__ BatchArgs<S> T) {
    pdl_wait();
    const unsigned before = min((unsigned)T.bblocks, (blockIdx.x + (1u << T.bshift) - 1u) >> T.bshift);
    if ((blockIdx.x & ((1u << T.bshift) - 1u)) == 0u && (blockIdx.x >> T.bshift) < (unsigned)T.bblocks) {
        batch_boundary<S>(T, (int)(blockIdx.x >> T.bshift));
        return;
    }
    const BulkRun R = T.runs[blockIdx.x - before];
    batch_bulk<S, ZC>(T, R, R.item + (int)threadIdx.x);
}

// -------------------------------------------------------------------- remap
// Refill of the uncovered cell (i, j, k) = flat index c of one simulation by
// the whole warp (Sec. 2.3): lane q = 1..18 takes the periodic neighbour
// (i, j, k) + c_q, counted when it is fluid before (fc) and after (the ball
// predicate) the move, with its density 1 + sum_p g_p and momentum
// sum_p c_p g_p (for Grad's strain rate from the face neighbours).  The mean
// density and the rigid-body velocity give the equilibrium, plus Grad's
// term when grad is set; lane q < 19 writes population q.  Every lane calls
// it with the same cell.
template <typename S>
__device__ __forceinline__ void batch_refill_warp(S* p0, const uint8_t* fc, const GridDesc& G,
                                                  const int n3[3], const BoxFrame& F, const ParticleState& P, int i,
                                                  int j, int k, size_t c, typename Store<S>::A scale,
                                                  typename Store<S>::A inv, int grad, double sp) {
    using A = typename Store<S>::A;
    const int lane = threadIdx.x & 31;
    const size_t n = (size_t)G.n;
    bool ok = false;
    A r = A(0), mo[3] = {A(0), A(0), A(0)};
    if (lane >= 1 && lane < 19) {
        int v[3] = {i + cx(lane), j + cy(lane), k + cz(lane)};
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = v[a] < 0 ? v[a] + n3[a] : (v[a] >= n3[a] ? v[a] - n3[a] : v[a]);
        if (!ball_flag(v, n3, G.periodic, F, P)) {
            const size_t y = (size_t)v[0] + (size_t)G.nx * ((size_t)v[1] + (size_t)G.ny * (size_t)v[2]);
            {   // the populations are loaded beside the flag (not after it): a solid neighbour's are dropped
                ok = fc[y] != FLAG_SOLID;
                A gp[19];
#pragma unroll
                for (int q2 = 0; q2 < 19; ++q2) gp[q2] = Store<S>::fetch(p0 + (size_t)q2 * n + y, inv);
                r = A(1);
#pragma unroll
                for (int q2 = 0; q2 < 19; ++q2) r += gp[q2];
                if (grad) {
#pragma unroll
                    for (int q2 = 1; q2 < 19; ++q2) {
                        if (cx(q2)) mo[0] += cx(q2) > 0 ? gp[q2] : -gp[q2];
                        if (cy(q2)) mo[1] += cy(q2) > 0 ? gp[q2] : -gp[q2];
                        if (cz(q2)) mo[2] += cz(q2) > 0 ? gp[q2] : -gp[q2];
                    }
                }
            }
        }
    }
    const unsigned okm = __ballot_sync(0xffffffffu, ok);
    A rs = ok ? r : A(0);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, off);
    const int cnt = __popc(okm);
    const A rho = cnt > 0 ? rs / A(cnt) : A(1);
    const double d[3] = {wrap_diff((i + 0.5) - P.x[0], G.nx, 1), wrap_diff((j + 0.5) - P.x[1], G.ny, 1),
                         wrap_diff((k + 0.5) - P.x[2], G.nz, 1)};
    const A u[3] = {A(P.u[0] + (P.w[1] * d[2] - P.w[2] * d[1])), A(P.u[1] + (P.w[2] * d[0] - P.w[0] * d[2])),
                    A(P.u[2] + (P.w[0] * d[1] - P.w[1] * d[0]))};
    const A uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    A Sr[6] = {A(0), A(0), A(0), A(0), A(0), A(0)};
    A gcoef = A(0);
    if (grad) {   // face neighbour q = 1 + 2 a (+1 for -e_a), fluid before and after the move
        gcoef = A(-3.0 * (1.0 - sp) / sp);
        auto nb = [&](int a, int sgn, A uo[3]) {
            const int q = 1 + 2 * a + (sgn > 0 ? 0 : 1);
#pragma unroll
            for (int m = 0; m < 3; ++m) uo[m] = __shfl_sync(0xffffffffu, mo[m], q);
            return ((okm >> q) & 1u) != 0;
        };
        refill_strain<A>(nb, u, Sr);
    }
    if (lane < 19) {
        const int q = lane;
        const A cu = A(cx(q)) * u[0] + A(cy(q)) * u[1] + A(cz(q)) * u[2];
        A e = wgt<A>(q) * ((rho - A(1)) + A(3) * cu + A(4.5) * cu * cu - A(1.5) * uu);
        if (grad) e += grad_term<A>(q, Sr, gcoef);
        Store<S>::store(p0 + (size_t)q * n + c, e, scale);
    }
}

// Remap of Sec. 2.3 over each simulation's box, a block per segment (seg_sim names its simulation): the new flag of
// every cell (the exact ball predicate; 2 for fluid cells with a solid neighbour, evaluated from the same predicate),
// covered cells zeroed, the boundary cells into the segment; uncovered cells are listed in shared memory and refilled
// by the block's warps in turn (batch_refill_warp). 
template <typename S>
__global__ void __launch_bounds__(BW)
    k_batch_remap(S* pops, const uint8_t* fcur, uint8_t* fnext, const SimDev* sims, const int* seg_sim,
                  const ParticleState* ps, const PFrames* frames, typename Store<S>::A scale, typename Store<S>::A inv,
                  int* seg, int* seg_count, int grad) {
    using A = typename Store<S>::A;
    static_assert(BW == SEG, "a block is a segment");
    __shared__ BoxFrame F;
    __shared__ int s_n;
    __shared__ int s_g[3][BW];   // uncovered cells
    pdl_wait();
    const int sim = seg_sim[blockIdx.x];
    const SimDev& D = sims[sim];
    const GridDesc& G = D.G;
    const int n3[3] = {G.nx, G.ny, G.nz};
    if (threadIdx.x == 0) {
        F = frames[sim].bf;   // formed by the particle update that moved the sphere
        s_n = 0;
    }
    __syncthreads();
    const int t = ((int)blockIdx.x - D.seg_off) * BW + threadIdx.x;
    const ParticleState& P = ps[sim];
    const uint8_t* fc = fcur + D.flag_off;
    uint8_t* fn = fnext + D.flag_off;
    S* p0 = pops + D.pop_off;
    const size_t n = (size_t)G.n;
    bool is_b = false;
    int c = 0, p[3] = {0, 0, 0};
    // periodic: box_cell fails only for a corrupt centre
    if (t < D.box.cells && box_cell(t, n3, G.periodic, D.box, F, p)) {
        c = p[0] + G.nx * (p[1] + G.ny * p[2]);
        const bool was_solid = fc[c] == FLAG_SOLID;
        bool any_nb = false;
        const bool solid = ball_flag_and_neighbours(p, n3, G.periodic, F, P, &any_nb);
        is_b = !solid && any_nb;
        fn[c] = solid ? FLAG_SOLID : (is_b ? FLAG_BOUNDARY : FLAG_FLUID);
        if (solid && !was_solid) {   // (the bulk kernel stores the cells that were solid before as zero)
#pragma unroll
            for (int q = 0; q < 19; ++q) Store<S>::store(p0 + (size_t)q * n + c, A(0), scale);
        } else if (!solid && was_solid) {
            const int k = atomicAdd(&s_n, 1);
#pragma unroll
            for (int a = 0; a < 3; ++a) s_g[a][k] = p[a];
        }
    }
    write_segment(is_b, c, (int)blockIdx.x, seg, seg_count);   // its barrier also completes the shared list
    for (int k = (int)(threadIdx.x >> 5); k < s_n; k += BW / 32) {
        const int i = s_g[0][k], j = s_g[1][k], m = s_g[2][k];
        batch_refill_warp<S>(p0, fc, G, n3, F, P, i, j, m, (size_t)(i + G.nx * (j + G.ny * m)), scale, inv, grad, D.P.sp);
    }
}

// Frames of every simulation's start position (one block of 128 threads each).
__global__ void k_batch_frames(const SimDev* __restrict__ sims, const ParticleState* __restrict__ ps,
                               PFrames* __restrict__ frames) {
    const SimDev& D = sims[blockIdx.x];
    const int n3[3] = {D.G.nx, D.G.ny, D.G.nz};
    pframes_form(frames + blockIdx.x, ps[blockIdx.x], n3, D.G.periodic, D.box);
}

__global__ void k_batch_flags_full(uint8_t* __restrict__ f0, uint8_t* __restrict__ f1, const SimDev* __restrict__ sims,
                                   const ParticleState* __restrict__ ps, const long long* __restrict__ cell_off,
                                   int nsims, long long total) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= total) return;
    int sim = 0;
    while (sim + 1 < nsims && cell_off[sim + 1] <= g) ++sim;
    const SimDev& D = sims[sim];
    const int c = (int)(g - cell_off[sim]);
    const int e = D.G.nx;
    const uint8_t v = inside_ball(c % e, (c / e) % e, c / (e * e), D.G, ps[sim]) ? 1 : 0;
    f0[D.flag_off + c] = v;
    f1[D.flag_off + c] = v;
}

// Stored populations as FP64 deviations, for the read-back.
template <typename S>
__global__ void k_batch_to_f64(const S* __restrict__ pops, double* __restrict__ out, long long count,
                               typename Store<S>::A inv) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = (double)Store<S>::load(pops + i, inv);
}

struct Shape {
    int zc, dense;   // cells per thread along z; more resident CTAs (fewer registers)
};

}  // namespace

// =================================================================== engine
struct BatchEngine {
    int nsims = 0;
    std::vector<SimDev> sims;
    SimDev* d_sims = nullptr;
    long long total_cells = 0;
    std::vector<long long> cell_off;
    long long* d_cell_off = nullptr;
    void* pops[2] = {nullptr, nullptr};
    int cur = 0;
    uint8_t* flags[2] = {nullptr, nullptr};
    int fcur = 0;
    ParticleState* d_ps = nullptr;
    std::vector<ParticleState> h_ps;   // host copies: of the start, then of what was read back
    std::vector<char> read;            // per RECORDS records: h_ps holds them as they are on the device
    int* seg = nullptr;         // boundary cells by segment (an entry per box cell of every simulation)
    int* seg_count = nullptr;   // and their number
    int* d_seg_sim = nullptr;   // simulation of each segment
    int segments = 0;
    int bnd_segs = 1, bnd_parts = 1;   // segments of a boundary CTA, CTAs that share them
    PFrames* frames = nullptr;  // frames of every simulation's sphere
    int* done = nullptr;        // last-block-done counter per simulation
    double* partials = nullptr;
    int bnd_blocks = 1;     // boundary-kernel blocks of all simulations
    int* d_bnd_sim = nullptr;   // simulation of each boundary CTA
    double* history = nullptr;
    // runs of items per bulk CTA for every candidate shape
    BulkRun* d_runs[2] = {nullptr, nullptr};   // with one and with two cells a thread
    int nruns[2] = {0, 0};
    int shape = 0;
    float shape_ms[4] = {0, 0, 0, 0};
    cudaGraphExec_t graph = nullptr;
    cudaStream_t capture_stream = nullptr;
    long long graph_launches = 0;
};

namespace {

const Shape SHAPES[4] = {{1, 0}, {2, 0}, {1, 1}, {2, 1}};

template <typename F>
void with_storage_batch(int prec, F&& f) {
    if (prec == LBMP_FP64) f((double*)nullptr);
    else if (prec == LBMP_FP32) f((float*)nullptr);
    else f((__half*)nullptr);
}

template <typename S>
void batch_scales(const lbmp_handle* h, typename Store<S>::A* scale, typename Store<S>::A* inv) {
    const bool f16 = h->cfg.precision == LBMP_FP16;
    *scale = (typename Store<S>::A)(f16 ? std::ldexp(1.0, h->cfg.fp16_scale_log2) : 1.0);
    *inv = (typename Store<S>::A)(f16 ? std::ldexp(1.0, -h->cfg.fp16_scale_log2) : 1.0);
}

// One step's stream-collide launch in a candidate shape; coupled: with the boundary CTAs.
template <typename S>
void launch_step_shape(lbmp_handle* h, BatchEngine* B, int shape, const S* src, S* dst, bool coupled) {
    BatchArgs<S> T;
    batch_scales<S>(h, &T.scale, &T.inv);
    T.src = src;
    T.dst = dst;
    T.flags = B->flags[B->fcur];
    const Shape s = SHAPES[shape];
    T.runs = B->d_runs[s.zc - 1];
    T.sims = B->d_sims;
    T.status = h->status;
    T.bblocks = coupled ? B->bnd_blocks : 0;
    T.bshift = 0;
    T.segs = B->bnd_segs;
    T.parts = B->bnd_parts;
    T.seg = B->seg;
    T.seg_count = B->seg_count;
    T.bnd_sim = B->d_bnd_sim;
    T.ps = B->d_ps;
    T.frames = B->frames;
    T.cli = h->cfg.boundary == LBMP_CLI ? 1 : 0;
    T.hist_cap = h->cfg.history_capacity;
    T.partials = B->partials;
    T.done = B->done;
    T.history = B->history;
    const unsigned grid = (unsigned)(T.bblocks + B->nruns[s.zc - 1]);
    while (T.bshift < 5 && (unsigned)T.bblocks << (T.bshift + 2) <= grid) ++T.bshift;   // in the first half of the grid
    auto go = [&](auto kernel) { launch_pdl(kernel, grid, BW, 0, h->stream, T); };
    constexpr int FEW = sizeof(S) == 8 ? 1 : 5, MORE = sizeof(S) == 8 ? 2 : 6;
    if (s.zc == 1 && !s.dense) go(k_batch_step<S, 1, FEW>);
    else if (!s.dense) go(k_batch_step<S, 2, FEW>);
    else if (s.zc == 1) go(k_batch_step<S, 1, MORE>);
    else go(k_batch_step<S, 2, MORE>);
}

template <typename S>
void enqueue_batch_step(lbmp_handle* h) {
    using A = typename Store<S>::A;
    BatchEngine* B = h->batch;
    A scale, inv;
    batch_scales<S>(h, &scale, &inv);
    const S* src = (const S*)B->pops[B->cur];
    S* dst = (S*)B->pops[1 - B->cur];
    const long long ev = profile_mark(h);
    launch_step_shape<S>(h, B, B->shape, src, dst, true);
    profile_kernel(h, ev, profile_mark(h), 38.0 * sizeof(S) * (double)B->total_cells, (double)B->total_cells);
    launch_pdl(k_batch_remap<S>, (unsigned)B->segments, BW, 0, h->stream, dst, (const uint8_t*)B->flags[B->fcur],
               B->flags[1 - B->fcur], (const SimDev*)B->d_sims, (const int*)B->d_seg_sim, (const ParticleState*)B->d_ps,
               (const PFrames*)B->frames, scale, inv, B->seg, B->seg_count, h->cfg.refill == LBMP_REFILL_GRAD ? 1 : 0);
    B->cur = 1 - B->cur;
    B->fcur = 1 - B->fcur;
    h->launches += 2;
    h->updates += B->total_cells;
}

}  // namespace

void batch_destroy(lbmp_handle* h) {
    BatchEngine* B = h->batch;
    if (!B) return;
    if (B->graph) cudaGraphExecDestroy(B->graph);
    if (B->capture_stream) cudaStreamDestroy(B->capture_stream);
    delete B;
    h->batch = nullptr;   // device memory is released with the handle's allocations
}

lbmp_status batch_create(lbmp_handle* h, const lbmp_batch_sim* sims, int n) {
    BatchEngine* B = new (std::nothrow) BatchEngine();
    if (!B) return LBMP_ERR_OOM;
    h->batch = B;
    B->nsims = n;
    B->sims.resize(n);
    B->h_ps.resize(n);
    B->read.assign((size_t)((n + RECORDS - 1) / RECORDS), 0);
    B->cell_off.resize(n + 1, 0);
    const size_t es = h->cfg.precision == LBMP_FP64 ? 8 : (h->cfg.precision == LBMP_FP32 ? 4 : 2);
    long long cells = 0;
    std::vector<int> bnd_sim, seg_sim;
    for (int s = 0; s < n; ++s) {
        const lbmp_batch_sim& in = sims[s];
        SimDev& D = B->sims[s];
        D.G.nx = D.G.ny = D.G.nz = in.edge;
        D.G.periodic[0] = D.G.periodic[1] = D.G.periodic[2] = 1;
        D.G.n = (long long)in.edge * in.edge * in.edge;
        D.pop_off = 19 * cells;
        D.flag_off = cells;
        B->cell_off[s] = cells;
        cells += D.G.n;
        relaxation_rates(in.tau, h->cfg.magic, &D.P.sp, &D.P.sm);
        D.P.db = bulk_rate_offset(in.tau, h->cfg.bulk_factor);
        D.P.F[0] = D.P.F[1] = D.P.F[2] = 0.0;
        D.P.forced = 0;
        D.P.scale = D.P.inv_scale = 1.0;
        collide_consts(D.P);
        ParticleState& P = B->h_ps[s];
        std::memset(&P, 0, sizeof(P));
        for (int a = 0; a < 3; ++a) {
            P.x[a] = in.pos[a];
            P.g[a] = in.gravity[a];
        }
        P.D = in.diameter;
        P.r = 0.5 * in.diameter;
        P.rho_p = in.density_ratio;
        P.cv = in.cv;
        P.cvw = in.cv_omega;
        P.V = M_PI * in.diameter * in.diameter * in.diameter / 6.0;
        P.present = 1;
        P.force_average = h->cfg.force_average ? 1 : 0;
        BoxDesc& X = D.box;
        X.R = (int)std::ceil(P.r) + 3;
        X.cells = 1;
        for (int a = 0; a < 3; ++a) {
            X.E[a] = 2 * X.R + 2;
            if (X.E[a] >= in.edge) X.E[a] = in.edge;
            X.cells *= X.E[a];
        }
        D.by_edge.set((unsigned)in.edge);
        D.seg_off = (int)seg_sim.size();
        D.nseg = (int)((X.cells + SEG - 1) / SEG);
        seg_sim.insert(seg_sim.end(), (size_t)D.nseg, s);
        D.hist_off = (long long)s * std::max(1, h->cfg.history_capacity);
    }
    // boundary CTAs: two segments each where that is two or more CTAs per SM, else one, shared by up to BND_PARTS CTAs
    B->bnd_segs = (int)seg_sim.size() >= 2 * SMS * BND_SEGS ? BND_SEGS : 1;
    while (B->bnd_segs == 1 && B->bnd_parts < BND_PARTS && (int)seg_sim.size() * B->bnd_parts < 2 * SMS) B->bnd_parts *= 2;
    for (int s = 0; s < n; ++s) {
        SimDev& D = B->sims[s];
        D.bnd_off = (int)bnd_sim.size();
        D.bnd_n = (D.nseg + B->bnd_segs - 1) / B->bnd_segs * B->bnd_parts;
        bnd_sim.insert(bnd_sim.end(), (size_t)D.bnd_n, s);
    }
    B->cell_off[n] = cells;
    B->total_cells = cells;
    B->segments = (int)seg_sim.size();
    B->bnd_blocks = (int)bnd_sim.size();
    const size_t pop_bytes = es * 19 * (size_t)cells;
    B->pops[0] = handle_alloc(h, pop_bytes);
    B->pops[1] = handle_alloc(h, pop_bytes);
    B->flags[0] = (uint8_t*)handle_alloc(h, (size_t)cells);
    B->flags[1] = (uint8_t*)handle_alloc(h, (size_t)cells);
    B->d_sims = (SimDev*)handle_alloc(h, sizeof(SimDev) * n);
    B->d_cell_off = (long long*)handle_alloc(h, sizeof(long long) * (n + 1));
    B->d_ps = (ParticleState*)handle_alloc(h, sizeof(ParticleState) * n);
    B->seg = (int*)handle_alloc(h, sizeof(int) * SEG * seg_sim.size());
    B->seg_count = (int*)handle_alloc(h, sizeof(int) * seg_sim.size());
    B->d_seg_sim = (int*)handle_alloc(h, sizeof(int) * seg_sim.size());
    B->frames = (PFrames*)handle_alloc(h, sizeof(PFrames) * (size_t)n);
    B->done = (int*)handle_alloc(h, sizeof(int) * n);
    B->partials = (double*)handle_alloc(h, sizeof(double) * 6 * (size_t)B->bnd_blocks);
    B->d_bnd_sim = (int*)handle_alloc(h, sizeof(int) * (size_t)B->bnd_blocks);
    B->history = (double*)handle_alloc(h, sizeof(double) * 15 * (size_t)n * std::max(1, h->cfg.history_capacity));
    if (!B->pops[0] || !B->pops[1] || !B->flags[0] || !B->flags[1] || !B->d_sims || !B->d_cell_off || !B->d_ps ||
        !B->seg || !B->seg_count || !B->d_seg_sim || !B->frames || !B->done || !B->partials || !B->d_bnd_sim || !B->history)
        return LBMP_ERR_OOM;
    cudaMemcpyAsync(B->d_bnd_sim, bnd_sim.data(), sizeof(int) * bnd_sim.size(), cudaMemcpyHostToDevice, h->stream);
    cudaMemcpyAsync(B->d_seg_sim, seg_sim.data(), sizeof(int) * seg_sim.size(), cudaMemcpyHostToDevice, h->stream);
    // bulk runs with zc = c + 1 cells a thread: a CTA takes BW consecutive items (edges are multiples of 16, e^3 / zc
    // of 2,048, so runs are whole)
    long long run_bytes = 0;
    for (int c = 0; c < 2; ++c) {
        std::vector<BulkRun> runs;
        for (int s = 0; s < n; ++s) {
            const SimDev& D = B->sims[s];
            BulkRun R = {};
            R.pop_off = D.pop_off;
            R.sim = s;
            R.edge = D.G.nx;
            R.by_edge = D.by_edge;
            R.sp = (float)D.P.sp;
            R.sm = (float)D.P.sm;
            R.db = (float)D.P.db;
            for (long long i = 0; i < D.G.n / (c + 1); i += BW) {
                R.item = (int)i;
                runs.push_back(R);
            }
        }
        B->nruns[c] = (int)runs.size();
        B->d_runs[c] = (BulkRun*)handle_alloc(h, sizeof(BulkRun) * runs.size());
        if (!B->d_runs[c]) return LBMP_ERR_OOM;
        cudaMemcpyAsync(B->d_runs[c], runs.data(), sizeof(BulkRun) * runs.size(), cudaMemcpyHostToDevice, h->stream);
        run_bytes += (long long)(sizeof(BulkRun) * runs.size());
    }
    cudaMemcpyAsync(B->d_sims, B->sims.data(), sizeof(SimDev) * n, cudaMemcpyHostToDevice, h->stream);
    cudaMemcpyAsync(B->d_cell_off, B->cell_off.data(), sizeof(long long) * (n + 1), cudaMemcpyHostToDevice, h->stream);
    cudaMemcpyAsync(B->d_ps, B->h_ps.data(), sizeof(ParticleState) * n, cudaMemcpyHostToDevice, h->stream);
    cudaMemsetAsync(B->pops[0], 0, pop_bytes, h->stream);
    cudaMemsetAsync(B->pops[1], 0, pop_bytes, h->stream);
    cudaMemsetAsync(B->done, 0, sizeof(int) * n, h->stream);
    // flags, zero solid (fluid at rest everywhere else), initial boundary lists
    const unsigned gcells = (unsigned)((cells + 255) / 256);
    k_batch_flags_full<<<gcells, 256, 0, h->stream>>>(B->flags[0], B->flags[1], B->d_sims, B->d_ps, B->d_cell_off, n,
                                                       cells);
    with_storage_batch(h->cfg.precision, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        using A = typename Store<S>::A;
        A scale, inv;
        batch_scales<S>(h, &scale, &inv);
        // frames, boundary flags and segments of the start position (both flag buffers hold its solid cells)
        k_batch_frames<<<n, 128, 0, h->stream>>>(B->d_sims, B->d_ps, B->frames);
        k_batch_remap<S><<<B->segments, BW, 0, h->stream>>>((S*)B->pops[0], B->flags[1], B->flags[0], B->d_sims,
                                                            B->d_seg_sim, B->d_ps, B->frames, scale, inv, B->seg,
                                                            B->seg_count, 0);   // nothing is uncovered here
    });
    h->h2d += (long long)(sizeof(SimDev) + sizeof(ParticleState) + sizeof(long long)) * n +
              (long long)(sizeof(int) * (bnd_sim.size() + seg_sim.size())) + run_bytes;
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(h->stream) != cudaSuccess) return LBMP_ERR_CUDA;
    h->has_particle = true;
    return LBMP_OK;
}

lbmp_status batch_autotune(lbmp_handle* h, int reps) {
    BatchEngine* B = h->batch;
    if (B->graph) {
        cudaGraphExecDestroy(B->graph);
        B->graph = nullptr;
    }
    cudaEvent_t a, b;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) return LBMP_ERR_CUDA;
    float best = 1e30f;
    with_storage_batch(h->cfg.precision, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        // candidates read the current field and write the other buffer, which
        // the next step overwrites: the simulation state is not advanced
        const S* src = (const S*)B->pops[B->cur];
        S* dst = (S*)B->pops[1 - B->cur];
        for (int c = 0; c < 4; ++c) {
            launch_step_shape<S>(h, B, c, src, dst, false);   // warm-up
            cudaEventRecord(a, h->stream);
            for (int r = 0; r < reps; ++r) launch_step_shape<S>(h, B, c, src, dst, false);
            cudaEventRecord(b, h->stream);
            cudaEventSynchronize(b);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, a, b);
            B->shape_ms[c] = ms / reps;
            if (B->shape_ms[c] < best) {
                best = B->shape_ms[c];
                B->shape = c;
            }
        }
    });
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return cudaGetLastError() == cudaSuccess ? LBMP_OK : LBMP_ERR_CUDA;
}

lbmp_status batch_step(lbmp_handle* h, int n) {
    BatchEngine* B = h->batch;
    std::fill(B->read.begin(), B->read.end(), 0);
    auto one = [&]() {
        with_storage_batch(h->cfg.precision, [&](auto tag) {
            using S = std::remove_pointer_t<decltype(tag)>;
            enqueue_batch_step<S>(h);
        });
        h->steps += 1;
    };
    int i = 0;
    while (i < n) {
        // the captured graph holds two steps starting from buffer 0
        if (h->profiling || n - i < 2 || B->cur != 0 || B->fcur != 0) {
            one();
            ++i;
            continue;
        }
        if (!B->graph) {
            if (!B->capture_stream && cudaStreamCreateWithFlags(&B->capture_stream, cudaStreamNonBlocking) != cudaSuccess)
                return LBMP_ERR_CUDA;
            cudaStream_t user = h->stream;
            const long long l0 = h->launches, u0 = h->updates;
            h->stream = B->capture_stream;
            if (cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) {
                h->stream = user;
                return LBMP_ERR_CUDA;
            }
            with_storage_batch(h->cfg.precision, [&](auto tag) {
                using S = std::remove_pointer_t<decltype(tag)>;
                enqueue_batch_step<S>(h);
                enqueue_batch_step<S>(h);
            });
            cudaGraph_t g = nullptr;
            const cudaError_t e = cudaStreamEndCapture(h->stream, &g);
            h->stream = user;
            if (e != cudaSuccess) return LBMP_ERR_CUDA;
            const cudaError_t e2 = cudaGraphInstantiate(&B->graph, g, 0);
            cudaGraphDestroy(g);
            if (e2 != cudaSuccess) return LBMP_ERR_CUDA;
            B->graph_launches = h->launches - l0;
            h->launches = l0;
            h->updates = u0;
        }
        if (cudaGraphLaunch(B->graph, h->stream) != cudaSuccess) return LBMP_ERR_CUDA;
        h->launches += B->graph_launches;
        h->updates += 2 * B->total_cells;
        h->steps += 2;
        i += 2;
    }
    return cudaGetLastError() == cudaSuccess ? LBMP_OK : LBMP_ERR_CUDA;
}

lbmp_status batch_get_particle(lbmp_handle* h, int sim, ParticleState* out) {
    BatchEngine* B = h->batch;
    if (sim < 0 || sim >= B->nsims) return LBMP_ERR_INVALID_ARG;
    const int block = sim / RECORDS, first = block * RECORDS;
    if (!B->read[block]) {
        const size_t bytes = sizeof(ParticleState) * (size_t)std::min(RECORDS, B->nsims - first);
        if (cudaMemcpyAsync(B->h_ps.data() + first, B->d_ps + first, bytes, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
            cudaStreamSynchronize(h->stream) != cudaSuccess)
            return LBMP_ERR_CUDA;
        h->d2h += (long long)bytes;
        B->read[block] = 1;
    }
    *out = B->h_ps[sim];
    return LBMP_OK;
}

const double* batch_history(const lbmp_handle* h, int sim) {
    return h->batch->history + (size_t)h->batch->sims[sim].hist_off * 15;
}

lbmp_status batch_populations(lbmp_handle* h, int sim, double* out, size_t cap) {
    BatchEngine* B = h->batch;
    if (sim < 0 || sim >= B->nsims) return LBMP_ERR_INVALID_ARG;
    const SimDev& D = B->sims[sim];
    const long long count = 19 * D.G.n;
    if ((long long)cap < count) return LBMP_ERR_INVALID_ARG;
    double* tmp = (double*)handle_alloc(h, sizeof(double) * (size_t)count);
    if (!tmp) return LBMP_ERR_OOM;
    with_storage_batch(h->cfg.precision, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        using A = typename Store<S>::A;
        A scale, inv;
        batch_scales<S>(h, &scale, &inv);
        k_batch_to_f64<S><<<(unsigned)((count + 255) / 256), 256, 0, h->stream>>>((const S*)B->pops[B->cur] + D.pop_off,
                                                                                  tmp, count, inv);
    });
    cudaError_t e = cudaMemcpyAsync(out, tmp, sizeof(double) * (size_t)count, cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    h->d2h += (long long)sizeof(double) * count;
    handle_free(h, tmp);
    return e == cudaSuccess ? LBMP_OK : LBMP_ERR_CUDA;
}

void batch_info(const lbmp_handle* h, int64_t out[8]) {
    const BatchEngine* B = h->batch;
    out[0] = B->nsims;
    out[1] = B->total_cells;
    out[2] = BW;
    out[3] = SHAPES[B->shape].zc;
    for (int c = 0; c < 4; ++c) out[4 + c] = (int64_t)(B->shape_ms[c] * 1e6);   // ns per launch
}

}  // namespace lbmp
