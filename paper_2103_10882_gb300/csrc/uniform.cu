// Uniform-grid kernels of the coupled step (Algorithm 1), two launches per step:
//   k_step       stream (pull) + TRT collide of every cell (Sec. 2.1, Eq. LBE); its first CTAs take the cells
//                next to the sphere (CLI links, momentum-exchange force and torque, Sec. 2.3), and the last of
//                those to finish runs the particle update (force averaging, gravity, virtual mass, Velocity
//                Verlet, Sec. 2.2, 3.3)
//   k_remap      flags, refill and marks of the boundary cells after the sphere moved (Sec. 2.3)
// Populations are stored as deviations g = f - w in SoA layout [q][z][y][x].
#include <cuda_fp16.h>

#include <type_traits>

#include "internal.h"
#include "physics.cuh"

namespace lbmp {
namespace {

constexpr int STEP_THREADS = 256;
constexpr unsigned BULK_LONG = 40 * SMS;   // bulk CTAs: eight waves in FP32, ten in FP16, twenty in FP64
// Marks of the box cells around the sphere, written by the remap: plain fluid cell, fluid cell with a solid
// D3Q19 neighbour (taken by the boundary CTAs), cell with its centre inside the sphere.
constexpr uint8_t MARK_PLAIN = 0, MARK_BOUNDARY = 1, MARK_SOLID = 2;

// One coupled step of a uniform grid.
template <typename S>
struct StepArgs {
    using A = typename Store<S>::A;
    const S* src;
    S* dst;
    GridDesc G;
    CollideParams<A> P;
    FastDiv dx, dy;        // by nx (FP16 pairs: nx / 2) and ny
    unsigned items;        // cells (FP16 pairs: pairs of cells)
    int per_cta;           // of them per bulk CTA
    int* status;
    // the sphere's part (bblocks = 0 without a sphere)
    int bblocks;           // boundary CTAs: every 2^bshift-th CTA from the first on
    int bshift;
    int thin;              // a warp of every boundary CTA before a second one of any
    int finish;            // last boundary CTA: 0 the particle update, 1 the force into force_out, 2 nothing
    int cli, hist_cap;
    const uint8_t* flags;
    const uint8_t* mark;
    const int* seg;        // boundary cells (linear indices) by segment of the box, and their numbers
    const int* seg_count;
    const int* list;       // boundary cells as a list, for boxes of more than SEG_CELLS_MAX cells; else null
    FastDiv fx, fy;        // by nx and ny
    const int* count;
    BoxDesc B;
    ParticleState* ps;
    double* partials;
    int* done;
    double* history;
    const PFrames* frames;   // of the sphere's position in this step
    PFrames* frames_next;    // of the position that the particle update reaches
    double* force_out;
};

// Mark of cell (x, y, z): outside the sphere's box every cell is plain.  The box origin lies on the device;
// o, n and E per axis as in box_cell.
__device__ __forceinline__ int box_coord(int v, int o, int n, int periodic, int E) {
    int t = v - o;
    if (periodic) t = t < 0 ? t + n : (t >= n ? t - n : t);
    return (t >= 0 && t < E) ? t : -1;
}

// Index of the box cells of row (y, z), -1 outside the sphere's box (and without a sphere).  Most rows lie outside, so
// only there a cell's own place in the row is looked for, after its loads: 256^3 in FP16 storage 237 -> 228 us a step,
// the 64^3 gradient 15.7 -> 15.5 ms, 512^3 2989 -> 2976 us.
template <typename S>
__device__ __forceinline__ int box_row(const StepArgs<S>& T, int y, int z) {
    if (T.bblocks == 0) return -1;
    const int* o = T.frames->bf.o;
    const int tz = box_coord(z, o[2], T.G.nz, T.G.periodic[2], T.B.E[2]);
    const int ty = box_coord(y, o[1], T.G.ny, T.G.periodic[1], T.B.E[1]);
    return (ty | tz) < 0 ? -1 : T.B.E[0] * (ty + T.B.E[1] * tz);
}

// ------------------------------------------------------------------ bulk
// One thread per cell, pull form: g_q(x, t+1) = g~_q(x - c_q, t), then TRT; solid cells are stored as zero and
// boundary cells left to the boundary CTAs.  Cells are taken in memory order, so full warps touch whole lines
// whatever the extents (a 2-D tile of a 75-cell row left two threads in five idle).  WALLS: some axis has
// no-slip walls (bounce-back at the domain edge, by the address of the load, not by a branch around it: 256 x 128 x 96
// 87.0 -> 81.3 us a step, 61 x 53 x 75 in FP64 82.4 -> 79.2); FORCED: fluid body force present.
template <typename S, bool WALLS, bool FORCED>
__device__ __forceinline__ void bulk_cells(const StepArgs<S>& T, unsigned item) {
    using A = typename Store<S>::A;
    const GridDesc& G = T.G;
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const unsigned row = T.dx.div(item), plane = T.dy.div(row);
    const int x = (int)(item - row * (unsigned)nx), y = (int)(row - plane * (unsigned)ny), z = (int)plane;
    const size_t n = (size_t)G.n;
    const int cell = (int)item;
    // source coordinate x - c for c = -1, 0, +1 (-1 marks a wall)
    int xs[3], ys[3], zs[3];
    xs[1] = x;
    ys[1] = y;
    zs[1] = z;
    xs[0] = x + 1 < nx ? x + 1 : (WALLS && !G.periodic[0] ? -1 : 0);
    xs[2] = x > 0 ? x - 1 : (WALLS && !G.periodic[0] ? -1 : nx - 1);
    ys[0] = y + 1 < ny ? y + 1 : (WALLS && !G.periodic[1] ? -1 : 0);
    ys[2] = y > 0 ? y - 1 : (WALLS && !G.periodic[1] ? -1 : ny - 1);
    zs[0] = z + 1 < nz ? z + 1 : (WALLS && !G.periodic[2] ? -1 : 0);
    zs[2] = z > 0 ? z - 1 : (WALLS && !G.periodic[2] ? -1 : nz - 1);
    A g[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        const int sx = xs[cx(q) + 1], sy = ys[cy(q) + 1], sz = zs[cz(q) + 1];
        const bool wall = WALLS && (sx < 0 || sy < 0 || sz < 0);   // no-slip wall: bounce-back
        const size_t at = wall ? (size_t)opp(q) * n + (size_t)cell : (size_t)q * n + (size_t)(sx + nx * (sy + ny * sz));
        g[q] = Store<S>::fetch(T.src + at, T.P.inv_scale);
    }
    uint8_t mark = MARK_PLAIN;   // beside the pulls, not before them
    const int box = box_row(T, y, z);
    if (box >= 0) {
        const int tx = box_coord(x, T.frames->bf.o[0], nx, G.periodic[0], T.B.E[0]);
        if (tx >= 0) mark = T.mark[box + tx];
    }
    if (mark != MARK_PLAIN) {
        if (mark == MARK_SOLID)
#pragma unroll
            for (int q = 0; q < 19; ++q) Store<S>::store(T.dst + (size_t)q * n + cell, A(0), T.P.scale);
        return;
    }
    if (WALLS && G.moving && ((xs[0] | xs[2] | ys[0] | ys[2] | zs[0] | zs[2]) < 0)) {   // moving walls: Ladd's term
        const int xyz[3] = {x, y, z};
#pragma unroll
        for (int q = 1; q < 19; ++q)
            if ((xs[cx(q) + 1] | ys[cy(q) + 1] | zs[cz(q) + 1]) < 0) g[q] += wall_term<A>(G, q, xyz);
    }
    trt_collide<A, FORCED>(g, T.P, T.status);
#pragma unroll
    for (int q = 0; q < 19; ++q) Store<S>::store(T.dst + (size_t)q * n + cell, g[q], T.P.scale);
}

// Two cells side by side in the packed FP32 arithmetic of the part (PTX f32x2): one instruction for both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Coefficients of collide_pair, each twice (c...: of the quadratic terms, with the FP16 storage factor).
struct PairConsts {
    float2 one_m, half, three, c15, c45;   // -1, 1/2, 3, -3/2, 9/2
    float2 w0, wF, wE;                     // lattice weights, negated
    float2 sp, sm, sm_m;                   // -s+, s-, -s-
    float2 two, h15, d0, dF, dE;           // MRT: -2, 3/2, -db w of rest, 2 db w of faces, -db w of edges
};
inline PairConsts pair_consts(const CollideParams<float>& P) {
    auto both = [](float v) { return make_float2(v, v); };
    const float w0 = wgt<float>(0), wF = wgt<float>(1), wE = wgt<float>(7);
    PairConsts c;
    c.one_m = both(-1.0f);
    c.half = both(0.5f);
    c.three = both(3.0f);
    c.c15 = both(-1.5f * P.inv_scale);
    c.c45 = both(4.5f * P.inv_scale);
    c.w0 = both(-w0);
    c.wF = both(-wF);
    c.wE = both(-wE);
    c.sp = both(-P.sp);
    c.sm = both(P.sm);
    c.sm_m = both(-P.sm);
    c.two = both(-2.0f);
    c.h15 = both(1.5f);
    c.d0 = both(-(P.db * w0));
    c.dF = both(2.0f * (P.db * wF));
    c.dE = both(-(P.db * wE));
    return c;
}

// trt_collide (unforced, scaled) of two cells at once, the moments from the sums and differences of the opposite pairs;
// check0, check1: the cell's velocity is looked at.  A population relaxes by s+ and s- times its distance from the
// equilibrium, g - s+ (g+ - e+) - s- (g- - e-), so that the rounding of the rates is multiplied by that distance: the
// momentum, which a collision keeps, is scaled by 1 + 2e-10 (tau 0.506) to 1 + 1.5e-8 in a step, by the rounding of the
// weights.  Sums and differences multiplied by rounded coefficients (1 - s+)/2 and (1 - s-)/2 take 116 instructions
// instead of 177 (a step of 256^3 cells 224 us and 229; 256 x 128 x 96 with walls, where the instructions are the time,
// 57 and 67), but scale it by 1 + 1.5e-8 to 1 + 6e-8.  Every product and sum is rounded as written.
template <bool MRT>
__device__ __forceinline__ void collide_pair(f32x2 (&g)[19], const PairConsts& C, float inv_scale, bool check0, bool check1,
                                             int* status) {
    auto K = [](const float2& v) { return pack2(v.x, v.y); };
    auto sub2 = [&](f32x2 a, f32x2 b) { return fma2(b, K(C.one_m), a); };
    f32x2 ps[9], pd[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        ps[k] = add2(g[2 * k + 1], g[2 * k + 2]);
        pd[k] = sub2(g[2 * k + 1], g[2 * k + 2]);
    }
    f32x2 drho = g[0];
#pragma unroll
    for (int k = 0; k < 9; ++k) drho = add2(drho, ps[k]);
    // pairs 3..8: (+x+y), (+x-y), (+x+z), (+x-z), (+y+z), (+y-z)
    const f32x2 u[3] = {add2(add2(add2(add2(pd[0], pd[3]), pd[4]), pd[5]), pd[6]),
                        add2(add2(sub2(add2(pd[1], pd[3]), pd[4]), pd[7]), pd[8]),
                        sub2(add2(sub2(add2(pd[2], pd[5]), pd[6]), pd[7]), pd[8])};
    const f32x2 uu = fma2(u[2], u[2], fma2(u[1], u[1], mul2(u[0], u[0])));
    const float2 v = unpack2(uu);
    const float limit = inv_scale * inv_scale;
    if ((check0 && !(v.x * limit <= 0.09f)) || (check1 && !(v.y * limit <= 0.09f))) atomicOr(status, STATUS_UNSTABLE_FLUID);
    // MRT: sums of f - f_eq over the rest, face and edge populations
    f32x2 nR, nF, nE;
    {
        const f32x2 n0 = fma2(K(C.w0), fma2(K(C.c15), uu, drho), g[0]);
        if (MRT) nR = n0;
        g[0] = fma2(K(C.sp), n0, g[0]);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int q = 2 * k + 1;
        const float2 &w = k < 3 ? C.wF : C.wE;
        f32x2 cu;
        if (k < 3) {
            cu = u[k];
        } else {
            const int a = k < 7 ? 0 : 1, b = k < 5 ? 1 : 2;
            cu = (k & 1) ? add2(u[a], u[b]) : sub2(u[a], u[b]);
        }
        const f32x2 ep = mul2(K(w), fma2(K(C.c15), uu, fma2(mul2(K(C.c45), cu), cu, drho)));   // -e+
        const f32x2 em = mul2(K(w), mul2(K(C.three), cu));                                      // -e-
        // g+ - e+ and g- - e-, the sum and difference formed again: kept, they spill.  (As sums of two such terms, not
        // as fma2 with one half, the assembler would fuse them with the products before them.)
        const f32x2 np = fma2(K(C.half), add2(g[q + 1], g[q]), ep);
        const f32x2 nm = fma2(K(C.half), fma2(K(C.one_m), g[q + 1], g[q]), em);
        if (MRT) {
            if (k == 0) nF = add2(np, np);
            else if (k < 3) nF = add2(nF, add2(np, np));
            else if (k == 3) nE = add2(np, np);
            else nE = add2(nE, add2(np, np));
        }
        g[q] = fma2(K(C.sm_m), nm, fma2(K(C.sp), np, g[q]));
        g[q + 1] = fma2(K(C.sm), nm, fma2(K(C.sp), np, g[q + 1]));
    }
    if (MRT) {   // as in trt_collide
        const f32x2 s4 = sub2(nE, nR), c16 = mul2(K(C.half), add2(fma2(K(C.two), nF, nR), nE));
        const f32x2 r = fma2(K(C.h15), mul2(K(C.one_m), s4), c16), e = fma2(K(C.h15), s4, c16);
        g[0] = fma2(K(C.d0), r, g[0]);
#pragma unroll
        for (int q = 1; q < 7; ++q) g[q] = fma2(K(C.dF), c16, g[q]);
#pragma unroll
        for (int q = 7; q < 19; ++q) g[q] = fma2(K(C.dE), e, g[q]);
    }
}

// FP16 storage, unforced: the same update, two cells (x, x + 1, x even) per
// thread.  Every population is read as the aligned pair of halves of its
// source row; the populations shifted along x take their outer half from the
// neighbouring lane (a shuffle); the first lane of a warp or row and the last
// pair of a warp or row load that one half themselves.  The collision runs on
// the stored, scaled values (collide_pair), so neither the loads nor the
// stores multiply by the scale, and TRT or MRT is chosen at compile time.  nx
// is even; rows hold whole pairs.  Every lane of the warp calls it (valid:
// the lane has a pair).
// Bound by what it issues as much as by HBM (188 us at 256^3): 262 us a step
// with two scalar collisions, 255 packed, 251 with ordinary stores, 235 with
// one load for the outer halves of a population and its mirror image, 224 with
// the marks after the loads (box_row), 229 with the collision's rounding as it
// is now.  With walls the bounced populations are chosen by their address, the
// moving walls' term added after the loads: 256 x 128 x 96 74.7 us a step with a
// branch around every load, 70.4 packed, 62.0 so, 57.3 with box_row, now 66.8.
template <bool WALLS, bool MRT>
__device__ __forceinline__ void bulk_pairs(const StepArgs<__half>& T, const PairConsts& K, unsigned pair, bool valid) {
    const GridDesc& G = T.G;
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int lane = threadIdx.x & 31;
    const unsigned item = valid ? pair : 0u;
    const unsigned row0 = T.dx.div(item), plane = T.dy.div(row0);
    const int x = 2 * (int)(item - row0 * T.dx.d), yy = (int)(row0 - plane * (unsigned)ny), z = (int)plane;
    const size_t n = (size_t)G.n;
    const __half* src = T.src;
    const int cell = x + nx * (yy + ny * z);
    int ys[3], zs[3];
    ys[1] = yy;
    zs[1] = z;
    ys[0] = yy + 1 < ny ? yy + 1 : (WALLS && !G.periodic[1] ? -1 : 0);
    ys[2] = yy > 0 ? yy - 1 : (WALLS && !G.periodic[1] ? -1 : ny - 1);
    zs[0] = z + 1 < nz ? z + 1 : (WALLS && !G.periodic[2] ? -1 : 0);
    zs[2] = z > 0 ? z - 1 : (WALLS && !G.periodic[2] ? -1 : nz - 1);
    // x - 1 of the pair's first cell and x + 2 of its second (-1: beyond a wall)
    const int xm = x > 0 ? x - 1 : (WALLS && !G.periodic[0] ? -1 : nx - 1);
    const int xq = x + 2 < nx ? x + 2 : (WALLS && !G.periodic[0] ? -1 : 0);
    const bool first = lane == 0 || x == 0, last = lane == 31 || x + 2 >= nx;   // warp or row ends
    // all loads first (the pairs, then the outer halves of the shifted populations, every lane
    // loading one: the lanes that need none read their own pair's first half), then the shuffles
    __half2 pr[19];
    __half ex[19];
    auto behind = [&](int q) { return WALLS && (ys[cy(q) + 1] < 0 || zs[cz(q) + 1] < 0); };   // a wall in y or z
    auto row_of = [&](int q) { return nx * (ys[cy(q) + 1] + ny * zs[cz(q) + 1]); };
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        const bool yw = behind(q);
        const int row = yw ? nx * (yy + ny * z) : row_of(q);
        pr[q] = *reinterpret_cast<const __half2*>(src + (size_t)(yw ? opp(q) : q) * n + row + x);
        if (cx(q) == 1) {
            // its mirror image along x reads the same row: one load for the two, few lanes need both
            const int m = q == 1 ? 2 : (q == 7 ? 10 : (q == 9 ? 8 : (q == 11 ? 14 : 12)));
            const bool wall = WALLS && (first ? xm : xq) < 0;   // bounce-back: the cell's own opposite population
            const int pop = wall ? (first ? opp(q) : opp(m)) : (first ? q : m);
            ex[q] = src[(size_t)pop * n + (size_t)(wall ? cell + (first ? 0 : 1) : row + (first ? xm : (last ? xq : x)))];
            ex[m] = ex[q];
        }
    }
    if (first && last) {
#pragma unroll
        for (int q = 1; q < 19; ++q)
            if (cx(q) == -1) {
                const bool wall = WALLS && xq < 0;
                ex[q] = src[(size_t)(wall ? opp(q) : q) * n + (size_t)(wall ? cell + 1 : (behind(q) ? nx * (yy + ny * z) : row_of(q)) + xq)];
            }
    }
    uint8_t mark0 = MARK_PLAIN, mark1 = MARK_PLAIN;
    const int box = box_row(T, yy, z);
    if (box >= 0) {
        const int t0 = box_coord(x, T.frames->bf.o[0], nx, G.periodic[0], T.B.E[0]);
        const int t1 = box_coord(x + 1, T.frames->bf.o[0], nx, G.periodic[0], T.B.E[0]);
        if (t0 >= 0) mark0 = T.mark[box + t0];
        if (t1 >= 0) mark1 = T.mark[box + t1];
    }
    f32x2 g[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        const __half2 p = pr[q];
        float a, b;
        if (cx(q) == 0) {
            a = __low2float(p);
            b = __high2float(p);
        } else {
            if (cx(q) == 1) {   // sources x - 1 and x
                const float prev = __shfl_up_sync(0xffffffffu, __high2float(p), 1);
                a = first ? __half2float(ex[q]) : prev;
                b = __low2float(p);
            } else {            // sources x + 1 and x + 2
                const float next = __shfl_down_sync(0xffffffffu, __low2float(p), 1);
                a = __high2float(p);
                b = last ? __half2float(ex[q]) : next;
            }
            if (behind(q)) {
                a = __low2float(p);
                b = __high2float(p);
            }
        }
        g[q] = pack2(a, b);
    }
    if (!valid) return;
    __half* dst = T.dst;
    if (WALLS && G.moving && ((xm | xq | ys[0] | ys[2] | zs[0] | zs[2]) < 0)) {   // Ladd's term, scaled like the stored values
        const int xyz0[3] = {x, yy, z}, xyz1[3] = {x + 1, yy, z};
#pragma unroll
        for (int q = 1; q < 19; ++q) {
            const bool wa = behind(q) || (cx(q) == 1 && xm < 0), wb = behind(q) || (cx(q) == -1 && xq < 0);
            if (wa || wb)
                g[q] = add2(g[q], pack2(wa ? wall_term<float>(G, q, xyz0) * T.P.scale : 0.0f,
                                        wb ? wall_term<float>(G, q, xyz1) * T.P.scale : 0.0f));
        }
    }
    collide_pair<MRT>(g, K, T.P.inv_scale, mark0 == MARK_PLAIN, mark1 == MARK_PLAIN, T.status);
    if ((mark0 | mark1) == MARK_PLAIN) {
#pragma unroll
        for (int q = 0; q < 19; ++q) {
            const float2 v = unpack2(g[q]);
            *reinterpret_cast<__half2*>(dst + (size_t)q * n + cell) = __floats2half2_rn(v.x, v.y);
        }
        return;
    }
    // one of the two is solid or a boundary cell: each by itself
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        const float2 v = unpack2(g[q]);
        if (mark0 != MARK_BOUNDARY) dst[(size_t)q * n + cell] = __float2half_rn(mark0 == MARK_SOLID ? 0.0f : v.x);
        if (mark1 != MARK_BOUNDARY) dst[(size_t)q * n + cell + 1] = __float2half_rn(mark1 == MARK_SOLID ? 0.0f : v.y);
    }
}

// -------------------------------------------------------------- boundary
// The cells next to the sphere, one warp per cell, lane q handling population q: pulls from solid cells are
// replaced by the CLI rule of Sec. 2.3 (link geometry in the population arithmetic), then the warp collides the
// cell cooperatively and writes it.  The boundary cells are spread evenly over the warps of the boundary CTAs:
// every CTA turns the remap's numbers per segment into a prefix, and warp w of W takes the cells w, w + W, ...
// in box order (or the entries of the list, for large boxes).  The block sums of force and torque go into one
// FP64 partial per CTA; the CTA that finishes last sums them.  Runs beside the bulk CTAs, which skip these cells.
template <typename S, bool FORCED>
__device__ __forceinline__ void boundary_cells(const StepArgs<S>& T, int bid, int* pre) {
    using A = typename Store<S>::A;
    const GridDesc& G = T.G;
    const CollideParams<A>& P = T.P;
    const S* src = T.src;
    __shared__ LinkFrame<A> Fr;
    const int nseg = (int)((T.B.cells + SEG - 1) / SEG);
    __shared__ double sX[3];
    if (threadIdx.x == STEP_THREADS - 1) Fr = pframe_link<A>(*T.frames);
    if (threadIdx.x >= STEP_THREADS - 32 && threadIdx.x < STEP_THREADS - 29)
        sX[threadIdx.x - (STEP_THREADS - 32)] = T.ps->x[threadIdx.x - (STEP_THREADS - 32)];
    const int i2 = 2 * (int)threadIdx.x;
    int total;
    if (T.list) {
        total = *T.count;
        __syncthreads();
    } else {
        const int first0 = i2 < nseg ? T.seg_count[i2] : 0, first1 = i2 + 1 < nseg ? T.seg_count[i2 + 1] : 0;
        total = block_prefix<STEP_THREADS>(T.seg_count, nseg, pre, first0, first1);
    }
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int W = T.bblocks * (STEP_THREADS / 32);
    const size_t n = (size_t)G.n;
    const int n3[3] = {G.nx, G.ny, G.nz};
    const int q = lane < 19 ? lane : 0, k = opp(q);
    const int c[3] = {cx(q), cy(q), cz(q)};
    LinkSums<A> acc;
    // a warp's last cell is stored after the hand-off: the hand-off's release waits for the stores before it
    A kept = A(0);
    S* kept_at = nullptr;
    for (int j = sizeof(S) == 8 && T.thin ? wib * T.bblocks + bid : bid * (STEP_THREADS / 32) + wib; j < total; j += W) {
        if (kept_at) Store<S>::store(kept_at, kept, P.scale);
        int at = j;
        if (!T.list) {
            const int sg = find_segment(pre, nseg, j);
            at = sg * SEG + (j - pre[sg]);
        }
        const int ci = T.list ? T.list[at] : T.seg[at];
        const unsigned row = T.fx.div((unsigned)ci), plane = T.fy.div(row);
        const int xyz[3] = {ci - (int)row * G.nx, (int)row - (int)plane * G.ny, (int)plane};
        const size_t cell = (size_t)ci;
        A gq = A(0);
        if (lane < 19) {
            int s3[3], f3[3];
            bool wall = false, far_ok = true;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                s3[a] = src_coord(xyz[a], c[a], n3[a], G.periodic[a]);    // x - c_q
                f3[a] = src_coord(xyz[a], -c[a], n3[a], G.periodic[a]);   // x + c_q
                wall |= s3[a] < 0;
                far_ok &= f3[a] >= 0;
            }
            // everything the pull or the link can need at once: one memory round trip instead of three
            const size_t sidx = wall ? cell : (size_t)s3[0] + (size_t)G.nx * ((size_t)s3[1] + (size_t)G.ny * (size_t)s3[2]);
            const size_t far = far_ok ? (size_t)f3[0] + (size_t)G.nx * ((size_t)f3[1] + (size_t)G.ny * (size_t)f3[2]) : cell;
            const uint8_t fsrc = T.flags[sidx], ffar = T.flags[far];
            const A pull = Store<S>::fetch(src + (size_t)q * n + sidx, P.inv_scale);
            const A gt_k = Store<S>::fetch(src + (size_t)k * n + cell, P.inv_scale);
            const A gt_q = Store<S>::fetch(src + (size_t)q * n + cell, P.inv_scale);
            const A vfar = Store<S>::fetch(src + (size_t)k * n + far, P.inv_scale);
            // the link's geometry while they are on their way, as if the far cell were fluid (it nearly always is)
            A d[3];
            int pu[3];
            Fr.offset(xyz, n3, G.periodic, d, pu);
            CliGeometry<A> L = cli_geometry<A>(q, d, T.cli != 0, Fr);
            gq = pull;
            if (wall) {
                gq = gt_k + wall_term<A>(G, q, xyz);
            } else if (q != 0 && fsrc != 0) {
                far_ok = far_ok && ffar == 0;
                if (T.cli && !far_ok) L = cli_geometry<A>(q, d, false, Fr);
                A fl[3], tl[3];
                gq = cli_apply<A>(q, L, gt_k, gt_q, far_ok ? vfar : A(0), fl, tl);
                acc.add(k, pu, fl, tl);
            }
        }
        kept = warp_trt_collide<A, FORCED>(gq, lane, P, T.status);
        if (lane < 19) kept_at = T.dst + (size_t)lane * n + cell;
    }
    if (T.finish == 2) {   // the force is not wanted
        if (kept_at) Store<S>::store(kept_at, kept, P.scale);
        return;
    }
    block_link_sums<STEP_THREADS>(acc, sX, T.partials + bid, T.bblocks);
    const bool last = last_block_done(T.done, T.bblocks);
    if (kept_at) Store<S>::store(kept_at, kept, P.scale);
    if (!last) return;
    if (T.finish == 1) {
        // the next step's launch beside this sum: 32^3 gradient 18.7 -> 17.7 us a step (before the particle update it does
        // not pay: 32^3 2% slower, the remap's CTAs take the SM's slots from it)
        pdl_trigger();
        if (wib < 3) {
            const double f = sum_partials(T.partials, T.bblocks, wib);
            if (lane == 0) T.force_out[wib] = f;
        }
        return;
    }
    // with it the frames of the moved sphere, in the other copy: bulk CTAs of this launch still read this one
    particle_block_update<STEP_THREADS>(T.ps, T.partials, T.bblocks, G, T.history, T.hist_cap, T.status, T.frames->inv,
                                        [&](const ParticleState& Q, int a, int part) {
                                            pframes_axis(T.frames_next, Q, n3, T.B, a, part);
                                        });
}

// CTA b of the grid: boundary CTA b >> bshift (true), or the bulk CTA *bulk.
template <typename S>
__device__ __forceinline__ bool is_boundary_cta(const StepArgs<S>& T, unsigned b, unsigned* bulk) {
    const unsigned before = min((unsigned)T.bblocks, (b + (1u << T.bshift) - 1u) >> T.bshift);
    *bulk = b - before;
    return (b & ((1u << T.bshift) - 1u)) == 0u && (b >> T.bshift) < (unsigned)T.bblocks;
}

// One launch: boundary CTAs among the first bulk CTAs (launch_step).  The chain boundary cells -> force sum -> particle update
// (11 + 5 us as two launches of their own) runs beside the bulk update instead of after it.  With k_remap for the four
// remap launches: a 32^3 FP32 step 46.1 -> 23.4 us, 256 x 128 x 96 with walls 123.6 -> 94.2, 61 x 53 x 75 in FP64
// 175 -> 92 (with collide_direct), 512^3 3066 -> 2997.  With what the parts below took off since: 14.7, 81.3, 79.2 and 2990.
// CTAS: resident CTAs of 256 threads per SM asked of the compiler (launch_step): FP64 2, FP16 4, FP32 4 or 5.  FP16
// pairs: 4, with walls 3 (80 registers; four spill 100 bytes, 256 x 128 x 96 68.2 us a step instead of 66.8).
template <typename S, bool WALLS, bool FORCED, int CTAS>
__global__ void __launch_bounds__(STEP_THREADS, CTAS) k_step(const __grid_constant__ StepArgs<S> T) {
    extern __shared__ int pre[];   // prefix of the segments' numbers (boundary CTAs)
    pdl_wait();
    unsigned bulk;
    if (is_boundary_cta(T, blockIdx.x, &bulk)) {
        boundary_cells<S, FORCED>(T, (int)(blockIdx.x >> T.bshift), pre);
        return;
    }
    const unsigned t = threadIdx.x, item = bulk * (unsigned)T.per_cta + t;
    if ((int)t >= T.per_cta || item >= T.items) return;
    bulk_cells<S, WALLS, FORCED>(T, item);
}

template <bool WALLS, bool MRT>
__global__ void __launch_bounds__(STEP_THREADS, WALLS ? 3 : 4) k_step_h2(const __grid_constant__ StepArgs<__half> T, const __grid_constant__ PairConsts K) {
    extern __shared__ int pre[];
    pdl_wait();
    unsigned bulk;
    if (is_boundary_cta(T, blockIdx.x, &bulk)) {
        boundary_cells<__half, false>(T, (int)(blockIdx.x >> T.bshift), pre);
        return;
    }
    const unsigned t = threadIdx.x, item = bulk * (unsigned)T.per_cta + t;
    if ((int)t >= T.per_cta) return;   // whole warps
    bulk_pairs<WALLS, MRT>(T, K, item, item < T.items);
}

// ------------------------------------------------------------------ remap
__global__ void k_flags_full(uint8_t* __restrict__ flags, GridDesc G, const ParticleState* __restrict__ ps) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= G.n) return;
    const int ij = c % (G.nx * G.ny);
    const int i = ij % G.nx, j = ij / G.nx, k = c / (G.nx * G.ny);
    flags[c] = (ps->present && inside_ball(i, j, k, G, *ps)) ? 1 : 0;
}

// Both copies of the frames of the current record, after the host changed it (128 threads).
__global__ void k_frames(const ParticleState* __restrict__ ps, PFrames* __restrict__ frames, GridDesc G, BoxDesc B) {
    const int n3[3] = {G.nx, G.ny, G.nz};
    pframes_form(frames, *ps, n3, G.periodic, B);
    pframes_form(frames + 1, *ps, n3, G.periodic, B);
}

// Refill of the uncovered cell (i, j, k) = index c by the whole warp
// (Sec. 2.3): lane q = 1..18 takes the neighbour (i, j, k) + c_q (wrapped on
// periodic axes; none beyond a wall), counted when it is fluid before (fcur)
// and after (the ball predicate) the move, with its density 1 + sum_p g_p and
// momentum sum_p c_p g_p (for Grad's strain rate from the face neighbours).
// The mean density and the rigid-body velocity u_p + omega_p x (x - x_p) give
// the equilibrium, plus Grad's term when gcoef != 0; lane q < 19 writes
// population q.  Every lane calls it with the same cell.
template <typename S>
__device__ __forceinline__ void refill_warp(S* pops, const uint8_t* fcur, const GridDesc& G,
                                            const int n3[3], const BoxFrame& F, const ParticleState& P, int i, int j,
                                            int k, typename Store<S>::A scale, typename Store<S>::A inv_scale,
                                            typename Store<S>::A gcoef) {
    using A = typename Store<S>::A;
    const int lane = threadIdx.x & 31;
    const size_t n = (size_t)G.n;
    const size_t c = (size_t)i + (size_t)G.nx * ((size_t)j + (size_t)G.ny * (size_t)k);
    bool ok = false;
    A r = A(0), mo[3] = {A(0), A(0), A(0)};
    if (lane >= 1 && lane < 19) {
        int v[3] = {i + cx(lane), j + cy(lane), k + cz(lane)};
        bool in = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (v[a] < 0 || v[a] >= n3[a]) {
                if (!G.periodic[a]) in = false;
                v[a] = (v[a] + n3[a]) % n3[a];
            }
        }
        if (in && !ball_flag(v, n3, G.periodic, F, P)) {
            const size_t y = (size_t)v[0] + (size_t)G.nx * ((size_t)v[1] + (size_t)G.ny * (size_t)v[2]);
            // the populations are loaded beside the flag (not after it): a solid neighbour's are dropped
            A gp[19];
#pragma unroll
            for (int q = 0; q < 19; ++q) gp[q] = Store<S>::fetch(pops + (size_t)q * n + y, inv_scale);
            ok = fcur[y] == 0;
            r = A(1);
#pragma unroll
            for (int q = 0; q < 19; ++q) r += gp[q];
#pragma unroll
            for (int q = 1; q < 19; ++q) {
                if (cx(q)) mo[0] += cx(q) > 0 ? gp[q] : -gp[q];
                if (cy(q)) mo[1] += cy(q) > 0 ? gp[q] : -gp[q];
                if (cz(q)) mo[2] += cz(q) > 0 ? gp[q] : -gp[q];
            }
        }
    }
    const unsigned okm = __ballot_sync(0xffffffffu, ok);
    A rs = ok ? r : A(0);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, off);
    const int cnt = __popc(okm);
    const A rho = cnt > 0 ? rs / A(cnt) : A(1);
    const double d[3] = {wrap_diff((i + 0.5) - P.x[0], G.nx, G.periodic[0]),
                         wrap_diff((j + 0.5) - P.x[1], G.ny, G.periodic[1]),
                         wrap_diff((k + 0.5) - P.x[2], G.nz, G.periodic[2])};
    const A u[3] = {A(P.u[0] + (P.w[1] * d[2] - P.w[2] * d[1])), A(P.u[1] + (P.w[2] * d[0] - P.w[0] * d[2])),
                    A(P.u[2] + (P.w[0] * d[1] - P.w[1] * d[0]))};
    const A uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    A Sr[6] = {A(0), A(0), A(0), A(0), A(0), A(0)};
    if (gcoef != A(0)) {   // Grad refill: face neighbour q = 1 + 2 a (+1 for -e_a), fluid before and after the move
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
        if (gcoef != A(0)) e += grad_term<A>(q, Sr, gcoef);
        Store<S>::store(pops + (size_t)q * n + c, e, scale);
    }
}

// Remap of Sec. 2.3 after the particle moved, one pass over the box: the new flag of every box cell (the exact
// ball predicate) and its mark; newly covered cells drop their populations (the step stores the cells that were
// solid before as zero); uncovered cells are listed in shared memory and refilled afterwards, each by one warp
// of the block in turn (refill_warp reads only cells that are fluid before and after the move, which nothing
// here writes).  Neighbour flags are evaluated from the same predicate instead of being read back, so flags,
// refill and boundary marks (four launches of 4 to 6 us before) take one pass.  mark_only: only marks and counts
// (flags and populations already belong to the current position).
constexpr int REMAP_THREADS = SEG;
template <typename S>
__global__ void __launch_bounds__(REMAP_THREADS)
    k_remap(S* pops, const uint8_t* fcur, uint8_t* fnext, const __grid_constant__ GridDesc G,
            const __grid_constant__ BoxDesc B, const ParticleState* ps, const PFrames* frames, typename Store<S>::A scale,
            typename Store<S>::A inv_scale, typename Store<S>::A gcoef, uint8_t* mark, int* seg, int* seg_count,
            int mark_only) {
    using A = typename Store<S>::A;
    __shared__ BoxFrame F;
    __shared__ int s_n;
    __shared__ int s_g[3][REMAP_THREADS];   // uncovered cells
    const int n3[3] = {G.nx, G.ny, G.nz};
    pdl_wait();
    if (threadIdx.x == 0) {
        F = frames->bf;
        s_n = 0;
    }
    __syncthreads();
    const ParticleState& P = *ps;
    const size_t n = (size_t)G.n;
    const int t = blockIdx.x * REMAP_THREADS + threadIdx.x;
    bool is_b = false;
    size_t c = 0;
    if (t < B.cells) {
        uint8_t m = MARK_PLAIN;
        int p[3];
        if (box_cell(t, n3, G.periodic, B, F, p)) {
            c = (size_t)p[0] + (size_t)G.nx * ((size_t)p[1] + (size_t)G.ny * (size_t)p[2]);
            const bool was_solid = fcur[c] != 0;
            bool any_nb = false;
            const bool solid = ball_flag_and_neighbours(p, n3, G.periodic, F, P, &any_nb);
            is_b = !solid && any_nb;
            m = solid ? MARK_SOLID : (is_b ? MARK_BOUNDARY : MARK_PLAIN);
            if (!mark_only) {
                fnext[c] = solid ? 1 : 0;
                if (solid && !was_solid) {
#pragma unroll
                    for (int q = 0; q < 19; ++q) Store<S>::store(pops + (size_t)q * n + c, A(0), scale);
                } else if (!solid && was_solid) {
                    const int k = atomicAdd(&s_n, 1);
                    s_g[0][k] = p[0];
                    s_g[1][k] = p[1];
                    s_g[2][k] = p[2];
                }
            }
        }
        mark[t] = m;
    }
    write_segment(is_b, (int)c, (int)blockIdx.x, seg, seg_count);   // its barrier also completes the shared list
    const int wid = threadIdx.x >> 5;
    for (int k = wid; k < s_n; k += REMAP_THREADS / 32)
        refill_warp<S>(pops, fcur, G, n3, F, P, s_g[0][k], s_g[1][k], s_g[2][k], scale, inv_scale, gcoef);
}

// The boundary cells as one list in box order: every block copies its segment behind the cells of the segments before
// it.  Read back for inspection, and by the step itself for boxes with too many segments for a prefix of their numbers
// in shared memory (SEG_CELLS_MAX).
__global__ void __launch_bounds__(SEG)
    k_list_segments(const int* __restrict__ seg, const int* __restrict__ seg_count, int* __restrict__ list,
                    int* __restrict__ count, int capacity, int* __restrict__ status) {
    __shared__ int red[SEG];
    int s = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += SEG) s += seg_count[b];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = SEG / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    const int base = red[0], mine = seg_count[blockIdx.x];
    if ((int)threadIdx.x < mine) {
        const int pos = base + (int)threadIdx.x;
        if (pos >= capacity) atomicOr(status, STATUS_LINK_OVERFLOW);
        else list[pos] = seg[(size_t)blockIdx.x * SEG + threadIdx.x];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *count = min(base + mine, capacity);
}

// Link export for inspection: slot (i*18 + q-1) of the i-th boundary cell
// holds q and delta_q when x + c_q is solid, q = -1 otherwise.
__global__ void k_export_links(const uint8_t* __restrict__ flags, const int* __restrict__ list,
                               const int* __restrict__ count, GridDesc G, const ParticleState* __restrict__ ps,
                               int32_t* __restrict__ q_out, double* __restrict__ delta_out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= *count) return;
    const int cell = list[i];
    const int x = cell % G.nx, y = (cell / G.nx) % G.ny, z = cell / (G.nx * G.ny);
    const ParticleState& P = *ps;
    const double d[3] = {wrap_diff((x + 0.5) - P.x[0], G.nx, G.periodic[0]),
                         wrap_diff((y + 0.5) - P.x[1], G.ny, G.periodic[1]),
                         wrap_diff((z + 0.5) - P.x[2], G.nz, G.periodic[2])};
    const int n3[3] = {G.nx, G.ny, G.nz};
    for (int q = 1; q < 19; ++q) {
        int v[3] = {x + cx(q), y + cy(q), z + cz(q)};
        bool ok = true;
        for (int a = 0; a < 3; ++a) {
            if (v[a] < 0 || v[a] >= n3[a]) {
                if (!G.periodic[a]) ok = false;
                v[a] = (v[a] + n3[a]) % n3[a];
            }
        }
        const size_t slot = (size_t)i * 18 + (q - 1);
        const size_t yy = ok ? (size_t)v[0] + (size_t)G.nx * ((size_t)v[1] + (size_t)G.ny * (size_t)v[2]) : 0;
        if (ok && flags[yy] != 0) {
            q_out[slot] = q;
            delta_out[slot] = link_delta(d, q, P.r);
        } else {
            q_out[slot] = -1;
            delta_out[slot] = 0.0;
        }
    }
}

template <typename S>
__global__ void k_init_eq(S* __restrict__ pops, const uint8_t* __restrict__ flags, GridDesc G, double rho,
                          double u0, double u1, double u2, const double* __restrict__ ufield,
                          typename Store<S>::A scale) {
    using A = typename Store<S>::A;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= G.n) return;
    const size_t n = (size_t)G.n;
    const bool fluid = flags == nullptr || flags[c] == 0;
    double u[3] = {u0, u1, u2};
    if (ufield) {
        u[0] = ufield[c];
        u[1] = ufield[n + c];
        u[2] = ufield[2 * n + c];
    }
    const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        const double cu = dir_dot<double>(q, u[0], u[1], u[2]);
        const double e = wgt<double>(q) * ((rho - 1.0) + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu);
        Store<S>::store(pops + (size_t)q * n + c, fluid ? A(e) : A(0), scale);
    }
}

template <typename S>
__global__ void k_to_f64(const S* __restrict__ pops, double* __restrict__ out, long long count,
                         typename Store<S>::A inv_scale) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = (double)Store<S>::load(pops + i, inv_scale);
}

template <typename S>
__global__ void k_from_f64(const double* __restrict__ in, S* __restrict__ pops, long long count,
                           typename Store<S>::A scale) {
    using A = typename Store<S>::A;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) Store<S>::store(pops + i, (A)in[i], scale);
}

template <typename S>
__global__ void k_gather(const S* __restrict__ pops, long long ncells, const int64_t* __restrict__ cells,
                         long long n, double* __restrict__ out, typename Store<S>::A inv_scale) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * 19) return;
    const long long i = t / 19;
    const int q = (int)(t % 19);
    const long long c = cells[i];
    out[t] = (c >= 0 && c < ncells) ? (double)Store<S>::load(pops + (size_t)q * ncells + c, inv_scale) : 0.0;
}

template <typename S>
__global__ void k_zero_solid(S* __restrict__ pops, const uint8_t* __restrict__ flags, GridDesc G) {
    using A = typename Store<S>::A;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= G.n || flags[c] == 0) return;
    for (int q = 0; q < 19; ++q) Store<S>::store(pops + (size_t)q * G.n + c, A(0), A(1));
}

inline unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ------------------------------------------------------------- launchers
// One coupled step (StepArgs); without a sphere only its bulk part.
template <typename S>
void launch_step(const lbmp_handle* h, const S* src, S* dst, const CollideParams<typename Store<S>::A>& p, int finish,
                 double* force_out, cudaStream_t stream) {
    const GridDesc& g = h->G;
    StepArgs<S> T;
    T.src = src;
    T.dst = dst;
    T.G = g;
    T.P = p;
    T.status = h->status;
    T.bblocks = 0;
    T.finish = finish;
    T.cli = h->cfg.boundary == LBMP_CLI ? 1 : 0;
    T.hist_cap = h->cfg.history_capacity;
    T.flags = h->flags[h->fcur];
    T.mark = h->link_mask;
    T.seg = h->seg;
    T.seg_count = h->seg_count;
    T.fx.set((unsigned)g.nx);
    T.fy.set((unsigned)g.ny);
    T.bshift = 0;
    T.list = nullptr;
    T.count = h->count;
    T.B = h->box;
    T.ps = h->d_ps;
    T.partials = h->partials;
    T.done = h->d_done;
    T.history = h->history;
    T.frames = h->frames + h->frame_cur;
    T.frames_next = h->frames + (1 - h->frame_cur);
    T.force_out = force_out;
    const bool walls = !(g.periodic[0] && g.periodic[1] && g.periodic[2]);
    const bool pairs = std::is_same<S, __half>::value && !p.forced && g.nx % 2 == 0;   // FP16: two cells per thread
    T.dx.set((unsigned)(pairs ? g.nx / 2 : g.nx));
    T.dy.set((unsigned)g.ny);
    T.items = (unsigned)(pairs ? g.n / 2 : g.n);
    // Small grids are spread over the SMs: CTAs of fewer cells until there is one per SM (with two per SM 24^3 cells
    // take 14.5 us a step instead of 13.7, 32^3 15.5 instead of 15.2).
    // FP64: an SM runs one instruction in 19 cycles and a warp of its own one in 64, so three or four busy warps fill
    // it, and two CTAs' registers.  As long as the launch is resident at once, CTAs are made smaller; and up to 2.5
    // rounds the boundary cells go to many CTAs of few busy warps each, not eight warps to an SM: 32^3 cells 38.1 to
    // 25.7 us a step, 40^3 43 to 38, a forward step of the 24^3 gradient 20 to 14.  In longer launches the bulk update
    // fills the SMs anyway (60^3: 66.9 us with one CTA per 32 entries, 71.5 with one per 8).
    auto ctas = [&](int per_cta) { return (T.items + (unsigned)per_cta - 1) / (unsigned)per_cta; };
    T.per_cta = STEP_THREADS;
    if (sizeof(S) != 8)
        while (T.per_cta > 32 && T.items / (unsigned)T.per_cta < SMS) T.per_cta /= 2;
    unsigned bulk = ctas(T.per_cta);
    size_t smem = 0;
    if (h->has_particle) {
        if constexpr (sizeof(S) == 8) {
            T.bblocks = step_boundary_blocks(h->list_cap, BOUNDARY_PER_FP64);
            T.thin = bulk + (unsigned)T.bblocks <= 5 * SMS;
            if (!T.thin) T.bblocks = step_boundary_blocks(h->list_cap, bulk >= BULK_LONG ? 40 : 32);
        } else {
            T.bblocks = step_boundary_blocks(h->list_cap, bulk >= BULK_LONG ? 40 : BOUNDARY_PER);
        }
        if (step_uses_list(h->box)) T.list = h->list;
        else smem = sizeof(int) * (size_t)((h->box.cells + SEG - 1) / SEG + 1);
    }
    if (sizeof(S) == 8) {
        while (T.per_cta > 32 && (unsigned)T.bblocks + ctas(T.per_cta / 2) <= 2 * SMS) T.per_cta /= 2;
        bulk = ctas(T.per_cta);
    }
    const unsigned grid = (unsigned)T.bblocks + bulk;
    // Boundary CTAs wait on latencies: up to three bulk CTAs between two of them keep the memory busy meanwhile (a
    // sphere of 40 cells has 900, more than a wave).
    while (T.bshift < 2 && (unsigned)T.bblocks << (T.bshift + 1) <= grid) ++T.bshift;
    auto go = [&](auto kernel) { launch_pdl(kernel, grid, STEP_THREADS, smem, stream, T); };
    if constexpr (std::is_same<S, __half>::value) {
        if (pairs) {
            const bool mrt = p.db != 0.0f;
            const PairConsts K = pair_consts(p);
            auto go2 = [&](auto kernel) { launch_pdl(kernel, grid, STEP_THREADS, smem, stream, T, K); };
            if (walls && mrt) go2(k_step_h2<true, true>);
            else if (walls) go2(k_step_h2<true, false>);
            else if (mrt) go2(k_step_h2<false, true>);
            else go2(k_step_h2<false, false>);
            return;
        }
    }
    // FP32: a bulk update of more than four waves waits on HBM and wants five CTAs per SM (48 registers, some spilled in
    // the boundary cells: 512^3 2990 us a step, 3095 with four; 88^3 21.3 and 21.7).  In a shorter one the boundary
    // cells' chain counts, which four (64 registers) shorten: 32^3 15.2 -> 14.8 us a step, 64 x 64 x 128 with MRT 20.9
    // -> 19.5, 84^3 20.0 -> 19.3.
    auto pick = [&](auto ctas) {
        constexpr int C = decltype(ctas)::value;
        if (walls && p.forced) go(k_step<S, true, true, C>);
        else if (walls) go(k_step<S, true, false, C>);
        else if (p.forced) go(k_step<S, false, true, C>);
        else go(k_step<S, false, false, C>);
    };
    if constexpr (std::is_same<S, float>::value) {
        if (bulk > 4 * 4 * SMS) pick(std::integral_constant<int, 5>());
        else pick(std::integral_constant<int, 4>());
    } else {
        pick(std::integral_constant<int, sizeof(S) == 8 ? 2 : 4>());
    }
}

void launch_flags_full(uint8_t* flags, const GridDesc& g, const ParticleState* ps, cudaStream_t stream) {
    k_flags_full<<<blocks_for(g.n, 256), 256, 0, stream>>>(flags, g, ps);
}

size_t frames_bytes() { return 2 * sizeof(PFrames); }

void launch_frames(const lbmp_handle* h, cudaStream_t stream) {
    k_frames<<<1, 128, 0, stream>>>(h->d_ps, h->frames, h->G, h->box);
}

// Remap to the position of frames[frame] (fcur -> fnext); mark_only for the marks alone.  Large boxes: also the list.
template <typename S>
int launch_remap(const lbmp_handle* h, S* pops, const uint8_t* fcur, uint8_t* fnext, int frame, bool mark_only,
                 typename Store<S>::A scale, typename Store<S>::A inv_scale, typename Store<S>::A gcoef,
                 cudaStream_t stream) {
    const PFrames* F = h->frames + frame;
    launch_pdl(k_remap<S>, blocks_for(h->box.cells, REMAP_THREADS), REMAP_THREADS, 0, stream, pops, fcur, fnext, h->G,
               h->box, (const ParticleState*)h->d_ps, F, scale, inv_scale, gcoef, h->link_mask, h->seg, h->seg_count,
               mark_only ? 1 : 0);
    if (!step_uses_list(h->box)) return 1;
    launch_list_segments(h, stream);
    return 2;
}

void launch_list_segments(const lbmp_handle* h, cudaStream_t stream) {
    k_list_segments<<<blocks_for(h->box.cells, SEG), SEG, 0, stream>>>(h->seg, h->seg_count, h->list, h->count, h->list_cap,
                                                                      h->status);
}

void launch_export_links(const uint8_t* flags, const int* list, const int* count, int max_cells, const GridDesc& g,
                         const ParticleState* ps, int cli, int32_t* q_out, double* delta_out, cudaStream_t stream) {
    (void)cli;
    if (max_cells <= 0) return;
    k_export_links<<<blocks_for(max_cells, 128), 128, 0, stream>>>(flags, list, count, g, ps, q_out, delta_out);
}

template <typename S>
void launch_init_equilibrium(S* pops, const uint8_t* flags, const GridDesc& g, double rho, const double u[3],
                             const double* u_field, typename Store<S>::A scale, cudaStream_t stream) {
    k_init_eq<S><<<blocks_for(g.n, 256), 256, 0, stream>>>(pops, flags, g, rho, u[0], u[1], u[2], u_field, scale);
}

template <typename S>
void launch_to_f64(const S* pops, double* out, long long count, typename Store<S>::A inv_scale,
                   cudaStream_t stream) {
    k_to_f64<S><<<blocks_for(count, 256), 256, 0, stream>>>(pops, out, count, inv_scale);
}

template <typename S>
void launch_from_f64(const double* in, S* pops, long long count, typename Store<S>::A scale, cudaStream_t stream) {
    k_from_f64<S><<<blocks_for(count, 256), 256, 0, stream>>>(in, pops, count, scale);
}

template <typename S>
void launch_gather(const S* pops, long long ncells, const int64_t* cells, long long n, double* out,
                   typename Store<S>::A inv_scale, cudaStream_t stream) {
    if (n <= 0) return;
    k_gather<S><<<blocks_for(n * 19, 256), 256, 0, stream>>>(pops, ncells, cells, n, out, inv_scale);
}

template <typename S>
void launch_zero_solid(S* pops, const uint8_t* flags, const GridDesc& g, cudaStream_t stream) {
    k_zero_solid<S><<<blocks_for(g.n, 256), 256, 0, stream>>>(pops, flags, g);
}

#define LBMP_INSTANTIATE(S)                                                                                        \
    template void launch_step<S>(const lbmp_handle*, const S*, S*, const CollideParams<Store<S>::A>&, int, double*, \
                                 cudaStream_t);                                                                    \
    template int launch_remap<S>(const lbmp_handle*, S*, const uint8_t*, uint8_t*, int, bool, Store<S>::A,         \
                                 Store<S>::A, Store<S>::A, cudaStream_t);                                          \
    template void launch_init_equilibrium<S>(S*, const uint8_t*, const GridDesc&, double, const double*,           \
                                             const double*, Store<S>::A, cudaStream_t);                            \
    template void launch_to_f64<S>(const S*, double*, long long, Store<S>::A, cudaStream_t);                       \
    template void launch_from_f64<S>(const double*, S*, long long, Store<S>::A, cudaStream_t);                      \
    template void launch_zero_solid<S>(S*, const uint8_t*, const GridDesc&, cudaStream_t);                       \
    template void launch_gather<S>(const S*, long long, const int64_t*, long long, double*, Store<S>::A,           \
                                   cudaStream_t);

LBMP_INSTANTIATE(double)
LBMP_INSTANTIATE(float)
LBMP_INSTANTIATE(__half)

}  // namespace lbmp
