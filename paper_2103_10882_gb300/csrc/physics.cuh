// Device arithmetic shared by the uniform and the refined-grid kernels:
// TRT collision on deviations (Sec. 2.1) and the sphere-link geometry of
// the CLI boundary (Sec. 2.3).
#pragma once

#include <cstddef>

#include "internal.h"

namespace lbmp {

// Programmatic dependent launch (PTX griddepcontrol): the CTAs of a kernel launched with the attribute may become
// resident once every CTA of the kernel ahead has ended or called pdl_trigger; pdl_wait returns when that kernel has
// completed and its writes are visible.  Every thread waits before it reads or writes global memory, so only the
// launch itself overlaps; loads are ordinary ones (Store::fetch).
// No kernel triggers at its start: CTAs that become resident while the kernel ahead still runs take the slots that
// happen to be free, several of the first, longest ones on one SM, instead of one on each.  Without the attribute, with
// a trigger at the start, and with none, a 32^3 FP32 step takes 19.3, 16.9 and 15.5 us, a 24^3 FP64 gradient 1.80, 2.92
// and 1.79 ms, 256 x 128 x 96 with walls 91.8, 89.2 and 87.4 us a step.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Minimum-image difference for periodic axes.
__device__ __forceinline__ double wrap_diff(double d, int n, int periodic) {
    if (!periodic) return d;
    double L = (double)n;
    if (d > 0.5 * L) d -= L;
    else if (d < -0.5 * L) d += L;
    return d;
}

// Wall distance fraction along c_q from the fluid cell centre (Sec. 2.3):
// smallest root in (0,1] of |d + s c|^2 = r^2.
__device__ __forceinline__ double link_delta(const double d[3], int q, double r) {
    double c0 = cx(q), c1 = cy(q), c2 = cz(q);
    double cc = c0 * c0 + c1 * c1 + c2 * c2;
    double dc = d[0] * c0 + d[1] * c1 + d[2] * c2;
    double dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    double disc = dc * dc - cc * (dd - r * r);
    disc = disc < 0.0 ? 0.0 : disc;
    double s = (-dc - sqrt(disc)) / cc;
    return s < 0.0 ? 0.0 : (s > 1.0 ? 1.0 : s);
}

// c_q . u for a direction known at compile time, without the products by zero (which the compiler may
// not drop in IEEE arithmetic: 0 * inf); the value is the same.
template <typename A>
__device__ __forceinline__ A dir_dot(int q, A x, A y, A z) {
    const int a = cx(q), b = cy(q), c = cz(q);
    A t = A(0);
    bool any = false;
    if (a) {
        t = a > 0 ? x : -x;
        any = true;
    }
    if (b) {
        t = any ? (b > 0 ? t + y : t - y) : (b > 0 ? y : -y);
        any = true;
    }
    if (c) t = any ? (c > 0 ? t + z : t - z) : (c > 0 ? z : -z);
    return t;
}

// The collision of trt_collide with the fewest instructions, for FP64, whose time is instructions (an SM issues one FP64
// warp instruction in 19 cycles, a warp by itself one in 64: at 242 of them per cell the update ran at that rate,
// 0.51e12 a second).  With the sums ps and differences pd of the opposite pairs, both new populations of a pair are
// S + D and S - D,
//   S = (1 - s+)/2 ps + s+ e+ + (1 - s+/2) S+,   D = (1 - s-)/2 pd + s- e- + (1 - s-/2) S-,
// the coefficients and the direction's part of the Guo source come from the host (collide_consts), the density part of
// e+ and the MRT correction are one number per class of directions: 121 instructions per cell unforced (13 more forced).
// (1 - s+)/2 is exact for s+ in [1/2, 2] (below, tau above 2, its rounding scales a cell's density by up to 6e-17 a
// step, where that of the weights does by 1.1e-16 at tau 0.5); (1 - s-)/2 is not for s- < 1/2, and its rounding would
// change every cell's momentum by the same relative 6e-17 in every step, so pd/2 - (s-/2) pd takes two operations.
// Measured: a coupled FP64 step of 61 x 53 x 75 cells 175 -> 129 us, a refined FP64 step (1.1 M updates) 394 -> 261 us.
// The MRT sums over a class follow from ps alone: sum_faces 2 e+ = rho/3, sum_edges 2 e+ = rho/3 + uu/2, and the half
// source sums to -uF/2, 0 and uF/2 over rest, faces and edges.
// FP32 and FP16 storage keep the plain form below (collide_pair: two cells in one): their kernels wait on memory as much
// as on instructions, and in FP32 arithmetic the rounded coefficient would be a relative 1.5e-8 to 6e-8 a step.
template <typename A, bool FORCED>
__device__ __forceinline__ void collide_direct(A (&g)[19], const CollideParams<A>& P, int* status) {
    const CollideConsts<A>& K = P.k;
    A ps[9], pd[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        ps[k] = g[2 * k + 1] + g[2 * k + 2];
        pd[k] = g[2 * k + 1] - g[2 * k + 2];
    }
    const A pF = ps[0] + ps[1] + ps[2];
    const A pE = ((ps[3] + ps[4]) + (ps[5] + ps[6])) + (ps[7] + ps[8]);
    const A drho = g[0] + pF + pE;
    // pairs 3..8 are (+x+y), (+x-y), (+x+z), (+x-z), (+y+z), (+y-z)
    A ux = pd[0] + ((pd[3] + pd[4]) + (pd[5] + pd[6]));
    A uy = pd[1] + ((pd[3] - pd[4]) + (pd[7] + pd[8]));
    A uz = pd[2] + ((pd[5] - pd[6]) + (pd[7] - pd[8]));
    if (FORCED) {
        ux += A(0.5) * P.F[0];
        uy += A(0.5) * P.F[1];
        uz += A(0.5) * P.F[2];
    }
    const A u2[3] = {ux * ux, uy * uy, uz * uz};
    const A uu = u2[0] + u2[1] + u2[2];
    if (!(uu <= A(0.09))) atomicOr(status, STATUS_UNSTABLE_FLUID);
    A R = P.sp * (drho - K.c15 * uu);
    A uF = A(0);
    if (FORCED) {
        uF = ux * P.F[0] + uy * P.F[1] + uz * P.F[2];
        R -= K.cF * uF;
    }
    A bF = wgt<A>(1) * R, bE = wgt<A>(7) * R, b0 = wgt<A>(0) * R;
    if (P.db != A(0)) {   // MRT, as in trt_collide
        const A t = drho * (A(1) / A(3)), u3 = K.c15 * (A(1) / A(3)) * uu;   // u3 = uu / 2
        A nR = g[0] - t + u3;
        const A nF = pF - t;
        A nE = pE - t - u3;
        if (FORCED) {
            nR -= A(0.5) * uF;
            nE += A(0.5) * uF;
        }
        const A c4 = A(1.5) * (nE - nR);
        const A c16 = A(0.5) * (nR - A(2) * nF + nE);
        b0 -= P.db * wgt<A>(0) * (c16 - c4);
        bF -= P.db * wgt<A>(1) * (A(-2) * c16);
        bE -= P.db * wgt<A>(7) * (c4 + c16);
    }
    g[0] = K.r0 * g[0] + b0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int q = 2 * k + 1;
        const bool face = k < 3;
        const A cu = dir_dot<A>(q, ux, uy, uz);
        A e, d;
        if (FORCED) {
            e = ((face ? K.kF : K.kE) * cu + K.gs[k]) * cu + (face ? bF : bE);
            d = (face ? K.mF : K.mE) * cu + K.ga[k];
        } else {
            e = face ? K.kF * u2[k < 3 ? k : 0] + bF : (K.kE * cu) * cu + bE;
            d = (face ? K.mF : K.mE) * cu;
        }
        const A Sy = K.hp * ps[k] + e;
        const A Da = (A(0.5) * pd[k] + d) - K.hsm * pd[k];
        g[q] = Sy + Da;
        g[q + 1] = Sy - Da;
    }
}

// TRT collision on deviations (Sec. 2.1, Lambda_b = 1): the symmetric part of
// each pair relaxes with s+, the antisymmetric part with s-; incompressible
// equilibrium with rho_0 = 1; optional Guo-type source split the same way.
// SCALED: g holds the deviations times 2^s (FP16 storage kept in its scaled
// form); the collision is linear in g except for the equilibrium's two
// quadratic terms, which then take one factor 2^-s (P.inv_scale).
template <typename A, bool FORCED, bool SCALED = false>
__device__ __forceinline__ void trt_collide(A (&g)[19], const CollideParams<A>& P, int* status) {
    static_assert(!(FORCED && SCALED), "the scaled form is for the unforced collision");
    if constexpr (sizeof(A) == 8) {
        collide_direct<A, FORCED>(g, P, status);
        return;
    }
    const A q2 = SCALED ? P.inv_scale : A(1);
    A drho = A(0), jx = A(0), jy = A(0), jz = A(0);
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        drho += g[q];
        if (cx(q) == 1) jx += g[q];
        if (cx(q) == -1) jx -= g[q];
        if (cy(q) == 1) jy += g[q];
        if (cy(q) == -1) jy -= g[q];
        if (cz(q) == 1) jz += g[q];
        if (cz(q) == -1) jz -= g[q];
    }
    A ux = jx, uy = jy, uz = jz;
    if (FORCED) {
        ux += A(0.5) * P.F[0];
        uy += A(0.5) * P.F[1];
        uz += A(0.5) * P.F[2];
    }
    const A uu = (ux * ux + uy * uy + uz * uz) * q2;
    if (!(uu * q2 <= A(0.09))) atomicOr(status, STATUS_UNSTABLE_FLUID);
    const A sp = P.sp, sm = P.sm;
    const bool mrt = P.db != A(0);
    // MRT bulk correction: sums of (f - f_eq + source/2) over the rest,
    // face and edge populations (the even modes' inputs)
    A nR = A(0), nF = A(0), nE = A(0);
    {
        const A e0 = wgt<A>(0) * (drho - A(1.5) * uu);
        if (mrt) nR = g[0] - e0;
        A o = g[0] - sp * (g[0] - e0);
        if (FORCED) {
            const A uF = ux * P.F[0] + uy * P.F[1] + uz * P.F[2];
            o += (A(1) - A(0.5) * sp) * wgt<A>(0) * (A(-3) * uF);
            if (mrt) nR += A(0.5) * wgt<A>(0) * (A(-3) * uF);
        }
        g[0] = o;
    }
#pragma unroll
    for (int q = 1; q < 19; q += 2) {
        const A cu = dir_dot<A>(q, ux, uy, uz);
        const A w = wgt<A>(q);
        const A ep = w * (drho + A(4.5) * q2 * cu * cu - A(1.5) * uu);
        const A em = w * (A(3) * cu);
        const A gp = A(0.5) * (g[q] + g[q + 1]);
        const A gm = A(0.5) * (g[q] - g[q + 1]);
        const A dp = sp * (gp - ep);
        const A dm = sm * (gm - em);
        if (mrt) {
            if (q < 7) nF += A(2) * (gp - ep);
            else nE += A(2) * (gp - ep);
        }
        A a = g[q] - dp - dm;
        A b = g[q + 1] - dp + dm;
        if (FORCED) {
            const A cF = dir_dot<A>(q, P.F[0], P.F[1], P.F[2]);
            const A uF = ux * P.F[0] + uy * P.F[1] + uz * P.F[2];
            const A Sp = (A(1) - A(0.5) * sp) * w * (A(9) * cu * cF - A(3) * uF);
            const A Sm = (A(1) - A(0.5) * sm) * w * (A(3) * cF);
            a += Sp + Sm;
            b += Sp - Sm;
            if (mrt) {   // half the symmetric source of the pair
                const A hs = w * (A(9) * cu * cF - A(3) * uF);
                if (q < 7) nF += hs;
                else nE += hs;
            }
        }
        g[q] = a;
        g[q + 1] = b;
    }
    if (mrt) {
        // MRT of Sec. 2.1 = TRT with the bulk mode e4 = |c|^2 - 1 and the
        // isotropic fourth-order mode e16 = 3|c|^4 - 6|c|^2 + 1 relaxed at s_b
        // instead of s+: subtract (s_b - s+) w_q sum_k e_k(q) c_k with
        // c_k = sum_p e_k(p) (f - f_eq + source/2)_p / sum_p w_p e_k(p)^2
        // (e4: rest -1, faces 0, edges 1, norm 2/3; e16: rest 1, faces -2,
        // edges 1, norm 2).
        const A c4 = A(1.5) * (nE - nR);
        const A c16 = A(0.5) * (nR - A(2) * nF + nE);
        g[0] -= P.db * wgt<A>(0) * (c16 - c4);
        const A df = P.db * wgt<A>(1) * (A(-2) * c16);
        const A de = P.db * wgt<A>(7) * (c4 + c16);
#pragma unroll
        for (int q = 1; q < 7; ++q) g[q] -= df;
#pragma unroll
        for (int q = 7; q < 19; ++q) g[q] -= de;
    }
}

}  // namespace lbmp

namespace lbmp {

// Warp-cooperative TRT collision: lane q (< 19) holds population q of one
// cell; lanes 19..31 hold 0 and take part in the shuffles.  Returns the
// post-collision value of the lane's population (same arithmetic as
// trt_collide, reduced across the warp).
template <typename A>
__device__ __forceinline__ A warp_sum(A v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

__device__ __forceinline__ int lane_c(int lane, int axis) {
    const int q = lane < 19 ? lane : 0;   // c_q component (0 for idle lanes)
    return axis == 0 ? cx(q) : (axis == 1 ? cy(q) : cz(q));
}

template <typename A, bool FORCED>
__device__ __forceinline__ A warp_trt_collide(A gq, int lane, const CollideParams<A>& P, int* status) {
    const int c0 = lane_c(lane, 0), c1 = lane_c(lane, 1), c2 = lane_c(lane, 2);
    const A drho = warp_sum<A>(gq);
    A ux = warp_sum<A>(A(c0) * gq), uy = warp_sum<A>(A(c1) * gq), uz = warp_sum<A>(A(c2) * gq);
    if (FORCED) {
        ux += A(0.5) * P.F[0];
        uy += A(0.5) * P.F[1];
        uz += A(0.5) * P.F[2];
    }
    const A uu = ux * ux + uy * uy + uz * uz;
    if (lane == 0 && !(uu <= A(0.09))) atomicOr(status, STATUS_UNSTABLE_FLUID);
    const int partner = lane == 0 ? 0 : (lane < 19 ? ((lane & 1) ? lane + 1 : lane - 1) : lane);
    const A gb = __shfl_sync(0xffffffffu, gq, partner);
    const A w = lane == 0 ? A(1) / A(3) : (lane <= 6 ? A(1) / A(18) : A(1) / A(36));
    const A cu = A(c0) * ux + A(c1) * uy + A(c2) * uz;
    const A ep = w * (drho + A(4.5) * cu * cu - A(1.5) * uu);
    const A em = w * (A(3) * cu);
    const A gp = A(0.5) * (gq + gb), gm = A(0.5) * (gq - gb);
    A out = gq - P.sp * (gp - ep) - P.sm * (gm - em);
    A v = gq - ep - em;   // f - f_eq of the lane (the odd part drops out of the even sums below)
    if (FORCED) {
        const A cF = A(c0) * P.F[0] + A(c1) * P.F[1] + A(c2) * P.F[2];
        const A uF = ux * P.F[0] + uy * P.F[1] + uz * P.F[2];
        out += (A(1) - A(0.5) * P.sp) * w * (A(9) * cu * cF - A(3) * uF) + (A(1) - A(0.5) * P.sm) * w * (A(3) * cF);
        v += A(0.5) * w * (A(9) * cu * cF - A(3) * uF);
    }
    if (P.db != A(0)) {   // MRT bulk correction, as in trt_collide (uniform across the warp)
        const A e4 = lane == 0 ? A(-1) : (lane <= 6 ? A(0) : (lane < 19 ? A(1) : A(0)));
        const A e16 = lane == 0 ? A(1) : (lane <= 6 ? A(-2) : (lane < 19 ? A(1) : A(0)));
        const A c4 = A(1.5) * warp_sum<A>(e4 * v);
        const A c16 = A(0.5) * warp_sum<A>(e16 * v);
        out -= P.db * w * (e4 * c4 + e16 * c16);
    }
    return lane < 19 ? out : A(0);
}

// Particle quantities the link kernels need, converted once per block
// (thread 0 fills a shared copy): Xi = floor(X) and Xh = 1/2 - (X - Xi), so
// the offset of a cell centre p + 1/2 from the centre X is (p - Xi) + Xh
// without cancellation in A; radius and velocities u(t + 1/2), omega(t + 1/2) in A.
template <typename A>
struct LinkFrame {
    int Xi[3];
    A Xh[3], r, u[3], w[3];
    __device__ __forceinline__ void init(const ParticleState& P) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double f = floor(P.x[a]);
            Xi[a] = (int)f;
            Xh[a] = A(0.5 - (P.x[a] - f));
            u[a] = A(P.u[a]);
            w[a] = A(P.w[a]);
        }
        r = A(P.r);
    }
    // d = p + 1/2 - X for cell p (minimum image on periodic axes) and the
    // matching unwrapped coordinate pu, with d = pu + 1/2 - X.
    __device__ __forceinline__ void offset(const int p[3], const int n[3], const int periodic[3], A d[3],
                                           int pu[3]) const {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int v = p[a];
            if (periodic[a]) {
                const A t = A(v - Xi[a]) + Xh[a];
                const A half = A(0.5) * A(n[a]);
                v += t > half ? -n[a] : (t < -half ? n[a] : 0);
            }
            pu[a] = v;
            d[a] = A(v - Xi[a]) + Xh[a];
        }
    }
};

// CLI link of Sec. 2.3 for the fluid cell at offset d from the sphere
// centre, incoming direction q (k = opp(q) points into the solid): returns
// the new deviation g_q and the link's momentum-exchange force and torque
// without their lattice-weight part.  On full populations f = w + g the
// link force is (c_k - v) f~_k + (c_k + v) f_q = 2 w_k c_k + fl with
// fl = (c_k - v) g~_k + (c_k + v) g_q; the 2 w_k c_k part (and its torque
// d x 2 w_k c_k) is summed exactly by LinkSums.  Geometry and fl are
// evaluated in the arithmetic type A of the populations (FP64 on the FP64
// path); use_delta = false takes the wall half-way (delta = 1/2).
// Every product and sum of the link is rounded as written (fma_rn, mul_rn: the compiler neither contracts nor splits
// them), so the uniform, refined and batched steps get the same bits from the same populations.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// Wall distance delta along c_k (k = opp(q)) from the cell at offset d and
// the CLI coefficients kappa0 = (1 - 2 delta) / (1 + 2 delta) and
// alpha = 4 / (1 + 2 delta) of Sec. 2.3; use_delta = false takes delta = 1/2.
template <typename A>
__device__ __forceinline__ void cli_coeffs(int q, const A d[3], bool use_delta, A r, A* delta_out, A* kappa0,
                                           A* alpha) {
    const int k = opp(q);
    A delta = A(0.5);
    if (use_delta) {   // smallest root in (0,1] of |d + s c_k|^2 = r^2 (|c_k|^2 is 1 or 2)
        const A dc = d[0] * A(cx(k)) + d[1] * A(cy(k)) + d[2] * A(cz(k));   // products by 0 and +-1 are exact
        const A e = fma_rn(-r, r, fma_rn(d[2], d[2], fma_rn(d[0], d[0], mul_rn(d[1], d[1]))));
        const bool face = k <= 6;
        A disc = fma_rn(dc, dc, face ? -e : A(-2) * e);
        disc = disc < A(0) ? A(0) : disc;
        const A s = (-dc - sqrt(disc)) * (face ? A(1) : A(0.5));
        delta = s < A(0) ? A(0) : (s > A(1) ? A(1) : s);
    }
    const A inv = A(1) / fma_rn(A(2), delta, A(1));
    *delta_out = delta;
    *kappa0 = mul_rn(fma_rn(A(-2), delta, A(1)), inv);
    *alpha = A(4) * inv;
}

// The part of a link that needs no populations: kappa0, alpha 3 w_k, v.c_k, the arm and the wall velocity v at the
// link's wall point.  A caller forms it while the populations are still on their way.
template <typename A>
struct CliGeometry {
    A kappa0, aw, vc, arm[3], vb[3];
};

template <typename A>
__device__ __forceinline__ A cross_term(A a, A b, A c, A d) { return fma_rn(a, b, -mul_rn(c, d)); }   // ab - cd

template <typename A>
__device__ __forceinline__ CliGeometry<A> cli_geometry(int q, const A d[3], bool use_delta, const LinkFrame<A>& Fr) {
    const int k = opp(q);
    const A c[3] = {A(cx(k)), A(cy(k)), A(cz(k))};
    CliGeometry<A> L;
    A delta, alpha;
    cli_coeffs<A>(q, d, use_delta, Fr.r, &delta, &L.kappa0, &alpha);
#pragma unroll
    for (int a = 0; a < 3; ++a) L.arm[a] = fma_rn(delta, c[a], d[a]);
    L.vb[0] = Fr.u[0] + cross_term(Fr.w[1], L.arm[2], Fr.w[2], L.arm[1]);
    L.vb[1] = Fr.u[1] + cross_term(Fr.w[2], L.arm[0], Fr.w[0], L.arm[2]);
    L.vb[2] = Fr.u[2] + cross_term(Fr.w[0], L.arm[1], Fr.w[1], L.arm[0]);
    L.vc = L.vb[0] * c[0] + L.vb[1] * c[1] + L.vb[2] * c[2];
    const A wk3 = k <= 6 ? A(1) / A(6) : A(1) / A(12);   // 3 w_k
    L.aw = mul_rn(alpha, wk3);
    return L;
}

template <typename A>
__device__ __forceinline__ A cli_apply(int q, const CliGeometry<A>& L, A gt_k, A gt_q, A gt_far, A fl[3], A tl[3]) {
    const int k = opp(q);
    const A c[3] = {A(cx(k)), A(cy(k)), A(cz(k))};
    const A gnew = fma_rn(-L.aw, L.vc, fma_rn(-L.kappa0, gt_q, fma_rn(L.kappa0, gt_far, gt_k)));
#pragma unroll
    for (int a = 0; a < 3; ++a) fl[a] = fma_rn(c[a] - L.vb[a], gt_k, mul_rn(c[a] + L.vb[a], gnew));
    tl[0] = cross_term(L.arm[1], fl[2], L.arm[2], fl[1]);
    tl[1] = cross_term(L.arm[2], fl[0], L.arm[0], fl[2]);
    tl[2] = cross_term(L.arm[0], fl[1], L.arm[1], fl[0]);
    return gnew;
}

// Per-lane sums of the link forces and torques of one particle.  fl and tl
// of every link are added in the arithmetic type A; in FP32 each running
// sum carries its rounding error (Knuth's TwoSum, exact for every
// addition), so a lane's sum is exact to far below FP32 resolution without
// the slow FP64 pipe.  The block sum is formed in FP64.  The lattice-weight part
// 2 w_k c_k is summed in integers: 36 * 2 w_k is 4 on faces and 2 on edges,
// and its torque (pu + 1/2 - X) x 2 w_k c_k is carried as
// (2 pu + 1) x (36 * 2 w_k c_k) over 72 minus X x (the force part), so it
// cancels exactly wherever the links close around the body.
template <typename A>
struct LinkSums {
    A F[3] = {A(0), A(0), A(0)}, T[3] = {A(0), A(0), A(0)};
    A eF[3] = {A(0), A(0), A(0)}, eT[3] = {A(0), A(0), A(0)};   // FP32: rounding errors of F and T
    int iF[3] = {0, 0, 0};
    long long iT[3] = {0, 0, 0};

    __device__ static __forceinline__ void sum2(A& s, A& e, A x) {
        if constexpr (sizeof(A) == 8) {
            s += x;
        } else {
            const A t = s + x, xv = t - s;
            e += (s - (t - xv)) + (x - xv);
            s = t;
        }
    }
    __device__ __forceinline__ void add(int k, const int pu[3], const A fl[3], const A tl[3]) {
        const int m = k <= 6 ? 4 : 2;
        const int mc[3] = {m * cx(k), m * cy(k), m * cz(k)};
        const long long p2[3] = {2LL * pu[0] + 1, 2LL * pu[1] + 1, 2LL * pu[2] + 1};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            sum2(F[a], eF[a], fl[a]);
            sum2(T[a], eT[a], tl[a]);
            iF[a] += mc[a];
        }
        iT[0] += p2[1] * mc[2] - p2[2] * mc[1];
        iT[1] += p2[2] * mc[0] - p2[0] * mc[2];
        iT[2] += p2[0] * mc[1] - p2[1] * mc[0];
    }
};

__device__ __forceinline__ double pick3(const double v[3], int i) { return i == 0 ? v[0] : (i == 1 ? v[1] : v[2]); }

// Double-float addition (h, l) += (bh, bl): Knuth's TwoSum of the leading
// parts, the trailing parts added to its error, renormalised (Fast2Sum).
// About 44 significant bits, in FP32 arithmetic.
__device__ __forceinline__ void df_add(float& h, float& l, float bh, float bl) {
    const float s = h + bh, v = s - h;
    const float e = ((h - (s - v)) + (bh - v)) + (l + bl);
    h = s + e;
    l = e - (h - s);
}

// Deterministic block sum of the threads' link sums into out[c * stride], c = 0..5: force,
// and torque about X (best in shared memory: it is read last).  Every thread of the block must call it.  FP64
// additions, and conversions to FP64, are slow and narrow on this GPU, so
// in FP32 the lanes' sums (each with its TwoSum error) are reduced as
// double-float pairs, a butterfly within each warp and, after one barrier,
// one across the warps' results by warps 0..5 (one component each); only
// lane 0 of those warps converts to FP64.  In FP64 the six components are
// staged in shared memory and warp c adds column l of the warp rows
// pairwise in lane l, then across the lanes.  The integer parts are summed
// exactly by shuffles, and the constant divisions are multiplications by
// the reciprocals.  A last-block hand-off after this call is ordered by its
// barrier and release (the writers need no fence of their own).
template <int NT, typename A>
__device__ __forceinline__ void block_link_sums(const LinkSums<A>& acc, const double X[3], double* __restrict__ out,
                                                int stride) {
    static_assert(NT % 32 == 0 && NT >= 192 && NT <= 1024, "six warps take the six components");
    constexpr int NW = NT / 32;
    constexpr int SPAN = NW <= 8 ? 8 : (NW <= 16 ? 16 : 32);   // lanes of the cross-warp butterfly
    __shared__ long long si[6][NW];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    // integers: exact warp sums by redux.sync, the torque parts in two halves of 16 low bits and the rest
    long long iv[6];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        iv[a] = __reduce_add_sync(0xffffffffu, acc.iF[a]);
        const int lo = __reduce_add_sync(0xffffffffu, (int)(acc.iT[a] & 0xffff));
        const int hi = __reduce_add_sync(0xffffffffu, (int)(acc.iT[a] >> 16));
        iv[3 + a] = ((long long)hi << 16) + lo;
    }
    if (lane == 0)
#pragma unroll
        for (int c = 0; c < 6; ++c) si[c][wid] = iv[c];
    double t;
    int c;
    if constexpr (sizeof(A) == 4) {
        __shared__ float sh[6][NW], sl[6][NW];
        // eight slots (six used) exchanged so that each step halves what a lane carries: 9 additions and 18 shuffles
        // where six butterflies take 30 and 60; component c ends in lane 4 c
        float h[8], l[8];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            h[a] = acc.F[a] + acc.eF[a];
            l[a] = acc.eF[a] - (h[a] - acc.F[a]);
            h[3 + a] = acc.T[a] + acc.eT[a];
            l[3 + a] = acc.eT[a] - (h[3 + a] - acc.T[a]);
        }
        h[6] = h[7] = l[6] = l[7] = 0.0f;
#pragma unroll
        for (int off = 16, m = 4; m >= 1; off >>= 1, m >>= 1) {
            const bool up = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < m; ++i) {
                const float sh_ = up ? h[i] : h[i + m], sl_ = up ? l[i] : l[i + m];
                if (up) {
                    h[i] = h[i + m];
                    l[i] = l[i + m];
                }
                const float oh = __shfl_xor_sync(0xffffffffu, sh_, off), ol = __shfl_xor_sync(0xffffffffu, sl_, off);
                df_add(h[i], l[i], oh, ol);
            }
        }
#pragma unroll
        for (int off = 2; off > 0; off >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, h[0], off), ol = __shfl_xor_sync(0xffffffffu, l[0], off);
            df_add(h[0], l[0], oh, ol);
        }
        if ((lane & 3) == 0 && lane < 24) {
            sh[lane >> 2][wid] = h[0];
            sl[lane >> 2][wid] = l[0];
        }
        __syncthreads();
        if (wid >= 6) return;
        c = wid;
        float th = lane < NW ? sh[c][lane] : 0.0f, tl = lane < NW ? sl[c][lane] : 0.0f;
#pragma unroll
        for (int off = SPAN / 2; off > 0; off >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, th, off), ol = __shfl_xor_sync(0xffffffffu, tl, off);
            df_add(th, tl, oh, ol);
        }
        if (lane != 0) return;
        t = (double)th + (double)tl;
    } else {
        __shared__ double sd[6][NT];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            sd[a][tid] = acc.F[a];
            sd[3 + a][tid] = acc.T[a];
        }
        __syncthreads();
        if (wid >= 6) return;
        c = wid;
        double v[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) v[w] = sd[c][lane + 32 * w];
#pragma unroll
        for (int st = 1; st < NW; st <<= 1)
#pragma unroll
            for (int w = 0; w + st < NW; w += 2 * st) v[w] += v[w + st];
        t = v[0];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (lane != 0) return;
    }
    long long iF[3] = {0, 0, 0}, iT = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        iF[0] += si[0][w];
        iF[1] += si[1][w];
        iF[2] += si[2][w];
        iT += si[c][w];
    }
    const double r36 = 1.0 / 36.0, r72 = 1.0 / 72.0;
    const double fr[3] = {(double)iF[0] * r36, (double)iF[1] * r36, (double)iF[2] * r36};
    if (c < 3) {
        out[(size_t)c * stride] = t + pick3(fr, c);
    } else {
        const int a1 = c == 3 ? 1 : (c == 4 ? 2 : 0), a2 = c == 3 ? 2 : (c == 4 ? 0 : 1);
        out[(size_t)c * stride] = t + ((double)iT * r72 - (X[a1] * pick3(fr, a2) - X[a2] * pick3(fr, a1)));
    }
}

__device__ __forceinline__ int src_coord(int x, int c, int n, int periodic) {
    int s = x - c;
    if (s < 0) return periodic ? s + n : -1;
    if (s >= n) return periodic ? s - n : -1;
    return s;
}

// Cell centre p + 1/2 inside the closed ball |p + 1/2 - X| <= r: the flag
// definition, evaluated in FP64 with explicit round-to-nearest products and
// sums (no contraction), minimum image on periodic axes.
__device__ __forceinline__ bool inside_ball_exact(const int p[3], const int n[3], const int periodic[3],
                                                  const ParticleState& P) {
    const double dx = wrap_diff(__dsub_rn((double)p[0] + 0.5, P.x[0]), n[0], periodic[0]);
    const double dy = wrap_diff(__dsub_rn((double)p[1] + 0.5, P.x[1]), n[1], periodic[1]);
    const double dz = wrap_diff(__dsub_rn((double)p[2] + 0.5, P.x[2]), n[2], periodic[2]);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return d2 <= __dmul_rn(P.r, P.r);
}

__device__ __forceinline__ bool inside_ball(int i, int j, int k, const GridDesc& G, const ParticleState& P) {
    const int p[3] = {i, j, k}, n[3] = {G.nx, G.ny, G.nz};
    return inside_ball_exact(p, n, G.periodic, P);
}

// Per-block constants of the kernels that walk the box of cells around the
// sphere (cell o + t for t in [0, E) per axis, o from the current centre),
// filled once by thread 0 (all of their FP64 set-up work): the box
// origin and an FP32 pre-test of the ball predicate.  The FP32 squared
// distance (p - Xi + Xh)^2 differs from the FP64 one by less than
// 1e-6 (|d|^2 + 1); cells whose estimate lies below lo = r^2 - 1e-5 (r^2 + 1)
// are inside, above hi = r^2 + 1e-5 (r^2 + 1) outside, and only the thin shell
// in between evaluates inside_ball_exact, so every flag equals the FP64
// definition.
struct BoxFrame {
    int o[3];      // first box cell per axis (0 where the box spans a periodic axis)
    int Xi[3];     // floor(X)
    float Xh[3];   // 1/2 - (X - Xi)
    float lo, hi;
};

__device__ __forceinline__ void box_frame_init(BoxFrame& F, const int n[3], const int periodic[3], const BoxDesc& B,
                                               const ParticleState& P) {
    bool wide = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // a centre that is not finite or absurdly far (only after an unstable step, which the
        // status word reports) is replaced so that the integer box arithmetic stays in range
        const double x = fabs(P.x[a]) < 1e9 ? P.x[a] : 0.0;
        F.o[a] = (B.E[a] >= n[a]) ? 0 : (int)floor(x - 0.5) - B.R;
        const double f = floor(x);
        F.Xi[a] = (int)f;
        F.Xh[a] = (float)(0.5 - (x - f));
        // a sphere reaching within two cells of half a period: the FP32 tests skip minimum images
        wide |= periodic[a] && (P.r > 0.4 * n[a] || P.r + 2.0 >= 0.5 * n[a]);
    }
    const double rr = P.r * P.r, m = 1e-5 * (rr + 1.0);
    F.lo = wide ? -1.0f : (float)(rr - m);   // a sphere this wide takes the FP64 path everywhere
    F.hi = wide ? 3.0e38f : (float)(rr + m);
}

// Both frames of the sphere's current state (the link frame in FP32 and in
// FP64, and the box frame), formed once per step by the particle update, or
// after the host changed the record, and read by the box kernels of the
// refined step instead of each of their blocks forming them from the FP64
// record (FP64 is slow on this part, and every block waited for it).
__device__ __forceinline__ double particle_mass(const ParticleState& P);
__device__ __forceinline__ double particle_inertia(const ParticleState& P);

struct PFrames {
    LinkFrame<float> lf;
    LinkFrame<double> ld;
    BoxFrame bf;
    double inv[2];   // 1/m and 1/I (particle_mass, particle_inertia): fixed between changes by the host
};

template <typename A>
__device__ __forceinline__ const LinkFrame<A>& pframe_link(const PFrames& F) {
    if constexpr (sizeof(A) == 8) return F.ld;
    else return F.lf;
}

// Forms F from the record P: the three frames by lane 0 of warps 0, 1 and 2
// of the calling block (each is one FP64 sequence), the inverses by lanes 0
// and 1 of warp 3; every thread of a block of at least 128 calls it.
__device__ __forceinline__ void pframes_form(PFrames* __restrict__ F, const ParticleState& P, const int n[3],
                                             const int periodic[3], const BoxDesc& B) {
    if (threadIdx.x == 0) F->lf.init(P);
    else if (threadIdx.x == 32) F->ld.init(P);
    else if (threadIdx.x == 64) box_frame_init(F->bf, n, periodic, B, P);
    else if (threadIdx.x == 96) F->inv[0] = 1.0 / particle_mass(P);
    else if (threadIdx.x == 97) F->inv[1] = 1.0 / particle_inertia(P);
}

// |v| as an integer that orders like it (NaN above infinity).
__device__ __forceinline__ long long abs_bits(double v) { return __double_as_longlong(v) & 0x7fffffffffffffffll; }

// The parts of F that follow the sphere along axis a after the particle update, positions (part 0) and velocities
// (part 1) by different warps: the same values as pframes_form, from a shorter FP64 sequence (floor by one conversion,
// the box origin from the fraction); the radius and the FP32 pre-test bounds do not change during a run and keep the
// values pframes_form gave them.
__device__ __forceinline__ void pframes_axis(PFrames* __restrict__ F, const ParticleState& P, const int n[3],
                                             const BoxDesc& B, int a, int part) {
    if (part == 1) {
        F->lf.u[a] = (float)P.u[a];
        F->lf.w[a] = (float)P.w[a];
        F->ld.u[a] = P.u[a];
        F->ld.w[a] = P.w[a];
        return;
    }
    const double xr = P.x[a];
    const bool sane = abs_bits(xr) < abs_bits(1e9);   // as box_frame_init: keep the box arithmetic in range
    const int xi = __double2int_rd(xr);
    const double frac = xr - (double)xi;
    const int bi = sane ? xi : 0;
    const double bfrac = sane ? frac : 0.0;
    const double xh = 0.5 - frac;
    F->lf.Xi[a] = xi;
    F->ld.Xi[a] = xi;
    F->ld.Xh[a] = xh;
    F->lf.Xh[a] = (float)xh;
    F->bf.Xi[a] = bi;
    F->bf.Xh[a] = (float)(0.5 - bfrac);
    // floor(x - 1/2): x - 1/2 and x - floor(x) are exact
    F->bf.o[a] = (B.E[a] >= n[a]) ? 0 : (bfrac < 0.5 ? bi - 1 : bi) - B.R;
}

// Box cell t (x fastest) -> cell p; false where the box leaves a wall-bounded axis.
__device__ __forceinline__ bool box_cell(int t, const int n[3], const int periodic[3], const BoxDesc& B,
                                         const BoxFrame& F, int p[3]) {
    const int e0 = B.E[0], e1 = B.E[1];
    const int tk = t / (e0 * e1);
    const int r = t - tk * e0 * e1;
    const int tj = r / e0;
    const int tt[3] = {r - tj * e0, tj, tk};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int v = F.o[a] + tt[a];
        if (v < 0 || v >= n[a]) {
            if (!periodic[a]) return false;
            v = v < 0 ? v + n[a] : v - n[a];   // the box is never wider than the domain
            if (v < 0 || v >= n[a]) return false;   // a centre outside the domain: touch nothing
        }
        p[a] = v;
    }
    return true;
}

__device__ __forceinline__ bool ball_flag(const int p[3], const int n[3], const int periodic[3], const BoxFrame& F,
                                          const ParticleState& P) {
    float e = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int v = p[a] - F.Xi[a];
        if (periodic[a]) {
            const float t = (float)v + F.Xh[a], half = 0.5f * (float)n[a];
            v += t > half ? -n[a] : (t < -half ? n[a] : 0);
        }
        const float t = (float)v + F.Xh[a];
        e = fmaf(t, t, e);
    }
    if (e < F.lo) return true;
    if (e > F.hi) return false;
    return inside_ball_exact(p, n, periodic, P);
}

// Solid flag of cell p and whether any of its 18 D3Q19 neighbours is solid,
// both as defined by the exact ball predicate.  The neighbours' FP32
// squared distances follow from the cell's own FP32 offset t as
// (t + c_q)^2, one more rounding per component than ball_flag, well inside
// the same margin; undecided cells take the FP64 expression at the wrapped
// neighbour position.  A box wider than half a period takes the FP64 path
// everywhere (lo < 0, see box_frame_init), so no minimum image is needed for
// the neighbours here.
__device__ __forceinline__ bool ball_flag_and_neighbours(const int p[3], const int n[3], const int periodic[3],
                                                         const BoxFrame& F, const ParticleState& P, bool* any_nb) {
    float t[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int v = p[a] - F.Xi[a];
        if (periodic[a]) {
            const float u = (float)v + F.Xh[a], half = 0.5f * (float)n[a];
            v += u > half ? -n[a] : (u < -half ? n[a] : 0);
        }
        t[a] = (float)v + F.Xh[a];
    }
    const float e0 = fmaf(t[2], t[2], fmaf(t[1], t[1], t[0] * t[0]));
    const bool own = e0 < F.lo ? true : (e0 > F.hi ? false : inside_ball_exact(p, n, periodic, P));
    bool any = false;
#pragma unroll
    for (int q = 1; q < 19; ++q) {
        const float a0 = t[0] + (float)cx(q), a1 = t[1] + (float)cy(q), a2 = t[2] + (float)cz(q);
        const float e = fmaf(a2, a2, fmaf(a1, a1, a0 * a0));
        if (e < F.lo) any = true;
        else if (e <= F.hi && !any) {
            int v[3] = {p[0] + cx(q), p[1] + cy(q), p[2] + cz(q)};
            bool ok = true;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (v[a] < 0 || v[a] >= n[a]) {
                    if (!periodic[a]) ok = false;
                    v[a] = v[a] < 0 ? v[a] + n[a] : v[a] - n[a];
                }
            }
            if (ok && inside_ball_exact(v, n, periodic, P)) any = true;
        }
    }
    *any_nb = any;
    return own;
}

// m = (rho_p + C_v) V and I = 2/5 (rho_p + C_vw) V r^2 (Sec. 2.2: virtual mass and moment of inertia).
__device__ __forceinline__ double particle_mass(const ParticleState& P) { return (P.rho_p + P.cv) * P.V; }
__device__ __forceinline__ double particle_inertia(const ParticleState& P) {
    return 0.4 * (P.rho_p + P.cvw) * P.V * P.r * P.r;
}

// One axis a of Algorithm 1's particle update, translation and rotation each by a thread of its own (of different
// warps: a scheduler issues one FP64 instruction in about 76 cycles): average of the hydrodynamic force or torque over
// two steps, gravity/buoyancy (Fg) and the virtual force (Fv) or torque (Tv) from the previous accelerations, and the
// kick-drift-kick update with the virtually increased mass or moment of inertia, whose inverses the caller passes.
// A held group (translation; rotation) keeps its velocity and records zero acceleration, so the virtual force or
// torque after it is zero; a group released in this step starts afresh, with no half kick completing a previous step.
// Both return false for a jump or a non-finite state (!(|x - xold| <= 1/2), !(|u| < 1/2); !(|w| < 1e30)), compared as
// integers, which order non-negative doubles alike and put NaN above infinity.

__device__ __forceinline__ void wrap_centre(ParticleState& P, int a, const GridDesc& G) {   // into the periodic box
    const int n = a == 0 ? G.nx : (a == 1 ? G.ny : G.nz);
    if (G.periodic[a]) {
        const double L = (double)n;
        if (P.x[a] >= L) P.x[a] -= L;
        else if (P.x[a] < 0.0) P.x[a] += L;
    }
}

__device__ __forceinline__ bool advance_translation(ParticleState& P, int a, double Fh, double Fg, double Fv, double inv_m,
                                                    const GridDesc& G) {
    const bool avg = P.force_average && P.steps > 0;
    const double Fbar = avg ? 0.5 * (Fh + P.Fh_old[a]) : Fh;
    P.Fh[a] = Fh;
    P.Fh_old[a] = Fh;
    const double Fp = Fbar + Fg + Fv;
    P.Fp[a] = Fp;
    const double xold = P.x[a];
    const double acc = Fp * inv_m;
    if (P.fixed == 0) {
        double u = P.u[a];
        if (P.steps > 0 && P.prev_fixed == 0) u += 0.5 * acc;   // second half kick of the previous step completes u(t)
        u += 0.5 * acc;   // first half kick, then drift with u(t + 1/2)
        P.a[a] = acc;
        P.u[a] = u;
        P.x[a] = xold + u;
    } else {
        P.a[a] = 0.0;
    }
    const bool ok = abs_bits(P.x[a] - xold) <= abs_bits(0.5) && abs_bits(P.u[a]) < abs_bits(0.5);
    if (ok) wrap_centre(P, a, G);
    return ok;
}

__device__ __forceinline__ bool advance_rotation(ParticleState& P, int a, double Th, double Tv, double inv_I) {
    const bool avg = P.force_average && P.steps > 0;
    const double Tbar = avg ? 0.5 * (Th + P.Th_old[a]) : Th;
    P.Th[a] = Th;
    P.Th_old[a] = Th;
    const double Tp = Tbar + Tv;
    const double bet = Tp * inv_I;
    if (P.fixed != 1) {
        double w = P.w[a];
        if (P.steps > 0 && P.prev_fixed != 1) w += 0.5 * bet;
        w += 0.5 * bet;
        P.b[a] = bet;
        P.w[a] = w;
    } else {
        P.b[a] = 0.0;
    }
    return abs_bits(P.w[a]) < abs_bits(1e30);
}

// Sum of component comp over the nblocks force partials ([component][block]) by one warp, in a fixed order (every lane
// gets it).
__device__ __forceinline__ double sum_partials(const double* partials, int nblocks, int comp) {
    const int lane = threadIdx.x & 31;
    // Lane l sums partials l, l + 64, ... into s0 and l + 32, l + 96, ... into s1, in that
    // order; eight loads at a time are issued before their sums
    double s0 = 0.0, s1 = 0.0;
    for (int base = 0; base < nblocks; base += 256) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int b = base + lane + 32 * k;
            v[k] = b < nblocks ? __ldcg(partials + (size_t)comp * nblocks + b) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            if (base + lane + 32 * k < nblocks) s0 += v[k];
            if (base + lane + 32 * (k + 1) < nblocks) s1 += v[k + 1];
        }
    }
    double t = s0 + s1;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
}

// Particle update by one block of NT >= 256 threads once the nblocks force
// partials ([component][block]) are complete: warps 0..5 sum one component
// each in a fixed order (lane l takes partials l, l + 32, ... in two
// alternating sums, then a butterfly runs across the lanes), warp 6 forms
// 1/m, 1/I and the forces known beforehand, warp 7 stages the record in
// shared memory.  Then warp 0 advances the translation and warp 1 the
// rotation, a lane per axis, and all of the block writes record and history.
// The partials may come from other blocks of the same launch: they are read
// through L2.  Every thread of the block must call it.
// after(P, a, part): called with the advanced record (in shared memory) by the lanes of warp 2 (part 0, for what
// follows the position) and of warp 3 (part 1, the velocities), a lane per axis.
// Measured on the rising sphere's boundary launch: 3.7 us when one warp advanced both groups and all else followed it.
struct NoAfter {
    __device__ __forceinline__ void operator()(const ParticleState&, int, int) const {}
};
template <int NT, typename After = NoAfter>
__device__ __forceinline__ void particle_block_update(ParticleState* __restrict__ ps, const double* partials,
                                                      int nblocks, const GridDesc& G, double* __restrict__ history,
                                                      int hist_cap, int* __restrict__ status,
                                                      const double* __restrict__ inv = nullptr, After after = After{}) {
    static_assert(NT % 32 == 0 && NT >= 256, "eight warps share the work");
    constexpr int words = (int)(sizeof(ParticleState) / sizeof(int));
    __shared__ double sFT[6], sinv[2], sFg[3], sFv[3], sTv[3];
    __shared__ ParticleState sP;
    __shared__ double xold[3];
    __shared__ int bad[2][3];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < 6) {
        const double t = sum_partials(partials, nblocks, wid);
        if (lane == 0) sFT[wid] = t;
    } else if (wid == 6) {
        if (lane < 2) {
            sinv[lane] = inv ? inv[lane] : 1.0 / (lane == 0 ? particle_mass(*ps) : particle_inertia(*ps));
        } else if (lane >= 8 && lane < 11) {
            const int a = lane - 8;
            const double V = ps->V, r = ps->r;
            sFg[a] = (ps->rho_p - 1.0) * ps->g[a] * V;
            sFv[a] = ps->cv * V * ps->a[a];
            sTv[a] = 0.4 * ps->cvw * V * r * r * ps->b[a];
            xold[a] = ps->x[a];
        }
    } else if (wid == 7) {
        const int* srcw = reinterpret_cast<const int*>(ps);
        int* dstw = reinterpret_cast<int*>(&sP);
#pragma unroll 4
        for (int i = lane; i < words; i += 32) dstw[i] = __ldcg(srcw + i);
    }
    __syncthreads();
    if (wid == 0 && lane < 3) bad[0][lane] = !advance_translation(sP, lane, sFT[lane], sFg[lane], sFv[lane], sinv[0], G);
    if (wid == 1 && lane < 3) bad[1][lane] = !advance_rotation(sP, lane, sFT[3 + lane], sTv[lane], sinv[1]);
    __syncthreads();
    if ((bad[0][0] | bad[0][1] | bad[0][2] | bad[1][0] | bad[1][1] | bad[1][2]) != 0) {   // uniform across the block
        // a jump or a non-finite state: flag it, and keep the sphere where it was and at rest, so that
        // the box kernels that follow until the host reads the status stay inside the domain
        const int a = threadIdx.x;
        if (a < 3 && (bad[0][a] | bad[1][a])) {
            atomicOr(status, STATUS_PARTICLE_JUMP);
            sP.x[a] = xold[a];
            sP.u[a] = sP.w[a] = sP.a[a] = sP.b[a] = 0.0;
            wrap_centre(sP, a, G);
        }
        __syncthreads();
    }
    if (wid == 2 && lane < 3) after(sP, lane, 0);
    if (wid == 3 && lane < 3) after(sP, lane, 1);
    if (wid == 0 && lane < 15 && hist_cap > 0) {   // F_hyd, T_hyd, x_p, u_p, omega_p
        const int a = lane % 3, f = lane / 3;
        const double v = f == 0 ? sP.Fh[a] : (f == 1 ? sP.Th[a] : (f == 2 ? sP.x[a] : (f == 3 ? sP.u[a] : sP.w[a])));
        history[(size_t)(sP.steps % hist_cap) * 15 + lane] = v;
    }
    {
        const int* srcw = reinterpret_cast<const int*>(&sP);
        int* dstw = reinterpret_cast<int*>(ps);
        constexpr int at_steps = (int)(offsetof(ParticleState, steps) / sizeof(int));
        constexpr int at_prev = (int)(offsetof(ParticleState, prev_fixed) / sizeof(int));
        for (int i = (int)threadIdx.x - 128; i >= 0 && i < words; i += NT - 128) {
            int v = srcw[i];
            if (i == at_steps) v = (int)(unsigned)(unsigned long long)(sP.steps + 1);
            if (i == at_steps + 1) v = (int)((sP.steps + 1) >> 32);
            if (i == at_prev) v = sP.fixed;
            dstw[i] = v;
        }
    }
}


// Grad refill of an uncovered cell (Sec. 2.3: the paper uses Dorschner et
// al.'s approach, read as Grad's approximation from the local strain rate).
// Strain rate S (xx, yy, zz, xy, yz, xz) from the six face neighbours'
// velocities: central differences where both are fluid, one-sided against
// the wall velocity uw where one is, zero where neither is.  nb(a, sgn, u)
// returns whether the face neighbour x + sgn e_a is fluid (before and after
// the move) and, if so, its velocity in u.
template <typename A, typename NB>
__device__ __forceinline__ void refill_strain(NB&& nb, const A uw[3], A S[6]) {
    A G[3][3];   // G[a][b] = d u_b / d x_a
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        A up[3], um[3];
        const bool okp = nb(a, 1, up), okm = nb(a, -1, um);
#pragma unroll
        for (int b = 0; b < 3; ++b)
            G[a][b] = (okp && okm) ? A(0.5) * (up[b] - um[b]) : (okp ? up[b] - uw[b] : (okm ? uw[b] - um[b] : A(0)));
    }
    S[0] = G[0][0];
    S[1] = G[1][1];
    S[2] = G[2][2];
    S[3] = A(0.5) * (G[0][1] + G[1][0]);
    S[4] = A(0.5) * (G[1][2] + G[2][1]);
    S[5] = A(0.5) * (G[0][2] + G[2][0]);
}

// Grad's non-equilibrium part of population q of a refilled post-collision
// state: gcoef w_q Q_q:S with Q_q = c_q c_q - I/3 and gcoef = -3 (1 - s+)/s+
// (the first-order Chapman-Enskog stress after one collision).
template <typename A>
__device__ __forceinline__ A grad_term(int q, const A S[6], A gcoef) {
    const A x = A(cx(q)), y = A(cy(q)), z = A(cz(q));
    const A qs = x * x * S[0] + y * y * S[1] + z * z * S[2] + A(2) * (x * y * S[3] + y * z * S[4] + x * z * S[5]) -
                 (S[0] + S[1] + S[2]) / A(3);
    return gcoef * wgt<A>(q) * qs;
}

// Last-block-done hand-off: each of nblocks blocks calls it after writing
// its partials; the block that finishes last (a device counter, reset by
// that block) gets true.  No block waits for another.  The block barrier
// followed by thread 0's acquire-release atomic at GPU scope publishes the
// partials of all the block's threads and, in the last block, makes the
// other blocks' partials visible (read them through L2).
__device__ __forceinline__ bool last_block_done(int* counter, int nblocks) {
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        int old;
        asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(counter) : "memory");
        last = old == nblocks - 1;
        if (last) *counter = 0;
    }
    __syncthreads();
    return last != 0;
}

// Exclusive prefix of n counts into pre[0..n] (pre[n] = total), computed by
// the whole CTA (NT threads, two consecutive counts per thread and pass);
// every thread must call it.  first0, first1: counts 2 threadIdx.x and
// 2 threadIdx.x + 1 (0 beyond n), loaded by the caller ahead.
template <int NT>
__device__ __forceinline__ int block_prefix(const int* __restrict__ count, int n, int* pre, int first0, int first1) {
    __shared__ int wsum[NT / 32];
    __shared__ int carry;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < n; base += 2 * NT) {
        const int i = base + 2 * (int)threadIdx.x;
        const int c0 = base == 0 ? first0 : (i < n ? count[i] : 0);
        const int c1 = base == 0 ? first1 : (i + 1 < n ? count[i + 1] : 0);
        int v = c0 + c1;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, v, off);
            if (lane >= off) v += y;
        }
        if (lane == 31) wsum[wid] = v;
        __syncthreads();
        if (wid == 0) {
            int w = lane < NT / 32 ? wsum[lane] : 0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, w, off);
                if (lane >= off) w += y;
            }
            if (lane < NT / 32) wsum[lane] = w;
        }
        __syncthreads();
        const int incl = carry + (wid > 0 ? wsum[wid - 1] : 0) + v;   // through count i + 1
        if (i < n) pre[i + 1] = incl - c1;
        if (i + 1 < n) pre[i + 2] = incl;
        __syncthreads();
        if (threadIdx.x == 0) carry += wsum[NT / 32 - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) pre[0] = 0;
    __syncthreads();
    return pre[n];
}

// Boundary cells in segments: the remap CTA of 256 box cells writes its marked cells, in box order, to the first
// entries of its own 256, and their number.  A prefix of the numbers then gives the j-th boundary cell in one look-up
// (a mask byte per box cell and a count per 64 took a binary search, two mask loads and a bit scan: 2,000 cycles of
// the 5,500 that a boundary cell took).
constexpr int SEG = 256;

// The segment of boundary cell j: the largest s with pre[s] <= j, by the whole warp (two or a few ballots).
__device__ __forceinline__ int find_segment(const int* pre, int nseg, int j) {
    const int lane = threadIdx.x & 31;
    const int step = (nseg + 31) >> 5;
    const int at = lane * step;
    const unsigned b = __ballot_sync(0xffffffffu, at < nseg && pre[at] <= j);
    const int base = (__popc(b) - 1) * step;   // pre[0] = 0 <= j
    int s = base;
    for (int off = 0; off < step; off += 32) {
        const int i = base + off + lane;
        const unsigned m = __ballot_sync(0xffffffffu, off + lane < step && i < nseg && pre[i] <= j);
        if (m == 0u) break;
        s = base + off + __popc(m) - 1;
    }
    return s;
}

// Writes the block's marked cells (is_b, entry) into its segment.  Every thread of a block of SEG calls it.
__device__ __forceinline__ void write_segment(bool is_b, int entry, int segment, int* __restrict__ seg,
                                              int* __restrict__ seg_count) {
    __shared__ int wsum[SEG / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned ballot = __ballot_sync(0xffffffffu, is_b);
    if (lane == 0) wsum[wid] = __popc(ballot);
    __syncthreads();
    int base = 0, total = 0;
#pragma unroll
    for (int w = 0; w < SEG / 32; ++w) {
        if (w < wid) base += wsum[w];
        total += wsum[w];
    }
    if (is_b) seg[(size_t)segment * SEG + base + __popc(ballot & ((1u << lane) - 1u))] = entry;
    if (threadIdx.x == 0) seg_count[segment] = total;
}

}  // namespace lbmp
