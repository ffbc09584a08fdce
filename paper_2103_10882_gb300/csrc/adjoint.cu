// Reverse-mode derivative of the mean drag on a fixed sphere.
//
// Objective: J = (1/N) sum_{n=1..N} F_a^n, the mean over N steps of one
// component of the momentum-exchange force (Sec. 2.3) on a sphere held at
// rest in a periodic box, with respect to the relaxation time tau (through
// s+ = 1/tau and s- of the magic parameter, Sec. 2.1), the fluid body force
// F and the initial velocity field u0 (the fluid starts at the equilibrium
// of u0).
//
// With h^n = S(g^{n-1}) the streamed (pre-collision) field, g^n = C(h^n) the
// post-collision field and F^n = sum over links (x, q) of
// c_k (2 w_k + g^{n-1}_k(x) + h^n_q(x)), k = opp(q), the adjoint fields
// nu^n = dJ/dh^n and lambda^n = dJ/dg^n obey
//     lambda^n = S^T nu^{n+1} + (1/N) sum_links c_k,a e_(x,k)      (n < N)
//     nu^n     = (dC/dh (h^n))^T lambda^n + (1/N) sum_links c_k,a e_(x,q)
// with lambda^N = 0, and
//     dJ/dtau = sum_n lambda^n . dC/dtau (h^n),  dJ/dF = sum_n lambda^n . dC/dF (h^n),
//     dJ/du0  = (dE/du0)^T lambda^0.
// S^T is streaming run backwards: a pull along -c_q, with the CLI terms of
// every link moved to the cells they read.  One kernel per reverse step
// forms lambda and nu cell by cell: it gathers nu^{n+1} from x + c_q and
// recomputes h^n from the stored g^{n-1}, so only the post-collision
// fields are kept: every interval-th one from the forward pass, the rest
// recomputed segment by segment (checkpoint and recompute).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "adjoint.h"
#include "internal.h"
#include "physics.cuh"

namespace lbmp {
namespace {

constexpr int AT = 256;   // threads per block of the cell kernels
constexpr int NEAR_WARPS_MAX = 32 * SMS;   // warps for the cells next to the sphere (4,864, each takes several of a large sphere's)

// Threads of a reverse-step CTA, and resident CTAs per SM asked of the compiler: 56 registers in FP32 (64^3
// 2% faster per gradient than 64), 128 in FP64.
// In FP64 an SM runs one instruction in 19 cycles and a warp of its own one in 64, so three or four busy warps fill it:
// CTAs of two warps, all resident, even out what each SM gets, 25 us a step of 24^3 cells (1,700 instructions on an SM,
// 17 us).  Of 256 threads, one per SM, its 500 CTAs took 3.3 rounds, 57 us.  FP32 at 64^3 16.2 ms per gradient with
// CTAs of 128 threads, 16.6 with 256.
template <typename S>
constexpr int ADJ_THREADS = sizeof(S) == 8 ? 64 : 128;
template <typename S>
constexpr int ADJ_MIN_CTAS = sizeof(S) == 8 ? 8 : 9;

enum : uint8_t { KIND_PLAIN = 0, KIND_SOLID = 1, KIND_NEAR = 2 };

template <typename A>
struct AdjParams {
    A sp, sm, F[3];
    A seed;      // 1/N
    int axis;    // force component of the objective
};

__device__ __forceinline__ int wrapc(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

__device__ __forceinline__ long long cell_at(const GridDesc& G, int i, int j, int k) {
    return (long long)wrapc(i, G.nx) + (long long)G.nx * ((long long)wrapc(j, G.ny) + (long long)G.ny * wrapc(k, G.nz));
}

// Moments that the transposed collision needs: of h the density and velocity (with half the force), of lambda
//   L0 = sum w lambda, L1 = sum w lambda c, L2 = sum w lambda c c^T (xx yy zz xy xz yz).
template <typename A>
struct AdjMoments {
    A drho, u[3], L0, L1[3], L2[6];
};

// What every population of the cell shares: a0 and b of
//   (dC/dh)^T lambda = lambda - s+ lambda+ - s- lambda- + a0 + b.c with
//   a0 = s+ L0, b = s+ (9 L2 u - 3 L0 u) + 3 s- L1 + (1 - s+/2)(9 L2 F - 3 L0 F),
// and the force parts lambda . dC/dF.  The source is always differentiated, also where F = 0.
template <typename A>
__device__ __forceinline__ void adj_shared(const AdjMoments<A>& M, const AdjParams<A>& P, A* a0, A b[3], A dF[3]) {
    const A* L2 = M.L2;
    const A* u = M.u;
    const A L2u[3] = {L2[0] * u[0] + L2[3] * u[1] + L2[4] * u[2], L2[3] * u[0] + L2[1] * u[1] + L2[5] * u[2],
                      L2[4] * u[0] + L2[5] * u[1] + L2[2] * u[2]};
    const A L2F[3] = {L2[0] * P.F[0] + L2[3] * P.F[1] + L2[4] * P.F[2],
                      L2[3] * P.F[0] + L2[1] * P.F[1] + L2[5] * P.F[2],
                      L2[4] * P.F[0] + L2[5] * P.F[1] + L2[2] * P.F[2]};
    *a0 = P.sp * M.L0;
    const A L03 = A(3) * M.L0, hs = A(1) - A(0.5) * P.sp, hm = A(3) * (A(1) - A(0.5) * P.sm);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const A du = A(9) * L2u[a] - L03 * u[a];
        b[a] = P.sp * du + A(3) * P.sm * M.L1[a] + hs * (A(9) * L2F[a] - L03 * P.F[a]);
        dF[a] = A(0.5) * b[a] + hs * du + hm * M.L1[a];
    }
}

// Transpose of the TRT collision with the Guo-type source (the derivative of trt_collide at h, applied to lambda) on
// one cell, and the parameter parts part = (lambda . dC/ds+, lambda . dC/ds-, lambda . dC/dF), with
//   C_q(h) = h_q - s+ (h+_q - e+_q) - s- (h-_q - e-_q) + (1 - s+/2) S+_q + (1 - s-/2) S-_q,
//   dC_q/ds+ = -(h+_q - e+_q) - S+_q / 2, dC_q/ds- = -(h-_q - e-_q) - S-_q / 2.
// All on the sums and differences of the opposite pairs, without products by zero components: about 300
// instructions instead of 470, which is the time in FP64.
template <typename A>
__device__ __forceinline__ void trt_adjoint(const A (&h)[19], A (&lam)[19], const AdjParams<A>& P, A part[5]) {
    A hp[9], hm[9], lp[9], lm[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        hp[k] = h[2 * k + 1] + h[2 * k + 2];
        hm[k] = h[2 * k + 1] - h[2 * k + 2];
        lp[k] = lam[2 * k + 1] + lam[2 * k + 2];
        lm[k] = lam[2 * k + 1] - lam[2 * k + 2];
    }
    // pairs 0..2 are the faces, 3..8 (+x+y), (+x-y), (+x+z), (+x-z), (+y+z), (+y-z)
    AdjMoments<A> M;
    M.drho = h[0] + (((hp[0] + hp[1]) + hp[2]) + (((hp[3] + hp[4]) + (hp[5] + hp[6])) + (hp[7] + hp[8])));
    M.u[0] = (hm[0] + ((hm[3] + hm[4]) + (hm[5] + hm[6]))) + A(0.5) * P.F[0];
    M.u[1] = (hm[1] + ((hm[3] - hm[4]) + (hm[7] + hm[8]))) + A(0.5) * P.F[1];
    M.u[2] = (hm[2] + ((hm[5] - hm[6]) + (hm[7] - hm[8]))) + A(0.5) * P.F[2];
    const A wF = wgt<A>(1), wE = wgt<A>(7);
    const A exy = lp[3] + lp[4], exz = lp[5] + lp[6], eyz = lp[7] + lp[8];
    M.L0 = wgt<A>(0) * lam[0] + wF * ((lp[0] + lp[1]) + lp[2]) + wE * ((exy + exz) + eyz);
    M.L1[0] = wF * lm[0] + wE * ((lm[3] + lm[4]) + (lm[5] + lm[6]));
    M.L1[1] = wF * lm[1] + wE * ((lm[3] - lm[4]) + (lm[7] + lm[8]));
    M.L1[2] = wF * lm[2] + wE * ((lm[5] - lm[6]) + (lm[7] - lm[8]));
    M.L2[0] = wF * lp[0] + wE * (exy + exz);
    M.L2[1] = wF * lp[1] + wE * (exy + eyz);
    M.L2[2] = wF * lp[2] + wE * (exz + eyz);
    M.L2[3] = wE * (lp[3] - lp[4]);
    M.L2[4] = wE * (lp[5] - lp[6]);
    M.L2[5] = wE * (lp[7] - lp[8]);
    A a0, b[3];
    adj_shared<A>(M, P, &a0, b, part + 2);
    const A* u = M.u;
    const A uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const A uF = u[0] * P.F[0] + u[1] * P.F[1] + u[2] * P.F[2];
    const A r = M.drho - A(1.5) * uu + A(1.5) * uF;   // e+ - S+/2 without its direction-dependent part, over w
    A tsp = lam[0] * (wgt<A>(0) * r - h[0]), tsm = A(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int q = 2 * k + 1;
        const A w = wgt<A>(q);
        const A cu = dir_dot<A>(q, u[0], u[1], u[2]);
        const A cF = dir_dot<A>(q, P.F[0], P.F[1], P.F[2]);   // the same in every cell
        const A v = A(4.5) * (cu - cF);
        tsp += lp[k] * (w * (v * cu + r) - A(0.5) * hp[k]);
        tsm += lm[k] * ((A(3) * w) * (cu - A(0.5) * cF) - A(0.5) * hm[k]);
        const A bc = dir_dot<A>(q, b[0], b[1], b[2]);
        // x, y = lambda+ (1 - s+) + a0 +- (lambda- (1 - s-) + b.c)
        const A hl = A(0.5) * lp[k];
        const A Sy = hl - P.sp * hl + a0;
        const A gl = A(0.5) * lm[k];
        const A Da = gl - P.sm * gl + bc;
        lam[q] = Sy + Da;
        lam[q + 1] = Sy - Da;
    }
    part[0] = tsp;
    part[1] = tsm;
    lam[0] = lam[0] - P.sp * lam[0] + a0;
}

// Sums of N = 16 or 8 values over the warp's lanes: each exchange halves the values a lane still carries, 16 shuffles
// where 16 separate sums take 80.  Value i ends in the 32 / N lanes from lane 32 / N * i on.
template <int N, typename A>
__device__ __forceinline__ A warp_sums(A (&v)[N]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16, m = N / 2; m >= 1; off >>= 1, m >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const A keep = up ? v[i + m] : v[i], send = up ? v[i] : v[i + m];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (int off = 16 / N; off >= 1; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    return v[0];
}
__host__ __device__ constexpr int sum16_lane(int i) { return 2 * i; }

// trt_adjoint by a whole warp: lane q < 19 holds h_q and lambda_q (the others zero) and gets the new lambda_q; sp and
// sm parts are added up per lane, the force parts in lane 0.
template <typename A>
__device__ __forceinline__ A warp_trt_adjoint(A h, A lam, int lane, const AdjParams<A>& P, A part[5]) {
    const int c0 = lane_c(lane, 0), c1 = lane_c(lane, 1), c2 = lane_c(lane, 2);
    const A w = lane >= 19 ? A(0) : (lane == 0 ? A(1) / A(3) : (lane <= 6 ? A(1) / A(18) : A(1) / A(36)));
    const A f0 = A(c0), f1 = A(c1), f2 = A(c2), wl = w * lam;
    A v[16] = {h,           f0 * h,      f1 * h,      f2 * h,       wl,           f0 * wl,      f1 * wl, f2 * wl,
               f0 * f0 * wl, f1 * f1 * wl, f2 * f2 * wl, f0 * f1 * wl, f0 * f2 * wl, f1 * f2 * wl, A(0),    A(0)};
    const A mine = warp_sums<16>(v);
    A s[14];
#pragma unroll
    for (int i = 0; i < 14; ++i) s[i] = __shfl_sync(0xffffffffu, mine, sum16_lane(i));
    AdjMoments<A> M;
    M.drho = s[0];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        M.u[a] = s[1 + a] + A(0.5) * P.F[a];
        M.L1[a] = s[5 + a];
    }
    M.L0 = s[4];
#pragma unroll
    for (int i = 0; i < 6; ++i) M.L2[i] = s[8 + i];
    A a0, b[3], dF[3];
    adj_shared<A>(M, P, &a0, b, dF);
    const int partner = lane == 0 ? 0 : (lane < 19 ? ((lane & 1) ? lane + 1 : lane - 1) : lane);
    const A ho = __shfl_sync(0xffffffffu, h, partner), lo = __shfl_sync(0xffffffffu, lam, partner);
    const A* u = M.u;
    const A uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const A uF = u[0] * P.F[0] + u[1] * P.F[1] + u[2] * P.F[2];
    const A cu = f0 * u[0] + f1 * u[1] + f2 * u[2];
    const A cF = f0 * P.F[0] + f1 * P.F[1] + f2 * P.F[2];
    const A ep = w * (M.drho + A(4.5) * cu * cu - A(1.5) * uu), em = w * (A(3) * cu);
    const A Sp = w * (A(9) * cu * cF - A(3) * uF), Sm = w * (A(3) * cF);
    const A hp = A(0.5) * (h + ho), hm = A(0.5) * (h - ho);
    part[0] += lam * (-(hp - ep) - A(0.5) * Sp);
    part[1] += lam * (-(hm - em) - A(0.5) * Sm);
    if (lane == 0)
#pragma unroll
        for (int a = 0; a < 3; ++a) part[2 + a] += dF[a];
    const A lp = A(0.5) * (lam + lo), lm = A(0.5) * (lam - lo);
    const A bc = f0 * b[0] + f1 * b[1] + f2 * b[2];
    return lam - P.sp * lp - P.sm * lm + a0 + bc;
}

// Block sum of the per-thread parameter parts, added to this block's FP64
// accumulator (one slot per block, so the order of additions is fixed).  In
// FP32 the warps' sums are added as a double-float pair (TwoSum, exact to
// far below FP32 resolution) and converted once: FP64 arithmetic is slow on
// this part and every block ends with it.
template <int THREADS, typename A>
__device__ __forceinline__ void accumulate_parts(const A part[5], bool busy, double* __restrict__ acc) {
    __shared__ A red[5][THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (busy) {
        A v[8] = {part[0], part[1], part[2], part[3], part[4], A(0), A(0), A(0)};
        const A s = warp_sums<8>(v);
        const int c = lane >> 2;
        if ((lane & 3) == 0 && c < 5) red[c][wid] = s;
    } else if (lane < 5) {
        red[lane][wid] = A(0);
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        double s;
        if constexpr (sizeof(A) == 4) {
            float h = 0.0f, l = 0.0f;
            for (int w = 0; w < THREADS / 32; ++w) df_add(h, l, red[threadIdx.x][w], 0.0f);
            s = (double)h + (double)l;
        } else {
            s = 0.0;
            for (int w = 0; w < THREADS / 32; ++w) s += red[threadIdx.x][w];
        }
        acc[(size_t)blockIdx.x * 5 + threadIdx.x] += s;
    }
}

// Cells whose reverse step involves a solid cell: some x + c_q, x - c_q or
// x + 2 c_q is solid.  Counts per block for the ordered compaction.
__global__ void __launch_bounds__(AT)
    k_adj_kind(const uint8_t* __restrict__ flags, GridDesc G, uint8_t* __restrict__ kind, int* __restrict__ block_count) {
    const long long x = (long long)blockIdx.x * AT + threadIdx.x;
    int near = 0;
    if (x < G.n) {
        const int i = (int)(x % G.nx), j = (int)((x / G.nx) % G.ny), k = (int)(x / ((long long)G.nx * G.ny));
        uint8_t v = KIND_SOLID;
        if (flags[x] == 0) {
            v = KIND_PLAIN;
            for (int q = 1; q < 19; ++q) {
                const bool s = flags[cell_at(G, i + cx(q), j + cy(q), k + cz(q))] != 0 ||
                               flags[cell_at(G, i - cx(q), j - cy(q), k - cz(q))] != 0 ||
                               flags[cell_at(G, i + 2 * cx(q), j + 2 * cy(q), k + 2 * cz(q))] != 0;
                if (s) v = KIND_NEAR;
            }
        }
        kind[x] = v;
        near = v == KIND_NEAR;
    }
    const unsigned ballot = __ballot_sync(0xffffffffu, near);
    __shared__ int wsum[AT / 32];
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = __popc(ballot);
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < AT / 32; ++w) s += wsum[w];
        block_count[blockIdx.x] = s;
    }
}

// Ordered list of the near cells.  The block offsets are an exclusive scan
// of the per-block counts, done by every block over the blocks before it.
__global__ void __launch_bounds__(AT)
    k_adj_near_list(const uint8_t* __restrict__ kind, const int* __restrict__ block_count, GridDesc G,
                    int* __restrict__ list, int* __restrict__ count) {
    __shared__ int red[AT];
    __shared__ int wsum[AT / 32];
    int s = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += AT) s += block_count[b];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = AT / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    const int base = red[0];
    const long long x = (long long)blockIdx.x * AT + threadIdx.x;
    const int near = x < G.n && kind[x] == KIND_NEAR;
    const unsigned ballot = __ballot_sync(0xffffffffu, near);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) wsum[warp] = __popc(ballot);
    __syncthreads();
    int wbase = 0;
    for (int w = 0; w < warp; ++w) wbase += wsum[w];
    if (near) list[base + wbase + __popc(ballot & ((1u << lane) - 1u))] = (int)x;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        int tot = base;
        for (int w = 0; w < AT / 32; ++w) tot += wsum[w];
        *count = tot;
    }
}

// One reverse step; its first nblocks CTAs take the cells next to the sphere, the others the plain cells in memory
// order.
template <typename S>
struct ReverseArgs {
    using A = typename Store<S>::A;
    const S* gprev;
    const A* nu_next;
    A* nu_out;
    const uint8_t* kind;
    const uint8_t* flags;
    const int* list;       // the near cells
    const int* count;
    GridDesc G;
    FastDiv dx, dy;        // by nx and ny
    int per_cta;           // plain cells per CTA
    int nblocks;
    AdjParams<A> P;
    const ParticleState* ps;
    int cli, with_seed;
    double* acc;           // [CTA][5]
};

// Reverse step on the cells that see no solid: h_q = g_q(x - c_q),
// lambda_q = nu_q(x + c_q).  Solid cells get nu = 0; near cells are left to
// the first CTAs.
template <typename S>
__device__ __forceinline__ void reverse_plain(const ReverseArgs<S>& T, unsigned item, typename Store<S>::A part[5]) {
    using A = typename Store<S>::A;
    const GridDesc& G = T.G;
    const size_t n = (size_t)G.n;
    // the cell's kind is loaded beside the 38 loads of the plain case (a branch on it would
    // hold them back by one memory round trip); a cell of another kind drops them
    const uint8_t kd = T.kind[item];
    const unsigned row = T.dx.div(item), plane = T.dy.div(row);
    const int i = (int)(item - row * (unsigned)G.nx), j = (int)(row - plane * (unsigned)G.ny), k = (int)plane;
    // xs[1 + d] = i - d: the pull source x - c_q at index 1 + c, x + c_q at 1 - c
    const int xs[3] = {wrapc(i + 1, G.nx), i, wrapc(i - 1, G.nx)};
    const int ys[3] = {wrapc(j + 1, G.ny), j, wrapc(j - 1, G.ny)};
    const int zs[3] = {wrapc(k + 1, G.nz), k, wrapc(k - 1, G.nz)};
    A h[19], lam[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        const int src = xs[1 + cx(q)] + G.nx * (ys[1 + cy(q)] + G.ny * zs[1 + cz(q)]);
        const int dn = xs[1 - cx(q)] + G.nx * (ys[1 - cy(q)] + G.ny * zs[1 - cz(q)]);
        h[q] = Store<S>::fetch(T.gprev + (size_t)q * n + src, A(1));
        lam[q] = T.nu_next[(size_t)q * n + dn];
    }
    if (kd == KIND_SOLID) {
#pragma unroll
        for (int q = 0; q < 19; ++q) T.nu_out[(size_t)q * n + item] = A(0);
    } else if (kd == KIND_PLAIN) {
        trt_adjoint<A>(h, lam, T.P, part);
#pragma unroll
        for (int q = 0; q < 19; ++q) T.nu_out[(size_t)q * n + item] = lam[q];
    }
}

// Reverse step of the cells next to the sphere, one warp per cell, lane q on population q: h_q is the forward pull
// with the CLI rule on links (wall at rest), lambda_q the pull run backwards with the terms of every link moved to the
// cells it reads (near_lambda), and the force's own dependence on both.  Everything a population can need is loaded at
// once; a thread per cell followed 19 chains of flag and value loads one after another (43 us at 64^3 in FP32, 142 us
// at 24^3 in FP64).
template <typename S>
__device__ __forceinline__ void reverse_near(const ReverseArgs<S>& T, typename Store<S>::A part[5]) {
    using A = typename Store<S>::A;
    __shared__ LinkFrame<A> Fr;
    if (threadIdx.x == 0) Fr.init(*T.ps);
    const GridDesc& G = T.G;
    const size_t n = (size_t)G.n;
    const int n3[3] = {G.nx, G.ny, G.nz}, per[3] = {1, 1, 1};
    const int lane = threadIdx.x & 31;
    const int total = *T.count, W = T.nblocks * (ADJ_THREADS<S> / 32);
    __syncthreads();
    for (int t = (int)blockIdx.x * (ADJ_THREADS<S> / 32) + (int)(threadIdx.x >> 5); t < total; t += W) {
        const int x = T.list[t];
        const unsigned row = T.dx.div((unsigned)x), plane = T.dy.div(row);
        const int p[3] = {x - (int)row * G.nx, (int)row - (int)plane * G.ny, (int)plane};
        A h = A(0), l = A(0);
        bool link = false;
        const int q = lane < 19 ? lane : 0, k = opp(q);
        const int c[3] = {cx(q), cy(q), cz(q)};
        if (lane < 19) {
            const long long s = cell_at(G, p[0] - c[0], p[1] - c[1], p[2] - c[2]);
            const long long y = cell_at(G, p[0] + c[0], p[1] + c[1], p[2] + c[2]);
            const long long yy = cell_at(G, p[0] + 2 * c[0], p[1] + 2 * c[1], p[2] + 2 * c[2]);
            const bool s_solid = T.flags[s] != 0, y_solid = T.flags[y] != 0, yy_solid = T.flags[yy] != 0;
            const A g_s = Store<S>::fetch(T.gprev + (size_t)q * n + s, A(1));
            const A g_k = Store<S>::fetch(T.gprev + (size_t)k * n + x, A(1));
            const A g_q = Store<S>::fetch(T.gprev + (size_t)q * n + x, A(1));
            const A g_far = Store<S>::fetch(T.gprev + (size_t)k * n + y, A(1));
            const A nu_y = T.nu_next[(size_t)q * n + y], nu_yk = T.nu_next[(size_t)k * n + y];
            const A nu_k = T.nu_next[(size_t)k * n + x], nu_q = T.nu_next[(size_t)q * n + x];
            const int ca = c[T.P.axis];
            h = g_s;
            if (q == 0) {
                l = nu_q;
            } else {
                link = s_solid;
                A dx[3], delta, kappa0, alpha;
                int pu[3];
                if (!y_solid) {
                    l = nu_y;   // plain pull at y reads g_q(x)
                    if (yy_solid) {   // link at y, incoming opp(q): its far cell is x
                        const int py[3] = {wrapc(p[0] + c[0], G.nx), wrapc(p[1] + c[1], G.ny), wrapc(p[2] + c[2], G.nz)};
                        Fr.offset(py, n3, per, dx, pu);
                        cli_coeffs<A>(k, dx, T.cli != 0, Fr.r, &delta, &kappa0, &alpha);
                        l += kappa0 * nu_yk;
                    }
                } else {   // link at x, incoming opp(q): g_q(x) is its g~_k, also in the force
                    l = nu_k;
                    if (T.with_seed) l += T.P.seed * A(ca);
                }
                if (link) {   // link at x, incoming q
                    Fr.offset(p, n3, per, dx, pu);
                    cli_coeffs<A>(q, dx, T.cli && !y_solid, Fr.r, &delta, &kappa0, &alpha);
                    h = g_k + kappa0 * (y_solid ? A(0) : g_far) - kappa0 * g_q;
                    l -= kappa0 * nu_q;
                }
            }
        }
        A out = warp_trt_adjoint<A>(h, l, lane, T.P, part);
        if (lane < 19) {
            if (link) out -= T.P.seed * A(c[T.P.axis]);   // the force's own dependence on h^n at the link: c_k = -c_q
            T.nu_out[(size_t)q * n + x] = out;
        }
    }
}

template <typename S>
__global__ void __launch_bounds__(ADJ_THREADS<S>, ADJ_MIN_CTAS<S>)
    k_adj_step(const __grid_constant__ ReverseArgs<S> T) {
    using A = typename Store<S>::A;
    pdl_wait();
    A part[5] = {A(0), A(0), A(0), A(0), A(0)};
    bool busy = true;
    if ((int)blockIdx.x < T.nblocks) {
        reverse_near<S>(T, part);
    } else {
        const unsigned cta = blockIdx.x - (unsigned)T.nblocks;
        const unsigned t = threadIdx.x, item = cta * (unsigned)T.per_cta + t;
        busy = (int)t < T.per_cta;   // whole warps
        if (busy && item < (unsigned)T.G.n) reverse_plain<S>(T, item, part);
    }
    accumulate_parts<ADJ_THREADS<S>>(part, busy, T.acc);
}

// lambda at a fluid cell next to the sphere: S^T nu with the link terms,
// plus (with_seed) the force's own dependence on g at the links.
template <typename A>
__device__ __forceinline__ void near_lambda(const A* __restrict__ nu, const uint8_t* __restrict__ flags,
                                            const GridDesc& G, int i, int j, int k, const LinkFrame<A>& Fr, int cli,
                                            bool with_seed, A seed, int axis, A (&lam)[19]) {
    const size_t n = (size_t)G.n;
    const long long x = cell_at(G, i, j, k);
    const int n3[3] = {G.nx, G.ny, G.nz}, per[3] = {1, 1, 1};
    const int px[3] = {i, j, k};
    A dx[3];
    int pu[3];
    Fr.offset(px, n3, per, dx, pu);
    lam[0] = nu[x];
    for (int q = 1; q < 19; ++q) {
        const int c[3] = {cx(q), cy(q), cz(q)};
        const long long y = cell_at(G, i + c[0], j + c[1], k + c[2]);
        A l;
        if (flags[y] == 0) {
            l = nu[(size_t)q * n + y];   // plain pull at y reads g_q(x)
            if (flags[cell_at(G, i + 2 * c[0], j + 2 * c[1], k + 2 * c[2])] != 0) {
                // link at y, incoming opp(q): its far cell is x
                const int py[3] = {wrapc(i + c[0], G.nx), wrapc(j + c[1], G.ny), wrapc(k + c[2], G.nz)};
                A dy[3], delta, kappa0, alpha;
                int pv[3];
                Fr.offset(py, n3, per, dy, pv);
                cli_coeffs<A>(opp(q), dy, cli != 0, Fr.r, &delta, &kappa0, &alpha);
                l += kappa0 * nu[(size_t)opp(q) * n + y];
            }
        } else {
            // link at x, incoming opp(q): g_q(x) is its g~_k, also in the force
            l = nu[(size_t)opp(q) * n + x];
            if (with_seed) l += seed * A(c[axis]);
        }
        if (flags[cell_at(G, i - c[0], j - c[1], k - c[2])] != 0) {
            // link at x, incoming q: -kappa0 g_q(x)
            const bool far_ok = flags[y] == 0;
            A delta, kappa0, alpha;
            cli_coeffs<A>(q, dx, cli && far_ok, Fr.r, &delta, &kappa0, &alpha);
            l -= kappa0 * nu[(size_t)q * n + x];
        }
        lam[q] = l;
    }
}

// lambda^0 and dJ/du0 = (dE/du0)^T lambda^0 with
// dE_q/du = w_q (3 c_q + 9 (c_q.u0) c_q - 3 u0), times the incoming dJ.  In
// FP64 (u0's type) whatever the field's: bound by its instructions, about 100
// a cell on the sums and differences of the opposite pairs instead of 320,
// and in CTAs of two warps for all SMs of a small grid: 63 -> 41 us for 24^3
// FP64 cells (what is left are the link quotients of the cells by the sphere).
constexpr int INIT_THREADS = 64;
template <typename A>
__global__ void __launch_bounds__(INIT_THREADS)
    k_adj_init_grad(const A* __restrict__ nu, const uint8_t* __restrict__ flags, const uint8_t* __restrict__ kind,
                    GridDesc G, const double* __restrict__ u0, const ParticleState* __restrict__ ps, int cli, A seed,
                    int axis, const double* __restrict__ dJ, double* __restrict__ grad_u0) {
    __shared__ LinkFrame<A> Fr;
    if (threadIdx.x == 0) Fr.init(*ps);
    __syncthreads();
    const long long x = (long long)blockIdx.x * INIT_THREADS + threadIdx.x;
    if (x >= G.n) return;
    const size_t n = (size_t)G.n;
    if (kind[x] == KIND_SOLID) {
        for (int a = 0; a < 3; ++a) grad_u0[(size_t)a * n + x] = 0.0;
        return;
    }
    const int i = (int)(x % G.nx), j = (int)((x / G.nx) % G.ny), k = (int)(x / ((long long)G.nx * G.ny));
    A lam[19];
    if (kind[x] == KIND_PLAIN) {
        for (int q = 0; q < 19; ++q) lam[q] = nu[(size_t)q * n + cell_at(G, i + cx(q), j + cy(q), k + cz(q))];
    } else {
        near_lambda<A>(nu, flags, G, i, j, k, Fr, cli, true, seed, axis, lam);
    }
    const double u[3] = {u0[x], u0[n + x], u0[2 * n + x]};
    double p[9], m[9];   // pairs 0..2 are the faces, 3..8 (+x+y), (+x-y), (+x+z), (+x-z), (+y+z), (+y-z)
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const double a = (double)lam[2 * q + 1], b = (double)lam[2 * q + 2];
        p[q] = a + b;
        m[q] = a - b;
    }
    const double wF = wgt<double>(1), wE = wgt<double>(7);
    const double exy = p[3] + p[4], exz = p[5] + p[6], eyz = p[7] + p[8];
    const double L0 = wgt<double>(0) * (double)lam[0] + wF * ((p[0] + p[1]) + p[2]) + wE * ((exy + exz) + eyz);
    const double L1[3] = {wF * m[0] + wE * ((m[3] + m[4]) + (m[5] + m[6])), wF * m[1] + wE * ((m[3] - m[4]) + (m[7] + m[8])),
                          wF * m[2] + wE * ((m[5] - m[6]) + (m[7] - m[8]))};
    const double xy = wE * (p[3] - p[4]), xz = wE * (p[5] - p[6]), yz = wE * (p[7] - p[8]);
    const double L2u[3] = {(wF * p[0] + wE * (exy + exz)) * u[0] + xy * u[1] + xz * u[2],
                           xy * u[0] + (wF * p[1] + wE * (exy + eyz)) * u[1] + yz * u[2],
                           xz * u[0] + yz * u[1] + (wF * p[2] + wE * (exz + eyz)) * u[2]};
    const double s = *dJ;
    for (int a = 0; a < 3; ++a) grad_u0[(size_t)a * n + x] = s * (3.0 * L1[a] + 9.0 * L2u[a] - 3.0 * L0 * u[a]);
}

__global__ void k_adj_mean(const double* __restrict__ forces, int nsteps, int axis, double* __restrict__ J) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int n = 0; n < nsteps; ++n) s += forces[(size_t)n * 3 + axis];
        *J = s / (double)nsteps;
    }
}

// Parameter gradients from the per-block accumulators:
// dJ/dtau = ds+/dtau sum part0 + ds-/dtau sum part1 with ds+/dtau = -s+^2 and
// ds-/dtau = s-^2 Lambda / (tau - 1/2)^2; dJ/dF_a = sum part_{2+a}.
__global__ void k_adj_params(const double* __restrict__ acc, int nblocks, double tau, double magic,
                             const double* __restrict__ dJ, double* __restrict__ grad_tau,
                             double* __restrict__ grad_force) {
    __shared__ double red[5][AT];
    double v[5] = {0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nblocks; b += AT)
        for (int c = 0; c < 5; ++c) v[c] += acc[(size_t)b * 5 + c];
    for (int c = 0; c < 5; ++c) red[c][threadIdx.x] = v[c];
    __syncthreads();
    for (int h = AT / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h)
            for (int c = 0; c < 5; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double sp = 1.0 / tau, sm = 1.0 / (0.5 + magic / (tau - 0.5));
        const double dsp = -sp * sp, dsm = sm * sm * magic / ((tau - 0.5) * (tau - 0.5));
        const double s = *dJ;
        if (grad_tau) *grad_tau = s * (dsp * red[0][0] + dsm * red[1][0]);
        if (grad_force)
            for (int a = 0; a < 3; ++a) grad_force[a] = s * red[2 + a][0];
    }
}

template <typename F>
void with_adj_storage(int prec, F&& f) {
    if (prec == LBMP_FP64) f((double*)nullptr);
    else f((float*)nullptr);
}

}  // namespace

struct AdjointEngine {
    int nsteps = 0, interval = 0, nckpt = 0, axis = 0;
    size_t state_bytes = 0, nu_bytes = 0;
    void* ckpt = nullptr;     // nckpt states
    void* seg = nullptr;      // interval states (slot 0 unused: it is the checkpoint)
    void* nu[2] = {nullptr, nullptr};
    double* u0 = nullptr;     // copy of the initial velocity field [3][n]
    double* forces = nullptr; // [nsteps][3]
    double* acc = nullptr;    // [acc_blocks][5]
    int acc_blocks = 0, near_blocks = 0, near_cells = 0;
    int cell_blocks = 0;                   // blocks of AT cells
    int threads = AT;                      // of a reverse-step CTA
    int per_cta = AT, plain_blocks = 0;    // plain cells per reverse-step CTA, and those CTAs
    uint8_t* kind = nullptr;
    int* blk = nullptr;
    int* near_list = nullptr;
    int* near_count = nullptr;
    bool forward_done = false;
    bool geometry_done = false;   // kind bytes and near list of the (fixed) sphere
    long long placed = -1;        // the handle's `placed` that they, the graphs and the forward pass belong to
    double tau = 0, F[3] = {0, 0, 0};
    // the forward pass (one per parity of the handle's buffers) and the reverse
    // sweep replayed from CUDA graphs; dropped when tau, the body force, the
    // objective's axis or the sphere's place (with it the flag buffer) change
    cudaGraphExec_t gfwd[2] = {nullptr, nullptr};
    cudaGraphExec_t gbwd = nullptr;
    double graph_tau = -1.0, graph_F[3] = {0, 0, 0};
    int graph_axis = -1;
    cudaStream_t capture_stream = nullptr;
};

namespace {

// The step's frames after the host changed the record.
void renew_frames(lbmp_handle* h) {
    if (!h->frames_stale) return;
    launch_frames(h, h->stream);
    h->frames_stale = false;
    h->launches += 1;
}

// One forward step with the sphere held at rest; the force of the step into force_out (null: not wanted).
template <typename S>
void forward_step(lbmp_handle* h, const S* src, S* dst, double* force_out) {
    launch_step<S>(h, src, dst, collide_params<typename Store<S>::A>(h), force_out ? 1 : 2, force_out, h->stream);
}

template <typename S>
S* state(AdjointEngine* E, int m, int j, size_t n) {
    if (j == 0) return (S*)E->ckpt + (size_t)m * 19 * n;
    return (S*)E->seg + (size_t)j * 19 * n;
}

void drop_graphs(AdjointEngine* E) {
    for (auto& g : E->gfwd)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    if (E->gbwd) {
        cudaGraphExecDestroy(E->gbwd);
        E->gbwd = nullptr;
    }
}

// Enqueues `body` on the handle's stream: replayed from *graph, captured on a
// private stream the first time (the caller's stream may be the legacy
// default stream, which cannot be captured).  Profiling runs plain launches.
template <typename F>
lbmp_status captured(lbmp_handle* h, AdjointEngine* E, cudaGraphExec_t* graph, F&& body) {
    if (h->profiling) {
        body();
        return LBMP_OK;
    }
    if (!*graph) {
        if (!E->capture_stream && cudaStreamCreateWithFlags(&E->capture_stream, cudaStreamNonBlocking) != cudaSuccess)
            return LBMP_ERR_CUDA;
        // the capture stream starts after the work already queued on the caller's stream
        cudaEvent_t ev;
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return LBMP_ERR_CUDA;
        cudaEventRecord(ev, h->stream);
        cudaStreamWaitEvent(E->capture_stream, ev, 0);
        cudaEventDestroy(ev);
        cudaStream_t user = h->stream;
        h->stream = E->capture_stream;
        if (cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) {
            h->stream = user;
            return LBMP_ERR_CUDA;
        }
        body();
        cudaGraph_t g = nullptr;
        const cudaError_t e = cudaStreamEndCapture(h->stream, &g);
        h->stream = user;
        if (e != cudaSuccess) return LBMP_ERR_CUDA;
        const cudaError_t e2 = cudaGraphInstantiate(graph, g, 0);
        cudaGraphDestroy(g);
        if (e2 != cudaSuccess) return LBMP_ERR_CUDA;
    }
    return cudaGraphLaunch(*graph, h->stream) == cudaSuccess ? LBMP_OK : LBMP_ERR_CUDA;
}

void release(lbmp_handle* h, AdjointEngine* E) {
    drop_graphs(E);
    if (E->capture_stream) cudaStreamDestroy(E->capture_stream);
    void* ptrs[] = {E->ckpt, E->seg, E->nu[0], E->nu[1], E->u0, E->forces, E->acc, E->kind, E->blk, E->near_list,
                    E->near_count};
    for (void* p : ptrs)
        if (p) handle_free(h, p);
    *E = AdjointEngine();
}

}  // namespace

void adjoint_destroy(lbmp_handle* h) {
    if (!h->adj) return;
    drop_graphs(h->adj);
    if (h->adj->capture_stream) cudaStreamDestroy(h->adj->capture_stream);
    delete h->adj;   // device memory is released with the handle's allocations
    h->adj = nullptr;
}

lbmp_status adjoint_check(const lbmp_handle* h, std::string* why) {
    if (h->amr || h->batch) return *why = "the drag adjoint runs on a single uniform grid", LBMP_ERR_UNSUPPORTED;
    if (!h->has_particle) return *why = "the drag adjoint needs a sphere", LBMP_ERR_INVALID_ARG;
    if (h->h_ps.fixed != 1) return *why = "the drag adjoint needs the sphere held fixed", LBMP_ERR_UNSUPPORTED;
    for (int a = 0; a < 3; ++a) {
        if (!h->G.periodic[a]) return *why = "the drag adjoint needs a periodic box", LBMP_ERR_UNSUPPORTED;
        if (h->h_ps.u[a] != 0.0 || h->h_ps.w[a] != 0.0)
            return *why = "the drag adjoint needs the sphere at rest", LBMP_ERR_UNSUPPORTED;
    }
    if (h->cfg.precision == LBMP_FP16) return *why = "the drag adjoint runs in FP32 or FP64", LBMP_ERR_UNSUPPORTED;
    if (h->cfg.bulk_factor != 1.0) return *why = "the drag adjoint is the reverse of the TRT step (bulk factor 1)", LBMP_ERR_UNSUPPORTED;
    return LBMP_OK;
}

lbmp_status adjoint_forward(lbmp_handle* h, const double* u0, int nsteps, int interval, int axis, double* J,
                            double* forces) {
    if (!h->adj) h->adj = new AdjointEngine();
    AdjointEngine* E = h->adj;
    const size_t n = (size_t)h->G.n;
    const size_t es = h->cfg.precision == LBMP_FP64 ? 8 : 4;
    const int nckpt = (nsteps + interval - 1) / interval;
    if (E->nsteps != nsteps || E->interval != interval) {
        release(h, E);
        E->nsteps = nsteps;
        E->interval = interval;
        E->nckpt = nckpt;
        E->state_bytes = es * 19 * n;
        E->nu_bytes = es * 19 * n;
        E->cell_blocks = (int)((n + AT - 1) / AT);
        E->threads = h->cfg.precision == LBMP_FP64 ? ADJ_THREADS<double> : ADJ_THREADS<float>;
        E->per_cta = E->threads;   // small grids over all SMs: four CTAs on each (32^3 FP32 0.3 us a step less than two)
        while (E->per_cta > 32 && (int)n / E->per_cta < 4 * SMS) E->per_cta /= 2;
        E->plain_blocks = (int)((n + (size_t)E->per_cta - 1) / (size_t)E->per_cta);
        E->near_blocks = 0;
        E->acc_blocks = NEAR_WARPS_MAX / (E->threads / 32) + E->plain_blocks;
        E->ckpt = handle_alloc(h, E->state_bytes * (size_t)nckpt);
        E->seg = handle_alloc(h, E->state_bytes * (size_t)interval);
        E->nu[0] = handle_alloc(h, E->nu_bytes);
        E->nu[1] = handle_alloc(h, E->nu_bytes);
        E->u0 = (double*)handle_alloc(h, sizeof(double) * 3 * n);
        E->forces = (double*)handle_alloc(h, sizeof(double) * 3 * (size_t)nsteps);
        E->acc = (double*)handle_alloc(h, sizeof(double) * 5 * (size_t)E->acc_blocks);
        E->kind = (uint8_t*)handle_alloc(h, n);
        E->blk = (int*)handle_alloc(h, sizeof(int) * (size_t)E->cell_blocks);
        E->near_list = (int*)handle_alloc(h, sizeof(int) * n);
        E->near_count = (int*)handle_alloc(h, sizeof(int));
        if (!E->ckpt || !E->seg || !E->nu[0] || !E->nu[1] || !E->u0 || !E->forces || !E->acc || !E->kind || !E->blk ||
            !E->near_list || !E->near_count) {
            release(h, E);
            return LBMP_ERR_OOM;
        }
    }
    E->axis = axis;
    E->tau = h->tau;
    for (int a = 0; a < 3; ++a) E->F[a] = h->body_force[a];
    if (E->graph_tau != h->tau || E->graph_F[0] != h->body_force[0] || E->graph_F[1] != h->body_force[1] ||
        E->graph_F[2] != h->body_force[2] || E->graph_axis != axis) {
        drop_graphs(E);
        E->graph_tau = h->tau;
        E->graph_axis = axis;
        for (int a = 0; a < 3; ++a) E->graph_F[a] = h->body_force[a];
    }
    if (E->placed != h->placed) {   // released, moved and held again, or another one loaded
        drop_graphs(E);
        E->geometry_done = false;
        E->placed = h->placed;
    }
    renew_frames(h);
    if (!E->geometry_done) {   // cells of the reverse step next to the (fixed) sphere
        const unsigned gb = (unsigned)E->cell_blocks;
        k_adj_kind<<<gb, AT, 0, h->stream>>>(h->flags[h->fcur], h->G, E->kind, E->blk);
        k_adj_near_list<<<gb, AT, 0, h->stream>>>(E->kind, E->blk, h->G, E->near_list, E->near_count);
        h->launches += 2;
        if (cudaMemcpyAsync(&E->near_cells, E->near_count, sizeof(int), cudaMemcpyDeviceToHost, h->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(h->stream) != cudaSuccess)
            return LBMP_ERR_CUDA;
        h->d2h += sizeof(int);
        const int warps = E->threads / 32;
        E->near_blocks = std::min(NEAR_WARPS_MAX / warps, std::max(1, (E->near_cells + warps - 1) / warps));
        E->geometry_done = true;
    }
    cudaMemcpyAsync(E->u0, u0, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, h->stream);
    const int par = h->cur;
    const lbmp_status st = captured(h, E, &E->gfwd[par], [&]() {
        with_adj_storage(h->cfg.precision, [&](auto tag) {
            using S = std::remove_pointer_t<decltype(tag)>;
            const double zero[3] = {0.0, 0.0, 0.0};
            S* a = (S*)h->pops[par];
            S* b = (S*)h->pops[1 - par];
            launch_init_equilibrium<S>(a, h->flags[h->fcur], h->G, 1.0, zero, E->u0, (typename Store<S>::A)1,
                                       h->stream);
            cudaMemcpyAsync(E->ckpt, a, E->state_bytes, cudaMemcpyDeviceToDevice, h->stream);
            for (int s = 1; s <= nsteps; ++s) {
                forward_step<S>(h, a, b, E->forces + (size_t)(s - 1) * 3);
                std::swap(a, b);
                if (s % interval == 0 && s / interval < nckpt)
                    cudaMemcpyAsync((char*)E->ckpt + E->state_bytes * (size_t)(s / interval), a, E->state_bytes,
                                    cudaMemcpyDeviceToDevice, h->stream);
            }
        });
    });
    if (st != LBMP_OK) return st;
    h->cur = (par + nsteps) & 1;
    h->steps += nsteps;
    h->launches += 1 + (long long)nsteps;
    h->updates += (long long)nsteps * h->G.n;
    k_adj_mean<<<1, 32, 0, h->stream>>>(E->forces, nsteps, axis, J);
    h->launches += 1;
    if (forces)
        cudaMemcpyAsync(forces, E->forces, sizeof(double) * 3 * (size_t)nsteps, cudaMemcpyDeviceToDevice, h->stream);
    E->forward_done = true;
    if (cudaGetLastError() != cudaSuccess) return LBMP_ERR_CUDA;
    return LBMP_OK;
}

lbmp_status adjoint_backward(lbmp_handle* h, const double* dJ, double* grad_tau, double* grad_force, double* grad_u0,
                             std::string* why) {
    AdjointEngine* E = h->adj;
    if (!E || !E->forward_done) return *why = "lbmp_drag_backward needs a preceding lbmp_drag_forward", LBMP_ERR_INVALID_ARG;
    if (E->tau != h->tau || E->F[0] != h->body_force[0] || E->F[1] != h->body_force[1] || E->F[2] != h->body_force[2])
        return *why = "tau or the body force changed since lbmp_drag_forward", LBMP_ERR_INVALID_ARG;
    if (E->placed != h->placed) return *why = "the sphere moved since lbmp_drag_forward", LBMP_ERR_INVALID_ARG;
    renew_frames(h);   // the held sphere's velocities may have been others in between
    const size_t n = (size_t)h->G.n;
    const int N = E->nsteps, K = E->interval;
    const int cli = h->cfg.boundary == LBMP_CLI ? 1 : 0;
    lbmp_status st = LBMP_OK;
    with_adj_storage(h->cfg.precision, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        using A = typename Store<S>::A;
        AdjParams<A> P;
        double sp, sm;
        relaxation_rates(h->tau, h->magic, &sp, &sm);
        P.sp = (A)sp;
        P.sm = (A)sm;
        for (int a = 0; a < 3; ++a) P.F[a] = (A)h->body_force[a];
        P.seed = (A)(1.0 / (double)N);
        P.axis = E->axis;
        ReverseArgs<S> T;
        T.kind = E->kind;
        T.flags = h->flags[h->fcur];
        T.list = E->near_list;
        T.count = E->near_count;
        T.G = h->G;
        T.dx.set((unsigned)h->G.nx);
        T.dy.set((unsigned)h->G.ny);
        T.per_cta = E->per_cta;
        T.nblocks = E->near_blocks;
        T.P = P;
        T.ps = h->d_ps;
        T.cli = cli;
        T.acc = E->acc;
        st = captured(h, E, &E->gbwd, [&]() {
            cudaMemsetAsync(E->acc, 0, sizeof(double) * 5 * (size_t)E->acc_blocks, h->stream);
            cudaMemsetAsync(E->nu[0], 0, E->nu_bytes, h->stream);
            int cur = 0;   // nu[cur] holds nu^{n+1}
            for (int m = E->nckpt - 1; m >= 0; --m) {
                const int s0 = m * K, len = std::min(K, N - s0);
                for (int j = 1; j < len; ++j)
                    forward_step<S>(h, state<S>(E, m, j - 1, n), state<S>(E, m, j, n), nullptr);
                for (int s = s0 + len; s > s0; --s) {
                    const S* gprev = state<S>(E, m, s - 1 - s0, n);
                    const A* nu_next = (const A*)E->nu[cur];
                    A* nu_out = (A*)E->nu[1 - cur];
                    const long long ev = profile_mark(h);
                    T.gprev = gprev;
                    T.nu_next = nu_next;
                    T.nu_out = nu_out;
                    T.with_seed = s < N ? 1 : 0;
                    launch_pdl(k_adj_step<S>, (unsigned)(E->near_blocks + E->plain_blocks), ADJ_THREADS<S>, 0, h->stream, T);
                    // algorithmic bytes: 19 populations of g^{n-1} read, 19 adjoint values read and written per cell
                    const double cells = (double)n;
                    profile_kernel(h, ev, profile_mark(h), cells * (19.0 * sizeof(S) + 38.0 * sizeof(A)), cells);
                    cur = 1 - cur;
                }
            }
        });
        h->launches += (long long)(N - E->nckpt) + (long long)N;
        if (st == LBMP_OK && grad_u0) {   // nu^1 sits in nu[N % 2] after N reverse steps
            k_adj_init_grad<A><<<(unsigned)((n + INIT_THREADS - 1) / INIT_THREADS), INIT_THREADS, 0, h->stream>>>(
                (const A*)E->nu[N & 1], h->flags[h->fcur], E->kind, h->G, E->u0, h->d_ps, cli, P.seed, E->axis, dJ, grad_u0);
            h->launches += 1;
        }
    });
    if (st != LBMP_OK) return st;
    k_adj_params<<<1, AT, 0, h->stream>>>(E->acc, E->plain_blocks + E->near_blocks, h->tau, h->magic, dJ, grad_tau,
                                          grad_force);
    h->launches += 1;
    if (cudaGetLastError() != cudaSuccess) return LBMP_ERR_CUDA;
    return LBMP_OK;
}

}  // namespace lbmp
