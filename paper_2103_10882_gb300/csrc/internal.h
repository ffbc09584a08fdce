// Internal declarations shared by the host API and the kernel launchers.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <cmath>
#include <stdint.h>

#include <string>
#include <utility>
#include <vector>

#include "../../include/lbmp.h"
#include "lattice.cuh"

namespace lbmp {

constexpr int SMS = 152;   // streaming multiprocessors of the part, by which launches are sized

struct GridDesc {
    int nx, ny, nz;
    int periodic[3];
    long long n;   // nx * ny * nz
    // velocities of the no-slip domain walls [axis][0 low face, 1 high face] (uniform grids);
    // moving != 0 when any is nonzero
    double uw[3][2][3] = {};
    int moving = 0;
};

// Moving-wall term of a pull from beyond a no-slip domain wall half-way
// between cells: bounce-back plus Ladd's 2 w_q rho_0 c_q.u_w / c_s^2 = 6 w_q
// c_q.u_w (the CLI rule of Sec. 2.3 at delta = 1/2), summed over the faces
// the link from the cell xyz against c_q crosses.
template <typename A>
__device__ __forceinline__ A wall_term(const GridDesc& G, int q, const int xyz[3]) {
    if (!G.moving) return A(0);
    const int n3[3] = {G.nx, G.ny, G.nz};
    const int c3[3] = {cx(q), cy(q), cz(q)};
    A t = A(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int s = xyz[a] - c3[a];
        if (G.periodic[a] || (s >= 0 && s < n3[a])) continue;
        const double* u = G.uw[a][s < 0 ? 0 : 1];
        t += A(6) * wgt<A>(q) * (A(c3[0]) * A(u[0]) + A(c3[1]) * A(u[1]) + A(c3[2]) * A(u[2]));
    }
    return t;
}

// Coefficients of collide_direct, formed once on the host in FP64 (collide_consts): the relaxation and
// equilibrium factors of a pair's sum and difference, and per pair of directions the constant part of the
// Guo source.
template <typename A>
struct CollideConsts {
    A hp, hsm, r0;        // (1 - s+)/2, s-/2, 1 - s+
    A kF, kE, mF, mE;     // s+ 9/2 w, s- 3 w on faces and edges
    A c15, cF;            // 3/2, 3 (1 - s+/2)
    A gs[9], ga[9];       // 9 (1 - s+/2) w c_q.F, 3 (1 - s-/2) w c_q.F for q = 1, 3, ..., 17
};

// Collision parameters in the arithmetic precision A of the storage type.
template <typename A>
struct CollideParams {
    A sp, sm;          // s+ = 1/tau, s- from the magic parameter
    A db;              // MRT: s_b - s+ (bulk factor Lambda_b != 1), 0 for TRT
    A F[3];            // fluid body force
    int forced;
    A scale, inv_scale;   // FP16 storage scaling (1 otherwise)
    CollideConsts<A> k;
};

// Fills p.k from the rates and the force of p (already rounded to A: the coefficients belong to them).
template <typename A>
inline void collide_consts(CollideParams<A>& p) {
    const double sp = p.sp, sm = p.sm;
    const double wF = 1.0 / 18.0, wE = 1.0 / 36.0;
    CollideConsts<A>& k = p.k;
    k.hp = (A)(0.5 * (1.0 - sp));
    k.hsm = (A)(0.5 * sm);
    k.r0 = (A)(1.0 - sp);
    k.kF = (A)(4.5 * sp * wF);
    k.kE = (A)(4.5 * sp * wE);
    k.mF = (A)(3.0 * sm * wF);
    k.mE = (A)(3.0 * sm * wE);
    k.c15 = (A)1.5;
    k.cF = (A)(3.0 * (1.0 - 0.5 * sp));
    for (int i = 0; i < 9; ++i) {
        const int q = 2 * i + 1;
        const double w = q < 7 ? wF : wE;
        const double c = (double)p.F[0] * kCX[q] + (double)p.F[1] * kCY[q] + (double)p.F[2] * kCZ[q];
        k.gs[i] = (A)(9.0 * (1.0 - 0.5 * sp) * w * c);
        k.ga[i] = (A)(3.0 * (1.0 - 0.5 * sm) * w * c);
    }
}

// Axis-aligned box of cells around the sphere, fixed extent, origin read
// from the particle state on the device.
struct BoxDesc {
    int R;        // half width in cells
    int E[3];     // extent per axis (clamped to the domain for periodic axes)
    long long cells;
};

// Boundary CTAs of a coupled uniform step, also the number of force partials (8 warps each, taking the boundary
// cells in turn).  The list's capacity is two to three times the boundary cells: one CTA per 20 entries gives every
// warp about one cell, and the chain of a cell, the sums and the particle update is the step where the bulk update is
// short (one per 40 costs a 32^3 step 10%, one per 10 4%).  Where the bulk update runs for 6,080 CTAs or more (BULK_LONG)
// the chain hides behind it and half as many cost it less (256 x 128 x 96: 92.0 and 91.3 us; 256^3 in FP16 storage 272
// and 270).  FP64 in launch_step.  At most eight per SM.
// Boxes of up to SEG_CELLS_MAX cells (spheres up to about 70 cells) find their cells through a prefix of the segments'
// numbers, 8 KB of shared memory at most; larger ones read a list that a further launch makes.
constexpr int BOUNDARY_PER = 20, BOUNDARY_PER_FP64 = 8;   // list entries per CTA where there are most CTAs
constexpr long long SEG_CELLS_MAX = 2048 * 256;
inline bool step_uses_list(const BoxDesc& b) { return b.cells > SEG_CELLS_MAX; }
inline int step_boundary_blocks(int list_capacity, int per) {
    const int n = (list_capacity + per - 1) / per;
    return n < 1 ? 1 : (n > 8 * SMS ? 8 * SMS : n);
}

// n / d for n < 2^31 by one high multiplication (Granlund & Montgomery, "Division by invariant integers
// using multiplication", 1994, Fig. 4.1): d >= 1.
struct FastDiv {
    unsigned d, m, s;
    __host__ void set(unsigned v) {
        d = v;
        s = 0;
        while ((1ull << s) < v) ++s;
        m = (unsigned)(((1ull << 32) * ((1ull << s) - v)) / v + 1);
    }
    __device__ __forceinline__ unsigned div(unsigned n) const {
        const unsigned t = __umulhi(m, n);
        return (t + n) >> s;   // t <= n < 2^31: no overflow
    }
};

// Launch that may start before the kernel ahead of it on the stream has ended (pdl_wait).
template <typename K, typename... Args>
inline void launch_pdl(K kernel, unsigned grid, int threads, size_t smem, cudaStream_t stream, const Args&... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = stream;
    cudaLaunchAttribute a = {};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, args...);
}

struct PFrames;

// Launchers (uniform.cu).  All are asynchronous on `stream`.
template <typename S>
void launch_step(const lbmp_handle* h, const S* src, S* dst, const CollideParams<typename Store<S>::A>& p, int finish,
                 double* force_out, cudaStream_t stream);
void launch_flags_full(uint8_t* flags, const GridDesc& g, const ParticleState* ps, cudaStream_t stream);
void launch_frames(const lbmp_handle* h, cudaStream_t stream);
size_t frames_bytes();
// Returns the number of launches.
template <typename S>
int launch_remap(const lbmp_handle* h, S* pops, const uint8_t* fcur, uint8_t* fnext, int frame, bool mark_only,
                 typename Store<S>::A scale, typename Store<S>::A inv_scale, typename Store<S>::A gcoef,
                 cudaStream_t stream);
// The segments' boundary cells as one list (h->list, h->count).
void launch_list_segments(const lbmp_handle* h, cudaStream_t stream);
void launch_export_links(const uint8_t* flags, const int* list, const int* count, int max_cells,
                         const GridDesc& g, const ParticleState* ps, int cli, int32_t* q_out, double* delta_out,
                         cudaStream_t stream);
template <typename S>
void launch_init_equilibrium(S* pops, const uint8_t* flags, const GridDesc& g, double rho, const double u[3],
                             const double* u_field, typename Store<S>::A scale, cudaStream_t stream);
template <typename S>
void launch_to_f64(const S* pops, double* out, long long count, typename Store<S>::A inv_scale,
                   cudaStream_t stream);
template <typename S>
void launch_from_f64(const double* in, S* pops, long long count, typename Store<S>::A scale, cudaStream_t stream);
template <typename S>
void launch_gather(const S* pops, long long ncells, const int64_t* cells, long long n, double* out,
                   typename Store<S>::A inv_scale, cudaStream_t stream);
template <typename S>
void launch_zero_solid(S* pops, const uint8_t* flags, const GridDesc& g, cudaStream_t stream);

struct AmrEngine;
struct BatchEngine;
struct AdjointEngine;

// Profiling events on the handle's stream (api.cu); -1 when profiling is off.
long long profile_mark(lbmp_handle* h);
void profile_kernel(lbmp_handle* h, long long start, long long end, double bytes, double updates);
void profile_step(lbmp_handle* h, long long start, long long end);

// Device allocation through the handle's allocator (api.cu).
void* handle_alloc(lbmp_handle* h, size_t bytes);
void handle_free(lbmp_handle* h, void* p);

}  // namespace lbmp

namespace lbmp {
// The particle record and the status word, side by side on the device so that one copy brings both back.
struct RecordStatus {
    ParticleState ps;
    int status;
};
}  // namespace lbmp

// One simulation (opaque to callers of the C ABI).
struct lbmp_handle {
    lbmp_config cfg;
    lbmp::GridDesc G;
    cudaStream_t stream = nullptr;
    void* pops[2] = {nullptr, nullptr};
    int cur = 0;                         // pops[cur] holds the post-collision field
    uint8_t* flags[2] = {nullptr, nullptr};
    int fcur = 0;                        // flags[fcur] are the flags of pops[cur]
    int* list = nullptr;                 // boundary cells
    int* count = nullptr;
    int list_cap = 0;
    uint8_t* link_mask = nullptr;        // uniform grids: marks of the box cells around the sphere (one byte each)
    int* seg = nullptr;                  // boundary cells by segment of the box (an entry per box cell)
    int* seg_count = nullptr;            // and their number per segment
    double* partials = nullptr;
    int* d_done = nullptr;               // last-block-done counter of the boundary CTAs (uniform grids)
    lbmp::PFrames* frames = nullptr;     // uniform grids: two copies of the sphere's frames, a step reads one
    int frame_cur = 0;                   // (frame_cur) while its particle update writes the other
    lbmp::ParticleState* d_ps = nullptr;       // of a RecordStatus, as status
    lbmp::ParticleState h_ps;                  // host copy of the parameters
    double* history = nullptr;
    int* status = nullptr;
    lbmp::BoxDesc box;
    bool has_particle = false;
    bool frames_stale = true;            // the host changed the particle record since the refined step formed its frames
    long long placed = 0;                // uniform grids: raised where the sphere's place may change (a step that does not
                                         // hold it, a load)
    bool ps_current = false;             // h_ps equals the device record (read with the status after a step)
    double tau = 0.6, magic = 3.0 / 16.0;
    double body_force[3] = {0, 0, 0};
    long long steps = 0, updates = 0, launches = 0, h2d = 0, d2h = 0;
    bool profiling = false;
    std::vector<cudaEvent_t> ev_pool;    // events of the current measurement
    size_t ev_used = 0;
    // (start, end) event indices of stream-collide launches with their algorithmic bytes and cell updates
    std::vector<std::pair<size_t, size_t>> prof_kernel;
    std::vector<double> prof_bytes, prof_updates;
    std::vector<std::pair<size_t, size_t>> prof_step;
    std::vector<std::pair<void*, size_t>> allocations;
    std::string err;
    lbmp::AmrEngine* amr = nullptr;     // refined hierarchy (levels > 1), else null
    lbmp::BatchEngine* batch = nullptr; // batched sweep, else null
    lbmp::AdjointEngine* adj = nullptr; // drag adjoint workspace, else null
};

namespace lbmp {

// s- from the magic parameter: Lambda = (1/s+ - 1/2)(1/s- - 1/2)  (Sec. 2.1)
inline void relaxation_rates(double tau, double magic, double* sp, double* sm) {
    *sp = 1.0 / tau;
    *sm = 1.0 / (0.5 + magic / (tau - 0.5));
}

// Coefficient of Grad's refill term for relaxation time tau (-3 (1 - s+)/s+,
// see refill_strain and grad_term), or 0 for the equilibrium refill.
inline double grad_refill_coef(int refill, double tau) {
    if (refill != LBMP_REFILL_GRAD) return 0.0;
    const double sp = 1.0 / tau;
    return -3.0 * (1.0 - sp) / sp;
}

// MRT bulk rate from the bulk factor: Lambda_b = (1/s_b - 1/2)/(1/s_nu - 1/2)
// (Sec. 2.1); returns s_b - s+, exactly 0 for Lambda_b = 1 (TRT).
inline double bulk_rate_offset(double tau, double bulk) {
    if (bulk == 1.0) return 0.0;
    return 1.0 / (0.5 + bulk * (tau - 0.5)) - 1.0 / tau;
}

template <typename A>
inline CollideParams<A> collide_params(const lbmp_handle* h) {
    CollideParams<A> p;
    double sp, sm;
    relaxation_rates(h->tau, h->magic, &sp, &sm);
    p.sp = (A)sp;
    p.sm = (A)sm;
    p.db = (A)bulk_rate_offset(h->tau, h->cfg.bulk_factor);
    for (int a = 0; a < 3; ++a) p.F[a] = (A)h->body_force[a];
    p.forced = (h->body_force[0] != 0.0 || h->body_force[1] != 0.0 || h->body_force[2] != 0.0) ? 1 : 0;
    if (h->cfg.precision == LBMP_FP16) {
        p.scale = (A)std::ldexp(1.0, h->cfg.fp16_scale_log2);
        p.inv_scale = (A)std::ldexp(1.0, -h->cfg.fp16_scale_log2);
    } else {
        p.scale = (A)1;
        p.inv_scale = (A)1;
    }
    collide_consts(p);
    return p;
}

}  // namespace lbmp

