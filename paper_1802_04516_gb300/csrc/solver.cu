// Per-step solve of the Schur velocity system, entirely on the device (Sec. 4,
// "... we can still solve the system using a matrix-free GMRES algorithm ..."; CG for the
// symmetric positive definite Crank-Nicolson case, Theorems 1-2).
//
// Every Krylov scalar (dot products, Hessenberg column, Givens rotations, residual
// estimate, loop flags) lives in device memory; loops are CUDA-graph WHILE nodes whose
// condition a small kernel sets with cudaGraphSetConditional, so one graph launch runs
// a whole time step with no host round trip.  With use_graph = 0 the same kernels run
// from a host loop that reads the flag after each body (a debugging aid).
//
// Several shots (right-hand sides on one mesh) are solved together: their vectors are
// stacked shot-major, the operator and preconditioner kernels load each face's and
// element's blocks once for all shots, and every Krylov scalar is kept PER SHOT, so each
// shot runs its own CG / GMRES recurrence (the same iterates as a solve of that shot
// alone) and stops at ||r_s|| <= rel_tol ||b_s||.  A shot that has converged is frozen
// (zero step length) while the others continue; the loops end when every shot has.
//
// Solvers
//   CG        (Crank-Nicolson)  r = b - A x; standard recurrences; FP64 dots.
//   GMRES(m)  (space-time DG)   restarted, classical Gram-Schmidt with a second
//                               pass only where the first one cancelled more than 99%
//                               of ||w||^2, Givens rotations on the device,
//                               true residual checked at every restart.
//   Mixed     FP64 iterative refinement around an FP32 CG / GMRES: r = b - A64 x in FP64,
//             solve A32 d = r/|r| to inner_tol, x += |r| d, stop at rel_tol in FP64.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "krylov.h"
#include "stdg_internal.h"

namespace stdg {

struct Workspace {
    int m = 30;
    int ns = 1;                   // shots
    int64_t nvec = 0;             // values per shot (velocity DOFs)
    int64_t n = 0, ldv = 0;       // stacked length, basis leading dimension
    unsigned G = 1;               // blocks per shot of the streaming kernels (grid G x ns)
    unsigned Gd = 1;              // blocks per shot of the multi-dot kernels
    unsigned red_blocks = 1;      // blocks of the single-vector streaming kernels
    DevScalars* sc = nullptr;
    ShotScalars* ss = nullptr;    // [ns]
    double* partials = nullptr;   // [slot][shot][block], (kMaxRestart + 2) slots
    unsigned* done = nullptr;     // [ns] blocks of a shot, [1] shots that have finished a reducing kernel
    double* dparams = nullptr;    // t^n, dt, step index
    double *pb = nullptr;         // second search direction of the fused CG
    float *pb32 = nullptr;
    double *V = nullptr, *w = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *z = nullptr, *t = nullptr;   // FP64
    float *V32 = nullptr, *w32 = nullptr, *b32 = nullptr, *x32 = nullptr, *r32 = nullptr, *p32 = nullptr, *q32 = nullptr;
    float *z32 = nullptr, *t32 = nullptr;
    cudaStream_t side[6] = {};
    int depth = 0;
    // cached graphs: [0] one whole step, [1] the solve alone (adjoint)
    cudaGraph_t graph[2] = {};
    cudaGraphExec_t exec[2] = {};
    double graph_dt[2] = {-1.0, -1.0};
    long body_kernels[2][kBodies] = {};   // kernels of each body, as recorded
    std::vector<void*> owned;   // device buffers of this workspace
    dim3 grid() const { return dim3(G, (unsigned)ns); }
    dim3 dot_grid() const { return dim3(Gd, (unsigned)ns); }
    // threads of the single-block control kernels: one per shot, at least a warp per ten shots
    int fin_threads() const { return std::min(kFinThreads, std::max(128, (ns + 31) / 32 * 96)); }
};

static Workspace* W(stdg_ctx* c) { return reinterpret_cast<Workspace*>(c->ws); }

// 16-byte vector access: VW = 4 floats or 2 doubles per load/store.  Every pointer that is
// vectorised is 16-byte aligned (separate allocations, or basis columns at a leading
// dimension that is a multiple of 64 elements).
template <typename R> struct VL;
template <> struct VL<float> {
    static constexpr int W = 4;
    __device__ __forceinline__ static void ld(const float* p, float (&o)[4]) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    }
    __device__ __forceinline__ static void st(float* p, const float (&o)[4]) {
        *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
    }
};
template <> struct VL<double> {
    static constexpr int W = 2;
    __device__ __forceinline__ static void ld(const double* p, double (&o)[2]) {
        const double2 t = *reinterpret_cast<const double2*>(p);
        o[0] = t.x; o[1] = t.y;
    }
    __device__ __forceinline__ static void st(double* p, const double (&o)[2]) {
        *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
    }
};

// Streaming over one shot's segment [s*nvec, (s+1)*nvec), s = blockIdx.y, by the
// gridDim.x blocks of that shot: fv(i) handles the VW values from i (i a multiple of VW),
// fs(i) one value of the unaligned head or tail (thread 0 of the shot's first block).
template <typename R, class FV, class FS>
__device__ __forceinline__ void seg_loop(int64_t nvec, FV&& fv, FS&& fs) {
    constexpr int VW = VL<R>::W;
    const int64_t lo = (int64_t)blockIdx.y * nvec, hi = lo + nvec;
    const int64_t a0 = min(hi, (lo + VW - 1) / VW * VW);
    const int64_t a1 = max(a0, hi / VW * VW);
    for (int64_t g = a0 / VW + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < a1 / VW;
         g += (int64_t)gridDim.x * blockDim.x)
        fv(g * VW);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int64_t i = lo; i < a0; ++i) fs(i);
        for (int64_t i = a1; i < hi; ++i) fs(i);
    }
}

// block's partial sum into slot k of its shot
__device__ __forceinline__ void put_partial(double* part, int k, double v) {
    const double s = block_sum(v);
    if (threadIdx.x == 0) part[((int64_t)k * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
}

template <typename R>
__device__ __forceinline__ void put_acc(double* part, int k, const Acc<R>& v) {
    const double s = block_sum1(v);
    if (threadIdx.x == 0) part[((int64_t)k * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
}

// per-shot dot products a_s . b_s into slot k
template <typename A, typename B>
__global__ void dot_partial_kernel(int64_t nvec, const A* __restrict__ a, const B* __restrict__ b, double* __restrict__ part,
                                   int k) {
    Acc<A> acc;
    const int64_t lo = (int64_t)blockIdx.y * nvec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x)
        acc.add(a[lo + i], b[lo + i]);
    put_acc(part, k, acc);
}

// x_s = 0 for the shots whose right-hand side is zero (level 0: Krylov, 1: refinement)
__global__ void zero_if_kernel(int64_t nvec, double* x, const ShotScalars* ss, int level) {
    if (!(level ? ss[blockIdx.y].ir_zero : ss[blockIdx.y].zero_x)) return;
    const int64_t lo = (int64_t)blockIdx.y * nvec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x)
        x[lo + i] = 0;
}

// ---------------------------------------------------------------------------------
// (Preconditioned) CG kernels (R = vector type, scalars FP64, one recurrence per shot).
// Without a preconditioner z aliases r and rz = rr.
// ---------------------------------------------------------------------------------
template <typename R>
__global__ void cg_res_kernel(int64_t nvec, const R* __restrict__ b, const R* __restrict__ Ax, R* __restrict__ r,
                              double* __restrict__ part) {
    double rr = 0, bb = 0;
    const int64_t lo = (int64_t)blockIdx.y * nvec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x) {
        const R ri = b[lo + i] - Ax[lo + i];
        r[lo + i] = ri;
        rr += (double)ri * (double)ri;
        bb += (double)b[lo + i] * (double)b[lo + i];
    }
    put_partial(part, 0, rr);
    put_partial(part, 1, bb);
}

// bnorm_given < 0: use ||b_s|| from the partials; slots: 0 rr, 1 bb, 2 rz
__global__ void __launch_bounds__(kFinThreads) cg_init_final_kernel(DevScalars* sc, ShotScalars* ss, const double* part,
                                                                    int ns, int G, double rel_tol, int max_iters,
                                                                    double bnorm_given, int gate_ir,
                                                                    cudaGraphConditionalHandle h, int use_h) {
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int q = warp; q < 3 * ns; q += nw) {
        const double v = warp_sum(slot(part, q % 3, q / 3, ns, G), G);
        if ((threadIdx.x & 31) == 0) ss[q / 3].red[q % 3] = v;
    }
    __syncthreads();
    const int active = gate_ir ? sc->ir_flag : 1;
    int any = 0;
    for (int s = threadIdx.x; s < ns; s += blockDim.x) {
        ShotScalars& t = ss[s];
        t.rr = t.red[0];
        t.pq = t.red[2];                   // holds r.z between iterations
        t.bnorm = bnorm_given >= 0 ? bnorm_given : sqrt(t.red[1]);
        t.tol_abs = rel_tol * t.bnorm;
        t.zero_x = active && t.bnorm == 0.0;
        t.converged = !active || sqrt(t.rr) <= t.tol_abs;
        t.active = !t.converged && isfinite(t.rr) && isfinite(t.bnorm);   // a NaN/Inf residual stops the shot
        t.alpha = t.beta = 0.0;
        any |= t.active;
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
        sc->iters = 0;
        sc->max_iters = max_iters;
        sc->flag_inner = any && max_iters > 0;
        set_cond(h, use_h, sc->flag_inner);
    }
}

template <typename R>
__global__ void copy_kernel(int64_t n, const R* __restrict__ a, R* __restrict__ b) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) b[i] = a[i];
}

// p.q of each shot; the shot's last block forms alpha_s = (r.z)_s / (p.q)_s (0 for a frozen shot)
template <typename R>
__global__ void cg_dot_alpha_kernel(int64_t nvec, const R* __restrict__ p, const R* __restrict__ q, double* part,
                                    ShotScalars* ss, unsigned* done) {
    const int s = blockIdx.y, G = gridDim.x;
    if (!ss[s].active) return;
    Acc<R> acc;
    const int64_t lo = (int64_t)s * nvec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)G * blockDim.x)
        acc.add(p[lo + i], q[lo + i]);
    put_acc(part, 0, acc);
    if (!last_block(done + s, G) || threadIdx.x >= 32) return;
    const double pq = warp_sum(slot(part, 0, s, gridDim.y, G), G);
    if (threadIdx.x == 0) ss[s].alpha = pq != 0.0 ? ss[s].pq / pq : 0.0;
}

template <typename R>
__global__ void cg_update_kernel(int64_t nvec, const ShotScalars* __restrict__ ss, R* __restrict__ x, R* __restrict__ r,
                                 const R* __restrict__ p, const R* __restrict__ q, double* __restrict__ part) {
    if (!ss[blockIdx.y].active) return;
    const double a = ss[blockIdx.y].alpha;
    const int64_t lo = (int64_t)blockIdx.y * nvec;
    double rr = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x) {
        x[lo + i] = (R)((double)x[lo + i] + a * (double)p[lo + i]);
        const R ri = (R)((double)r[lo + i] - a * (double)q[lo + i]);
        r[lo + i] = ri;
        rr += (double)ri * (double)ri;
    }
    put_partial(part, 0, rr);
}

// r.z of each shot (slot 2; slot 0 holds the parts of r.r); the shot's last block forms beta_s and
// the convergence test, and the last shot to get there advances the loop
template <typename R>
__global__ void cg_dot_beta_kernel(int64_t nvec, const R* __restrict__ r, const R* __restrict__ z, double* part,
                                   DevScalars* sc, ShotScalars* ss, unsigned* done, cudaGraphConditionalHandle h, int use_h) {
    const int s = blockIdx.y, ns = gridDim.y, G = gridDim.x;
    ShotScalars& t = ss[s];
    if (t.active) {
        Acc<R> acc;
        const int64_t lo = (int64_t)s * nvec;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)G * blockDim.x)
            acc.add(r[lo + i], z[lo + i]);
        put_acc(part, 2, acc);
    }
    if (!last_block(done + s, G) || threadIdx.x >= 32) return;
    if (t.active) {
        const double rr = warp_sum(slot(part, 0, s, ns, G), G);
        const double rz = warp_sum(slot(part, 2, s, ns, G), G);
        if (threadIdx.x == 0) {
            t.beta = t.pq != 0.0 ? rz / t.pq : 0.0;
            t.pq = rz;
            t.rr = rr;
            t.converged = sqrt(rr) <= t.tol_abs;
            t.active = !t.converged && isfinite(rr);
        }
    }
    if (threadIdx.x != 0) return;
    if (t.active) atomicOr(&sc->any, 1);
    __threadfence();
    if (atomicInc(done + ns, ns - 1) != (unsigned)ns - 1) return;
    sc->iters += 1;
    sc->runs[kBodyInner] += 1;
    sc->flag_inner = atomicExch(&sc->any, 0) && sc->iters < sc->max_iters;
    set_cond(h, use_h, sc->flag_inner);
}

template <typename R>
__global__ void cg_p_kernel(int64_t nvec, const ShotScalars* __restrict__ ss, const R* __restrict__ z, R* __restrict__ p) {
    if (!ss[blockIdx.y].active) return;
    const double b = ss[blockIdx.y].beta;
    const int64_t lo = (int64_t)blockIdx.y * nvec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x)
        p[lo + i] = (R)((double)z[lo + i] + b * (double)p[lo + i]);
}

// ---------------------------------------------------------------------------------
// GMRES kernels (one Arnoldi process and one Hessenberg matrix per shot)
// ---------------------------------------------------------------------------------
// r = b - A x into v0; with start != 0 the last block of each shot also opens a restart cycle:
// beta_s = ||r_s|| (the true residual), convergence test, g = beta_s e_1
template <typename R>
__global__ void gm_res_kernel(int64_t nvec, const R* __restrict__ b, const R* __restrict__ Ax, R* __restrict__ v0,
                             double* __restrict__ part, int start, DevScalars* sc, ShotScalars* ss, unsigned* done,
                             cudaGraphConditionalHandle h, int use_h) {
    constexpr int VW = VL<R>::W;
    Acc<R> rr;
    seg_loop<R>(nvec,
        [&](int64_t i) {
            R bb[VW], aa[VW];
            VL<R>::ld(b + i, bb);
            VL<R>::ld(Ax + i, aa);
#pragma unroll
            for (int u = 0; u < VW; ++u) { bb[u] -= aa[u]; rr.add(bb[u], bb[u]); }
            VL<R>::st(v0 + i, bb);
        },
        [&](int64_t i) { const R ri = b[i] - Ax[i]; v0[i] = ri; rr.add(ri, ri); });
    put_acc(part, 0, rr);
    if (!start) return;
    const int s = blockIdx.y, ns = gridDim.y, G = gridDim.x;
    if (!last_block(done + s, G)) return;
    ShotScalars& t = ss[s];
    for (int k = threadIdx.x; k <= sc->m; k += blockDim.x) t.g[k] = 0.0;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const double beta = sqrt(warp_sum(slot(part, 0, s, ns, G), G));
    if (threadIdx.x != 0) return;
    t.gbeta = beta;
    t.resid = beta;
    t.jj = 0;
    if (!t.converged) t.converged = beta <= t.tol_abs;
    t.active = !t.converged && isfinite(beta) && isfinite(t.tol_abs);   // a NaN/Inf residual stops the shot
    t.g[0] = beta;
    if (t.active) atomicOr(&sc->any, 1);
    __threadfence();
    if (atomicInc(done + ns, ns - 1) != (unsigned)ns - 1) return;
    sc->j = 0;
    sc->flag_inner = atomicExch(&sc->any, 0) && sc->iters < sc->max_iters;
    set_cond(h, use_h, sc->flag_inner);
}

// set up one GMRES solve: ||b_s|| (from slot 0, or given), tolerances, counters
__global__ void __launch_bounds__(kFinThreads) gm_init_kernel(DevScalars* sc, ShotScalars* ss, const double* part, int ns,
                                                              int G, double rel_tol, int max_iters, int m,
                                                              double bnorm_given, int gate_ir,
                                                              cudaGraphConditionalHandle h, int use_h) {
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (bnorm_given < 0)
        for (int s = warp; s < ns; s += nw) {
            const double v = warp_sum(slot(part, 0, s, ns, G), G);
            if ((threadIdx.x & 31) == 0) ss[s].red[0] = v;
        }
    __syncthreads();
    const int active = gate_ir ? sc->ir_flag : 1;
    int any = 0;
    for (int s = threadIdx.x; s < ns; s += blockDim.x) {
        ShotScalars& t = ss[s];
        t.bnorm = bnorm_given >= 0 ? bnorm_given : sqrt(t.red[0]);
        t.tol_abs = rel_tol * t.bnorm;
        t.zero_x = active && t.bnorm == 0.0;
        t.converged = !active || t.zero_x;
        t.active = 0;
        t.jj = 0;
        any |= !t.converged;
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
        sc->iters = 0;
        sc->max_iters = max_iters;
        sc->m = m;
        sc->j = 0;
        sc->flag_outer = any;
        set_cond(h, use_h, sc->flag_outer);
    }
}

template <typename R>
__global__ void gm_scale0_kernel(int64_t nvec, const DevScalars* __restrict__ sc, const ShotScalars* __restrict__ ss,
                                 R* __restrict__ v0) {
    if (!sc->flag_inner) return;
    constexpr int VW = VL<R>::W;
    const double gb = ss[blockIdx.y].gbeta;
    const R s = (R)(gb > 0.0 ? 1.0 / gb : 0.0);
    seg_loop<R>(nvec,
        [&](int64_t i) {
            R a[VW];
            VL<R>::ld(v0 + i, a);
#pragma unroll
            for (int u = 0; u < VW; ++u) a[u] *= s;
            VL<R>::st(v0 + i, a);
        },
        [&](int64_t i) { v0[i] *= s; });
}

// Accumulates V_k . w over the values at i for the kn <= kDotChunk columns from k0.  The columns
// are loaded kDotLoads at a time before the first is used: with one 16-byte load per column in
// flight the kernel waited on memory (long scoreboard) at 0.4-0.5 of the DRAM rate.
template <typename R, int VW>
__device__ __forceinline__ void dot_columns(const R* __restrict__ V, int64_t ldv, int64_t i, int kn, const R (&wv)[VW],
                                            Acc<R> (&acc)[kDotChunk]) {
#pragma unroll
    for (int g = 0; g < kDotChunk; g += kDotLoads) {
        if (g >= kn) break;
        R vv[kDotLoads][VW];
#pragma unroll
        for (int kk = 0; kk < kDotLoads; ++kk)
            if (g + kk < kn) VL<R>::ld(V + (int64_t)(g + kk) * ldv + i, vv[kk]);
#pragma unroll
        for (int kk = 0; kk < kDotLoads; ++kk)
            if (g + kk < kn) {
#pragma unroll
                for (int u = 0; u < VW; ++u) acc[g + kk].add(vv[kk][u], wv[u]);
            }
    }
}

// the block's sums of acc[0..kn) into slots k0.. of its shot
template <typename R>
__device__ __forceinline__ void put_chunk(double* part, int k0, int kn, Acc<R> (&acc)[kDotChunk]) {
    const double s = block_sum16(acc);
    if ((int)threadIdx.x < kn) part[((int64_t)(k0 + threadIdx.x) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
}

// v[i] - sum_k h_k V_k[i], four columns loaded before the first is used
template <typename R, int VW>
__device__ __forceinline__ void subtract_columns(const R* __restrict__ V, int64_t ldv, int64_t i, int n, const R* h,
                                                 R (&wv)[VW]) {
    int k = 0;
    for (; k + 4 <= n; k += 4) {
        R vv[4][VW];
#pragma unroll
        for (int q = 0; q < 4; ++q) VL<R>::ld(V + (int64_t)(k + q) * ldv + i, vv[q]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < VW; ++u) wv[u] = fma(-h[k + q], vv[q][u], wv[u]);
    }
    for (; k < n; ++k) {
        R vv[VW];
        VL<R>::ld(V + (int64_t)k * ldv + i, vv);
#pragma unroll
        for (int u = 0; u < VW; ++u) wv[u] = fma(-h[k], vv[u], wv[u]);
    }
}

// First classical Gram-Schmidt pass: V_k . w (k = 0..j) and ||w||^2 of every shot still iterating;
// the shot's last block sums the blocks' parts, starts the Hessenberg column and decides whether
// the second pass is needed: one pass leaves w orthogonal to the basis to about
// eps ||w|| / ||w - V h||, so the pass is repeated when that ratio would exceed 10, i.e. when
// ||w - V h||^2 = ||w||^2 - |h|^2 < 1e-2 ||w||^2 (V orthonormal; the dots are FP64-accurate).
// The grid is sized by the vector: one 16-byte item a thread, at most two blocks an SM (128
// registers, eight columns in flight a thread).  Measured with 13 FP64 columns of 291,600 values:
// 24 us, where a fixed grid of 1,216 blocks with one block-wide reduction per column and a
// single-block final kernel took 78 + 13 us; with ten FP32 columns of 16,056,320 values 127 us
// (5.6 TB/s) against 210 + 13 us.  Short vectors stay at the chain of its dependent accesses, 8 us.
template <typename R>
__global__ void __launch_bounds__(256, 2) gm_mdot_kernel(int64_t nvec, int64_t ldv, const DevScalars* __restrict__ sc,
                                                      ShotScalars* ss, const R* __restrict__ V, const R* __restrict__ w,
                                                      double* part, unsigned* done) {
    constexpr int VW = VL<R>::W;
    const int J = sc->j, s = blockIdx.y, ns = gridDim.y, G = gridDim.x;
    if (!ss[s].active) return;
    for (int k0 = 0; k0 <= J; k0 += kDotChunk) {
        Acc<R> acc[kDotChunk];
        Acc<R> ww;                                // ||w||^2, first chunk only
        const int kn = min(kDotChunk, J + 1 - k0);
        const R* Vk = V + (int64_t)k0 * ldv;
        seg_loop<R>(nvec,
            [&](int64_t i) {
                R wv[VW];
                VL<R>::ld(w + i, wv);
                dot_columns<R, VW>(Vk, ldv, i, kn, wv, acc);
                if (k0 == 0) {
#pragma unroll
                    for (int u = 0; u < VW; ++u) ww.add(wv[u], wv[u]);
                }
            },
            [&](int64_t i) {
                if (k0 == 0) ww.add(w[i], w[i]);
#pragma unroll
                for (int kk = 0; kk < kDotChunk; ++kk)
                    if (kk < kn) acc[kk].add(Vk[(int64_t)kk * ldv + i], w[i]);
            });
        put_chunk<R>(part, k0, kn, acc);
        if (k0 == 0) put_acc(part, J + 1, ww);
    }
    if (!last_block(done + s, G)) return;
    ShotScalars& t = ss[s];
    __shared__ double h[kMaxRestart + 2];
    for (int k = threadIdx.x >> 5; k <= J + 1; k += blockDim.x >> 5) {
        const double v = warp_sum(slot(part, k, s, ns, G), G);
        if ((threadIdx.x & 31) == 0) {
            h[k] = v;
            if (k <= J) t.hpass[k] = t.hcol[k] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double h2 = 0.0;
    for (int k = threadIdx.x; k <= J; k += 32) h2 += h[k] * h[k];
    for (int o = 16; o > 0; o >>= 1) h2 += __shfl_xor_sync(0xffffffffu, h2, o);
    if (threadIdx.x == 0) t.reorth = h[J + 1] - h2 < 1e-2 * h[J + 1];
}

// Second Gram-Schmidt pass fused with the first subtraction, only for the shots that need it:
// w_s <- w_s - sum_k h1_s[k] V_k, then V_k . w_s for the re-orthogonalisation; the shot's last
// block adds the second pass to the Hessenberg column.
template <typename R>
__global__ void __launch_bounds__(256, 2) gm_orth_fused_kernel(int64_t nvec, int64_t ldv, const DevScalars* __restrict__ sc,
                                                            ShotScalars* ss, const R* __restrict__ V,
                                                            R* __restrict__ w, double* part, unsigned* done) {
    constexpr int VW = VL<R>::W;
    const int J = sc->j, s = blockIdx.y, ns = gridDim.y, G = gridDim.x;
    if (!ss[s].active || !ss[s].reorth) return;   // this shot's first pass was enough
    __shared__ R h[kMaxRestart + 2];
    for (int k = threadIdx.x; k <= J; k += blockDim.x) h[k] = (R)ss[s].hpass[k];
    __syncthreads();
    for (int k0 = 0; k0 <= J; k0 += kDotChunk) {
        Acc<R> acc[kDotChunk];
        const int kn = min(kDotChunk, J + 1 - k0);
        const R* Vk = V + (int64_t)k0 * ldv;
        seg_loop<R>(nvec,
            [&](int64_t i) {
                R wv[VW];
                VL<R>::ld(w + i, wv);
                if (k0 == 0) {   // first chunk: form and store the projected w (in the vector precision)
                    subtract_columns<R, VW>(V, ldv, i, J + 1, h, wv);
                    VL<R>::st(w + i, wv);
                }
                dot_columns<R, VW>(Vk, ldv, i, kn, wv, acc);
            },
            [&](int64_t i) {
                R wi = w[i];
                if (k0 == 0) {
                    for (int k = 0; k <= J; ++k) wi = fma(-h[k], V[(int64_t)k * ldv + i], wi);
                    w[i] = wi;
                }
#pragma unroll
                for (int kk = 0; kk < kDotChunk; ++kk)
                    if (kk < kn) acc[kk].add(Vk[(int64_t)kk * ldv + i], wi);
            });
        put_chunk<R>(part, k0, kn, acc);
    }
    if (!last_block(done + s, G)) return;
    ShotScalars& t = ss[s];
    for (int k = threadIdx.x >> 5; k <= J; k += blockDim.x >> 5) {
        const double v = warp_sum(slot(part, k, s, ns, G), G);
        if ((threadIdx.x & 31) == 0) {
            t.hpass[k] = v;
            t.hcol[k] += v;
        }
    }
}

// w_s -= sum_k hpass_s[k] V_k and ||w_s||.  The shot's last block closes the Arnoldi step: Givens
// rotations of the new Hessenberg column, residual estimate; the shot stops at its residual
// estimate or on breakdown and keeps the columns it has (jj).  The last shot to get there advances
// the loop.  For short vectors the kernel is a chain of dependent memory accesses (about 0.6 us
// each), so everything that the closing needs is loaded beside the coefficients, before the vector:
// 9 us for 2,352 values, against 18 + 9 + 10 us for the subtraction and its two single-block kernels.
template <typename R>
__global__ void __launch_bounds__(256) gm_maxpy_kernel(int64_t nvec, int64_t ldv, DevScalars* sc, ShotScalars* ss,
                                                       const R* __restrict__ V, R* __restrict__ w, double* part,
                                                       unsigned* done, cudaGraphConditionalHandle handle, int use_h) {
    constexpr int VW = VL<R>::W;
    const int J = sc->j, s = blockIdx.y, ns = gridDim.y, G = gridDim.x;
    const int iters = sc->iters, max_iters = sc->max_iters, m = sc->m;
    const unsigned runs = sc->runs[kBodyInner];
    __shared__ R h[kMaxRestart + 2];
    __shared__ double hc[kMaxRestart + 2], cs[kMaxRestart], sn[kMaxRestart];
    ShotScalars& t = ss[s];
    int active = t.active;
    const double g = t.g[J], tol = t.tol_abs;
    if (active) {
        for (int k = threadIdx.x; k <= J; k += blockDim.x) {
            h[k] = (R)t.hpass[k];
            hc[k] = t.hcol[k];
            cs[k] = t.cs[k];
            sn[k] = t.sn[k];
        }
        __syncthreads();
        Acc<R> nn;
        seg_loop<R>(nvec,
            [&](int64_t i) {
                R wv[VW];
                VL<R>::ld(w + i, wv);
                subtract_columns<R, VW>(V, ldv, i, J + 1, h, wv);
                VL<R>::st(w + i, wv);
#pragma unroll
                for (int u = 0; u < VW; ++u) nn.add(wv[u], wv[u]);
            },
            [&](int64_t i) {
                R wi = w[i];
                for (int k = 0; k <= J; ++k) wi = fma(-h[k], V[(int64_t)k * ldv + i], wi);
                w[i] = wi;
                nn.add(wi, wi);
            });
        put_acc(part, 0, nn);
    }
    if (!last_block(done + s, G)) return;
    if (active) {
        double v = 0;
        const double* p = slot(part, 0, s, ns, G);
        for (int i = threadIdx.x; i < G; i += blockDim.x) v += __ldcg(p + i);
        v = block_sum(v);   // ||w||^2 in thread 0
        if (threadIdx.x < 32) {
            v = __shfl_sync(0xffffffffu, v, 0);
            double hi = hc[0];
            for (int i = 0; i < J; ++i) {   // every lane alike
                const double hn = hc[i + 1];
                const double u = cs[i] * hi + sn[i] * hn;
                hi = -sn[i] * hi + cs[i] * hn;
                __syncwarp();
                if (threadIdx.x == 0) hc[i] = u;
            }
            // one square root and one division for the warp: lane 0 the rotated diagonal, lane 1 ||w||
            const double root = sqrt(threadIdx.x == 0 ? fma(hi, hi, v) : v);
            const double den = __shfl_sync(0xffffffffu, root, 0), b = __shfl_sync(0xffffffffu, root, 1);
            const double bot = threadIdx.x == 2 ? b : den;
            const double quo = (threadIdx.x == 0 ? hi : threadIdx.x == 1 ? b : 1.0) / (bot > 0.0 ? bot : 1.0);
            const double q0 = __shfl_sync(0xffffffffu, quo, 0), q1 = __shfl_sync(0xffffffffu, quo, 1);
            const double q2 = __shfl_sync(0xffffffffu, quo, 2);
            const double c = den > 0.0 ? q0 : 1.0, q = den > 0.0 ? q1 : 0.0, resid = fabs(q * g);
            if (resid <= tol || den == 0.0 || !isfinite(resid)) active = 0;
            if (threadIdx.x == 0) {
                hc[J] = den;
                t.cs[J] = c;
                t.sn[J] = q;
                t.vscale = b > 0.0 ? q2 : 0.0;
                t.g[J + 1] = -q * g;
                t.g[J] = c * g;
                t.resid = resid;
                t.jj = J + 1;
                t.active = active;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i <= J; i += blockDim.x) t.H[i * kMaxRestart + J] = hc[i];
    }
    if (threadIdx.x != 0) return;
    if (ns > 1) {
        if (active) atomicOr(&sc->any, 1);
        __threadfence();
        if (atomicInc(done + ns, ns - 1) != (unsigned)ns - 1) return;
        active = atomicExch(&sc->any, 0);
    }
    sc->iters = iters + 1;
    sc->j = J + 1;
    sc->runs[kBodyInner] = runs + 1;
    const int go = active && J + 1 < m && iters + 1 < max_iters;
    sc->flag_inner = go;
    set_cond(handle, use_h, go);
}

// V_{j} = w / ||w|| for the next step (j already advanced), while the cycle goes on
template <typename R>
__global__ void gm_next_kernel(int64_t nvec, int64_t ldv, const DevScalars* __restrict__ sc,
                               const ShotScalars* __restrict__ ss, const R* __restrict__ w, R* __restrict__ V) {
    constexpr int VW = VL<R>::W;
    if (!sc->flag_inner || !ss[blockIdx.y].active) return;
    const R s = (R)ss[blockIdx.y].vscale;
    R* vn = V + (int64_t)sc->j * ldv;
    seg_loop<R>(nvec,
        [&](int64_t i) {
            R a[VW];
            VL<R>::ld(w + i, a);
#pragma unroll
            for (int u = 0; u < VW; ++u) a[u] *= s;
            VL<R>::st(vn + i, a);
        },
        [&](int64_t i) { vn[i] = w[i] * s; });
}

// y = R^{-1} g (upper triangular, size J) of one shot, by every block that needs it: the triangle
// through shared memory, then one warp eliminates column by column (two unknowns a lane).
__device__ __forceinline__ void triangular_solve(const ShotScalars& t, int J, double* sH, double* y) {
    for (int q = threadIdx.x; q < J * J; q += blockDim.x) sH[q] = t.H[(q / J) * kMaxRestart + q % J];
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        double g[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) g[u] = lane + 32 * u < J ? t.g[lane + 32 * u] : 0.0;
        for (int k = J - 1; k >= 0; --k) {
            const double d = sH[k * J + k];
            const double gk = __shfl_sync(0xffffffffu, k < 32 ? g[0] : g[1], k & 31);
            const double yk = d != 0.0 ? gk / d : 0.0;
            if (lane == 0) y[k] = yk;
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (lane + 32 * u < k) g[u] -= sH[(lane + 32 * u) * J + k] * yk;
        }
    }
    __syncthreads();
}

// x_s += sum_{k<jj_s} y_s[k] V_k  (accumulate = 1), or t_s = sum_k y_s[k] V_k (accumulate = 0;
// right preconditioning applies P^{-1} to t afterwards), y_s = R_s^{-1} g_s
template <typename R>
__global__ void __launch_bounds__(256) gm_combine_kernel(int64_t nvec, int64_t ldv, const ShotScalars* __restrict__ ss,
                                                         const R* __restrict__ V, R* __restrict__ x, int accumulate) {
    constexpr int VW = VL<R>::W;
    const int J = ss[blockIdx.y].jj;
    if (accumulate && J == 0) return;
    __shared__ double sH[kMaxRestart * kMaxRestart], yd[kMaxRestart];
    __shared__ R y[kMaxRestart];
    triangular_solve(ss[blockIdx.y], J, sH, yd);
    for (int k = threadIdx.x; k < J; k += blockDim.x) y[k] = (R)(-yd[k]);
    __syncthreads();
    seg_loop<R>(nvec,
        [&](int64_t i) {
            R a[VW];
            if (accumulate) VL<R>::ld(x + i, a);
            else {
#pragma unroll
                for (int u = 0; u < VW; ++u) a[u] = 0;
            }
            subtract_columns<R, VW>(V, ldv, i, J, y, a);
            VL<R>::st(x + i, a);
        },
        [&](int64_t i) {
            R a = accumulate ? x[i] : (R)0;
            for (int k = 0; k < J; ++k) a = fma(-y[k], V[(int64_t)k * ldv + i], a);
            x[i] = a;
        });
}

template <typename R>
__global__ void axpy_kernel(int64_t n, R* __restrict__ x, const R* __restrict__ z) {
    constexpr int VW = VL<R>::W;
    const int64_t nv = n / VW;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < nv; g += (int64_t)gridDim.x * blockDim.x) {
        R a[VW], b[VW];
        VL<R>::ld(x + g * VW, a);
        VL<R>::ld(z + g * VW, b);
#pragma unroll
        for (int u = 0; u < VW; ++u) a[u] += b[u];
        VL<R>::st(x + g * VW, a);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        for (int64_t i = nv * VW; i < n; ++i) x[i] += z[i];
}

__global__ void __launch_bounds__(kFinThreads) gm_cycle_end_kernel(DevScalars* sc, const ShotScalars* ss, int ns,
                                                                   cudaGraphConditionalHandle h, int use_h) {
    int any = 0;
    for (int s = threadIdx.x; s < ns; s += blockDim.x) any |= !ss[s].converged;
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
        // a cycle without an Arnoldi step (every unconverged shot has a NaN or Inf residual) left x as it
        // was: the next one could do no better
        const int go = any && sc->j > 0 && sc->iters < sc->max_iters;
        sc->j = 0;
        sc->runs[kBodyCycle] += 1;
        sc->flag_outer = go;
        set_cond(h, use_h, sc->flag_outer);
    }
}

// ---------------------------------------------------------------------------------
// FP64 iterative refinement around the FP32 solver (per shot)
// ---------------------------------------------------------------------------------
__global__ void __launch_bounds__(kFinThreads) ir_init_kernel(DevScalars* sc, ShotScalars* ss, const double* part, int ns,
                                                              int G, double rel_tol, int ir_max,
                                                              cudaGraphConditionalHandle h, int use_h) {
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int s = warp; s < ns; s += nw) {
        const double v = warp_sum(slot(part, 0, s, ns, G), G);
        if ((threadIdx.x & 31) == 0) ss[s].red[0] = v;
    }
    __syncthreads();
    int any = 0;
    for (int s = threadIdx.x; s < ns; s += blockDim.x) {
        ShotScalars& t = ss[s];
        t.ir_bnorm = sqrt(t.red[0]);
        t.ir_tol_abs = rel_tol * t.ir_bnorm;
        t.ir_rnorm = t.ir_bnorm;
        t.ir_zero = t.ir_bnorm == 0.0;
        t.ir_conv = t.ir_zero;
        any |= !t.ir_conv && isfinite(t.ir_bnorm);
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
        sc->ir_count = 0;
        sc->ir_max = ir_max;
        sc->ir_flag = any;
        set_cond(h, use_h, sc->ir_flag);
    }
}

__global__ void __launch_bounds__(kFinThreads) ir_check_kernel(DevScalars* sc, ShotScalars* ss, const double* part, int ns,
                                                               int G, int max_total) {
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int s = warp; s < ns; s += nw) {
        const double v = warp_sum(slot(part, 0, s, ns, G), G);
        if ((threadIdx.x & 31) == 0) ss[s].red[0] = v;
    }
    __syncthreads();
    int any = 0;
    for (int s = threadIdx.x; s < ns; s += blockDim.x) {
        ShotScalars& t = ss[s];
        t.ir_rnorm = sqrt(t.red[0]);
        t.ir_conv = t.ir_zero || t.ir_rnorm <= t.ir_tol_abs;
        t.ir_scale = !t.ir_conv && t.ir_rnorm > 0.0 ? 1.0 / t.ir_rnorm : 0.0;
        any |= !t.ir_conv && isfinite(t.ir_rnorm) && isfinite(t.ir_bnorm);   // no refinement of a NaN/Inf residual
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) sc->ir_flag = any && sc->ir_count < sc->ir_max && sc->st_total < max_total;
}

// r32_s = r64_s * scale_s (0 for converged shots); x32 = 0   (when the refinement continues)
__global__ void ir_convert_kernel(int64_t nvec, const DevScalars* __restrict__ sc, const ShotScalars* __restrict__ ss,
                                  const double* __restrict__ r64, float* __restrict__ r32, float* __restrict__ x32) {
    if (!sc->ir_flag) return;
    const double s = ss[blockIdx.y].ir_scale;
    const int64_t lo = (int64_t)blockIdx.y * nvec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x) {
        r32[lo + i] = (float)(r64[lo + i] * s);
        x32[lo + i] = 0.0f;
    }
}

// x_s += |r_s| x32_s
__global__ void ir_update_kernel(int64_t nvec, const DevScalars* __restrict__ sc, const ShotScalars* __restrict__ ss,
                                 const float* __restrict__ x32, double* __restrict__ x) {
    if (!sc->ir_flag || ss[blockIdx.y].ir_conv) return;
    const double s = ss[blockIdx.y].ir_rnorm;
    const int64_t lo = (int64_t)blockIdx.y * nvec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x)
        x[lo + i] += s * (double)x32[lo + i];
}

__global__ void ir_end_kernel(DevScalars* sc, cudaGraphConditionalHandle h, int use_h) {
    if (threadIdx.x != 0) return;
    sc->runs[kBodyIr] += 1;
    if (sc->ir_flag) {
        sc->ir_count += 1;
        sc->st_total += sc->iters;
    }
    set_cond(h, use_h, sc->ir_flag);
}

// per-solve statistics (worst shot); mode 0 = GMRES, 1 = CG, 2 = mixed (refinement level)
__global__ void __launch_bounds__(kFinThreads) solve_stats_kernel(DevScalars* sc, const ShotScalars* ss, int ns, int mode) {
    __shared__ double worst[kFinThreads];
    double rel = 0.0;
    int notconv = 0, nonfinite = 0;
    for (int s = threadIdx.x; s < ns; s += blockDim.x) {
        const ShotScalars& t = ss[s];
        double r, bn;
        if (mode == 2) { r = t.ir_zero ? 0.0 : t.ir_rnorm; bn = t.ir_bnorm; notconv |= !t.ir_conv; }
        else { r = t.zero_x ? 0.0 : mode == 1 ? sqrt(t.rr) : t.resid; bn = t.bnorm; notconv |= !t.converged; }
        nonfinite |= !isfinite(r) || !isfinite(bn);
        rel = fmax(rel, bn > 0 ? r / bn : 0.0);
    }
    worst[threadIdx.x] = rel;
    notconv = __syncthreads_or(notconv);
    nonfinite = __syncthreads_or(nonfinite);
    if (threadIdx.x != 0) return;
    for (int i = 1; i < (int)blockDim.x; ++i) rel = fmax(rel, worst[i]);
    int it;
    if (mode == 2) {
        it = sc->st_total;          // accumulated by ir_end over the refinement sweeps
        sc->st_total = 0;
        sc->st_refine += sc->ir_count;
    } else {
        it = sc->iters;
    }
    sc->runs[kBodyStraight] += 1;
    if (notconv) sc->st_notconv = 1;
    if (nonfinite) sc->st_nonfinite = 1;
    sc->st_final_rel = rel;
    sc->st_max = max(sc->st_max, it);
    sc->st_iters_sum += (double)it;
}

__global__ void step_begin_kernel(double* dparams, double dt) {
    if (threadIdx.x == 0) dparams[1] = dt;
}
__global__ void step_end_kernel(double* dparams, double dt) {
    if (threadIdx.x == 0) { dparams[0] += dt; dparams[2] += 1.0; }
}

// ---------------------------------------------------------------------------------
// control flow: a WHILE loop either as a graph conditional node (during capture) or a
// host loop that reads the flag after each body.
// ---------------------------------------------------------------------------------
struct Flow {
    stdg_ctx* c;
    Workspace* ws;
    bool graph;
    long* kernels;      // kernels of each recorded body
    cudaError_t err = cudaSuccess;

    template <class Init, class Rec>
    void loop(Body id, const int* d_flag, Init init, Rec body) {
        if (err != cudaSuccess) return;
        if (!graph) {
            init(cudaGraphConditionalHandle(0), 0);
            for (long guard = 0; guard < 100000000L; ++guard) {
                int f = 0;
                err = cudaMemcpyAsync(&f, d_flag, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
                if (err == cudaSuccess) err = cudaStreamSynchronize(c->stream);
                if (err != cudaSuccess || !f) break;
                run_body(id, body, cudaGraphConditionalHandle(0), 0);
            }
            return;
        }
        cudaStream_t s = c->stream;
        cudaStreamCaptureStatus st;
        cudaGraph_t g;
        const cudaGraphNode_t* deps = nullptr;
        size_t nd = 0;
        if ((err = cudaStreamGetCaptureInfo(s, &st, nullptr, &g, &deps, nullptr, &nd)) != cudaSuccess) return;
        cudaGraphConditionalHandle h;
        if ((err = cudaGraphConditionalHandleCreate(&h, g, 0, 0)) != cudaSuccess) return;
        init(h, 1);
        if ((err = cudaStreamGetCaptureInfo(s, &st, nullptr, &g, &deps, nullptr, &nd)) != cudaSuccess) return;
        cudaGraphNodeParams p = {cudaGraphNodeTypeConditional};
        p.conditional.handle = h;
        p.conditional.type = cudaGraphCondTypeWhile;
        p.conditional.size = 1;
        cudaGraphNode_t node;
        if ((err = cudaGraphAddNode(&node, g, deps, nullptr, nd, &p)) != cudaSuccess) return;
        cudaGraph_t body_g = p.conditional.phGraph_out[0];
        cudaStream_t s2 = ws->side[ws->depth++];
        err = cudaStreamBeginCaptureToGraph(s2, body_g, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
        if (err == cudaSuccess) {
            c->stream = s2;
            run_body(id, body, h, 1);
            c->stream = s;
            cudaGraph_t tmp;
            cudaError_t e2 = cudaStreamEndCapture(s2, &tmp);
            if (err == cudaSuccess) err = e2;
        }
        ws->depth--;
        if (err == cudaSuccess) err = cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
    }
    void check(cudaError_t e) { if (err == cudaSuccess && e != cudaSuccess) err = e; }

    // one loop body in its own launch-count scope (the device counts its executions)
    template <class Rec>
    void run_body(Body id, Rec& body, cudaGraphConditionalHandle h, int use) {
        c->scopes.push_back(0);
        body(h, use);
        kernels[id] = c->scopes.back();
        c->scopes.pop_back();
    }
};


// ---- (P)CG on vectors of type R; apply(x, y): y = A x; prec(r, z): z = P^{-1} r or null --------
template <typename R, class Apply, class Prec>
static void solve_cg(Flow& F, double dt, Apply apply, Prec prec, bool use_prec, const R* b, R* x, R* r, R* p, R* pb, R* q, R* z,
                     double rel_tol, int max_iters, double bnorm_given, int gate_ir) {
    stdg_ctx* c = F.c;
    Workspace* ws = F.ws;
    const int64_t n = ws->n, nv = ws->nvec;
    const int ns = ws->ns, G = (int)ws->G;
    const dim3 grid = ws->grid();
    R* zz = use_prec ? z : r;
    const bool fused = use_prec && cg_fused_applies(c, ns, sizeof(R) == 4);   // two kernels an iteration
    F.loop(kBodyInner, &ws->sc->flag_inner,
           [&](cudaGraphConditionalHandle h, int use) {
               F.check(apply(x, q));
               cg_res_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, b, q, r, ws->partials); note_launch(c);
               if (use_prec) F.check(prec(r, zz));
               dot_partial_kernel<R, R><<<grid, kRedThreads, 0, c->stream>>>(nv, r, zz, ws->partials, 2); note_launch(c);
               cg_init_final_kernel<<<1, ws->fin_threads(), 0, c->stream>>>(ws->sc, ws->ss, ws->partials, ns, G, rel_tol, max_iters,
                                                                      bnorm_given, gate_ir, h, use); note_launch(c);
               copy_kernel<R><<<ws->red_blocks, kRedThreads, 0, c->stream>>>(n, zz, p); note_launch(c);
           },
           [&](cudaGraphConditionalHandle h, int use) {
               if (fused) {
                   F.check(launch_cg_fused(c, dt, x, r, zz, p, pb, q, ws->sc, ws->ss, ws->partials, ws->done, h, use));
                   return;
               }
               F.check(apply(p, q));
               cg_dot_alpha_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, p, q, ws->partials, ws->ss, ws->done); note_launch(c);
               cg_update_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, ws->ss, x, r, p, q, ws->partials); note_launch(c);
               if (use_prec) F.check(prec(r, zz));
               cg_dot_beta_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, r, zz, ws->partials, ws->sc, ws->ss, ws->done, h,
                                                                          use); note_launch(c);
               cg_p_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, ws->ss, zz, p); note_launch(c);
               F.check(cudaGetLastError());
           });
}

// ---- GMRES(m) on vectors of type R -----------------------------------------------------
// apply_prec(z, V, j, ld, w): w = A z for z = prec(V_j)
template <typename R, class Apply, class ApplyIdx, class ApplyPrec, class Prec>
static void solve_gmres(Flow& F, Apply apply, ApplyIdx apply_idx, ApplyPrec apply_prec, Prec prec, bool use_prec, const R* b,
                        R* x, R* V, R* w,
                        R* zbuf, R* tbuf, double rel_tol, int max_iters, double bnorm_given, int gate_ir) {
    stdg_ctx* c = F.c;
    Workspace* ws = F.ws;
    const int64_t n = ws->n, nv = ws->nvec, ldv = ws->ldv;
    const int m = ws->m;
    const int ns = ws->ns, G = (int)ws->G;
    const dim3 grid = ws->grid();
    DevScalars* sc = ws->sc;
    ShotScalars* ss = ws->ss;
    double* part = ws->partials;
    const dim3 dot_grid = ws->dot_grid();
    unsigned* done = ws->done;
    F.loop(kBodyCycle, &sc->flag_outer,
           [&](cudaGraphConditionalHandle h, int use) {
               if (bnorm_given < 0) {
                   dot_partial_kernel<R, R><<<grid, kRedThreads, 0, c->stream>>>(nv, b, b, part, 0); note_launch(c);
               }
               gm_init_kernel<<<1, ws->fin_threads(), 0, c->stream>>>(sc, ss, part, ns, G, rel_tol, max_iters, m, bnorm_given,
                                                                      gate_ir, h, use); note_launch(c);
           },
           [&](cudaGraphConditionalHandle h_outer, int use_outer) {
               // restart cycle: true residual, then Arnoldi
               F.check(apply(x, w));
               F.loop(kBodyInner, &sc->flag_inner,
                      [&](cudaGraphConditionalHandle h, int use) {
                          gm_res_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, b, w, V, part, 1, sc, ss, done, h, use);
                          note_launch(c);
                          gm_scale0_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, sc, ss, V); note_launch(c);
                      },
                      [&](cudaGraphConditionalHandle h, int use) {
                          if (use_prec) {   // right preconditioning: w = A P^{-1} v_j
                              F.check(prec(V, zbuf, &sc->j, ldv));
                              F.check(apply_prec(zbuf, V, &sc->j, ldv, w));
                          } else {
                              F.check(apply_idx(V, &sc->j, w));
                          }
                          // classical Gram-Schmidt: dots and ||w||^2; a second pass (with the first
                          // subtraction fused in) only for the shots that need it; subtraction, norm,
                          // Givens rotations and loop control
                          gm_mdot_kernel<R><<<dot_grid, kRedThreads, 0, c->stream>>>(nv, ldv, sc, ss, V, w, part, done);
                          note_launch(c);
                          gm_orth_fused_kernel<R><<<dot_grid, kRedThreads, 0, c->stream>>>(nv, ldv, sc, ss, V, w, part, done);
                          note_launch(c);
                          gm_maxpy_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, ldv, sc, ss, V, w, part, done, h, use);
                          note_launch(c);
                          gm_next_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, ldv, sc, ss, w, V); note_launch(c);
                          F.check(cudaGetLastError());
                      });
               if (use_prec) {   // x += P^{-1} (V y)
                   gm_combine_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, ldv, ss, V, tbuf, 0); note_launch(c);
                   F.check(prec(tbuf, zbuf, nullptr, 0));
                   axpy_kernel<R><<<ws->red_blocks, kRedThreads, 0, c->stream>>>(n, x, zbuf); note_launch(c);
               } else {
                   gm_combine_kernel<R><<<grid, kRedThreads, 0, c->stream>>>(nv, ldv, ss, V, x, 1); note_launch(c);
               }
               gm_cycle_end_kernel<<<1, ws->fin_threads(), 0, c->stream>>>(sc, ss, ns, h_outer, use_outer); note_launch(c);
               F.check(cudaGetLastError());
           });
}

// ---- all shots, one slab -----------------------------------------------------------------
static void record_solve(Flow& F, double dt, double* b, double* x) {
    stdg_ctx* c = F.c;
    Workspace* ws = F.ws;
    const int64_t nv = ws->nvec;
    const int ns = ws->ns, G = (int)ws->G;
    const dim3 grid = ws->grid();
    // CG for the SPD Crank-Nicolson system unless the preconditioner is the (non-symmetric) stencil one
    const bool cn = c->opt.scheme == STDG_SCHEME_CN && c->opt.preconditioner != 2;
    const bool pre = c->opt.preconditioner != 0;
    const bool p2 = c->opt.preconditioner == 2;
    const int64_t ldv = ws->ldv;
    auto A64 = [&](const double* xx, double* yy) { return launch_apply(c, dt, xx, yy, 1.0, nullptr, 0, ns); };
    auto A64i = [&](const double* V, const int* idx, double* yy) { return launch_apply(c, dt, V, yy, 1.0, idx, ldv, ns); };
    auto A32 = [&](const float* xx, float* yy) { return launch_apply32(c, dt, xx, yy, 1.0, nullptr, 0, ns); };
    auto A32i = [&](const float* V, const int* idx, float* yy) { return launch_apply32(c, dt, V, yy, 1.0, idx, ldv, ns); };
    auto AP64 = [&](const double* z, const double* V, const int* idx, int64_t ld, double* w) {
        return p2 ? launch_apply(c, dt, z, w, 1.0, nullptr, 0, ns) : launch_apply_pre1(c, dt, z, V, idx, ld, w, ns);
    };
    auto AP32 = [&](const float* z, const float* V, const int* idx, int64_t ld, float* w) {
        return p2 ? launch_apply32(c, dt, z, w, 1.0, nullptr, 0, ns) : launch_apply_pre1_32(c, dt, z, V, idx, ld, w, ns);
    };
    auto P64 = [&](const double* r, double* z, const int* idx, int64_t ld) {
        return p2 ? launch_pre2_apply(c, r, z, idx, ld, ns) : launch_pre1_apply(c, r, z, idx, ld, ns);
    };
    auto P32 = [&](const float* r, float* z, const int* idx, int64_t ld) {
        return p2 ? launch_pre2_apply32(c, r, z, idx, ld, ns) : launch_pre1_apply32(c, r, z, idx, ld, ns);
    };
    auto P64c = [&](const double* r, double* z) { return launch_pre1_apply(c, r, z, nullptr, 0, ns); };
    auto P32c = [&](const float* r, float* z) { return launch_pre1_apply32(c, r, z, nullptr, 0, ns); };
    const double tol = c->opt.rel_tol;
    const int maxit = c->opt.max_iters;
    if (c->opt.precision == STDG_FP64) {
        if (cn) solve_cg<double>(F, dt, A64, P64c, pre, b, x, ws->r, ws->p, ws->pb, ws->q, ws->z, tol, maxit, -1.0, 0);
        else solve_gmres<double>(F, A64, A64i, AP64, P64, pre, b, x, ws->V, ws->w, ws->z, ws->t, tol, maxit, -1.0, 0);
        zero_if_kernel<<<grid, kRedThreads, 0, c->stream>>>(nv, x, ws->ss, 0); note_launch(c);
        solve_stats_kernel<<<1, ws->fin_threads(), 0, c->stream>>>(ws->sc, ws->ss, ns, cn ? 1 : 0); note_launch(c);
        return;
    }
    // mixed: FP64 refinement, FP32 inner solve with zero initial guess and unit RHS per shot
    F.loop(kBodyIr, &ws->sc->ir_flag,
           [&](cudaGraphConditionalHandle h, int use) {
               dot_partial_kernel<double, double><<<grid, kRedThreads, 0, c->stream>>>(nv, b, b, ws->partials, 0); note_launch(c);
               ir_init_kernel<<<1, ws->fin_threads(), 0, c->stream>>>(ws->sc, ws->ss, ws->partials, ns, G, tol, 64, h, use); note_launch(c);
           },
           [&](cudaGraphConditionalHandle h, int use) {
               F.check(A64(x, ws->w));
               gm_res_kernel<double><<<grid, kRedThreads, 0, c->stream>>>(nv, b, ws->w, ws->r, ws->partials, 0, ws->sc, ws->ss,
                                                                          ws->done, 0, 0); note_launch(c);
               ir_check_kernel<<<1, ws->fin_threads(), 0, c->stream>>>(ws->sc, ws->ss, ws->partials, ns, G, maxit); note_launch(c);
               ir_convert_kernel<<<grid, kRedThreads, 0, c->stream>>>(nv, ws->sc, ws->ss, ws->r, ws->b32, ws->x32); note_launch(c);
               if (cn)
                   solve_cg<float>(F, dt, A32, P32c, pre, ws->b32, ws->x32, ws->r32, ws->p32, ws->pb32, ws->q32, ws->z32, c->opt.inner_tol,
                                   maxit, 1.0, 1);
               else
                   solve_gmres<float>(F, A32, A32i, AP32, P32, pre, ws->b32, ws->x32, ws->V32, ws->w32, ws->z32, ws->t32,
                                      c->opt.inner_tol, maxit, 1.0, 1);
               ir_update_kernel<<<grid, kRedThreads, 0, c->stream>>>(nv, ws->sc, ws->ss, ws->x32, x); note_launch(c);
               ir_end_kernel<<<1, 32, 0, c->stream>>>(ws->sc, h, use); note_launch(c);
               F.check(cudaGetLastError());
           });
    zero_if_kernel<<<grid, kRedThreads, 0, c->stream>>>(nv, x, ws->ss, 1); note_launch(c);
    solve_stats_kernel<<<1, ws->fin_threads(), 0, c->stream>>>(ws->sc, ws->ss, ns, 2); note_launch(c);
}

// One slab for every shot: per-shot right-hand sides and initial guesses, ONE stacked
// (block-diagonal) solve whose operator and preconditioner kernels load each face's and
// element's blocks once for all shots, then per-shot stress, traces and receivers.
static void record_step(Flow& F, double dt) {
    stdg_ctx* c = F.c;
    Workspace* ws = F.ws;
    c->scopes.assign(1, 0);
    step_begin_kernel<<<1, 32, 0, c->stream>>>(ws->dparams, dt); note_launch(c);
    for (int shot = 0; shot < c->n_shots && F.err == cudaSuccess; ++shot) {
        F.check(launch_rhs(c, dt, ws->dparams, shot, c->d_b + (int64_t)shot * c->nvel));
        F.check(launch_initial_guess(c, shot, c->d_x + (int64_t)shot * c->nvel));
    }
    record_solve(F, dt, c->d_b, c->d_x);
    for (int shot = 0; shot < c->n_shots && F.err == cudaSuccess; ++shot) {
        F.check(launch_stress_update(c, dt, shot, c->d_x + (int64_t)shot * c->nvel));
        F.check(launch_traces(c, shot, c->d_x + (int64_t)shot * c->nvel));
        F.check(launch_receivers(c, ws->dparams, shot));
    }
    step_end_kernel<<<1, 32, 0, c->stream>>>(ws->dparams, dt); note_launch(c);
    F.kernels[kBodyStraight] = c->scopes.back();
    c->scopes.clear();
    F.check(cudaGetLastError());
}

int solver_setup(stdg_ctx* c) {
    solver_free(c);
    Workspace* ws = new Workspace();
    c->ws = ws;
    ws->m = std::max(2, std::min(c->opt.gmres_restart > 0 ? c->opt.gmres_restart : 30, kMaxRestart));
    ws->ns = c->n_shots;
    ws->nvec = c->nvel;
    ws->n = c->nvel * (int64_t)c->n_shots;
    // Grids by vector length: one 16-byte item a thread, up to the blocks that keep every SM busy.
    // (A fixed grid made every launch on a 2,352-value vector start 1,216 blocks and every reduction
    // sum as many parts: 49 us per CG iteration.)
    const int64_t item = c->opt.precision == STDG_FP64 ? 2 : 4;
    auto blocks = [&](int64_t values, int per_sm, int shots) {
        const int64_t want = (values + item * kRedThreads - 1) / (item * kRedThreads);
        return (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)per_sm * c->n_sm / shots));
    };
    const int64_t n = ws->n;
    ws->red_blocks = blocks(n, 8, 1);
    ws->G = blocks(ws->nvec, 4, ws->ns);
    ws->Gd = blocks(ws->nvec, 2, ws->ns);
    const bool cn = c->opt.scheme == STDG_SCHEME_CN && c->opt.preconditioner != 2;   // CG workspace
    const bool mixed = c->opt.precision != STDG_FP64;
    const bool pre = c->opt.preconditioner != 0;
    int rc;
#define ALLOC(ptr, bytes) do { if ((rc = dev_alloc(c, (void**)&(ptr), (bytes))) != STDG_OK) return rc; \
                               ws->owned.push_back((void*)(ptr)); } while (0)
    ALLOC(ws->sc, sizeof(DevScalars));
    ALLOC(ws->ss, sizeof(ShotScalars) * ws->ns);
    ALLOC(ws->partials, sizeof(double) * (kMaxRestart + 2) * std::max(ws->G * ws->ns, (unsigned)(4 * c->n_sm)));
    ALLOC(ws->done, sizeof(unsigned) * (ws->ns + 1));
    ALLOC(ws->dparams, sizeof(double) * 4);
    ALLOC(c->d_b, sizeof(double) * n);
    ALLOC(c->d_x, sizeof(double) * n);
    ALLOC(ws->w, sizeof(double) * n);
    ALLOC(ws->r, sizeof(double) * n);
    ws->ldv = (n + 63) / 64 * 64;   // 16-byte aligned basis columns for vector loads
    if (cn && !mixed && pre) ALLOC(ws->pb, sizeof(double) * n);
    if (cn && mixed && pre) ALLOC(ws->pb32, sizeof(float) * n);
    if (cn && !mixed) { ALLOC(ws->p, sizeof(double) * n); ALLOC(ws->q, sizeof(double) * n); }
    if (!cn && !mixed) ALLOC(ws->V, sizeof(double) * ws->ldv * (ws->m + 1));
    if (pre && !mixed) { ALLOC(ws->z, sizeof(double) * n); if (!cn) ALLOC(ws->t, sizeof(double) * n); }
    if (mixed) {
        ALLOC(ws->b32, sizeof(float) * n);
        ALLOC(ws->x32, sizeof(float) * n);
        if (cn) { ALLOC(ws->r32, sizeof(float) * n); ALLOC(ws->p32, sizeof(float) * n); ALLOC(ws->q32, sizeof(float) * n); }
        else { ALLOC(ws->V32, sizeof(float) * ws->ldv * (ws->m + 1)); ALLOC(ws->w32, sizeof(float) * n); }
        if (pre) { ALLOC(ws->z32, sizeof(float) * n); if (!cn) ALLOC(ws->t32, sizeof(float) * n); }
    }
#undef ALLOC
    cudaMemsetAsync(ws->sc, 0, sizeof(DevScalars), c->stream);
    cudaMemsetAsync(ws->ss, 0, sizeof(ShotScalars) * ws->ns, c->stream);
    cudaMemsetAsync(ws->done, 0, sizeof(unsigned) * (ws->ns + 1), c->stream);
    cudaMemsetAsync(ws->dparams, 0, sizeof(double) * 4, c->stream);
    for (auto& s : ws->side) cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    return STDG_OK;
}

void solver_free(stdg_ctx* c) {
    Workspace* ws = W(c);
    if (!ws) return;
    for (int k = 0; k < 2; ++k) {
        if (ws->exec[k]) cudaGraphExecDestroy(ws->exec[k]);
        if (ws->graph[k]) cudaGraphDestroy(ws->graph[k]);
    }
    for (auto& s : ws->side) if (s) cudaStreamDestroy(s);
    cudaStreamSynchronize(c->stream);
    for (void* p : ws->owned) dev_release(c, p);
    c->d_b = c->d_x = nullptr;
    delete ws;
    c->ws = nullptr;
}

void solver_invalidate_graph(stdg_ctx* c) {
    Workspace* ws = W(c);
    if (!ws) return;
    for (int k = 0; k < 2; ++k) {
        if (ws->exec[k]) cudaGraphExecDestroy(ws->exec[k]);
        if (ws->graph[k]) cudaGraphDestroy(ws->graph[k]);
        ws->exec[k] = nullptr;
        ws->graph[k] = nullptr;
        ws->graph_dt[k] = -1.0;
    }
}

double* solver_dparams(stdg_ctx* c) { return W(c) ? W(c)->dparams : nullptr; }

// the solve alone: A x = b on the stacked c->d_b / c->d_x (x holds the initial guess)
static void record_solve_only(Flow& F, double dt) {
    stdg_ctx* c = F.c;
    c->scopes.assign(1, 0);
    record_solve(F, dt, c->d_b, c->d_x);
    F.kernels[kBodyStraight] = c->scopes.back();
    c->scopes.clear();
    F.check(cudaGetLastError());
}

// Runs `n` repetitions of a recorded body (kind 0: a whole step, 1: the solve alone), as one
// cached CUDA graph per kind and dt, or from the host loop; then reads the statistics.
static int run_body_n(stdg_ctx* c, double dt, int n, int kind, stdg_stats* st) {
    Workspace* ws = W(c);
    STDG_CUDA(c, cudaMemsetAsync(&ws->sc->st_total, 0, sizeof(int) * 5, c->stream));
    STDG_CUDA(c, cudaMemsetAsync(&ws->sc->st_final_rel, 0, sizeof(double) * 2, c->stream));
    STDG_CUDA(c, cudaMemsetAsync(ws->sc->runs, 0, sizeof(ws->sc->runs), c->stream));
    auto record = [&](Flow& F) {
        if (kind == 0) record_step(F, dt);
        else record_solve_only(F, dt);
    };
    if (c->opt.use_graph) {
        if (!ws->exec[kind] || ws->graph_dt[kind] != dt) {
            if (ws->exec[kind]) cudaGraphExecDestroy(ws->exec[kind]);
            if (ws->graph[kind]) cudaGraphDestroy(ws->graph[kind]);
            ws->exec[kind] = nullptr;
            ws->graph[kind] = nullptr;
            cudaStream_t s0 = c->stream;
            STDG_CUDA(c, cudaStreamBeginCapture(s0, cudaStreamCaptureModeRelaxed));
            Flow F{c, ws, true, ws->body_kernels[kind]};
            record(F);
            c->stream = s0;
            cudaGraph_t g = nullptr;
            cudaError_t e = cudaStreamEndCapture(s0, &g);
            if (F.err != cudaSuccess || e != cudaSuccess) {
                if (g) cudaGraphDestroy(g);
                c->err = std::string("graph capture failed: ") + cudaGetErrorString(F.err != cudaSuccess ? F.err : e);
                cudaGetLastError();
                return STDG_ECUDA;
            }
            ws->graph[kind] = g;
            STDG_CUDA(c, cudaGraphInstantiate(&ws->exec[kind], g, 0));
            ws->graph_dt[kind] = dt;
        }
        for (int s = 0; s < n; ++s) STDG_CUDA(c, cudaGraphLaunch(ws->exec[kind], c->stream));
    } else {
        for (int s = 0; s < n; ++s) {
            Flow F{c, ws, false, ws->body_kernels[kind]};
            record(F);
            if (F.err != cudaSuccess) STDG_CUDA(c, F.err);
        }
    }
    STDG_CUDA(c, cudaStreamSynchronize(c->stream));
    STDG_CUDA(c, cudaGetLastError());
    DevScalars h;
    STDG_CUDA(c, cudaMemcpy(&h, ws->sc, sizeof(DevScalars), cudaMemcpyDeviceToHost));
    if (st) {
        st->iters_total = (int)h.st_iters_sum;
        st->iters_max = h.st_max;
        st->refinements = h.st_refine;
        st->final_rel_res = h.st_final_rel;
        st->status = h.st_nonfinite ? STDG_ENONFINITE : h.st_notconv ? STDG_ENOTCONV : STDG_OK;
    }
    c->last_launches = 0;
    for (int i = 0; i < kBodies; ++i) c->last_launches += (int64_t)h.runs[i] * ws->body_kernels[kind][i];
    {
        const int rc = take_device_error(c);
        if (rc != STDG_OK) return rc;
    }
    if (h.st_nonfinite) STDG_FAIL(c, STDG_ENONFINITE, "a residual or right-hand-side norm is NaN or Inf (input overflow?)");
    if (h.st_notconv) STDG_FAIL(c, STDG_ENOTCONV, "Krylov solve reached max_iters");
    return STDG_OK;
}

int solver_step(stdg_ctx* c, double dt, int n_steps, stdg_stats* st) {
    Workspace* ws = W(c);
    if (!ws) STDG_FAIL(c, STDG_ESTATE, "solver not set up");
    {
        const int rc = precond_for_dt(c, dt);
        if (rc != STDG_OK) return rc;
    }
    const double t0 = c->t;
    STDG_CUDA(c, cudaMemcpyAsync(ws->dparams, &t0, sizeof(double), cudaMemcpyHostToDevice, c->stream));
    {
        double stepidx = (double)c->rec_steps;
        STDG_CUDA(c, cudaMemcpyAsync(ws->dparams + 2, &stepidx, sizeof(double), cudaMemcpyHostToDevice, c->stream));
    }
    c->wait_gave_up = false;
    const int rc = run_body_n(c, dt, n_steps, 0, st);
    // the state advanced when the solve did not converge and when a bounded wait gave up
    // (then with invalid values); a CUDA error proper leaves time and records where they were
    if (rc == STDG_OK || rc == STDG_ENOTCONV || rc == STDG_ENONFINITE || c->wait_gave_up) {
        c->t = t0 + n_steps * dt;
        c->rec_steps += n_steps;
    }
    return rc;
}

int solver_solve(stdg_ctx* c, double dt, stdg_stats* st) {
    Workspace* ws = W(c);
    if (!ws) STDG_FAIL(c, STDG_ESTATE, "solver not set up");
    const int rc = precond_for_dt(c, dt);
    if (rc != STDG_OK) return rc;
    return run_body_n(c, dt, 1, 1, st);
}

}  // namespace stdg
