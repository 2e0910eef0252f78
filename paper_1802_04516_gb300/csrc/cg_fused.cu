// Conjugate gradients of the Crank-Nicolson system with block-Jacobi preconditioning, one shot, two
// kernels per iteration:
//   cg_apply    p = z + beta p' (formed where it is read, for the element and its neighbours), q = A p from
//               the assembled couplings with the mass term, p . q; the last block forms alpha
//   cg_update   x += alpha p, r -= alpha q, z = P_1 r, r . r and r . z; the last block forms beta, tests the
//               convergence and advances the loop
// Both work element by element, so the vector updates need no passes of their own.  The systems that
// the scheme solves this way are often small (2,352 unknowns in the plane-wave problem), where an
// iteration is a chain of launches and of dependent memory accesses: six kernels took 29 us there, two
// take 23 us.  p' is read while p is written, so the two alternate between two buffers by iteration.
// N_gamma = 1 throughout, so a row of an element is one value.
//
// Systems of up to 512 unknowns in whole elements per SM (8,192 in all; 8,160 or 7,680 where d N_phi does not
// divide 512) run in one cluster of 16 SMs for all their iterations: a thread per
// unknown keeps x, r, z, p and q in registers, only p crosses SMs (through L2), and the two reductions
// of an iteration meet in distributed shared memory behind cluster barriers (three an iteration), which cost less than the
// end of a kernel (9 us per iteration in the plane-wave problem).  Above that size 16 SMs are too few
// (FP64 runs at two lanes an SM).
#include <algorithm>
#include <cstdint>

#include <cooperative_groups.h>

#include "compensated.h"
#include "krylov.h"
#include "stdg_internal.h"

namespace stdg {

template <typename R> struct CgPair;
template <> struct CgPair<float> { using T = float2; };
template <> struct CgPair<double> { using T = double2; };

template <typename R, int DIM, int NP>
__global__ void __launch_bounds__(160) cg_apply_kernel(int64_t n_elem, int EB, const int2* __restrict__ adj,
                                                       const R* __restrict__ Ke, const R* __restrict__ Kf,
                                                       const R* __restrict__ rhoJ, const RefTables* __restrict__ rtp, double scale,
                                                       const R* __restrict__ z, const R* p0, const R* p1, R* pw0, R* pw1,
                                                       R* __restrict__ q, const DevScalars* __restrict__ sc, ShotScalars* ss,
                                                       double* part, unsigned* done) {
    constexpr int N = DIM * NP, FACES = DIM + 1, SLOTS = FACES + 1;
    constexpr bool BOTH = sizeof(R) == 4;                     // the FP32 faces' blocks are kept in both orientations
    constexpr int CH = N % 10 == 0 ? 10 : 6;                  // columns loaded together
    using P = typename CgPair<R>::T;
    extern __shared__ __align__(16) unsigned char smraw[];
    R* sx = reinterpret_cast<R*>(smraw);                      // [slot][element][row]
    __shared__ R sM[NP * NP];
    const bool odd = sc->iters & 1;
    const double beta = ss->beta, rz = ss->pq;
    const R* po = odd ? p1 : p0;
    R* pn = odd ? pw0 : pw1;
    const R S = (R)(scale * rtp->S[0]), T = (R)rtp->T[0];   // rounded once
    for (int t = threadIdx.x; t < NP * NP; t += blockDim.x) sM[t] = (R)rtp->Mref[t];
    const int le = threadIdx.x / N, row = threadIdx.x % N;
    Acc<R> pq;
    for (int64_t e0 = (int64_t)blockIdx.x * EB; e0 < n_elem; e0 += (int64_t)gridDim.x * EB) {
        const bool act = le < min((int64_t)EB, n_elem - e0);
        const int64_t e = e0 + le;
        int2 nb[FACES];
#pragma unroll
        for (int i = 0; i < FACES; ++i) nb[i] = act ? adj[e * FACES + i] : make_int2(-1, 0);
        __syncthreads();                                      // the values of the group before have been read
        R own = (R)0;
        if (act) {
            R zv[SLOTS], pv[SLOTS];
#pragma unroll
            for (int sl = 0; sl < SLOTS; ++sl) {
                const int64_t en = sl == 0 ? e : nb[sl ? sl - 1 : 0].x;
                zv[sl] = en >= 0 ? z[en * N + row] : (R)0;
                pv[sl] = en >= 0 ? po[en * N + row] : (R)0;
            }
#pragma unroll
            for (int sl = 0; sl < SLOTS; ++sl) {
                const R v = (R)((double)zv[sl] + beta * (double)pv[sl]);
                sx[(sl * EB + le) * N + row] = v;
                if (sl == 0) own = v;
            }
            pn[e * N + row] = own;
        }
        __syncthreads();
        if (!act) continue;
        RowSum<R> acc;
#pragma unroll
        for (int sl = 0; sl < SLOTS; ++sl) {
            const R* kp = Ke + e * (N * N);
            bool by_rows = false;
            if (sl) {
                const int2 a = nb[sl ? sl - 1 : 0];
                if (a.x < 0) continue;
                by_rows = !BOTH && !(a.y & 1);
                kp = Kf + (int64_t)(BOTH ? a.y : a.y >> 1) * (N * N);
            }
            const R* xp = sx + (sl * EB + le) * N;
            for (int jc = 0; jc < N; jc += CH) {
                R kv[CH];
                if (by_rows) {
#pragma unroll
                    for (int j = 0; j < CH; j += 2) {
                        const P t = __ldg(reinterpret_cast<const P*>(kp + row * N + jc + j));
                        kv[j] = t.x;
                        kv[j + 1] = t.y;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < CH; ++j) kv[j] = __ldg(kp + (jc + j) * N + row);
                }
                acc.columns(kv, [&](int j) { return xp[jc + j]; });
            }
            acc.end_slot();
        }
        const int k = row / NP, nn = row % NP;
        R u = (R)0;
#pragma unroll
        for (int j = 0; j < NP; ++j) u = fma(sM[nn * NP + j], sx[le * N + k * NP + j], u);
        const R o = fma(T, u * rhoJ[e], acc.scaled(S));
        q[e * N + row] = o;
        pq.add(own, o);
    }
    const double mine = block_sum1(pq);
    if (threadIdx.x == 0) part[blockIdx.x] = mine;
    if (!last_block(done, gridDim.x)) return;
    double v = 0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) v += __ldcg(part + i);
    v = block_sum(v);
    if (threadIdx.x == 0) ss->alpha = v != 0.0 ? rz / v : 0.0;
}

template <typename R, int DIM, int NP>
__global__ void __launch_bounds__(160) cg_update_kernel_fused(int64_t n_elem, int EB, const R* __restrict__ V,
                                                              const R* __restrict__ B, R* __restrict__ x, R* __restrict__ r,
                                                              R* __restrict__ z, const R* __restrict__ p0, const R* __restrict__ p1,
                                                              const R* __restrict__ q, DevScalars* sc, ShotScalars* ss,
                                                              double* part, unsigned* done, cudaGraphConditionalHandle h,
                                                              int use_h) {
    constexpr int N = DIM * NP;
    using P = typename CgPair<R>::T;
    extern __shared__ __align__(16) unsigned char smraw[];
    R* sr = reinterpret_cast<R*>(smraw);                      // [element][row]: r, then w = B V^T r
    R* sw = sr + EB * N;
    const int iters = sc->iters, max_iters = sc->max_iters;
    const unsigned runs = sc->runs[kBodyInner];
    const double a = ss->alpha, rz_old = ss->pq, tol = ss->tol_abs;
    const R* p = iters & 1 ? p0 : p1;
    const int le = threadIdx.x / N, row = threadIdx.x % N;
    double rr = 0;
    Acc<R> rz;
    for (int64_t e0 = (int64_t)blockIdx.x * EB; e0 < n_elem; e0 += (int64_t)gridDim.x * EB) {
        const bool act = le < min((int64_t)EB, n_elem - e0);
        const int64_t e = e0 + le, at = e * N + row;
        const R* Ve = V + (act ? e : e0) * (N * N);
        __syncthreads();
        R ri = (R)0, b = (R)0;
        if (act) {
            b = B[at];
            x[at] = (R)((double)x[at] + a * (double)p[at]);
            ri = (R)((double)r[at] - a * (double)q[at]);
            r[at] = ri;
            rr += (double)ri * (double)ri;
            sr[le * N + row] = ri;
        }
        __syncthreads();
        if (act) {
            R u = (R)0;
#pragma unroll 10
            for (int j = 0; j < N; ++j) u = fma(__ldg(Ve + j * N + row), sr[le * N + j], u);
            sw[le * N + row] = b * u;
        }
        __syncthreads();
        if (act) {
            R o = (R)0;
#pragma unroll 5
            for (int j = 0; j < N; j += 2) {
                const P v = __ldg(reinterpret_cast<const P*>(Ve + row * N + j));
                o = fma(v.x, sw[le * N + j], o);
                o = fma(v.y, sw[le * N + j + 1], o);
            }
            z[at] = o;
            rz.add(ri, o);
        }
    }
    const double srr = block_sum(rr), srz = block_sum1(rz);
    const int G = gridDim.x;
    if (threadIdx.x == 0) {
        part[blockIdx.x] = srr;
        part[G + blockIdx.x] = srz;
    }
    if (!last_block(done, G)) return;
    double v = 0, w = 0;
    for (int i = threadIdx.x; i < G; i += blockDim.x) {
        v += __ldcg(part + i);
        w += __ldcg(part + G + i);
    }
    v = block_sum(v);
    w = block_sum(w);
    if (threadIdx.x != 0) return;
    const bool conv = sqrt(v) <= tol, active = !conv && isfinite(v);
    ss->beta = active && rz_old != 0.0 ? w / rz_old : 0.0;
    ss->pq = w;
    ss->rr = v;
    ss->converged = conv;
    ss->active = active;
    sc->iters = iters + 1;
    sc->runs[kBodyInner] = runs + 1;
    const int go = active && iters + 1 < max_iters;
    sc->flag_inner = go;
    set_cond(h, use_h, go);
}

// A thread's row of the element couplings and of V, in registers where they are few.
template <typename R, int DIM, int NP>
struct CgRow {
    static constexpr int N = DIM * NP, SLOTS = DIM + 2;
    static constexpr bool KEEP = N <= 6;
};

constexpr int kClusterSize = 16;

template <typename R, int DIM, int NP>
__global__ void __launch_bounds__(512, 1) cg_cluster_kernel(int64_t n_elem, int EPC, const int2* __restrict__ adj,
                                                            const R* __restrict__ Ke, const R* __restrict__ Kf,
                                                            const R* __restrict__ rhoJ, const RefTables* __restrict__ rtp, double scale,
                                                            const R* __restrict__ V, const R* __restrict__ B, R* x, R* r, R* z,
                                                            R* p, DevScalars* sc, ShotScalars* ss, cudaGraphConditionalHandle h,
                                                            int use_h) {
    namespace cg = cooperative_groups;
    using C = CgRow<R, DIM, NP>;
    constexpr int N = C::N, FACES = DIM + 1, SLOTS = C::SLOTS;
    constexpr bool BOTH = sizeof(R) == 4;
    constexpr int CH = N % 10 == 0 ? 10 : 6;
    using P = typename CgPair<R>::T;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ R sp[512], sr[512], sw[512], sM[NP * NP];
    __shared__ double part[3], bc[2];
    const int rank = blockIdx.x, CT = gridDim.x;
    for (int t = threadIdx.x; t < NP * NP; t += blockDim.x) sM[t] = (R)rtp->Mref[t];
    const R S = (R)(scale * rtp->S[0]), T = (R)rtp->T[0];   // rounded once
    const int le = threadIdx.x / N, row = threadIdx.x % N, k = row / NP, nn = row % NP;
    const int64_t e = (int64_t)rank * EPC + le, at = e * N + row;
    const bool act = le < EPC && e < n_elem;
    const int max_iters = sc->max_iters;
    const double tol = ss->tol_abs;
    double rz = ss->pq, beta = 0.0, rr = ss->rr;
    int2 nb[FACES];
#pragma unroll
    for (int i = 0; i < FACES; ++i) nb[i] = act ? adj[e * FACES + i] : make_int2(-1, 0);
    R xv = (R)0, rv = (R)0, zv = (R)0, pv = (R)0, rj = (R)0, bq = (R)0;
    if (act) {
        xv = x[at];
        rv = r[at];
        zv = z[at];
        rj = rhoJ[e];
        bq = B[at];
    }
    const R* Ve = V + (act ? e : 0) * (N * N);
    auto load_k = [&](int sl, int jc, R (&kv)[CH]) {   // columns jc.. of the thread's row of slot sl
        const R* kp = Ke + e * (N * N);
        bool by_rows = false;
        if (sl) {
            int2 a = nb[0];
#pragma unroll
            for (int i = 1; i < FACES; ++i)
                if (sl - 1 == i) a = nb[i];
            by_rows = !BOTH && !(a.y & 1);
            kp = Kf + (int64_t)(BOTH ? a.y : a.y >> 1) * (N * N);
        }
        if (by_rows) {
#pragma unroll
            for (int j = 0; j < CH; j += 2) {
                const P t = __ldg(reinterpret_cast<const P*>(kp + row * N + jc + j));
                kv[j] = t.x;
                kv[j + 1] = t.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < CH; ++j) kv[j] = __ldg(kp + (jc + j) * N + row);
        }
    };
    R kk[C::KEEP ? SLOTS : 1][CH], vc[C::KEEP ? N : 1], vr[C::KEEP ? N : 1];
    if constexpr (C::KEEP) {
        if (act) {
#pragma unroll
            for (int sl = 0; sl < SLOTS; ++sl)
                if (sl == 0 || nb[sl ? sl - 1 : 0].x >= 0) load_k(sl, 0, kk[sl]);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                vc[j] = Ve[j * N + row];
                vr[j] = Ve[row * N + j];
            }
        }
    }
    // sums of the blocks' parts in rank order, the same in every block
    auto gather = [&](int i) {
        double v = 0;
        if (threadIdx.x < 32) {
            if ((int)threadIdx.x < CT) v = *cl.map_shared_rank(&part[i], threadIdx.x);
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        }
        return v;   // valid in the first warp
    };
    int it = 0;
    bool go = true;
    while (go) {
        if (act) {
            pv = (R)((double)zv + beta * (double)pv);
            sp[threadIdx.x] = pv;
            p[at] = pv;
        }
        cl.sync();
        R q = (R)0;
        Acc<R> pq;
        if (act) {
            R pn[FACES][N <= 6 ? N : 1];
            if constexpr (N <= 6) {
#pragma unroll
                for (int i = 0; i < FACES; ++i)
#pragma unroll
                    for (int j = 0; j < N; ++j) pn[i][j] = nb[i].x >= 0 ? __ldcg(p + (int64_t)nb[i].x * N + j) : (R)0;
            }
            RowSum<R> acc;
#pragma unroll
            for (int sl = 0; sl < SLOTS; ++sl) {
                if (sl && nb[sl ? sl - 1 : 0].x < 0) continue;
#pragma unroll 1
                for (int jc = 0; jc < N; jc += CH) {
                    R kv[CH];
                    if constexpr (C::KEEP) {
#pragma unroll
                        for (int j = 0; j < CH; ++j) kv[j] = kk[sl][j];
                    } else {
                        load_k(sl, jc, kv);
                    }
                    acc.columns(kv, [&](int j) {
                        if (sl == 0) return sp[le * N + jc + j];
                        if constexpr (N <= 6) return pn[sl ? sl - 1 : 0][j];
                        else return __ldcg(p + (int64_t)nb[sl ? sl - 1 : 0].x * N + jc + j);
                    });
                }
                acc.end_slot();
            }
            R u = (R)0;
#pragma unroll
            for (int j = 0; j < NP; ++j) u = fma(sM[nn * NP + j], sp[le * N + k * NP + j], u);
            q = fma(T, u * rj, acc.scaled(S));
            pq.add(pv, q);
        }
        {
            const double v = block_sum1(pq);
            if (threadIdx.x == 0) part[0] = v;
        }
        cl.sync();
        {
            const double v = gather(0);
            if (threadIdx.x == 0) bc[0] = v != 0.0 ? rz / v : 0.0;
        }
        __syncthreads();
        const double alpha = bc[0];
        double rr1 = 0;
        if (act) {
            xv = (R)((double)xv + alpha * (double)pv);
            rv = (R)((double)rv - alpha * (double)q);
            rr1 = (double)rv * (double)rv;
            sr[threadIdx.x] = rv;
        }
        __syncthreads();
        if (act) {
            R u = (R)0;
#pragma unroll
            for (int j = 0; j < N; ++j) u = fma(C::KEEP ? vc[C::KEEP ? j : 0] : __ldg(Ve + j * N + row), sr[le * N + j], u);
            sw[threadIdx.x] = bq * u;
        }
        __syncthreads();
        Acc<R> rza;
        if (act) {
            R o = (R)0;
#pragma unroll
            for (int j = 0; j < N; ++j) o = fma(C::KEEP ? vr[C::KEEP ? j : 0] : __ldg(Ve + row * N + j), sw[le * N + j], o);
            zv = o;
            rza.add(rv, o);
        }
        {
            const double a = block_sum(rr1), b = block_sum1(rza);
            if (threadIdx.x == 0) { part[1] = a; part[2] = b; }
        }
        cl.sync();
        {
            const double a = gather(1), b = gather(2);
            if (threadIdx.x == 0) { bc[0] = a; bc[1] = b; }
        }
        __syncthreads();
        rr = bc[0];
        beta = rz != 0.0 ? bc[1] / rz : 0.0;
        rz = bc[1];
        ++it;
        go = !(sqrt(rr) <= tol) && isfinite(rr) && it < max_iters;   // alike in every thread of the cluster
    }
    if (act) {
        x[at] = xv;
        r[at] = rv;
    }
    if (rank == 0 && threadIdx.x == 0) {
        ss->beta = beta;
        ss->pq = rz;
        ss->rr = rr;
        ss->converged = sqrt(rr) <= tol;
        ss->active = 0;
        sc->iters = it;
        sc->runs[kBodyInner] += 1;
        sc->flag_inner = 0;
        set_cond(h, use_h, 0);
    }
    cl.sync();   // no block leaves while its parts may be read
}

// Elements per SM of the cluster kernel; 0 where the system is too large for it.
static int cluster_elements(const stdg_ctx* c) {
    const int N = c->dim * c->Nphi;
    const int64_t epc = (c->n_elem + kClusterSize - 1) / kClusterSize;
    return epc * N <= 512 ? (int)epc : 0;
}

bool cg_fused_applies(const stdg_ctx* c, int nshots, bool fp32) {
    return nshots == 1 && c->Ng == 1 && c->opt.scheme == STDG_SCHEME_CN && c->opt.preconditioner == 1 &&
           (fp32 ? c->d_Kf32 != nullptr : c->d_Kf != nullptr);
}

template <typename R, int DIM, int NP>
static cudaError_t go(stdg_ctx* c, double dt, const R* Ke, const R* Kf, const R* rhoJ, const R* V, const R* B, R* x, R* r, R* z,
                      R* p, R* pb, R* q, DevScalars* sc, ShotScalars* ss, double* part, unsigned* done,
                      cudaGraphConditionalHandle h, int use_h) {
    constexpr int N = DIM * NP;
    if (const int epc = cluster_elements(c)) {
        auto kern = cg_cluster_kernel<R, DIM, NP>;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kClusterSize;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kClusterSize);
        cfg.blockDim = dim3((epc * N + 31) / 32 * 32);
        cfg.stream = c->stream;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        // 16 blocks are more than the portable cluster size: a partition of the GPU, or one whose clusters hold
        // fewer free SMs, cannot schedule them, and the two kernels below serve every size
        int fit = 0;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) == cudaSuccess && fit > 0) {
            note_launch(c);
            return cudaLaunchKernelEx(&cfg, kern, c->n_elem, epc, (const int2*)c->d_adj, Ke, Kf, rhoJ, (const RefTables*)c->d_rt,
                                      0.25 * dt * dt, V, B, x, r, z, p, sc, ss, h, use_h);
        }
        cudaGetLastError();
    }
    // whole warps of rows, at most 160 threads; at least one block per SM on small meshes, and on large
    // ones at most four, so that the reductions stay short
    const int most = (int)std::max<int64_t>(1, std::min<int64_t>(160 / N, c->n_elem / c->n_sm));
    double best = 0.0;
    int EB = 1;
    for (int e = 1; e <= most; ++e) {
        const double eff = (double)(e * N) / ((e * N + 31) / 32 * 32);
        if (eff >= best) { best = eff; EB = e; }
    }
    const unsigned grid = (unsigned)std::min<int64_t>((c->n_elem + EB - 1) / EB, (int64_t)c->n_sm * 4);
    const int threads = (EB * N + 31) / 32 * 32;
    cg_apply_kernel<R, DIM, NP><<<grid, threads, sizeof(R) * (DIM + 2) * EB * N, c->stream>>>(
        c->n_elem, EB, c->d_adj, Ke, Kf, rhoJ, c->d_rt, 0.25 * dt * dt, z, p, pb, p, pb, q, sc, ss, part, done);
    note_launch(c);
    cg_update_kernel_fused<R, DIM, NP><<<grid, threads, sizeof(R) * 2 * EB * N, c->stream>>>(
        c->n_elem, EB, V, B, x, r, z, p, pb, q, sc, ss, part, done, h, use_h);
    note_launch(c);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t dispatch(stdg_ctx* c, double dt, const R* Ke, const R* Kf, const R* rhoJ, const R* V, const R* B, R* x, R* r,
                            R* z, R* p, R* pb, R* q, DevScalars* sc, ShotScalars* ss, double* part, unsigned* done,
                            cudaGraphConditionalHandle h, int use_h) {
#define STDG_CG(D_, N_) return go<R, D_, N_>(c, dt, Ke, Kf, rhoJ, V, B, x, r, z, p, pb, q, sc, ss, part, done, h, use_h)
    switch (c->dim * 100 + c->Nphi) {
        case 203: STDG_CG(2, 3);
        case 206: STDG_CG(2, 6);
        case 210: STDG_CG(2, 10);
        case 215: STDG_CG(2, 15);
        case 304: STDG_CG(3, 4);
        case 310: STDG_CG(3, 10);
        case 320: STDG_CG(3, 20);
        default: return cudaErrorInvalidValue;
    }
#undef STDG_CG
}

cudaError_t launch_cg_fused(stdg_ctx* c, double dt, double* x, double* r, double* z, double* p, double* pb, double* q,
                            DevScalars* sc, ShotScalars* ss, double* part, unsigned* done, cudaGraphConditionalHandle h, int use_h) {
    return dispatch<double>(c, dt, c->d_Ke, c->d_Kf, c->d_rhoJ, c->d_preV, c->d_preB, x, r, z, p, pb, q, sc, ss, part, done, h, use_h);
}
cudaError_t launch_cg_fused(stdg_ctx* c, double dt, float* x, float* r, float* z, float* p, float* pb, float* q, DevScalars* sc,
                            ShotScalars* ss, double* part, unsigned* done, cudaGraphConditionalHandle h, int use_h) {
    return dispatch<float>(c, dt, c->d_Ke32, c->d_Kf32, c->d_rhoJ32, c->d_preV32, c->d_preB32, x, r, z, p, pb, q, sc, ss, part, done,
                           h, use_h);
}

}  // namespace stdg
