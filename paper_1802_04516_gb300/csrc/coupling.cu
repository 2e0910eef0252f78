// The Schur velocity operator from assembled element couplings.
//
// The face term of Eq. velocity.sys couples element i with itself and its face neighbours through
//   (A v)_i = rho_i |J_i| (T (x) M_ref) v_i + c dt^2 [ K_ii (x) S v_i + sum_e K_ie (x) S v_e ],
//   K_ie[(k,n),(k',n')] = lam_j P(k,k') + mu_j P(k',k) + delta_kk' mu_j sum_l P(l,l),
//   P(a,b) = D~_{i,j}[a] D~_{e,j}[b]^T   (j the shared face; K_ii sums its own faces; K_ei = K_ie^T).
// K depends on the mesh and the medium alone (not on dt), so it is laid out once per medium: one
// d N_phi x d N_phi block per face and one per element.  Against the gather - E_j : - scatter form
// of the face kernels that is (d + 2)(d N_phi)^2 N_gamma products per element instead of
// 2 (d + 1)(d N_phi)^2 N_gamma plus the E_j : and S stages, no atomics, and one launch with the mass
// term in it.  FP64 runs at two lanes a clock and SM, so there the number of products decides; in
// FP32 the shapes without a specialised face kernel gain as well, since that generic kernel reads
// two shared-memory values per product.
//
// Because D_i y_i = r_i for y = P_1 r, the operator on a block-Jacobi preconditioned vector is
// A y = r + (off-diagonal part) y: neither the diagonal blocks nor the mass term are needed there.
#include <algorithm>
#include <cstdint>

#include "stdg_internal.h"

namespace stdg {

// ---------------------------------------------------------------------------------
// Set-up, FP64.  A thread takes a pair (n, n') of nodes: the d^2 products P(a,b)[n][n'] give the
// pair's entries of all component pairs (k, k').
// ---------------------------------------------------------------------------------
template <int DIM>
__device__ __forceinline__ void add_pair(const double* Da, const double* Db, int NP, int nn, int n2, double lam, double mu,
                                         double (&K)[DIM][DIM]) {
    double P[DIM][DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a)
#pragma unroll
        for (int b = 0; b < DIM; ++b) P[a][b] = 0.0;
    for (int m = 0; m < NP; ++m) {
        double u[DIM], v[DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            u[a] = Da[(a * NP + nn) * NP + m];
            v[a] = Db[(a * NP + n2) * NP + m];
        }
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
            for (int b = 0; b < DIM; ++b) P[a][b] = fma(u[a], v[b], P[a][b]);
    }
    double tr = 0.0;
#pragma unroll
    for (int l = 0; l < DIM; ++l) tr += P[l][l];
#pragma unroll
    for (int k = 0; k < DIM; ++k)
#pragma unroll
        for (int k2 = 0; k2 < DIM; ++k2) K[k][k2] += lam * P[k][k2] + mu * P[k2][k] + (k == k2 ? mu * tr : 0.0);
}

// K_lr of every interior face, rows of l(j), columns of r(j): one block per face
template <int DIM>
__global__ void __launch_bounds__(128) coupling_face_kernel(int64_t n_face, int NP, const int32_t* __restrict__ fr,
                                                            const double* __restrict__ D, const double* __restrict__ lamf,
                                                            const double* __restrict__ muf, double* __restrict__ K) {
    extern __shared__ double sD[];
    const int nD = DIM * NP * NP, n = DIM * NP;
    for (int64_t f = blockIdx.x; f < n_face; f += gridDim.x) {
        if (fr[f] < 0) continue;
        __syncthreads();
        for (int t = threadIdx.x; t < 2 * nD; t += blockDim.x) sD[t] = D[f * 2 * nD + t];
        __syncthreads();
        const double lam = lamf[f], mu = muf[f];
        for (int q = threadIdx.x; q < NP * NP; q += blockDim.x) {
            const int nn = q / NP, n2 = q % NP;
            double Kp[DIM][DIM] = {};
            add_pair<DIM>(sD, sD + nD, NP, nn, n2, lam, mu, Kp);
#pragma unroll
            for (int k = 0; k < DIM; ++k)
#pragma unroll
                for (int k2 = 0; k2 < DIM; ++k2) K[f * n * n + (k * NP + nn) * n + k2 * NP + n2] = Kp[k][k2];
        }
    }
}

// K_ii of every element, the sum over its faces: one block per element
template <int DIM>
__global__ void __launch_bounds__(128) coupling_diag_kernel(int64_t n_elem, int NP, const int32_t* __restrict__ elem_face,
                                                            const int32_t* __restrict__ fl, const double* __restrict__ D,
                                                            const double* __restrict__ lamf, const double* __restrict__ muf,
                                                            double* __restrict__ K) {
    extern __shared__ double sD[];
    const int nD = DIM * NP * NP, n = DIM * NP;
    for (int64_t e = blockIdx.x; e < n_elem; e += gridDim.x) {
        double lam[DIM + 1], mu[DIM + 1];
        __syncthreads();
#pragma unroll
        for (int i = 0; i <= DIM; ++i) {
            const int64_t f = elem_face[e * (DIM + 1) + i];
            const double* Df = D + (f * 2 + (fl[f] == (int)e ? 0 : 1)) * nD;
            for (int t = threadIdx.x; t < nD; t += blockDim.x) sD[i * nD + t] = Df[t];
            lam[i] = lamf[f];
            mu[i] = muf[f];
        }
        __syncthreads();
        for (int q = threadIdx.x; q < NP * NP; q += blockDim.x) {
            const int nn = q / NP, n2 = q % NP;
            double Kp[DIM][DIM] = {};
#pragma unroll
            for (int i = 0; i <= DIM; ++i) add_pair<DIM>(sD + i * nD, sD + i * nD, NP, nn, n2, lam[i], mu[i], Kp);
#pragma unroll
            for (int k = 0; k < DIM; ++k)
#pragma unroll
                for (int k2 = 0; k2 < DIM; ++k2) K[e * n * n + (k * NP + nn) * n + k2 * NP + n2] = Kp[k][k2];
        }
    }
}

cudaError_t launch_coupling_setup(stdg_ctx* c) {
    const int NP = c->Nphi;
    const size_t side = sizeof(double) * c->dim * NP * NP;
    const unsigned gf = (unsigned)std::min<int64_t>(c->n_face, (int64_t)c->n_sm * 64);
    const unsigned ge = (unsigned)std::min<int64_t>(c->n_elem, (int64_t)c->n_sm * 64);
    auto go = [&](auto face, auto diag) {
        cudaFuncSetAttribute(diag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)((c->dim + 1) * side));
        face<<<gf, 128, 2 * side, c->stream>>>(c->n_face, NP, c->d_face_r, c->d_D, c->d_lamf, c->d_muf, c->d_Kf); note_launch(c);
        diag<<<ge, 128, (c->dim + 1) * side, c->stream>>>(c->n_elem, NP, c->d_elem_face, c->d_face_l, c->d_D, c->d_lamf,
                                                          c->d_muf, c->d_Ke); note_launch(c);
    };
    if (c->dim == 2) go(coupling_face_kernel<2>, coupling_diag_kernel<2>);
    else go(coupling_face_kernel<3>, coupling_diag_kernel<3>);
    return cudaGetLastError();
}

// FP32 copies: K_ii as it is, the faces' blocks in both orientations by columns:
// out[2 f][j][i] = K_lr[i][j] for the l side, out[2 f + 1][j][i] = K_lr[j][i] for the r side.
__global__ void coupling_cast_kernel(int64_t n_face, int n, const double* __restrict__ K, float* __restrict__ out) {
    for (int64_t f = blockIdx.x; f < n_face; f += gridDim.x)
        for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
            const float v = (float)K[f * n * n + t];
            out[(2 * f + 1) * n * n + t] = v;
            out[2 * f * n * n + (t % n) * n + t / n] = v;
        }
}

cudaError_t launch_coupling_cast(stdg_ctx* c) {
    const int n = c->dim * c->Nphi;
    coupling_cast_kernel<<<(unsigned)std::min<int64_t>(c->n_face, (int64_t)c->n_sm * 64), 128, 0, c->stream>>>(c->n_face, n, c->d_Kf,
                                                                                                      c->d_Kf32); note_launch(c);
    return launch_cast32(c, c->d_Ke, c->d_Ke32, c->n_elem * n * n);
}

// ---------------------------------------------------------------------------------
// Application: dispatch over the shapes
// ---------------------------------------------------------------------------------
template <typename R>
cudaError_t coupling_2d(stdg_ctx*, const R*, const R*, const R*, const R*, const int*, int64_t, const R*, const int*, int64_t,
                        R*, double, int);
template <typename R>
cudaError_t coupling_3d(stdg_ctx*, const R*, const R*, const R*, const R*, const int*, int64_t, const R*, const int*, int64_t,
                        R*, double, int);

cudaError_t launch_coupling(stdg_ctx* c, const double* x, const int* xidx, int64_t ld, const double* base, const int* bidx,
                            int64_t bld, double* y, double scale, int nshots) {
    auto go = c->dim == 2 ? coupling_2d<double> : coupling_3d<double>;
    return go(c, c->d_Ke, c->d_Kf, c->d_rhoJ, x, xidx, ld, base, bidx, bld, y, scale, nshots);
}
cudaError_t launch_coupling32(stdg_ctx* c, const float* x, const int* xidx, int64_t ld, const float* base, const int* bidx,
                              int64_t bld, float* y, double scale, int nshots) {
    if (coupling_shots_applies(c, nshots, x, ld, base, bld, y))
        return launch_coupling_shots(c, x, xidx, ld, base, bidx, bld, y, scale, nshots);
    auto go = c->dim == 2 ? coupling_2d<float> : coupling_3d<float>;
    return go(c, c->d_Ke32, c->d_Kf32, c->d_rhoJ32, x, xidx, ld, base, bidx, bld, y, scale, nshots);
}

}  // namespace stdg
