// Block-Jacobi apply with one thread per (element, row): z = V (blockdiag B) V^T r (see precond.cu),
// instantiated per shape in pre1_rows.cu (FP64) and pre1_rows_f32.cu.
//
// FP64 is bound by the FP64 pipe, where an instruction takes 16 cycles of the SM however few lanes are
// active: one element per warp left 20 of 32 lanes idle at p = 2.  Here consecutive threads are
// consecutive rows of consecutive elements, so whole warps of a block work.  V goes straight to
// registers: columns (consecutive across the threads) for u = V^T r, pieces of the thread's row, now in
// cache, for z = V w.  Every V value feeds N_gamma products for SC shots.  The sums run in ascending
// order, as in the warp-per-element kernels that this replaces.
// Measured (warp per element -> here): FP64 2D p = 2 on 40,000 triangles 175 -> 68 us, p = 1 73 -> 15 us, 3D
// p = 3 on 3,072 tetrahedra 533 -> 179 us; FP32 2D p = 4 on 10,000 triangles 57 -> 14 us, 3D p = 3 89 -> 26 us,
// 2D p = 2 with 15 shots on 6,400 triangles 25 -> 16 us.
#pragma once
#include <algorithm>
#include <cstdint>

#include "stdg_internal.h"

namespace stdg {

template <typename R> struct Pair;
template <> struct Pair<float> { using T = float2; };
template <> struct Pair<double> { using T = double2; };

template <typename R, int DIM, int NP, int NG, int SC>
__global__ void __launch_bounds__(256) pre1_rows_kernel(int64_t n_elem, int EB, const R* __restrict__ V, const R* __restrict__ B,
                                                        const R* __restrict__ r, const int* __restrict__ ridx, int64_t ld,
                                                        R* __restrict__ z, int nshots, int64_t nvec) {
    constexpr int N = DIM * NP, NV = N * NG;
    using P = typename Pair<R>::T;
    static_assert(N % 2 == 0, "d N_phi is even for every supported order");
    extern __shared__ __align__(16) unsigned char smraw[];
    R* sr = reinterpret_cast<R*>(smraw);          // [shot of the chunk][element][row (k,n)][time]
    R* sw = sr + SC * EB * NV;                    // [shot of the chunk][element][q][time]
    if (ridx) r += (int64_t)(*ridx) * ld;
    const int64_t e0 = (int64_t)blockIdx.x * EB;
    const int ne = (int)min((int64_t)EB, n_elem - e0);
    const int le = threadIdx.x / N, q = threadIdx.x % N;
    const bool act = le < ne;
    const R* Ve = V + (e0 + (act ? le : 0)) * (N * N);
    R Bq[NG * NG];
    if (act) {
#pragma unroll
        for (int t = 0; t < NG * NG; ++t) Bq[t] = B[((e0 + le) * N + q) * (NG * NG) + t];
    }
    for (int s0 = 0; s0 < nshots; s0 += SC) {
        if (s0) __syncthreads();
        if (act) {
#pragma unroll
            for (int c = 0; c < SC; ++c) {
                if (SC > 1 && s0 + c >= nshots) break;
                const R* src = r + (int64_t)(s0 + c) * nvec + (e0 + le) * NV;
#pragma unroll
                for (int i = 0; i < NG; ++i) {
                    const int t = i * N + q, ka = t / NP, nn = t % NP, k = ka / NG, a = ka % NG;
                    sr[(c * EB + le) * NV + (k * NP + nn) * NG + a] = src[t];
                }
            }
        }
        __syncthreads();
        R u[SC][NG];
        if (act) {
#pragma unroll
            for (int c = 0; c < SC; ++c)
#pragma unroll
                for (int a = 0; a < NG; ++a) u[c][a] = (R)0;
#pragma unroll 6
            for (int row = 0; row < N; ++row) {
                const R v = __ldg(Ve + row * N + q);
#pragma unroll
                for (int c = 0; c < SC; ++c)
#pragma unroll
                    for (int a = 0; a < NG; ++a) u[c][a] = fma(v, sr[(c * EB + le) * NV + row * NG + a], u[c][a]);
            }
#pragma unroll
            for (int c = 0; c < SC; ++c)
#pragma unroll
                for (int a = 0; a < NG; ++a) {
                    R s = 0;
#pragma unroll
                    for (int b = 0; b < NG; ++b) s = fma(Bq[a * NG + b], u[c][b], s);
                    sw[(c * EB + le) * NV + q * NG + a] = s;
                }
        }
        __syncthreads();
        if (!act) continue;
#pragma unroll
        for (int c = 0; c < SC; ++c)
#pragma unroll
            for (int a = 0; a < NG; ++a) u[c][a] = (R)0;
#pragma unroll 3
        for (int j = 0; j < N; j += 2) {
            const P v = __ldg(reinterpret_cast<const P*>(Ve + q * N + j));
#pragma unroll
            for (int c = 0; c < SC; ++c)
#pragma unroll
                for (int a = 0; a < NG; ++a) {
                    u[c][a] = fma(v.x, sw[(c * EB + le) * NV + j * NG + a], u[c][a]);
                    u[c][a] = fma(v.y, sw[(c * EB + le) * NV + (j + 1) * NG + a], u[c][a]);
                }
        }
        const int k = q / NP, nn = q % NP;
#pragma unroll
        for (int c = 0; c < SC; ++c) {
            if (SC > 1 && s0 + c >= nshots) break;
#pragma unroll
            for (int a = 0; a < NG; ++a) z[(int64_t)(s0 + c) * nvec + (e0 + le) * NV + (k * NG + a) * NP + nn] = u[c][a];
        }
    }
}

// Elements per block, at most 160 threads: the size that fills its warps best.  FP64 is bound by the pipe of
// the SM that gets the most warps, so there only sizes count that give it at most 1/16 more than the best one
// does (1,000 elements of 30 rows: 10 warps in blocks of five, 7 of one).  1,444 triangles at p = 3: 38.3 -> 30.2 us,
// five shots 136.9 -> 112.3 us; 1,296 tetrahedra at p = 2 37.9 -> 36.3 us; sizes that already spread evenly keep their
// block.  In FP32 these calls take the launch's 17 to 26 us either way.
template <typename R, int DIM, int NP, int NG, int SC>
static cudaError_t pre1_rows_go(stdg_ctx* c, const R* V, const R* B, const R* r, const int* ridx, int64_t ld, R* z, int nshots) {
    constexpr int N = DIM * NP;
    const int most = (int)std::max<int64_t>(1, std::min<int64_t>(160 / N, c->n_elem / c->n_sm));
    auto busiest = [&](int e) {
        const int64_t blocks = (c->n_elem + e - 1) / e;
        return (blocks + c->n_sm - 1) / c->n_sm * ((e * N + 31) / 32);
    };
    int64_t least = busiest(1);
    for (int e = 2; e <= most; ++e) least = std::min(least, busiest(e));
    double best = 0.0;
    int EB = 1;
    for (int e = 1; e <= most; ++e) {
        const double eff = (double)(e * N) / ((e * N + 31) / 32 * 32);
        if ((sizeof(R) == 4 || busiest(e) * 16 <= least * 17) && eff >= best) { best = eff; EB = e; }
    }
    const size_t smem = sizeof(R) * 2 * (size_t)SC * EB * N * NG;
    auto kern = pre1_rows_kernel<R, DIM, NP, NG, SC>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<(unsigned)((c->n_elem + EB - 1) / EB), (EB * N + 31) / 32 * 32, smem, c->stream>>>(c->n_elem, EB, V, B, r, ridx, ld, z,
                                                                                             nshots, c->nvel);
    note_launch(c);
    return cudaGetLastError();
}

template <typename R, int DIM, int NP>
static cudaError_t pre1_rows_shape(stdg_ctx* c, const R* V, const R* B, const R* r, const int* ridx, int64_t ld, R* z, int ns) {
#define STDG_NG(NG_)                                                                           \
    case NG_:                                                                                  \
        return ns == 1 ? pre1_rows_go<R, DIM, NP, NG_, 1>(c, V, B, r, ridx, ld, z, ns)         \
                       : pre1_rows_go<R, DIM, NP, NG_, 4>(c, V, B, r, ridx, ld, z, ns);
    switch (c->Ng) {
        STDG_NG(1)
        STDG_NG(2)
        STDG_NG(3)
        STDG_NG(4)
        STDG_NG(5)
        default: return cudaErrorInvalidValue;
    }
#undef STDG_NG
}

template <typename R>
static cudaError_t pre1_rows(stdg_ctx* c, const R* V, const R* B, const R* r, const int* ridx, int64_t ld, R* z, int ns) {
    switch (c->dim * 100 + c->Nphi) {
        case 203: return pre1_rows_shape<R, 2, 3>(c, V, B, r, ridx, ld, z, ns);
        case 206: return pre1_rows_shape<R, 2, 6>(c, V, B, r, ridx, ld, z, ns);
        case 210: return pre1_rows_shape<R, 2, 10>(c, V, B, r, ridx, ld, z, ns);
        case 215: return pre1_rows_shape<R, 2, 15>(c, V, B, r, ridx, ld, z, ns);
        case 304: return pre1_rows_shape<R, 3, 4>(c, V, B, r, ridx, ld, z, ns);
        case 310: return pre1_rows_shape<R, 3, 10>(c, V, B, r, ridx, ld, z, ns);
        case 320: return pre1_rows_shape<R, 3, 20>(c, V, B, r, ridx, ld, z, ns);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace stdg
