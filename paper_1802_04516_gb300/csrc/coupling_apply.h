// Application of the assembled element couplings (see coupling.cu), instantiated per shape and
// precision in coupling_2d.cu, coupling_3d.cu and their FP32 counterparts.
#pragma once
#include <algorithm>
#include <cstdint>

#include "compensated.h"
#include "stdg_internal.h"

namespace stdg {

// ---------------------------------------------------------------------------------
// Application.  A block takes EB elements; the values of the elements and of their neighbours come
// into shared memory as [row][time].  Thread (element, rows) forms the N_gamma sums of its rows for
// SC shots at a time.  A value of K is used by one thread alone, so it goes straight from memory to a
// register.
// FP64: bound by the pipe (0.97 busy at p = 4; an FP64 instruction takes 16 cycles of the SM however few lanes are
// active), so a thread has one row and at most one lane in 16 is idle (17,956 triangles, p = 4,
// p_gamma = 2: 642 us with the face and mass kernels, 410 us here; 40,000 at p = 2: 398 and 163 us).  K_ii and the r
// side's K_lr^T are read by columns (consecutive across the threads), the l side's K_lr by pieces of
// its rows; the two ways of loading differ between the elements of a warp, the products do not.
// FP32: bound by the latency of K from memory (3D p = 3, 7,986 tetrahedra: 605 MB at 0.54 of the DRAM peak, 0.22 of the
// warps resident, 6.9 of 9.5 cycles an instruction waits on a long scoreboard; L1 data pipe 0.37).  A thread has two
// consecutive rows, so that one 16-byte read of the staged values feeds them all, and the faces' blocks are
// kept in both orientations, so that every load is a vector load of consecutive columns (reading rows of
// one copy cost a wavefront per lane).
// Smooth vectors: the face term of a constant vanishes, which the face form sees before it multiplies by the
// stiffness and the couplings only in the sum of their products.  So the value of the element's first node is
// taken off its own and its neighbours' values, per component and time node, wherever every one of these
// subtractions is exact; the mass term adds it again.  Otherwise (rough vectors, a change of binade) the values
// stay as they are.  FP32 error on smooth vectors 1.1 to 2.0 times the face form's without this, 0.7 to 1.2 with
// it, on constants 1.3 to 2.2 and 0.03 to 0.7; it costs 1 to 10% of a call (FP64 p = 4 on 17,956 triangles: 406 -> 410 us, p = 2 on 40,000
// 163 -> 172 us; FP32 3D p = 3 on 7,986 tetrahedra 149 -> 153 us, p = 1 on 131,712 91 -> 102 us), 17% with one time node in FP32.
// ---------------------------------------------------------------------------------
template <typename R, int DIM, int NP, int NG, int SC>
struct Coupling {
    static constexpr int N = DIM * NP, FACES = DIM + 1, NV = N * NG;
    static constexpr bool BOTH = sizeof(R) == 4;                          // the faces' blocks are kept in both orientations
    static constexpr int RPT = BOTH ? 2 : 1, TPE = N / RPT;   // rows per thread, threads per element
    static constexpr int NGP = NG <= 2 ? NG : (NG <= 4 ? 4 : 6);          // row stride of the staged values
    static constexpr int VJ = !BOTH || SC > 1 ? 2 : (N % 10 == 0 ? 10 : 6);   // columns loaded together
    static constexpr int BL = !BOTH ? N : (N % 10 == 0 ? 10 : 6);         // columns per turn of the loop
    // FP32: columns summed before they join the total (compensated.h)
    static constexpr int CH = !BOTH || SC > 1 ? BL : BL / 2;
    static_assert(N % BL == 0 && BL % VJ == 0 && (CH == BL || (VJ == BL && VJ % CH == 0)), "chunks of whole loads");
    static_assert(N % 2 == 0, "d N_phi is even for every supported order");
    __host__ __device__ static constexpr int slots(bool own) { return FACES + (own ? 1 : 0); }
    static constexpr int KA = DIM * NG;                       // constants of an element
    // resident blocks of 160 threads that the compiler has to leave registers for, one shot with the element's own
    // block: as many as fit without spills, fewer where ten columns are loaded together (FP32 3D p = 2, p_gamma = 1 204 -> 162 us,
    // p = 3, p_gamma = 2 211 -> 150 us against the compiler's own choice; at p = 1 and 2 the same limit costs 20 to 40%)
    __host__ __device__ static constexpr int blocks() {
        if (!BOTH) return NG == 1 ? 7 : NG == 2 ? 5 : NG == 3 ? 4 : 3;
        if (NG == 5) return DIM == 2 && N == 30 ? 3 : 2;
        return N % 10 == 0 || NG == 4 ? 3 : NG == 3 ? 5 : NG == 2 ? 6 : 8;
    }
    static size_t smem(int EB, bool own) {
        return sizeof(R) * (size_t)SC * slots(own) * EB * N * NGP + (own ? (sizeof(R) + sizeof(int)) * (size_t)SC * EB * KA : 0);
    }
};

// v - c is exact: c finite, v of the same sign and exponent (then c / 2 < v < 2 c, Sterbenz 1974)
__device__ __forceinline__ bool exact_difference(float v, float c) {
    const unsigned cb = __float_as_uint(c);
    return (__float_as_uint(v) ^ cb) >> 23 == 0 && (cb & 0x7f800000u) != 0x7f800000u;
}
__device__ __forceinline__ bool exact_difference(double v, double c) {
    const unsigned cb = (unsigned)__double2hiint(c);
    return ((unsigned)__double2hiint(v) ^ cb) >> 20 == 0 && (cb & 0x7ff00000u) != 0x7ff00000u;
}

template <typename R, int W> struct Piece;
template <> struct Piece<float, 2> { using T = float2; };
template <> struct Piece<double, 2> { using T = double2; };

template <typename R, int DIM, int NP, int NG, int SC, bool OWN>
__global__ void __launch_bounds__(OWN && SC == 1 ? 160 : 256, OWN && SC == 1 ? Coupling<R, DIM, NP, NG, SC>::blocks() : 0) coupling_apply_kernel(int64_t n_elem, int EB, const int2* __restrict__ adj,
                                                             const R* __restrict__ Ke, const R* __restrict__ Kf,
                                                             const R* __restrict__ rhoJ, const RefTables* __restrict__ rtp,
                                                             const R* __restrict__ x, const int* __restrict__ xidx, int64_t ld,
                                                             const R* __restrict__ base, const int* __restrict__ bidx,
                                                             int64_t bld, R* __restrict__ y, double scale, int nshots,
                                                             int64_t nvec) {
    using C = Coupling<R, DIM, NP, NG, SC>;
    constexpr int N = C::N, FACES = C::FACES, NV = C::NV, RPT = C::RPT, TPE = C::TPE, NGP = C::NGP, VJ = C::VJ;
    constexpr int SLOTS = C::slots(OWN), OFF = OWN ? 1 : 0;   // slot 0: the element itself, unless a base vector stands for it
    using P = typename Piece<R, 2>::T;   // two rows of a column (FP32), two columns of a row (FP64)
    extern __shared__ __align__(16) unsigned char smraw[];
    constexpr int KA = C::KA;
    __shared__ R sM[OWN ? NP * NP : 1], sM1[OWN ? NP : 1], sT[NG * NG], sS[NG * NG];
    R* sx = reinterpret_cast<R*>(smraw);                      // [shot of the chunk][slot][element][row (k,n)][time]
    R* sc = sx + SC * SLOTS * EB * N * NGP;                   // [shot of the chunk][element][k][time]: the first node's value
    int* sb = reinterpret_cast<int*>(sc + SC * EB * KA);      // the same: some subtraction would not be exact, nothing is taken off
    if (xidx) x += (int64_t)(*xidx) * ld;
    if (!OWN && bidx) base += (int64_t)(*bidx) * bld;
    const int64_t e0 = (int64_t)blockIdx.x * EB;
    const int ne = (int)min((int64_t)EB, n_elem - e0);
    if (OWN)
        for (int t = threadIdx.x; t < NP * NP; t += blockDim.x) sM[t] = (R)rtp->Mref[t];
    if (OWN)
        for (int t = threadIdx.x; t < NP; t += blockDim.x) sM1[t] = (R)rtp->Mrow[t];
    for (int t = threadIdx.x; t < NG * NG; t += blockDim.x) {
        if (OWN) sT[t] = (R)rtp->T[t];
        sS[t] = (R)(scale * rtp->S[t]);   // rounded once: its error is common to all elements
    }
    const int le = threadIdx.x / TPE, row = threadIdx.x % TPE;
    const bool act = le < ne;
    int2 nb[FACES];                                           // the thread's element: neighbours, face and side
#pragma unroll
    for (int i = 0; i < FACES; ++i) nb[i] = act ? adj[(e0 + le) * FACES + i] : make_int2(-1, 0);
    for (int s0 = 0; s0 < nshots; s0 += SC) {
        if (s0) __syncthreads();                              // the chunk before has been read
        if (OWN) {
            for (int t = threadIdx.x; t < SC * EB * KA; t += blockDim.x) sb[t] = 0;
            __syncthreads();
        }
        if (act) {   // the threads of an element stage its slots
            static_assert(NV % TPE == 0, "a thread stages whole rounds of values");
            constexpr int NVT = NV / TPE;
            R first[SC == 1 ? NVT : 1];                       // of the values that the thread stages (one shot: loaded once)
            unsigned rough[SC] = {};                          // bit i: a subtraction of value i's constant would round
            if constexpr (OWN && SC == 1) {
#pragma unroll
                for (int i = 0; i < NVT; ++i) first[i] = x[(int64_t)s0 * nvec + (e0 + le) * NV + (i * TPE + row) / NP * NP];
            }
#pragma unroll
            for (int sl = 0; sl < SLOTS; ++sl) {
                const int64_t e = sl < OFF ? e0 + le : nb[sl < OFF ? 0 : sl - OFF].x;
                if (e < 0) continue;
#pragma unroll
                for (int c = 0; c < SC; ++c) {
                    if (SC > 1 && s0 + c >= nshots) break;
                    const R* src = x + (int64_t)(s0 + c) * nvec + e * NV;
                    R* dst = sx + ((c * SLOTS + sl) * EB + le) * (N * NGP);
#pragma unroll
                    for (int t0 = 0; t0 < NV; t0 += TPE) {
                        const int t = t0 + row, ka = t / NP, nn = t % NP, k = ka / NG, a = ka % NG;
                        const R v = src[t];
                        dst[(k * NP + nn) * NGP + a] = v;
                        if (OWN) {
                            if (sl == 0 && nn == 0) sc[(c * EB + le) * KA + ka] = v;
                            const R f = SC == 1 ? first[SC == 1 ? t0 / TPE : 0] : x[(int64_t)(s0 + c) * nvec + (e0 + le) * NV + ka * NP];
                            rough[c] |= (exact_difference(v, f) ? 0u : 1u) << (t0 / TPE);
                        }
                    }
                }
            }
            if (OWN) {
#pragma unroll
                for (int c = 0; c < SC; ++c)
#pragma unroll
                    for (int i = 0; i < NVT; ++i)
                        if (rough[c] >> i & 1) sb[(c * EB + le) * KA + (i * TPE + row) / NP] = 1;
            }
        }
        __syncthreads();
        if (OWN) {
            if (act) {
#pragma unroll 1
                for (int q = row; q < SC * NV; q += TPE) {
                    const int c = q / NV, t = q % NV, ka = t / NP, nn = t % NP, k = ka / NG, a = ka % NG;
                    const int at = (c * EB + le) * KA + ka;
                    if (sb[at]) continue;
                    const R off = sc[at];
                    R* v = sx + (c * SLOTS * EB + le) * (N * NGP) + (k * NP + nn) * NGP + a;
#pragma unroll
                    for (int sl = 0; sl < SLOTS; ++sl) v[sl * EB * N * NGP] -= off;   // (slots of missing neighbours are not read)
                }
            }
            __syncthreads();
        }
        if (!act) continue;
        R bs[OWN || SC > 1 ? 1 : RPT][NG];   // the base values, loaded ahead of the sums
        if constexpr (!OWN && SC == 1) {
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int i = row * RPT + r, k = i / NP, nn = i % NP;
#pragma unroll
                for (int a = 0; a < NG; ++a) bs[r][a] = base[(int64_t)s0 * nvec + (e0 + le) * NV + (k * NG + a) * NP + nn];
            }
        }
        R acc[RPT][SC][NG], low[C::BOTH ? RPT : 1][C::BOTH ? SC : 1][C::BOTH ? NG : 1];   // totals, what their joins rounded away
#pragma unroll
        for (int r = 0; r < RPT; ++r)
#pragma unroll
            for (int c = 0; c < SC; ++c)
#pragma unroll
                for (int a = 0; a < NG; ++a) {
                    acc[r][c][a] = (R)0;
                    if constexpr (C::BOTH) low[r][c][a] = (R)0;
                }
        for (int sl = 0; sl < SLOTS; ++sl) {
            const R* kp = Ke + (e0 + le) * (N * N);
            bool by_rows = false, on = true;
            if (sl >= OFF) {
                int2 a = nb[0];
#pragma unroll
                for (int i = 1; i < FACES; ++i)
                    if (sl - OFF == i) a = nb[i];
                on = a.x >= 0;
                by_rows = !C::BOTH && !(a.y & 1);
                kp = Kf + (int64_t)(C::BOTH ? a.y : a.y >> 1) * (N * N);
            }
            if (!on) continue;
            const R* xp = sx + (sl * EB + le) * (N * NGP);
#pragma unroll 1
            for (int jc = 0; jc < N; jc += C::BL) {
                R sum[RPT][SC][NG];   // short sums first: rounding grows with the square root of a chain's length
#pragma unroll
                for (int r = 0; r < RPT; ++r)
#pragma unroll
                    for (int c = 0; c < SC; ++c)
#pragma unroll
                        for (int a = 0; a < NG; ++a) sum[r][c][a] = (R)0;
                auto join_all = [&]() {
#pragma unroll
                    for (int r = 0; r < RPT; ++r)
#pragma unroll
                        for (int c = 0; c < SC; ++c)
#pragma unroll
                            for (int a = 0; a < NG; ++a) {
                                if constexpr (C::BOTH) join(acc[r][c][a], low[r][c][a], sum[r][c][a]);
                                else acc[r][c][a] += sum[r][c][a];
                                sum[r][c][a] = (R)0;
                            }
                };
#pragma unroll 3
                for (int j = jc; j < jc + C::BL; j += VJ) {
                    R kv[VJ][RPT];
                    if constexpr (C::BOTH) {
#pragma unroll
                        for (int q = 0; q < VJ; ++q)
                            *reinterpret_cast<P*>(kv[q]) = __ldg(reinterpret_cast<const P*>(kp + (j + q) * N + row * RPT));
                    } else if (by_rows) {
                        const P t = __ldg(reinterpret_cast<const P*>(kp + row * N + j));
                        kv[0][0] = t.x;
                        kv[1][0] = t.y;
                    } else {
#pragma unroll
                        for (int q = 0; q < VJ; ++q) kv[q][0] = __ldg(kp + (j + q) * N + row);
                    }
#pragma unroll
                    for (int q = 0; q < VJ; ++q) {
#pragma unroll
                        for (int c = 0; c < SC; ++c) {
                            R xv[NGP];
                            const R* xq = xp + c * (SLOTS * EB * N * NGP) + (j + q) * NGP;
                            if constexpr (sizeof(R) == 4 && NGP == 4) {
                                *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(xq);
                            } else {
#pragma unroll
                                for (int a = 0; a < NG; ++a) xv[a] = xq[a];
                            }
#pragma unroll
                            for (int r = 0; r < RPT; ++r)
#pragma unroll
                                for (int a = 0; a < NG; ++a) sum[r][c][a] = fma(kv[q][r], xv[a], sum[r][c][a]);
                        }
                        if constexpr (C::CH < C::BL)
                            if ((q + 1) % C::CH == 0) join_all();
                    }
                }
                if constexpr (C::CH == C::BL) join_all();
            }
        }
        const R rj = OWN ? rhoJ[e0 + le] : (R)0;
#pragma unroll
        for (int c = 0; c < SC; ++c) {
            if (SC > 1 && s0 + c >= nshots) break;
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int i = row * RPT + r, k = i / NP, nn = i % NP;
                const int64_t at = (int64_t)(s0 + c) * nvec + (e0 + le) * NV + k * (NG * NP) + nn;
                R u[NG];
#pragma unroll
                for (int a = 0; a < NG; ++a) u[a] = (R)0;
                if (OWN) {
                    const R* xp = sx + (c * SLOTS * EB + le) * (N * NGP) + k * (NP * NGP);
                    for (int q = 0; q < NP; ++q) {
                        const R mv = sM[nn * NP + q];
#pragma unroll
                        for (int a = 0; a < NG; ++a) u[a] = fma(mv, xp[q * NGP + a], u[a]);
                    }
#pragma unroll
                    for (int a = 0; a < NG; ++a) {
                        const int at = (c * EB + le) * KA + k * NG + a;
                        u[a] = fma(sM1[nn], sb[at] ? (R)0 : sc[at], u[a]);
                    }
#pragma unroll
                    for (int a = 0; a < NG; ++a) u[a] *= rj;
                }
#pragma unroll
                for (int a = 0; a < NG; ++a) {
                    R o = OWN ? (R)0 : SC == 1 ? bs[OWN || SC > 1 ? 0 : r][a] : base[at + a * NP];
#pragma unroll
                    for (int b = 0; b < NG; ++b) {
                        if constexpr (C::BOTH) o = fma(sS[a * NG + b], rest(acc[r][c][b], low[r][c][b]), o);
                        o = fma(sS[a * NG + b], acc[r][c][b], o);
                        if (OWN) o = fma(sT[a * NG + b], u[b], o);
                    }
                    y[at + a * NP] = o;
                }
            }
        }
    }
}

// Elements per block: whole warps of threads (an idle lane costs as much as a busy one), at most
// 160 threads and 48 KB, and at least one block per SM on small meshes.
template <typename R, int DIM, int NP, int NG, int SC, bool OWN>
static cudaError_t coupling_go(stdg_ctx* c, const R* Ke, const R* Kf, const R* rhoJ, const R* x, const int* xidx, int64_t ld,
                               const R* base, const int* bidx, int64_t bld, R* y, double scale, int nshots) {
    using C = Coupling<R, DIM, NP, NG, SC>;
    const int most = (int)std::max<int64_t>(1, std::min<int64_t>(160 / C::TPE, c->n_elem / c->n_sm));
    double best = 0.0;
    int EB = 1;
    for (int e = 1; e <= most && (e == 1 || C::smem(e, OWN) <= 48 * 1024); ++e) {
        const double eff = (double)(e * C::TPE) / ((e * C::TPE + 31) / 32 * 32);
        if (eff >= best) { best = eff; EB = e; }
    }
    const size_t smem = C::smem(EB, OWN);
    auto kern = coupling_apply_kernel<R, DIM, NP, NG, SC, OWN>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<(unsigned)((c->n_elem + EB - 1) / EB), (EB * C::TPE + 31) / 32 * 32, smem, c->stream>>>(
        c->n_elem, EB, c->d_adj, Ke, Kf, rhoJ, c->d_rt, x, xidx, ld, base, bidx, bld, y, scale, nshots, c->nvel);
    note_launch(c);
    return cudaGetLastError();
}

template <typename R, int DIM, int NP, int NG>
static cudaError_t coupling_ng(stdg_ctx* c, const R* Ke, const R* Kf, const R* rhoJ, const R* x, const int* xidx, int64_t ld,
                               const R* base, const int* bidx, int64_t bld, R* y, double scale, int ns) {
    if (base) return ns == 1 ? coupling_go<R, DIM, NP, NG, 1, false>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns)
                             : coupling_go<R, DIM, NP, NG, 4, false>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
    return ns == 1 ? coupling_go<R, DIM, NP, NG, 1, true>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns)
                   : coupling_go<R, DIM, NP, NG, 4, true>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
}

// (the FP32 shapes with a tiled face kernel keep no FP32 couplings: coupling32_wanted)
template <typename R, int DIM, int NP>
static cudaError_t coupling_shape(stdg_ctx* c, const R* Ke, const R* Kf, const R* rhoJ, const R* x, const int* xidx, int64_t ld,
                                  const R* base, const int* bidx, int64_t bld, R* y, double scale, int ns) {
    switch (c->Ng) {
        case 1: return coupling_ng<R, DIM, NP, 1>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        case 2: return coupling_ng<R, DIM, NP, 2>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        case 3:
            if constexpr (sizeof(R) == 8 || DIM != 3 || NP != 10)
                return coupling_ng<R, DIM, NP, 3>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
            return cudaErrorInvalidValue;
        case 4:
            if constexpr (sizeof(R) == 8 || DIM != 2 || NP != 10)
                return coupling_ng<R, DIM, NP, 4>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
            return cudaErrorInvalidValue;
        case 5: return coupling_ng<R, DIM, NP, 5>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace stdg
