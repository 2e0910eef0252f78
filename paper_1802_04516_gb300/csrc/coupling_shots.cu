// The FP32 operator from assembled couplings for stacked shots, 2D at p = p_gamma = 2 (the multi-shot
// and inversion workloads): one lane per shot.  A warp takes 32 / SH elements with SH shots each; a
// lane keeps its shot's 12 x 3 sums and the 36 values of the current slot (a neighbour, or the
// element itself) in registers, and the slot's 12 x 12 block of K is read from shared memory by all
// lanes of the element at once: three 16-byte reads feed 36 products.  Products run on the packed
// FP32 FMA over pairs of rows.  Against the face kernel with one lane per shot (gather, stress and
// scatter with 72 inputs and 72 outputs per face, 1.5 faces per element, atomics, a mass kernel ahead)
// a shot and element costs 1,728 products instead of 4,050 and no vector is updated in memory: the
// off-diagonal part of 64 shots on 12,544 triangles takes 139 us (282 us with the face and mass
// kernels), of 32 shots on 4,096 triangles 33 us (67 us), of 8 on 3,844 11.5 us (30 us).  Plain sums took 113, 25
// and 9.4 us, with up to a third more error.  Bound by latency at eight warps an SM (0.12 of the warps: 254 registers and
// 21 KB of ring a warp; 64 shots on 12,544 triangles: issue 0.45 busy, DRAM 0.33, L1 0.35 of their peaks, the longest
// stall a fixed-latency dependency); shared-memory reads and the joins of the compensated sums come next.
//
// Every warp runs a ring of four slot buffers (the shots' rows and K; buffer = slot), filled by
// cp.async three slots ahead across element boundaries: three neighbours, then the element's own
// values (or the base vector's in the off-diagonal form).  The sums leave through the last buffer so
// that the stores are consecutive along each shot's row.
#include <algorithm>
#include <cstdint>

#include "stdg_internal.h"
#include "tma.h"

namespace stdg {

struct CouplingShots {
    static constexpr int NP = 6, NG = 3, N = 12, NV = 36, NK = N * N;
    static constexpr int CPR = NV / 4;                        // 16-byte pieces of a row (9: an odd stride, no bank conflicts)
    static constexpr int ROWS = 32 * NV;
    static constexpr int CH = 6;                              // columns summed before they join the total
    template <int SH> static constexpr int buf() { return ROWS + 32 / SH * NK; }
    template <int SH> static constexpr size_t warp_bytes() { return sizeof(float) * 4 * buf<SH>(); }
};

__device__ __forceinline__ void cs_cp16(float* dst, const float* src, bool on) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 16u : 0u)
                 : "memory");
}

// compensated sum (Kahan 1965): the error of a total of 48 products stays that of its short sums.  Kahan's own
// arrangement holds one value less than that of compensated.h, and registers are what this kernel lacks (64
// shots on 12,544 triangles: preconditioner 332 us, 380 us with the other).  It makes NaN of an infinite total, which
// no caller sees: these results go through S^{-1} or into a solve, which ends alike on either.
__device__ __forceinline__ void cs_join(float& acc, float& lost, float sum) {
    const float add = sum - lost, t = acc + add;
    lost = (t - acc) - add;
    acc = t;
}

template <int SH, bool OWN>
__global__ void __launch_bounds__(128) coupling_shots_kernel(int64_t n_elem, const int2* __restrict__ adj,
                                                             const float* __restrict__ Ke, const float* __restrict__ Kf,
                                                             const float* __restrict__ rhoJ, const RefTables* __restrict__ rtp,
                                                             const float* __restrict__ x, const int* __restrict__ xidx, int64_t ld,
                                                             const float* __restrict__ base, const int* __restrict__ bidx,
                                                             int64_t bld, float* __restrict__ y, double scale, int nshots,
                                                             int64_t nvec) {
    using C = CouplingShots;
    constexpr int NP = C::NP, NG = C::NG, N = C::N, NV = C::NV, NK = C::NK, CPR = C::CPR, EPW = 32 / SH, BUF = C::ROWS + EPW * NK;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ float sM[NP * NP];
    if (xidx) x += (int64_t)(*xidx) * ld;
    if (!OWN && bidx) base += (int64_t)(*bidx) * bld;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    float* ring = reinterpret_cast<float*>(smraw) + warp * 4 * BUF;
    if (OWN)
        for (int t = threadIdx.x; t < NP * NP; t += blockDim.x) sM[t] = (float)rtp->Mref[t];
    float Sm[NG][NG], Tm[NG][NG];
#pragma unroll
    for (int a = 0; a < NG; ++a)
#pragma unroll
        for (int b = 0; b < NG; ++b) {
            Sm[a][b] = (float)(scale * rtp->S[a * NG + b]);   // rounded once: its error is common to all elements
            Tm[a][b] = OWN ? (float)rtp->T[a * NG + b] : 0.f;
        }
    __syncthreads();
    const int sub = lane / SH;                                // the lane's element of the warp's group
    const int nc = (nshots + SH - 1) / SH;                    // chunks of SH shots
    const int64_t n_grp = (n_elem + EPW - 1) / EPW;
    const int64_t gw = blockIdx.x * (int64_t)wpb + warp, W = (int64_t)gridDim.x * wpb;
    const int64_t n_items = (gw < n_grp ? (n_grp - 1 - gw) / W + 1 : 0) * nc;
    struct Item { int e; int2 nb[3]; };                       // e < 0: the lane has no element
    auto fetch = [&](int64_t t) {
        Item it;
        const int64_t e = t < n_items ? (gw + t / nc * W) * EPW + sub : n_elem;
        it.e = e < n_elem ? (int)e : -1;
#pragma unroll
        for (int i = 0; i < 3; ++i) it.nb[i] = it.e >= 0 ? adj[e * 3 + i] : make_int2(-1, 0);
        return it;
    };
    // copies of slot sl of an item into buffer sl: the 32 lanes' rows in order (consecutive pieces of a
    // shot's row are consecutive in memory), then each element's block of K
    auto issue = [&](const Item& it, int64_t t, int sl) {
        if (t < n_items) {
            float* buf = ring + sl * BUF;
            const int c0 = (int)(t % nc) * SH;
            const int e = sl == 3 ? it.e : it.nb[sl].x;
            const float* v = (sl == 3 && !OWN) ? base : x;
#pragma unroll
            for (int u = 0; u < CPR; ++u) {
                const int ci = lane + 32 * u, r = ci / CPR, j = ci % CPR;
                const int er = EPW == 1 ? e : __shfl_sync(FULL, e, r);
                const int shot = c0 + r % SH;
                const bool ok = er >= 0 && shot < nshots;
                cs_cp16(buf + r * NV + 4 * j, v + (ok ? (int64_t)shot * nvec + (int64_t)er * NV + 4 * j : 0), ok);
            }
            if (sl < 3 || OWN) {
                const int64_t blk = sl == 3 ? it.e : it.nb[sl].y;
#pragma unroll
                for (int u = 0; u < (EPW * NK / 4 + 31) / 32; ++u) {
                    const int ci = lane + 32 * u, q = ci / (NK / 4), j = ci % (NK / 4);
                    const int from = min(q, EPW - 1) * SH;
                    const int er = EPW == 1 ? e : __shfl_sync(FULL, e, from);
                    const int64_t bk = EPW == 1 ? blk : __shfl_sync(FULL, blk, from);
                    const bool ok = q < EPW && er >= 0;
                    if (q < EPW) cs_cp16(buf + C::ROWS + q * NK + 4 * j, (sl == 3 ? Ke : Kf) + (ok ? bk * NK + 4 * j : 0), ok);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    Item cur = fetch(0), nxt = fetch(1);
    issue(cur, 0, 0);
    issue(cur, 0, 1);
    issue(cur, 0, 2);
    for (int64_t t = 0; t < n_items; ++t) {
        const Item far = fetch(t + 2);
        float2 acc[N / 2][NG], lost[N / 2][NG];                // totals, what their last join rounded away
#pragma unroll
        for (int i = 0; i < N / 2; ++i)
#pragma unroll
            for (int a = 0; a < NG; ++a) acc[i][a] = lost[i][a] = make_float2(0.f, 0.f);
        float out[N][NG];
#pragma unroll
        for (int sl = 0; sl < 4; ++sl) {
            if (sl == 0) {
                issue(cur, t, 3);                              // free since the end of the item before
            } else {
                __syncwarp();                                  // every lane has read the slot before: its buffer is free
                issue(nxt, t + 1, sl - 1);
            }
            asm volatile("cp.async.wait_group 3;" ::: "memory");
            __syncwarp();
            const float* buf = ring + sl * BUF;
            float v[NV];                                       // canonical order [k][time][n]
#pragma unroll
            for (int q = 0; q < CPR; ++q) {
                const float4 f = reinterpret_cast<const float4*>(buf + lane * NV)[q];
                v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
            }
            if (sl < 3 || OWN) {   // rows of a missing neighbour are zero (zero-filled copies)
                const float4* kp = reinterpret_cast<const float4*>(buf + C::ROWS + sub * NK);
#pragma unroll
                for (int g = 0; g < N / 4; ++g)                // four rows at a time: short sums, few registers
#pragma unroll
                    for (int j0 = 0; j0 < N; j0 += C::CH) {
                        float2 sum[2][NG];
#pragma unroll
                        for (int j = j0; j < j0 + C::CH; ++j) {
                            const float4 f = kp[j * (N / 4) + g];
#pragma unroll
                            for (int a = 0; a < NG; ++a) {
                                const float xv = v[(j / NP * NG + a) * NP + j % NP];
                                sum[0][a] = ffma2(make_float2(f.x, f.y), make_float2(xv, xv), j > j0 ? sum[0][a] : make_float2(0.f, 0.f));
                                sum[1][a] = ffma2(make_float2(f.z, f.w), make_float2(xv, xv), j > j0 ? sum[1][a] : make_float2(0.f, 0.f));
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int a = 0; a < NG; ++a) {
                                cs_join(acc[2 * g + i][a].x, lost[2 * g + i][a].x, sum[i][a].x);
                                cs_join(acc[2 * g + i][a].y, lost[2 * g + i][a].y, sum[i][a].y);
                            }
                    }
            }
            if (sl == 3) {
                const float rj = OWN && cur.e >= 0 ? rhoJ[cur.e] : 0.f;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int k = i / NP, nn = i % NP;
                    float m[NG];
                    if (OWN) {
#pragma unroll
                        for (int a = 0; a < NG; ++a) {
                            m[a] = 0.f;
#pragma unroll
                            for (int q = 0; q < NP; ++q) m[a] = fmaf(sM[nn * NP + q], v[(k * NG + a) * NP + q], m[a]);
                            m[a] *= rj;
                        }
                    }
#pragma unroll
                    for (int a = 0; a < NG; ++a) {
                        float o = OWN ? 0.f : v[(k * NG + a) * NP + nn];
#pragma unroll
                        for (int b = 0; b < NG; ++b) {
                            o = fmaf(Sm[a][b], -(i % 2 ? lost[i / 2][b].y : lost[i / 2][b].x), o);
                            o = fmaf(Sm[a][b], i % 2 ? acc[i / 2][b].y : acc[i / 2][b].x, o);
                            if (OWN) o = fmaf(Tm[a][b], m[b], o);
                        }
                        out[i][a] = o;
                    }
                }
            }
        }
        // out through buffer 3 (each lane has read its own row of it), then along the shots' rows
        float* row = ring + 3 * BUF + lane * NV;
#pragma unroll
        for (int q = 0; q < CPR; ++q) {
            float f[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int at = 4 * q + u, k = at / (NG * NP), a = (at / NP) % NG, nn = at % NP;
                f[u] = out[k * NP + nn][a];
            }
            reinterpret_cast<float4*>(row)[q] = make_float4(f[0], f[1], f[2], f[3]);
        }
        __syncwarp();
        const int c0 = (int)(t % nc) * SH;
#pragma unroll
        for (int u = 0; u < CPR; ++u) {
            const int ci = lane + 32 * u, r = ci / CPR, j = ci % CPR;
            const int er = EPW == 1 ? cur.e : __shfl_sync(FULL, cur.e, r);
            const int shot = c0 + r % SH;
            if (er >= 0 && shot < nshots)
                *reinterpret_cast<float4*>(y + (int64_t)shot * nvec + (int64_t)er * NV + 4 * j) =
                    *reinterpret_cast<const float4*>(ring + 3 * BUF + r * NV + 4 * j);
        }
        __syncwarp();   // buffer 3 is free for the next item
        cur = nxt;
        nxt = far;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int SH, bool OWN>
static cudaError_t go(stdg_ctx* c, const float* x, const int* xidx, int64_t ld, const float* base, const int* bidx, int64_t bld,
                      float* y, double scale, int nshots) {
    constexpr int wpb = 4;
    constexpr size_t smem = wpb * CouplingShots::warp_bytes<SH>();
    auto kern = coupling_shots_kernel<SH, OWN>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int64_t grp = (c->n_elem + 32 / SH - 1) / (32 / SH);
    // two blocks an SM are resident (21 KB a warp): several rounds of them even out the tail
    const int64_t blocks = std::min<int64_t>((grp + wpb - 1) / wpb, (int64_t)c->n_sm * 8);
    kern<<<(unsigned)blocks, 32 * wpb, smem, c->stream>>>(c->n_elem, c->d_adj, c->d_Ke32, c->d_Kf32, c->d_rhoJ32, c->d_rt, x, xidx,
                                                         ld, base, bidx, bld, y, scale, nshots, c->nvel);
    note_launch(c);
    return cudaGetLastError();
}

bool coupling_shots_applies(const stdg_ctx* c, int nshots, const float* x, int64_t ld, const float* base, int64_t bld,
                            const float* y) {
    auto al = [](const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    return c->dim == 2 && c->Nphi == 6 && c->Ng == 3 && nshots >= 2 && c->d_Kf32 && al(x) && al(base) && al(y) && ld % 4 == 0 &&
           bld % 4 == 0;
}

cudaError_t launch_coupling_shots(stdg_ctx* c, const float* x, const int* xidx, int64_t ld, const float* base, const int* bidx,
                                  int64_t bld, float* y, double scale, int nshots) {
#define STDG_SH(SH_)                                                                                     \
    return base ? go<SH_, false>(c, x, xidx, ld, base, bidx, bld, y, scale, nshots)                      \
                : go<SH_, true>(c, x, xidx, ld, nullptr, nullptr, 0, y, scale, nshots)
    // the fewest lanes per element that waste no more lanes on the last chunk than a wider one
    const int pad8 = (nshots + 7) / 8 * 8, pad16 = (nshots + 15) / 16 * 16, pad32 = (nshots + 31) / 32 * 32;
    if (pad32 == pad8) { STDG_SH(32); }
    if (pad16 == pad8) { STDG_SH(16); }
    STDG_SH(8);
#undef STDG_SH
}

}  // namespace stdg
