// Device-side state of the Krylov solvers and the reductions that their kernels share (solver.cu,
// cg_fused.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "compensated.h"

namespace stdg {

constexpr int kMaxRestart = 64;
constexpr int kRedThreads = 256;
constexpr int kFinThreads = 1024;   // single-block reduction / control kernels
constexpr int kDotChunk = 16;       // basis vectors per pass of the multi-dot kernels
constexpr int kDotLoads = 8;        // basis vectors whose values a thread has in flight at once

// Krylov state of one shot
struct ShotScalars {
    double bnorm, tol_abs;
    double rr, pq, alpha, beta;                   // CG
    double gbeta, resid;                          // GMRES
    double hcol[kMaxRestart + 2], hpass[kMaxRestart + 2];
    double H[(kMaxRestart + 1) * kMaxRestart];
    double cs[kMaxRestart], sn[kMaxRestart], g[kMaxRestart + 1], y[kMaxRestart];
    double red[3];                                // reduced sums handed between warps
    double vscale;                                // 1 / ||w||, the scale of the next basis vector
    int jj;            // basis columns this shot uses in the current cycle
    int active;        // still iterating in the current cycle / CG solve
    int reorth;        // this Arnoldi step needs the second Gram-Schmidt pass
    int converged, zero_x;                        // zero_x: b_s = 0, so x_s = 0
    // FP64 refinement level (mixed precision)
    double ir_bnorm, ir_tol_abs, ir_rnorm, ir_scale;
    int ir_conv, ir_zero;
};

// Recorded bodies whose executions are counted on the device: the kernels launched by a call are
// sum_i runs[i] * (kernels of body i), the second factor known from recording.
enum Body { kBodyStraight, kBodyIr, kBodyCycle, kBodyInner, kBodies };

// loop control shared by all shots
struct DevScalars {
    int j, iters, flag_outer, flag_inner, max_iters, m;
    int any;           // a shot still iterates (collected by the shots' last blocks)
    int ir_flag, ir_count, ir_max;
    // statistics, reset by the host before a batch of steps
    int st_total, st_max, st_refine, st_notconv, st_nonfinite;
    double st_final_rel, st_iters_sum;
    unsigned int runs[kBodies];       // executions of each recorded body since the last reset
};

// ---------------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------------
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double s = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    return s;   // valid in thread 0
}

// sum of p[0..n) by one warp; valid in every lane (read past L1: the values may come from other
// blocks of the same kernel)
__device__ __forceinline__ double warp_sum(const double* p, int n) {
    double v = 0;
    for (int i = threadIdx.x & 31; i < n; i += 32) v += __ldcg(p + i);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// partial sums of slot k, shot s: part + (k * ns + s) * G
__device__ __forceinline__ const double* slot(const double* part, int k, int s, int ns, int G) {
    return part + ((int64_t)k * ns + s) * G;
}

// Per-thread dot-product accumulator: FP64 for FP64 vectors; for FP32 vectors an error-free
// (TwoProduct + TwoSum) pair of floats, so FP32 inner products carry FP64-level accuracy
// without FP64 arithmetic (GB300's FP64 rate is 1/64 of FP32).
template <typename R> struct Acc;
template <> struct Acc<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ double value() const { return s; }
    __device__ __forceinline__ void plus_xor(const Acc& give, int o) { s += __shfl_xor_sync(0xffffffffu, give.s, o); }
};
template <> struct Acc<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float a, float b) {
        const float p = a * b;
        const float pe = fmaf(a, b, -p);
        const float t = s + p;
        const float z = t - s;
        const float te = (s - (t - z)) + (p - z);
        s = t;
        c += te + pe;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};
// FP32 accumulators in the tree over the lanes.  At two FP64 lanes an SM the conversions and FP64
// additions of 16 sums per thread took 5 us a block, more than the products; three floats lose no
// bit of an FP64 tree (compensated.h)
template <> struct Acc<Triple> {
    Triple t;
    __device__ __forceinline__ double value() const { return t.value(); }
    __device__ __forceinline__ void plus_xor(const Acc& give, int o) {
        t.plus(Triple{__shfl_xor_sync(0xffffffffu, give.t.s, o), __shfl_xor_sync(0xffffffffu, give.t.c, o),
                      __shfl_xor_sync(0xffffffffu, give.t.d, o)});
    }
};

// True in every thread of the block that arrives last of `total` (its reads then see what the
// others wrote before arriving).  Reductions finish in that block, in a fixed order, instead of in
// a single-block kernel of their own: a dependent launch costs 2-3 us and such a kernel took
// 8-13 us, five of them per GMRES iteration.  The counter is back at zero afterwards.
__device__ __forceinline__ bool last_block(unsigned* counter, unsigned total) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(counter, total - 1) == total - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Sums over the lanes of a warp of the 16 accumulators that each thread holds: the lanes halve their set at
// every exchange (16 exchanges instead of 80).  Lanes 2 i and 2 i + 1 end with the sum of accumulator
// lane_of16(lane).
__device__ __forceinline__ int lane_of16(int lane) {
    return (lane & 16 ? 8 : 0) + (lane & 8 ? 4 : 0) + (lane & 4 ? 2 : 0) + (lane & 2 ? 1 : 0);
}
template <typename R>
__device__ __forceinline__ double lane_sums16(Acc<R> (&v)[kDotChunk], int lane) {
#pragma unroll
    for (int o = 16, n = kDotChunk / 2; o > 1; o >>= 1, n >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const Acc<R> give = up ? v[i] : v[i + n];
            if (up) v[i] = v[i + n];
            v[i].plus_xor(give, o);
        }
    }
    v[0].plus_xor(v[0], 1);
    return v[0].value();
}
__device__ __forceinline__ double lane_sums16(Acc<float> (&v)[kDotChunk], int lane) {
    bool fits = true;
#pragma unroll
    for (int k = 0; k < kDotChunk; ++k) fits = fits && fabsf(v[k].s) <= kTripleMax;
    if (__all_sync(0xffffffffu, fits)) {
        Acc<Triple> t[kDotChunk];
#pragma unroll
        for (int k = 0; k < kDotChunk; ++k) t[k].t = Triple{v[k].s, v[k].c, 0.f};
        return lane_sums16<Triple>(t, lane);
    }
    Acc<double> t[kDotChunk];   // values that FP32 cannot add, infinities and NaN
#pragma unroll
    for (int k = 0; k < kDotChunk; ++k) t[k].s = v[k].value();
    return lane_sums16<double>(t, lane);
}

// Block-wide sums of the 16 accumulators: over the lanes, then FP64 sums over the warps through shared
// memory.  The sum of accumulator k is valid in thread k < 16.
template <typename R>
__device__ __forceinline__ double block_sum16(Acc<R> (&v)[kDotChunk]) {
    __shared__ double red[32][kDotChunk];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double mine = lane_sums16(v, lane);
    __syncthreads();
    if ((lane & 1) == 0) red[warp][lane_of16(lane)] = mine;
    __syncthreads();
    double s = 0;
    if (threadIdx.x < kDotChunk)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w][threadIdx.x];
    return s;
}

// Sum of one accumulator over the lanes of a warp.
template <typename R>
__device__ __forceinline__ double lane_sum1(Acc<R> v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v.plus_xor(v, o);
    return v.value();
}
__device__ __forceinline__ double lane_sum1(Acc<float> v) {
    if (__all_sync(0xffffffffu, fabsf(v.s) <= kTripleMax)) return lane_sum1<Triple>(Acc<Triple>{{v.s, v.c, 0.f}});
    return lane_sum1<double>(Acc<double>{v.value()});
}

// Block-wide sum of one accumulator; valid in thread 0.
template <typename R>
__device__ __forceinline__ double block_sum1(Acc<R> v) {
    __shared__ double red[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double mine = lane_sum1(v);
    __syncthreads();
    if (lane == 0) red[warp] = mine;
    __syncthreads();
    double s = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    return s;
}

__device__ __forceinline__ void set_cond(cudaGraphConditionalHandle h, int use, int v) {
    if (use) cudaGraphSetConditional(h, v ? 1u : 0u);
}

}  // namespace stdg
