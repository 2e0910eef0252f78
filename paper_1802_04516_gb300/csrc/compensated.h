// FP32 sums that keep what rounding drops.  The assembled couplings sum d N_phi products per neighbour,
// several times the length of the face form's chains, so plain FP32 totals had up to a third more error.
// Short chains join a total whose rounding errors are summed beside it (Kahan 1965; Neumaier's
// arrangement, in which the total itself is the plain sum: four additions a join as in Kahan's, but an
// infinite total stays infinite instead of turning into Inf - Inf).
// Plain C++ for the host as well, so that the arithmetic can be tested without a GPU.
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define STDG_HD __host__ __device__ __forceinline__
#else
#define STDG_HD inline
#endif

namespace stdg {

// total += sum; low collects what the additions round away
STDG_HD void join(float& total, float& low, float sum) {
    const float t = total + sum;
    low += sum - (t - total);
    total = t;
}

// the collected errors, to be added to the total last (none where the total is not finite)
STDG_HD float rest(float total, float low) { return total - total == 0.f ? low : 0.f; }

// Three floats whose sum is the value.  Additions carry the rounding errors of the two leading terms on
// (Knuth's two-sum), so that a tree over 32 lanes errs by some 2^-70 of the magnitudes: below an FP64 tree,
// without its arithmetic (an FP64 instruction takes 16 cycles of the SM).  The leading terms must not overflow
// in the sum: kTripleMax each for 32 of them.
constexpr float kTripleMax = 5.3e36f;
struct Triple {
    float s, c, d;
    STDG_HD void plus(const Triple& o) {
        const float a = s + o.s, av = a - s, ae = (s - (a - av)) + (o.s - av);
        const float b = c + o.c, bv = b - c, be = (c - (b - bv)) + (o.c - bv);
        const float g = b + ae, gv = g - b, ge = (b - (g - gv)) + (ae - gv);
        s = a;
        c = g;
        d += o.d + (be + ge);
    }
    STDG_HD double value() const { return (double)s + ((double)c + (double)d); }
};

// Sum of a row's products over the couplings, CH columns at a time.  FP64: a chain per neighbour, then their
// sum.  FP32: as the operator by itself (coupling_apply.h), chains of half as many columns joined with
// compensation; plain totals had 4% (2D p = 1) to 7% (3D p = 1) more error than the face form's.
template <typename R> struct RowSum;
template <> struct RowSum<double> {
    double total = 0.0, slot = 0.0;
    template <int CH, class F> STDG_HD void columns(const double (&kv)[CH], F&& x) {
        double sum = 0.0;
#pragma unroll
        for (int j = 0; j < CH; ++j) sum = fma(kv[j], x(j), sum);
        slot += sum;
    }
    STDG_HD void end_slot() { total += slot; slot = 0.0; }
    STDG_HD double scaled(double S) const { return S * total; }
};
template <> struct RowSum<float> {
    float total = 0.f, low = 0.f;
    template <int CH, class F> STDG_HD void columns(const float (&kv)[CH], F&& x) {
#pragma unroll
        for (int c = 0; c < CH; c += CH / 2) {
            float sum = 0.f;
#pragma unroll
            for (int j = c; j < c + CH / 2; ++j) sum = fmaf(kv[j], x(j), sum);
            join(total, low, sum);
        }
    }
    STDG_HD void end_slot() {}
    STDG_HD float scaled(float S) const { return fmaf(S, total, S * rest(total, low)); }
};

}  // namespace stdg
