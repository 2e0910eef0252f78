// FP32 sums that keep what rounding drops.  The assembled couplings sum d N_phi products per neighbour,
// several times the length of the face form's chains, so plain FP32 totals had up to a third more error.
// Short chains join a total whose rounding errors are summed beside it (Kahan 1965; Neumaier's
// arrangement, in which the total itself is the plain sum: four additions a join as in Kahan's, but an
// infinite total stays infinite instead of turning into Inf - Inf).
// Plain C++ for the host as well, so that the arithmetic can be tested without a GPU.
#pragma once

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

}  // namespace stdg
