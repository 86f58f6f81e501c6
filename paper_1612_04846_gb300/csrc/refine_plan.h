// The plan of the iterative refinement, for host and device code.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define BURA_HD __host__ __device__ __forceinline__
#else
#define BURA_HD inline
#endif

namespace bura {

constexpr int kPlanPowers = 8;  // step counts that plan_steps finds by multiplication

// The number of steps in which a relative reduction t of the residual is reached when one step is asked for a factor
// inner_rtol at most: n = ceil(log t / log inner_rtol - 1e-9), at least 1 and at most 2^31 - 1 (0 <= t < 1, 0 < inner_rtol
// < 1).  slack = inner_rtol^1e-9 and log_rtol = log(inner_rtol) are the caller's constants.  Plans of up to kPlanPowers
// steps (any t above 1e-40 with the default 1e-5) compare t with the powers of inner_rtol, because an FP64 logarithm on
// GB300 is a chain of some thousand SM clocks; the count grows without bound as inner_rtol approaches 1, so longer plans
// take the logarithm.
BURA_HD double plan_steps(double t, double inner_rtol, double slack, double log_rtol) {
    double r = inner_rtol;
    for (int n = 1; n <= kPlanPowers; ++n) {
        if (!(t < r * slack)) return n;
        r *= inner_rtol;
    }
    return fmin(fmax(ceil(log(t) / log_rtol - 1e-9), kPlanPowers + 1.0), 2147483647.0);
}

}  // namespace bura
