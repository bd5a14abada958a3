// Acceptance test of the Gamma draws (also compiled for the host, where it is tested).
#pragma once
#include <math.h>

namespace bp {

// Marsaglia & Tsang (2000): accept d v with v = t^3, t = 1 + c g > 0, if log u < g^2/2 + d (1 - v + log v).
// Decided in FP32 where its two sides are further apart than FP32 can err, which spares two FP64
// logarithms in all but ~1e-3 of the draws; the decision is the same.  FP32 is within 1e-5 sqrt(d) of
// exact for |g| < 7 and t > 0.01; the error of log t grows as 1 / t below (shapes under 6 only).
__host__ __device__ inline bool gamma_accept(double g, double t, double c, double d, double u) {
    const float df = (float)d, margin = 2.0e-4f + 2.0e-4f * sqrtf(df);
    // g^2/2 + d (1 - v + log v) - log u with v = (1 + w)^3
    const float w = (float)(c * g), gf = (float)g;
    const float gap = fmaf(0.5f * gf, gf, df * (3.0f * log1pf(w) - w * fmaf(w, w + 3.0f, 3.0f))) - logf((float)u);
    if (t > 0.01 && fabsf(gap) > margin) return gap > 0.0f;
    const double v = t * t * t;
    return log(u) < 0.5 * g * g + d - d * v + d * log(v);
}

}  // namespace bp
