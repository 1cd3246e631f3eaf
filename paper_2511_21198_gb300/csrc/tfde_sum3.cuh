// Sums of FP32 values in at least FP64 precision without FP64 arithmetic: an
// unevaluated sum hi + mid + lo of FP32 values, each far below the one before.
// GB300 issues FP64 additions and conversions at two lanes per clock and SM,
// FP32 additions at 128: an addition here is 20 of the latter.  The two leading
// parts are added without error (two-sum), so an addition errs by a few 2^-72
// of the largest value it has met; a pair of FP32 values errs by 2^-45 and an
// FP64 sum by 2^-53.
#pragma once

#include "tfde_pow2conv.cuh"

namespace tfde {

struct Sum3 {
    float hi = 0.f, mid = 0.f, lo = 0.f;

    // Knuth's two-sum: a + b = sum + the value returned, exactly
    TFDE_HD static float two_sum(float a, float b, float* sum) {
        const float s = a + b, t = s - a;
        *sum = s;
        return (a - (s - t)) + (b - t);
    }
    TFDE_HD void operator+=(const Sum3 o) {
        const float e = two_sum(hi, o.hi, &hi);
        const float f = two_sum(mid, o.mid, &mid);
        const float g = two_sum(mid, e, &mid);
        lo += o.lo + (f + g);
    }
    TFDE_HD void add(float v) {
        const float e = two_sum(hi, v, &hi);
        lo += two_sum(mid, e, &mid);
    }
    // an infinite or undefined sum is hi's (the other parts are NaN then)
    TFDE_HD double value() const {
        const double t = (double)hi;
        return t - t == 0.0 ? t + ((double)mid + (double)lo) : t;
    }
};

}  // namespace tfde
