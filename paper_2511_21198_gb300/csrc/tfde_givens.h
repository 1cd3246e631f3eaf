// Givens-rotated least-squares state of one GMRES cycle (FP64): the small
// (m+1) x m Hessenberg problem min || beta e_1 - H y || of the Arnoldi process
// (Sec. 3.2).  The host form is shared by the FP64 and the mixed-precision
// PGMRES; the device-side cycles take the same rotation.
#pragma once

#include <cmath>
#include <vector>

#include "tfde_pow2conv.cuh"

namespace tfde {

// The rotation (c, s) that takes (a, b) to (den, 0); the identity for (0, 0).
// The norm is formed between powers of two that keep its squares in range, with
// the larger one's square unrounded: less than 2 ulp off, as CUDA's hypot is, in
// fewer dependent operations: one thread runs them while a GMRES cycle waits (40 x
// 32 x 24, eight steps: 10.68 ms with hypot, 10.25 so).
TFDE_HD void givens_rotation(double a, double b, double* c, double* s, double* den) {
    const double m = fmax(fabs(a), fabs(b));
    int e = 0;
    if (m > 0.0 && m < INFINITY && !(m > 1e-140 && m < 1e140)) {
        frexp(m, &e);
        a = ldexp(a, -e);
        b = ldexp(b, -e);
    }
    const bool swap = fabs(a) < fabs(b);   // false for a NaN, which either place keeps
    const double hi = swap ? b : a, lo = swap ? a : b;
    const double d = sqrt(fma(hi, hi, lo * lo));
    *c = d > 0.0 ? a / d : 1.0;
    *s = d > 0.0 ? b / d : 0.0;
    *den = e ? ldexp(d, e) : d;
}

struct GivensLS {
    int m;
    std::vector<double> R, cs, sn, g;
    explicit GivensLS(int m_) : m(m_), R((size_t)(m_ + 1) * m_, 0.0), cs(m_), sn(m_), g(m_ + 1, 0.0) {}
    double& at(int i, int j) { return R[(size_t)i * m + j]; }
    // column j of the Hessenberg matrix (entries 0..j+1) -> rotated; returns |g_{j+1}|
    double add_column(int j, const double* h) {
        for (int i = 0; i <= j + 1; ++i) at(i, j) = h[i];
        for (int i = 0; i < j; ++i) {
            const double t = cs[i] * at(i, j) + sn[i] * at(i + 1, j);
            at(i + 1, j) = -sn[i] * at(i, j) + cs[i] * at(i + 1, j);
            at(i, j) = t;
        }
        givens_rotation(at(j, j), at(j + 1, j), &cs[j], &sn[j], &at(j, j));
        at(j + 1, j) = 0.0;
        g[j + 1] = -sn[j] * g[j];
        g[j] = cs[j] * g[j];
        return std::fabs(g[j + 1]);
    }
    void solve(int k, std::vector<double>& y) {
        y.assign(k, 0.0);
        for (int i = k - 1; i >= 0; --i) {
            double t = g[i];
            for (int j = i + 1; j < k; ++j) t -= at(i, j) * y[j];
            y[i] = t / at(i, i);
        }
    }
};

}  // namespace tfde
