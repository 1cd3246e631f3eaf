// Three-part FP32 sums (tfde_sum3.cuh) against exact sums and against FP64
// sums in the same tree: butterflies over 32 lanes, then eight warps.  Values
// as the Gram-Schmidt sweeps close them (a Kahan sum and its correction), of
// one size, of mixed sizes, and cancelling.  Prints the worst errors relative
// to the sum of magnitudes; exit status 1 when one exceeds 2^-53.
#include <cmath>
#include <cstdio>
#include <random>

#include "tfde_sum3.cuh"

using tfde::Sum3;

template <typename T>
T tree(T (&v)[8][32]) {
    for (int w = 0; w < 8; ++w)
        for (int off = 16; off > 0; off >>= 1)
            for (int l = 0; l < off; ++l) v[w][l] += v[w][l + off];
    for (int w = 1; w < 8; ++w) v[0][0] += v[w][0];
    return v[0][0];
}

int main() {
    std::mt19937_64 g(7);
    std::normal_distribution<float> nd;
    double worst = 0.0, worst64 = 0.0;
    for (int it = 0; it < 60000; ++it) {
        Sum3 a[8][32];
        double b[8][32];
        __float128 exact = 0, mag = 0;
        for (int i = 0; i < 256; ++i) {
            Sum3& t = a[i / 32][i % 32];
            const int mode = it % 3;
            t.hi = std::ldexp(nd(g), mode == 1 ? (int)(g() % 40) - 20 : 0);
            t.mid = std::ldexp(nd(g), std::ilogb(t.hi) - 25);
            if (mode == 2 && i % 2) {   // the value before it, nearly cancelled
                t.hi = -a[i / 32][i % 32 - 1].hi;
            }
            b[i / 32][i % 32] = (double)t.hi + (double)t.mid;
            exact += (__float128)t.hi + (__float128)t.mid;
            mag += fabsl((long double)t.hi);
        }
        const double e = (double)((__float128)tree(a).value() - exact), e64 = (double)((__float128)tree(b) - exact);
        // the rounding of the result to a double is not the sum's
        const double half = 0.5 * (std::nextafter(std::fabs((double)exact), INFINITY) - std::fabs((double)exact));
        worst = std::fmax(worst, std::fmax(0.0, std::fabs(e) - half) / (double)mag);
        worst64 = std::fmax(worst64, std::fabs(e64) / (double)mag);
    }
    // 53 bits between the largest and the smallest value: exact in FP64 in any order
    Sum3 s;
    const float v[5] = {0x1p40f, 0x1p14f, 0x1p-12f, -0x1p14f, -0x1p40f};
    for (float x : v) {
        Sum3 t;
        t.hi = x;
        s += t;
    }
    Sum3 inf;
    for (float x : {1.f, INFINITY, -2.f}) {
        Sum3 t;
        t.hi = x;
        inf += t;
    }
    std::printf("three-part %.3g, FP64 %.3g, cancelled %a\n", worst, worst64, s.value());
    return !(worst <= 0x1p-53 && worst <= worst64 && s.value() == 0x1p-12 && inf.value() == INFINITY);
}
