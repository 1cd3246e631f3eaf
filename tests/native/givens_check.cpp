// The Givens rotation of the GMRES cycles against extended precision: random
// values of every size and ratio, the ends of the double range, zeros.  Prints
// the worst errors in ulps; exit status 1 on a special value that is not what it
// should be, or beyond the bounds of the operations' roundings (u = 2^-53): the
// sum of squares (1 + 1/2) u, its root 3/4 u + u, a quotient u more, and u is
// between half an ulp and one.
#include <cstdio>
#include <limits>
#include <random>

#include "tfde_givens.h"

#ifdef __SIZEOF_FLOAT128__
typedef __float128 wide;
#else
typedef long double wide;   // 113 bits where the type above is missing
#endif

static wide root(wide x) {   // of a value near 1: two Newton steps from the double
    wide r = std::sqrt((double)x);
    for (int i = 0; i < 3; ++i) r = (r + x / r) / 2;
    return r;
}
static double ulps(double got, wide want) {
    const double w = std::fabs((double)want);
    const double u = std::nextafter(w, INFINITY) - w;
    return std::fabs((double)(((wide)got - want) / (wide)u));
}

int main() {
    std::mt19937_64 g(3);
    std::uniform_real_distribution<double> ud(0.5, 1.0);
    double wd = 0.0, wc = 0.0;
    bool ok = true;
    for (int it = 0; it < 2000000; ++it) {
        const int scale = it % 2 ? (int)(g() % 1800) - 900 : 0, ratio = (int)(g() % 60) - 30;
        const double a0 = (g() & 1 ? 1 : -1) * ud(g), b0 = std::ldexp(ud(g), ratio);   // hn >= 0
        const wide d0 = root((wide)a0 * a0 + (wide)b0 * b0);
        double c, s, d;
        tfde::givens_rotation(std::ldexp(a0, scale), std::ldexp(b0, scale), &c, &s, &d);
        wd = std::fmax(wd, ulps(std::ldexp(d, -scale), d0));
        wc = std::fmax(wc, std::fmax(ulps(c, a0 / d0), ulps(s, b0 / d0)));
    }
    auto is = [&](double a, double b, double ec, double es, double ed) {
        double c, s, d;
        tfde::givens_rotation(a, b, &c, &s, &d);
        ok = ok && c == ec && s == es && d == ed;
    };
    const double big = std::numeric_limits<double>::max(), tiny = std::numeric_limits<double>::denorm_min();
    is(0, 0, 1, 0, 0);
    is(-2, 0, -1, 0, 2);
    is(0, 3, 0, 1, 3);
    is(big, 0, 1, 0, big);
    is(0, tiny, 0, 1, tiny);
    is(0x1.8p-999, 0x1p-998, 0.6, 0.8, 0x1.4p-998);
    is(0x1.8p1000, 0x1p1001, 0.6, 0.8, 0x1.4p1001);
    double c, s, d;
    tfde::givens_rotation(NAN, 1.0, &c, &s, &d);
    ok = ok && c == 1.0 && s == 0.0 && std::isnan(d);
    std::printf("norm %.3f ulp, entries %.3f ulp, special values %s\n", wd, wc, ok ? "ok" : "WRONG");
    return !(ok && wd <= 1.75 && wc <= 2.75);
}
