// The double-float radii, cosines and sines of the Gaussian draws (host code of ddmath.cuh) against long double: their errors
// have to stay well inside the 2^-39 that the rounding test of a draw allows for.  Random arguments, the smallest and largest
// ones and the neighbourhood of every octant.
#include <cmath>
#include <cstdio>
#include <random>

#include "ddmath.cuh"

using namespace pb;

static long double err(dd::F2 a, long double ref) { return fabsl(((long double)a.h + (long double)a.l) / ref - 1.0L); }

int main() {
    std::mt19937_64 gen(1);
    long double er = 0, ec = 0, es = 0;
    for (long i = 0; i < 1500000; ++i) {
        unsigned long long v = 2ull * (uint32_t)gen() + 1;
        if (i < 50000) v = 2ull * i + 1;
        else if (i < 100000) v = (1ull << 33) - 1 - 2ull * (i - 50000);
        else if (i < 400000) v = ((unsigned long long)(1 + i % 7) << 30) + 1 + 2 * ((i / 7) % 40000) - 40000;
        const long double q = 0.785398163397448309615660845819875721L;   // pi / 4
        er = fmaxl(er, err(dd::radius(v), sqrtl(-2.0L * logl((long double)v / 8589934592.0L))));
        const int o = (int)(v >> 30);
        const unsigned long long rem = v & 0x3FFFFFFFull, w = (o & 1) ? 0x40000000ull - rem : rem;
        long double c = cosl((long double)w / 1073741824.0L * q), s = sinl((long double)w / 1073741824.0L * q);
        if ((o + 1) & 2) std::swap(c, s);
        if (o >= 2 && o < 6) c = -c;
        if (o >= 4) s = -s;
        dd::F2 dc, ds;
        dd::sincos_turn(v, dc, ds);
        ec = fmaxl(ec, err(dc, c));
        es = fmaxl(es, err(ds, s));
    }
    std::printf("radius %.2Le cos %.2Le sin %.2Le\n", er, ec, es);
    return er < 4e-13L && ec < 1e-13L && es < 1e-13L ? 0 : 1;
}
