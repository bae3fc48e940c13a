// Host-side driver for the fixed-point separations of the FP64 real space.  Reads lines
//   rc L x0 y0 z0 x1 y1 z1   (hexadecimal floats; the second particle's x moved by -L first)
// and prints the unit's exponent, the three separations and r^2 in units, and the cutoff's square.
#include <cstdio>
#include <cstring>

#include "../../paper_2110_14362_gb300/csrc/rbe_pair64.cuh"

using namespace rbe;

static unsigned long long bits(double x)
{
    unsigned long long b;
    std::memcpy(&b, &x, 8);
    return b;
}

int main()
{
    double v[8];
    for (;;) {
        for (double& x : v)
            if (std::scanf("%la", &x) != 1) return 0;
        const PairUnit u = pair_unit(v[0], 0);
        long long d[3];
        for (int t = 0; t < 3; ++t) d[t] = (long long)(pair_fixed(bits(v[5 + t]), u.s) - pair_fixed(bits(v[2 + t]), u.s));
        d[0] = (long long)((unsigned long long)d[0] - pair_fixed(bits(v[1]), u.s));
        std::printf("%d %lld %lld %lld %llu %llu\n", u.s, d[0], d[1], d[2], pair_r2(d[0], d[1], d[2]), u.rc2);
    }
}
