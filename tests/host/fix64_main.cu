// Host-side driver for the 64-bit fixed-point arithmetic of the FP64 path.  Reads commands from stdin:
//   T p (hex)       -> sine and cosine of the phase p 2^-64 revolutions, in units of 2^-62
//   F r l           -> round(r / l 2^64) mod 2^64
//   M a b e         -> the product of the fixed-point value a 2^-62 (an integer) and |b| as a fraction of
//                      2^(e + 1), in units of 2^-57
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../paper_2110_14362_gb300/csrc/rbe_fix64.cuh"

using namespace rbe;

static unsigned long long bits(double x)
{
    unsigned long long b;
    std::memcpy(&b, &x, 8);
    return b;
}

int main()
{
    std::vector<TrigEntry> tab(kTrigLen);
    for (int i = 0; i < kTrigLen; ++i) tab[i] = trig_entry(i);
    char op;
    while (std::scanf(" %c", &op) == 1) {
        if (op == 'T') {
            unsigned long long p;
            if (std::scanf("%llx", &p) != 1) return 1;
            const unsigned long long t = p + kPhaseStart;
            const PhaseX x = phase_x((uint32_t)(t >> 32), (uint32_t)t);
            const TrigEntry s = tab[t >> 53], c = tab[(t >> 53) + kTrigN / 4];
            std::printf("%lld %lld\n", (long long)(trig_value<1>(s.v, s.h, s.l, c.h, c.l, x) - kMulBias),
                        (long long)(trig_value<-1>(c.v, c.h, c.l, s.h, s.l, x) - kMulBias));
        } else if (op == 'F') {
            double r, l;
            if (std::scanf("%lf %lf", &r, &l) != 2) return 1;
            std::printf("%llu\n", fixed_frac64(bits(r), fix_scale64(l, 1.0 / l)));
        } else if (op == 'M') {
            long long a;
            double b;
            int e;
            if (std::scanf("%lld %lf %d", &a, &b, &e) != 3) return 1;
            const unsigned long long u = (unsigned long long)a + kMulBias, v = fix_magnitude(bits(b), e + 1023) + kMulBias;
            std::printf("%lld\n", (long long)(mul_fix(fx_hi(u), fx_lo(u), fx_hi(v), fx_lo(v)) - kMulBias));
        }
    }
    return 0;
}
