// Host-side driver for the 64-bit fixed-point arithmetic of the FP64 path.  Reads commands from stdin:
//   T p (hex)       -> sine and cosine of the phase p 2^-64 revolutions, each as an integer in units of
//                      2^-30, the remainder as a float and the remainder in units of 2^-54
//   F r l           -> round(r / l 2^64) mod 2^64
//   M h l b         -> (h + l 2^-24) b 2^-30 for integers h, l and b (0 <= b < 2^60)
//   Q q e           -> |q| as a fraction of 2^(e + 1), in units of 2^-55
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
    std::vector<TrigEntry> tab(kTrigN);
    for (int i = 0; i < kTrigN; ++i) tab[i] = trig_entry(i);
    char op;
    while (std::scanf(" %c", &op) == 1) {
        if (op == 'T') {
            unsigned long long p;
            if (std::scanf("%llx", &p) != 1) return 1;
            const Frac f = frac_of(p);
            const uint32_t hi = (uint32_t)f.hi + kPhaseStart;
            const PhaseX x = phase_x(hi, f.lo);
            const TrigEntry e = tab[hi >> 21];
            const TrigLow w = trig_low(e);
            const float sf = fx_i2f(e.sa), cf = fx_i2f(e.ca);
            int sh, ch;
            float sl, cl;
            trig_value<1>(e.sa, sf, w.s, cf, w.c, x, sh, sl);
            trig_value<-1>(e.ca, cf, w.c, sf, w.s, x, ch, cl);
            std::printf("%d %.17g %d %d %.17g %d\n", sh, (double)trig_low_f(e.sr, sl), trig_low_i(e.sr, sl), ch,
                        (double)trig_low_f(e.cr, cl), trig_low_i(e.cr, cl));
        } else if (op == 'F') {
            double r, l;
            if (std::scanf("%lf %lf", &r, &l) != 2) return 1;
            std::printf("%llu\n", fixed_frac64(bits(r), fix_scale64(l, 1.0 / l)));
        } else if (op == 'M') {
            int h, l;
            unsigned long long b;
            if (std::scanf("%d %d %llu", &h, &l, &b) != 3) return 1;
            const unsigned long long c = b + (1ull << 29);
            std::printf("%lld\n", (long long)(mul_fix(h, l, (int)(c >> 30), (int)(c & 0x3FFFFFFFull) - (1 << 29)) - kMulBias));
        } else if (op == 'Q') {
            double q;
            int e;
            if (std::scanf("%lf %d", &q, &e) != 2) return 1;
            std::printf("%llu\n", fix_magnitude(bits(q), e + 1023));
        }
    }
    return 0;
}
