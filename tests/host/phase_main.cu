// Host-side driver for the phases of the FP64 path.  Reads lines
//   mx my mz rx ry rz lx ly lz   (reals as hexadecimal floats)
// and prints sine and cosine of 2 pi m.(r / l), summed as the rho pass does, in units of 2^-30 (an integer and a
// remainder each), and the sine times 2^60 - 2^29 - 1 by the force pass's product.
#include <cstdio>
#include <cstring>

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
    int m[3];
    double r[3], l[3];
    while (std::scanf("%d %d %d %la %la %la %la %la %la", m, m + 1, m + 2, r, r + 1, r + 2, l, l + 1, l + 2) == 9) {
        Frac f[3];
        for (int t = 0; t < 3; ++t) f[t] = frac_of(fixed_frac64(bits(r[t]), fix_scale64(l[t], 1.0 / l[t])));
        uint32_t hi = kPhaseStart;
        for (int t = 0; t < 3; ++t) hi += (uint32_t)m[t] * (uint32_t)f[t].hi;
        float lo = fmaf((float)m[0], f[0].lo, fmaf((float)m[1], f[1].lo, (float)m[2] * f[2].lo));
        if (phase_is_wide(m[0], m[1], m[2])) phase_whole(hi, lo);
        const PhaseX x = phase_x(hi, lo);
        const TrigEntry e = trig_entry((int)(hi >> 21));
        const TrigLow w = trig_low(e);
        const float sf = fx_i2f(e.sa), cf = fx_i2f(e.ca);
        int sh, ch;
        float sl, cl;
        trig_value<1>(e.sa, sf, w.s, cf, w.c, x, sh, sl);
        trig_value<-1>(e.ca, cf, w.c, sf, w.s, x, ch, cl);
        const unsigned long long c = (1ull << 60) - 1;  // b = 2^60 - 2^29 - 1, as the force pass holds an amplitude
        const unsigned long long p = mul_fix(sh, trig_low_i(e.sr, sl), (int)(c >> 30), (int)(c & 0x3FFFFFFFull) - (1 << 29));
        std::printf("%d %.17g %d %.17g %lld\n", sh, (double)trig_low_f(e.sr, sl), ch, (double)trig_low_f(e.cr, cl),
                    (long long)(p - kMulBias));
    }
}
