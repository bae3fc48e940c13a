// Host-side driver for the range of the FP64 real space's tables.  Reads from stdin lines
//   alpha rc sigma eps r2 ...   (r2 values to the end of the line)
// and prints for each r2 the Coulomb and the Lennard-Jones energy of the table, or "direct" where the pair kernels
// evaluate the pair directly.
#include <cmath>
#include <cstdio>
#include <iostream>
#include <sstream>
#include <string>
#include <vector>

#include "../../paper_2110_14362_gb300/csrc/rbe_pair64.cuh"

using namespace rbe;

int main()
{
    std::string line;
    while (std::getline(std::cin, line)) {
        std::istringstream in(line);
        double alpha, rc, sigma, eps, u;
        in >> alpha >> rc >> sigma >> eps;
        const int top = std::ilogb(rc * rc) + 1;
        const bool fits = eps == 0.0 || pair_lj_fits(sigma * sigma, 24.0 * eps, top);
        const int segs = fits ? pair_segs(alpha, top) : 0;
        std::vector<PairWord> t(kPairTabBytes / sizeof(PairWord));
        for (int i = 0; i < kPairSegs; ++i) pair_segment(t.data(), i, top, alpha, sigma * sigma, 24.0 * eps, 4.0 * eps);
        while (in >> u) {
            const PairUnit unit = pair_unit(rc, top);
            const PairArg a = pair_arg((unsigned long long)std::ldexp(u, 2 * unit.s - 64), unit.e, unit.base);
            if ((unsigned)a.seg >= (unsigned)segs) {
                std::printf("direct\n");
                continue;
            }
            double f;
            FF e, l, q;
            pair_eval<0>(t.data(), a, f, q, e);
            pair_eval<1>(t.data(), a, f, q, l);
            std::printf("%.17g %.17g\n", (double)e.h + (double)e.l, (double)l.h + (double)l.l);
        }
    }
    return 0;
}
