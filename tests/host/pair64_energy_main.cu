// Host-side driver for the energies of the FP64 real space's tables as the pair kernels sum them.  Reads from stdin lines
//   alpha rc sigma eps r2 ...   (r2 values to the end of the line)
// and prints for each r2 the Coulomb and the Lennard-Jones energy, each as its constant term and the rest; or lines
//   R x y z   (separations in units)
// and prints their square sum as the pair kernels form it.
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
        if (line[0] == 'R') {
            long long x, y, z;
            if (std::sscanf(line.c_str(), "R %lld %lld %lld", &x, &y, &z) != 3) return 1;
            std::printf("%llu\n", pair_r2(x, y, z, kPairHalf));
            continue;
        }
        std::istringstream in(line);
        double alpha, rc, sigma, eps, u;
        in >> alpha >> rc >> sigma >> eps;
        const int top = std::ilogb(rc * rc) + 1;
        std::vector<PairWord> t(kPairTabBytes / sizeof(PairWord));
        for (int i = 0; i < kPairSegs; ++i) pair_segment(t.data(), i, top, alpha, sigma * sigma, 24.0 * eps, 4.0 * eps);
        while (in >> u) {
            const PairUnit unit = pair_unit(rc, top);
            const PairArg a = pair_arg((unsigned long long)std::ldexp(u, 2 * unit.s - 64), unit.e, unit.base);
            double f, ec, el;
            FF q, dc, dl;
            pair_eval<0>(t.data(), a, f, q, ec, dc);
            pair_eval<1>(t.data(), a, f, q, el, dl);
            std::printf("%.17g %.17g %.17g %.17g\n", ec, (double)dc.h + (double)dc.l, el, (double)dl.h + (double)dl.l);
        }
    }
    return 0;
}
