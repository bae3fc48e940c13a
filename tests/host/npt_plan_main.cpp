// Prints, per particle count of the arguments after the SM count: blocks of the FP32 pair kernel, of the
// flexible cell's FP64 pairs, of the FP64 pair kernels, of the finishing kernel, and the rows of the partial sums.
#include <cstdio>
#include <cstdlib>

#include "../../paper_2110_14362_gb300/csrc/rbe_npt_plan.h"

int main(int argc, char** argv)
{
    const int sms = std::atoi(argv[1]);
    for (int64_t N = std::atoll(argv[2]); N <= std::atoll(argv[3]); ++N)
        std::printf("%lld %d %d %d %d %lld\n", (long long)N, rbe::pair_blocks_of(N, sms, rbe::kPairBlocksPerSM),
                    rbe::pair_blocks_of(N, sms, rbe::kPairBlocksPerSM64), rbe::pair_blocks64_of(N, sms),
                    rbe::npt_blocks(N), (long long)rbe::npt_partial_rows(N, sms));
    return argc == 4 ? 0 : 1;
}
