// Block counts of the NPT step's pair kernels and the rows of its partial sums (host arithmetic only).
#pragma once

#include <algorithm>
#include <cstdint>

namespace rbe {

constexpr int kNptThreads = 256;
constexpr int kPairWarps = 8;        // k_pair: warps (particles in flight) per block
constexpr int kPairBlocksPerSM = 4;  // k_pair (FP32): resident blocks per SM the grid is sized for
constexpr int kPairBlocksPerSM64 = 2;  // the flexible cell's FP64 pairs: more registers per thread

// Grid of the pair search: enough blocks for one particle per warp, at most per_sm per SM (the warps stride
// over the rest).
inline int pair_blocks_of(int64_t N, int sms, int per_sm)
{
    const int64_t want = (N + kPairWarps - 1) / kPairWarps;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * per_sm));
}

// Blocks of the FP64 pair kernels: one per SM (its warps share the table), every SM from few particles on.
inline int pair_blocks64_of(int64_t N, int sms)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>(sms, (N + 3) / 4));
}

// Blocks of the finishing kernel (and of the other one-thread-per-particle kernels).
inline int npt_blocks(int64_t N) { return (int)std::max<int64_t>(1, (N + kNptThreads - 1) / kNptThreads); }

// Rows of the partial sums: the pair kernel's blocks, of either precision (below eight particles per SM the FP64
// kernels have more blocks than the FP32 ones), then the finishing kernel's.
inline int64_t npt_partial_rows(int64_t N, int sms)
{
    return (int64_t)std::max(pair_blocks_of(N, sms, kPairBlocksPerSM), pair_blocks64_of(N, sms)) + npt_blocks(N);
}

}  // namespace rbe
