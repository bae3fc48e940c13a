// Dynamic shared memory beyond 48 KB has to be asked for, kernel by kernel, on the device that launches it.  Each
// context asks for itself, at its first launch of a kernel: contexts of one process may be on several devices, and a
// request that failed is made again.
#pragma once

#include <cstdint>

namespace rbe {

// The kernels that ask (bits of SmemOptIn).
enum SmemKernel { kSmemRho64 = 0 /* + CHECK */, kSmemForce64 = 2 /* + 2 log2(slices) + CHECK */, kSmemPair64 = 10 /* + 2 list + diagonal */,
                  kSmemWaterPair = 14 };

struct SmemOptIn {
    uint32_t asked = 0;

    // ask() once per kernel, until it returns 0 (cudaSuccess); its result.
    template <typename Ask>
    auto once(int kernel, Ask ask) -> decltype(ask())
    {
        if (asked >> kernel & 1u) return {};
        const auto e = ask();
        if (e == decltype(ask()){}) asked |= 1u << kernel;
        return e;
    }
};

}  // namespace rbe
