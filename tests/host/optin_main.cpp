// Host-side driver for the per-context requests of dynamic shared memory: prints the calls that reach the device for a
// sequence of launches "context kernel result" read from stdin, and the result that the launch sees.
#include <cstdio>

#include "../../paper_2110_14362_gb300/csrc/rbe_optin.h"

int main()
{
    rbe::SmemOptIn ctx[4];
    int c, kernel, result;
    while (std::scanf("%d %d %d", &c, &kernel, &result) == 3) {
        int calls = 0;
        const int got = ctx[c].once(kernel, [&] {
            ++calls;
            return result;
        });
        std::printf("%d %d\n", calls, got);
    }
}
