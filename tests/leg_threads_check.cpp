// The CTAs that the batched legs are launched with fit what their kernels are
// compiled for, and are whole rows of lanes.
#include <cstdio>

#include "batch_tiles.h"

using namespace gmg::batch;

int main() {
    for (int n = 4; n <= 1024; n *= 2)
        for (int down = 0; down < 2; ++down) {
            const int th = leg_threads(n, down);
            if (th < 32 || th > kLegThreads || th % 32 || th % std::min(n / 4, 32)) {
                std::printf("n %d down %d: %d threads\n", n, down, th);
                return 1;
            }
        }
    return kLegThreads > 1024;
}
