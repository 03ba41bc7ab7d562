// quarter_turns against the exact angle: prints the largest error in units of 2^-55 of a quarter turn.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "fft_core.cuh"

int main() {
    double worst = 0;
    for (uint32_t ro : {1u, 3u, 5u, 9u}) {
        for (int lg = 12; (uint64_t)ro << lg <= 1u << 28; lg += 3) {
            const uint32_t L = ro << lg;
            const uint32_t step = L > 200000 ? L / 199999 : 1;
            for (uint32_t e = 0; e < L; e += step) {
                uint32_t q;
                const double x = pa::quarter_turns(e, L, &q);
                // 4 e / L = q + x: the remainder x L is an integer below 2^31 in exact arithmetic
                const long double off = (long double)x - (long double)((int64_t)4 * e - (int64_t)q * L) / (long double)L;
                worst = std::max(worst, (double)fabsl(off));
                if (q > 4 || fabs(x) > 0.5) worst = 1;
            }
        }
    }
    std::printf("%.3f\n", worst * 0x1p55);
}
