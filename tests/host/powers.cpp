// The powers that single precision stages form from their table entries, against the exact roots of unity: prints the
// largest distance over every forward stage of every pass and row length, in units of 2^-24.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "fft_core.cuh"

using namespace pa;

static double worst = 0;

static void exact(uint64_t e, uint64_t n, double *c, double *s) {
    const double a = 2 * acos(-1.0) * ((double)(e % n) / (double)n);
    *c = cos(a);
    *s = -sin(a);
}
// A radix-R stage whose table has P butterflies: entries of w = w_{R P}^k, level l's power is w^(R / 2^(l+1)).
template <int R> void stage(int P) {
    const uint64_t n = (uint64_t)R * P;
    for (int k = 0; k < P; ++k) {
        float2 w[2], pw[4];
        double c, s;
        for (int r = 0; r < stage_rows(R, Rows::SINGLE, false); ++r) {
            exact(stage_exponent(R, P, r, k, n, Rows::SINGLE), n, &c, &s);
            w[r] = {(float)c, (float)s};
        }
        entry_powers<float, R, true>(w, pw);
        for (int l = 0; l < ilog2(R); ++l) {
            exact((uint64_t)(R >> (l + 1)) * k, n, &c, &s);
            worst = std::max(worst, hypot(pw[l].x - c, pw[l].y - s));
        }
    }
}
static void any(int R, int P) {
    if (R == 2) stage<2>(P);
    if (R == 4) stage<4>(P);
    if (R == 8) stage<8>(P);
    if (R == 16) stage<16>(P);
}

int main() {
    for (int ro : {1, 3, 5, 9}) {
        for (int lg = 6; ro << lg <= 16384; ++lg) {
            const StagePlan p = stage_plan(ro << lg, 16, Rows::SINGLE);
            for (int i = ro > 1 ? 1 : 0; i < p.n; ++i) {
                any(p.R[i], p.P[i]);
            }
        }
    }
    std::printf("%.3f\n", worst * 0x1p24);
}
