// The stage multipliers of the double precision inverse column passes, against the exact roots of unity: prints the
// largest distance over every stage of every pass length, in units of 2^-53.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "fft_core.cuh"

using namespace pa;
using ld = long double;

// exp(-2 pi i e / n): the angle reduced exactly, by integers, before it is taken
static void exact(uint64_t e, uint64_t n, ld *c, ld *s) {
    const ld a = 2 * acosl(-1.0L) * ((ld)(e % n) / (ld)n);
    *c = cosl(a);
    *s = -sinl(a);
}
static double2 rounded(uint64_t e, uint64_t n) {
    ld c, s;
    exact(e, n, &c, &s);
    return {(double)c, (double)s};
}

// Stage I of a column of LEN values in a pass of stride S: the multiplier of row r is
// w_{LEN S}^{(R / 2^(l+1)) P (S j + u)} w_{2^(l+1)}^p for the row's level l and position p.
template <int LEN, int I> ld stage_error(uint32_t S) {
    using M = StageMap<double, LEN, 8, I>;
    constexpr StagePlan plan = Plan<double, LEN, 8>::p;
    constexpr int R = M::R;
    const StageRow row = plan.inv[I];
    std::vector<double2> st(plan.total);
    for (int r = 0; r < row.rows; ++r)
        for (int j = 0; j < plan.s[I]; ++j)
            st[row.off + (row.rows == 1 ? j : 2 * (r / 2 * plan.s[I] + j) + r % 2)] =
                rounded(stage_exponent(R, plan.s[I], r, j, LEN, Rows::DOUBLE), LEN);
    const int first = first_col_table(plan, I, Rows::DOUBLE), count = stage_col_tables(R, Rows::DOUBLE);
    const uint64_t n = (uint64_t)LEN * S;
    ld worst = 0;
    for (uint32_t u = 0; u < S; u += 1 + u * 7 % 13) {
        double2 hu[8];
        for (int l = 0; l < count; ++l) hu[l] = rounded(col_exponent(plan, first + l, Rows::DOUBLE) * u, n);
        for (uint32_t t = 0; t < (uint32_t)M::threads; ++t) {
            for (int g = 0; g < M::groups; ++g) {
                double2 m[level_rows(R)];
                col_multipliers<double, LEN, 8, I>(t, g, st.data(), hu, m);
                for (int r = 0; r < level_rows(R); ++r) {
                    const int l = row_level(r);
                    const uint64_t k = (uint64_t)(R >> (l + 1)) * plan.P[I] * ((uint64_t)S * M::offset(t, g) + u);
                    ld c, s;
                    exact(k + (uint64_t)row_pos(r) * (n >> (l + 1)), n, &c, &s);
                    worst = std::max(worst, hypotl(m[r].x - c, m[r].y - s));
                }
            }
        }
    }
    return worst * 0x1p53L;
}
template <int LEN, int I = 0> ld length_error(uint32_t S) {
    if constexpr (I < Plan<double, LEN, 8>::n) {
        return std::max(stage_error<LEN, I>(S), length_error<LEN, I + 1>(S));
    } else {
        return 0;
    }
}

int main() {
    for (uint32_t S : {64u, 384u, 2304u})
        std::printf("%.3Lf %.3Lf %.3Lf %.3Lf %.3Lf\n", length_error<64>(S), length_error<128>(S), length_error<256>(S),
                    length_error<512>(S), length_error<1024>(S));
}
