// tables.cuh -- twiddle tables of a transform: which entries a plan needs, where they sit,
// and how a stage reads them.
//
// Every entry is a power w_L^e of the transform's root, rounded once from its exact value,
// and every table is laid out in the order the reading threads need it, so a warp's
// lookups are whole 128-byte lines. (The passes used to gather from one table of powers:
// on rows of 256 values those gathers were 150 of the 271 shared-memory/L1 wavefronts a
// warp of the first pass needs.) Three kinds:
//   hi, lo       w_L^e = hi[e >> B] * lo[e mod 2^B], for single powers at any e (the half-length form only);
//   stage tables (one per pass length): the multipliers of every in-CTA butterfly stage
//                (stage_plan gives the stages, stage_exponent what each row holds);
//   pass tables  (one set per strided pass): the pass twiddle w^{k u} of frequency k = f + s*TC in
//                column u = blk*COLS + col. Forward: a[f][blk] * c[f][col] * g[u]^s. Inverse, complex
//                arithmetic: it goes into the stages' multipliers (inv_col_stages in fft_core.cuh),
//                stage i needing w^{P_i u} (single precision) or its powers for every butterfly level
//                (double) beside its stage table: the column tables. The exact transform of
//                zq.cuh, whose multipliers cannot be multiplied with each other: a[f][u] and g[s][u].
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace pa {

__host__ __device__ constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v >> 1); }
__host__ __device__ constexpr int bitrev(int v, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((v >> b) & 1) << (bits - 1 - b);
    return r;
}
__host__ __device__ constexpr int odd_part(int v) { return (v & 1) ? v : odd_part(v >> 1); }
constexpr int kMaxCompositeRadix = 24;

// Stage plan of an in-CTA transform of length LEN = RO * 2^k2 (RO odd: 1, 3, 5 or 9) with E
// values per thread (TC = LEN / E threads per column). The forward transform runs stages
// 0 .. n-1 of radix R[i], the inverse n-1 .. 0; stage i combines, within blocks of N[i]
// elements (block P[i] of them), the R[i] elements s[i] = N[i] / R[i] apart, in place. Radices:
// [RC], r0, E, ..., E with r0 * E^(q-1) = 2^k2. The odd radix RC exists only in transforms that
// read their input from, and write their output to, memory (the innermost pass), because its
// groups do not divide a thread's E values; it absorbs the radix-r0 stage when r0 < E and
// RC = RO * r0 stays within a register budget.
constexpr int kMaxStages = 6;
struct StageRow {
    int rows, off;  // twiddle rows of a stage and where they start
};
struct StagePlan {
    int n, RO, R0C, RC, TC, r0;
    int R[kMaxStages], N[kMaxStages], s[kMaxStages], P[kMaxStages];
    // Twiddle tables: butterfly (block b, offset j) of forward stage i reads rows at index b < P[i],
    // of inverse stage i at index j < s[i]. Rows are stored in pairs, entry (row, x) at
    // off + 2*((row/2)*count + x) + row%2 (one row: off + x), so that a pair takes one wide
    // load; single precision's at off + row*count + x, most readers taking the first alone. rows = 0: no twiddles
    // (forward stage 0, inverse stage n-1).
    StageRow fwd[kMaxStages], inv[kMaxStages];
    int total;  // entries
};

// The three arithmetics' table rows. A complex stage needs the multipliers of its butterfly levels
// (dft_rows in fft_core.cuh), R/2 of a radix-R power-of-two stage, RO-1 + RO*R0/2 of an odd one.
// Double precision reads them all: its passes are bound by the FP64 pipe, the load path is idle. Single
// precision reads w alone and forms the others (squarings and constant turns): its innermost
// pass is bound by the load/store data path (78 % busy with all rows read, a 16-byte load costing four
// wavefronts whatever the addresses) and has multiply-add slots to spare. Its forward stages with R >= 8 also have a row of
// w^4, for the passes that need the powers closer to their roots (entry_powers in fft_core.cuh). The exact transforms
// read w^r, r = 1 .. R-1 (EXACT), or every level's multipliers, R-1 as well, no two of which are a free quarter
// turn apart (LEVELS).
enum class Rows { SINGLE, DOUBLE, EXACT, LEVELS };
__host__ __device__ constexpr bool is_complex(Rows kind) { return kind == Rows::SINGLE || kind == Rows::DOUBLE; }
__host__ __device__ constexpr int level_rows(int R) { return R / 2; }
__host__ __device__ constexpr int odd_level_rows(int RO, int R0) { return RO - 1 + RO * (R0 / 2); }
__host__ __device__ constexpr int stage_rows(int R, Rows kind, bool inverse) {
    return kind == Rows::SINGLE ? (R >= 8 && !inverse ? 2 : 1) : kind == Rows::DOUBLE ? level_rows(R) : R - 1;
}
__host__ __device__ constexpr int odd_rows(int RO, int R0, Rows kind) {
    return kind == Rows::SINGLE ? 1 : odd_level_rows(RO, R0);
}

// Entries of a stage's rows (whole pairs, except a single row; even, so that every table starts on a pair).
__host__ __device__ constexpr int row_entries(int rows, int count) {
    return rows == 1 ? (count + 1) / 2 * 2 : (rows + 1) / 2 * 2 * count;
}

__host__ __device__ constexpr StagePlan stage_plan(int len, int E, Rows kind) {
    StagePlan l{};
    l.RO = odd_part(len);
    const int k = ilog2(len / l.RO), e = ilog2(E);
    const int q = (k + e - 1) / e;  // power-of-two stages
    l.r0 = 1 << (k - (q - 1) * e);
    const bool fold = l.RO > 1 && l.r0 < E && l.RO * l.r0 <= kMaxCompositeRadix;
    l.R0C = fold ? l.r0 : 1;
    l.RC = l.RO * l.R0C;
    l.TC = len / E;
    if (l.RO > 1) l.R[l.n++] = l.RC;
    for (int S = fold ? 1 : 0; S < q; ++S) l.R[l.n++] = S == 0 ? l.r0 : E;
    int P = 1, off = 0;
    for (int i = 0; i < l.n; ++i) {
        l.P[i] = P;
        l.N[i] = len / P;
        l.s[i] = l.N[i] / l.R[i];
        const int rows = i == 0 ? 0 : stage_rows(l.R[i], kind, false);
        l.fwd[i] = StageRow{rows, off};
        off += row_entries(rows, P);
        P *= l.R[i];
    }
    for (int i = 0; i < l.n; ++i) {
        const int rows = i == l.n - 1 ? 0 : i == 0 && l.RO > 1 ? odd_rows(l.RO, l.R0C, kind) : stage_rows(l.R[i], kind, true);
        l.inv[i] = StageRow{rows, off};
        off += row_entries(rows, l.s[i]);
    }
    l.total = off;
    return l;
}

// Frequency of block b of stage i: b's digits, outermost first, are the output digits k_0, ...,
// k_{i-1} of the earlier stages, and the frequency is k_0 + R[0] (k_1 + R[1] (...)).
__host__ __device__ constexpr uint32_t block_freq(const StagePlan &l, int i, uint32_t b) {
    uint32_t f = 0;
    for (int t = i - 1; t >= 0; --t) {  // the last digit of b is k_{i-1}
        f += (b % (uint32_t)l.R[t]) * (uint32_t)l.P[t];
        b /= (uint32_t)l.R[t];
    }
    return f;
}
// Level and position of row `row` of a complex radix-R stage: level l >= 0 has rows
// (l == 0: row 0; else rows 2^(l-1) .. 2^l - 1, p = row - 2^(l-1)).
__host__ __device__ constexpr int row_level(int row) { return row == 0 ? 0 : ilog2(row) + 1; }
__host__ __device__ constexpr int row_pos(int row) { return row == 0 ? 0 : row - (1 << ilog2(row)); }

// Exponent e (of w_L) held by row `row` of a radix-R stage for the twiddle base w_{R P}^k.
__host__ __device__ inline uint64_t stage_exponent(int R, uint64_t P, int row, uint64_t k, uint64_t L, Rows kind) {
    const uint64_t unit = L / ((uint64_t)R * P);  // w_{R P} = w_L^unit
    if (kind == Rows::LEVELS) {  // level l: rows 2^l - 1 .., one per sub-transform p
        const int l = ilog2(row + 1), p = row + 1 - (1 << l);
        return (uint64_t)(R >> (l + 1)) * k * unit + (uint64_t)p * (L >> (l + 1));
    }
    if (kind == Rows::SINGLE) return (row ? 4 : 1) * k * unit;
    if (kind != Rows::DOUBLE) return (uint64_t)(row + 1) * k * unit;
    const int l = row_level(row);
    return (uint64_t)(R >> (l + 1)) * k * unit + (uint64_t)row_pos(row) * (L >> (l + 1));
}
__host__ __device__ inline uint64_t odd_exponent(int RO, int R0, uint64_t P, int row, uint64_t k, uint64_t L, Rows kind) {
    const uint64_t RC = (uint64_t)RO * R0, unit = L / (RC * P);
    if (kind == Rows::SINGLE) return k * unit;
    if (row < RO - 1) return (uint64_t)R0 * (row + 1) * k * unit;
    const int t = row - (RO - 1), k1 = t % RO, r = t / RO;  // level row r of the radix-R0 stage of k1
    const int l = row_level(r);
    return (uint64_t)(R0 >> (l + 1)) * (k * unit + (uint64_t)k1 * (L / RC)) + (uint64_t)row_pos(r) * (L >> (l + 1));
}

// e of L parts of a turn (e < L <= 2^28, 4 | L) as (q + x) quarter turns with |x| <= 1/2: integers reduce the angle, so that
// x, the only rounded number, is off by 2^-55 of a quarter turn at most. (e / L, near 1, was off by eight times that in angle
// for lengths with an odd factor.)
__host__ __device__ inline double quarter_turns(uint32_t e, uint32_t L, uint32_t *q) {
    *q = (4u * e + L / 2u) / L;
    return (double)((int32_t)(4u * e) - (int32_t)(*q * L)) / (double)L;
}

// Column tables (complex arithmetic): stage i has one (SINGLE, w^{P_i u}) or one per level l of its butterflies
// (DOUBLE, w^{(R_i / 2^(l+1)) P_i u}), stage after stage. The factor of u in table t's exponent is col_exponent.
__host__ __device__ constexpr int stage_col_tables(int R, Rows kind) { return kind == Rows::SINGLE ? 1 : ilog2(R); }
__host__ __device__ constexpr int first_col_table(const StagePlan &l, int i, Rows kind) {
    int t = 0;
    for (int s = 0; s < i; ++s) t += stage_col_tables(l.R[s], kind);
    return t;
}
__host__ __device__ constexpr int col_tables(const StagePlan &l, Rows kind) { return first_col_table(l, l.n, kind); }
__host__ __device__ constexpr uint64_t col_exponent(const StagePlan &l, int t, Rows kind) {
    int i = 0;
    while (t >= stage_col_tables(l.R[i], kind)) t -= stage_col_tables(l.R[i++], kind);
    return (uint64_t)l.P[i] * (kind == Rows::SINGLE ? 1u : (uint32_t)l.R[i] >> (t + 1));
}

// Where every table of one transform sits in its block of memory (offsets in elements).
struct PassShape {
    uint32_t tc = 0, cols = 0;  // threads per column, columns per CTA
    uint64_t stride = 0;        // S: distance of a column's elements
    uint64_t a = 0, c = 0, g = 0;      // forward pass tables
    uint64_t ai = 0, ci = 0, gi = 0;   // inverse ones (the exact transforms)
    uint64_t h = 0;                    // complex arithmetic: column tables of `stride` entries for the inverse stages
};
struct TwLayout {
    uint64_t L = 0;
    uint32_t B = 0;
    int len[3] = {0, 0, 0};  // pass lengths: first, middle strided (0: none), innermost
    int E = 0;
    uint64_t hi = 0, lo = 0, nhi = 0, nlo = 0;
    uint64_t st[3] = {0, 0, 0};
    PassShape pass[2];
    uint64_t total = 0;  // elements
};

}  // namespace pa
