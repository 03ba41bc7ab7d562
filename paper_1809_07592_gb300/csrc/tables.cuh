// tables.cuh -- twiddle tables of a transform: which entries a plan needs, where they sit,
// and how a stage reads them.
//
// Every entry is a power w_L^e of the transform's root, rounded once from its exact value,
// and every table is laid out in the order the reading threads need it, so a warp's
// lookups are whole 128-byte lines. (The passes used to gather from one table of powers:
// on rows of 256 values those gathers were 150 of the 271 shared-memory/L1 wavefronts a
// warp of the first pass needs.) Three kinds:
//   hi, lo       w_L^e = hi[e >> B] * lo[e mod 2^B], for single powers at any e;
//   stage tables (one per pass length): the multipliers of every in-CTA butterfly stage
//                (stage_list gives the stages, stage_exponent what each row holds);
//   pass tables  (one set per strided pass): w^{k u} for output k = tq + s*TC of column
//                u = blk*COLS + col as a[tq][blk] * c[tq][col] * g[u]^s.
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

// Stage plan of a Stockham FFT of length LEN = RO * 2^k2 (RO odd: 1, 3, 5 or 9)
// with E values per thread (TC = LEN / E threads per column). Radices:
//   forward  [RC], R0, E, ..., E        inverse  E, ..., E, R0, [RC]
// so the forward's output distribution over threads equals the inverse's input
// distribution (the two chain in registers). An odd stage exists only in
// transforms that read their input from, and write their output to, memory
// (the innermost pass), because its E / RO groups per thread do not divide. It
// absorbs the radix-r0 stage when r0 < E and the composite radix RC = RO * r0
// stays within a register budget.
struct StageShape {
    int RO, K2, q, r0, TC, R0C, RC;
    bool fold;
};
__host__ __device__ constexpr StageShape stage_shape(int len, int E) {
    StageShape s{};
    s.RO = odd_part(len);
    s.K2 = len / s.RO;
    const int k = ilog2(s.K2), e = ilog2(E);
    s.q = (k + e - 1) / e;  // power-of-two stages
    s.r0 = 1 << (k - (s.q - 1) * e);
    s.TC = len / E;
    s.fold = s.RO > 1 && s.r0 < E && s.RO * s.r0 <= kMaxCompositeRadix;
    s.R0C = s.fold ? s.r0 : 1;
    s.RC = s.RO * s.R0C;
    return s;
}

// The twiddled stages of one pass length: radix R at span P reads `rows` multipliers per
// butterfly k < P. Rows are stored in pairs, entry (row, k) at off + 2*((row/2)*P + k) + row%2,
// so that one 16-byte load of single-precision values brings two multipliers.
struct StageRow {
    int R, P, rows, off;
};
constexpr int kMaxStages = 6;
struct StageList {
    StageRow fwd[kMaxStages];  // power-of-two stage S of the forward transform (span 1 stages have no rows)
    StageRow inv[kMaxStages];  // power-of-two stage S of the inverse transform
    StageRow odd;              // the inverse transform's odd stage
    int total;                 // entries
};

// Rows of a radix-R power-of-two stage. Complex arithmetic: the distinct multipliers of the
// log2 R butterfly levels (dft_tw in fft_core.cuh); the exact transform: w^r, r = 1 .. R-1.
__host__ __device__ constexpr int stage_rows(int R, bool complex_) { return complex_ ? R / 2 : R - 1; }
// Rows of the odd stage of radix RO * R0: w^{R0 n1}, then the levels of a radix-R0 stage per k1 < RO.
__host__ __device__ constexpr int odd_rows(int RO, int R0) { return RO - 1 + RO * (R0 / 2); }

__host__ __device__ constexpr StageList stage_list(int len, int E, bool complex_) {
    StageList l{};
    const StageShape s = stage_shape(len, E);
    int off = 0;
    int P = s.RO > 1 ? s.RC : 1;
    for (int S = s.fold ? 1 : 0; S < s.q; ++S) {
        const int R = S == 0 ? s.r0 : E;
        const int rows = P > 1 ? stage_rows(R, complex_) : 0;
        l.fwd[S] = StageRow{R, P, rows, off};
        off += (rows + 1) / 2 * 2 * P;
        P *= R;
    }
    P = 1;
    for (int S = 0; S < (s.fold ? s.q - 1 : s.q); ++S) {
        const int R = S == s.q - 1 ? s.r0 : E;
        const int rows = P > 1 ? stage_rows(R, complex_) : 0;
        l.inv[S] = StageRow{R, P, rows, off};
        off += (rows + 1) / 2 * 2 * P;
        P *= R;
    }
    if (s.RO > 1) {
        const int K = len / s.RC, rows = odd_rows(s.RO, s.R0C);
        l.odd = StageRow{s.RC, K, rows, off};
        off += (rows + 1) / 2 * 2 * K;
    }
    l.total = off;
    return l;
}

// Level and position of row `row` of a complex radix-R stage: level l >= 0 has rows
// (l == 0: row 0; else rows 2^(l-1) .. 2^l - 1, p = row - 2^(l-1)).
__host__ __device__ constexpr int row_level(int row) { return row == 0 ? 0 : ilog2(row) + 1; }
__host__ __device__ constexpr int row_pos(int row) { return row == 0 ? 0 : row - (1 << ilog2(row)); }

// Exponent e (of w_L) held by row `row` of butterfly k of the stage `s` (pass length len).
__host__ __device__ inline uint64_t stage_exponent(const StageRow &s, int row, uint32_t k, uint64_t L, bool complex_) {
    const uint64_t unit = L / ((uint64_t)s.R * s.P);  // w_{R P} = w_L^unit
    if (!complex_) return (uint64_t)(row + 1) * k * unit;
    const int l = row_level(row);
    return (uint64_t)(s.R >> (l + 1)) * k * unit + (uint64_t)row_pos(row) * (L >> (l + 1));
}
__host__ __device__ inline uint64_t odd_exponent(const StageRow &s, int RO, int R0, int row, uint32_t k, uint64_t L) {
    const uint64_t unit = L / ((uint64_t)s.R * s.P);
    if (row < RO - 1) return (uint64_t)R0 * (row + 1) * k * unit;
    const int t = row - (RO - 1), k1 = t % RO, r = t / RO;  // level row r of the radix-R0 stage of k1
    const int l = row_level(r);
    return (uint64_t)(R0 >> (l + 1)) * ((uint64_t)k * unit + (uint64_t)k1 * (L / s.R)) +
           (uint64_t)row_pos(r) * (L >> (l + 1));
}

// Where every table of one transform sits in its block of memory (offsets in elements).
struct PassShape {
    uint32_t tc = 0, cols = 0;  // threads per column, columns per CTA
    uint64_t stride = 0;        // S: distance of a column's elements
    uint64_t a = 0, c = 0, g = 0;      // forward pass tables
    uint64_t ai = 0, ci = 0, gi = 0;   // inverse ones (the exact transform; else the same)
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
