// pa_kernels.cuh -- the pass kernels of the FFT Toeplitz hash.
//
// Index conventions for a transform of complex length L = L1 * L2 (two
// levels) or L1 * L2 * L3 (three levels). Element t of a length-L vector lives
// at offset t of its work slot; a pass at level j with transform length LEN and
// stride S treats the slot as blocks of LEN*S elements, each holding S
// interleaved columns of LEN elements (element a of column u at a*S + u).
//
//   forward level j (decimation in frequency, paper Algorithm 1's "row FFT
//   then twiddle W[i*j]"): X[k] = sum_a x[a] w_LEN^{a k}, then
//   X[k] *= w_{LEN*S}^{k u}, stored back at k*S + u.
//   inverse level j: x[k] *= w_{LEN*S}^{-k u}, then the unscaled inverse DFT.
//
// The innermost level (S = 1, contiguous) fuses the last forward step, the
// pointwise product with the cached seed spectrum (Eq. 4's FFT(V) . FFT(X))
// and the first inverse step. The seed spectrum already carries the 1/L of
// the inverse transform.
//
// Encoding (the value that is rounded): key bits x_j in {0,1}; seed bits
// enter as sigma = 1 - 2 s in {+1,-1} and are rotated so the wanted window of
// the linear convolution lands at positions 0..m-1:
//     r_i = sum_j sigma[i - j + n - 1] x_j = P - 2 c_i,
// where c_i = sum_j s[i-j+n-1] x_j is the GF(2) row count and P = popcount(x).
// So y_i = c_i mod 2 = rint((P - r_i)/2) mod 2, and since 4 | (P - P mod 4)
// only P mod 4 enters: y_i = rint(w_i) mod 2 with w_i = ((P mod 4) - r_i)/2.
// |r_i| grows like sqrt(n) instead of n, which keeps FP32 rounding far from
// the 0.5 cliff (the precision concern of the paper's Section 5).
#pragma once

#include "bulk.cuh"
#include "fft_core.cuh"
#include "pa_launch.h"

namespace pa {

// Resident CTAs requested per SM for a CTA of `threads` threads: enough for 1024
// threads, so the register allocation stays <= 64 per thread and at least two
// CTAs overlap their load, transform and store phases.
__host__ __device__ constexpr int min_blocks(int threads) { return threads >= 1024 ? 1 : (1024 / threads > 16 ? 16 : 1024 / threads); }
// The fused innermost passes ask for 512 resident threads per SM (<= 128 registers each; at most 16 CTAs).
// In single precision they ask for 768, at most 8 CTAs (more CTAs overlap their barrier and load phases), with at most 8
// bytes of spills. Rows of 5120 values (CTAs of 320 threads) ask for three CTAs and rows of 4608 (288 threads)
// for four. Over 2^25 values (us, k_middle alone): rows of 4096 122 (with 512 threads 139), 6144 133 (193), 2304 125 (135),
// 3072 120 (133); 5120 with two, three CTAs 140, 124, four took 32 pairs from 156 to 213; 4608 with three, four 125, 121.
// Asking for 1024 threads is faster on 2304, 2560, 3072 and 4096 (117, 114, 114, 114; 2560 takes 126 with 768) and on
// 8192 (176, 209 with 768), and the same on the shorter rows: not taken yet.
__host__ __device__ constexpr int min_blocks_inner(int threads, int elem_bytes = 16) {
    return elem_bytes > 8 ? (threads >= 512 ? 1 : (512 / threads > 16 ? 16 : 512 / threads))
                          : (threads >= 768 ? 1
                                            : threads == 288 ? 4
                                            : threads == 320 ? 3
                                                             : (768 / threads > 8 ? 8 : 768 / threads));
}

// The two-row kernels in single precision (double precision keeps the 512 threads of the rule above). The
// split kernel asks for 1024 threads: the 256-block uneven batch took 9.99 ms, with 768, 640 and 512
// threads 10.06, 10.25 and 10.47. By row length (2^25 values, us with 1024 and 768): 1280 117 and 131, 1536 115 and 121,
// 2304 125 and 158, 2560 123 and 150, 4096 128 and 158; 512 54 and 51, 640 82 and 79, 768 85 and 80, 1024 103 and 98, 2048
// 115 and 112, others alike. Rows of 384 to 2048 and 8192 values spill 24-112 bytes for it. The half-length kernel asks
// for 640: the 2^27-bit block took 1.179 ms, with 512 and 768 threads 1.210 and 1.190.
__host__ __device__ constexpr int min_blocks_split(int threads, int elem_bytes) {
    return elem_bytes > 8 ? min_blocks_inner(threads) : min_blocks(threads);
}
__host__ __device__ constexpr int min_blocks_real(int threads, int elem_bytes) {
    return elem_bytes > 8 ? min_blocks_inner(threads) : threads >= 640 ? 1 : 640 / threads > 16 ? 16 : 640 / threads;
}

// Rounding to the nearest integer (ties to even) by adding and subtracting
// 1.5 * 2^(mantissa bits): exact for |x| < 2^22 (float) / 2^51 (double); the
// integer's parity is the lowest bit of the sum's encoding.
template <typename T> struct Magic;
template <> struct Magic<float> {
    static constexpr float v = 12582912.0f, limit = 2097152.0f;
    static __device__ __forceinline__ float from_high(uint32_t hi) { return __uint_as_float(hi); }
};
template <> struct Magic<double> {
    static constexpr double v = 6755399441055744.0, limit = 1125899906842624.0;
    static __device__ __forceinline__ double from_high(uint32_t hi) { return __hiloint2double((int)hi, 0); }
};
__device__ __forceinline__ uint32_t low_bit(float x) { return __float_as_uint(x) & 1u; }
__device__ __forceinline__ uint32_t low_bit(double x) { return (uint32_t)__double_as_longlong(x) & 1u; }

// Encoding of inputs and decoding of outputs per arithmetic.
// Complex: key bits in the real (key 2p) and imaginary (key 2p+1) parts,
// seed as +-1; the decoded value is w = ((P mod 4) - r)/2 (see above).
// Zp: key 2p + 2^32 * key 2p+1 packed in one residue, seed as 0/1; the
// convolution counts c_a, c_b < 2^32 come out exactly as the low and high
// halves of the canonical residue.
template <typename T> struct Enc {
    using E = cx<T>;
    using M = T;  // margin accumulator
    // Bit 30 alone is the encoding of 2.0f (and of the high word of 2.0), so a shift and a mask
    // make a key bit the value 0 or 2, and one more of each a seed bit +-2. The spectra are
    // scaled back by kSpecScale: powers of two, so no rounding changes.
    static __device__ __forceinline__ uint32_t two_if(uint32_t x, int bit) {
        return (bit <= 30 ? x << (30 - bit) : x >> 1) & 0x40000000u;
    }
    static __device__ __forceinline__ T pm_two(uint32_t x, int bit, uint32_t in, int j) {
        return Magic<T>::from_high(two_if(in, j) | ((x << (31 - bit)) & 0x80000000u));
    }
    // bit j of x: real part, bit 16 + j: imaginary part (key a and key b, or a key's even and odd bits)
    static __device__ __forceinline__ E keys(uint32_t x, int j) {
        return Arith<T>::mk(Magic<T>::from_high(two_if(x, j)), Magic<T>::from_high(two_if(x, 16 + j)));
    }
    // bit j of x: key, bit 16 + j: seed; bit j of in: the position is inside the seed
    static __device__ __forceinline__ E key_seed(uint32_t x, uint32_t in, int j) {
        return Arith<T>::mk(Magic<T>::from_high(two_if(x, j)), pm_two(x, 16 + j, in, j));
    }
    // seed bits in both parts
    static __device__ __forceinline__ E seed(uint32_t x, uint32_t in_re, uint32_t in_im, int j) {
        return Arith<T>::mk(pm_two(x, j, in_re, j), pm_two(x, 16 + j, in_im, j));
    }
    // bits and margins of the two values carried by v (valid_b: the imaginary part's own range)
    static __device__ __forceinline__ void decode2(E v, uint32_t popa, uint32_t popb, bool valid_a, bool valid_b,
                                                   bool &bit_a, bool &bit_b, M &ma, M &mb) {
        const T wa = ((T)(popa & 3u) - v.x) * (T)0.5, wb = ((T)(popb & 3u) - v.y) * (T)0.5;
        const T fa = wa + Magic<T>::v, fb = wb + Magic<T>::v;  // rint via the 1.5*2^p addition
        bit_a = valid_a && low_bit(fa);
        bit_b = valid_b && low_bit(fb);
        // beyond the limit the parity is not resolvable: report a margin of 1 so the guard escalates
        if (valid_a) ma = fmax(ma, fabs(wa) < Magic<T>::limit ? fabs(wa - (fa - Magic<T>::v)) : (T)1);
        if (valid_b) mb = fmax(mb, fabs(wb) < Magic<T>::limit ? fabs(wb - (fb - Magic<T>::v)) : (T)1);
    }
};
template <> struct Enc<Zp> {
    using E = cx<Zp>;
    using M = float;
    static __device__ __forceinline__ E keys(uint32_t x, int j) {
        return (E)((x >> j) & 1u) | ((E)((x >> (16 + j)) & 1u) << 32);
    }
    // (the exact transform has no half-length packing and no key+seed form: its values are not complex)
    static __device__ __forceinline__ E seed(uint32_t x, uint32_t, uint32_t, int j) { return (E)((x >> j) & 1u); }
    static __device__ __forceinline__ void decode2(E v, uint32_t, uint32_t, bool valid_a, bool valid_b, bool &bit_a,
                                                   bool &bit_b, M &, M &) {
        bit_a = valid_a && (v & 1ull);
        bit_b = valid_b && ((v >> 32) & 1ull);
    }
};

template <> struct Enc<Zq> {
    using E = cx<Zq>;
    using M = float;
    static __device__ __forceinline__ E keys(uint32_t x, int j) { return make_uint2((x >> j) & 1u, (x >> (16 + j)) & 1u); }
    static __device__ __forceinline__ E seed(uint32_t x, uint32_t, uint32_t, int j) { return make_uint2((x >> j) & 1u, 0u); }
    static __device__ __forceinline__ void decode2(E v, uint32_t, uint32_t, bool valid_a, bool valid_b, bool &bit_a,
                                                   bool &bit_b, M &, M &) {
        bit_a = valid_a && (Arith<Zq>::canonical(v.x) & 1u);
        bit_b = valid_b && (Arith<Zq>::canonical(v.y) & 1u);
    }
};

// A value of the seed's spectrum as the product takes it.
template <typename T>
__device__ __forceinline__ cx<T> spectrum_value(cx<T> v) {
    if constexpr (std::is_same<T, Zq>::value) {
        return Arith<Zq>::multiplier(v);
    } else {
        return v;
    }
}

// Input bits of the level-1 forward passes. Thread (tq, col) of column block blk transforms the
// rows tq + j*TC, j < E, of column blk*COLS + col, whose bits lie E/32 of a row apart in memory:
// a CTA would touch LEN lines for LEN words of 16 bits each (32 wavefronts per load and warp). The
// bits are therefore transposed once, by k_key_bits and its kin (pa_prep.cu), into one 32-bit word per thread:
// bit j: the real part's bit of row j, bit 16 + j: the imaginary part's, word (blk, tq, col) of a
// slot in thread order, so a pass reads one coalesced word per thread and makes every element
// with two shift-and-mask instructions at constant positions.
// Position j of the row of register slot s (elem_of): row = tq + j*TC.
template <typename T, int LEN, int E>
constexpr int slot_pos(int s) {
    constexpr int r0 = Plan<T, LEN, E>::r0;
    return s / r0 + (s % r0) * (E / r0);
}

// Two per-thread counters reduced over the CTA (sum, or max when MAX): warp reductions into
// scratch (64 words of shared memory; cta_reduce_put), a barrier of the caller's, then warp 0
// over the warps' partial results (cta_reduce_get: the totals are valid in thread 0). The
// per-key counters of a batch (key popcounts, rounding margins) are accumulated with one
// atomic per key and CTA this way: one atomic per warp on the same few words from thousands
// of CTAs at once queues up in the memory system and measurably slows the whole pass.
template <bool MAX>
__device__ __forceinline__ void cta_reduce_put(uint32_t a, uint32_t b, uint32_t *scratch) {
    a = MAX ? __reduce_max_sync(0xffffffffu, a) : __reduce_add_sync(0xffffffffu, a);
    b = MAX ? __reduce_max_sync(0xffffffffu, b) : __reduce_add_sync(0xffffffffu, b);
    if ((threadIdx.x & 31) == 0) {
        scratch[threadIdx.x >> 5] = a;
        scratch[32 + (threadIdx.x >> 5)] = b;
    }
}
template <bool MAX>
__device__ __forceinline__ void cta_reduce_get(uint32_t &a, uint32_t &b, const uint32_t *scratch) {
    if (threadIdx.x >= 32) return;
    const uint32_t lane = threadIdx.x, nw = blockDim.x >> 5;
    a = lane < nw ? scratch[lane] : 0u;
    b = lane < nw ? scratch[32 + lane] : 0u;
    a = MAX ? __reduce_max_sync(0xffffffffu, a) : __reduce_add_sync(0xffffffffu, a);
    b = MAX ? __reduce_max_sync(0xffffffffu, b) : __reduce_add_sync(0xffffffffu, b);
}

// Single keys in half-length transforms: transform element t carries key bits 2t
// (real part) and 2t+1 (imaginary part). spread_bits moves the low 16 bits of x to the even positions.
__device__ __forceinline__ uint32_t spread_bits(uint32_t x) {
    x &= 0x0000FFFFu;
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}

// COLS bits of v starting at bit t0 (t0 % COLS == 0, so they sit in one word);
// bits at or past nbits read as 0.
template <int COLS>
__device__ __forceinline__ uint32_t aligned_bits(const uint64_t *v, uint64_t nbits, uint64_t t0) {
    if (t0 >= nbits) return 0u;
    uint32_t w = (uint32_t)(__ldg(v + (t0 >> 6)) >> (t0 & 63)) & ((1u << COLS) - 1u);
    const uint64_t left = nbits - t0;
    if (left < COLS) w &= (1u << left) - 1u;
    return w;
}

// cnt <= 32 bits of v starting at an arbitrary bit position pos; bits at or past nbits read as 0.
__device__ __forceinline__ uint32_t bits_at(const uint64_t *v, uint64_t nbits, uint64_t pos, uint32_t cnt) {
    if (pos >= nbits || cnt == 0) return 0u;
    const uint64_t q = pos >> 6;
    const uint32_t r = (uint32_t)(pos & 63);
    uint64_t x = __ldg(v + q) >> r;
    if (r + cnt > 64 && ((q + 1) << 6) < nbits) x |= __ldg(v + q + 1) << (64 - r);
    uint32_t w = (uint32_t)x & (cnt == 32 ? 0xffffffffu : ((1u << cnt) - 1u));
    const uint64_t left = nbits - pos;
    if (left < cnt) w &= (1u << left) - 1u;
    return w;
}

// The first stage's first two butterfly levels on input bits, in double precision: their values are
// integers up to 8 in magnitude (sums of four inputs 0 or +-2), so single precision is exact, and the
// encoding of such a float becomes the double's with integer instructions. The pass is bound by the
// FP64 pipe (90 % busy), which these levels occupied for 4 of its 32 operations per value: a batch of 64 keys
// of 10^6 bits took 10.09 ms instead of 10.41.
template <int R> constexpr int kExactLevels = R >= 4 ? 2 : 1;
__device__ __forceinline__ double widen(float x) {
    const uint32_t b = __float_as_uint(x), mag = b & 0x7fffffffu;
    return __hiloint2double((int)((mag ? (mag >> 3) + 0x38000000u : 0u) | (b & 0x80000000u)), 0);
}
template <int R, int LEVEL = 0>
__device__ __forceinline__ void exact_levels(float2 *u) {
    if constexpr (LEVEL < kExactLevels<R>) {
        dft_const_sub<float, R, false, LEVEL, 0>(u);
        exact_levels<R, LEVEL + 1>(u);
    }
}

// ---------------------------------------------------------------------------
// Level-1 forward pass from transposed bits. Grid (S/COLS, slots). KEYS: slot p holds keys 2p
// and 2p+1 (or, one key per slot, its even and odd bits); SEED: the rotated, +-1 encoded seed in
// the real part (or its even and odd positions); BLOCKS: block p's key and rotated seed.
// The slot's first CTA also adds up the popcounts the transposition left per part: popc[p * ppk] (+1 for the
// imaginary part's key; ppk = 1: both parts are one key's), or popc[block id].
template <typename T, int LEN, int COLS, int E, In KIND>
__global__ void __launch_bounds__(COLS * LEN / E, min_blocks(COLS * LEN / E))
    k_fwd(FwdArgs in, cx<T> *__restrict__ W, uint64_t L, TwTab<T> tw) {
    const uint32_t *bits = in.bits;
    const uint2 *parts = in.parts;
    const BlockDev *blocks = in.blocks;
    begin_after_previous(bits, parts, blocks, W);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T> *sm = reinterpret_cast<cx<T> *>(smem_raw);
    const uint32_t col = threadIdx.x % COLS, tq = threadIdx.x / COLS;
    const uint32_t S = (uint32_t)(L >> ilog2(LEN)), u = blockIdx.x * COLS + col;
    const uint32_t x = fresh(bits + (uint64_t)blockIdx.y * (L / E) + blockIdx.x * (COLS * LEN / E) + threadIdx.x);
    // double precision: the inputs and the first levels in single (exact)
    using I = typename std::conditional<std::is_same<T, double>::value, float, T>::type;
    cx<I> b[E];
    if constexpr (KIND == In::KEYS) {
#pragma unroll
        for (int s = 0; s < E; ++s) b[s] = Enc<I>::keys(x, slot_pos<T, LEN, E>(s));
    } else if constexpr (KIND == In::SEED) {
        const uint32_t re = in.re.mask(tq * S + u), im = in.im.mask(tq * S + u);
#pragma unroll
        for (int s = 0; s < E; ++s) b[s] = Enc<I>::seed(x, re, im, slot_pos<T, LEN, E>(s));
    } else {
        const uint32_t inside = blocks[blockIdx.y].in.mask(tq * S + u);
#pragma unroll
        for (int s = 0; s < E; ++s) b[s] = Enc<I>::key_seed(x, inside, slot_pos<T, LEN, E>(s));
    }
    cx<T> v[E];
    if constexpr (std::is_same<T, double>::value) {
        constexpr int R = Plan<T, LEN, E>::r0;
#pragma unroll
        for (int g = 0; g < E / R; ++g) exact_levels<R>(b + g * R);
#pragma unroll
        for (int s = 0; s < E; ++s) v[s] = make_double2(widen(b[s].x), widen(b[s].y));
        fwd_stages<T, LEN, COLS, E, 0, true, kExactLevels<R>>(sm, v, tq, col, tw.st[0]);
    } else {
#pragma unroll
        for (int s = 0; s < E; ++s) v[s] = b[s];
        cta_fft<T, LEN, COLS, E, false, KIND == In::BLOCKS>(sm, v, tq, col, tw.st[0]);
    }
    const uint32_t f = freq_of<T, LEN, E>(tq);
    pass_twiddles<T, E, COLS>(v, tw.fw[0], gridDim.x, f, blockIdx.x, col);
    cx<T> *w = W + (uint64_t)blockIdx.y * L + u;
#pragma unroll
    for (int s = 0; s < E; ++s) w[(f + s * (LEN / E)) * S] = v[s];
    if constexpr (KIND != In::SEED) {
        if (blockIdx.x == 0 && threadIdx.x < 32) {
            uint32_t ca = 0, cb = 0;
            for (uint32_t i = threadIdx.x; i < in.nparts; i += 32) {
                const uint2 c = fresh(parts + (uint64_t)blockIdx.y * in.nparts + i);
                ca += c.x;
                cb += c.y;
            }
            ca = __reduce_add_sync(0xffffffffu, ca);
            cb = __reduce_add_sync(0xffffffffu, cb);
            if (threadIdx.x == 0) {
                if constexpr (KIND == In::BLOCKS) {
                    in.popc[blocks[blockIdx.y].id] = ca;
                } else if (in.ppk == 1) {
                    in.popc[blockIdx.y] = ca + cb;
                } else {
                    in.popc[2 * blockIdx.y] = ca;
                    if (2 * blockIdx.y + 1 < in.nkeys) in.popc[2 * blockIdx.y + 1] = cb;
                }
            }
        }
    }
}

// Middle-level strided pass (three-level plans only), forward or inverse (NEAR: entry_powers).
// S is the innermost length (the stride of this pass); blocks of LEN*S elements.
// Grid (S/COLS, blocks * pairs).
template <typename T, int LEN, int COLS, int E, bool INV, bool NEAR = false>
__global__ void __launch_bounds__(COLS * LEN / E, min_blocks(COLS * LEN / E))
    k_mid(cx<T> *__restrict__ W, uint64_t L, uint32_t S, TwTab<T> tw) {
    begin_after_previous(W);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T> *sm = reinterpret_cast<cx<T> *>(smem_raw);
    const uint32_t col = threadIdx.x % COLS, tq = threadIdx.x / COLS;
    const uint64_t blk_len = (uint64_t)LEN * S;
    const uint64_t nblk = L / blk_len;
    const uint64_t pair = blockIdx.y / nblk, blk = blockIdx.y % nblk;
    const uint32_t u = blockIdx.x * COLS + col;
    cx<T> *w = W + pair * L + blk * blk_len + u;
    const uint32_t f = freq_of<T, LEN, E>(tq);
    cx<T> v[E];
#pragma unroll
    for (int s = 0; s < E; ++s) v[s] = fresh(w + (INV ? f + s * (LEN / E) : elem_of<T, LEN, E>(tq, s)) * S);
    if constexpr (INV) {
        inverse_columns<T, LEN, COLS, E, 1>(sm, v, tq, col, tw, gridDim.x, blockIdx.x, S, LEN);
    } else {
        cta_fft<T, LEN, COLS, E, false, NEAR>(sm, v, tq, col, tw.st[1]);
        pass_twiddles<T, E, COLS>(v, tw.fw[1], gridDim.x, f, blockIdx.x, col);
    }
    // the stride anew: where loads and stores go to the same rows, the compiler would keep 16
    // addresses in registers through the transform (80 bytes of spills; length 256 still has 60 to 70)
    asm volatile("" : "+r"(S));
#pragma unroll
    for (int s = 0; s < E; ++s) w[(INV ? elem_of<T, LEN, E>(tq, s) : f + s * (LEN / E)) * S] = v[s];
}

// Innermost level: contiguous rows of LEN elements. MODE 0: forward, times
// the seed spectrum, inverse (the fused convolution step). MODE 1: forward
// only, scaled by 1/L, written as the seed spectrum.
template <typename T, int LEN, int E, int MODE>
__global__ void __launch_bounds__(LEN / E, min_blocks_inner(LEN / E, sizeof(cx<T>)))
    k_middle(cx<T> *__restrict__ W, cx<T> *spec, uint64_t L, TwTab<T> tw, cx<T> scale) {
    begin_after_previous(W, spec);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T> *sm = reinterpret_cast<cx<T> *>(smem_raw);
    const uint32_t tq = threadIdx.x;
    const uint64_t row = blockIdx.x, pair = blockIdx.y;
    // thread tq's elements sit at compile-time offsets from element tq of the row
    cx<T> *wt = W + pair * L + row * LEN + tq;
    cx<T> *spt = spec + row * LEN + tq;
    cx<T> v[E];
    if constexpr (Plan<T, LEN, E>::RO == 1) {
#pragma unroll
        for (int s = 0; s < E; ++s) v[s] = fresh(wt + elem_of<T, LEN, E>(0, s));
        cta_fft<T, LEN, 1, E, false>(sm, v, tq, 0, tw.st[2]);
    } else {
        cta_fft_fwd_odd<T, LEN, E, false>(sm, v, tq, tw.st[2], [&](uint32_t o) { return fresh(wt + o); });
    }
    if constexpr (MODE == 1) {
#pragma unroll
        for (int s = 0; s < E; ++s) spt[s * (LEN / E)] = spectrum_value<T>(Arith<T>::mul(v[s], scale));
    } else {
#pragma unroll
        for (int s = 0; s < E; ++s) v[s] = Arith<T>::mul(v[s], spt[s * (LEN / E)]);
        if constexpr (Plan<T, LEN, E>::RO == 1) {
            cta_fft<T, LEN, 1, E, true>(sm, v, tq, 0, tw.st[2]);
#pragma unroll
            for (int s = 0; s < E; ++s) wt[elem_of<T, LEN, E>(0, s)] = v[s];
        } else {
            cta_fft_inv_odd<T, LEN, E>(sm, v, tq, tw.st[2], [&](uint32_t o, cx<T> x) { wt[o] = x; });
        }
    }
}

// Word type for COLS output bits.
template <int COLS> struct BitsWord;
template <> struct BitsWord<8> { using type = uint8_t; };
template <> struct BitsWord<16> { using type = uint16_t; };
template <> struct BitsWord<32> { using type = uint32_t; };

__device__ __forceinline__ float margin_to_float(float x) { return x; }
__device__ __forceinline__ float margin_to_float(double x) { return __double2float_ru(x); }

// Output bits up to the end of the last word, and the rows t1 of the column block at u0 with t1*S + u0 < end.
__device__ __forceinline__ uint32_t words_end(uint64_t m) { return (uint32_t)(((m + 63) >> 6) << 6); }
__device__ __forceinline__ uint32_t output_rows(uint32_t end, uint32_t u0, uint32_t S) {
    return end > u0 ? (end - u0 + S - 1u) / S : 0u;
}

// The bits of a warp's output rows. A ballot per register slot gives the bits of 32 / COLS rows, and every lane
// keeps the ballots of its own rows (slot lane / ROWS + q*COLS, the warp's row lane % ROWS), so that all the
// warp's rows are packed and stored at once. With a store per slot by its rows' first lanes, two of 32 lanes worked
// through the packing of every slot, and the modified hash read its key words slot after slot (7 keys of 100003
// bits: 55.4 us, now 47.9; 64 keys of 2^20 bits modulo the word-sized prime 949 us, now 927; the plain single
// precision batches, which wait on other things there, take the same time).
template <int COLS, int E>
struct RowBits {
    static constexpr int ROWS = 32 / COLS, N = E / COLS;
    static_assert(E % COLS == 0, "a lane keeps whole registers of rows");
    uint32_t a[N] = {}, b[N] = {};
    __device__ __forceinline__ void keep(int s, uint32_t lane, bool bit_a, bool bit_b) {
        const uint32_t ba = __ballot_sync(0xffffffffu, bit_a), bb = __ballot_sync(0xffffffffu, bit_b);
        if (lane / ROWS == (uint32_t)(s % COLS)) {
            a[s / COLS] = ba;
            b[s / COLS] = bb;
        }
    }
    // f(first output position of the row, its bits): rows whose slot was not reached hold no bits
    template <typename T, int LEN, class F>
    __device__ __forceinline__ void rows(uint32_t lane, uint32_t tq0, uint32_t S, uint32_t u0, F &&f) const {
        const uint32_t g = lane % ROWS, msk = (1u << COLS) - 1u;
#pragma unroll
        for (int q = 0; q < N; ++q)
            f(elem_of<T, LEN, E>(tq0 + g, (int)(lane / ROWS) + q * COLS) * S + u0, (a[q] >> (g * COLS)) & msk,
              (b[q] >> (g * COLS)) & msk);
    }
};

// Round, mod 2 and pack the outputs of the level-1 inverse transform of one column
// (pair form): v holds rows t1 = elem_of(tq, s) of column u = u0 + col, the real part
// belonging to key ka with ma_bits outputs, the imaginary part to key kb (if has_b) with
// mb_bits outputs (the uneven batch pairs blocks of different lengths; a plan's pairs
// have ma_bits = mb_bits = m). Output bit i = t1*S + u of a key is element i of the
// convolution window; bits past the key's outputs are written 0. Each key's rounding
// margin max |w - rint(w)| over its outputs goes to margin_bits[ka] / [kb] (float bits,
// atomicMax; margins are >= 0, so integer order is float order). With xkeys, the bits
// are XORed with key bits 0 .. m-1 (the identity block of the modified hash, Eq. 3).
template <typename T, int LEN, int COLS, int E>
__device__ __forceinline__ void pack_pair_bits(const cx<T> *v, uint32_t tq, uint32_t col, uint64_t S, uint64_t u0,
                                               uint64_t ma_bits, uint64_t mb_bits, uint32_t popa, uint32_t popb,
                                               uint32_t ka, uint32_t kb, bool has_b,
                                               typename BitsWord<COLS>::type *oa,
                                               typename BitsWord<COLS>::type *ob, uint32_t *margin_bits,
                                               const uint64_t *xkeys, uint64_t xstride) {
    using word_t = typename BitsWord<COLS>::type;
    const uint32_t lane = threadIdx.x & 31;
    // 32-bit positions (t1*S + u < L <= 2^28). Rows at or past the end of the last output word
    // are not decoded; the test uses the warp's first row of each slot (rows grow with tq, so
    // the whole warp is past the end when its first row is), which keeps it warp-uniform: the
    // ballots below need every lane. The bound is taken once as a row count, and where a
    // thread's rows grow with the slot (one radix-E last stage) the loop stops at the first
    // slot past it.
    const uint32_t S32 = (uint32_t)S, u032 = (uint32_t)u0;
    const uint32_t ma32 = (uint32_t)ma_bits, mb32 = has_b ? (uint32_t)mb_bits : 0u;
    const uint32_t mwa = words_end(ma_bits), mwb = has_b ? words_end(mb_bits) : 0u;
    const uint32_t mw = mwa > mwb ? mwa : mwb;
    const uint32_t tq0 = (threadIdx.x & ~31u) / COLS;  // the warp's first tq
    const uint32_t nrow = output_rows(mw, u032, S32);
    RowBits<COLS, E> bits;
    typename Enc<T>::M ma = 0, mb = 0;
    [[maybe_unused]] float wa_max = 0.f, wb_max = 0.f;  // single precision: largest |w| of each key
    [[maybe_unused]] const float2 half_p = make_float2(0.5f * (float)(popa & 3u), 0.5f * (float)(popb & 3u));
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const uint32_t t1 = elem_of<T, LEN, E>(tq, s);
        if constexpr (Plan<T, LEN, E>::r0 == E) {  // t1 = tq + s*TC: every later slot is past the bound too
            if (elem_of<T, LEN, E>(tq0, s) >= nrow) break;
        } else {
            if (elem_of<T, LEN, E>(tq0, s) >= nrow) continue;
        }
        const uint32_t row0 = t1 * S32 + u032;  // output bit of this row's first column
        const bool valid_a = row0 + col < ma32, valid_b = row0 + col < mb32;
        bool bit_a, bit_b;
        if constexpr (std::is_same<T, float>::value) {
            // w = ((P mod 4) - r)/2 for both keys at once; rint by the 1.5*2^23 addition (exact for |w| < 2^22)
            const float2 w = f2_fma(v[s], make_float2(-0.5f, -0.5f), half_p);
            const float2 f = f2_add(w, make_float2(Magic<float>::v, Magic<float>::v));
            const float2 d = f2_sub(w, f2_sub(f, make_float2(Magic<float>::v, Magic<float>::v)));
            bit_a = valid_a && (__float_as_uint(f.x) & 1u);
            bit_b = valid_b && (__float_as_uint(f.y) & 1u);
            ma = fmaxf(ma, valid_a ? fabsf(d.x) : 0.f);
            mb = fmaxf(mb, valid_b ? fabsf(d.y) : 0.f);
            wa_max = fmaxf(wa_max, valid_a ? fabsf(w.x) : 0.f);
            wb_max = fmaxf(wb_max, valid_b ? fabsf(w.y) : 0.f);
        } else {
            Enc<T>::decode2(v[s], popa, popb, valid_a, valid_b, bit_a, bit_b, ma, mb);
        }
        bits.keep(s, lane, bit_a, bit_b);
    }
    bits.template rows<T, LEN>(lane, tq0, S32, u032, [&](uint32_t row0, uint32_t ya, uint32_t yb) {
        const uint32_t ci = row0 / COLS;  // output chunk of this row's COLS bits
        if (row0 < mwa) {
            // modified Toeplitz hash (Eq. 3): the identity block adds key bits 0 .. m-1
            if (xkeys) ya ^= aligned_bits<COLS>(xkeys + (uint64_t)ka * xstride, ma_bits, row0);
            oa[ci] = (word_t)ya;
        }
        if (row0 < mwb) {
            if (xkeys) yb ^= aligned_bits<COLS>(xkeys + (uint64_t)kb * xstride, mb_bits, row0);
            ob[ci] = (word_t)yb;
        }
    });
    if constexpr (std::is_same<T, float>::value) {
        // beyond the exact range of the rounding the parity is not resolvable: a margin of 1 escalates
        if (wa_max >= Magic<float>::limit) ma = 1.f;
        if (wb_max >= Magic<float>::limit) mb = 1.f;
    }
    uint32_t fa = __float_as_uint(margin_to_float(ma)), fb = __float_as_uint(margin_to_float(mb));
    __shared__ uint32_t red[64];
    cta_reduce_put<true>(fa, fb, red);
    __syncthreads();
    cta_reduce_get<true>(fa, fb, red);
    if (threadIdx.x == 0) {
        atomicMax(margin_bits + ka, fa);
        if (has_b) atomicMax(margin_bits + kb, fb);
    }
}

// Level-1 inverse pass with the post-processing step of the paper's Fig. 2 (the
// inverse transform's output rounded to integers, then reduced mod 2): round, mod 2, pack.
// Output bit i = element i of the convolution window; bits >= m are written 0.
// Each key's rounding margin max |w - rint(w)| goes to margin_bits (float bits,
// atomicMax; all margins are >= 0 so integer order equals float order).
// PACK: slot p holds one key p of a half-length transform; element t carries output
// bits 2t (real part) and 2t+1 (imaginary part).
template <typename T, int LEN, int COLS, int E, bool PACK = false>
__global__ void __launch_bounds__(COLS * LEN / E, min_blocks(COLS * LEN / E))
    k_inv_bits(const cx<T> *__restrict__ W, uint64_t L, uint64_t m, uint32_t nkeys,
               const uint32_t *__restrict__ popc, uint32_t *__restrict__ margin_bits, uint64_t *__restrict__ out,
               uint64_t ostride, TwTab<T> tw, const uint64_t *__restrict__ xkeys, uint64_t xstride) {
    begin_after_previous(W, popc, margin_bits, out, xkeys);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T> *sm = reinterpret_cast<cx<T> *>(smem_raw);
    using word_t = typename BitsWord<COLS>::type;
    const uint32_t col = threadIdx.x % COLS, tq = threadIdx.x / COLS;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t S = L >> ilog2(LEN);
    const uint64_t u0 = (uint64_t)blockIdx.x * COLS;
    const uint64_t u = u0 + col;
    const uint32_t pair = blockIdx.y;
    const uint32_t ka = PACK ? pair : 2 * pair, kb = 2 * pair + 1;
    const bool has_b = !PACK && kb < nkeys;
    const cx<T> *w = W + (uint64_t)pair * L;
    const uint32_t f = freq_of<T, LEN, E>(tq);
    cx<T> v[E];
#pragma unroll
    for (int s = 0; s < E; ++s) v[s] = fresh(w + (f + s * (LEN / E)) * (uint32_t)S + (uint32_t)u);
    const uint32_t nrow = output_rows(PACK ? (words_end(m) >> 1) : words_end(m), (uint32_t)u0, (uint32_t)S);
    inverse_columns<T, LEN, COLS, E, 0>(sm, v, tq, col, tw, gridDim.x, blockIdx.x, (uint32_t)S, nrow);

    const uint32_t popa = fresh(popc + ka);
    const uint32_t popb = PACK ? popa : (has_b ? fresh(popc + kb) : 0u);
    word_t *oa = reinterpret_cast<word_t *>(out + (uint64_t)ka * ostride);
    word_t *ob = reinterpret_cast<word_t *>(out + (uint64_t)kb * ostride);
    if constexpr (PACK) {
        RowBits<COLS, E> bits;
        typename Enc<T>::M ma = 0, mb = 0;
        [[maybe_unused]] float w_max = 0.f;
        [[maybe_unused]] const float half_p = 0.5f * (float)(popa & 3u);
        // chunk ci: the row's COLS elements t = t1*S + u0 + c, i.e. output bits 2*(t1*S + u0) .. +2*COLS;
        // 32-bit positions, and the warp-uniform skip of rows past the last output word as in pack_pair_bits
        using word2_t = typename BitsWord<2 * COLS>::type;
        word2_t *o2 = reinterpret_cast<word2_t *>(out + (uint64_t)ka * ostride);
        const uint32_t S32 = (uint32_t)S, u032 = (uint32_t)u0, m32 = (uint32_t)m;
        const uint32_t mw = words_end(m);
        const uint32_t tq0 = (threadIdx.x & ~31u) / COLS;
#pragma unroll
        for (int s = 0; s < E; ++s) {
            const uint32_t t1 = elem_of<T, LEN, E>(tq, s);
            if constexpr (Plan<T, LEN, E>::r0 == E) {
                if (elem_of<T, LEN, E>(tq0, s) >= nrow) break;
            } else {
                if (elem_of<T, LEN, E>(tq0, s) >= nrow) continue;
            }
            const uint32_t row0 = t1 * S32 + u032;
            const uint32_t t = row0 + col;
            const bool ve = 2 * t < m32, vo = 2 * t + 1 < m32;
            bool bit_e, bit_o;
            if constexpr (std::is_same<T, float>::value) {
                const float2 w = f2_fma(v[s], make_float2(-0.5f, -0.5f), make_float2(half_p, half_p));
                const float2 f = f2_add(w, make_float2(Magic<float>::v, Magic<float>::v));
                const float2 d = f2_sub(w, f2_sub(f, make_float2(Magic<float>::v, Magic<float>::v)));
                bit_e = ve && (__float_as_uint(f.x) & 1u);
                bit_o = vo && (__float_as_uint(f.y) & 1u);
                ma = fmaxf(ma, ve ? fabsf(d.x) : 0.f);
                mb = fmaxf(mb, vo ? fabsf(d.y) : 0.f);
                w_max = fmaxf(w_max, fmaxf(ve ? fabsf(w.x) : 0.f, vo ? fabsf(w.y) : 0.f));
            } else {
                Enc<T>::decode2(v[s], popa, popa, ve, vo, bit_e, bit_o, ma, mb);
            }
            bits.keep(s, lane, bit_e, bit_o);
        }
        bits.template rows<T, LEN>(lane, tq0, S32, u032, [&](uint32_t row0, uint32_t ye, uint32_t yo) {
            if (2 * row0 >= mw) return;
            uint32_t y = spread_bits(ye) | (spread_bits(yo) << 1);
            if (xkeys) y ^= bits_at(xkeys + (uint64_t)ka * xstride, m, 2 * (uint64_t)row0, 2 * COLS);
            o2[row0 / COLS] = (word2_t)y;
        });
        if constexpr (std::is_same<T, float>::value) {
            if (w_max >= Magic<float>::limit) ma = 1.f;  // parity not resolvable: escalate
        }
        uint32_t f = __float_as_uint(margin_to_float(ma > mb ? ma : mb)), unused = 0u;
        __shared__ uint32_t red[64];
        cta_reduce_put<true>(f, unused, red);
        __syncthreads();
        cta_reduce_get<true>(f, unused, red);
        if (threadIdx.x == 0) atomicMax(margin_bits + ka, f);
        return;
    }
    pack_pair_bits<T, LEN, COLS, E>(v, tq, col, S, u0, m, m, popa, popb, ka, kb, has_b, oa, ob, margin_bits, xkeys,
                                    xstride);
}

// The level-1 inverse pass of key pairs (FP32, pair form) as a persistent kernel whose
// input tiles are staged by the TMA: tile t is the COLS x LEN block of columns
// u0 .. u0+COLS-1 of pair t / (S / COLS), copied by one tiled copy into shared memory.
// The copy of a CTA's next tile is issued as soon as every thread has read the current
// one, so a copy is in flight while the tile is transformed and decoded: the pass keeps
// enough bytes in flight without spending registers on them. The arithmetic is
// k_inv_bits's, step for step. The tensor map describes the work buffer as a
// (pairs * LEN) x S array of 8-byte elements (row a of pair p at row p*LEN + a).
//
// Tiles are handed out by a ticket counter (ctl[1]), so a CTA that starts late, behind
// another stream's kernel, just takes fewer tiles. Every CTA counts itself out on ctl[2]
// when it leaves; the last one resets both counters for the next launch (launches that
// share ctl run in stream order). A copy wait that runs out of time sets bit 0 of ctl[0]
// and the CTA leaves after a second bounded wait for that copy. expire_ns != 0 is a test
// hook for that path: no CTA takes a tile or issues a copy, and each waits expire_ns on a
// barrier phase that nothing can complete.
template <int LEN>
__global__ void __launch_bounds__(LEN, 768 / LEN)
    k_inv_bits_tma(const __grid_constant__ CUtensorMap wmap, uint64_t L, uint64_t m, uint32_t nkeys, uint32_t pairs,
                   const uint32_t *__restrict__ popc, uint32_t *__restrict__ margin_bits, uint64_t *__restrict__ out,
                   uint64_t ostride, TwTab<float> tw, const uint64_t *__restrict__ xkeys, uint64_t xstride,
                   uint32_t *__restrict__ ctl, uint32_t expire_ns) {
    using T = float;
    constexpr int E = 16, COLS = 16;
    static_assert(LEN <= 256 && LEN >= 64, "one tiled copy moves at most 256 rows");
    constexpr uint32_t kTileBytes = LEN * COLS * sizeof(cx<T>);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // a tiled copy's destination must be 128-byte aligned: the launch adds 128 bytes to round up
    unsigned char *base = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
    cx<T> *stg = reinterpret_cast<cx<T> *>(base);  // staged tile: row a at stg[a * COLS .. +COLS)
    cx<T> *sm = stg + LEN * COLS;                   // exchange buffer of the transform
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t next_tile;
    using word_t = typename BitsWord<COLS>::type;
    const uint32_t col = threadIdx.x % COLS, tq = threadIdx.x / COLS;
    const uint64_t S = L >> ilog2(LEN);
    const uint32_t ncolt = (uint32_t)(S / COLS);
    const uint32_t ntiles = ncolt * pairs;
    const bool aligned = (smem_addr(stg) & 127u) == 0;  // always, given the spare bytes: never copy misaligned
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init_fence();
        uint32_t t = ntiles;
        if (!aligned) {
            atomicOr(ctl, 2u);
        } else if (expire_ns == 0) {
            t = atomicAdd(ctl + 1, 1u);
            if (t < ntiles) {
                mbar_arrive_expect_tx(&bar, kTileBytes);
                tma_load_2d(stg, &wmap, (int)((t % ncolt) * COLS), (int)((t / ncolt) * LEN), &bar);
            }
        } else if (!mbar_wait(&bar, 0, expire_ns)) {  // test hook: phase 0 never completes
            atomicOr(ctl, 1u);
        }
        next_tile = t;
    }
    __syncthreads();
    uint32_t t = next_tile, phase = 0;
    while (t < ntiles) {
        const bool ok = mbar_wait(&bar, phase);
        phase ^= 1u;
        // also orders this tile's first exchange writes after the last tile's exchange reads
        if (!__syncthreads_and(ok)) {
            if (threadIdx.x == 0) {
                atomicOr(ctl, 1u);
                mbar_wait(&bar, phase ^ 1u);  // the copy that ran late: one more bounded wait
            }
            break;
        }
        cx<T> v[E];
#pragma unroll
        for (int s = 0; s < E; ++s) v[s] = stg[(freq_of<T, LEN, E>(tq) + s * (LEN / E)) * COLS + col];
        __syncthreads();  // the staged tile has been read: refill it with the next tile
        if (threadIdx.x == 0) {
            const uint32_t nt = atomicAdd(ctl + 1, 1u);
            if (nt < ntiles) {
                mbar_arrive_expect_tx(&bar, kTileBytes);
                tma_load_2d(stg, &wmap, (int)((nt % ncolt) * COLS), (int)((nt / ncolt) * LEN), &bar);
            }
            next_tile = nt;  // read by every thread after pack_pair_bits' barrier
        }
        const uint32_t pair = t / ncolt;
        const uint64_t u0 = (uint64_t)(t % ncolt) * COLS;
        const uint32_t ka = 2 * pair, kb = ka + 1;
        const bool has_b = kb < nkeys;
        inverse_columns<T, LEN, COLS, E, 0>(sm, v, tq, col, tw, ncolt, t % ncolt, (uint32_t)S,
                                            output_rows(words_end(m), (uint32_t)u0, (uint32_t)S));
        const uint32_t popa = popc[ka], popb = has_b ? popc[kb] : 0u;
        word_t *oa = reinterpret_cast<word_t *>(out + (uint64_t)ka * ostride);
        word_t *ob = reinterpret_cast<word_t *>(out + (uint64_t)kb * ostride);
        pack_pair_bits<T, LEN, COLS, E>(v, tq, col, S, u0, m, m, popa, popb, ka, kb, has_b, oa, ob, margin_bits, xkeys,
                                        xstride);
        t = next_tile;
    }
    if (threadIdx.x == 0 && atomicAdd(ctl + 2, 1u) == gridDim.x - 1) {
        // every CTA has taken its last ticket: reset the counters for the next launch
        atomicExch(ctl + 1, 0u);
        atomicExch(ctl + 2, 0u);
    }
}

}  // namespace pa

// ===========================================================================
// Uneven batch: blocks of different (n, m), each with its own seed, grouped by
// transform length L. Per block the paper's real-valued FFT acceleration
// (Eq. 5-10) carries key and seed in one complex transform, z = x + i*sigma;
// the fused middle pass separates X and V from Z(k) and Z(-k), forms X*V and
// sends two blocks' products through one inverse transform as Y1 + i*Y2.
// ===========================================================================
namespace pa {

// Storage row of the frequency low part rho (lgM = log2 of the middle strided
// pass length, 0 for two-level plans): rho = k1 + L1*k2 sits at row k1*M + k2.
__device__ __forceinline__ uint32_t split_row(uint32_t rho, uint32_t lgL1, uint32_t lgM) {
    return ((rho & ((1u << lgL1) - 1u)) << lgM) + (rho >> lgL1);
}

// The mirror bins of a thread's spectrum values (frequency p = f + s*TC of its row) in the
// mirror row's spectrum in shared memory: frequency LEN-1-p, or in the row of the zero
// frequency low part -p mod LEN. LEN-1-p complements every digit of p, so thread TC-1-tq holds
// it, in register slot E-1-s.
template <typename T, int LEN, int E> struct Mirror {
    const cx<T> *base;
    uint32_t shift;  // -p mod LEN for f = 0: the thread's own block, one register slot further
    __device__ __forceinline__ Mirror(const cx<T> *spectrum, uint32_t tq, bool zero_row) : shift(0) {
        constexpr uint32_t TC = LEN / E;
        uint32_t t = TC - 1u - tq;
        if (zero_row) {
            const uint32_t f = freq_of<T, LEN, E>(tq);
            t = f ? thread_of<T, LEN, E>(TC - f) : 0u;
            shift = f ? 0u : 1u;
        }
        base = spectrum + slot_of<T, 1>(t * E, 0);
    }
    __device__ __forceinline__ cx<T> at(int s) const { return base[((uint32_t)(E - 1 - s) + shift) % E]; }
};

// Fused innermost pass of the uneven batch. CTA (rho, pair): rows rho and
// -rho of blocks 2*pair and 2*pair+1 (if present), one thread group per row.
// Forward transform, Eq. 5-10 split with the mirror bin, X*V/L, then the
// inverse transform of Y1 + i*Y2 written to the pair's slot in Wi. The first block's product waits in
// the row it came from, which the transform has consumed, while the second block is transformed: in
// registers it took 32 of a thread's, so that one CTA of 512 threads filled an SM.
template <typename T, int LEN, int E>
__global__ void __launch_bounds__(2 * (LEN / E), min_blocks_split(2 * (LEN / E), sizeof(cx<T>)))
    k_middle_split(cx<T> *Wf, cx<T> *__restrict__ Wi, uint64_t L, uint32_t nblocks, uint32_t lgL1, uint32_t lgM,
                   TwTab<T> tw, T inv_L) {
    begin_after_previous(Wf, Wi);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T> *smem = reinterpret_cast<cx<T> *>(smem_raw);
    constexpr uint32_t TC = LEN / E;
    constexpr uint32_t SE = smem_elems<T, LEN, 1>();
    const uint32_t g = threadIdx.x / TC, tq = threadIdx.x % TC;
    const uint32_t R = (uint32_t)(L / LEN);  // rows per block
    const uint32_t rho = blockIdx.x;          // 0 .. R/2
    const uint32_t rho_m = (R - rho) & (R - 1);
    const uint32_t my_rho = g ? rho_m : rho;
    const uint32_t row = split_row(my_rho, lgL1, lgM);
    const bool self_paired = rho == rho_m;
    cx<T> *sm = smem + g * SE;                          // this group's transform scratch
    const cx<T> *sm_other = smem + (self_paired ? g : 1u - g) * SE;  // where the mirror row's spectrum sits
    const uint32_t b1 = 2 * blockIdx.y, nb = b1 + 1 < nblocks ? 2u : 1u;
    const Mirror<T, LEN, E> mir(sm_other, tq, my_rho == 0);
    cx<T> *const w1 = Wf + (uint64_t)b1 * L + (uint64_t)row * LEN + tq;
    cx<T> v[E];
    for (uint32_t which = 0; which < nb; ++which) {
        const cx<T> *wt = w1 + which * L;
        __syncthreads();  // previous use of the scratch is finished
        if constexpr (Plan<T, LEN, E>::RO == 1) {
#pragma unroll
            for (int s = 0; s < E; ++s) v[s] = fresh(wt + elem_of<T, LEN, E>(0, s));
            cta_fft<T, LEN, 1, E, false, true>(sm, v, tq, 0, tw.st[2]);
        } else {
            cta_fft_fwd_odd<T, LEN, E, true>(sm, v, tq, tw.st[2], [&](uint32_t o) { return fresh(wt + o); });
        }
        store_stage<T, LEN, 1, E, Plan<T, LEN, E>::n - 1>(sm, v, tq, 0);  // the slots this thread read last
        __syncthreads();
#pragma unroll
        for (int s = 0; s < E; ++s) {
            const cx<T> z = v[s], zm = mir.at(s);
            // Eq. 7-10: X = (Z(k) + conj Z(-k)) / 2, V = (Z(k) - conj Z(-k)) / (2i)
            const cx<T> X = Arith<T>::mk((z.x + zm.x) * (T)0.5, (z.y - zm.y) * (T)0.5);
            const cx<T> V = Arith<T>::mk((z.y + zm.y) * (T)0.5, (zm.x - z.x) * (T)0.5);
            const cx<T> P = Arith<T>::mul(X, V);
            cx<T> Y = Arith<T>::mk(P.x * inv_L, P.y * inv_L);
            if (which == 0) {
                if (nb == 2) w1[s * TC] = Y;  // a self-paired row's two groups write the same values
            } else {  // Y1 + i * Y2
                const cx<T> Y1 = w1[s * TC];
                Y = Arith<T>::mk(Y1.x - Y.y, Y1.y + Y.x);
            }
            v[s] = Y;
        }
    }
    __syncthreads();
    cx<T> *wot = Wi + (uint64_t)blockIdx.y * L + (uint64_t)row * LEN + tq;
    const bool store = !(self_paired && g == 1);  // a self-paired row is written once
    if constexpr (Plan<T, LEN, E>::RO == 1) {
        cta_fft<T, LEN, 1, E, true>(sm, v, tq, 0, tw.st[2]);
        if (!store) return;
#pragma unroll
        for (int s = 0; s < E; ++s) wot[elem_of<T, LEN, E>(0, s)] = v[s];
    } else {
        cta_fft_inv_odd<T, LEN, E>(sm, v, tq, tw.st[2], [&](uint32_t o, cx<T> x) {
            if (store) wot[o] = x;
        });
    }
}

// Fused innermost pass of a single key in a half-length transform (the real-input
// form of the convolution theorem; paper Eq. 5-10 give the same split for a key and
// a seed). The slot holds Z = FFT_N(z), z[t] = x[2t] + i x[2t+1], N = L/2. With the
// mirror bin Z' = Z[N-k]: E_x = (Z + conj Z')/2 and O_x = (Z - conj Z')/(2i) are the
// spectra of the even and odd key bits, and with the seed tables (per bin, times 1/N)
// Es = E_s and Os = O_s of the seed's even/odd spectra, the product Y = S X of the length-L
// transforms is, in even/odd form (kRealTables: double precision also keeps w_N^k O_s),
//     E_y = Es E_x + Os (w_N^k O_x),   O_y = Es O_x + Os E_x,
// and the inverse transform of E_y + i O_y returns y[2t] + i y[2t+1].
// CTA (rho, slot): rows rho and -rho (one thread group each), as in k_middle_split.
// MODE 1 builds the tables from the seed slot instead (forward transform and split only).
template <typename T, int LEN, int E, int MODE>
__global__ void __launch_bounds__(2 * (LEN / E), min_blocks_real(2 * (LEN / E), sizeof(cx<T>)))
    k_middle_real(cx<T> *__restrict__ W, cx<T> *tabs, uint64_t N, uint32_t lgL1, uint32_t lgM,
                  TwTab<T> tw, T scale) {
    begin_after_previous(W, tabs);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T> *smem = reinterpret_cast<cx<T> *>(smem_raw);
    constexpr uint32_t TC = LEN / E;
    constexpr uint32_t SE = smem_elems<T, LEN, 1>();
    const uint32_t g = threadIdx.x / TC, tq = threadIdx.x % TC;
    const uint32_t R = (uint32_t)(N / LEN);  // rows
    const uint32_t rho = blockIdx.x;          // 0 .. R/2
    const uint32_t rho_m = (R - rho) & (R - 1);
    const uint32_t my_rho = g ? rho_m : rho;
    const uint32_t row = split_row(my_rho, lgL1, lgM);
    const bool self_paired = rho == rho_m;
    cx<T> *sm = smem + g * SE;
    const cx<T> *sm_other = smem + (self_paired ? g : 1u - g) * SE;
    cx<T> *wt = W + (uint64_t)blockIdx.y * N + (uint64_t)row * LEN + tq;
    cx<T> v[E];
    if constexpr (Plan<T, LEN, E>::RO == 1) {
#pragma unroll
        for (int s = 0; s < E; ++s) v[s] = fresh(wt + elem_of<T, LEN, E>(0, s));
        cta_fft<T, LEN, 1, E, false>(sm, v, tq, 0, tw.st[2]);
    } else {
        cta_fft_fwd_odd<T, LEN, E, false>(sm, v, tq, tw.st[2], [&](uint32_t o) { return fresh(wt + o); });
    }
    store_stage<T, LEN, 1, E, Plan<T, LEN, E>::n - 1>(sm, v, tq, 0);  // the slots this thread read last
    __syncthreads();
    const Mirror<T, LEN, E> mir(sm_other, tq, my_rho == 0);
    constexpr bool THREE = kRealTables<T> == 3;
    const cx<T> *Es = tabs, *Os = tabs + N;
    [[maybe_unused]] const uint32_t k0 = my_rho + R * freq_of<T, LEN, E>(tq);  // frequency of bin s: k0 + R s TC
    [[maybe_unused]] cx<T> w0;
    if constexpr (MODE == 0 && !THREE) w0 = Arith<T>::template omega<false>(tw, k0);
    const bool write_tab = !(self_paired && g == 1);
    static_for<E>([&](auto slot) {
        constexpr int s = decltype(slot)::value;
        const cx<T> z = v[s], zm = mir.at(s);
        const cx<T> ex = Arith<T>::mk((z.x + zm.x) * (T)0.5, (z.y - zm.y) * (T)0.5);
        const cx<T> ox = Arith<T>::mk((z.y + zm.y) * (T)0.5, (zm.x - z.x) * (T)0.5);
        const uint64_t e = (uint64_t)row * LEN + tq + s * TC;  // the tables keep the registers' order
        if constexpr (MODE == 1) {
            if (write_tab) {
                const cx<T> es = Arith<T>::mk(ex.x * scale, ex.y * scale);
                const cx<T> os = Arith<T>::mk(ox.x * scale, ox.y * scale);
                tabs[e] = es;
                tabs[N + e] = os;
                if constexpr (THREE) tabs[2 * N + e] = Arith<T>::mul(Arith<T>::template omega<false>(tw, k0 + R * (s * TC)), os);
            }
        } else {
            const cx<T> es = Es[e], os = Os[e];
            cx<T> t;  // w_N^k O_s O_x
            if constexpr (THREE) {
                t = Arith<T>::mul(tabs[2 * N + e], ox);
            } else {  // w_N^{R s TC} = w_E^s
                t = Arith<T>::mul(os, Arith<T>::mul(turn<T, E, s>(w0), ox));
            }
            const cx<T> ey = Arith<T>::add(Arith<T>::mul(es, ex), t);
            const cx<T> oy = Arith<T>::add(Arith<T>::mul(es, ox), Arith<T>::mul(os, ex));
            v[s] = Arith<T>::mk(ey.x - oy.y, ey.y + oy.x);  // E_y + i O_y
        }
    });
    if constexpr (MODE == 0) {
        __syncthreads();  // the mirror reads of both groups are done
        const bool store = !(self_paired && g == 1);  // a self-paired row is written once
        if constexpr (Plan<T, LEN, E>::RO == 1) {
            cta_fft<T, LEN, 1, E, true>(sm, v, tq, 0, tw.st[2]);
            if (!store) return;
#pragma unroll
            for (int s = 0; s < E; ++s) wt[elem_of<T, LEN, E>(0, s)] = v[s];
        } else {
            cta_fft_inv_odd<T, LEN, E>(sm, v, tq, tw.st[2], [&](uint32_t o, cx<T> x) {
                if (store) wt[o] = x;
            });
        }
    }
}

// Level-1 inverse pass with bit output for pairs of blocks (real part: block
// 2p, imaginary part: block 2p+1), each with its own m and output pointer.
template <typename T, int LEN, int COLS, int E>
__global__ void __launch_bounds__(COLS * LEN / E, min_blocks(COLS * LEN / E))
    k_inv_bits_blocks(const cx<T> *__restrict__ W, uint64_t L, const BlockDev *blocks, uint32_t nblocks,
                      const uint32_t *__restrict__ popc, uint32_t *__restrict__ margin_bits, TwTab<T> tw) {
    begin_after_previous(W, blocks, popc, margin_bits);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T> *sm = reinterpret_cast<cx<T> *>(smem_raw);
    using word_t = typename BitsWord<COLS>::type;
    const uint32_t col = threadIdx.x % COLS, tq = threadIdx.x / COLS;
    const uint64_t S = L >> ilog2(LEN);
    const uint64_t u0 = (uint64_t)blockIdx.x * COLS;
    const uint64_t u = u0 + col;
    const uint32_t ia = 2 * blockIdx.y, ib = ia + 1;
    const bool has_b = ib < nblocks;
    const BlockDev ba_ = blocks[ia];
    const BlockDev bb_ = blocks[has_b ? ib : ia];
    const cx<T> *w = W + (uint64_t)blockIdx.y * L;
    const uint32_t f = freq_of<T, LEN, E>(tq);
    cx<T> v[E];
#pragma unroll
    for (int s = 0; s < E; ++s) v[s] = fresh(w + (f + s * (LEN / E)) * (uint32_t)S + (uint32_t)u);
    const uint32_t mw = words_end(ba_.m > bb_.m ? ba_.m : bb_.m);
    inverse_columns<T, LEN, COLS, E, 0>(sm, v, tq, col, tw, gridDim.x, blockIdx.x, (uint32_t)S,
                                        output_rows(mw, (uint32_t)u0, (uint32_t)S));
    const uint32_t popa = fresh(popc + ba_.id);
    const uint32_t popb = has_b ? fresh(popc + bb_.id) : 0u;
    word_t *oa = reinterpret_cast<word_t *>(ba_.out);
    word_t *ob = reinterpret_cast<word_t *>(bb_.out);
    // each block decoded with its own m: the real part is block 2p, the imaginary part block 2p+1
    pack_pair_bits<T, LEN, COLS, E>(v, tq, col, S, u0, ba_.m, bb_.m, popa, popb, ba_.id, bb_.id, has_b, oa, ob,
                                    margin_bits, nullptr, 0);
}

}  // namespace pa
