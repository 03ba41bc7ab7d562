// pa_prep.cu -- preparation of a batch: transposed input bits, popcounts, margin reset.
#include <mutex>
#include <cuda.h>
#include <set>
#include <type_traits>
#include <utility>

#include "pa_kernels.cuh"
#include "pa_launch.h"

namespace pa {

namespace {
std::mutex g_smem_mu;
std::set<std::pair<const void *, int>> g_smem_done;
}  // namespace

bool encode_tile_map(CUtensorMap *map, const void *base, uint64_t cols, uint64_t rows, uint32_t box_cols,
                     uint32_t box_rows) {
    using Encode = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static Encode encode = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            encode = reinterpret_cast<Encode>(f);
        cudaGetLastError();
    });
    if (!encode) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * 8};  // bytes between rows (a multiple of 16: cols is even)
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool smem_configured(const void *kernel, int device) {
    std::lock_guard<std::mutex> lk(g_smem_mu);
    return g_smem_done.count({kernel, device}) != 0;
}

void smem_mark_configured(const void *kernel, int device) {
    std::lock_guard<std::mutex> lk(g_smem_mu);
    g_smem_done.insert({kernel, device});
}

// ---- transposed input bits -------------------------------------------------------------------
// w[j] = the 32 bits of p (nbits long) from bit at(j) on, j < E; bits at or past nbits read as 0. All
// positions share their offset in a word. The loads are branch free (addresses clamped to the last
// word) and leave together: with each row's load behind the last one's, a thread took 16 memory
// latencies (16 us for 32 keys of 2^20 bits).
template <int E, class At>
__device__ __forceinline__ void bits_rows(const uint32_t *__restrict__ p, uint32_t nbits, At at, uint32_t *w) {
    const uint32_t last = (nbits - 1) >> 5, r = at(0) & 31u;
#pragma unroll
    for (int j = 0; j < E; ++j) w[j] = fresh(p + min(at(j) >> 5, last));
    if (r) {
        uint32_t hi[E];
#pragma unroll
        for (int j = 0; j < E; ++j) hi[j] = fresh(p + min((at(j) >> 5) + 1, last));
#pragma unroll
        for (int j = 0; j < E; ++j) w[j] = __funnelshift_r(w[j], hi[j], r);
    }
#pragma unroll
    for (int j = 0; j < E; ++j)  // a mask of the bits left, none to 32
        w[j] &= __funnelshift_lc(0xffffffffu, 0u, (uint32_t)max((int)(nbits - at(j)), 0));
}
// The even-position bits of x in the low 16 bits.
__device__ __forceinline__ uint32_t even_bits(uint32_t x) {
    x &= 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0F0F0F0Fu;
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return (x | (x >> 8)) & 0x0000FFFFu;
}
// Transposes, in each 16-bit half (E = 16) or byte (E = 8) of the words, the E x E bit matrix whose
// row j is word j: afterwards bit j of word c is what bit c of word j was.
template <int E, int D = E / 2>
__device__ __forceinline__ void transpose_words(uint32_t *x) {
    if constexpr (D >= 1) {
        constexpr uint32_t m = D == 8 ? 0x00FF00FFu : D == 4 ? 0x0F0F0F0Fu : D == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const int lo = i / D * 2 * D + i % D, hi = lo + D;
            const uint32_t t = ((x[lo] >> D) ^ x[hi]) & m;
            x[hi] ^= t;
            x[lo] ^= t << D;
        }
        transpose_words<E, D / 2>(x);
    }
}

// Where a slot's bits come from: words(x, D, out) gives, for the 16 elements x + j*D .. +15 of every
// row j < E, the real part's bits in the low and the imaginary part's in the high half (x < D). D and
// the cyclic lengths are multiples of 64; positions stay below 2^30.
struct KeySource {
    const uint32_t *a, *b;  // b: null without a second key
    uint32_t n, koff;
    template <int E> __device__ __forceinline__ void words(uint32_t x, uint32_t D, uint32_t *out) const {
        const auto at = [&](int j) { return (x & ~31u) + koff + (uint32_t)j * D; };
        uint32_t wa[E], wb[E];
        bits_rows<E>(a, n + koff, at, wa);
        if (b) {
            bits_rows<E>(b, n + koff, at, wb);
        } else {
#pragma unroll
            for (int j = 0; j < E; ++j) wb[j] = 0u;
        }
        const int sel = (x & 16u) ? 0x7632 : 0x5410;
#pragma unroll
        for (int j = 0; j < E; ++j) out[j] = __byte_perm(wa[j], wb[j], sel);
    }
};
// Seed bits of rotated positions: position t of the cyclic length holds seed bit t + n - 1.
struct Rotated {
    const uint32_t *p;
    uint32_t nbits, rot, len;
    __device__ Rotated(const uint64_t *seed, uint64_t n, uint64_t m, uint64_t length)
        : p(reinterpret_cast<const uint32_t *>(seed)), nbits((uint32_t)(n + m - 1)), rot((uint32_t)n - 1u), len((uint32_t)length) {}
    template <int E> __device__ __forceinline__ void rows(uint32_t t, uint32_t step, uint32_t *w) const {
        const auto at = [&](int j) {
            const uint32_t s = t + (uint32_t)j * step + rot;
            return s >= len ? s - len : s;
        };
        bits_rows<E>(p, nbits, at, w);
        const uint32_t r = rot & 31u;
        const uint32_t first = r ? fresh(p) & __funnelshift_lc(0xffffffffu, 0u, nbits) : 0u;  // the seed's first 32 bits
#pragma unroll
        for (int j = 0; j < E; ++j)  // the 32 positions may wrap to the seed's start
            if (at(j) + 32 > len) w[j] |= first << (len - at(j));
    }
};
// 32 bits split into their even ones (low half) and odd ones (high half).
__device__ __forceinline__ uint32_t even_odd(uint32_t c) { return even_bits(c) | (even_bits(c >> 1) << 16); }
struct PackedKeySource {
    const uint32_t *a;
    uint32_t n, koff;
    template <int E> __device__ __forceinline__ void words(uint32_t x, uint32_t D, uint32_t *out) const {
        bits_rows<E>(a, n + koff, [&](int j) { return 2 * (x + (uint32_t)j * D) + koff; }, out);
#pragma unroll
        for (int j = 0; j < E; ++j) out[j] = even_odd(out[j]);
    }
};
struct SeedSource {
    Rotated s;
    template <int E> __device__ __forceinline__ void words(uint32_t x, uint32_t D, uint32_t *out) const {
        s.rows<E>(x, D, out);
#pragma unroll
        for (int j = 0; j < E; ++j) out[j] &= 0xffffu;
    }
};
struct PackedSeedSource {
    Rotated s;
    template <int E> __device__ __forceinline__ void words(uint32_t x, uint32_t D, uint32_t *out) const {
        s.rows<E>(2 * x, 2 * D, out);
#pragma unroll
        for (int j = 0; j < E; ++j) out[j] = even_odd(out[j]);
    }
};
struct BlockSource {
    const uint32_t *key;
    uint32_t n;
    Rotated s;
    template <int E> __device__ __forceinline__ void words(uint32_t x, uint32_t D, uint32_t *out) const {
        uint32_t wk[E], ws[E];
        bits_rows<E>(key, n, [&](int j) { return (x & ~31u) + (uint32_t)j * D; }, wk);
        s.rows<E>(x, D, ws);
#pragma unroll
        for (int j = 0; j < E; ++j) out[j] = __byte_perm(wk[j] >> (x & 16u), ws[j], 0x5410);
    }
};

// Shape of a transposition: column stride S, threads per column TC, columns per CTA of the pass
// 2^lgc, and lgh (transpose_slot).
struct BitShape {
    uint32_t S, TC, lgc, lgh;
};

// One thread transposes 16 columns of the E rows tq + j*TC: E words in, 16 words out, in groups of 2^lgc
// consecutive ones. Threads run over 2^lgh neighbouring groups of 16 columns (a 32-byte sector of every
// row), then over tq (neighbouring groups of words), so reads and writes are whole sectors. The pass
// reads the packed bits once and writes L/E words per slot, a 32nd of the pass it feeds.
template <int E, class Src>
__device__ __forceinline__ void transpose_slot(const Src &src, const BitShape &h, uint32_t idx, uint32_t *out,
                                               uint32_t &ca, uint32_t &cb) {
    const uint32_t rest = idx >> h.lgh, tq = rest & (h.TC - 1u);
    const uint32_t c0 = 16u * ((rest / h.TC << h.lgh) + (idx & ((1u << h.lgh) - 1u)));  // first column
    uint32_t x[E];
    src.template words<E>(tq * h.S + c0, h.S * h.TC, x);
    ca = cb = 0;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        ca += __popc(x[j] & 0xffffu);
        cb += __popc(x[j] >> 16);
    }
    transpose_words<E>(x);
    uint32_t w[16];
#pragma unroll
    for (int c = 0; c < 16; ++c)  // E = 8: bytes hold columns 0-7 and 8-15 of the real part, then of the imaginary part
        w[c] = E == 16 ? x[c % E] : (c < 8 ? x[c % E] : x[c % E] >> 8) & 0x00FF00FFu;
#pragma unroll
    for (int c = 0; c < 16; c += 4) {
        const uint32_t col = c0 + c, blk = col >> h.lgc;
        *reinterpret_cast<uint4 *>(out + (((uint64_t)blk * h.TC + tq) << h.lgc) + (col - (blk << h.lgc))) =
            make_uint4(w[c], w[c + 1], w[c + 2], w[c + 3]);
    }
}
// The CTA's popcounts as one part.
__device__ __forceinline__ void store_part(uint2 *parts, uint32_t ca, uint32_t cb) {
    __shared__ uint32_t red[2][kBitThreads / 32];
    ca = __reduce_add_sync(0xffffffffu, ca);
    cb = __reduce_add_sync(0xffffffffu, cb);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = ca;
        red[1][threadIdx.x >> 5] = cb;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (uint32_t i = 1; i < kBitThreads / 32; ++i) {
            ca += red[0][i];
            cb += red[1][i];
        }
        parts[(uint64_t)blockIdx.y * gridDim.x + blockIdx.x] = make_uint2(ca, cb);
    }
}

template <int E, bool PACK>
__global__ void __launch_bounds__(kBitThreads) k_key_bits(KeyBits k, BitShape h, BitScratch out,
                                                          uint32_t *__restrict__ margin_bits) {
    begin_after_previous(k.keys, out.bits, out.parts, margin_bits);
    const uint32_t idx = blockIdx.x * kBitThreads + threadIdx.x, slot = blockIdx.y;
    uint32_t *bits = out.bits + (uint64_t)slot * h.S * h.TC;
    uint32_t ca = 0, cb = 0;
    const bool two = !PACK && 2 * slot + 1 < k.nkeys;
    if (idx < h.S / 16 * h.TC) {
        const uint64_t *a = k.keys + (PACK ? 1 : 2) * (uint64_t)slot * k.kstride;
        if constexpr (PACK) {
            const PackedKeySource src{reinterpret_cast<const uint32_t *>(a), (uint32_t)k.n, (uint32_t)k.koff};
            transpose_slot<E>(src, h, idx, bits, ca, cb);
        } else {
            const KeySource src{reinterpret_cast<const uint32_t *>(a),
                                two ? reinterpret_cast<const uint32_t *>(a + k.kstride) : nullptr, (uint32_t)k.n,
                                (uint32_t)k.koff};
            transpose_slot<E>(src, h, idx, bits, ca, cb);
        }
    }
    store_part(out.parts, ca, cb);
    if (idx == 0) {  // the last pass accumulates the rounding margins
        margin_bits[(PACK ? 1 : 2) * slot] = 0u;
        if (two) margin_bits[2 * slot + 1] = 0u;
    }
}

// The seed for a length-L transform (grid row 0) and, with a second grid row, packed for the
// half-length form: even and odd rotated positions of the cyclic length 2 * len[1].
template <int E>
__global__ void __launch_bounds__(kBitThreads) k_seed_bits(const uint64_t *__restrict__ seed, uint64_t n, uint64_t m,
                                                           BitShape h0, uint64_t len0, uint32_t *out0, BitShape h1,
                                                           uint64_t len1, uint32_t *out1) {
    begin_after_previous(seed, out0, out1);
    const uint32_t idx = blockIdx.x * kBitThreads + threadIdx.x;
    uint32_t ca, cb;
    if (blockIdx.y == 0) {
        if (idx < h0.S / 16 * h0.TC) transpose_slot<E>(SeedSource{Rotated(seed, n, m, len0)}, h0, idx, out0, ca, cb);
    } else {
        if (idx < h1.S / 16 * h1.TC)
            transpose_slot<E>(PackedSeedSource{Rotated(seed, n, m, 2 * len1)}, h1, idx, out1, ca, cb);
    }
}

template <int E>
__global__ void __launch_bounds__(kBitThreads) k_block_bits(const BlockDev *blocks, BitShape h, uint64_t L,
                                                            BitScratch out, uint32_t *__restrict__ margin_bits) {
    begin_after_previous(blocks, out.bits, out.parts, margin_bits);
    const uint32_t idx = blockIdx.x * kBitThreads + threadIdx.x;
    const BlockDev &b = blocks[blockIdx.y];
    uint32_t ca = 0, cb = 0;
    if (idx < h.S / 16 * h.TC) {
        const BlockSource src{reinterpret_cast<const uint32_t *>(b.key), (uint32_t)b.n, Rotated(b.seed, b.n, b.m, L)};
        transpose_slot<E>(src, h, idx, out.bits + (uint64_t)blockIdx.y * h.S * h.TC, ca, cb);
    }
    store_part(out.parts, ca, 0u);
    if (idx == 0) margin_bits[b.id] = 0u;
}

static BitShape bit_shape(const BitForm &f) {
    BitShape h{(uint32_t)(f.L >> f.lgLEN), (1u << f.lgLEN) / (uint32_t)f.E, f.cols == 16 ? 4u : 3u, 4u};
    while ((h.S / 16) & ((1u << h.lgh) - 1u)) --h.lgh;  // S is a multiple of 64
    return h;
}

cudaError_t launch_key_bits(const KeyBits &k, const BitForm &f, BitScratch scratch, uint32_t *margin_bits,
                            uint32_t *nparts, cudaStream_t st) {
    const BitShape h = bit_shape(f);
    *nparts = (uint32_t)parts_count(f.L, f.E);
    const dim3 grid(*nparts, k.slots);
    cudaError_t e;
    if (f.E == 16 && k.pack) e = launch_chained(k_key_bits<16, true>, grid, kBitThreads, 0, st, k, h, scratch, margin_bits);
    else if (f.E == 16) e = launch_chained(k_key_bits<16, false>, grid, kBitThreads, 0, st, k, h, scratch, margin_bits);
    else if (k.pack) e = launch_chained(k_key_bits<8, true>, grid, kBitThreads, 0, st, k, h, scratch, margin_bits);
    else e = launch_chained(k_key_bits<8, false>, grid, kBitThreads, 0, st, k, h, scratch, margin_bits);
    return e;
}

cudaError_t launch_seed_bits(const uint64_t *seed, uint64_t n, uint64_t m, const BitForm &f, uint32_t *out,
                             const BitForm *packed, uint32_t *packed_out, cudaStream_t st) {
    const BitShape h0 = bit_shape(f), h1 = bit_shape(packed ? *packed : f);
    const uint64_t L1 = packed ? packed->L : 0;
    uint64_t x = parts_count(f.L, f.E);
    if (packed && parts_count(L1, f.E) > x) x = parts_count(L1, f.E);
    const dim3 grid((unsigned)x, packed ? 2 : 1);
    // an ordinary launch: the tables that the passes behind it read may be the kernel's before it
    if (f.E == 16) k_seed_bits<16><<<grid, kBitThreads, 0, st>>>(seed, n, m, h0, f.L, out, h1, L1, packed_out);
    else k_seed_bits<8><<<grid, kBitThreads, 0, st>>>(seed, n, m, h0, f.L, out, h1, L1, packed_out);
    return cudaGetLastError();
}

cudaError_t launch_block_bits(const BlockDev *blocks, uint32_t nblocks, const BitForm &f, BitScratch scratch,
                              uint32_t *margin_bits, uint32_t *nparts, cudaStream_t st) {
    const BitShape h = bit_shape(f);
    *nparts = (uint32_t)parts_count(f.L, f.E);
    const dim3 grid(*nparts, nblocks);
    cudaError_t e;
    if (f.E == 16) e = launch_chained(k_block_bits<16>, grid, kBitThreads, 0, st, blocks, h, f.L, scratch, margin_bits);
    else e = launch_chained(k_block_bits<8>, grid, kBitThreads, 0, st, blocks, h, f.L, scratch, margin_bits);
    return e;
}

// Round every float of x[0 .. count) to `bits` explicit significand bits (round to
// nearest, ties to even, on the float's encoding), as if the values had been stored in a
// format with that significand and FP32's exponent range.
__global__ void k_round_significand(float *__restrict__ x, uint64_t count, uint32_t bits) {
    const uint32_t drop = 23u - bits;
    const uint32_t half = (1u << (drop - 1)) - 1u, mask = ~((1u << drop) - 1u);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t u = __float_as_uint(x[i]);
        u = (u + half + ((u >> drop) & 1u)) & mask;
        x[i] = __uint_as_float(u);
    }
}

cudaError_t launch_round_significand(float *x, uint64_t count, uint32_t bits, cudaStream_t st) {
    if (bits == 0 || bits >= 23 || count == 0) return cudaSuccess;
    k_round_significand<<<1184, 256, 0, st>>>(x, count, bits);
    return cudaGetLastError();
}

}  // namespace pa
