// pa_launch.h -- host-side launchers of the pass kernels (declarations).
//
// Each launcher picks the kernel instance for its pass length, sets its dynamic
// shared memory and launches it on the given stream. Strided passes have
// power-of-two lengths 2^lgLEN; innermost passes have lengths RO * 2^lg with an
// odd factor RO in {1, 3, 5, 9} (smooth transform lengths). The definitions live
// in pa_launch.cuh, instantiated per arithmetic type (pa_f32.cu, pa_f64.cu,
// pa_zp.cu) and, for the odd innermost lengths, per (type, RO) (pa_*_r*.cu).
#pragma once

#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "fft_core.cuh"

namespace pa {

// Whether this thread's launch_chained makes ordinary launches: under stream capture. A graph launches its next kernel
// without delay, and CTAs that start early there crowd onto the SMs the running kernel leaves free instead of
// spreading over all of them. Two FP64 blocks of a class of length 262144 replay in 126 us with ordinary edges and in 236
// with overlapped ones (launched one by one: 150), eight of length 65536 in 114 and 189; batches from 2^21 values
// on take the same time either way (256 uneven blocks 9.99 and 9.96 ms), the smallest replay 2 us more (one FP32 block of
// 65536: 35.5 and 33.2). Overlapping only grids of at most 16, 32 or 64 CTAs gained nothing (one FP64 block of 65536
// 62.6, 79.1 and 79.1 us; with ordinary edges 62.6). The calls that can be captured set this for their duration: asking
// the stream at every launch cost a call of eight launches 1.2 us.
inline thread_local bool t_ordinary_launches = false;
struct LaunchesFor {
    bool before = t_ordinary_launches;
    explicit LaunchesFor(cudaStream_t st) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) cudaGetLastError();
        t_ordinary_launches = capture != cudaStreamCaptureStatusNone;
    }
    ~LaunchesFor() { t_ordinary_launches = before; }
    LaunchesFor(const LaunchesFor &) = delete;
    LaunchesFor &operator=(const LaunchesFor &) = delete;
};

// Launches a kernel whose first instruction is begin_after_previous (fft_core.cuh): its CTAs may
// start filling the SMs while the last CTAs of the stream's previous kernel still run.
template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kern)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st,
                           Args... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = t_ordinary_launches ? 0 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // reported here: the next <<<>>> launch must not find it again
    return e;
}

// Per-type kernel shape: E complex values per thread, COLS columns per CTA in
// the strided passes. FP64 halves both to keep registers and shared memory
// within one SM's budget.
template <typename T> struct Shape;
template <> struct Shape<float> { static constexpr int E = 16, COLS = 16; };
template <> struct Shape<double> { static constexpr int E = 8, COLS = 8; };
template <> struct Shape<Zp> { static constexpr int E = 8, COLS = 8; };
template <> struct Shape<Zq> { static constexpr int E = 16, COLS = 16; };
// Seed tables of the half-length form. Single precision forms w_N^k (a third table would be a fifth of the
// innermost pass's memory traffic, and that pass runs at 0.8 of the HBM rate on the 2^27-bit block);
// double precision, bound by the FP64 pipe, reads w_N^k O_s.
template <typename T> constexpr int kRealTables = std::is_same<T, float>::value ? 2 : 3;
template <typename T> constexpr bool kExact = std::is_same<T, Zp>::value || std::is_same<T, Zq>::value;
// Columns per CTA of a strided pass of length LEN: the types with 16 values per thread take 8 instead of 16 at
// LEN = 1024 (512 threads, two CTAs per SM instead of one).
constexpr int strided_cols_of(bool wide, int len) { return wide ? (len >= 1024 ? 8 : 16) : 8; }
template <typename T, int LEN>
constexpr int strided_cols() {
    static_assert(Shape<T>::COLS == (Shape<T>::E == 16 ? 16 : 8), "the width goes with the values per thread");
    return strided_cols_of(Shape<T>::E == 16, LEN);
}

// The kernels' view of a transform's tables at mem (layout y).
template <typename T>
TwTab<T> tw_tab(const TwLayout &y, const void *mem) {
    const cx<T> *m = static_cast<const cx<T> *>(mem);
    TwTab<T> t;
    t.hi = m + y.hi;
    t.lo = m + y.lo;
    t.B = y.B;
    for (int p = 0; p < 3; ++p) t.st[p] = m + y.st[p];
    for (int p = 0; p < 2; ++p) {
        t.fw[p] = PassTw<T>{m + y.pass[p].a, m + y.pass[p].c, m + y.pass[p].g};
        t.iv[p] = PassTw<T>{m + y.pass[p].ai, m + y.pass[p].ci, m + y.pass[p].gi};
        t.col[p] = m + y.pass[p].h;
    }
    return t;
}

// The complex passes take key bits as 0 / 2 and seed bits as +-2 (Enc in pa_kernels.cuh); products are scaled back by this.
constexpr double kSpecScale = 0.25;

// Supported pass lengths (log2).
constexpr int kMinLgStrided = 6, kMaxLgStrided = 10;
template <typename T> struct MaxLgMiddle;
template <> struct MaxLgMiddle<float> { static constexpr int v = 14; };
template <> struct MaxLgMiddle<double> { static constexpr int v = 13; };
template <> struct MaxLgMiddle<Zp> { static constexpr int v = 13; };
template <> struct MaxLgMiddle<Zq> { static constexpr int v = 13; };
constexpr int kMinLgMiddle = 6;

// Which elements of a rotated seed are inside the seed: element t holds a seed value iff t < M or
// t >= Z. For a thread's elements x + j*D (D = L / E, x < D), j < E, that is j < M/D + (x < M%D) or
// j >= Z/D + (x < Z%D).
struct SeedRange {
    uint32_t mr, zr;
    uint16_t mq, zq;  // at most E
    __host__ __device__ SeedRange() : mr(0), zr(0), mq(0), zq(0) {}
    __host__ __device__ SeedRange(uint64_t M, uint64_t Z, uint64_t D)
        : mr((uint32_t)(M % D)), zr((uint32_t)(Z % D)), mq((uint16_t)(M / D)), zq((uint16_t)(Z / D)) {}
    __device__ __forceinline__ uint32_t mask(uint32_t x) const {
        const uint32_t below = (1u << (mq + (x < mr))) - 1u, from = (1u << (zq + (x < zr))) - 1u;  // both counts <= 16
        return below | ~from;
    }
};

// Device-side block descriptor of the uneven batch.
struct BlockDev {
    const uint64_t *key;   // ceil(n/64) words
    const uint64_t *seed;  // ceil((n+m-1)/64) words
    uint64_t *out;         // ceil(m/64) words
    uint32_t n, m;         // at most 2^27
    uint32_t id;           // index of the block in the caller's list (popcount / margin slot)
    SeedRange in;          // seed window of the block in its class's transform
};
static_assert(sizeof(BlockDev) == 48, "counted into a served block's scratch, which callers cap to the byte");

// Scratch of the level-1 forward passes: transposed input bits (bits_words per slot) and partial
// popcounts (parts_count per slot).
struct BitScratch {
    uint32_t *bits = nullptr;
    uint2 *parts = nullptr;
};
inline uint64_t bits_words(uint64_t L, int E) { return L / (uint64_t)E; }
constexpr uint32_t kBitThreads = 128;  // threads of a transposition CTA, 16 columns of E rows each
inline uint64_t parts_count(uint64_t L, int E) { return (L / 16 / (uint64_t)E + kBitThreads - 1) / kBitThreads; }
// Bytes of scratch for `slots` slots, parts first.
inline size_t bit_scratch_bytes(uint64_t L, int E, uint64_t slots) {
    return (size_t)((parts_count(L, E) * slots * sizeof(uint2) + 255) / 256 * 256 + bits_words(L, E) * slots * sizeof(uint32_t));
}
inline BitScratch bit_scratch_at(void *mem, uint64_t L, int E, uint64_t slots) {
    BitScratch b;
    b.parts = static_cast<uint2 *>(mem);
    b.bits = reinterpret_cast<uint32_t *>(static_cast<unsigned char *>(mem) +
                                          (parts_count(L, E) * slots * sizeof(uint2) + 255) / 256 * 256);
    return b;
}

// Keys of a batch: slot p holds keys 2p (real part) and 2p+1, if any (imaginary part), or, with
// pack, key p's even and odd bits (a half-length transform). The transform input is key bits
// koff .. koff+n-1 (koff = m for the modified Toeplitz hash).
struct KeyBits {
    const uint64_t *keys = nullptr;
    uint32_t nkeys = 0, slots = 0;
    uint64_t kstride = 0, n = 0, koff = 0;
    bool pack = false;
};

// The first pass whose bits are transposed: length 2^lgLEN of a length-L transform, E values per
// thread, cols columns per CTA.
struct BitForm {
    uint64_t L;
    int lgLEN, E, cols;
};
template <typename T>
BitForm bit_form(int lgLEN, uint64_t L) {
    return BitForm{L, lgLEN, Shape<T>::E, strided_cols_of(Shape<T>::E == 16, 1 << lgLEN)};
}

// Transpose input bits (layout: see "Input bits" in pa_kernels.cuh). The key forms also leave
// partial popcounts (*nparts per slot) and zero the margins of their keys (blocks: margin_bits[id]).
cudaError_t launch_key_bits(const KeyBits &k, const BitForm &f, BitScratch scratch, uint32_t *margin_bits,
                            uint32_t *nparts, cudaStream_t st);
// packed (or null): also for the half-length form, a length-packed->L transform whose element t holds
// rotated positions 2t and 2t+1.
cudaError_t launch_seed_bits(const uint64_t *seed, uint64_t n, uint64_t m, const BitForm &f, uint32_t *out,
                             const BitForm *packed, uint32_t *packed_out, cudaStream_t st);
cudaError_t launch_block_bits(const BlockDev *blocks, uint32_t nblocks, const BitForm &f, BitScratch scratch,
                              uint32_t *margin_bits, uint32_t *nparts, cudaStream_t st);

// Round x[0 .. count) in place to `bits` explicit significand bits (1 <= bits <= 22; other
// values leave x as it is): the storage-precision study of pa_plan_set_storage_bits.
cudaError_t launch_round_significand(float *x, uint64_t count, uint32_t bits, cudaStream_t st);

// What the level-1 forward pass transforms: slots of keys, a seed, or the blocks of a class. The pass
// also adds up the partial popcounts of its slots: popc[slot * ppk] (+1 for the imaginary part's
// key; ppk = 1: both parts are one key's), or popc[id] of a block.
enum class In { KEYS, SEED, BLOCKS };
struct FwdArgs {
    const uint32_t *bits;   // L / E words per slot
    const uint2 *parts;     // popcounts (real, imaginary part): nparts per slot
    uint32_t nparts, ppk, nkeys;
    uint32_t *popc;
    SeedRange re, im;       // SEED
    const BlockDev *blocks; // BLOCKS
};
template <typename T>
cudaError_t launch_fwd(int lgLEN, In kind, const FwdArgs &in, uint32_t slots, cx<T> *W, uint64_t L, TwTab<T> tw,
                       cudaStream_t st);

// Transpose the bits of keys or blocks for launch_fwd, which takes *in.
template <typename T>
cudaError_t prepare_keys(int lgLEN, const KeyBits &k, uint64_t L, BitScratch scratch, uint32_t *popc,
                         uint32_t *margin_bits, cudaStream_t st, FwdArgs *in) {
    *in = FwdArgs();
    in->bits = scratch.bits;
    in->parts = scratch.parts;
    in->ppk = k.pack ? 1 : 2;
    in->nkeys = k.nkeys;
    in->popc = popc;
    return launch_key_bits(k, bit_form<T>(lgLEN, L), scratch, margin_bits, &in->nparts, st);
}
template <typename T>
cudaError_t prepare_blocks(int lgLEN, const BlockDev *blocks, uint32_t nblocks, uint64_t L, BitScratch scratch,
                           uint32_t *popc, uint32_t *margin_bits, cudaStream_t st, FwdArgs *in) {
    *in = FwdArgs();
    in->bits = scratch.bits;
    in->parts = scratch.parts;
    in->popc = popc;
    in->blocks = blocks;
    return launch_block_bits(blocks, nblocks, bit_form<T>(lgLEN, L), scratch, margin_bits, &in->nparts, st);
}
// The first pass's input from transposed seed bits. Rotated position t holds seed bit t + n - 1 (mod
// the cyclic length): a seed value for t < m or t > length - n.
template <typename T>
FwdArgs seed_args(const uint32_t *bits, uint64_t n, uint64_t m, bool pack, uint64_t L) {
    FwdArgs in{};
    in.bits = bits;
    const uint64_t D = L / Shape<T>::E;
    if (pack) {
        in.re = SeedRange((m + 1) / 2, (2 * L - n + 2) / 2, D);
        in.im = SeedRange(m / 2, (2 * L - n + 1) / 2, D);
    } else {
        in.re = SeedRange(m, L - n + 1, D);
        in.im = SeedRange(0, L, D);
    }
    return in;
}
// S: innermost length (the stride of the middle strided pass). near_roots: the forward pass's stages read w^4 (entry_powers).
template <typename T>
cudaError_t launch_mid(int lgLEN, bool inverse, cx<T> *W, uint64_t L, uint32_t S, uint32_t pairs, TwTab<T> tw,
                       cudaStream_t st, bool near_roots = false);
// Innermost pass of length ro * 2^lg. mode 0: the fused convolution step; mode 1:
// the seed spectrum.
template <typename T>
cudaError_t launch_middle(int ro, int lg, int mode, cx<T> *W, cx<T> *spec, uint64_t L, uint32_t pairs, TwTab<T> tw,
                          cx<T> scale, cudaStream_t st);
template <typename T, int RO>
cudaError_t launch_middle_odd(int lg, int mode, cx<T> *W, cx<T> *spec, uint64_t L, uint32_t pairs, TwTab<T> tw,
                              cx<T> scale, cudaStream_t st);

// Limits of the odd innermost lengths RO * 2^lg: a CTA has RO * 2^lg / E threads
// (at most 1024, or 512 per row for the two-row split kernel).
constexpr int kMinLgOdd = 7, kMaxLgOdd = 11;
template <typename T>
constexpr bool odd_inner_ok(int ro, int lg, bool split) {
    return lg >= kMinLgOdd && lg <= kMaxLgOdd && (long long)ro * (1ll << lg) / Shape<T>::E <= (split ? 512 : 1024);
}
// Level-1 inverse pass with the bit output. With xkeys, output bit i of key k is
// XORed with bit i of xkeys + k*xstride (the identity block of the modified hash).
// With ctl != nullptr (three device words, zero before the first launch: error bits,
// tile ticket, CTAs done), FP32 pairs with pass lengths up to 256 run the persistent
// TMA-staged kernel; a copy wait there that runs out of time sets bit 0 of ctl[0].
// expire_ns != 0 (test hook) makes that kernel copy nothing and let its wait run out.
template <typename T>
cudaError_t launch_inv_bits(int lgLEN, const cx<T> *W, uint64_t L, uint64_t m, uint32_t nkeys,
                            const uint32_t *popc, uint32_t *margin_bits, uint64_t *out, uint64_t ostride,
                            uint32_t pairs, TwTab<T> tw, cudaStream_t st, const uint64_t *xkeys = nullptr,
                            uint64_t xstride = 0, bool pack = false, uint32_t *ctl = nullptr,
                            uint32_t expire_ns = 0);
// Whether launch_inv_bits runs the TMA-staged kernel for this type and pass length.
constexpr bool inv_bits_staged(uint64_t elem_bytes, int lgLEN) { return elem_bytes == 8 && lgLEN <= 8; }

// Tiled-copy descriptor of a row-major array of rows x cols 8-byte elements at base, copied
// in boxes of box_cols x box_rows (the cuTensorMapEncodeTiled encoder, resolved from the
// driver at run time). false if the driver offers no encoder or rejects the layout.
bool encode_tile_map(CUtensorMap *map, const void *base, uint64_t cols, uint64_t rows, uint32_t box_cols,
                     uint32_t box_rows);

// ---- uneven batch (complex arithmetic only: the Eq. 5-10 split needs conjugation) ----
template <typename T> struct MaxLgSplit;
template <> struct MaxLgSplit<float> { static constexpr int v = 13; };
template <> struct MaxLgSplit<double> { static constexpr int v = 12; };

template <typename T>
cudaError_t launch_middle_split(int ro, int lg, cx<T> *Wf, cx<T> *Wi, uint64_t L, uint32_t nblocks,
                                uint32_t lgL1, uint32_t lgM, TwTab<T> tw, cudaStream_t st);
template <typename T, int RO>
cudaError_t launch_middle_split_odd(int lg, cx<T> *Wf, cx<T> *Wi, uint64_t L, uint32_t nblocks, uint32_t lgL1,
                                    uint32_t lgM, TwTab<T> tw, cudaStream_t st);
template <typename T>
cudaError_t launch_inv_bits_blocks(int lgLEN, const cx<T> *Wi, uint64_t L, const BlockDev *blocks, uint32_t nblocks,
                                   const uint32_t *popc, uint32_t *margin_bits, TwTab<T> tw, cudaStream_t st);

// ---- single keys in half-length transforms (complex arithmetic only) ----
// Innermost pass of length ro * 2^lg over a length-N slot (slots of N elements from W):
// mode 0 multiplies with the seed tables (kRealTables * N values: E_s, O_s, w_N^k O_s, times 1/N) and
// transforms back; mode 1 builds those tables from the packed seed's transform (scale 1/N).
template <typename T>
cudaError_t launch_middle_real(int ro, int lg, int mode, cx<T> *W, cx<T> *tabs, uint64_t N, uint32_t lgL1,
                               uint32_t lgM, TwTab<T> tw, T scale, uint32_t slots, cudaStream_t st);
template <typename T, int RO>
cudaError_t launch_middle_real_odd(int lg, int mode, cx<T> *W, cx<T> *tabs, uint64_t N, uint32_t lgL1, uint32_t lgM,
                                   TwTab<T> tw, T scale, uint32_t slots, cudaStream_t st);

}  // namespace pa
