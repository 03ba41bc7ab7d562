// zq.cuh -- arithmetic modulo the prime q = 7 * 2^26 + 1 for the exact transform of lengths up
// to 2^26.
//
// The hash only needs the convolution's counts c_i <= n exactly (y_i = c_i mod 2), so any prime above
// n with roots of unity of the transform's order gives the same bits as the 64-bit prime of
// zp.cuh: q = 469762049 > 2^27 >= n, and 2^26 divides q - 1. A 64-bit element holds two residues, one per
// key of a pair. Products with a known multiplier w take three 32-bit multiplications (Shoup's
// method: with w' = floor(w 2^32 / q), b w - floor(b w' / 2^32) q lies in [0, 2q) for any b < 2^32),
// and butterflies keep their values in [0, 4q) with one conditional subtraction (Harvey, "Faster
// arithmetic for number-theoretic transforms", 2014; 4q < 2^32). The 64-bit prime's product and its
// reduction take about 20 instructions, its canonical additions about 8.
#pragma once

#include <cstdint>

namespace pa {

struct Zq {};  // tag type: two residues modulo q per element

constexpr uint32_t kQ = 469762049u;  // 7 * 2^26 + 1, prime; 3 generates the multiplicative group
constexpr int kMaxLgZq = 26;
static_assert(kQ > (1u << 27), "above every count of a key of up to 2^27 bits");
static_assert((kQ - 1) % (1u << kMaxLgZq) == 0, "roots of unity of order 2^kMaxLgZq");
static_assert(4ull * kQ <= 1ull << 32, "lazy residues below 4q fit a word");

__host__ __device__ constexpr uint32_t zq_mul(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b % kQ); }
__host__ __device__ constexpr uint32_t zq_pow(uint32_t a, uint64_t e) {
    uint32_t r = 1;
    for (; e; e >>= 1) {
        if (e & 1) r = zq_mul(r, a);
        a = zq_mul(a, a);
    }
    return r;
}
// w' of a multiplier w < q.
__host__ __device__ constexpr uint32_t zq_quotient(uint32_t w) { return (uint32_t)(((uint64_t)w << 32) / kQ); }
// w_32^j of the root w_32 = 3^((q-1)/32) (the tables' w_L = 3^((q-1)/L): one root system).
__host__ __device__ constexpr uint32_t zq_root32(int j) { return zq_pow(zq_pow(3u, (kQ - 1) / 32), (uint64_t)j); }

// Multipliers are pairs (w, w'), data elements pairs of residues (key a, key b); both are uint2.
template <> struct Arith<Zq> {
    using E = uint2;
    static __device__ __forceinline__ uint32_t below2q(uint32_t x) { return min(x, x - 2u * kQ); }  // [0, 4q) -> [0, 2q)
    static __device__ __forceinline__ uint32_t product(uint32_t b, uint32_t w, uint32_t wq) {       // in [0, 2q)
        return b * w - __umulhi(b, wq) * kQ;
    }
    static __device__ __forceinline__ E mul(E b, E w) { return make_uint2(product(b.x, w.x, w.y), product(b.y, w.x, w.y)); }
    // (a, b) -> (a + w b, a - w b); t = w b in [0, 2q)
    static __device__ __forceinline__ void combine(E &a, E &b, E t) {
        const uint32_t ax = below2q(a.x), ay = below2q(a.y);
        b = make_uint2(ax - t.x + 2u * kQ, ay - t.y + 2u * kQ);
        a = make_uint2(ax + t.x, ay + t.y);
    }
    static __device__ __forceinline__ void bfly(E &a, E &b, E w) { combine(a, b, mul(b, w)); }
    static __device__ __forceinline__ void bfly1(E &a, E &b) { combine(a, b, make_uint2(below2q(b.x), below2q(b.y))); }
    // the value of a residue in [0, 4q)
    static __device__ __forceinline__ uint32_t canonical(uint32_t x) {
        x = below2q(x);
        return min(x, x - kQ);
    }
    // the multiplier (w, w') of the first residue
    static __device__ __forceinline__ E multiplier(E v) {
        const uint32_t w = canonical(v.x);
        return make_uint2(w, zq_quotient(w));
    }
};

}  // namespace pa
