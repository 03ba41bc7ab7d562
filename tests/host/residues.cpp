// Arith<Zq> as the kernels use it, on given operands. Reads lines "b w" (a residue below 2^32, a multiplier below q) and
// "a b w" and prints the results for Python to check: first the constants, then for every line the multiplier's
// quotient, product, butterfly and canonical value.
#include <cinttypes>
#include <cstdio>

#include "fft_core.cuh"

using namespace pa;

int main() {
    std::printf("%u %d %u\n", kQ, kMaxLgZq, zq_root32(1));
    uint32_t a, b, w;
    while (std::scanf("%" SCNu32 " %" SCNu32 " %" SCNu32, &a, &b, &w) == 3) {
        const uint2 m = make_uint2(w, zq_quotient(w));
        const uint2 t = Arith<Zq>::mul(make_uint2(b, a), m);
        uint2 u = make_uint2(a, a), v = make_uint2(b, b), x = make_uint2(a, a), y = make_uint2(b, b);
        Arith<Zq>::bfly(u, v, m);
        Arith<Zq>::bfly1(x, y);
        const uint2 back = Arith<Zq>::multiplier(make_uint2(a, 0));
        std::printf("%u %u %u %u %u %u %u %u %u\n", t.x, t.y, u.x, v.x, x.x, y.x, Arith<Zq>::canonical(a), back.x, back.y);
    }
}
