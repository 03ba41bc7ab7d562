// fft_core.cuh -- device building blocks of the FFT passes.
//
// The hash is evaluated through the convolution theorem (paper Eq. 4). A long
// transform of length L is split into passes of short transforms in the spirit
// of the paper's Algorithm 1 (row FFTs, twiddle factors W[i*j], column FFTs).
// Unlike Algorithm 1 the passes never transpose: each forward pass is a
// decimation-in-frequency step that leaves the spectrum in digit-reversed
// order, the pointwise product does not care about order (the seed spectrum
// is stored in the same order), and the inverse passes undo the steps in
// reverse so the convolution comes out in natural order. This is the GPU form
// of Algorithm 2's observation that the spectrum's order is irrelevant to PA,
// without Algorithm 2's permutation of the final key.
//
// Inside a CTA every thread of a short transform of length LEN holds E complex values in
// registers, does radix-R butterflies (R <= E) on them, and exchanges through shared memory
// between stages, in place.
// A CTA works on COLS transforms at once, interleaved column-wise in shared
// memory, so that a warp's global accesses touch COLS consecutive elements.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "tables.cuh"

namespace pa {

// First statement of every pass kernel but the staged last pass (they are launched with launch_chained): waits until the stream's
// previous kernel has finished and its writes are visible, then lets the next kernel start once
// every CTA of this one has got here. A chain of small launches loses the launch latency between its
// kernels, and a large one's first CTAs fill the SMs that the last wave of the kernel before leaves
// empty. What earlier kernels of the stream write is read with fresh() or plain loads, never as
// constant memory (__ldg, const __restrict__): the compiler and the assembler move constant loads
// above the wait (then a key read another launch's popcount, and escalated without need), and the
// pointers pass through the wait for the same reason.
template <typename... P>
__device__ __forceinline__ void begin_after_previous(P &...p) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const auto behind = [](auto &q) { asm volatile("" : "+l"(q)::"memory"); };
    (behind(p), ...);
}
// A load from L2, past L1.
template <typename V> __device__ __forceinline__ V fresh(const V *p) { return __ldcg(p); }

// Element arithmetic of the transforms. Arith<float> / Arith<double> work on
// complex numbers (x = real, y = imaginary); Arith<Zp> (zp.cuh) on residues
// modulo the prime p = 2^64 - 2^32 + 1. The FFT engine below only uses add,
// sub, mul, the in-register roots rot32 and the table twiddles omega.
template <typename T> struct Arith;
template <typename T> using cx = typename Arith<T>::E;

// cos(pi*j/16), j = 0..8, to 20 significant digits.
__host__ __device__ constexpr double cos_pi16(int j) {
    return j == 0   ? 1.0
           : j == 1 ? 0.98078528040323044913
           : j == 2 ? 0.92387953251128675613
           : j == 3 ? 0.83146961230254523708
           : j == 4 ? 0.70710678118654752440
           : j == 5 ? 0.55557023301960222474
           : j == 6 ? 0.38268343236508977173
           : j == 7 ? 0.19509032201612826785
                    : 0.0;
}
// cos and sin of 2*pi*j/32 for 0 <= j < 16.
__host__ __device__ constexpr double cos32(int j) { return j <= 8 ? cos_pi16(j) : -cos_pi16(16 - j); }
__host__ __device__ constexpr double sin32(int j) { return j <= 8 ? cos_pi16(8 - j) : cos_pi16(j - 8); }

// In-register DFT of RO = 3, 5 or 9 complex values (odd factors of smooth
// transform lengths), natural order in and out. Forward roots w_R = exp(-2 pi i / R).
// Constants: cos/sin of 2 pi j / R to 20 significant digits.
template <typename T, bool INV>
__device__ __forceinline__ void dft3(cx<T> &x0, cx<T> &x1, cx<T> &x2) {
    constexpr T s3 = (T)0.86602540378443864676;  // sin(2 pi / 3)
    const cx<T> a = Arith<T>::add(x1, x2), b = Arith<T>::sub(x1, x2);
    const cx<T> c = Arith<T>::mk(x0.x - (T)0.5 * a.x, x0.y - (T)0.5 * a.y);
    // forward: y1 = c - i s3 b, y2 = c + i s3 b (inverse swaps the signs)
    const T sb_x = (INV ? -s3 : s3) * b.x, sb_y = (INV ? -s3 : s3) * b.y;
    x0 = Arith<T>::add(x0, a);
    x1 = Arith<T>::mk(c.x + sb_y, c.y - sb_x);
    x2 = Arith<T>::mk(c.x - sb_y, c.y + sb_x);
}

template <typename T, bool INV>
__device__ __forceinline__ void dft5(cx<T> *x) {
    constexpr T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;  // cos(2pi/5), cos(4pi/5)
    constexpr T s1 = (T)0.95105651629515357212, s2 = (T)0.58778525229247312917;   // sin(2pi/5), sin(4pi/5)
    const cx<T> a1 = Arith<T>::add(x[1], x[4]), b1 = Arith<T>::sub(x[1], x[4]);
    const cx<T> a2 = Arith<T>::add(x[2], x[3]), b2 = Arith<T>::sub(x[2], x[3]);
    const cx<T> x0 = x[0];
    // real-coefficient parts
    const cx<T> p1 = Arith<T>::mk(x0.x + c1 * a1.x + c2 * a2.x, x0.y + c1 * a1.y + c2 * a2.y);
    const cx<T> p2 = Arith<T>::mk(x0.x + c2 * a1.x + c1 * a2.x, x0.y + c2 * a1.y + c1 * a2.y);
    // q1 = s1 b1 + s2 b2, q2 = s2 b1 - s1 b2; y1 = p1 - i q1, y4 = p1 + i q1, y2 = p2 - i q2, y3 = p2 + i q2
    T q1x = s1 * b1.x + s2 * b2.x, q1y = s1 * b1.y + s2 * b2.y;
    T q2x = s2 * b1.x - s1 * b2.x, q2y = s2 * b1.y - s1 * b2.y;
    if (INV) { q1x = -q1x; q1y = -q1y; q2x = -q2x; q2y = -q2y; }
    x[0] = Arith<T>::add(x0, Arith<T>::add(a1, a2));
    x[1] = Arith<T>::mk(p1.x + q1y, p1.y - q1x);
    x[4] = Arith<T>::mk(p1.x - q1y, p1.y + q1x);
    x[2] = Arith<T>::mk(p2.x + q2y, p2.y - q2x);
    x[3] = Arith<T>::mk(p2.x - q2y, p2.y + q2x);
}

// x * w9^j for the radix-9 internal twiddles (j in 1, 2, 4).
template <typename T, bool INV>
__device__ __forceinline__ cx<T> rot9(cx<T> x, int j) {
    const T c = j == 1 ? (T)0.76604444311897803520 : j == 2 ? (T)0.17364817766693034885 : (T)-0.93969262078590838405;
    const T sn = j == 1 ? (T)0.64278760968653932632 : j == 2 ? (T)0.98480775301220805936 : (T)0.34202014332566873304;
    const T s = INV ? sn : -sn;
    return Arith<T>::mk(x.x * c - x.y * s, x.x * s + x.y * c);
}

template <typename T, int RO, bool INV>
__device__ __forceinline__ void dft_odd(cx<T> *x) {
    if constexpr (RO == 3) {
        dft3<T, INV>(x[0], x[1], x[2]);
    } else if constexpr (RO == 5) {
        dft5<T, INV>(x);
    } else {
        static_assert(RO == 9, "odd radix must be 3, 5 or 9");
        // 9 = 3 x 3: x[3m + r] -> DFT3 over m for each r, twiddle w9^{r k1}, DFT3 over r; X[k1 + 3 k2]
        cx<T> a[9];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            cx<T> u0 = x[r], u1 = x[3 + r], u2 = x[6 + r];
            dft3<T, INV>(u0, u1, u2);
            a[3 * r + 0] = u0;  // k1 = 0
            a[3 * r + 1] = r ? rot9<T, INV>(u1, r) : u1;
            a[3 * r + 2] = r ? rot9<T, INV>(u2, 2 * r) : u2;
        }
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            cx<T> v0 = a[k1], v1 = a[3 + k1], v2 = a[6 + k1];
            dft3<T, INV>(v0, v1, v2);
            x[k1] = v0;
            x[k1 + 3] = v1;
            x[k1 + 6] = v2;
        }
    }
}

// cos and sin of 2 pi a / b in double precision at compile time: the angle is
// reduced to [0, pi/4] by the symmetries of the circle, then summed as a Taylor
// series (terms up to x^27 / 27!, below 1e-30 for |x| <= pi/4).
__host__ __device__ constexpr double taylor_sin(double x) {
    double term = x, sum = x;
    for (int k = 1; k <= 13; ++k) {
        term *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double taylor_cos(double x) {
    double term = 1.0, sum = 1.0;
    for (int k = 1; k <= 13; ++k) {
        term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
        sum += term;
    }
    return sum;
}
constexpr double kPi = 3.14159265358979323846264338327950288;
// cos (SIN = false) or sin (SIN = true) of 2 pi a / b for 0 <= a < b: with 4a = q b + r,
// the angle is q pi/2 + psi, psi = (pi/2) r / b; psi above pi/4 is taken as
// pi/2 - (pi/2)(b - r)/b so the series always runs on [0, pi/4].
__host__ __device__ constexpr double trig_frac(int a, int b, bool want_sin) {
    const int q = (4 * a) / b, r = (4 * a) % b;
    const bool high = 2 * r > b;
    const double psi = (kPi / 2.0) * (double)(high ? b - r : r) / (double)b;
    const double c0 = high ? taylor_sin(psi) : taylor_cos(psi);
    const double s0 = high ? taylor_cos(psi) : taylor_sin(psi);
    // rotate (c0, s0) by q quarter turns
    const double c = q == 0 ? c0 : q == 1 ? -s0 : q == 2 ? -c0 : s0;
    const double sn = q == 0 ? s0 : q == 1 ? c0 : q == 2 ? -s0 : -c0;
    return want_sin ? sn : c;
}
__host__ __device__ constexpr double cos_frac(int a, int b) { return trig_frac(a, b, false); }
__host__ __device__ constexpr double sin_frac(int a, int b) { return trig_frac(a, b, true); }

// Twiddle tables of a length-L transform as the kernels take them (layout: tables.cuh).
// Complex roots are exp(-2*pi*i/L), the inverse transform takes the conjugates; the exact
// transform has tables of its own for the inverse passes.
template <typename T> struct PassTw {
    const cx<T> *a;  // a[tq * (S / COLS) + blk]
    const cx<T> *c;  // c[tq * COLS + col]
    const cx<T> *g;  // g[u]
};
template <typename T> struct TwTab {
    const cx<T> *hi;
    const cx<T> *lo;
    uint32_t B;              // w_L^e = hi[e >> B] * lo[e & (2^B - 1)]
    const cx<T> *st[3];      // stage tables: first pass, middle strided pass, innermost pass
    PassTw<T> fw[2], iv[2];  // pass tables of the first and the middle strided pass (iv: exact transform)
    const cx<T> *col[2];     // their inverse column tables (complex arithmetic)
};

template <typename T> struct ComplexArith {
    using E = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
    static __device__ __forceinline__ E mk(T x, T y) { E r; r.x = x; r.y = y; return r; }
    static __device__ __forceinline__ E add(E a, E b) { return mk(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ E sub(E a, E b) { return mk(a.x - b.x, a.y - b.y); }
    static __device__ __forceinline__ E mul(E a, E b) { return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
    // k*a + c for a real k
    static __device__ __forceinline__ E fmak(T k, E a, E c) { return mk(k * a.x + c.x, k * a.y + c.y); }
    static __device__ __forceinline__ E mulk(T k, E a) { return mk(k * a.x, k * a.y); }
    // (a, b) -> (a + w b, a - w b), w = c + i s: six fused multiply-adds, the difference
    // as 2a - (a + w b).
    static __device__ __forceinline__ E add_mul(E a, E b, T c, T s) {
        const E t = fmak(c, b, a);
        return mk(fma(-s, b.y, t.x), fma(s, b.x, t.y));
    }
    static __device__ __forceinline__ void bfly(E &a, E &b, T c, T s) {
        const E p = add_mul(a, b, c, s);
        b = mk(fma((T)2, a.x, -p.x), fma((T)2, a.y, -p.y));
        a = p;
    }
    template <bool INV> static __device__ __forceinline__ E omega(const TwTab<T> &t, uint32_t e) {
        E a = __ldg(t.hi + (e >> t.B));
        E b = __ldg(t.lo + (e & ((1u << t.B) - 1u)));
        E w = mul(a, b);
        if (INV) w.y = -w.y;
        return w;
    }
};
// FP32 complex add/sub as one packed f32x2 instruction each (sm_100+ packed FP32):
// the (re, im) pair sits in one 64-bit register pair.
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
// d = a * b + c on both lanes of an f32x2 pair (one packed instruction).
__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "mov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\t"
        "mov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
template <> struct Arith<float> : ComplexArith<float> {
    static __device__ __forceinline__ E add(E a, E b) { return f2_add(a, b); }
    static __device__ __forceinline__ E sub(E a, E b) { return f2_sub(a, b); }
    static __device__ __forceinline__ E fmak(float k, E a, E c) { return f2_fma(make_float2(k, k), a, c); }
    static __device__ __forceinline__ E mulk(float k, E a) { return f2_mul(make_float2(k, k), a); }
    static __device__ __forceinline__ E add_mul(E a, E b, float c, float s) {
        const E t = fmak(c, b, a);
        return mk(fmaf(-s, b.y, t.x), fmaf(s, b.x, t.y));
    }
    static __device__ __forceinline__ void bfly(E &a, E &b, float c, float s) {
        const E p = add_mul(a, b, c, s);
        b = mk(fmaf(2.f, a.x, -p.x), fmaf(2.f, a.y, -p.y));
        a = p;
    }
};
template <> struct Arith<double> : ComplexArith<double> {};

}  // namespace pa

#include "zp.cuh"
#include "zq.cuh"

namespace pa {

// f(0), ..., f(N-1) with compile-time arguments.
template <int N, int I = 0, class F>
__device__ __forceinline__ void static_for(F &&f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<N, I + 1>(f);
    }
}

// (a, b) -> (a + w b, a - w b) for w = w_32^J (forward root; the inverse uses the conjugate),
// the whole and quarter turns without multiplications.
template <typename T, int J, bool INV>
__device__ __forceinline__ void bfly32(cx<T> &a, cx<T> &b) {
    if constexpr (std::is_same<T, Zq>::value) {
        constexpr uint32_t w = zq_root32(INV ? (32 - J) % 32 : J), wq = zq_quotient(w);
        if constexpr (J == 0) {
            Arith<Zq>::bfly1(a, b);
        } else {
            Arith<Zq>::bfly(a, b, make_uint2(w, wq));
        }
    } else if constexpr (J == 0) {
        const cx<T> p = Arith<T>::add(a, b);
        b = Arith<T>::sub(a, b);
        a = p;
    } else if constexpr (J == 8) {  // w = -i (inverse: i)
        const cx<T> r = INV ? Arith<T>::mk(-b.y, b.x) : Arith<T>::mk(b.y, -b.x);
        b = Arith<T>::mk(a.x - r.x, a.y - r.y);
        a = Arith<T>::mk(a.x + r.x, a.y + r.y);
    } else {
        Arith<T>::bfly(a, b, (T)cos32(J), INV ? (T)sin32(J) : (T)-sin32(J));
    }
}

template <typename T, int R, bool INV, int LEVEL, int P>
__device__ __forceinline__ void dft_const_sub(cx<T> *v) {
    if constexpr (P < (1 << LEVEL)) {
        constexpr int h = R >> (LEVEL + 1), base = bitrev(P, LEVEL) * (R >> LEVEL);
#pragma unroll
        for (int r = 0; r < h; ++r) bfly32<T, (P << (4 - LEVEL)), INV>(v[base + r], v[base + r + h]);
        dft_const_sub<T, R, INV, LEVEL, P + 1>(v);
    }
}
template <typename T, int R, bool INV, int LEVEL>
__device__ __forceinline__ void dft_const(cx<T> *v) {
    if constexpr ((1 << LEVEL) < R) {
        dft_const_sub<T, R, INV, LEVEL, 0>(v);
        dft_const<T, R, INV, LEVEL + 1>(v);
    }
}

template <typename T, int R>
__device__ __forceinline__ void bitrev_regs(cx<T> *v) {
    cx<T> t[R];
#pragma unroll
    for (int k = 0; k < R; ++k) t[k] = v[bitrev(k, ilog2(R))];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = t[k];
}

// In-register DFT of R = 2^s <= 32 values, natural order in and out. Complex: radix-2
// decimation in time; level l combines the halves of the 2^l sub-transforms p (outputs
// k = p mod 2^l) with the root w_{2^(l+1)}^p, which the butterfly's multiply-adds absorb.
// Exact transform: decimation in frequency with the shift roots.
// FROM > 0: the values are those of the first FROM levels already (complex).
template <typename T, int R, bool INV, int FROM = 0>
__device__ __forceinline__ void dft(cx<T> *v) {
    static_assert(R >= 1 && R <= 32 && (R & (R - 1)) == 0, "radix must be a power of two <= 32");
    if constexpr (R > 1) {
        if constexpr (std::is_same<T, Zp>::value) {
#pragma unroll
            for (int len = R; len >= 2; len >>= 1) {
#pragma unroll
                for (int b = 0; b < R; b += len) {
#pragma unroll
                    for (int j = 0; j < len / 2; ++j) {
                        cx<T> a = v[b + j], c = v[b + j + len / 2];
                        v[b + j] = Arith<T>::add(a, c);
                        v[b + j + len / 2] = Arith<T>::template rot32<INV>(Arith<T>::sub(a, c), j * (32 / len));
                    }
                }
            }
        } else {
            dft_const<T, R, INV, FROM>(v);
        }
        bitrev_regs<T, R>(v);
    }
}

// Two consecutive table entries (a row pair).
__device__ __forceinline__ void load_pair(const float2 *p, float2 &a, float2 &b) {
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    a = make_float2(q.x, q.y);
    b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void load_pair(const double2 *p, double2 &a, double2 &b) {
    a = __ldg(p);
    b = __ldg(p + 1);
}
__device__ __forceinline__ void load_pair(const unsigned long long *p, unsigned long long &a, unsigned long long &b) {
    const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2 *>(p));
    a = q.x;
    b = q.y;
}
template <typename T>
constexpr Rows kRows = std::is_same<T, Zp>::value      ? Rows::EXACT
                       : std::is_same<T, Zq>::value    ? Rows::LEVELS
                       : std::is_same<T, float>::value ? Rows::SINGLE
                                                       : Rows::DOUBLE;
// Multipliers a thread holds for a radix-R stage.
template <typename T>
constexpr int multipliers(int R) { return is_complex(kRows<T>) ? level_rows(R) : R - 1; }
__device__ __forceinline__ void load_pair(const uint2 *p, uint2 &a, uint2 &b) {
    const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p));
    a = make_uint2(q.x, q.y);
    b = make_uint2(q.z, q.w);
}
// The ROWS multipliers at index k of a table of P butterflies.
template <typename T, int ROWS, int P>
__device__ __forceinline__ void load_rows(const cx<T> *tab, uint32_t k, cx<T> *w) {
    if constexpr (ROWS == 1) {
        w[0] = __ldg(tab + k);
    } else {
        const cx<T> *t = tab + 2 * k;
#pragma unroll
        for (int r = 0; r < ROWS; r += 2) {
            if (r + 1 < ROWS) {
                load_pair(t + r * P, w[r], w[r + 1]);
            } else {
                w[r] = __ldg(t + r * P);
            }
        }
    }
}

// w^2 of a root of unity: (1 - 2 s^2, 2 s c).
template <typename T>
__device__ __forceinline__ cx<T> square_root_of_unity(cx<T> w) {
    const T t = w.y + w.y;
    return Arith<T>::mk(fma(-t, w.y, (T)1), t * w.x);
}
// w * w_N^J for a compile-time turn.
template <typename T, int N, int J>
__device__ __forceinline__ cx<T> turn(cx<T> w) {
    if constexpr (J % N == 0) {
        return w;
    } else {
        constexpr T c = (T)cos_frac(J % N, N), s = -(T)sin_frac(J % N, N);
        const cx<T> t = Arith<T>::mulk(c, w);
        return Arith<T>::mk(fma(-s, w.y, t.x), fma(s, w.x, t.y));
    }
}
// m[] = the multipliers of the levels of a radix-R stage (dft_rows) for the root pw[l] * w_TURN_N^(TURN * R/2^(l+1))
// of level l, where pw[l] = w^(R / 2^(l+1)): rows p of a level are further turns by w_{2^(l+1)}^p.
template <typename T, int R, int N, int TURN, int LEVEL = 0, int P = 0>
__device__ __forceinline__ void level_multipliers(const cx<T> *pw, cx<T> *m) {
    if constexpr ((1 << LEVEL) < R) {
        constexpr int half = LEVEL ? 1 << (LEVEL - 1) : 1, h = R >> (LEVEL + 1);
        if constexpr (P < half) {
            // exponent of w_M, M = N * 2^(LEVEL+1): TURN h / N + P / 2^(LEVEL+1)
            constexpr int M = N << (LEVEL + 1);
            m[LEVEL ? half + P : 0] = turn<T, M, (TURN * h << (LEVEL + 1)) + P * N>(pw[LEVEL]);
            level_multipliers<T, R, N, TURN, LEVEL, P + 1>(pw, m);
        } else {
            level_multipliers<T, R, N, TURN, LEVEL + 1, 0>(pw, m);
        }
    }
}
// pw[l] = w^(R / 2^(l+1)), l = log2 R - 1 .. 0.
template <typename T, int R>
__device__ __forceinline__ void level_powers(cx<T> w, cx<T> *pw) {
#pragma unroll
    for (int l = ilog2(R) - 1; l >= 0; --l) {
        pw[l] = w;
        if (l) w = square_root_of_unity<T>(w);
    }
}
// The same from a stage's table entries in single precision: w and, NEAR, w^4 (R >= 8). At most one squaring away from a
// rounded root, a power is off by 3.2 units of 2^-24 at most; from w alone w^8 is off by up to 10.
// NEAR is for the uneven batch's forward stages, which separate a block's key and seed spectra afterwards: that carries an
// error of the key's large low frequencies into the seed's. Margins there fell to 0.5 of what they were in the geometric
// mean over 33 splits of eight lengths (four blocks of 2^24 bits to 2^23, 256 * 128 * 768: 7.8e-2, now 3.5e-2).
// It costs the split pass 5 and 8 % on rows of 3072 and 6144 values (registers) and saves it up to 6 % on others; 256
// uneven blocks take the same 10.0 ms. The passes of plans, whose margins are far below (0.42-0.83 of those with twiddled
// inputs), read w alone: a second row made the innermost pass 1-3.5 % slower on most row lengths (4096: 118.2 -> 122.5 us)
// and the middle strided pass of the 2^27-bit block 3 % (202.5 -> 209.0 us).
template <typename T, int R, bool NEAR>
__device__ __forceinline__ void entry_powers(const cx<T> *w, cx<T> *pw) {
    level_powers<T, R>(w[0], pw);
    if constexpr (NEAR && R >= 8) {
        pw[ilog2(R) - 3] = w[1];
        if constexpr (R == 16) pw[0] = square_root_of_unity<T>(w[1]);
    }
}

// The multipliers of a power-of-two stage at table index k.
template <typename T, int R, int P, bool NEAR>
__device__ __forceinline__ void stage_multipliers(const cx<T> *tab, uint32_t k, cx<T> *m) {
    if constexpr (kRows<T> == Rows::SINGLE) {
        cx<T> w[2], pw[ilog2(R)];
        w[0] = __ldg(tab + k);
        if constexpr (NEAR && R >= 8) w[1] = __ldg(tab + P + k);
        entry_powers<T, R, NEAR>(w, pw);
        level_multipliers<T, R, 1, 0>(pw, m);
    } else {
        load_rows<T, stage_rows(R, kRows<T>, false), P>(tab, k, m);
    }
}
// The multipliers of the odd stage (odd_exponent) at table index k.
template <typename T, int RO, int R0, int K1 = 0>
__device__ __forceinline__ void odd_level_multipliers(const cx<T> *pw, cx<T> *w) {
    if constexpr (K1 < RO) {
        cx<T> m[R0 / 2];
        level_multipliers<T, R0, RO * R0, K1>(pw, m);
#pragma unroll
        for (int r = 0; r < R0 / 2; ++r) w[RO - 1 + r * RO + K1] = m[r];
        odd_level_multipliers<T, RO, R0, K1 + 1>(pw, w);
    }
}
template <typename T, int RO, int R0, int P>
__device__ __forceinline__ void odd_multipliers(const cx<T> *tab, uint32_t k, cx<T> *w) {
    if constexpr (kRows<T> == Rows::SINGLE) {
        cx<T> b;  // w, then w^R0
        load_rows<T, 1, P>(tab, k, &b);
        if constexpr (R0 > 1) {
            cx<T> pw[ilog2(R0)];
            level_powers<T, R0>(b, pw);
            odd_level_multipliers<T, RO, R0>(pw, w);
            b = square_root_of_unity<T>(pw[0]);
        }
        // w[i] = b^(i + 1): even powers by squaring, odd ones by a product
        w[0] = b;
#pragma unroll
        for (int n = 2; n < RO; ++n)
            w[n - 1] = n % 2 == 0 ? square_root_of_unity<T>(w[n / 2 - 1]) : Arith<T>::mul(w[n / 2 - 1], w[(n + 1) / 2 - 1]);
    } else {
        load_rows<T, odd_rows(RO, R0, kRows<T>), P>(tab, k, w);
    }
}

// DFT of v[r] * w^r, r < R, natural order in and out, with the multipliers of
// stage_multipliers for this w: level l, sub-transform p needs (w w_R^p)^(R / 2^(l+1)), and the upper half
// of the p are a quarter turn away from the lower half, so R/2 multipliers do. Every
// butterfly absorbs its multiplier (bfly): a radix-16 stage takes 192 multiply-add slots,
// where twiddling first (15 products, and 14 more to form the powers) took 284.
// With FULL < log2 R only outputs k < 2^FULL are formed: from level FULL on the differences, which
// the other outputs need, are left out.
template <typename T, int R, bool INV, int FULL = ilog2(R)>
__device__ __forceinline__ void dft_rows(cx<T> *v, const cx<T> *w) {
    if constexpr (std::is_same<T, Zp>::value) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = Arith<T>::mul(v[r], w[r - 1]);
        dft<T, R, INV>(v);
    } else if constexpr (std::is_same<T, Zq>::value) {
#pragma unroll
        for (int l = 0; (1 << l) < R; ++l) {
#pragma unroll
            for (int p = 0; p < (1 << l); ++p) {
                const int h = R >> (l + 1), base = bitrev(p, l) * (R >> l);
#pragma unroll
                for (int r = 0; r < h; ++r) Arith<Zq>::bfly(v[base + r], v[base + r + h], w[(1 << l) - 1 + p]);
            }
        }
        bitrev_regs<T, R>(v);
    } else {
#pragma unroll
        for (int l = 0; (1 << l) < R; ++l) {
            const int h = R >> (l + 1);
#pragma unroll
            for (int p = 0; p < (1 << l) && p < (1 << FULL); ++p) {
                const int half = l ? (1 << (l - 1)) : 1;
                const cx<T> m = w[l ? half + (p % half) : 0];
                const bool turned = p >= half;  // a further factor -i (inverse: i)
                const T c = turned ? m.y : m.x, s = turned ? -m.x : m.y;
                const int base = bitrev(p, l) * (R >> l);
#pragma unroll
                for (int r = 0; r < h; ++r) {
                    if (l < FULL) {
                        Arith<T>::bfly(v[base + r], v[base + r + h], c, INV ? -s : s);
                    } else {
                        v[base + r] = Arith<T>::add_mul(v[base + r], v[base + r + h], c, INV ? -s : s);
                    }
                }
            }
        }
        bitrev_regs<T, R>(v);
    }
}

// (a, b) -> (a + w b, a - w b) for w = w_N^J (forward root; the inverse uses the conjugate).
template <typename T, int N, int J, bool INV>
__device__ __forceinline__ void bfly_const(cx<T> &a, cx<T> &b) {
    constexpr int j = J % N;
    if constexpr (j == 0) {
        bfly32<T, 0, INV>(a, b);
    } else if constexpr (4 * j == N) {
        bfly32<T, 8, INV>(a, b);
    } else {
        constexpr T c = (T)cos_frac(j, N), s = (T)sin_frac(j, N);
        Arith<T>::bfly(a, b, c, INV ? s : -s);
    }
}
// DFT of u[n2] * w_{RO R0}^{K1 n2}, n2 < R0, output in bit-reversed slots: level l,
// sub-transform p has the root w_RC^{K1 R0 / 2^(l+1)} w_{2^(l+1)}^p.
template <typename T, int RO, int R0, int K1, bool INV, int LEVEL, int P>
__device__ __forceinline__ void comp_sub(cx<T> *u) {
    if constexpr ((1 << LEVEL) < R0) {
        if constexpr (P < (1 << LEVEL)) {
            constexpr int h = R0 >> (LEVEL + 1), base = bitrev(P, LEVEL) * (R0 >> LEVEL);
#pragma unroll
            for (int r = 0; r < h; ++r)
                bfly_const<T, RO * R0, K1 * h + P * (RO * R0 >> (LEVEL + 1)), INV>(u[base + r], u[base + r + h]);
            comp_sub<T, RO, R0, K1, INV, LEVEL, P + 1>(u);
        } else {
            comp_sub<T, RO, R0, K1, INV, LEVEL + 1, 0>(u);
        }
    }
}
// The radix-R0 step of column k1 = K1, ..., RO-1 of dft_comp.
template <typename T, int RO, int R0, int K1, bool INV>
__device__ __forceinline__ void comp_cols(const cx<T> *a, cx<T> *x) {
    if constexpr (K1 < RO) {
        cx<T> u[R0];
#pragma unroll
        for (int n2 = 0; n2 < R0; ++n2) u[n2] = a[n2 * RO + K1];
        comp_sub<T, RO, R0, K1, INV, 0, 0>(u);
#pragma unroll
        for (int k2 = 0; k2 < R0; ++k2) x[K1 + RO * k2] = u[bitrev(k2, ilog2(R0))];
        comp_cols<T, RO, R0, K1 + 1, INV>(a, x);
    }
}

// In-register DFT of RC = RO * R0 values (RO in {3, 5, 9}, R0 a power of two),
// natural order in and out, by one Cooley-Tukey step: with n = R0 n1 + n2 and
// k = k1 + RO k2, X[k] = sum_n2 w_R0^{n2 k2} w_RC^{n2 k1} sum_n1 w_RO^{n1 k1} x[n].
// The twiddle between the two steps goes into the butterflies of the second.
template <typename T, int RO, int R0, bool INV>
__device__ __forceinline__ void dft_comp(cx<T> *x) {
    if constexpr (R0 == 1) {
        dft_odd<T, RO, INV>(x);
    } else {
        cx<T> a[RO * R0];  // a[n2 * RO + k1]
#pragma unroll
        for (int n2 = 0; n2 < R0; ++n2) {
            cx<T> u[RO];
#pragma unroll
            for (int n1 = 0; n1 < RO; ++n1) u[n1] = x[R0 * n1 + n2];
            dft_odd<T, RO, INV>(u);
#pragma unroll
            for (int k1 = 0; k1 < RO; ++k1) a[n2 * RO + k1] = u[k1];
        }
        comp_cols<T, RO, R0, 0, INV>(a, x);
    }
}

// dft_comp of x[n] * w^n (the inverse transform's last stage) with the multipliers of butterfly
// k of the odd stage (odd_exponent): w^{R0 n1} before the odd step, then radix-R0 stages whose
// multipliers carry w w_RC^{k1}.
template <typename T, int RO, int R0, int P, bool INV>
__device__ __forceinline__ void dft_comp_rows(cx<T> *x, const cx<T> *tab, uint32_t k) {
    cx<T> w[odd_level_rows(RO, R0)];
    odd_multipliers<T, RO, R0, P>(tab, k, w);
    if constexpr (INV) {
#pragma unroll
        for (int r = 0; r < RO - 1; ++r) w[r].y = -w[r].y;
    }
#pragma unroll
    for (int n1 = 1; n1 < RO; ++n1) {
#pragma unroll
        for (int n2 = 0; n2 < R0; ++n2) x[R0 * n1 + n2] = Arith<T>::mul(x[R0 * n1 + n2], w[n1 - 1]);
    }
    if constexpr (R0 == 1) {
        dft_odd<T, RO, INV>(x);
    } else {
        cx<T> a[RO * R0];
#pragma unroll
        for (int n2 = 0; n2 < R0; ++n2) {
            cx<T> u[RO];
#pragma unroll
            for (int n1 = 0; n1 < RO; ++n1) u[n1] = x[R0 * n1 + n2];
            dft_odd<T, RO, INV>(u);
#pragma unroll
            for (int k1 = 0; k1 < RO; ++k1) a[n2 * RO + k1] = u[k1];
        }
#pragma unroll
        for (int k1 = 0; k1 < RO; ++k1) {
            cx<T> u[R0], m[R0 / 2];
#pragma unroll
            for (int n2 = 0; n2 < R0; ++n2) u[n2] = a[n2 * RO + k1];
#pragma unroll
            for (int r = 0; r < R0 / 2; ++r) m[r] = w[RO - 1 + r * RO + k1];
            dft_rows<T, R0, INV>(u, m);
#pragma unroll
            for (int k2 = 0; k2 < R0; ++k2) x[k1 + RO * k2] = u[k2];
        }
    }
}

// The pass twiddles: v[s] *= w^{(tq + s*TC) u} for s = 0 .. N-1 and column u = blk*COLS + col
// (nblk column blocks): one product for s = 0, then a chain of products with g = w^{TC u}.
template <typename T, int N, int COLS>
__device__ __forceinline__ void pass_twiddles(cx<T> *v, const PassTw<T> &t, uint32_t nblk, uint32_t tq, uint32_t blk,
                                              uint32_t col) {
    if constexpr (std::is_same<T, Zq>::value) {  // multipliers do not multiply: one product per table
        const uint32_t S = nblk * COLS, u = blk * COLS + col;
        const cx<T> p = __ldg(t.a + (uint64_t)tq * S + u);
#pragma unroll
        for (int s = 0; s < N; ++s) {
            if (s) v[s] = Arith<T>::mul(v[s], __ldg(t.g + (uint64_t)s * S + u));
            v[s] = Arith<T>::mul(v[s], p);
        }
    } else {
        cx<T> w = Arith<T>::mul(__ldg(t.a + (uint64_t)tq * nblk + blk), __ldg(t.c + tq * COLS + col));
        const cx<T> g = __ldg(t.g + blk * COLS + col);
#pragma unroll
        for (int r = 0; r < N; ++r) {
            v[r] = Arith<T>::mul(v[r], w);
            if (r + 1 < N) w = Arith<T>::mul(w, g);
        }
    }
}

// ---- in-CTA transforms ---------------------------------------------------------------------
// A transform of LEN values per column lives in the CTA's registers, E per thread, and passes
// through shared memory between stages (stage_plan in tables.cuh). Every stage works in place:
// a thread writes the slots it has read, so an exchange needs one barrier, between the writes of
// one stage and the reads of the next, and the stage after it none. Stage i's exchange with stage
// i+1 stays inside blocks of N[i] elements, which N[i] / E neighbouring threads hold: with the last
// two stages of radix E that is half a warp (E = 16) or less, and the exchange needs no CTA
// barrier at all. A row of 20*16*16 values has two CTA barriers in the fused innermost pass,
// where a self-sorting (Stockham) order of the same stages had seven: the in-CTA transforms alone,
// with no global access, took 143 of that pass's 177 us there.
//
// In-place stages leave the spectrum in digit-reversed order. A column's frequency digits are put
// right where it leaves the CTA (freq_of); rows keep the order, since nothing but the pointwise
// product, stored in the same order, sees it.
// Twiddles sit on a stage's inputs in both directions: forward stage i multiplies element r of block b
// by w_{R P}^{r f} with f the frequency digits found so far (block_freq), inverse stage i by
// w_N^{-r j} at offset j.

// Shared-memory slot of element a of column col (COLS columns interleaved; one: a row), skewed by
// one slot every 128 bytes. A stage's r-th element sits at base + r*s with s a multiple of the skew's
// period, or (s = 1) base a multiple of E: slot(base + r*s) = slot(base) + slot(r*s).
template <typename T, int COLS>
constexpr int slot_lg() { return COLS == 1 && sizeof(cx<T>) == 16 ? 3 : 4; }
template <typename T, int COLS>
__host__ __device__ constexpr uint32_t slot_of(uint32_t a, uint32_t col) {
    const uint32_t i = a * COLS + col;
    return i + (i >> slot_lg<T, COLS>());
}
template <typename T, int LEN, int COLS>
constexpr uint32_t smem_elems() { return (uint32_t)LEN * COLS + ((uint32_t)LEN * COLS >> slot_lg<T, COLS>()) + 1; }

// The stage plan at compile time.
template <typename T, int LEN, int E> struct Plan {
    static constexpr StagePlan p = stage_plan(LEN, E, kRows<T>);
    static constexpr int RO = p.RO, TC = p.TC, r0 = p.r0, n = p.n;
    static_assert(RO == 1 || RO == 3 || RO == 5 || RO == 9, "odd factor must be 1, 3, 5 or 9");
    static_assert(n >= 2 && p.R[n - 1] == E, "at least two stages, the last of radix E");
};

// block_freq and freq_block (tables.cuh) of stage I with every radix a compile-time constant.
template <typename T, int LEN, int E, int I>
__device__ __forceinline__ uint32_t block_to_freq(uint32_t b) {
    if constexpr (I == 0) {
        return 0u;
    } else {
        constexpr uint32_t R = (uint32_t)Plan<T, LEN, E>::p.R[I - 1], P = (uint32_t)Plan<T, LEN, E>::p.P[I - 1];
        return b % R * P + block_to_freq<T, LEN, E, I - 1>(b / R);
    }
}
template <typename T, int LEN, int E, int I>
__device__ __forceinline__ uint32_t freq_to_block(uint32_t f, uint32_t b = 0u) {
    if constexpr (I == Plan<T, LEN, E>::n - 1) {
        return b;
    } else {
        constexpr uint32_t R = (uint32_t)Plan<T, LEN, E>::p.R[I];
        return freq_to_block<T, LEN, E, I + 1>(f / R, b * R + f % R);
    }
}
// Frequency (mod TC) of the values that thread tq holds at the end of a forward transform and at
// the start of an inverse one: register slot s is frequency freq_of(tq) + s*TC. thread_of is the inverse.
template <typename T, int LEN, int E>
__device__ __forceinline__ uint32_t freq_of(uint32_t tq) {
    return block_to_freq<T, LEN, E, Plan<T, LEN, E>::n - 1>(tq);
}
template <typename T, int LEN, int E>
__device__ __forceinline__ uint32_t thread_of(uint32_t f) {
    return freq_to_block<T, LEN, E, 0>(f);
}
// Index of the element in register slot s of thread tq at the start of a forward transform and at
// the end of an inverse one (no odd stage): stage 0's butterfly s / r0, element s % r0.
template <typename T, int LEN, int E>
__device__ __forceinline__ uint32_t elem_of(uint32_t tq, int s) {
    constexpr int r0 = Plan<T, LEN, E>::r0;
    return tq + (uint32_t)(s / r0) * (LEN / E) + (uint32_t)(s % r0) * (LEN / r0);
}

// Barrier of an exchange inside blocks of N elements.
template <int N, int E>
__device__ __forceinline__ void exchange_barrier() {
    constexpr int scope = N / E;  // threads per block
    if constexpr (scope <= 32 && 32 % scope == 0) {
        __syncwarp();
    } else {
        __syncthreads();
    }
}

// Butterfly g < E / R[I] of thread tq in stage I: block tq / T, offset j = tq % T + g*T, where the
// T = N[I] / E threads of a block share its butterflies (so that the next exchange stays among them).
template <typename T, int LEN, int E, int I> struct StageMap {
    static constexpr StagePlan p = Plan<T, LEN, E>::p;
    static constexpr int R = p.R[I], N = p.N[I], s = p.s[I], threads = N / E, groups = E / R;
    static_assert(threads * E == N, "a block is a whole number of threads");
    static __device__ __forceinline__ uint32_t block(uint32_t tq) { return tq / (uint32_t)threads; }
    static __device__ __forceinline__ uint32_t offset(uint32_t tq, int g) {
        return tq % (uint32_t)threads + (uint32_t)(g * threads);
    }
    template <int COLS> static __device__ __forceinline__ uint32_t slot(uint32_t tq, int g, uint32_t col) {
        return slot_of<T, COLS>(block(tq) * (uint32_t)N + offset(tq, g), col);
    }
};
template <typename T, int LEN, int COLS, int E, int I>
__device__ __forceinline__ void load_stage(const cx<T> *sm, cx<T> *v, uint32_t tq, uint32_t col) {
    using M = StageMap<T, LEN, E, I>;
#pragma unroll
    for (int g = 0; g < M::groups; ++g) {
        const uint32_t s0 = M::template slot<COLS>(tq, g, col);
#pragma unroll
        for (int r = 0; r < M::R; ++r) v[g * M::R + r] = sm[s0 + slot_of<T, COLS>((uint32_t)(r * M::s), 0)];
    }
}
template <typename T, int LEN, int COLS, int E, int I>
__device__ __forceinline__ void store_stage(cx<T> *sm, const cx<T> *v, uint32_t tq, uint32_t col) {
    using M = StageMap<T, LEN, E, I>;
#pragma unroll
    for (int g = 0; g < M::groups; ++g) {
        const uint32_t s0 = M::template slot<COLS>(tq, g, col);
#pragma unroll
        for (int r = 0; r < M::R; ++r) sm[s0 + slot_of<T, COLS>((uint32_t)(r * M::s), 0)] = v[g * M::R + r];
    }
}
// The butterflies of stage I on the thread's registers (NEAR: entry_powers).
template <typename T, int LEN, int E, int I, bool INV, int FROM = 0, bool NEAR = false>
__device__ __forceinline__ void stage_regs(cx<T> *v, uint32_t tq, const cx<T> *st) {
    using M = StageMap<T, LEN, E, I>;
    constexpr StagePlan p = Plan<T, LEN, E>::p;
    constexpr int COUNT = INV ? p.s[I] : p.P[I];
    constexpr StageRow row = INV ? p.inv[I] : p.fwd[I];
#pragma unroll
    for (int g = 0; g < M::groups; ++g) {
        if constexpr (row.rows == 0) {
            dft<T, M::R, INV, FROM>(v + g * M::R);
        } else {
            cx<T> w[multipliers<T>(M::R)];
            stage_multipliers<T, M::R, COUNT, NEAR && !INV>(st + row.off, INV ? M::offset(tq, g) : M::block(tq), w);
            dft_rows<T, M::R, INV>(v + g * M::R, w);
        }
    }
}

// Forward stages I .. n-1, stage I's inputs in shared memory (a barrier away) unless FROM_REGS;
// the outputs end in registers (frequencies freq_of(tq) + s*TC).
template <typename T, int LEN, int COLS, int E, int I, bool FROM_REGS, int FROM = 0, bool NEAR = false>
__device__ __forceinline__ void fwd_stages(cx<T> *sm, cx<T> *v, uint32_t tq, uint32_t col, const cx<T> *st) {
    using PL = Plan<T, LEN, E>;
    if constexpr (!FROM_REGS) {
        exchange_barrier<COLS * PL::p.N[I - 1], E>();
        load_stage<T, LEN, COLS, E, I>(sm, v, tq, col);
    }
    stage_regs<T, LEN, E, I, false, FROM, NEAR>(v, tq, st);
    if constexpr (I < PL::n - 1) {
        store_stage<T, LEN, COLS, E, I>(sm, v, tq, col);
        fwd_stages<T, LEN, COLS, E, I + 1, false, 0, NEAR>(sm, v, tq, col, st);
    }
}
// Inverse stages I .. LAST (counting down), stage I's inputs in registers; the outputs of stage LAST
// end in registers, or, with TO_SMEM, in shared memory.
template <typename T, int LEN, int COLS, int E, int I, int LAST, bool TO_SMEM>
__device__ __forceinline__ void inv_stages(cx<T> *sm, cx<T> *v, uint32_t tq, uint32_t col, const cx<T> *st) {
    using PL = Plan<T, LEN, E>;
    stage_regs<T, LEN, E, I, true>(v, tq, st);
    if constexpr (I > LAST || TO_SMEM) store_stage<T, LEN, COLS, E, I>(sm, v, tq, col);
    if constexpr (I > LAST) {
        exchange_barrier<COLS * PL::p.N[I - 1], E>();
        load_stage<T, LEN, COLS, E, I - 1>(sm, v, tq, col);
        inv_stages<T, LEN, COLS, E, I - 1, LAST, TO_SMEM>(sm, v, tq, col, st);
    }
}

// Full power-of-two transform of length LEN on COLS interleaved columns. Forward: v holds
// elements elem_of(tq, s) on entry and frequencies freq_of(tq) + s*TC on exit; inverse the
// other way round. A forward transform writes shared memory that other threads may still be
// reading (from an earlier one): the caller puts a barrier before it. An inverse transform
// first writes the slots the same thread read last in the forward one.
template <typename T, int LEN, int COLS, int E, bool INV, bool NEAR = false>
__device__ __forceinline__ void cta_fft(cx<T> *sm, cx<T> *v, uint32_t tq, uint32_t col, const cx<T> *st) {
    using PL = Plan<T, LEN, E>;
    static_assert(PL::RO == 1, "odd lengths use cta_fft_fwd_odd / cta_fft_inv_odd");
    if constexpr (!INV) {
        fwd_stages<T, LEN, COLS, E, 0, true, 0, NEAR>(sm, v, tq, col, st);
    } else {
        inv_stages<T, LEN, COLS, E, PL::n - 1, 0, false>(sm, v, tq, col, st);
    }
}

// Inverse transform of a strided pass's columns with the pass twiddle w^{-k u} (column u of stride S)
// in the stages' multipliers: frequency k = k_0 + R_0 (k_1 + ...), and stage i, which sums over k_i with
// w_{N_i}^{-j k_i}, takes w_{N_i S}^{-(S j + u) k_i} instead, the product of its table's entry and
// an entry of the column tables. Twiddling the inputs first cost a product for every value, another to form its twiddle
// (248 of a 256-point column thread's 866 instructions in single precision) and left the first stage's
// butterflies without multipliers to absorb. Only outputs of butterfly slots below `need` (of stage 0's
// radix) are wanted: with few of them stage 0 leaves out the butterflies of the others.
// Single precision reads one column table per stage, w^{P_i u}, and forms the stage's multipliers by squarings, as it
// does elsewhere. Double precision reads one per butterfly level: every multiplier is then the product of two
// rounded roots, off by 4.25 units of 2^-53 at most (2.1 seen). Formed by squarings they were off by up to 18: the
// rounding margins of a 2^23-bit key (512 * 64 * 384) were 8.2e-12 in the mean, now 4.0e-12 (with twiddled
// inputs 6.5e-12), and a batch of 64 keys of 10^6 bits takes 10.05 ms instead of 10.11.
// hu[l] = the entry of level l of stage I (SINGLE: hu[0], the last level's) in column u, h its entry in table 0.
template <typename T, int LEN, int E, int I>
__device__ __forceinline__ void load_col(const cx<T> *h, uint32_t S, cx<T> *hu) {
    constexpr StagePlan p = Plan<T, LEN, E>::p;
#pragma unroll
    for (int l = 0; l < stage_col_tables(p.R[I], kRows<T>); ++l) hu[l] = __ldg(h + (uint32_t)(first_col_table(p, I, kRows<T>) + l) * S);
}
template <typename T, int LEN, int E, int I>
__device__ __forceinline__ void col_multipliers(uint32_t tq, int g, const cx<T> *st, const cx<T> *hu, cx<T> *m) {
    using M = StageMap<T, LEN, E, I>;
    constexpr StagePlan p = Plan<T, LEN, E>::p;
    if constexpr (kRows<T> == Rows::SINGLE) {
        cx<T> w = hu[0], pw[ilog2(M::R)];
        if constexpr (I < p.n - 1) w = Arith<T>::mul(w, __ldg(st + p.inv[I].off + M::offset(tq, g)));
        level_powers<T, M::R>(w, pw);
        level_multipliers<T, M::R, 1, 0>(pw, m);
    } else if constexpr (I < p.n - 1) {
        load_rows<T, level_rows(M::R), M::s>(st + p.inv[I].off, M::offset(tq, g), m);
#pragma unroll
        for (int r = 0; r < level_rows(M::R); ++r) m[r] = Arith<T>::mul(m[r], hu[row_level(r)]);
    } else {
        level_multipliers<T, M::R, 1, 0>(hu, m);
    }
}
template <typename T, int LEN, int COLS, int E, int I>
__device__ __forceinline__ void inv_col_stages(cx<T> *sm, cx<T> *v, uint32_t tq, uint32_t col, const cx<T> *st,
                                               const cx<T> *h, uint32_t S, uint32_t need) {
    using PL = Plan<T, LEN, E>;
    using M = StageMap<T, LEN, E, I>;
    cx<T> hu[stage_col_tables(M::R, kRows<T>)];
    load_col<T, LEN, E, I>(h, S, hu);
#pragma unroll
    for (int g = 0; g < M::groups; ++g) {
        cx<T> m[level_rows(M::R)];
        col_multipliers<T, LEN, E, I>(tq, g, st, hu, m);
        cx<T> *x = v + g * M::R;
        if constexpr (I == 0 && M::R == 16) {
            if (need <= 2) dft_rows<T, 16, true, 1>(x, m);
            else if (need <= 4) dft_rows<T, 16, true, 2>(x, m);
            else dft_rows<T, 16, true>(x, m);
        } else if constexpr (I == 0 && M::R == 8 && M::groups == 1) {
            if (need <= 1) dft_rows<T, 8, true, 0>(x, m);
            else if (need <= 2) dft_rows<T, 8, true, 1>(x, m);
            else dft_rows<T, 8, true>(x, m);
        } else {
            dft_rows<T, M::R, true>(x, m);
        }
    }
    if constexpr (I > 0) {
        store_stage<T, LEN, COLS, E, I>(sm, v, tq, col);
        exchange_barrier<COLS * PL::p.N[I - 1], E>();
        load_stage<T, LEN, COLS, E, I - 1>(sm, v, tq, col);
        inv_col_stages<T, LEN, COLS, E, I - 1>(sm, v, tq, col, st, h, S, need);
    }
}
// The inverse transform of column u of a strided pass (pass 0 or 1 of tw; column block blk of nblk,
// stride S), pass twiddle included: v holds frequencies freq_of(tq) + s*TC on entry, elements
// elem_of(tq, s) on exit, of which the rows below nrow are wanted.
template <typename T, int LEN, int COLS, int E, int PASS>
__device__ __forceinline__ void inverse_columns(cx<T> *sm, cx<T> *v, uint32_t tq, uint32_t col, const TwTab<T> &tw,
                                                uint32_t nblk, uint32_t blk, uint32_t S, uint32_t nrow) {
    using PL = Plan<T, LEN, E>;
    if constexpr (!is_complex(kRows<T>)) {
        pass_twiddles<T, E, COLS>(v, tw.iv[PASS], nblk, freq_of<T, LEN, E>(tq), blk, col);
        cta_fft<T, LEN, COLS, E, true>(sm, v, tq, col, tw.st[PASS]);
    } else {
        constexpr uint32_t K = LEN / PL::r0;  // rows of one butterfly slot of stage 0
        inv_col_stages<T, LEN, COLS, E, PL::n - 1>(sm, v, tq, col, tw.st[PASS], tw.col[PASS] + blk * COLS + col, S,
                                                   (nrow + K - 1) / K);
    }
}

// Forward transform of a contiguous row of LEN = RO * 2^k elements (RO > 1).
// Stage 0 has the odd (or composite) radix RC: group b = tq + g TC < K = LEN / RC reads elements
// b + r K through ld(offset), the offset g TC + r K counted from element tq (a compile-time
// constant, so the caller's base pointer for thread tq takes immediate offsets).
template <typename T, int LEN, int E, bool NEAR, class Ld>
__device__ __forceinline__ void cta_fft_fwd_odd(cx<T> *sm, cx<T> *v, uint32_t tq, const cx<T> *st, Ld ld) {
    constexpr StagePlan p = Plan<T, LEN, E>::p;
    constexpr int RC = p.RC, K = LEN / RC, TC = p.TC;
    constexpr int G = (K + TC - 1) / TC;  // groups per thread (the last may be partial)
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const uint32_t b = tq + (uint32_t)g * TC;
        if (b < (uint32_t)K) {
            cx<T> u[RC];
#pragma unroll
            for (int r = 0; r < RC; ++r) u[r] = ld((uint32_t)(g * TC + r * K));
            dft_comp<T, p.RO, p.R0C, false>(u);
            const uint32_t s0 = slot_of<T, 1>(b, 0);
#pragma unroll
            for (int r = 0; r < RC; ++r) sm[s0 + slot_of<T, 1>((uint32_t)(r * K), 0)] = u[r];
        }
    }
    fwd_stages<T, LEN, 1, E, 1, false, 0, NEAR>(sm, v, tq, 0, st);
}

// Inverse transform of a row (RO > 1): the power-of-two stages from registers into shared memory,
// then stage 0: group b reads slots b + r K, and its output b + r K goes through
// put(g TC + r K, value) (offset from element tq, as for ld above).
template <typename T, int LEN, int E, class St>
__device__ __forceinline__ void cta_fft_inv_odd(cx<T> *sm, cx<T> *v, uint32_t tq, const cx<T> *st, St put) {
    constexpr StagePlan p = Plan<T, LEN, E>::p;
    constexpr int RC = p.RC, K = LEN / RC, TC = p.TC;
    constexpr int G = (K + TC - 1) / TC;
    inv_stages<T, LEN, 1, E, p.n - 1, 1, true>(sm, v, tq, 0, st);
    exchange_barrier<LEN, E>();
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const uint32_t b = tq + (uint32_t)g * TC;
        if (b < (uint32_t)K) {
            cx<T> u[RC];
            const uint32_t s0 = slot_of<T, 1>(b, 0);
#pragma unroll
            for (int r = 0; r < RC; ++r) u[r] = sm[s0 + slot_of<T, 1>((uint32_t)(r * K), 0)];
            dft_comp_rows<T, p.RO, p.R0C, K, true>(u, st + p.inv[0].off, b);
#pragma unroll
            for (int r = 0; r < RC; ++r) put((uint32_t)(g * TC + r * K), u[r]);
        }
    }
}

}  // namespace pa
