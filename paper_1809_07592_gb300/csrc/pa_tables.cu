// pa_tables.cu -- layout and filling of the twiddle tables (tables.cuh) of a transform.
#include "pa.h"
#include "pa_internal.h"
#include "pa_launch.h"

using namespace pa;

namespace {

constexpr uint64_t kAlignElems = 32;  // every table starts on a 256-byte boundary (8-byte elements)
uint64_t take(uint64_t *total, uint64_t n) {
    const uint64_t at = *total;
    *total += (n + kAlignElems - 1) / kAlignElems * kAlignElems;
    return at;
}

// The stage plans of a layout's passes (worked out once on the host: they are loops over divisions).
struct StagePlans {
    StagePlan pass[3];
};

// Exponent (of w_L, not reduced) of element i of the block; inverse tables of the exact
// transform come back with *neg set. Padding elements read as w^0.
__device__ uint64_t exponent_at(const TwLayout &y, const StagePlan *plans, uint64_t i, Rows kind, bool *neg) {
    const bool complex_ = is_complex(kind);
    *neg = false;
    if (i >= y.hi && i < y.hi + y.nhi) return (i - y.hi) << y.B;
    if (i >= y.lo && i < y.lo + y.nlo) return i - y.lo;
    for (int p = 0; p < 3; ++p) {
        if (y.len[p] == 0) continue;
        const StagePlan &l = plans[p];
        if (i < y.st[p] || i >= y.st[p] + (uint64_t)l.total) continue;
        const int o = (int)(i - y.st[p]);
        for (int j = 0; j < 2 * l.n; ++j) {
            const int stage = j % l.n;
            const bool inv = j >= l.n;
            const StageRow r = inv ? l.inv[stage] : l.fwd[stage];
            const int count = inv ? l.s[stage] : l.P[stage];
            if (r.rows == 0 || o < r.off || o >= r.off + row_entries(r.rows, count)) continue;
            const bool pairs = r.rows > 1 && kind != Rows::SINGLE;
            const int q = pairs ? (o - r.off) / 2 : o - r.off;
            const int row = pairs ? 2 * (q / count) + ((o - r.off) & 1) : q / count;
            const uint32_t x = (uint32_t)(q % count);
            if (row >= r.rows) return 0;
            *neg = !complex_ && inv;
            if (inv && stage == 0 && l.RO > 1) return odd_exponent(l.RO, l.R0C, count, row, x, y.L, kind);
            return stage_exponent(l.R[stage], count, row, inv ? x : block_freq(l, stage, x), y.L, kind);
        }
        return 0;
    }
    for (int p = 0; p < 2; ++p) {
        const PassShape &t = y.pass[p];
        if (t.stride == 0) continue;
        const uint64_t mult = p == 0 ? 1 : (uint64_t)y.len[0], nblk = t.stride / t.cols;
        for (int inv = 0; inv < (complex_ ? 1 : 2); ++inv) {
            const uint64_t a = inv ? t.ai : t.a, c = inv ? t.ci : t.c, g = inv ? t.gi : t.g;
            *neg = inv != 0;
            if (kind == Rows::LEVELS) {
                if (i >= a && i < a + t.tc * t.stride) return (i - a) / t.stride * ((i - a) % t.stride) * mult;
                if (i >= g && i < g + (uint64_t)y.E * t.stride)
                    return t.tc * ((i - g) / t.stride) * ((i - g) % t.stride) * mult;
                continue;
            }
            if (i >= a && i < a + t.tc * nblk) return (i - a) / nblk * ((i - a) % nblk) * t.cols * mult;
            if (i >= c && i < c + (uint64_t)t.tc * t.cols) return (i - c) / t.cols * ((i - c) % t.cols) * mult;
            if (i >= g && i < g + t.stride) return t.tc * (i - g) * mult;
        }
        if (complex_) {
            const StagePlan &l = plans[p];
            *neg = false;
            if (i >= t.h && i < t.h + (uint64_t)col_tables(l, kind) * t.stride)
                return col_exponent(l, (int)((i - t.h) / t.stride), kind) * ((i - t.h) % t.stride) * mult;
        }
    }
    *neg = false;
    return 0;
}

// exp(-2 pi i e / L), each part rounded once from double precision.
template <typename T>
__device__ cx<T> root_power(uint64_t e, uint64_t L, uint64_t) {
    uint32_t q;
    double s, c;
    sincospi(0.5 * quarter_turns((uint32_t)e, (uint32_t)L, &q), &s, &c);
    const double x = q & 1 ? -s : c, y = q & 1 ? -c : -s;  // the first quarter turn: times -i
    cx<T> w;
    w.x = (T)(q & 2 ? -x : x);
    w.y = (T)(q & 2 ? -y : y);
    return w;
}
template <>
__device__ cx<Zp> root_power<Zp>(uint64_t e, uint64_t, uint64_t w) {
    uint64_t r = 1;
    for (uint64_t b = w; e; e >>= 1) {
        if (e & 1) r = zp_mul(r, b);
        b = zp_mul(b, b);
    }
    return r;
}

template <>
__device__ cx<Zq> root_power<Zq>(uint64_t e, uint64_t, uint64_t w) {
    const uint32_t r = zq_pow((uint32_t)w, e);
    return make_uint2(r, zq_quotient(r));
}

template <typename T>
__global__ void k_fill_tables(cx<T> *mem, const __grid_constant__ TwLayout y, const __grid_constant__ StagePlans plans,
                              uint64_t root) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < y.total; i += (uint64_t)gridDim.x * blockDim.x) {
        bool neg;
        uint64_t e = exponent_at(y, plans.pass, i, kRows<T>, &neg) % y.L;
        if (neg && e) e = y.L - e;
        mem[i] = root_power<T>(e, y.L, root);
    }
}

uint64_t zp_mul_host(uint64_t a, uint64_t b) {
    unsigned __int128 x = (unsigned __int128)a * b;
    return zp_reduce((uint64_t)(x >> 64), (uint64_t)x);
}

// Root of unity of order L (a power of two, 32 <= L <= 2^32) whose L/32-th power
// is 2^6, the root the in-register DFTs use.
uint64_t zp_root(uint64_t L) {
    const uint64_t w = zp_pow_host(7, (kP - 1) / L);  // 7 generates the multiplicative group mod p
    const uint64_t w32 = zp_pow_host(w, L / 32);
    for (uint64_t j = 1; j < 64; j += 2) {
        if (zp_pow_host(w32, j) == 64ull) return zp_pow_host(w, j);
    }
    return 0;
}

}  // namespace

namespace pa {

uint64_t zp_pow_host(uint64_t a, uint64_t e) {
    uint64_t r = 1;
    for (; e; e >>= 1) {
        if (e & 1) r = zp_mul_host(r, a);
        a = zp_mul_host(a, a);
    }
    return r;
}

static Rows rows_of(pa_dtype_t dtype, uint64_t L) {
    return dtype == PA_FP32_GUARD       ? kRows<float>
           : dtype == PA_FP64           ? kRows<double>
           : narrow_exact(dtype, L) ? kRows<Zq>
                                        : kRows<Zp>;
}

TwLayout tw_layout(const Geometry &g, pa_dtype_t dtype, bool powers) {
    const Rows kind = rows_of(dtype, g.L);
    const bool complex_ = is_complex(kind);
    TwLayout y;
    y.L = g.L;
    if (powers) {
        int lgL = 0;
        while ((1ull << lgL) < g.L) ++lgL;
        y.B = (uint32_t)(lgL + 1) / 2;
        y.nlo = 1ull << y.B;
        y.nhi = (g.L + y.nlo - 1) >> y.B;
    }
    y.E = values_per_thread(dtype, g.L);
    y.len[0] = 1 << g.lg1;
    y.len[1] = g.lgM ? 1 << g.lgM : 0;
    y.len[2] = (int)g.inner();
    y.hi = take(&y.total, y.nhi);
    y.lo = take(&y.total, y.nlo);
    for (int p = 0; p < 3; ++p)
        if (y.len[p]) y.st[p] = take(&y.total, (uint64_t)stage_plan(y.len[p], y.E, kind).total);
    for (int p = 0; p < 2; ++p) {
        if (!y.len[p]) continue;
        PassShape &t = y.pass[p];
        t.tc = (uint32_t)(y.len[p] / y.E);
        t.cols = (uint32_t)strided_cols_of(y.E == 16, y.len[p]);
        t.stride = p == 0 ? g.L >> g.lg1 : (uint64_t)g.inner();
        if (kind == Rows::LEVELS) {
            t.a = take(&y.total, t.tc * t.stride);
            t.g = take(&y.total, (uint64_t)y.E * t.stride);
            t.ai = take(&y.total, t.tc * t.stride);
            t.gi = take(&y.total, (uint64_t)y.E * t.stride);
            continue;
        }
        t.a = take(&y.total, t.tc * (t.stride / t.cols));
        t.c = take(&y.total, (uint64_t)t.tc * t.cols);
        t.g = take(&y.total, t.stride);
        if (complex_) {
            t.h = take(&y.total, (uint64_t)col_tables(stage_plan(y.len[p], y.E, kind), kind) * t.stride);
        } else {  // residues have no conjugate: the inverse passes read tables of their own
            t.ai = take(&y.total, t.tc * (t.stride / t.cols));
            t.ci = take(&y.total, (uint64_t)t.tc * t.cols);
            t.gi = take(&y.total, t.stride);
        }
    }
    return y;
}

cudaError_t tw_fill(const TwLayout &y, pa_dtype_t dtype, void *mem, cudaStream_t st) {
    const Rows kind = rows_of(dtype, y.L);
    StagePlans plans{};
    for (int p = 0; p < 3; ++p)
        if (y.len[p]) plans.pass[p] = stage_plan(y.len[p], y.E, kind);
    const uint64_t want = (y.total + 255) / 256;
    const unsigned grid = (unsigned)(want < 1216 ? want : 1216);
    if (dtype == PA_FP32_GUARD) {
        k_fill_tables<float><<<grid, 256, 0, st>>>(static_cast<float2 *>(mem), y, plans, 0);
    } else if (dtype == PA_FP64) {
        k_fill_tables<double><<<grid, 256, 0, st>>>(static_cast<double2 *>(mem), y, plans, 0);
    } else if (narrow_exact(dtype, y.L)) {
        if (y.L & (y.L - 1)) return cudaErrorInvalidValue;  // the exact transforms keep power-of-two lengths
        k_fill_tables<Zq><<<grid, 256, 0, st>>>(static_cast<uint2 *>(mem), y, plans, zq_pow(3u, (kQ - 1) / y.L));
    } else {
        const uint64_t w = (y.L & (y.L - 1)) ? 0 : zp_root(y.L);  // the exact transform keeps power-of-two lengths
        if (!w) return cudaErrorInvalidValue;
        k_fill_tables<Zp><<<grid, 256, 0, st>>>(static_cast<unsigned long long *>(mem), y, plans, w);
    }
    return cudaGetLastError();
}

}  // namespace pa

int pa_internal_twiddles(const Geometry &g, pa_dtype_t dtype, TwSet *out, bool powers) {
    out->lay = tw_layout(g, dtype, powers);
    const size_t esz = dtype == PA_FP32_GUARD ? sizeof(float2) : dtype == PA_FP64 ? sizeof(double2) : sizeof(uint64_t);
    cudaError_t e = cudaMalloc(&out->mem, out->lay.total * esz);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        out->mem = nullptr;
        return PA_ENOMEM;
    }
    if (e == cudaSuccess) e = tw_fill(out->lay, dtype, out->mem, nullptr);
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);  // filled before any stream of the caller reads them
    if (e != cudaSuccess) {
        pa_internal_free_twiddles(out);
        return pa_internal_cuda_fail(e, "twiddle tables");
    }
    return PA_OK;
}

void pa_internal_free_twiddles(TwSet *t) {
    cudaFree(t->mem);
    t->mem = nullptr;
}
