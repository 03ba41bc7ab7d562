// pa_internal.h -- helpers shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "fft_core.cuh"

// Records "what: cuda error string" as the calling thread's last CUDA error and returns PA_ECUDA.
int pa_internal_cuda_fail(cudaError_t e, const char *what);

#include "pa.h"

namespace pa {

// Transform geometry: length L = 2^lg1 * 2^lgM * (ro * 2^lgI),
// strided level-1 pass 2^lg1, optional middle strided pass 2^lgM (lgM = 0: none),
// innermost pass ro * 2^lgI (ro in {1, 3, 5, 9}).
struct Geometry {
    uint64_t L = 0;
    int lg1 = 0, lgM = 0, ro = 1, lgI = 0;
    uint32_t inner() const { return (uint32_t)ro << lgI; }
};

// Whether the exact transform of length L runs modulo the word-sized prime of zq.cuh (lengths up to
// 2^kMaxLgZq, where it has roots of unity) instead of the 64-bit one, and the values a thread holds.
inline bool narrow_exact(pa_dtype_t dtype, uint64_t L) { return dtype == PA_NTT64 && L <= (1ull << kMaxLgZq); }
inline int values_per_thread(pa_dtype_t dtype, uint64_t L) { return dtype == PA_FP32_GUARD || narrow_exact(dtype, L) ? 16 : 8; }

// Every valid split of length L for the arithmetic `dtype` (split = the
// innermost pass is the two-row Eq. 5-10 kernel of the uneven batch).
std::vector<Geometry> geometry_candidates(uint64_t L, pa_dtype_t dtype, bool split);
// The preferred split of L (two levels when possible, innermost length near 2^12), or L = 0.
Geometry default_geometry(uint64_t L, pa_dtype_t dtype, bool split);
// The smallest supported transform length >= max(need, 2^12): ro * 2^k with ro in {1, 3, 5, 9}
// (ro = 1 only for the exact transform), together with its default split.
Geometry choose_geometry(uint64_t need, pa_dtype_t dtype, bool split);

// Twiddle tables of a transform: where they sit in one block of memory, and filling that
// block on `st` (cudaErrorInvalidValue if the arithmetic has no root of order L). powers: with the tables of
// single powers (TwTab hi, lo), which only the half-length form's innermost pass reads.
TwLayout tw_layout(const Geometry &g, pa_dtype_t dtype, bool powers = false);
cudaError_t tw_fill(const TwLayout &y, pa_dtype_t dtype, void *mem, cudaStream_t st);

// The tables of one transform in device memory of their own.
struct TwSet {
    TwLayout lay;
    void *mem = nullptr;
};

uint64_t zp_pow_host(uint64_t a, uint64_t e);  // a^e mod p (the exact transform's prime)

}  // namespace pa

// Allocate and fill the tables (waits for the fill) / release them.
int pa_internal_twiddles(const pa::Geometry &g, pa_dtype_t dtype, pa::TwSet *out, bool powers = false);
void pa_internal_free_twiddles(pa::TwSet *t);
