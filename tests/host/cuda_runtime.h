// A stand-in for the CUDA runtime header: what the device headers' arithmetic needs to compile as host C++.
#pragma once
#include <cmath>
#include <cstdint>
#define __CUDACC__
#define __host__
#define __device__
#define __global__
#define __forceinline__ inline
struct float2 { float x, y; };
struct double2 { double x, y; };
struct uint2 { uint32_t x, y; };
struct float4 { float x, y, z, w; };
struct uint4 { uint32_t x, y, z, w; };
struct ulonglong2 { unsigned long long x, y; };
inline float2 make_float2(float x, float y) { return {x, y}; }
inline double2 make_double2(double x, double y) { return {x, y}; }
inline uint2 make_uint2(uint32_t x, uint32_t y) { return {x, y}; }
inline uint32_t min(uint32_t a, uint32_t b) { return a < b ? a : b; }
inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return (unsigned long long)((unsigned __int128)a * b >> 64);
}
template <typename T> inline T __ldg(const T *p) { return *p; }
template <typename T> inline T __ldcg(const T *p) { return *p; }
inline void __syncwarp() {}
inline void __syncthreads() {}
using std::fma;
using std::fmaf;
