// Pairs of FP32 values held in one 64-bit register: the paired instructions
// (FADD2, FMUL2, FFMA2) advance both at once.  Used for two x-adjacent cells by
// the explicit kernel and for two adjacent lines by the column solvers.
#pragma once

#include "ch_kernels.cuh"

namespace chg {

template <typename T>
struct Pr;

template <>
struct Pr<float> {
    float2 v;
    __device__ __forceinline__ float x() const { return v.x; }
    __device__ __forceinline__ float y() const { return v.y; }
};

__device__ __forceinline__ Pr<float> mk(float a, float b) { return {make_float2(a, b)}; }
template <typename T>
__device__ __forceinline__ Pr<T> sp(T a) { return mk(a, a); }

__device__ __forceinline__ Pr<float> add(Pr<float> a, Pr<float> b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ Pr<float> mul(Pr<float> a, Pr<float> b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ Pr<float> fma2(Pr<float> a, Pr<float> b, Pr<float> c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ Pr<float> sub(Pr<float> a, Pr<float> b) {
    // a - b with one rounding (the paired subtraction; no constant operand)
    unsigned long long ra, rb, rd;
    memcpy(&ra, &a.v, 8);
    memcpy(&rb, &b.v, 8);
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    Pr<float> d;
    memcpy(&d.v, &rd, 8);
    return d;
}


// aligned pair load/store (address of the first element of the pair)
__device__ __forceinline__ Pr<float> ldp(const float* p) { return {*reinterpret_cast<const float2*>(p)}; }
__device__ __forceinline__ void stp(float* p, Pr<float> a) { *reinterpret_cast<float2*>(p) = a.v; }

template <typename T>
__device__ __forceinline__ Pr<T> psi_pp(Pr<T> c) {  // psi'(C) = C (C (C - 1.5) + 0.5)
    return mul(c, fma2(c, sub(c, sp<T>(T(1.5))), sp<T>(T(0.5))));
}

constexpr int kTX2 = 64;  // cells in x of the explicit kernel's tile (two per thread)
constexpr int kHL2 = 4;   // its left halo columns (a 16-byte chunk)

}  // namespace chg
