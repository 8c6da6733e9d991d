// Fixed-point diagonals and packed FMAs of the segment and Hubbard kernels.
#pragma once

#include <cuda_runtime.h>

namespace hphi {

constexpr int kFixShift = 29;  // 64-bit to 32-bit fixed point (diagonals are below 2^59 in 64 bits)

template <typename T>
struct FixInt { using type = int; };
template <>
struct FixInt<double> { using type = long long; };

// A 64-bit fixed-point value in T's fixed point (FP32: its upper bits, rounded).
template <typename T>
__host__ __device__ __forceinline__ typename FixInt<T>::type to_fix(long long v) {
    if constexpr (sizeof(T) == 4) return (int)((v + (1ll << (kFixShift - 1))) >> kFixShift);
    else return v;
}

// (a0, a1) += c (v0, v1), each rounded as a single fma
__device__ __forceinline__ void fma2(float &a0, float &a1, float c, float v0, float v1) {
    asm("{.reg .b64 a, b, d; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %4}; mov.b64 d, {%0, %1};\n\t"
        "fma.rn.f32x2 d, a, b, d; mov.b64 {%0, %1}, d;}"
        : "+f"(a0), "+f"(a1)
        : "f"(v0), "f"(v1), "f"(c));
}

}  // namespace hphi
