// Fixed-point diagonals and packed FMAs of the segment and Hubbard kernels.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace hphi {

// A diagonal is an integer times a power of two, below 2^BITS in 64 bits; 32-bit
// integers keep its upper bits (rounded), below 2^30.

// A 64-bit fixed-point value as an integer of type I.
template <typename I, int BITS>
__host__ __device__ __forceinline__ I to_fix(long long v) {
    constexpr int S = BITS - 30;
    if constexpr (sizeof(I) == 4) return (int)((long long)((unsigned long long)v + (1ull << (S - 1))) >> S);
    else return v;
}

// Does coupling v survive on the grid of `bits` bits below 2^e2 as it would in a
// floating-point number of `digits` digits: on the grid exactly, or with that many
// bits of it (an error of half a grid step is then no more than half an ulp)?
inline bool fix_keeps(double v, int e2, int bits, int digits) {
    const double f = fabs(ldexp(v, bits - e2));
    return f >= ldexp(1.0, digits - 1) || f == rint(f);
}

// (a0, a1) += c (v0, v1), each rounded as a single fma
__device__ __forceinline__ void fma2(float &a0, float &a1, float c, float v0, float v1) {
    asm("{.reg .b64 a, b, d; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %4}; mov.b64 d, {%0, %1};\n\t"
        "fma.rn.f32x2 d, a, b, d; mov.b64 {%0, %1}, d;}"
        : "+f"(a0), "+f"(a1)
        : "f"(v0), "f"(v1), "f"(c));
}

}  // namespace hphi
