// Two FP32 lanes per instruction: the packed add/sub/mul/fma of sm_100 and
// later on .b64 register pairs, each lane rounded to nearest as the scalar FP32
// instruction would round it.  A product whose only use is a packed sum or
// difference is not safe from fusion: ptxas makes one multiply-add of the two, .rn or
// not (x x - RN(x x) comes out as the product's rounding error).  Where the separate
// roundings matter, the scalar __fmul_rn and __fadd_rn keep them.
#pragma once

namespace tri {

using f2 = unsigned long long;

__device__ __forceinline__ f2 f2_pack(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
#define TRI_F2_OP(NAME, OP)                                                                                   \
    __device__ __forceinline__ f2 NAME(f2 a, f2 b)                                                           \
    {                                                                                                        \
        f2 r;                                                                                                \
        asm(OP ".rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));                                          \
        return r;                                                                                            \
    }
TRI_F2_OP(f2_add, "add")
TRI_F2_OP(f2_sub, "sub")
TRI_F2_OP(f2_mul, "mul")
#undef TRI_F2_OP
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Three-input minimum (a NaN is ignored, as by fminf).
__device__ __forceinline__ float min3(float a, float b, float c)
{
    float y;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// 1 / sqrt(x) by the MUFU unit, subnormal inputs taken as zero.
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

}  // namespace tri
