// Arithmetic on a pair of floats, one per fluid component: x for A, y for B.
//
// The two components of a node go through the same moments, force sums,
// relaxation and back-transform (arXiv:1909.01092, Section 2). On sm_103a a
// packed instruction (add, mul, fma .rn.f32x2) does one operation on both and
// takes one issue slot, and the collide is bound by its issue slots. Each
// half is rounded like the scalar operation. Every operation is written out
// (no contraction is left to the compiler), so all kernels that instantiate
// the same code form the same bits. On the host the halves are computed one
// by one (tests of the headers); the scalar overloads serve them too.
#pragma once

#include <cmath>

namespace flbm {

struct __align__(8) Pair {
    float x, y;
};

__host__ __device__ __forceinline__ Pair splat(float v) { return Pair{v, v}; }

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float2 as_f2(Pair a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ Pair as_pair(float2 a) { return Pair{a.x, a.y}; }
#endif

__host__ __device__ __forceinline__ Pair add(Pair a, Pair b)
{
#ifdef __CUDA_ARCH__
    return as_pair(__fadd2_rn(as_f2(a), as_f2(b)));
#else
    return Pair{a.x + b.x, a.y + b.y};
#endif
}
__host__ __device__ __forceinline__ Pair mul(Pair a, Pair b)
{
#ifdef __CUDA_ARCH__
    return as_pair(__fmul2_rn(as_f2(a), as_f2(b)));
#else
    return Pair{a.x * b.x, a.y * b.y};
#endif
}
// a b + c, rounded once
__host__ __device__ __forceinline__ Pair mad(Pair a, Pair b, Pair c)
{
#ifdef __CUDA_ARCH__
    return as_pair(__ffma2_rn(as_f2(a), as_f2(b), as_f2(c)));
#else
    return Pair{std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y)};
#endif
}
// a - b: the product with -1 is exact
__host__ __device__ __forceinline__ Pair sub(Pair a, Pair b) { return mad(b, splat(-1.0f), a); }

// s + e = a + b exactly, s = fl(a + b) (Knuth's two-sum)
__host__ __device__ __forceinline__ void two_sum(Pair a, Pair b, Pair& s, Pair& e)
{
    s = add(a, b);
    const Pair bb = sub(s, a);
    e = add(sub(a, sub(s, bb)), sub(b, bb));
}

__host__ __device__ __forceinline__ float add(float a, float b) { return a + b; }
__host__ __device__ __forceinline__ float sub(float a, float b) { return a - b; }
__host__ __device__ __forceinline__ float mul(float a, float b) { return a * b; }
__host__ __device__ __forceinline__ float mad(float a, float b, float c)
{
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fma(a, b, c);
#endif
}

__host__ __device__ __forceinline__ double add(double a, double b) { return a + b; }
__host__ __device__ __forceinline__ double sub(double a, double b) { return a - b; }
__host__ __device__ __forceinline__ double mul(double a, double b) { return a * b; }
__host__ __device__ __forceinline__ double mad(double a, double b, double c) { return std::fma(a, b, c); }

// A constant in the arithmetic of T.
template <class T>
__host__ __device__ __forceinline__ T lit(float v);
template <>
__host__ __device__ __forceinline__ float lit<float>(float v)
{
    return v;
}
template <>
__host__ __device__ __forceinline__ double lit<double>(float v)
{
    return v;
}
template <>
__host__ __device__ __forceinline__ Pair lit<Pair>(float v)
{
    return splat(v);
}

}  // namespace flbm
