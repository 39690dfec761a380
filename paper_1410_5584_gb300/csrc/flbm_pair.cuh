// flbm_pair.cuh -- two floats handled by one instruction: the packed FP32
// arithmetic of sm_100 and later (add, sub, mul, fma on .f32x2 operands).
// The collide uses it where both species run the same arithmetic on their
// own values (one lane per species).  Each lane is rounded exactly as the
// scalar instruction would round it.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace flbm {

struct F2 {
    unsigned long long v;
    F2() = default;
    __device__ __forceinline__ explicit F2(unsigned long long bits) : v(bits) {}
    __device__ __forceinline__ F2(float lo, float hi)
    {
        asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    }
    __device__ __forceinline__ explicit F2(float2 x) : F2(x.x, x.y) {}
    __device__ __forceinline__ float2 f2() const { return make_float2(lo(), hi()); }
    // the same value in both lanes; built from the bit patterns so that a
    // constant argument gives a compile-time constant
    __device__ __forceinline__ explicit F2(int k) : v(splat((float)k)) {}
    __device__ __forceinline__ static unsigned long long splat(float x)
    {
        const unsigned long long b = __float_as_uint(x);
        return (b << 32) | b;
    }
    __device__ __forceinline__ float lo() const
    {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        (void)b;
        return a;
    }
    __device__ __forceinline__ float hi() const
    {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        (void)a;
        return b;
    }
};

__device__ __forceinline__ F2 splat2(float x) { return F2(F2::splat(x)); }
// a float2 of the kernel parameters (or any 8-byte aligned pair) as one packed value
__device__ __forceinline__ F2 pair2(const float2 &x) { return F2(*reinterpret_cast<const unsigned long long *>(&x)); }
__device__ __forceinline__ F2 neg2(F2 a) { return F2(a.v ^ 0x8000000080000000ull); }

__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return d;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b)
{
    F2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
    F2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b)
{
    F2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}

// A product whose rounding is deferred, so that "c + k * x" and "c - k * x"
// (the forms of the factored transforms, with k a small integer constant)
// become one fused multiply-add, as the scalar compiler contracts them.
struct P2 {
    F2 a, b;
};
__device__ __forceinline__ P2 operator*(F2 a, F2 b) { return {a, b}; }
__device__ __forceinline__ F2 operator+(F2 c, P2 p) { return fma2(p.a, p.b, c); }
__device__ __forceinline__ F2 operator+(P2 p, F2 c) { return fma2(p.a, p.b, c); }
__device__ __forceinline__ F2 operator-(F2 c, P2 p) { return fma2(neg2(p.a), p.b, c); }
__device__ __forceinline__ F2 operator-(P2 p, F2 c) { return mul2(p.a, p.b) - c; }

// Sum of floats as three floats hi + mid + lo: the rounding error of each addition
// to hi (two-sum: D. E. Knuth, The Art of Computer Programming 2, 4.2.2, Thm. B)
// is added to mid in the same way, and that addition's error to lo (the sum with
// K = 3 of T. Ogita, S. M. Rump, S. Oishi, Accurate sum and dot product, SIAM J.
// Sci. Comput. 26 (2005), Alg. 4.8).  n values are summed to (2 n 2^-24)^3 of the
// sum of their magnitudes and the rounding of value(); up to kFold of them that is
// 2^-48, below the n 2^-53 of an FP64 sum in order.  This GPU does only a few
// FP64 operations a cycle and SM.
struct FloatSum {
    static constexpr int kFold = 128; // longer sums: value() into a double after that many
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
    __device__ __forceinline__ static float two_sum(float &s, float v)
    {
        const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b));
        s = t;
        return e;
    }
    __device__ __forceinline__ void add(float v) { lo = __fadd_rn(lo, two_sum(mid, two_sum(hi, v))); }
    __device__ __forceinline__ double value() const
    {
        return isfinite(hi) ? (double)hi + ((double)mid + (double)lo) : (double)hi;
    }
};

} // namespace flbm
