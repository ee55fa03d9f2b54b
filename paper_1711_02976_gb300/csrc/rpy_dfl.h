// Double-floats: a value held as the unevaluated sum h + l of two FP32 numbers, about 48 significant
// bits.  Sums by Knuth's two-sum, products with their error by FMA (Dekker 1971; Ogita, Rump and
// Oishi 2005).  The FP64 precision form computes in them wherever it was bound by the FP64 pipe
// of this part: 2 FP64 operations per SM and clock against 128 FP32 ones, so a multiply-add of
// 12 FP32 operations is five times as fast as one in FP64.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace rpy {

using ::fma;    // the overloads below join these, they do not hide them
using ::sqrt;

struct alignas(8) dfl {
    float h, l;
    dfl() = default;
    __host__ __device__ __forceinline__ dfl(float a, float b) : h(a), l(b) {}
    __host__ __device__ __forceinline__ dfl(int v) : h(float(v)), l(0.f) {}   // |v| < 2^24
    __host__ __device__ __forceinline__ dfl(float v) : h(v), l(0.f) {}
    __host__ __device__ __forceinline__ explicit dfl(double v) : h(float(v)), l(float(v - double(float(v)))) {}
    __host__ __device__ __forceinline__ explicit operator double() const { return double(h) + double(l); }
};

#ifdef __CUDACC__
// |h| >= |l| or h = 0: the same value with |l| at most half an ulp of h
__device__ __forceinline__ dfl renorm(float h, float l) {
    const float s = __fadd_rn(h, l);
    return dfl(s, __fsub_rn(l, __fsub_rn(s, h)));
}
__device__ __forceinline__ dfl renorm(dfl a) { return renorm(a.h, a.l); }
// s + e = a + b exactly
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}
// a b without the last normalisation (an addend, not a factor)
__device__ __forceinline__ dfl mul_raw(dfl a, dfl b) {
    const float p = __fmul_rn(a.h, b.h);
    return dfl(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
// a + b, normalised or (sum_raw) not
__device__ __forceinline__ dfl sum_raw(dfl a, dfl b) {
    float e;
    const float s = two_sum(a.h, b.h, e);
    return dfl(s, __fadd_rn(__fadd_rn(a.l, b.l), e));
}
__device__ __forceinline__ dfl operator-(dfl a) { return dfl(-a.h, -a.l); }
__device__ __forceinline__ dfl operator+(dfl a, dfl b) { return renorm(sum_raw(a, b)); }
__device__ __forceinline__ dfl operator-(dfl a, dfl b) { return a + (-b); }
__device__ __forceinline__ dfl operator*(dfl a, dfl b) { return renorm(mul_raw(a, b)); }
__device__ __forceinline__ void operator+=(dfl &a, dfl b) { a = a + b; }
__device__ __forceinline__ void operator-=(dfl &a, dfl b) { a = a - b; }
__device__ __forceinline__ void operator*=(dfl &a, dfl b) { a = a * b; }
__device__ __forceinline__ dfl fma(dfl a, dfl b, dfl c) { return renorm(sum_raw(c, mul_raw(a, b))); }
// 1 / a: the FP32 quotient and one residual step
__device__ __forceinline__ dfl recip(dfl a) {
    const float y = __frcp_rn(a.h);
    const float e = __fmaf_rn(-a.l, y, __fmaf_rn(-a.h, y, 1.f));   // 1 - a y
    return renorm(y, __fmul_rn(y, __fmaf_rn(e, e, e)));
}
__device__ __forceinline__ dfl operator/(dfl a, dfl b) { return a * recip(b); }
// sqrt(a), a > 0: the FP32 root s and half the exact residual a - s^2 over it
__device__ __forceinline__ dfl sqrt(dfl a) {
    const float s = __fsqrt_rn(a.h);
    const float e = __fadd_rn(__fmaf_rn(-s, s, a.h), a.l);
    const float c = __fdiv_rn(e, __fadd_rn(s, s));
    return renorm(s, __fmaf_rn(-__fmul_rn(c, c), __fdiv_rn(0.5f, s), c));
}

// Running sums: acc += a b without normalising; closed() before the sum is used as a factor.
__device__ __forceinline__ void macc(dfl &acc, dfl a, dfl b) { acc = sum_raw(acc, mul_raw(a, b)); }
__device__ __forceinline__ dfl closed(dfl acc) { return renorm(acc); }
// a b - c d
__device__ __forceinline__ dfl mul_diff(dfl a, dfl b, dfl c, dfl d) { return renorm(sum_raw(mul_raw(a, b), mul_raw(-c, d))); }
// a times a power of two (or any factor that keeps the products exact)
__device__ __forceinline__ dfl scale2(float s, dfl a) { return dfl(__fmul_rn(s, a.h), __fmul_rn(s, a.l)); }

template <typename T> __device__ __forceinline__ void macc(T &acc, T a, T b) { acc = fma(a, b, acc); }
template <typename T> __device__ __forceinline__ T closed(T acc) { return acc; }
template <typename T> __device__ __forceinline__ T mul_diff(T a, T b, T c, T d) { return fma(a, b, -c * d); }
template <typename T> __device__ __forceinline__ T scale2(float s, T a) { return T(s) * a; }

// Two double-floats in the lanes of packed FP32x2 operations (half the instructions of two scalar ones).
struct df2 {
    float2 h, l;
};
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// s + e = a + b exactly
__device__ __forceinline__ float2 two_sum2(float2 a, float2 b, float2 &e) {
    const float2 s = add2(a, b), bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
    return s;
}
// (a.h + a.l) (b.h + b.l)
__device__ __forceinline__ df2 mul_df(df2 a, df2 b) {
    df2 r;
    r.h = mul2(a.h, b.h);
    r.l = fma2(a.l, b.h, fma2(a.h, b.l, fma2(a.h, b.h, neg2(r.h))));
    return r;
}
// a + b, not normalised
__device__ __forceinline__ df2 sum_raw(df2 a, df2 b) {
    float2 e;
    df2 r;
    r.h = two_sum2(a.h, b.h, e);
    r.l = add2(add2(a.l, b.l), e);
    return r;
}
__device__ __forceinline__ df2 renorm(df2 a) {
    df2 r;
    r.h = add2(a.h, a.l);
    r.l = sub2(a.l, sub2(r.h, a.h));
    return r;
}
__device__ __forceinline__ df2 operator-(df2 a) { return df2{neg2(a.h), neg2(a.l)}; }
__device__ __forceinline__ df2 dup(dfl s) { return df2{dup(s.h), dup(s.l)}; }
__device__ __forceinline__ void macc(df2 &acc, df2 a, df2 b) { acc = sum_raw(acc, mul_df(a, b)); }
__device__ __forceinline__ df2 scale2(float s, df2 a) { return df2{mul2(dup(s), a.h), mul2(dup(s), a.l)}; }
__device__ __forceinline__ df2 as_df2(float4 v) { return df2{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 as_float4(df2 v) { return make_float4(v.h.x, v.h.y, v.l.x, v.l.y); }
#endif

}  // namespace rpy
