// The four charge sets of an item in packed FP32x2 operations: types, shared-memory planes and the factored
// rotation, for the translation kernels of both precision forms (rpy_waves.cu, rpy_shift.cu).
#pragma once

#include "rpy_far.h"

namespace rpy {

// ---------------------------------------------------------------- sets of one item in packed operations
// Quad<T>: N threads share the four sets of an item (pr = 0 .. N - 1), each holding V; a V stands as one
// float4 in memory: four floats, or two double-floats as (h, h', l, l').
struct f4 {
    float2 a, b;   // sets 0 1, 2 3
};
template <typename T> struct Quad;
template <> struct Quad<float> {
    using V = f4;
    static constexpr int N = 1, SH = 0;   // N = 1 << SH
};
template <> struct Quad<dfl> {
    using V = df2;
    static constexpr int N = 2, SH = 1;
};
__device__ __forceinline__ void get(float4 m, f4 &v) { v = f4{make_float2(m.x, m.y), make_float2(m.z, m.w)}; }
__device__ __forceinline__ void get(float4 m, df2 &v) { v = as_df2(m); }
__device__ __forceinline__ float4 put(f4 v) { return make_float4(v.a.x, v.a.y, v.b.x, v.b.y); }
__device__ __forceinline__ float4 put(df2 v) { return as_float4(v); }
template <typename V> __device__ __forceinline__ V zero();
template <> __device__ __forceinline__ f4 zero<f4>() { return f4{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
template <> __device__ __forceinline__ df2 zero<df2>() { return df2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
template <> __device__ __forceinline__ float2 zero<float2>() { return make_float2(0.f, 0.f); }

__device__ __forceinline__ df2 operator+(df2 a, df2 b) { return renorm(sum_raw(a, b)); }
__device__ __forceinline__ df2 operator-(df2 a, df2 b) { return renorm(sum_raw(a, -b)); }
__device__ __forceinline__ df2 closed(df2 a) { return renorm(a); }
__device__ __forceinline__ void macc(df2 &acc, dfl s, df2 b) { macc(acc, dup(s), b); }
__device__ __forceinline__ df2 times(dfl s, df2 a) { return renorm(mul_df(dup(s), a)); }
// a x + b y with scalar a, b
__device__ __forceinline__ df2 lin2(dfl a, df2 x, dfl b, df2 y) {
    return renorm(sum_raw(mul_df(dup(a), x), mul_df(dup(b), y)));
}

__device__ __forceinline__ float2 sum_raw(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 closed(float2 a) { return a; }
__device__ __forceinline__ void macc(float2 &acc, float s, float2 b) { acc = fma2(dup(s), b, acc); }
__device__ __forceinline__ float2 lin2(float a, float2 x, float b, float2 y) { return fma2(dup(a), x, mul2(dup(b), y)); }

__device__ __forceinline__ f4 operator-(f4 a) { return f4{neg2(a.a), neg2(a.b)}; }
__device__ __forceinline__ f4 operator+(f4 a, f4 b) { return f4{add2(a.a, b.a), add2(a.b, b.b)}; }
__device__ __forceinline__ f4 operator-(f4 a, f4 b) { return f4{sub2(a.a, b.a), sub2(a.b, b.b)}; }
__device__ __forceinline__ f4 sum_raw(f4 a, f4 b) { return a + b; }
__device__ __forceinline__ f4 closed(f4 a) { return a; }
__device__ __forceinline__ void macc(f4 &acc, float s, f4 b) {
    macc(acc.a, s, b.a);
    macc(acc.b, s, b.b);
}
__device__ __forceinline__ f4 scale2(float s, f4 a) { return f4{mul2(dup(s), a.a), mul2(dup(s), a.b)}; }
__device__ __forceinline__ f4 times(float s, f4 a) { return scale2(s, a); }
__device__ __forceinline__ f4 lin2(float a, f4 x, float b, f4 y) { return f4{lin2(a, x.a, b, y.a), lin2(a, x.b, b, y.b)}; }

__device__ __forceinline__ float neg1(float a) { return -a; }
__device__ __forceinline__ dfl neg1(dfl a) { return -a; }

// n complex coefficients of four sets in shared memory: real parts [n][N], then imaginary parts,
// 16 bytes each, so that consecutive threads touch consecutive banks.
template <typename T>
struct Planes {
    using V = typename Quad<T>::V;
    static constexpr int N = Quad<T>::N;
    float4 *p;
    int n;
    __device__ __forceinline__ V x(int pr, int i) const {
        V v;
        get(p[N * i + pr], v);
        return v;
    }
    __device__ __forceinline__ V y(int pr, int i) const {
        V v;
        get(p[N * (n + i) + pr], v);
        return v;
    }
    __device__ __forceinline__ void set(int pr, int i, V a, V b) const {
        p[N * i + pr] = put(a);
        p[N * (n + i) + pr] = put(b);
    }
};

// coefficient i of the thread's sets in global memory ([set][nc])
__device__ __forceinline__ void load_sets(const cpx<dfl> *g, int nc, int pr, int i, df2 &x, df2 &y) {
    const cpx<dfl> u = g[2 * pr * nc + i], v = g[(2 * pr + 1) * nc + i];
    x = df2{make_float2(u.x.h, v.x.h), make_float2(u.x.l, v.x.l)};
    y = df2{make_float2(u.y.h, v.y.h), make_float2(u.y.l, v.y.l)};
}
__device__ __forceinline__ void load_sets(const cpx<float> *g, int nc, int, int i, f4 &x, f4 &y) {
    const cpx<float> a = g[i], b = g[nc + i], c = g[2 * nc + i], d = g[3 * nc + i];
    x = f4{make_float2(a.x, b.x), make_float2(c.x, d.x)};
    y = f4{make_float2(a.y, b.y), make_float2(c.y, d.y)};
}
__device__ __forceinline__ void store_sets(cpx<dfl> *g, int nc, int pr, int i, df2 x, df2 y) {
    g[2 * pr * nc + i] = mk(dfl(x.h.x, x.l.x), dfl(y.h.x, y.l.x));
    g[(2 * pr + 1) * nc + i] = mk(dfl(x.h.y, x.l.y), dfl(y.h.y, y.l.y));
}
__device__ __forceinline__ void store_sets(cpx<float> *g, int nc, int, int i, f4 x, f4 y) {
    g[i] = mk(x.a.x, y.a.x);
    g[nc + i] = mk(x.a.y, y.a.y);
    g[2 * nc + i] = mk(x.b.x, y.b.x);
    g[3 * nc + i] = mk(x.b.y, y.b.y);
}
__device__ __forceinline__ void add_sets(cpx<dfl> *g, int nc, int pr, int i, df2 x, df2 y) {
    cpx<dfl> *d0 = g + 2 * pr * nc + i, *d1 = d0 + nc;
    cpx<dfl> u = *d0, v = *d1;
    u += mk(dfl(x.h.x, x.l.x), dfl(y.h.x, y.l.x));
    v += mk(dfl(x.h.y, x.l.y), dfl(y.h.y, y.l.y));
    *d0 = u;
    *d1 = v;
}
__device__ __forceinline__ void add_sets(cpx<float> *g, int nc, int, int i, f4 x, f4 y) {
    g[i] += mk(x.a.x, y.a.x);
    g[nc + i] += mk(x.a.y, y.a.y);
    g[2 * nc + i] += mk(x.b.x, y.b.x);
    g[3 * nc + i] += mk(x.b.y, y.b.y);
}

// The factored rotation of the four sets (a z rotation, the y block on real and imaginary parts, a z
// rotation) of one item: rotate_z forms tmp from (x, y), rotate_y the result from tmp.  rf: the rotation's table.
// COL: the y blocks stand as [k][m] (y_by_column).  QUARTER: the middle angle is pi/2 (the frame rotations):
// checkerboard y blocks (checked when the tables are built), Im of m = 0 zero.
template <typename T>
__device__ __forceinline__ void rotate_z(const T *rf, const int *foff, int i, int pr, typename Quad<T>::V x,
                                         typename Quad<T>::V y, Planes<T> tmp) {
    const int n = deg_of(i), m = i - tri(n, 0);
    const T *za = rf + foff[n];
    const T c = za[2 * m], sn = za[2 * m + 1];
    tmp.set(pr, i, lin2(c, x, neg1(sn), y), lin2(sn, x, c, y));
}
template <bool QUARTER, bool COL, typename T>
__device__ __forceinline__ void rotate_y(const T *rf, const int *foff, int i, int pr, Planes<T> tmp,
                                         typename Quad<T>::V &x, typename Quad<T>::V &y) {
    using V = typename Quad<T>::V;
    const int n = deg_of(i), m = i - tri(n, 0), q = n + 1, t0 = tri(n, 0);
    const T *o = rf + foff[n], *yre = o + 4 * q + (COL ? m : m * q), *yim = yre + q * q;
    const int sk = COL ? q : 1;
    V re = zero<V>(), im = re;
    if (QUARTER) {
        for (int k = (m + n) & 1; k < q; k += 2) macc(re, yre[k * sk], tmp.x(pr, t0 + k));
        if (m > 0)
            for (int k = 1 + ((m + n) & 1); k < q; k += 2) macc(im, yim[k * sk], tmp.y(pr, t0 + k));
    } else {
        for (int k = 0; k < q; ++k) {
            macc(re, yre[k * sk], tmp.x(pr, t0 + k));
            macc(im, yim[k * sk], tmp.y(pr, t0 + k));
        }
    }
    re = closed(re);
    im = closed(im);
    const T c = o[2 * q + 2 * m], sn = o[2 * q + 2 * m + 1];
    x = lin2(c, re, neg1(sn), im);
    y = lin2(sn, re, c, im);
}

}  // namespace rpy
