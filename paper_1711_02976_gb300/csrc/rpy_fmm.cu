// Far field of the RPY matvec: the four Laplace potentials of Sec. 2 through
// an adaptive FMM whose multipole-to-local step runs on plane-wave
// (exponential) expansions (M-to-I, I-to-I, I-to-L of Fig. "op").
//
// Charge sets (Sec. 2): q_1..q_3 = F^1..F^3, q_4 = F . (r - c0) with c0 the
// centre of the system's bounding cube (Eq. 2.8 holds for any common origin).
//
// Number types: T = float in the FP32 form, T = dfl (two FP32 numbers, about 48 bits: rpy_dfl.h) in the
// FP64 form, whose kernels were bound by the FP64 pipe (91 to 95% busy) at 64 times the cost of an FP32
// operation; a multiply-add is 12 FP32 operations in dfl.  Lengths are in units of a power of two at the root
// cube's side and forces in units of each system's largest (SysConst), so that every value lies well
// inside the FP32 exponent range.  Measured, matvec of the 1M-bead sphere and cube at 6 digits without its near field
// (ms), FP64 -> dfl -> now: 95 -> 37 -> 25.5 (M2X 23.4 -> 8.8 -> 5.4, X2L 20.1 -> 8.9 -> 7.3, X2X 11.9 -> 5.4 -> 3.6, L2P
// and M2P 16.6 -> 4.8 -> 2.4, P2M and P2L 14.5 -> 4.0 -> 3.65).  The velocities of whole matvecs move by
// 1e-14 ... 1.2e-13; the error of the expansions is 1e-10 at 9 digits.
//
// Kernels, in launch order:
//   k_p2x<0>   S->M   leaves: M_n^m = sum_j q_j conj(y_n^m(eta_j))
//   k_m2m, k_m2m_cluster  M->M   per child: rotate to the shift axis, z-shift, rotate back;
//                      per parent: add the children's shares in octant order (rpy_shift.cu)
//   k_m2x      M->I   rotate into the frame of each axis, outgoing plane waves
//                     W_kj = (w_k/M_k) sum_{n,m} M_n^m i^|m| lambda_k^n e^{i m a_kj} / sqrt((n-|m|)!(n+|m|)!)
//   k_x2x      I->I   merge-and-shift: per parent and direction, sources are
//                     shifted to the parent centre and summed per group of
//                     targets they serve, then shifted once to each child
//   k_x2l      I->L   L_n^m = i^|m| sum_k (-lambda_k)^n / sqrt(...) sum_j I_kj e^{-i m a_kj},
//                     rotated back to the world frame (the three: rpy_waves.cu)
//   k_p2x<1>   S->L   X list
//   k_l2l      L->L   the same for locals, level by level downward (rpy_shift.cu)
//   k_eval_prep, k_eval_apply  L->T   L2P: the gradients and Hessians of Theorems 1-2 formed as derivative
//                     expansions per leaf, combined by Eq. (2.8):
//                     u = C1 [L1 L2 L3] - C1 sum_k x_k grad L_k + C1 grad L4 - C2 grad L_C,
//                     six fields at each bead
//   k_far_eval M->T   M2P of a leaf's W list, by the same six fields
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <map>
#include <mutex>

#include "rpy_far.h"
#include "rpy_harmonics.h"

namespace rpy {

// ---------------------------------------------------------------- harmonics, several points per warp
__device__ __forceinline__ cpx<dfl> from_lane(unsigned mask, cpx<dfl> v, int lane) {
    return mk(dfl(__shfl_sync(mask, v.x.h, lane), __shfl_sync(mask, v.x.l, lane)),
              dfl(__shfl_sync(mask, v.y.h, lane), __shfl_sync(mask, v.y.l, lane)));
}

// Solid harmonics (regular, or irregular when IRREG) of one point into out[], by harm_lanes(P) consecutive lanes of
// a warp, c = 0, 1, ... : columns c and P - c each.  All lanes of the warp come here; those without a point
// (!act) store nothing.
// Double-floats: w^c by binary powers, w^(P - c) as w^(P - H) w^(H - c), H = P / 2, from the lane of column H - c, and
// the two columns as one sequence of P + 2 steps.  FP32: each lane raises w to both powers and runs its columns
// one after the other (1.5 P steps in the warp), for the shuffles and the longer loop body cost more there
// than the products they save.  Both ways in both forms, P2M: 1M mixed FP64 1.70 against 1.82 ms, 15M cube FP64 4.65
// against 5.12, 1M mixed FP32 0.52 against 0.39, 15M cube FP32 2.43 against 1.85.
template <typename T, bool IRREG>
__device__ void lane_harmonics(T x, T y, T z, int P, const T *ra, const T *rb, const T *cm, cpx<T> *out, int c,
                               bool act) {
    const T r2 = fma(z, z, fma(y, y, x * x));
    const T ir2 = IRREG ? T(1) / r2 : T(0);
    const cpx<T> w = IRREG ? mk(x * ir2, y * ir2) : mk(x, y);
    const T d0 = IRREG ? sqrt(ir2) : T(1);
    const T zz = IRREG ? z * ir2 : z;   // factor of the a-coefficients
    const T rr = IRREG ? ir2 : r2;      // factor of the b-coefficients
    if constexpr (kIsDf<T>) {
        const int H = P / 2, lane0 = (threadIdx.x & 31) - c;
        cpx<T> pw = c & 1 ? w : mk<T>(1, 0), base = w;
        for (int e = 2; e <= H; e <<= 1) {
            base = base * base;
            const cpx<T> t = pw * base;
            if (c & e) pw = t;
        }
        cpx<T> q = from_lane(0xffffffffu, pw, (lane0 + H) & 31);   // w^H
        if (P & 1) q = q * w;
        q = q * from_lane(0xffffffffu, pw, (lane0 + H - c) & 31);
        if (!act) return;
        int m = c, n = c;
        const T s0 = cm[c] * d0, s1 = cm[P - c] * d0;
        cpx<T> p1 = mk(s0 * pw.x, s0 * pw.y), p2 = mk<T>(0, 0);
        q = mk(s1 * q.x, s1 * q.y);
        for (int left = 2 * c == P ? P - c + 1 : P + 2; left > 0; --left) {
            out[tri(n, m)] = p1;
            if (n == P) {
                m = n = P - c;
                p1 = q;
                p2 = mk<T>(0, 0);
            } else {
                ++n;
                const int i = tri(n, m);
                const T A = ra[i] * zz, B = rb[i] * rr;
                const cpx<T> cn = mk(mul_diff(A, p1.x, B, p2.x), mul_diff(A, p1.y, B, p2.y));
                p2 = p1;
                p1 = cn;
            }
        }
    } else {
        if (!act) return;
        for (int h = 0; h < 2; ++h) {
            const int m = h ? P - c : c;
            if (h && m == c) break;
            cpx<T> pw = mk<T>(1, 0), base = w;   // w^m by binary powering
            for (int e = m; e; e >>= 1) {
                if (e & 1) pw = pw * base;
                base = base * base;
            }
            const T s0 = cm[m] * d0;
            cpx<T> p1 = mk(s0 * pw.x, s0 * pw.y), p2 = mk<T>(0, 0);
            out[tri(m, m)] = p1;
            for (int n = m + 1; n <= P; ++n) {
                const int i = tri(n, m);
                const T A = ra[i] * zz, B = rb[i] * rr;
                const cpx<T> cn = mk(mul_diff(A, p1.x, B, p2.x), mul_diff(A, p1.y, B, p2.y));
                out[i] = cn;
                p2 = p1;
                p1 = cn;
            }
        }
    }
}

// Streaming per-thread evaluation of NE real fields f_q = sum_{n<=P,m} w_m Re(E_q[n,m] h_n^m(v)),
// w_0 = 1, w_m = 2 (m > 0); W2: the coefficients already carry w_m.
template <typename T, int NE, bool IRREG, bool W2 = false>
__device__ void eval_fields(T x, T y, T z, int P, const cpx<T> *E, int stride, const T *ra, const T *rb,
                            const T *rc, T *acc) {
    const T r2 = fma(z, z, fma(y, y, x * x));
    const T ir2 = IRREG ? T(1) / r2 : T(0);
    const cpx<T> w = IRREG ? mk(x * ir2, y * ir2) : mk(x, y);
    const T zz = IRREG ? z * ir2 : z;
    const T rr = IRREG ? ir2 : r2;
    cpx<T> diag = IRREG ? mk<T>(sqrt(ir2), 0) : mk<T>(1, 0);
    for (int m = 0; m <= P; ++m) {
        if (m > 0) diag = rc[m] * (w * diag);
        const T wm = (W2 || m == 0) ? T(1) : T(2);
        cpx<T> p2 = mk<T>(0, 0), p1 = diag;
        {
            const int i = tri(m, m);
            const cpx<T> hw = W2 ? diag : mk(wm * diag.x, wm * diag.y);
#pragma unroll
            for (int q = 0; q < NE; ++q) {
                const cpx<T> e = E[q * stride + i];
                macc(acc[q], e.x, hw.x);
                macc(acc[q], -e.y, hw.y);
            }
        }
        for (int n = m + 1; n <= P; ++n) {
            const int i = tri(n, m);
            const T A = ra[i] * zz, B = rb[i] * rr;
            const cpx<T> c = mk(mul_diff(A, p1.x, B, p2.x), mul_diff(A, p1.y, B, p2.y));
            const cpx<T> hw = W2 ? c : mk(wm * c.x, wm * c.y);
#pragma unroll
            for (int q = 0; q < NE; ++q) {
                const cpx<T> e = E[q * stride + i];
                macc(acc[q], e.x, hw.x);
                macc(acc[q], -e.y, hw.y);
            }
            p2 = p1;
            p1 = c;
        }
    }
#pragma unroll
    for (int q = 0; q < NE; ++q) acc[q] = closed(acc[q]);
}

// Coefficient i of the six fields of fold_fields.
__device__ __forceinline__ void load_six(const cpx<float> *E, int i, cpx<float> (&e)[6]) {
    const float4 *q = reinterpret_cast<const float4 *>(E + 6 * i);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float4 v = q[k];
        e[2 * k] = mk(v.x, v.y);
        e[2 * k + 1] = mk(v.z, v.w);
    }
}
__device__ __forceinline__ void load_six(const cpx<dfl> *E, int i, cpx<dfl> (&e)[6]) {
    const float4 *q = reinterpret_cast<const float4 *>(E + 6 * i);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float4 v = q[k];
        e[k] = mk(dfl(v.x, v.y), dfl(v.z, v.w));
    }
}

// The six fields of fold_fields at one point.  AHEAD: each step's coefficients are loaded a step before, for few warps
// hide the loads where they come from global memory (k_eval_apply: 20,001 beads, 6 digits, FP64 0.16 -> 0.11 ms
// together with the bound on its registers) or the registers leave room for few (double-floats); the FP32 k_far_eval has
// warps enough and gains nothing.
template <typename T, bool IRREG, bool AHEAD>
__device__ void eval_six(T x, T y, T z, int P, const cpx<T> *E, const T *ra, const T *rb, const T *rc, T *acc) {
    const T r2 = fma(z, z, fma(y, y, x * x));
    const T ir2 = IRREG ? T(1) / r2 : T(0);
    const cpx<T> w = IRREG ? mk(x * ir2, y * ir2) : mk(x, y);
    const T zz = IRREG ? z * ir2 : z;
    const T rr = IRREG ? ir2 : r2;
    cpx<T> diag = IRREG ? mk<T>(sqrt(ir2), 0) : mk<T>(1, 0);
    cpx<T> e[6], f[6];
    if constexpr (AHEAD) load_six(E, 0, e);
    for (int m = 0; m <= P; ++m) {
        if (m > 0) diag = rc[m] * (w * diag);
        cpx<T> p2 = mk<T>(0, 0), p1 = diag;
#pragma unroll 2
        for (int n = m;;) {
            const bool last = n == P;
            T a, b;
            if constexpr (AHEAD) {
                const int i = last ? (m < P ? tri(m + 1, m + 1) : 0) : tri(n + 1, m);
                load_six(E, i, f);
                a = ra[i], b = rb[i];
            } else {
                load_six(E, tri(n, m), e);
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                macc(acc[q], e[q].x, p1.x);
                macc(acc[q], -e[q].y, p1.y);
            }
            if constexpr (AHEAD)
#pragma unroll
                for (int q = 0; q < 6; ++q) e[q] = f[q];
            if (last) break;
            ++n;
            if constexpr (!AHEAD) a = ra[tri(n, m)], b = rb[tri(n, m)];
            const T A = a * zz, B = b * rr;
            const cpx<T> c = mk(mul_diff(A, p1.x, B, p2.x), mul_diff(A, p1.y, B, p2.y));
            p2 = p1;
            p1 = c;
        }
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) acc[q] = closed(acc[q]);
}

// ---------------------------------------------------------------- derivative expansions
// Real-field derivative expansions (ladder relations of Sec. 2, Theorems 1-2),
// computed by the whole CTA.  src: degree ps coefficients.  dst: x, y, z
// derivatives, each zero-padded to stride.
template <typename T>
struct Lad {
    const T *lz, *lp, *lq, *mz, *mp, *mq;
};

template <typename T>
__device__ void d_local(const cpx<T> *src, int ps, cpx<T> *dx, cpx<T> *dy, cpx<T> *dz, int P, const Lad<T> &G) {
    // degree k <= ps-1 from L_{k+1}
    for (int i = threadIdx.x; i < ncoef(P); i += blockDim.x) {
        int k = deg_of(i), m = i - tri(k, 0);
        cpx<T> X = mk<T>(0, 0), Y = X, Z = X;
        if (k <= ps - 1) {
            Z = G.lz[i] * src[tri(k + 1, m)];
            cpx<T> Pv = m >= 1 ? G.lp[i] * src[tri(k + 1, m - 1)] : (-G.lq[i]) * conj(src[tri(k + 1, 1)]);
            cpx<T> Qv = (-G.lq[i]) * src[tri(k + 1, m + 1)];
            X = mk(T(0.5) * (Pv.x + Qv.x), T(0.5) * (Pv.y + Qv.y));
            Y = mk(T(0.5) * (Pv.y - Qv.y), T(-0.5) * (Pv.x - Qv.x));
        }
        dx[i] = X;
        dy[i] = Y;
        dz[i] = Z;
    }
}

template <typename T>
__device__ void d_multipole(const cpx<T> *src, int ps, cpx<T> *dx, cpx<T> *dy, cpx<T> *dz, int P, const Lad<T> &G) {
    // degree k <= ps+1 from M_{k-1}
    for (int i = threadIdx.x; i < ncoef(P); i += blockDim.x) {
        int k = deg_of(i), m = i - tri(k, 0);
        cpx<T> X = mk<T>(0, 0), Y = X, Z = X;
        if (k >= 1 && k <= ps + 1) {
            if (m <= k - 1) Z = (-G.mz[i]) * src[tri(k - 1, m)];
            cpx<T> Pv = mk<T>(0, 0), Qv = mk<T>(0, 0);
            if (m >= 1) Pv = G.mp[i] * src[tri(k - 1, m - 1)];
            else if (k >= 2) Pv = (-G.mp[i]) * conj(src[tri(k - 1, 1)]);
            if (m + 1 <= k - 1) Qv = (-G.mq[i]) * src[tri(k - 1, m + 1)];
            X = mk(T(0.5) * (Pv.x + Qv.x), T(0.5) * (Pv.y + Qv.y));
            Y = mk(T(0.5) * (Pv.y - Qv.y), T(-0.5) * (Pv.x - Qv.x));
        }
        dx[i] = X;
        dy[i] = Y;
        dz[i] = Z;
    }
}

// Coefficient i of one component c (0 = x, 1 = y, 2 = z) of the gradient of a
// local (d_loc_one) or multipole (d_mul_one) expansion of degree ps: the
// single-output forms of d_local and d_multipole.
template <typename T>
__device__ __forceinline__ cpx<T> d_loc_one(const cpx<T> *src, int ps, int c, int i, const Lad<T> &G) {
    const int k = deg_of(i), m = i - tri(k, 0);
    if (k > ps - 1) return mk<T>(0, 0);
    if (c == 2) return G.lz[i] * src[tri(k + 1, m)];
    const cpx<T> Pv = m >= 1 ? G.lp[i] * src[tri(k + 1, m - 1)] : (-G.lq[i]) * conj(src[tri(k + 1, 1)]);
    const cpx<T> Qv = (-G.lq[i]) * src[tri(k + 1, m + 1)];
    return c == 0 ? mk(T(0.5) * (Pv.x + Qv.x), T(0.5) * (Pv.y + Qv.y))
                  : mk(T(0.5) * (Pv.y - Qv.y), T(-0.5) * (Pv.x - Qv.x));
}

template <typename T>
__device__ __forceinline__ cpx<T> d_mul_one(const cpx<T> *src, int ps, int c, int i, const Lad<T> &G) {
    const int k = deg_of(i), m = i - tri(k, 0);
    if (k < 1 || k > ps + 1) return mk<T>(0, 0);
    if (c == 2) return m <= k - 1 ? (-G.mz[i]) * src[tri(k - 1, m)] : mk<T>(0, 0);
    cpx<T> Pv = mk<T>(0, 0), Qv = mk<T>(0, 0);
    if (m >= 1) Pv = G.mp[i] * src[tri(k - 1, m - 1)];
    else if (k >= 2) Pv = (-G.mp[i]) * conj(src[tri(k - 1, 1)]);
    if (m + 1 <= k - 1) Qv = (-G.mq[i]) * src[tri(k - 1, m + 1)];
    return c == 0 ? mk(T(0.5) * (Pv.x + Qv.x), T(0.5) * (Pv.y + Qv.y))
                  : mk(T(0.5) * (Pv.y - Qv.y), T(-0.5) * (Pv.x - Qv.x));
}

// ---------------------------------------------------------------- table access
template <typename T>
struct Rec {
    const T *a, *b, *c, *cm;
};

template <typename T>
__device__ Rec<T> load_rec(const DevTables<T> &D, T *sm) {
    int P = D.p + 2;
    int nc = ncoef(P);
    for (int i = threadIdx.x; i < nc; i += blockDim.x) {
        sm[i] = D.rec_a[i];
        sm[nc + i] = D.rec_b[i];
    }
    for (int i = threadIdx.x; i <= P; i += blockDim.x) {
        sm[2 * nc + i] = D.rec_c[i];
        sm[2 * nc + P + 1 + i] = D.rec_cm[i];
    }
    Rec<T> r{sm, sm + nc, sm + 2 * nc, sm + 2 * nc + P + 1};
    return r;
}

// ladder tables follow the recurrence tables in shared memory
template <typename T>
__device__ Lad<T> load_lad(const DevTables<T> &D, T *sm) {
    int nl = ncoef(D.p + 2);
    for (int i = threadIdx.x; i < 6 * nl; i += blockDim.x) sm[i] = D.lad[i];
    Lad<T> g{sm, sm + nl, sm + 2 * nl, sm + 3 * nl, sm + 4 * nl, sm + 5 * nl};
    return g;
}

template <typename T>
__host__ __device__ inline int rec_floats(int p) {
    return 2 * ncoef(p + 2) + 2 * (p + 3);
}

template <typename T>
__host__ __device__ inline int tab_floats(int p) {   // recurrences + ladders, rounded to an even count
    return ((rec_floats<T>(p) + 6 * ncoef(p + 2)) + 1) & ~1;
}


// ---------------------------------------------------------------- P2M / P2L

__device__ __forceinline__ float2 pair2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ df2 pair2(dfl a, dfl b) { return df2{make_float2(a.h, b.h), make_float2(a.l, b.l)}; }
__device__ __forceinline__ float first(float2 v) { return v.x; }
__device__ __forceinline__ float second(float2 v) { return v.y; }
__device__ __forceinline__ dfl first(df2 v) { return dfl(v.h.x, v.l.x); }
__device__ __forceinline__ dfl second(df2 v) { return dfl(v.h.y, v.l.y); }
__device__ __forceinline__ void macc2(float2 &s, float2 a, float2 b) { s = fma2(a, b, s); }
__device__ __forceinline__ void macc2(df2 &s, df2 a, df2 b) { macc(s, a, b); }
__device__ __forceinline__ void add_comp(float2 &s, float2 &c, float2 v) {   // s - c += v (Kahan)
    const float2 y = sub2(v, c), t = add2(s, y);
    c = sub2(sub2(t, s), y);
    s = t;
}

// Running sums of one coefficient for the four charge sets: re[h], im[h] of sets 2h and 2h + 1; in FP32 with the
// compensation of each (double-floats are only normalised).
template <typename T>
struct Sum4 {
    typename PairOf<T>::V v[4], c[sizeof(T) == 4 ? 4 : 1];
    __device__ void clear() {
        const auto z = pair2(T(0), T(0));
        for (auto &x : v) x = z;
        for (auto &x : c) x = z;
    }
    __device__ void add(const typename PairOf<T>::V *u) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if constexpr (sizeof(T) == 4) add_comp(v[k], c[k], u[k]);
            else v[k] = renorm(sum_raw(v[k], u[k]));
        }
    }
    __device__ void join(const Sum4 &o) {
        add(o.v);
        if constexpr (sizeof(T) == 4) {
            float2 m[4];
            for (int k = 0; k < 4; ++k) m[k] = neg2(o.c[k]);
            add(m);
        }
    }
};

// Threads of a P2M / P2L block: G = threads / ncoef groups of one thread per coefficient.  At low orders two warps, for
// the groups' joining costs as much as their sums (P2M, p = 6, 15M cube: FP64 4.10 ms, FP32 1.49 ms; four warps 4.65 and
// 1.86); four where there are too few boxes to fill the chip (585 boxes: 15 us against 17).
inline int p2x_threads(int p, int nbox) {
    const int nc = ncoef(p);
    return (std::max(1, (nbox < 1024 ? 128 : 64) / nc) * nc + 31) / 32 * 32;
}
// Beads per chunk: one round of harmonics (warps x points per warp) in at most kP2xBuf bytes (9 digits, p = 25, P2M: 32 KB
// 1.78 ms, 64 KB 1.24, 96 KB 1.10).
constexpr int kP2xStage = 128;   // beads staged at a time: coordinates and charges
constexpr int kP2xBuf = 96 * 1024;
template <typename T>
__host__ __device__ inline int p2x_chunk(int p, int threads) {
    const int most = kP2xBuf / int(ncoef(p) * sizeof(cpx<T>)), one = (threads / 32) * (32 / harm_lanes(p));
    return one < most ? one : most;
}
template <typename T>
__host__ __device__ inline int p2x_buf(int p, int threads) {   // harmonics of a chunk, later the groups' sums
    const int y = p2x_chunk<T>(p, threads) * ncoef(p) * int(sizeof(cpx<T>)), r = threads * int(sizeof(Sum4<T>));
    return ((y > r ? y : r) + 15) & ~15;
}

// Bound by the harmonics (a chain per lane) and, at low orders, by the synchronised phases of each leaf; in FP32 also by
// the FP64 coordinates, taken once per bead and box: every lane of a point's harmonics took them before.  A
// coefficient's four sums stay in registers and share each loaded harmonic; they stood in shared memory, a thread per
// coefficient and set, with two loads for every two products.  P2M and P2L before and now: 1M mixed FP64 1.97 -> 1.70
// and 2.06 -> 1.95 ms, FP32 0.49 -> 0.39 and 0.89 -> 0.73; 200k at 9 digits 1.21 -> 0.94 and 1.16 -> 0.83; 15M cube P2M
// FP64 5.05 -> 4.10 and FP32 2.02 -> 1.49; 256 systems FP32 2.57 -> 2.05 and 2.37 -> 2.02.
// MODE 0: P2M over the leaf's own beads (multipole about its centre)
// MODE 1: P2L over the beads of every box in X(b) (local about b's centre)
// The fourth charge q4 = F . (r - o) takes its origin o at the expansion's own
// centre when rb is set (box origin), else at the system's cube centre.
template <typename T, int MODE>
__global__ void __launch_bounds__(512) k_p2x(int b0, int nb, DevTables<T> D, const int *beg, const int *end,
                                             const double *ctr, const int *lvl, const int *leaf,
                                             const int *bsys, const int *xoff, const int *xidx, const double *pos,
                                             const double *fs, const double *lapq, int64_t n, SysConst sc, cpx<T> *out,
                                             int rb) {
    using V = typename PairOf<T>::V;
    const int chunk = p2x_chunk<T>(D.p, blockDim.x);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = b0 + blockIdx.x;
    if (b >= b0 + nb) return;
    if (lvl[b] < 2) return;
    if (MODE == 0 && !leaf[b]) return;
    int nsrc = MODE == 0 ? 1 : xoff[b + 1] - xoff[b];
    if (nsrc == 0) return;
    const int p = D.p, nc = ncoef(p);
    cpx<T> *ybuf = reinterpret_cast<cpx<T> *>(smem_raw);
    V *q = reinterpret_cast<V *>(smem_raw + p2x_buf<T>(p, blockDim.x));   // [bead][2]
    T *X = reinterpret_cast<T *>(q + 2 * kP2xStage);   // coordinates in box sides, [3][bead]
    Rec<T> R = load_rec(D, X + 3 * kP2xStage);
    int sy = bsys[b];
    double cx = ctr[3 * b], cy = ctr[3 * b + 1], cz = ctr[3 * b + 2];
    const double c0x = rb ? cx : sc.cube[4 * sy], c0y = rb ? cy : sc.cube[4 * sy + 1],
                 c0z = rb ? cz : sc.cube[4 * sy + 2];   // origin of q4
    const double ih = sc.pc[sy].icube * pow2i(lvl[b]);   // 1 / side[b], exactly
    // double-floats: the box centre in the split units of the positions, and 1 / side in them
    float c3[9];
    T ihs = T(0);
    double qs = 1.0;   // scale of given charges
    if constexpr (kIsDf<T>) {
        for (int k = 0; k < 9; ++k) c3[k] = sc.c3[9 * size_t(b) + k];
        ihs = T(inv_side_u(sc.pc[sy], lvl[b]));
        qs = force_scale(sc.fmax[sy]);
    }
    int warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    // harmonics: hG points per warp, lane -> (point hg, column pair hc)
    const int hL = harm_lanes(p), hG = 32 / hL, hg = (threadIdx.x & 31) / hL, hc = (threadIdx.x & 31) - hg * hL;
    // sums: this thread's coefficient i, and every G-th bead of a chunk from g on
    const int G = blockDim.x / nc, g = threadIdx.x / nc, i = threadIdx.x - g * nc;
    Sum4<T> sum;
    sum.clear();
    __syncthreads();
    for (int si = 0; si < nsrc; ++si) {
        int src = MODE == 0 ? b : xidx[xoff[b] + si];
        for (int js = beg[src], j1 = end[src]; js < j1; js += kP2xStage) {
            const int ns = min(kP2xStage, j1 - js);
            for (int t = threadIdx.x; t < ns; t += blockDim.x) {
                int j = js + t;
                if constexpr (kIsDf<T>) {
                    for (int a = 0; a < 3; ++a) X[a * kP2xStage + t] = coord_diff(sc.p3, n, j, a, c3) * ihs;
                } else {
                    X[t] = T((pos[j] - cx) * ih);
                    X[kP2xStage + t] = T((pos[n + j] - cy) * ih);
                    X[2 * kP2xStage + t] = T((pos[2 * n + j] - cz) * ih);
                }
                T c[kSets];
                if (lapq) {
                    for (int k = 0; k < kSets; ++k) c[k] = T(kIsDf<T> ? qs * lapq[4 * j + k] : lapq[4 * j + k]);
                } else if constexpr (kIsDf<T>) {
                    // scaled forces; q4 in the split units of length, its origin at the cube's or the box's centre
                    float o3[9];
                    for (int k = 0; k < 9; ++k) o3[k] = rb ? c3[k] : 0.f;
                    T q4 = T(0);
                    for (int a = 0; a < 3; ++a) {
                        c[a] = T(sc.f2[(2 * a) * n + j], sc.f2[(2 * a + 1) * n + j]);
                        macc(q4, c[a], coord_diff(sc.p3, n, j, a, o3));
                    }
                    c[3] = closed(q4);
                } else {
                    double fx = fs[j], fy = fs[n + j], fz = fs[2 * n + j];
                    c[0] = T(fx);
                    c[1] = T(fy);
                    c[2] = T(fz);
                    c[3] = T(fx * (pos[j] - c0x) + fy * (pos[n + j] - c0y) + fz * (pos[2 * n + j] - c0z));
                }
                q[2 * t] = pair2(c[0], c[1]);
                q[2 * t + 1] = pair2(c[2], c[3]);
            }
            __syncthreads();
            for (int jc = 0; jc < ns; jc += chunk) {
                const int cnt = min(chunk, ns - jc);
                for (int t0 = warp * hG; t0 < cnt; t0 += nwarp * hG) {
                    const int t = t0 + hg;
                    const bool act = hg < hG && t < cnt;
                    const T *x = X + jc + (act ? t : 0);
                    lane_harmonics<T, MODE == 1>(x[0], x[kP2xStage], x[2 * kP2xStage], p, R.a, R.b, R.cm, ybuf + t * nc, hc,
                                                 act);
                }
                __syncthreads();
                if (g < G) {
                    const V z = pair2(T(0), T(0));
                    V u[4] = {z, z, z, z};
                    for (int t = g; t < cnt; t += G) {
                        const cpx<T> yv = ybuf[t * nc + i];
                        const V re = pair2(yv.x, yv.x), im = pair2(-yv.y, -yv.y);   // conj
    #pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const V c = q[2 * (jc + t) + h];
                            macc2(u[2 * h], c, re);
                            macc2(u[2 * h + 1], c, im);
                        }
                    }
                    // a leaf (or an X-list source) may hold hundreds to thousands of beads: in FP32 the
                    // chunk's plain sum enters the running sum by compensated (Kahan) addition
                    sum.add(u);
                }
                __syncthreads();
            }
        }
    }
    if (G > 1) {
        Sum4<T> *red = reinterpret_cast<Sum4<T> *>(smem_raw);
        if (g > 0 && g < G) red[threadIdx.x] = sum;
        __syncthreads();
        if (g == 0)
            for (int h = 1; h < G; ++h) sum.join(red[h * nc + i]);
    }
    if (g > 0) return;
    cpx<T> *o = out + size_t(b) * kSets * nc + i;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const cpx<T> a = mk(first(sum.v[2 * h]), first(sum.v[2 * h + 1])),
                     c = mk(second(sum.v[2 * h]), second(sum.v[2 * h + 1]));
        if (MODE == 0) {
            o[2 * h * nc] = a;
            o[(2 * h + 1) * nc] = c;
        } else {
            o[2 * h * nc] += a;
            o[(2 * h + 1) * nc] += c;
        }
    }
}

// ---------------------------------------------------------------- far-field evaluation
constexpr int kNE = 18;   // evaluation expansions of Eq. (2.8) per box
constexpr int kNF = 12;   // evaluated per bead after the fold of k_eval_prep (per-potential form)
constexpr int kNF2 = 6;   // evaluated per bead in the one-expansion-per-component form
constexpr int kFarGroups = 4;   // source boxes per round of k_far_eval at most

// tables of k_far_eval (recurrences, ladders, 1 / (2k + 1)) and k_eval_prep (the last two), 16-byte multiples
template <typename T>
__host__ __device__ inline int far_tab_floats(int p) {
    return (tab_floats<T>(p) + p + 4 + 3) & ~3;
}
template <typename T>
__host__ __device__ inline int prep_tab_floats(int p) {
    return (6 * ncoef(p + 2) + p + 4 + 3) & ~3;
}

// Build the 18 evaluation expansions of Eq. (2.8) from 4 local expansions (the per-potential form).
template <typename T>
__device__ void build_eval_set(const cpx<T> *src, int p, int P, cpx<T> *EV, cpx<T> *tmp, T cbx, T cby, T cbz,
                               const Lad<T> &G) {
    const int st = ncoef(P);
    // 0..2 values
    for (int i = threadIdx.x; i < 3 * st; i += blockDim.x) {
        int k = i / st, c = i - k * st;
        EV[k * st + c] = c < ncoef(p) ? src[k * ncoef(p) + c] : mk<T>(0, 0);
    }
    // 3..11 gradients of sets 0..2 (index 3 + 3k + a), tmp[0..2] gradient of set 3
    for (int k = 0; k < 4; ++k) {
        cpx<T> *gx = k < 3 ? EV + (3 + 3 * k) * st : tmp;
        d_local(src + k * ncoef(p), p, gx, gx + st, gx + 2 * st, P, G);
    }
    __syncthreads();
    // 12..14: G4'_a = dL4_a - sum_k cb_k dL_k,a ; tmp[3] = L_C = dxL1 + dyL2 + dzL3
    const T cb[3] = {cbx, cby, cbz};
    for (int i = threadIdx.x; i < st; i += blockDim.x) {
        for (int a = 0; a < 3; ++a) {
            cpx<T> g = tmp[a * st + i];
            for (int k = 0; k < 3; ++k) {
                cpx<T> v = EV[(3 + 3 * k + a) * st + i];
                macc(g.x, -cb[k], v.x);
                macc(g.y, -cb[k], v.y);
            }
            EV[(12 + a) * st + i] = mk(closed(g.x), closed(g.y));
        }
        cpx<T> lc = EV[(3 + 0) * st + i] + EV[(3 + 3 + 1) * st + i] + EV[(3 + 6 + 2) * st + i];
        tmp[3 * st + i] = lc;
    }
    __syncthreads();
    d_local(tmp + 3 * st, p - 1, EV + 15 * st, EV + 16 * st, EV + 17 * st, P, G);
    __syncthreads();
}

// Eq. (2.8) of one expansion of degree p as six fields, with x the offset from the expansion's centre in box sides
// and o its centre relative to the origin of q4 (Approach 2 of Sec. 2, one expansion per velocity component):
//   u_d = L_d - sum_k x_k dL_k/dx_d + c4 dS/dx_d - cc dL_C/dx_d,  S = L4 - sum_k o_k L_k,  L_C = sum_k dL_k/dx_k
// in units of C1/h.  A coordinate times a harmonic function splits into harmonic ones (Kelvin transform): for each
// degree-n part h of a local expansion, with g = h / (2n + 1),
//   x_k h = [x_k h - |x|^2 d_k g] + |x|^2 d_k g,
// where the bracket is -|x|^(2n+3) d_k(g / |x|^(2n+1)): the coefficients of d_k g taken as a multipole expansion's,
// negated and read as a local one's.  For a multipole expansion the two swap, its local-form
// derivative being the bracket's part without |x|^2.  So
//   sum_k x_k L_k = U + |x|^2 V,  sum_k x_k dL_k/dx_d = d_d(U + |x|^2 V) - L_d = d_d U + 2 x_d V + |x|^2 d_d V - L_d,
// and with x_d V = Y_d + |x|^2 Z_d
//   u_d = [2 L_d + d_d(c4 S - U - cc L_C) - 2 Y_d] - |x|^2 [d_d V + 2 Z_d].
// V and Z are the native derivatives (L_C and d_d V) scaled by degree: two scalar expansions are differentiated where
// the gradients of all three L_k would be three times the work.  inv[k] = 1 / (2k + 1).  The fields
// carry the factor 2 of the m > 0 terms of Re(sum E h) and stand interleaved, [coefficient][6].
template <typename T, bool IRREG>
__device__ __forceinline__ cpx<T> d_native(const cpx<T> *src, int ps, int c, int i, const Lad<T> &G) {
    return IRREG ? d_mul_one(src, ps, c, i, G) : d_loc_one(src, ps, c, i, G);
}

template <typename T, bool IRREG>
__device__ __forceinline__ void fold_scalars(const cpx<T> *src, int p, int i, T c4, T cc, const T *o, const T *inv,
                                             const Lad<T> &G, cpx<T> *phi, cpx<T> *V) {
    const int nc = ncoef(p), k = deg_of(i);
    cpx<T> lc = mk<T>(0, 0), x = lc, S = lc;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lc += d_native<T, IRREG>(src + c * nc, p, c, i, G);
        x += d_native<T, !IRREG>(src + c * nc, p, c, i, G);
    }
    if (i < nc) {
        S = src[3 * nc + i];
        for (int c = 0; c < 3; ++c) {
            const cpx<T> v = src[c * nc + i];
            macc(S.x, -o[c], v.x);
            macc(S.y, -o[c], v.y);
        }
        S = mk(closed(S.x), closed(S.y));
    }
    const T up = inv[k + 1], dn = inv[max(k - 1, 0)];   // (no derivative raises to degree 0)
    V[i] = (IRREG ? -dn : up) * lc;
    const T u = IRREG ? -up : dn;
    cpx<T> f = mk(c4 * S.x, c4 * S.y);
    macc(f.x, u, x.x);
    macc(f.y, u, x.y);
    macc(f.x, -cc, lc.x);
    macc(f.y, -cc, lc.y);
    phi[i] = mk(closed(f.x), closed(f.y));
}

template <typename T, bool IRREG>
__device__ __forceinline__ void fold_fields(const cpx<T> *src, int p, int i, const T *inv, const Lad<T> &G,
                                            const cpx<T> *phi, const cpx<T> *V, cpx<T> *out) {
    const int nc = ncoef(p), k = deg_of(i), pv = IRREG ? p + 1 : p - 1;
    const T up = inv[k + 1], dn = inv[max(k - 1, 0)];
    const float w = i == tri(k, 0) ? 1.f : 2.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const cpx<T> a = d_native<T, IRREG>(V, pv, d, i, G), b = d_native<T, !IRREG>(V, pv, d, i, G);
        cpx<T> h = d_native<T, IRREG>(phi, p + 1, d, i, G);
        if (i < nc) {
            const cpx<T> v = src[d * nc + i];
            h += mk(scale2(2.f, v.x), scale2(2.f, v.y));
        }
        h += scale2(2.f, IRREG ? -up : dn) * b;
        const T z = T(1) + scale2(2.f, IRREG ? -dn : up);
        out[6 * i + d] = mk(scale2(w, h.x), scale2(w, h.y));
        const cpx<T> B = z * a;
        out[6 * i + 3 + d] = mk(scale2(w, B.x), scale2(w, B.y));
    }
}

template <typename T>
__device__ const T *load_inv(T *sm, int p) {   // p + 4 entries
    for (int k = threadIdx.x; k < p + 4; k += blockDim.x) {
        if constexpr (kIsDf<T>) sm[k] = recip(T(2 * k + 1));
        else sm[k] = T(1) / T(2 * k + 1);
    }
    return sm;
}

// M2P of the W lists, a near-field work item (at most kItemTargets beads of a leaf) per block: the six fields of
// `groups` source boxes at a time are formed in shared memory by the whole block, and each box then is evaluated
// by its own group of threads, one bead each.
// Bound by the FP32 pipe (the macc of the fields) and the loads of the fields from shared memory.  Eighteen fields per box,
// formed for every 64 beads of the leaf, took twice the arithmetic and three times the loads; a block per leaf left
// the large leaves of a cluster to run alone.  Evaluation stage before and now: 1M mixed, 6 digits, FP64 4.72 -> 2.40 ms,
// FP32 1.86 -> 0.82 ms; 256 systems FP32 4.77 -> 3.29 ms; a Plummer cluster of 30,001 beads 416 -> 180 us.  64 threads: FP32
// 0.96 ms; 256: 0.78 ms, but 256 systems 3.57 ms, most of whose items have no W list; two boxes a round instead of up to four:
// the same within 1%.
constexpr int kFarThreads = 128;
template <typename T>
struct FarBox {   // one source box of the round
    T c4, cc, o[3];
    double w;     // per velocity: C1 / side, with the force unit
    int box;
};
template <typename T>
__global__ void __launch_bounds__(kFarThreads) k_far_eval(const int4 *items, DevTables<T> D, const double *ctr,
                                                          const int *lvl, const int *bsys, const int *woff,
                                                          const int *widx, const double *pos, int64_t n, SysConst sc,
                                                          const cpx<T> *M, double *ufar, int rb, int groups) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ FarBox<T> sB[kFarGroups];
    __shared__ double sU[3][kItemTargets];
    const int4 item = items[blockIdx.x];
    const int w0 = woff[item.x], nw = woff[item.x + 1] - w0;
    if (nw == 0) return;
    const int p = D.p, nc = ncoef(p), n1 = ncoef(p + 1), P = p + 2, st = ncoef(P), sy = bsys[item.y];
    T *smr = reinterpret_cast<T *>(smem_raw);
    const Rec<T> R = load_rec(D, smr);
    const Lad<T> G = load_lad(D, smr + rec_floats<T>(p));
    const T *inv = load_inv(smr + tab_floats<T>(p), p);
    const int per = kSets * nc + 2 * n1 + 6 * st;
    cpx<T> *box0 = reinterpret_cast<cpx<T> *>(smr + far_tab_floats<T>(p));
    const PairConst &pc = sc.pc[sy];
    const int nt = item.w - item.z, rows = min(nt, kFarThreads), ng = min(min(groups, nw), kFarThreads / rows);
    const int tl = threadIdx.x % rows, g = threadIdx.x / rows;
    for (int e = threadIdx.x; e < 3 * kItemTargets; e += kFarThreads) sU[0][e] = 0.0;
    for (int wb = 0; wb < nw; wb += ng) {
        const int nb = min(ng, nw - wb);
        __syncthreads();
        if (threadIdx.x < nb) {
            FarBox<T> B;
            const int C = B.box = widx[w0 + wb + threadIdx.x];
            if constexpr (kIsDf<T>) {   // lengths in the split units: C2 / C1 = 2a^2/3 there
                const double ihd = inv_side_u(pc, lvl[C]);
                B.c4 = T(ihd);
                B.cc = T((double(pc.d_k23h) + double(pc.d_k23l)) * ihd * ihd);
                const float *c = sc.c3 + 9 * size_t(C);
                for (int a = 0; a < 3; ++a) B.o[a] = rb ? T(0) : dfl3(c[3 * a], c[3 * a + 1], c[3 * a + 2]);
                B.w = pc.C1 * pc.d_xs * force_unit(sc.fmax[sy]) * ihd;
            } else {
                const double ih = pc.icube * pow2i(lvl[C]);   // 1 / side[C], exactly
                B.c4 = T(ih);
                B.cc = T(pc.C2 / pc.C1 * ih * ih);
                for (int a = 0; a < 3; ++a) B.o[a] = rb ? T(0) : T(ctr[3 * C + a] - sc.cube[4 * sy + a]);
                B.w = pc.C1 * ih;
            }
            sB[threadIdx.x] = B;
        }
        for (int e = threadIdx.x; e < nb * kSets * nc; e += kFarThreads) {
            const int gg = e / (kSets * nc), r = e - gg * kSets * nc;
            box0[gg * per + r] = M[size_t(widx[w0 + wb + gg]) * kSets * nc + r];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < nb * n1; e += kFarThreads) {
            const int gg = e / n1;
            cpx<T> *src = box0 + gg * per, *phi = src + kSets * nc;
            fold_scalars<T, true>(src, p, e - gg * n1, sB[gg].c4, sB[gg].cc, sB[gg].o, inv, G, phi, phi + n1);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < nb * st; e += kFarThreads) {
            const int gg = e / st;
            cpx<T> *src = box0 + gg * per, *phi = src + kSets * nc;
            fold_fields<T, true>(src, p, e - gg * st, inv, G, phi, phi + n1, phi + 2 * n1);
        }
        __syncthreads();
        if (g < nb) {
            const int C = sB[g].box;
            const cpx<T> *E = box0 + g * per + kSets * nc + 2 * n1;
            const double w = sB[g].w;
            for (int t = tl; t < nt; t += rows) {   // one group takes more than one bead a thread
                const int j = item.z + t;
                double *u = &sU[0][g * rows + t];
                T acc[6];
#pragma unroll
                for (int q = 0; q < 6; ++q) acc[q] = T(0);
                if constexpr (kIsDf<T>) {
                    const float *c = sc.c3 + 9 * size_t(C);
                    const T ihs = sB[g].c4;
                    const T x = coord_diff(sc.p3, n, j, 0, c) * ihs, y = coord_diff(sc.p3, n, j, 1, c) * ihs,
                            z = coord_diff(sc.p3, n, j, 2, c) * ihs;
                    eval_six<T, true, kIsDf<T>>(x, y, z, P, E, R.a, R.b, R.c, acc);
                    const T r2 = fma(z, z, fma(y, y, x * x));
                    for (int d = 0; d < 3; ++d) u[d * kItemTargets] += w * double(acc[d] - r2 * acc[3 + d]);
                } else {
                    const double ih = pc.icube * pow2i(lvl[C]);
                    const double x = (pos[j] - ctr[3 * C]) * ih, y = (pos[n + j] - ctr[3 * C + 1]) * ih,
                                 z = (pos[2 * n + j] - ctr[3 * C + 2]) * ih;
                    eval_six<T, true, kIsDf<T>>(T(x), T(y), T(z), P, E, R.a, R.b, R.c, acc);
                    const double r2 = x * x + y * y + z * z;
                    for (int d = 0; d < 3; ++d) u[d * kItemTargets] += w * (double(acc[d]) - r2 * double(acc[3 + d]));
                }
            }
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * nt; e += kFarThreads) {
        const int t = e / 3, d = e - 3 * t;
        double v = 0.0;
        for (int gg = 0; gg < ng; ++gg) v += sU[d][gg * rows + t];
        ufar[3 * size_t(item.z) + e] += v;
    }
}

// Per leaf at level >= 2: the evaluated expansions of Eq. (2.8), written to global memory for the
// bead-parallel evaluation: six fields per leaf (per velocity component), or by request the twelve of the
// per-potential form.
// rb: the local expansions carry q4 about their own box centres (box origin),
// so set 4 needs no re-basing to the leaf centre.
template <typename T>
__global__ void k_eval_prep(const int *leaves, DevTables<T> D, const double *ctr, const int *lvl, const int *bsys,
                            SysConst sc, const cpx<T> *L, cpx<T> *EVg, int per_component, int rb) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int li = blockIdx.x;
    int b = leaves[li];
    if (lvl[b] < 2) return;
    const int p = D.p, nc = ncoef(p);
    T *smr = reinterpret_cast<T *>(smem_raw);
    Lad<T> G = load_lad(D, smr);
    const T *inv = load_inv(smr + 6 * ncoef(p + 2), p);
    cpx<T> *srcs = reinterpret_cast<cpx<T> *>(smr + prep_tab_floats<T>(p));
    cpx<T> *tmp = srcs + kSets * nc;
    const cpx<T> *E = L + size_t(b) * kSets * nc;
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) srcs[i] = E[i];
    int sy = bsys[b];
    T c4, cc, o[3] = {T(0), T(0), T(0)};
    if constexpr (kIsDf<T>) {   // lengths in the split units: C2 / C1 = 2a^2/3 there
        const double ihs = inv_side_u(sc.pc[sy], lvl[b]);
        c4 = T(ihs);
        cc = T((double(sc.pc[sy].d_k23h) + double(sc.pc[sy].d_k23l)) * ihs * ihs);
        const float *c = sc.c3 + 9 * size_t(b);
        if (!rb)
            for (int a = 0; a < 3; ++a) o[a] = dfl3(c[3 * a], c[3 * a + 1], c[3 * a + 2]);
    } else {
        const double ih = sc.pc[sy].icube * pow2i(lvl[b]);   // 1 / side[b], exactly
        c4 = T(ih);
        cc = T(sc.pc[sy].C2 / sc.pc[sy].C1 * ih * ih);
        if (!rb)
            for (int a = 0; a < 3; ++a) o[a] = T(ctr[3 * b + a] - sc.cube[4 * sy + a]);
    }
    __syncthreads();
    if (per_component) {
        cpx<T> *EV = EVg + size_t(li) * kNF2 * nc, *phi = tmp, *V = phi + ncoef(p + 1);
        for (int i = threadIdx.x; i < ncoef(p + 1); i += blockDim.x)
            fold_scalars<T, false>(srcs, p, i, c4, cc, o, inv, G, phi, V);
        __syncthreads();
        for (int i = threadIdx.x; i < nc; i += blockDim.x) fold_fields<T, false>(srcs, p, i, inv, G, phi, V, EV);
        return;
    }
    cpx<T> *EV = EVg + size_t(li) * kNE * nc;
    build_eval_set<T>(srcs, p, p, EV, tmp, o[0], o[1], o[2], G);
    // Fold the terms of Eq. (2.8) that are not multiplied by a coordinate into
    // fields 0..2 (in units of C1/h):  L_d + h^-1 dL4'_d - (C2/C1) h^-2 dL_C,d.
    // The bead evaluation then needs fields 0..11 only.
    for (int i = threadIdx.x; i < 3 * nc; i += blockDim.x) {
        int d = i / nc, c = i - d * nc;
        cpx<T> v = EV[d * nc + c], g4 = EV[(12 + d) * nc + c], gc = EV[(15 + d) * nc + c];
        macc(v.x, -cc, gc.x);
        macc(v.x, c4, g4.x);
        macc(v.y, -cc, gc.y);
        macc(v.y, c4, g4.y);
        v = mk(closed(v.x), closed(v.y));
        EV[d * nc + c] = v;
    }
    __syncthreads();
    // the evaluated fields carry the factor 2 of the m > 0 terms of Re(sum E h)
    for (int i = threadIdx.x; i < kNF * nc; i += blockDim.x) {
        int c = i % nc, n = deg_of(c);
        if (c != tri(n, 0)) {
            cpx<T> v = EV[i];
            EV[i] = mk(scale2(2.f, v.x), scale2(2.f, v.y));
        }
    }
}

// One thread per bead: L2P of the leaf's derived expansions and Eq. (2.8),
// per potential (NF = 12: folded values and nine gradients) or per velocity
// component (NF = 6: u_d = H_d - |x|^2 B_d).
// Bound by latency on small systems, by the FP32 pipe on large ones.  With k_eval_prep, before the six fields stood
// interleaved and came from two scalar expansions, and now: 15M-bead cube FP64 5.74 -> 4.71 ms, FP32 2.82 -> 2.36 ms; 200k
// mixed at 9 digits 1.83 -> 0.98 ms; 4,096 beads FP64 51 -> 40 us.
template <typename T, int NF>
__global__ void __launch_bounds__(128, 6) k_eval_apply(int64_t n, const int *bead_leaf, const int *leaves,
                                                       DevTables<T> D, const double *ctr,
                                                       const int *lvl, const int *bsys, const double *pos, SysConst sc,
                                                       const cpx<T> *EVg, double *ufar) {
    int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int li = bead_leaf[i];
    int b = leaves[li];
    double u[3] = {0, 0, 0};
    if (lvl[b] >= 2) {
        const int p = D.p, nc = ncoef(p);
        int sy = bsys[b];
        const double C1 = sc.pc[sy].C1;
        T acc[NF];
#pragma unroll
        for (int q = 0; q < NF; ++q) acc[q] = T(0);
        if constexpr (kIsDf<T>) {
            const float *c = sc.c3 + 9 * size_t(b);
            const double ihd = inv_side_u(sc.pc[sy], lvl[b]);
            const T ihs = T(ihd);
            const T xi[3] = {coord_diff(sc.p3, n, i, 0, c) * ihs, coord_diff(sc.p3, n, i, 1, c) * ihs,
                             coord_diff(sc.p3, n, i, 2, c) * ihs};
            if constexpr (NF == kNF2)
                eval_six<T, false, true>(xi[0], xi[1], xi[2], p, EVg + size_t(li) * kNF2 * nc, D.rec_a, D.rec_b,
                                         D.rec_c, acc);
            else
                eval_fields<T, NF, false, true>(xi[0], xi[1], xi[2], p, EVg + size_t(li) * kNE * nc, nc, D.rec_a,
                                                D.rec_b, D.rec_c, acc);
            const double w1 = C1 * sc.pc[sy].d_xs * force_unit(sc.fmax[sy]) * ihd;
            const T r2 = fma(xi[2], xi[2], fma(xi[1], xi[1], xi[0] * xi[0]));
            for (int d = 0; d < 3; ++d) {
                T v = acc[d];
                if constexpr (NF == kNF2) v -= r2 * acc[3 + d];
                else
                    for (int k = 0; k < 3; ++k) v -= xi[k] * acc[3 + 3 * k + d];
                u[d] = w1 * double(v);
            }
        } else {
        const double ih = sc.pc[sy].icube * pow2i(lvl[b]);   // 1 / side[b], exactly
        double xi[3] = {(pos[i] - ctr[3 * b]) * ih, (pos[n + i] - ctr[3 * b + 1]) * ih,
                        (pos[2 * n + i] - ctr[3 * b + 2]) * ih};
        if constexpr (NF == kNF2) {
            eval_six<T, false, true>(T(xi[0]), T(xi[1]), T(xi[2]), p, EVg + size_t(li) * kNF2 * nc, D.rec_a, D.rec_b,
                                     D.rec_c, acc);
            // fields 0..2: H_d; 3..5: B_d
            const double r2 = xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2];
            for (int d = 0; d < 3; ++d) u[d] = C1 * ih * (double(acc[d]) - r2 * double(acc[3 + d]));
        } else {
            eval_fields<T, NF, false, true>(T(xi[0]), T(xi[1]), T(xi[2]), p, EVg + size_t(li) * kNE * nc, nc, D.rec_a,
                                            D.rec_b, D.rec_c, acc);
            // fields 0..2: the folded value terms; 3..11: gradients dL_k / dx_d at 3 + 3k + d
            for (int d = 0; d < 3; ++d) {
                double v = double(acc[d]);
                for (int k = 0; k < 3; ++k) v -= xi[k] * double(acc[3 + 3 * k + d]);
                u[d] = C1 * ih * v;
            }
        }
        }
    }
    for (int d = 0; d < 3; ++d) ufar[3 * i + d] = u[d];
}

// Laplace diagnostic: potential, gradient and Hessian of each set from L2P and M2P.
template <typename T, bool IRREG>
__device__ void build_lap_set(const cpx<T> *src, int p, int P, cpx<T> *EV, cpx<T> *tmp, const Lad<T> &G) {
    const int st = ncoef(P);
    for (int i = threadIdx.x; i < st; i += blockDim.x) EV[i] = i < ncoef(p) ? src[i] : mk<T>(0, 0);
    if (IRREG) d_multipole(src, p, EV + st, EV + 2 * st, EV + 3 * st, P, G);
    else d_local(src, p, EV + st, EV + 2 * st, EV + 3 * st, P, G);
    __syncthreads();
    int pd = IRREG ? p + 1 : p - 1;
    // Hessian rows: d/dx of (x, y, z) derivatives -> 4..6, d/dy -> 7..9, d/dz -> 10..12
    for (int a = 0; a < 3; ++a) {
        if (IRREG) d_multipole(EV + (1 + a) * st, pd, tmp, tmp + st, tmp + 2 * st, P, G);
        else d_local(EV + (1 + a) * st, pd, tmp, tmp + st, tmp + 2 * st, P, G);
        __syncthreads();
        for (int i = threadIdx.x; i < st; i += blockDim.x)
            for (int c = 0; c < 3; ++c) EV[(4 + 3 * a + c) * st + i] = tmp[c * st + i];
        __syncthreads();
    }
}

template <typename T>
__global__ void k_lap_eval(const int *leaves, DevTables<T> D, const int *beg, const int *end, const double *ctr,
                           const double *side, const int *lvl, const int *woff, const int *widx, const double *pos,
                           int64_t n, const cpx<T> *L, const cpx<T> *M, double *out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int li = blockIdx.x;
    int b = leaves[li];
    const int p = D.p, nc = ncoef(p), P = p + 2, st = ncoef(P);
    T *smr = reinterpret_cast<T *>(smem_raw);
    Rec<T> R = load_rec(D, smr);   // recurrence tables cover degree p + 2
    Lad<T> G = load_lad(D, smr + rec_floats<T>(p));
    cpx<T> *EV = reinterpret_cast<cpx<T> *>(smr + tab_floats<T>(p));
    cpx<T> *tmp = EV + 13 * st;
    cpx<T> *srcs = tmp + 3 * st;
    double cbx = ctr[3 * b], cby = ctr[3 * b + 1], cbz = ctr[3 * b + 2];
    int j0 = beg[b], j1 = end[b];
    int nw = woff[li + 1] - woff[li];
    bool has_local = lvl[b] >= 2;
    for (int jc = j0; jc < j1; jc += blockDim.x) {
        int j = jc + threadIdx.x;
        bool act = j < j1;
        double x = act ? pos[j] : cbx, y = act ? pos[n + j] : cby, z = act ? pos[2 * n + j] : cbz;
        double res[kSets][13];
        for (int k = 0; k < kSets; ++k)
            for (int c = 0; c < 13; ++c) res[k][c] = 0;
        for (int w = -1; w < nw; ++w) {
            if (w < 0 && !has_local) continue;
            int C = w < 0 ? b : widx[woff[li] + w];
            const cpx<T> *E = w < 0 ? L + size_t(C) * kSets * nc : M + size_t(C) * kSets * nc;
            double h = side[C], ih = 1.0 / h;
            T vx = T((x - ctr[3 * C]) * ih), vy = T((y - ctr[3 * C + 1]) * ih), vz = T((z - ctr[3 * C + 2]) * ih);
            for (int k = 0; k < kSets; ++k) {
                __syncthreads();
                for (int i = threadIdx.x; i < nc; i += blockDim.x) srcs[i] = E[k * nc + i];
                __syncthreads();
                if (w < 0) build_lap_set<T, false>(srcs, p, P, EV, tmp, G);
                else build_lap_set<T, true>(srcs, p, P, EV, tmp, G);
                T acc[13];
#pragma unroll
                for (int q = 0; q < 13; ++q) acc[q] = 0;
                if (w < 0) eval_fields<T, 13, false>(vx, vy, vz, p, EV, st, R.a, R.b, R.c, acc);
                else eval_fields<T, 13, true>(vx, vy, vz, P, EV, st, R.a, R.b, R.c, acc);
                res[k][0] += ih * double(acc[0]);
                for (int c = 1; c < 4; ++c) res[k][c] += ih * ih * double(acc[c]);
                for (int c = 4; c < 13; ++c) res[k][c] += ih * ih * ih * double(acc[c]);
            }
        }
        if (act)
            for (int k = 0; k < kSets; ++k)
                for (int c = 0; c < 13; ++c) out[(size_t(j) * kSets + k) * 13 + c] = res[k][c];
    }
}

// ---------------------------------------------------------------- driver

// (never while a stream is being captured: the first, uncaptured matvec sets every limit it needs)
static std::mutex g_smem_mu;
static std::map<std::pair<int, const void *>, size_t> g_smem_done;

int raise_smem(const void *kernel, size_t bytes) {
    if (bytes <= 40 * 1024) return RPY_OK;   // below the default limit, static shared memory included
    int dev = 0;
    RPY_CHECK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_smem_mu);
    size_t &d = g_smem_done[{dev, kernel}];
    if (bytes > d) {
        RPY_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)));
        d = bytes;
    }
    return RPY_OK;
}

template <typename T>
static size_t smem_p2x(int p, int threads) {
    return size_t(p2x_buf<T>(p, threads)) + sizeof(T) * (7 * kP2xStage + rec_floats<T>(p));
}
template <typename T>
static size_t smem_far(int p, int groups) {
    return sizeof(T) * far_tab_floats<T>(p) +
           sizeof(cpx<T>) * groups * (kSets * ncoef(p) + 2 * ncoef(p + 1) + 6 * ncoef(p + 2));
}
template <typename T>
static size_t smem_lap(int p) {
    int st = ncoef(p + 2);
    return sizeof(T) * tab_floats<T>(p) + sizeof(cpx<T>) * (13 * st + 3 * st + ncoef(p)) + 64;
}

// With one origin of q4 per system, Eq. (2.8) cancels terms of size |c - c0| |grad L|, which rounds like 2^level.
// Double-floats, a cluster of 20,001 beads in a cube 2^0 ... 2^16 times its size, 9 digits, distance of the far field from
// the same one in FP64: cube centre 2.0e-13 at depth 9, 6.3e-13 at 11, 5e-12 at 12, 6.4e-11 at 16, 1.5e-9 at 20 (its
// truncation is 6e-10 ... 1.2e-9); box centres 1.5e-13 ... 1.9e-13 at every depth.  With the rules of fewer digits, which
// truncate at 6e-8 of the far field and more, 1.5e-9 is lost in it, and X2X pays for the moves (k_x2x4; matvec of 200,001 beads,
// depth 15, cube against box centres: 3 digits 7.5 against 10.8 ms, 6 digits 9.4 against 10.1, 9 digits 20.1 against 21.5).
constexpr int kBoxOriginDepth = 10;

template <typename T>
int run_far_t(Tree &t, const DevTables<T> &D, const double *fs, const double *lapq, double *ufar, double *lapout,
              const SysConst &sc, cudaStream_t st) {
    const int p = D.p, nc = ncoef(p);
    cpx<T> *M = static_cast<cpx<T> *>(t.M), *L = static_cast<cpx<T> *>(t.L);
    int nbx = t.nbox;
    RPY_CHECK(cudaMemsetAsync(L, 0, sizeof(cpx<T>) * size_t(nbx) * kSets * nc, st));
    if (t.nlevels <= 2) {
        // no box at level >= 2: nothing is far
        if (ufar) RPY_CHECK(cudaMemsetAsync(ufar, 0, sizeof(double) * 3 * size_t(t.n), st));
        if (lapout) RPY_CHECK(cudaMemsetAsync(lapout, 0, sizeof(double) * 52 * size_t(t.n), st));
        return RPY_OK;
    }
    int b2 = t.level_off[2];
    int n2 = nbx - b2;
    // origin of q4 (RPY charges only; the Laplace diagnostic takes its charges as given): each expansion's own box
    // centre by default in the FP32 form at 6 digits and in the FP64 form with the 9-digit plane waves on trees of
    // depth kBoxOriginDepth and more, the cube centre otherwise
    const int fl = t.params.flags;
    const int rb = lapq ? 0
                        : (fl & RPY_FLAG_BOX_ORIGIN) ? 1
                        : (fl & RPY_FLAG_CUBE_ORIGIN) ? 0
                        : kIsDf<T> ? t.params.quad == 9 && t.nlevels - 1 >= kBoxOriginDepth
                                   : t.params.digits >= 6;
    // upward pass
    const int tp = p2x_threads(p, n2);
    const size_t sp = smem_p2x<T>(p, tp);
    RPY_TRY(set_smem(k_p2x<T, 0>, sp));
    RPY_TRY(set_smem(k_p2x<T, 1>, sp));
    k_p2x<T, 0><<<n2, tp, sp, st>>>(b2, n2, D, t.b_begin, t.b_end, t.b_center, t.b_level, t.b_leaf,
                                     t.b_sys, t.x_off, t.x_idx, t.pos, fs, lapq, t.n, sc, M, rb);
    RPY_LAUNCHED(1);
    RPY_CHECK(cudaGetLastError());
    prof_mark(t, RPY_STAGE_M2M, st);
    RPY_TRY(run_m2m_t(t, D, M, rb, st));
    // plane-wave M2L: all three frames in one pass, or (large trees, where the
    // plane-wave buffers of six directions would not fit) one frame per pass,
    // each pass adding its frame's share into L (with profiling on, every pass's
    // M2X, X2X and X2L launches are timed under their own stages).
    RPY_TRY(run_waves_t(t, D, M, L, rb, st));
    // X list
    prof_mark(t, RPY_STAGE_P2L, st);
    // without X lists (a uniform system, or all of its X boxes summed directly) there is nothing to launch: matvec of
    // 4,096 beads 225.2 -> 223.9 us, 12 Lanczos steps of 50,000 6.99 -> 6.95 ms
    if (t.n_x > 0) {
        k_p2x<T, 1><<<n2, tp, sp, st>>>(b2, n2, D, t.b_begin, t.b_end, t.b_center, t.b_level, t.b_leaf,
                                         t.b_sys, t.x_off, t.x_idx, t.pos, fs, lapq, t.n, sc, L, rb);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
    }
    // downward pass
    prof_mark(t, RPY_STAGE_L2L, st);
    RPY_TRY(run_l2l_t(t, D, L, rb, st));
    prof_mark(t, RPY_STAGE_EVAL, st);
    if (ufar) {
        cpx<T> *EVg = static_cast<cpx<T> *>(t.EVg);
        const size_t sp2 = sizeof(T) * prep_tab_floats<T>(p) + sizeof(cpx<T>) * (kSets * nc + kSets * ncoef(p + 1));
        RPY_TRY(set_smem(k_eval_prep<T>, sp2));
        // one expansion per velocity component unless the per-potential form is asked for
        const int per_comp = (t.params.flags & RPY_FLAG_EVAL_PER_POTENTIAL) ? 0 : 1;
        k_eval_prep<T><<<t.nleaf, 128, sp2, st>>>(t.leaves, D, t.b_center, t.b_level, t.b_sys, sc, L, EVg, per_comp,
                                                  rb);
        RPY_LAUNCHED(1);
        const int ga = int((t.n + 127) / 128);
        if (per_comp)
            k_eval_apply<T, kNF2><<<ga, 128, 0, st>>>(t.n, t.bead_leaf, t.leaves, D, t.b_center, t.b_level,
                                                      t.b_sys, t.pos, sc, EVg, ufar);
        else
            k_eval_apply<T, kNF><<<ga, 128, 0, st>>>(t.n, t.bead_leaf, t.leaves, D, t.b_center, t.b_level,
                                                     t.b_sys, t.pos, sc, EVg, ufar);
        RPY_LAUNCHED(1);
        if (t.n_w > 0) {
            // source boxes per round: as many groups as fit a block of an average leaf, in 64 KB
            int groups = std::min(kFarGroups, std::max(1, int(int64_t(kFarThreads) * t.nleaf / t.n)));
            while (groups > 1 && smem_far<T>(p, groups) > 64 * 1024) --groups;
            const size_t sf = smem_far<T>(p, groups);
            RPY_TRY(set_smem(k_far_eval<T>, sf));
            k_far_eval<T><<<t.n_items, kFarThreads, sf, st>>>(t.u_items, D, t.b_center, t.b_level, t.b_sys, t.w_off,
                                                              t.w_idx, t.pos, t.n, sc, M, ufar, rb, groups);
            RPY_LAUNCHED(1);
        }
        RPY_CHECK(cudaGetLastError());
    }
    if (lapout) {
        size_t sl = smem_lap<T>(p);
        RPY_TRY(set_smem(k_lap_eval<T>, sl));
        k_lap_eval<T><<<t.nleaf, 64, sl, st>>>(t.leaves, D, t.b_begin, t.b_end, t.b_center, t.b_side, t.b_level,
                                                t.w_off, t.w_idx, t.pos, t.n, L, M, lapout);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
    }
    return RPY_OK;
}

template int run_far_t<dfl>(Tree &, const DevTables<dfl> &, const double *, const double *, double *, double *,
                               const SysConst &, cudaStream_t);
template int run_far_t<float>(Tree &, const DevTables<float> &, const double *, const double *, double *, double *,
                              const SysConst &, cudaStream_t);

}  // namespace rpy
