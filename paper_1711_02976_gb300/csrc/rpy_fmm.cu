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
// inside the FP32 exponent range.  Measured, matvec of the 1M-bead sphere and cube at 6 digits (ms), FP64 -> dfl ->
// dfl with packed plane waves: 104 -> 45.5 -> 38.1 (M2X 23.4 -> 8.8 -> 5.4, X2L 20.1 -> 8.9 -> 7.4, X2X 11.9 -> 5.4 ->
// 3.7, L2P and M2P 16.6 -> 4.8, P2M and P2L 14.5 -> 4.0).  The velocities of whole matvecs move by
// 1e-14 ... 1.2e-13; the error of the expansions is 1e-10 at 9 digits.
//
// Kernels, in launch order:
//   k_p2m      S->M   leaves: M_n^m = sum_j q_j conj(y_n^m(eta_j))
//   k_m2m_child, k_m2m_sum  M->M   per child: rotate to the shift axis, z-shift, rotate back;
//                      per parent: add the children's shares in octant order
//   k_m2x      M->I   rotate into the frame of each axis, outgoing plane waves
//                     W_kj = (w_k/M_k) sum_{n,m} M_n^m i^|m| lambda_k^n e^{i m a_kj} / sqrt((n-|m|)!(n+|m|)!)
//   k_x2x      I->I   merge-and-shift: per parent and direction, sources are
//                     shifted to the parent centre and summed per group of
//                     targets they serve, then shifted once to each child
//   k_x2l      I->L   L_n^m = i^|m| sum_k (-lambda_k)^n / sqrt(...) sum_j I_kj e^{-i m a_kj},
//                     rotated back to the world frame
//   k_p2l      S->L   X list
//   k_l2l_rot  L->L   the same for locals, level by level downward
//   k_far_eval L->T, M->T   L2P for the leaf and M2P for its W list, with the
//                     gradients and Hessians of Theorems 1-2 formed as
//                     derivative expansions per box, combined by Eq. (2.8):
//                     u = C1 [L1 L2 L3] - C1 sum_k x_k grad L_k + C1 grad L4 - C2 grad L_C.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <map>
#include <mutex>

#include "rpy_harmonics.h"

namespace rpy {

__device__ __forceinline__ int deg_of(int idx) {
    int n = int((sqrtf(8.0f * idx + 1.0f) - 1.0f) * 0.5f);
    while (tri(n + 1, 0) <= idx) ++n;
    while (tri(n, 0) > idx) --n;
    return n;
}

// ---------------------------------------------------------------- harmonics, several points per warp
// Lanes per point: columns m and P - m share a lane, so every lane runs P + 2
// recurrence steps (a column per lane would leave the lanes of high m idle
// while column 0 runs P + 1 steps, and lanes above P idle altogether; the
// arithmetic pipes are charged per warp instruction).
__host__ __device__ constexpr int harm_lanes(int P) { return P / 2 + 1; }

// Solid harmonics (regular, or irregular when IRREG) of one point into out[],
// columns c and P - c of it.
template <typename T, bool IRREG>
__device__ void lane_harmonics(T x, T y, T z, int P, const T *ra, const T *rb, const T *cm, cpx<T> *out, int c) {
    const T r2 = fma(z, z, fma(y, y, x * x));
    const T ir2 = IRREG ? T(1) / r2 : T(0);
    const cpx<T> w = IRREG ? mk(x * ir2, y * ir2) : mk(x, y);
    const T d0 = IRREG ? sqrt(ir2) : T(1);
    const T zz = IRREG ? z * ir2 : z;   // factor of the a-coefficients
    const T rr = IRREG ? ir2 : r2;      // factor of the b-coefficients
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

// Beads per chunk of P2M / P2L: one round of harmonics, (warps x points per warp).
__host__ __device__ inline int p2x_chunk(int p, int threads) { return (threads / 32) * (32 / harm_lanes(p)); }

// MODE 0: P2M over the leaf's own beads (multipole about its centre)
// MODE 1: P2L over the beads of every box in X(b) (local about b's centre)
// The fourth charge q4 = F . (r - o) takes its origin o at the expansion's own
// centre when rb is set (box origin), else at the system's cube centre.
template <typename T, int MODE>
__global__ void k_p2x(int b0, int nb, DevTables<T> D, const int *beg, const int *end, const double *ctr,
                      const double *side, const int *lvl, const int *leaf, const int *bsys, const int *xoff,
                      const int *xidx, const double *pos, const double *fs, const double *lapq, int64_t n,
                      SysConst sc, cpx<T> *out, int rb) {
    const int kChunkB = p2x_chunk(D.p, blockDim.x);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = b0 + blockIdx.x;
    if (b >= b0 + nb) return;
    if (lvl[b] < 2) return;
    if (MODE == 0 && !leaf[b]) return;
    int nsrc = MODE == 0 ? 1 : xoff[b + 1] - xoff[b];
    if (nsrc == 0) return;
    const int p = D.p, nc = ncoef(p);
    T *smr = reinterpret_cast<T *>(smem_raw);
    Rec<T> R = load_rec(D, smr);
    cpx<T> *ybuf = reinterpret_cast<cpx<T> *>(smr + ((rec_floats<T>(p) + 1) & ~1));
    cpx<T> *acc = ybuf + kChunkB * nc;
    cpx<T> *cmp = acc + kSets * nc;   // FP32: compensation of the running sums
    T *q = reinterpret_cast<T *>(cmp + kSets * nc);
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) acc[i] = cmp[i] = mk<T>(0, 0);
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
    __syncthreads();
    for (int si = 0; si < nsrc; ++si) {
        int src = MODE == 0 ? b : xidx[xoff[b] + si];
        int j0 = beg[src], j1 = end[src];
        for (int jc = j0; jc < j1; jc += kChunkB) {
            int cnt = min(kChunkB, j1 - jc);
            for (int t0 = warp * hG; t0 < cnt; t0 += nwarp * hG) {
                const int t = t0 + hg;
                if (hg < hG && t < cnt) {
                    int j = jc + t;
                    T ex, ey, ez;
                    if constexpr (kIsDf<T>) {
                        ex = coord_diff(sc.p3, n, j, 0, c3) * ihs;
                        ey = coord_diff(sc.p3, n, j, 1, c3) * ihs;
                        ez = coord_diff(sc.p3, n, j, 2, c3) * ihs;
                    } else {
                        ex = T((pos[j] - cx) * ih), ey = T((pos[n + j] - cy) * ih), ez = T((pos[2 * n + j] - cz) * ih);
                    }
                    lane_harmonics<T, MODE == 1>(ex, ey, ez, p, R.a, R.b, R.cm, ybuf + t * nc, hc);
                }
            }
            for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
                int j = jc + t;
                if (lapq) {
                    for (int k = 0; k < kSets; ++k) q[4 * t + k] = T(kIsDf<T> ? qs * lapq[4 * j + k] : lapq[4 * j + k]);
                } else if constexpr (kIsDf<T>) {
                    // scaled forces; q4 in the split units of length, its origin at the cube's or the box's centre
                    float o3[9];
                    for (int k = 0; k < 9; ++k) o3[k] = rb ? c3[k] : 0.f;
                    T q4 = T(0);
                    for (int a = 0; a < 3; ++a) {
                        const T fa(sc.f2[(2 * a) * n + j], sc.f2[(2 * a + 1) * n + j]);
                        q[4 * t + a] = fa;
                        macc(q4, fa, coord_diff(sc.p3, n, j, a, o3));
                    }
                    q[4 * t + 3] = closed(q4);
                } else {
                    double fx = fs[j], fy = fs[n + j], fz = fs[2 * n + j];
                    q[4 * t] = T(fx);
                    q[4 * t + 1] = T(fy);
                    q[4 * t + 2] = T(fz);
                    q[4 * t + 3] = T(fx * (pos[j] - c0x) + fy * (pos[n + j] - c0y) + fz * (pos[2 * n + j] - c0z));
                }
            }
            __syncthreads();
            for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
                int k = e / nc, i = e - k * nc;
                cpx<T> a = sizeof(T) == 4 ? mk<T>(0, 0) : acc[e];
                for (int t = 0; t < cnt; ++t) {
                    cpx<T> yv = ybuf[t * nc + i];
                    T qq = q[4 * t + k];
                    macc(a.x, qq, yv.x);
                    macc(a.y, -qq, yv.y);   // conj
                }
                if constexpr (sizeof(T) == 4) {
                    // a leaf (or an X-list source) may hold hundreds to thousands of beads: the
                    // chunk's plain sum enters the running sum by compensated (Kahan) addition
                    cpx<T> sum = acc[e], c = cmp[e];
                    const T yx = a.x - c.x, tx = sum.x + yx;
                    c.x = (tx - sum.x) - yx;
                    sum.x = tx;
                    const T yy = a.y - c.y, ty = sum.y + yy;
                    c.y = (ty - sum.y) - yy;
                    sum.y = ty;
                    acc[e] = sum;
                    cmp[e] = c;
                } else {
                    acc[e] = mk(closed(a.x), closed(a.y));
                }
            }
            __syncthreads();
        }
    }
    cpx<T> *o = out + size_t(b) * kSets * nc;
    for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
        if (MODE == 0) o[e] = acc[e];
        else o[e] += acc[e];
    }
}

// ---------------------------------------------------------------- M2M / L2L

// Dense per-octant operators (used by the FP32 form, where one streaming pass
// over the operator beats the rotation's extra synchronisation).
// M2M: parent M = sum over children of T_o [child M]; output degree n uses inputs of degree <= n.
// rb (box origin of q4): the child's set 4 moves its origin from the child's
// centre to the parent's first, M4 += (c_child - c_parent) . M_F (sets 1..3).
template <typename T>
__global__ void k_m2m(int b0, int nb, DevTables<T> D, const int *leaf, const int *child, const double *side,
                      int rb, cpx<T> *M) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = b0 + blockIdx.x;
    if (leaf[b]) return;
    const int nc = ncoef(D.p), Dd = 2 * nc;
    T *X = reinterpret_cast<T *>(smem_raw);
    int r = threadIdx.x;
    int kmax = r < Dd ? 2 * ncoef(deg_of(r >> 1)) : 0;
    T acc[kSets] = {0, 0, 0, 0};
    for (int o = 0; o < 8; ++o) {
        int c = child[8 * b + o];
        if (c < 0) continue;
        const T *src = reinterpret_cast<const T *>(M + size_t(c) * kSets * nc);
        __syncthreads();
        for (int i = threadIdx.x; i < kSets * Dd; i += blockDim.x) X[i] = src[i];
        __syncthreads();
        if (rb) {
            const double h = 0.5 * side[c];   // child centre - parent centre = h (2 bit - 1) per axis
            const T dx = T((o & 1) ? h : -h), dy = T((o & 2) ? h : -h), dz = T((o & 4) ? h : -h);
            for (int i = threadIdx.x; i < Dd; i += blockDim.x)
                X[3 * Dd + i] = fma(dz, X[2 * Dd + i], fma(dy, X[Dd + i], fma(dx, X[i], X[3 * Dd + i])));
            __syncthreads();
        }
        if (r < Dd) {
            const T *Tt = D.m2m_t + size_t(o) * Dd * Dd;
            for (int k = 0; k < kmax; ++k) {
                T t = Tt[size_t(k) * Dd + r];
#pragma unroll
                for (int s = 0; s < kSets; ++s) acc[s] += t * X[s * Dd + k];
            }
        }
    }
    if (r < Dd) {
        T *dst = reinterpret_cast<T *>(M + size_t(b) * kSets * nc);
        for (int s = 0; s < kSets; ++s) dst[s * Dd + r] = acc[s];
    }
}

// L2L: child L += S_o [parent L]; output degree k uses inputs of degree >= k.
// rb (box origin of q4): the shifted set 4 moves its origin from the parent's
// centre to the child's, L4 += (c_parent - c_child) . L_F.
template <typename T>
__global__ void k_l2l(int b0, int nb, DevTables<T> D, const int *par, const int *cell, const double *side, int rb,
                      cpx<T> *L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = b0 + blockIdx.x;
    int P = par[b];
    const int nc = ncoef(D.p), Dd = 2 * nc;
    T *X = reinterpret_cast<T *>(smem_raw);
    const T *src = reinterpret_cast<const T *>(L + size_t(P) * kSets * nc);
    for (int i = threadIdx.x; i < kSets * Dd; i += blockDim.x) X[i] = src[i];
    __syncthreads();
    int r = threadIdx.x;
    if (r >= Dd) return;
    int o = (cell[3 * b] & 1) | ((cell[3 * b + 1] & 1) << 1) | ((cell[3 * b + 2] & 1) << 2);
    int kdeg = deg_of(r >> 1);
    int k0 = 2 * tri(kdeg, 0);
    const T *St = D.l2l_t + size_t(o) * Dd * Dd;
    T acc[kSets] = {0, 0, 0, 0};
    for (int k = k0; k < Dd; ++k) {
        T t = St[size_t(k) * Dd + r];
#pragma unroll
        for (int s = 0; s < kSets; ++s) acc[s] += t * X[s * Dd + k];
    }
    if (rb) {
        const double h = 0.5 * side[b];   // parent centre - child centre = -h (2 bit - 1) per axis
        const T dx = T((o & 1) ? -h : h), dy = T((o & 2) ? -h : h), dz = T((o & 4) ? -h : h);
        acc[3] = fma(dz, acc[2], fma(dy, acc[1], fma(dx, acc[0], acc[3])));
    }
    T *dst = reinterpret_cast<T *>(L + size_t(b) * kSets * nc);
    for (int s = 0; s < kSets; ++s) dst[s * Dd + r] += acc[s];
}

// ---------------------------------------------------------------- rotations
// dst[s] = R src[s] per degree block (real 2-layout, block size 2(n+1)).
// The factorized rotation of the four sets: tmp <- za (src) (one 2x2 rotation per
// coefficient), then dst <- zc (Y tmp), Y acting on real and imaginary parts
// separately.  src and dst may not alias tmp; the caller synchronises after.
// COL: the y blocks stand as [k][m] (y_by_column).
template <typename T, bool QUARTER, bool COL>
__device__ void rotate_sets_f(const T *rf, const int *foff, int p, const cpx<T> *src, cpx<T> *tmp, cpx<T> *dst) {
    const int nc = ncoef(p);
    for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
        const int st = e / nc, i = e - st * nc, n = deg_of(i), m = i - tri(n, 0);
        const T *za = rf + foff[n];
        const T c = za[2 * m], sn = za[2 * m + 1];
        const cpx<T> v = src[st * nc + i];
        tmp[e] = mk(mul_diff(c, v.x, sn, v.y), mul_diff(sn, v.x, -c, v.y));
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
        const int st = e / nc, i = e - st * nc, n = deg_of(i), m = i - tri(n, 0), q = n + 1;
        const T *o = rf + foff[n];
        const T *yre = o + 4 * q + (COL ? m : m * q), *yim = yre + q * q;
        const int sk = COL ? q : 1;   // stride of k
        const cpx<T> *in = tmp + st * nc + tri(n, 0);
        T re = 0, im = 0;
        if (QUARTER) {
            // middle angle pi/2 (the frame rotations): the y blocks are checkerboards
            // (checked when the tables are built); Im of m = 0 is zero for real fields
            for (int k = (m + n) & 1; k < q; k += 2) macc(re, yre[k * sk], in[k].x);
            if (m > 0)
                for (int k = 1 + ((m + n) & 1); k < q; k += 2) macc(im, yim[k * sk], in[k].y);
        } else {
            for (int k = 0; k < q; ++k) {
                macc(re, yre[k * sk], in[k].x);
                macc(im, yim[k * sk], in[k].y);
            }
        }
        re = closed(re);
        im = closed(im);
        const T c = o[2 * q + 2 * m], sn = o[2 * q + 2 * m + 1];
        dst[st * nc + i] = mk(mul_diff(c, re, sn, im), mul_diff(sn, re, -c, im));
    }
}

// ---------------------------------------------------------------- rotation-based M2M / L2L
// Child octant o: rotate into the frame whose z axis is the shift direction,
// apply the m-diagonal z-shift, rotate back (O(p^3) per child instead of the
// O(p^4) dense operator).
// One child per block (the children of one level): rotate into the frame
// whose z axis is the shift direction, apply the m-diagonal z-shift, rotate back
// (O(p^3) per child instead of the O(p^4) dense operator), and write the
// child's share to its slot Sc[parent][octant]; k_m2m_sum adds the slots of each
// parent in octant order (a fixed order: the result does not depend on timing).
// rb (box origin of q4): the share's set 4 moves its origin from the child's
// centre to the parent's, M4 += (c_child - c_parent) . M_F.
template <typename T>
__global__ void k_m2m_child(int c0, int pb0, DevTables<T> D, const int *par, const int *cell, const double *side,
                            int rb, const cpx<T> *M, cpx<T> *Sc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int c = c0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p);
    cpx<T> *X = reinterpret_cast<cpx<T> *>(smem_raw);
    cpx<T> *Y = X + kSets * nc;
    cpx<T> *Tm = Y + kSets * nc;   // rotation scratch
    const int o = (cell[3 * c] & 1) | ((cell[3 * c + 1] & 1) << 1) | ((cell[3 * c + 2] & 1) << 2);
    const cpx<T> *src = M + size_t(c) * kSets * nc;
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) X[i] = src[i];
    __syncthreads();
    rotate_sets_f<T, false, true>(D.forot_fwd + size_t(o) * D.frot_len, D.frot_off, p, X, Tm, Y);
    __syncthreads();
    for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
        int st = e / nc, i = e - st * nc;
        int n = deg_of(i), m = i - tri(n, 0);
        const T *z = D.zm2m + i;   // stored [k][coefficient]
        cpx<T> a = mk<T>(0, 0);
        for (int k = m; k <= n; ++k) {
            const cpx<T> y = Y[st * nc + tri(k, m)];
            macc(a.x, z[k * nc], y.x);
            macc(a.y, z[k * nc], y.y);
        }
        X[e] = mk(closed(a.x), closed(a.y));
    }
    __syncthreads();
    rotate_sets_f<T, false, true>(D.forot_bwd + size_t(o) * D.frot_len, D.frot_off, p, X, Tm, Y);
    __syncthreads();
    cpx<T> *dst = Sc + (size_t(par[c] - pb0) * 8 + o) * kSets * nc;
    const double h = 0.5 * side[c];
    const T dx = T((o & 1) ? h : -h), dy = T((o & 2) ? h : -h), dz = T((o & 4) ? h : -h);
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) {
        cpx<T> v = Y[i];
        if (rb && i >= 3 * nc) {
            const int k = i - 3 * nc;
            const cpx<T> fx = Y[k], fy = Y[nc + k], fz = Y[2 * nc + k];
            v = mk(fma(dz, fz.x, fma(dy, fy.x, fma(dx, fx.x, v.x))), fma(dz, fz.y, fma(dy, fy.y, fma(dx, fx.y, v.y))));
        }
        dst[i] = v;
    }
}

template <typename T>
__global__ void k_m2m_sum(int b0, int nc4, const int *leaf, const int *child, const cpx<T> *Sc, cpx<T> *M) {
    const int b = b0 + blockIdx.x;
    if (leaf[b]) return;
    int ch[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) ch[o] = child[8 * b + o];
    const cpx<T> *src = Sc + size_t(blockIdx.x) * 8 * nc4;
    for (int i = threadIdx.x; i < nc4; i += blockDim.x) {
        cpx<T> acc = mk<T>(0, 0);
#pragma unroll
        for (int o = 0; o < 8; ++o)
            if (ch[o] >= 0) acc += src[size_t(o) * nc4 + i];
        M[size_t(b) * nc4 + i] = acc;
    }
}

// rb (box origin of q4): the shifted set 4 moves its origin from the parent's
// centre to the child's, L4 += (c_parent - c_child) . L_F.
template <typename T>
__global__ void k_l2l_rot(int b0, int nb, DevTables<T> D, const int *par, const int *cell, const double *side,
                          int rb, cpx<T> *L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = b0 + blockIdx.x;
    int P = par[b];
    const int p = D.p, nc = ncoef(p);
    cpx<T> *X = reinterpret_cast<cpx<T> *>(smem_raw);
    cpx<T> *Y = X + kSets * nc;
    cpx<T> *Tm = Y + kSets * nc;   // rotation scratch
    int o = (cell[3 * b] & 1) | ((cell[3 * b + 1] & 1) << 1) | ((cell[3 * b + 2] & 1) << 2);
    const cpx<T> *src = L + size_t(P) * kSets * nc;
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) X[i] = src[i];
    __syncthreads();
    rotate_sets_f<T, false, true>(D.forot_fwd + size_t(o) * D.frot_len, D.frot_off, p, X, Tm, Y);
    __syncthreads();
    for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
        int st = e / nc, i = e - st * nc;
        int n = deg_of(i), m = i - tri(n, 0);
        const T *z = D.zl2l + i;   // stored [k][coefficient]
        cpx<T> a = mk<T>(0, 0);
        for (int k = n; k <= p; ++k) {
            const cpx<T> y = Y[st * nc + tri(k, m)];
            macc(a.x, z[k * nc], y.x);
            macc(a.y, z[k * nc], y.y);
        }
        X[e] = mk(closed(a.x), closed(a.y));
    }
    __syncthreads();
    rotate_sets_f<T, false, true>(D.forot_bwd + size_t(o) * D.frot_len, D.frot_off, p, X, Tm, Y);
    __syncthreads();
    cpx<T> *dst = L + size_t(b) * kSets * nc;
    const double h = 0.5 * side[b];
    const T dx = T((o & 1) ? -h : h), dy = T((o & 2) ? -h : h), dz = T((o & 4) ? -h : h);
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) {
        cpx<T> v = Y[i];
        if (rb && i >= 3 * nc) {
            const int k = i - 3 * nc;
            const cpx<T> fx = Y[k], fy = Y[nc + k], fz = Y[2 * nc + k];
            v = mk(fma(dz, fz.x, fma(dy, fy.x, fma(dx, fx.x, v.x))), fma(dz, fz.y, fma(dy, fy.y, fma(dx, fx.y, v.y))));
        }
        dst[i] += v;
    }
}

// ---------------------------------------------------------------- M2X
template <typename T, bool COL>
__global__ void k_m2x(int b0, int nb, DevTables<T> D, const cpx<T> *M, cpx<T> *Xo, int f0, int nf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = b0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p), s = D.s, S = D.S, P1 = p + 1;
    // A per node k: [P1][4 sets] at stride NS = 4 P1 + 1, so that the units of
    // neighbouring nodes in one warp read different shared-memory banks
    const int NS = kSets * P1 + 1;
    cpx<T> *Mw = reinterpret_cast<cpx<T> *>(smem_raw);
    cpx<T> *Mf = Mw + kSets * nc;
    cpx<T> *AE = Mf + kSets * nc;       // [s][NS]
    cpx<T> *AO = AE + s * NS;
    cpx<T> *Tm = AO + s * NS;           // rotation scratch
    const cpx<T> *src = M + size_t(b) * kSets * nc;
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) Mw[i] = src[i];
    __syncthreads();
    size_t base = size_t(b) * (2 * nf) * kSets * S;   // frames f0 .. f0 + nf - 1 of this pass
    const int hP = harm_lanes(p);
    for (int f = f0; f < f0 + nf; ++f) {
        const cpx<T> *Mu = Mw;
        if (f > 0) {
            rotate_sets_f<T, true, COL>(D.frot_fwd + size_t(f - 1) * D.frot_len, D.frot_off, p, Mw, Tm, Mf);
            __syncthreads();
            Mu = Mf;
        }
        // A_k^m split by parity of n + m (the - direction is the reflection (-1)^{n+m}),
        // stored as 2 i^m A_k^m so that the wave sum below needs no sign logic:
        // even m feed the real part, odd m the imaginary part.  One thread per
        // (set, node k, column pair (m, p - m)): p + 2 terms each.
        for (int e = threadIdx.x; e < kSets * s * hP; e += blockDim.x) {
            const int st = e / (s * hP), r = e - st * s * hP, k = r / hP, c = r - k * hP;
            const T *cc = D.m2x_c + size_t(k) * nc;
            const cpx<T> *Ms = Mu + st * nc;
            for (int h = 0; h < 2; ++h) {
                const int m = h ? p - c : c;
                if (h && m == c) break;
                T evx = 0, evy = 0, odx = 0, ody = 0;
                for (int n = m; n <= p; n += 2) {
                    const int i = tri(n, m);
                    macc(evx, cc[i], Ms[i].x);
                    macc(evy, cc[i], Ms[i].y);
                }
                for (int n = m + 1; n <= p; n += 2) {
                    const int i = tri(n, m);
                    macc(odx, cc[i], Ms[i].x);
                    macc(ody, cc[i], Ms[i].y);
                }
                const float sg = m == 0 ? 1.f : (((m >> 1) & 1) ? -2.f : 2.f);   // 2 i^m up to i for odd m
                AE[k * NS + m * kSets + st] = mk(scale2(sg, closed(evx)), scale2(sg, closed(evy)));
                AO[k * NS + m * kSets + st] = mk(scale2(sg, closed(odx)), scale2(sg, closed(ody)));
            }
        }
        __syncthreads();
        {
            // FP32: one wave per thread (the kernel is not bound by its FMAs, and
            // twice the threads hide more latency)
            // W_j = (w_k/M_k) [A^0 + 2 sum_m i^m Re(A^m e^{i m a_j})], A = AE +- AO, all four
            // sets per wave (one root lookup and index update serve four sets)
            for (int j = threadIdx.x; j < S; j += blockDim.x) {
                const int k = D.e_k[j];
                const int j0 = D.k_start[k], jl = j - j0, Mk = 2 * (D.k_start[k + 1] - j0);
                const cpx<T> *rt = D.roots + 2 * j0;
                const cpx<T> *ae = AE + k * NS;
                const cpx<T> *ao = AO + k * NS;
                T er[kSets], orr[kSets], ei[kSets], oi[kSets];
    #pragma unroll
                for (int st = 0; st < kSets; ++st) {
                    er[st] = ae[st].x;
                    orr[st] = ao[st].x;
                    ei[st] = 0;
                    oi[st] = 0;
                }
                int step2 = 2 * jl;
                if (step2 >= Mk) step2 -= Mk;
                int idx = 0;   // (m jl) mod Mk for even m
                for (int m = 2; m <= p; m += 2) {
                    idx += step2;
                    if (idx >= Mk) idx -= Mk;
                    const cpx<T> z = rt[idx];
    #pragma unroll
                    for (int st = 0; st < kSets; ++st) {
                        const cpx<T> a = ae[m * kSets + st], o = ao[m * kSets + st];
                        er[st] = fma(-a.y, z.y, fma(a.x, z.x, er[st]));
                        orr[st] = fma(-o.y, z.y, fma(o.x, z.x, orr[st]));
                    }
                }
                idx = jl;      // odd m, starting at m = 1
                for (int m = 1; m <= p; m += 2) {
                    const cpx<T> z = rt[idx];
    #pragma unroll
                    for (int st = 0; st < kSets; ++st) {
                        const cpx<T> a = ae[m * kSets + st], o = ao[m * kSets + st];
                        ei[st] = fma(-a.y, z.y, fma(a.x, z.x, ei[st]));
                        oi[st] = fma(-o.y, z.y, fma(o.x, z.x, oi[st]));
                    }
                    idx += step2;
                    if (idx >= Mk) idx -= Mk;
                }
                const T wm = D.e_wm[j];
    #pragma unroll
                for (int st = 0; st < kSets; ++st) {
                    Xo[base + size_t(2 * (f - f0)) * kSets * S + st * S + j] =
                        mk(wm * (er[st] + orr[st]), wm * (ei[st] + oi[st]));
                    Xo[base + size_t(2 * (f - f0) + 1) * kSets * S + st * S + j] =
                        mk(wm * (er[st] - orr[st]), wm * (ei[st] - oi[st]));
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- X2X merge-and-shift
template <typename T, bool FAC>
__global__ void k_x2x(const int *parents, DevTables<T> D, const int *coll, const int *child, const int *leaf,
                      const cpx<T> *Xo, cpx<T> *Xi, int f0, int nf) {
    __shared__ int src[216];
    __shared__ int vsrc[216], vsh[216], vpre[217];   // the present sources, compacted in slot order
    __shared__ int vend[216];   // child mask of its group at the last present source of a group, else 0
    // FAC (FP32, few plane waves): the shift of a source as the product of its
    // per-axis factors, from shared memory (z offsets x S, x offsets, y offsets);
    // otherwise the shift table
    __shared__ int voz[216], vox[216], voy[216];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int P = parents[blockIdx.x];
    const int dl = blockIdx.y, d = 2 * f0 + dl;   // direction, and its slot in this pass's buffers
    const int S = D.S;
    for (int sl = threadIdx.x; sl < 216; sl += blockDim.x) {
        int q = sl >> 3, o = sl & 7;
        int Q = coll[27 * P + q];
        src[sl] = (Q >= 0 && !leaf[Q]) ? child[8 * Q + o] : -1;
    }
    __syncthreads();
    int ng = D.grp_n[d];
    const int *goff = D.grp_off + d * (kGroupMax + 1);
    const int *gmask = D.grp_mask + d * kGroupMax;
    const int *slots = D.slot_list + d * 216;
    // warp 0: keep the slots whose source box exists; vpre[z] = present slots before z,
    // so group g covers vsrc[vpre[goff[g]] .. vpre[goff[g + 1]])
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, nsl = goff[ng];
        int carry = 0;
        for (int z0 = 0; z0 < nsl; z0 += 32) {
            const int z = z0 + lane;
            int ent = 0, sb = -1;
            if (z < nsl) {
                ent = slots[z];
                sb = src[ent & 255];
            }
            const unsigned bal = __ballot_sync(0xffffffffu, sb >= 0);
            const int pos = carry + __popc(bal & ((1u << lane) - 1u));
            if (z < nsl) vpre[z] = pos;
            if (sb >= 0) {
                vsrc[pos] = sb;
                vsh[pos] = ent >> 8;
            }
            carry += __popc(bal);
        }
        if (lane == 0) vpre[nsl] = carry;
    }
    __syncthreads();
    const int nz = vpre[goff[ng]];
    for (int z = threadIdx.x; z < nz; z += blockDim.x) {
        vend[z] = 0;
        const int o = vsh[z];
        vox[z] = (o % 6) * S;
        voy[z] = ((o / 6) % 6) * S;
        voz[z] = (o / 36) * S;
    }
    T *sZ = reinterpret_cast<T *>(smem_raw);
    cpx<T> *sX = reinterpret_cast<cpx<T> *>(sZ + ((6 * S + 3) & ~3));
    cpx<T> *sY = sX + 6 * S;
    if constexpr (FAC) {
        for (int i = threadIdx.x; i < 6 * S; i += blockDim.x) {
            sZ[i] = D.shz[i];
            sX[i] = D.shx[i];
            sY[i] = D.shy[i];
        }
    }
    __syncthreads();
    for (int g = threadIdx.x; g < ng; g += blockDim.x) {
        const int z1 = vpre[goff[g + 1]];
        if (z1 > vpre[goff[g]]) vend[z1 - 1] = gmask[g];
    }
    __syncthreads();
    int ch[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) ch[t] = child[8 * P + t];
    const size_t dstride = size_t(2 * nf) * kSets * S;
    const cpx<T> *Xd = Xo + size_t(dl) * kSets * S;
    for (int e = threadIdx.x; e < kSets * S; e += blockDim.x) {
        int j = e % S;
        cpx<T> acc[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[t] = mk<T>(0, 0);
        // one pass over all present sources (group boundaries marked by vend), so
        // that the unrolled loads run ahead across groups (measured: 8 in flight for the
        // FP32 table form, 4 elsewhere)
        constexpr int kUnroll = (sizeof(T) == 4 && !FAC) ? 8 : 4;
        cpx<T> ga = mk<T>(0, 0);
#pragma unroll kUnroll
        for (int z = 0; z < nz; ++z) {
            const cpx<T> x = Xd[size_t(vsrc[z]) * dstride + e];
            cpx<T> sh;
            if constexpr (FAC) {
                const cpx<T> a = sX[vox[z] + j], b = sY[voy[z] + j];
                const T c = sZ[voz[z] + j];
                sh = mk(c * mul_diff(a.x, b.x, a.y, b.y), c * mul_diff(a.x, b.y, -a.y, b.x));
            } else {
                sh = D.shift[size_t(vsh[z]) * S + j];
            }
            macc(ga.x, x.x, sh.x);
            macc(ga.x, -x.y, sh.y);
            macc(ga.y, x.x, sh.y);
            macc(ga.y, x.y, sh.x);
            const int mask = vend[z];   // block-uniform
            if (mask) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if ((mask >> t) & 1) acc[t] += ga;
                ga = mk<T>(0, 0);
            }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            if (ch[t] < 0) continue;
            cpx<T> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
            Xi[(size_t(ch[t]) * (2 * nf) + dl) * kSets * S + e] = acc[t] * sh;
        }
    }
}

// Merge-and-shift with the four charge sets of a plane wave in one thread (the
// FP32 form, and the box-origin form in either precision).  With rb (box origin
// of q4 = F . (r - o)), set 4 travels with its origin at the centre of the box
// whose expansion it is: each source's set 4 moves to the parent centre as it is
// merged, X4 += (c_source - c_parent) . X_F, and each merged sum moves to the
// child as it is shifted there, X4 += (c_parent - c_child) . X_F, with X_F the
// force sets 1..3 of the same wave (rotations of the frames act on the plane-wave
// variables only, so the world offsets apply as they are).
template <typename T, bool FAC>
__global__ void k_x2x4(const int *parents, DevTables<T> D, const int *coll, const int *child, const int *leaf,
                       const double *side, const cpx<T> *Xo, cpx<T> *Xi, int f0, int nf, int rb) {
    __shared__ int src[216];
    __shared__ int vsrc[216], vsh[216], vpre[217], vend[216];
    __shared__ int voz[216], vox[216], voy[216];
    __shared__ T vd[3][216];   // source centre - parent centre (world axes), set-4 origin move
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = parents[blockIdx.x];
    const int dl = blockIdx.y, d = 2 * f0 + dl;
    const int S = D.S;
    const double hc = 0.5 * side[P];   // side of P's children (and of the sources)
    for (int sl = threadIdx.x; sl < 216; sl += blockDim.x) {
        int q = sl >> 3, o = sl & 7;
        int Q = coll[27 * P + q];
        src[sl] = (Q >= 0 && !leaf[Q]) ? child[8 * Q + o] : -1;
    }
    __syncthreads();
    const int ng = D.grp_n[d];
    const int *goff = D.grp_off + d * (kGroupMax + 1);
    const int *gmask = D.grp_mask + d * kGroupMax;
    const int *slots = D.slot_list + d * 216;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, nsl = goff[ng];
        int carry = 0;
        for (int z0 = 0; z0 < nsl; z0 += 32) {
            const int z = z0 + lane;
            int ent = 0, sb = -1;
            if (z < nsl) {
                ent = slots[z];
                sb = src[ent & 255];
            }
            const unsigned bal = __ballot_sync(0xffffffffu, sb >= 0);
            const int pos = carry + __popc(bal & ((1u << lane) - 1u));
            if (z < nsl) vpre[z] = pos;
            if (sb >= 0) {
                vsrc[pos] = sb;
                vsh[pos] = ent >> 8;
                // slot = colleague (dx, dy, dz in -1..1, index 9 dz + 3 dy + dx + 13) x 8 + child octant:
                // source centre - P's centre = hc (2 d + bit - 1/2) per axis, in world axes
                const int sl = ent & 255, q = sl >> 3, o = sl & 7;
                vd[0][pos] = T(hc * (2 * (q % 3 - 1) + (o & 1) - 0.5));
                vd[1][pos] = T(hc * (2 * ((q / 3) % 3 - 1) + ((o >> 1) & 1) - 0.5));
                vd[2][pos] = T(hc * (2 * (q / 9 - 1) + ((o >> 2) & 1) - 0.5));
            }
            carry += __popc(bal);
        }
        if (lane == 0) vpre[nsl] = carry;
    }
    __syncthreads();
    const int nz = vpre[goff[ng]];
    for (int z = threadIdx.x; z < nz; z += blockDim.x) {
        vend[z] = 0;
        const int o = vsh[z];
        vox[z] = (o % 6) * S;
        voy[z] = ((o / 6) % 6) * S;
        voz[z] = (o / 36) * S;
    }
    T *sZ = reinterpret_cast<T *>(smem_raw);
    cpx<T> *sX = reinterpret_cast<cpx<T> *>(sZ + ((6 * S + 3) & ~3));
    cpx<T> *sY = sX + 6 * S;
    if constexpr (FAC) {
        for (int i = threadIdx.x; i < 6 * S; i += blockDim.x) {
            sZ[i] = D.shz[i];
            sX[i] = D.shx[i];
            sY[i] = D.shy[i];
        }
    }
    __syncthreads();
    for (int g = threadIdx.x; g < ng; g += blockDim.x) {
        const int z1 = vpre[goff[g + 1]];
        if (z1 > vpre[goff[g]]) vend[z1 - 1] = gmask[g];
    }
    __syncthreads();
    int ch[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) ch[t] = child[8 * P + t];
    const size_t dstride = size_t(2 * nf) * kSets * S;
    const cpx<T> *Xd = Xo + size_t(dl) * kSets * S;
    for (int j = threadIdx.x; j < S; j += blockDim.x) {
        cpx<T> acc[8][kSets];
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int k = 0; k < kSets; ++k) acc[t][k] = mk<T>(0, 0);
        cpx<T> ga[kSets];
#pragma unroll
        for (int k = 0; k < kSets; ++k) ga[k] = mk<T>(0, 0);
#pragma unroll 2
        for (int z = 0; z < nz; ++z) {
            const cpx<T> *xs = Xd + size_t(vsrc[z]) * dstride + j;
            cpx<T> x[kSets];
#pragma unroll
            for (int k = 0; k < kSets; ++k) x[k] = xs[size_t(k) * S];
            if (rb) {
                const T ex = vd[0][z], ey = vd[1][z], ez = vd[2][z];
                x[3].x = fma(ez, x[2].x, fma(ey, x[1].x, fma(ex, x[0].x, x[3].x)));
                x[3].y = fma(ez, x[2].y, fma(ey, x[1].y, fma(ex, x[0].y, x[3].y)));
            }
            cpx<T> sh;
            if constexpr (FAC) {
                const cpx<T> a = sX[vox[z] + j], b = sY[voy[z] + j];
                const T c = sZ[voz[z] + j];
                sh = mk(c * mul_diff(a.x, b.x, a.y, b.y), c * mul_diff(a.x, b.y, -a.y, b.x));
            } else {
                sh = D.shift[size_t(vsh[z]) * S + j];
            }
#pragma unroll
            for (int k = 0; k < kSets; ++k) {
                macc(ga[k].x, x[k].x, sh.x);
                macc(ga[k].x, -x[k].y, sh.y);
                macc(ga[k].y, x[k].x, sh.y);
                macc(ga[k].y, x[k].y, sh.x);
            }
            const int mask = vend[z];   // block-uniform
            if (mask) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if ((mask >> t) & 1)
#pragma unroll
                        for (int k = 0; k < kSets; ++k) acc[t][k] += ga[k];
#pragma unroll
                for (int k = 0; k < kSets; ++k) ga[k] = mk<T>(0, 0);
            }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            if (ch[t] < 0) continue;
            if (rb) {   // P's centre - child t's centre = -(hc / 2) (2 bit - 1) per axis
                const double h = 0.5 * hc;
                const T ex = T((t & 1) ? -h : h), ey = T((t & 2) ? -h : h), ez = T((t & 4) ? -h : h);
                acc[t][3].x = fma(ez, acc[t][2].x, fma(ey, acc[t][1].x, fma(ex, acc[t][0].x, acc[t][3].x)));
                acc[t][3].y = fma(ez, acc[t][2].y, fma(ey, acc[t][1].y, fma(ex, acc[t][0].y, acc[t][3].y)));
            }
            const cpx<T> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
            cpx<T> *dst = Xi + (size_t(ch[t]) * (2 * nf) + dl) * kSets * S + j;
#pragma unroll
            for (int k = 0; k < kSets; ++k) dst[size_t(k) * S] = acc[t][k] * sh;
        }
    }
}

// ---------------------------------------------------------------- bulk copies and mbarriers
// One-dimensional bulk copies global -> shared (the TMA engine) completing on an
// mbarrier: a thread announces the bytes to arrive (expect_tx), issues the copies,
// and every thread waits for the barrier's phase.  Waits give up after about a
// second (a copy that never lands), so that no kernel can hang the device.
__device__ __forceinline__ unsigned smem_addr(const void *p) { return unsigned(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, uint64_t limit_ns = 1000000000ull) {
    if (mbar_test(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (!mbar_test(bar, parity))
        if (global_ns() - t0 > limit_ns) return false;
    return true;
}

// Self-test of the bounded wait: one thread waits for an mbarrier phase that no
// arrival will ever complete (no copy is issued), gives up after limit_ns and
// reports the timeout through the status word, as the pipelined kernels do.
__global__ void k_wait_selftest(uint64_t limit_ns, unsigned *status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    mbar_init_fence();
    if (!mbar_wait(&bar, 0, limit_ns)) atomicOr(status, DEVERR_TIMEOUT);
}

int wait_selftest(double limit_ms, cudaStream_t st) {
    unsigned *d = nullptr;
    RPY_CHECK(cudaMalloc(&d, sizeof(unsigned)));
    unsigned h = 0;
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(unsigned), st);
    if (e == cudaSuccess) {
        k_wait_selftest<<<1, 32, 0, st>>>(uint64_t(limit_ms * 1e6), d);
        RPY_LAUNCHED(1);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    if (e != cudaSuccess) return check_cuda("wait self-test", e);
    return (h & DEVERR_TIMEOUT) ? RPY_ERR_TIMEOUT : RPY_OK;
}
// orders this thread's earlier generic-proxy accesses to shared memory before later bulk copies
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Bulk-copy pipeline of the FP32 X2X: kX2XStages buffers, each holding one source's
// outgoing waves in one direction (4 S values) and its shift row (S values, rows
// padded to an even length).
constexpr int kX2XStages = 4;
__host__ __device__ inline int x2x_tma_stage_elems(int S) { return 4 * S + ((S + 1) & ~1); }
__host__ inline size_t x2x_tma_smem(int S) { return sizeof(cpx<float>) * size_t(kX2XStages) * x2x_tma_stage_elems(S); }

// FP32 merge-and-shift, one consumer thread per plane wave (the four charge sets
// and the box-origin move of set 4 as in k_x2x4), fed by a producer warp: the
// present sources are staged through shared memory by bulk copies (TMA) into
// kX2XStages buffers.  Buffer q is "full" when its copies have landed (an mbarrier
// with the transaction count) and "empty" when every consumer warp has read it
// (an mbarrier with one arrival per consumer warp); the producer refills a buffer
// as soon as it is empty, so the consumers never wait on a global load and the
// block needs no barrier per source.
__global__ void __launch_bounds__(512, 1) k_x2x_tma(const int *parents, DevTables<float> D, const int *coll,
                                                    const int *child, const int *leaf, const double *side,
                                                    const cpx<float> *Xo, cpx<float> *Xi, int f0, int nf, int rb,
                                                    unsigned *status) {
    __shared__ int src[216];
    __shared__ int vsrc[216], vsh[216], vpre[217], vend[216];
    __shared__ float vd[3][216];
    __shared__ __align__(8) uint64_t full[kX2XStages], empty[kX2XStages];
    __shared__ int bad, issued;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = parents[blockIdx.x];
    const int dl = blockIdx.y, d = 2 * f0 + dl;
    const int S = D.S, Sp = D.Sp;
    const int ncw = (S + 31) / 32;                 // consumer warps; the last warp produces
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double hc = 0.5 * side[P];
    for (int sl = threadIdx.x; sl < 216; sl += blockDim.x) {
        int q = sl >> 3, o = sl & 7;
        int Q = coll[27 * P + q];
        src[sl] = (Q >= 0 && !leaf[Q]) ? child[8 * Q + o] : -1;
    }
    if (threadIdx.x == 0) {
        bad = 0;
        issued = 0;
        for (int q = 0; q < kX2XStages; ++q) {
            mbar_init(&full[q], 1);
            mbar_init(&empty[q], unsigned(ncw));
        }
        mbar_init_fence();
    }
    __syncthreads();
    const int ng = D.grp_n[d];
    const int *goff = D.grp_off + d * (kGroupMax + 1);
    const int *gmask = D.grp_mask + d * kGroupMax;
    const int *slots = D.slot_list + d * 216;
    if (warp == 0) {
        const int nsl = goff[ng];
        int carry = 0;
        for (int z0 = 0; z0 < nsl; z0 += 32) {
            const int z = z0 + lane;
            int ent = 0, sb = -1;
            if (z < nsl) {
                ent = slots[z];
                sb = src[ent & 255];
            }
            const unsigned bal = __ballot_sync(0xffffffffu, sb >= 0);
            const int pos = carry + __popc(bal & ((1u << lane) - 1u));
            if (z < nsl) vpre[z] = pos;
            if (sb >= 0) {
                vsrc[pos] = sb;
                vsh[pos] = ent >> 8;
                const int sl = ent & 255, q = sl >> 3, o = sl & 7;
                vd[0][pos] = float(hc * (2 * (q % 3 - 1) + (o & 1) - 0.5));
                vd[1][pos] = float(hc * (2 * ((q / 3) % 3 - 1) + ((o >> 1) & 1) - 0.5));
                vd[2][pos] = float(hc * (2 * (q / 9 - 1) + ((o >> 2) & 1) - 0.5));
            }
            carry += __popc(bal);
        }
        if (lane == 0) vpre[nsl] = carry;
    }
    __syncthreads();
    const int nz = vpre[goff[ng]];
    for (int z = threadIdx.x; z < nz; z += blockDim.x) vend[z] = 0;
    __syncthreads();
    for (int g = threadIdx.x; g < ng; g += blockDim.x) {
        const int z1 = vpre[goff[g + 1]];
        if (z1 > vpre[goff[g]]) vend[z1 - 1] = gmask[g];
    }
    __syncthreads();
    const int stage_elems = x2x_tma_stage_elems(S);
    cpx<float> *stage0 = reinterpret_cast<cpx<float> *>(smem_raw);
    if (warp == ncw) {
        // producer: one lane issues the copies, refilling each buffer once it is empty
        if (lane == 0) {
            const size_t dstride = size_t(2 * nf) * kSets * S;
            const cpx<float> *Xd = Xo + size_t(dl) * kSets * S;
            const unsigned src_bytes = 32u * unsigned(S), sh_bytes = 8u * unsigned(Sp);
            for (int z = 0; z < nz; ++z) {
                const int q = z % kX2XStages;
                if (z >= kX2XStages && !mbar_wait(&empty[q], unsigned(z / kX2XStages - 1) & 1u)) {
                    bad = 1;
                    break;
                }
                if (*(volatile int *)&bad) break;
                cpx<float> *buf = stage0 + size_t(q) * stage_elems;
                mbar_expect(&full[q], src_bytes + sh_bytes);
                bulk_load(buf, Xd + size_t(vsrc[z]) * dstride, src_bytes, &full[q]);
                bulk_load(buf + 4 * S, D.shiftp + size_t(vsh[z]) * Sp, sh_bytes, &full[q]);
                issued = z + 1;
            }
        }
    } else {
        int ch[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) ch[t] = child[8 * P + t];
        const int j = threadIdx.x;
        const bool act = j < S;
        cpx<float> acc[8][kSets];
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int k = 0; k < kSets; ++k) acc[t][k] = mk(0.f, 0.f);
        cpx<float> ga[kSets];
#pragma unroll
        for (int k = 0; k < kSets; ++k) ga[k] = mk(0.f, 0.f);
        for (int z = 0; z < nz; ++z) {
            const int q = z % kX2XStages;
            if (!mbar_wait(&full[q], unsigned(z / kX2XStages) & 1u) || *(volatile int *)&bad) {
                bad = 1;
                break;
            }
            if (act) {
                const cpx<float> *buf = stage0 + size_t(q) * stage_elems;
                cpx<float> x[kSets];
#pragma unroll
                for (int k = 0; k < kSets; ++k) x[k] = buf[k * S + j];
                if (rb) {
                    const float ex = vd[0][z], ey = vd[1][z], ez = vd[2][z];
                    x[3].x = fmaf(ez, x[2].x, fmaf(ey, x[1].x, fmaf(ex, x[0].x, x[3].x)));
                    x[3].y = fmaf(ez, x[2].y, fmaf(ey, x[1].y, fmaf(ex, x[0].y, x[3].y)));
                }
                const cpx<float> sh = buf[4 * S + j];
#pragma unroll
                for (int k = 0; k < kSets; ++k) {
                    ga[k].x = fmaf(-x[k].y, sh.y, fmaf(x[k].x, sh.x, ga[k].x));
                    ga[k].y = fmaf(x[k].y, sh.x, fmaf(x[k].x, sh.y, ga[k].y));
                }
                const int mask = vend[z];   // block-uniform
                if (mask) {
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if ((mask >> t) & 1)
#pragma unroll
                            for (int k = 0; k < kSets; ++k) acc[t][k] += ga[k];
#pragma unroll
                    for (int k = 0; k < kSets; ++k) ga[k] = mk(0.f, 0.f);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[q]);   // this warp is done with buffer q
        }
        if (!*(volatile int *)&bad && act) {
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                if (ch[t] < 0) continue;
                if (rb) {   // P's centre - child t's centre = -(hc / 2) (2 bit - 1) per axis
                    const float h = float(0.5 * hc);
                    const float ex = (t & 1) ? -h : h, ey = (t & 2) ? -h : h, ez = (t & 4) ? -h : h;
                    acc[t][3].x = fmaf(ez, acc[t][2].x, fmaf(ey, acc[t][1].x, fmaf(ex, acc[t][0].x, acc[t][3].x)));
                    acc[t][3].y = fmaf(ez, acc[t][2].y, fmaf(ey, acc[t][1].y, fmaf(ex, acc[t][0].y, acc[t][3].y)));
                }
                const cpx<float> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
                cpx<float> *dst = Xi + (size_t(ch[t]) * (2 * nf) + dl) * kSets * S + j;
#pragma unroll
                for (int k = 0; k < kSets; ++k) dst[size_t(k) * S] = acc[t][k] * sh;
            }
        }
    }
    __syncthreads();
    if (bad && threadIdx.x == 0) {
        // a wait gave up: let every copy issued land (bounded) before the block's shared
        // memory is released, and flag the failure
        for (int q = 0; q < min(issued, kX2XStages); ++q) {
            const int zl = q + ((issued - 1 - q) / kX2XStages) * kX2XStages;   // last copy issued into buffer q
            mbar_wait(&full[q], unsigned(zl / kX2XStages) & 1u);
        }
        atomicOr(status, DEVERR_TIMEOUT);
    }
}

// ---------------------------------------------------------------- X2L
// FP32 form of X2L: the four charge sets in one pass.  The incoming waves of a
// frame are staged planar (real parts of the four sets in one float4, imaginary
// parts in another), so that the real DFT, which takes the real parts for even m
// and the imaginary parts for odd m, reads four sets with one 16-byte load per
// wave and direction; one root lookup then serves sixteen FMAs.
template <bool COL>
__global__ void k_x2l4(int b0, int nb, DevTables<float> D, const cpx<float> *Xi, cpx<float> *L, int f0, int nf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p), s = D.s, S = D.S, P1 = p + 1;
    float4 *PRe = reinterpret_cast<float4 *>(smem_raw);   // [S] + direction, real parts of sets 0..3
    float4 *PIm = PRe + S;
    float4 *MRe = PIm + S;                                  // - direction
    float4 *MIm = MRe + S;
    // b+ + b- (Bs) and b+ - b- (Bd) per (node, m), as planes of set pairs: (re, im) of sets
    // 0 and 1, then of sets 2 and 3, so that each thread's 16-byte stores are contiguous
    // across lanes (one [s][P1][4] array took four 8-byte stores 32 bytes apart)
    const int SP = s * P1;
    float4 *Bs01 = MIm + S, *Bs23 = Bs01 + SP, *Bd01 = Bs23 + SP, *Bd23 = Bd01 + SP;
    cpx<float> *Lf = reinterpret_cast<cpx<float> *>(Bd23 + SP);                  // [4][nc]
    cpx<float> *Lw = Lf + kSets * nc;
    cpx<float> *Lr = Lw + kSets * nc;
    cpx<float> *Tm = Lr + kSets * nc;                             // rotation scratch
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) Lw[i] = mk<float>(0, 0);
    for (int f = f0; f < f0 + nf; ++f) {
        __syncthreads();
        const cpx<float> *sp = Xi + (size_t(b) * (2 * nf) + 2 * (f - f0)) * kSets * S;
        const cpx<float> *sm = Xi + (size_t(b) * (2 * nf) + 2 * (f - f0) + 1) * kSets * S;
        for (int j = threadIdx.x; j < S; j += blockDim.x) {
            const cpx<float> p0 = sp[j], p1 = sp[S + j], p2 = sp[2 * S + j], p3 = sp[3 * S + j];
            const cpx<float> m0 = sm[j], m1 = sm[S + j], m2 = sm[2 * S + j], m3 = sm[3 * S + j];
            PRe[j] = make_float4(p0.x, p1.x, p2.x, p3.x);
            PIm[j] = make_float4(p0.y, p1.y, p2.y, p3.y);
            MRe[j] = make_float4(m0.x, m1.x, m2.x, m3.x);
            MIm[j] = make_float4(m0.y, m1.y, m2.y, m3.y);
        }
        __syncthreads();
        // b_k^m = 2 sum_j Re(I_j) e^{-i m a_j} (m even), 2i sum_j Im(I_j) e^{-i m a_j} (m odd)
        // (node, m) items at a stride of PA = 8 per node when p + 1 <= 8, so that a
        // quarter-warp never straddles two nodes (its wave loads are then broadcasts)
        const int PA = P1 <= 8 ? 8 : P1;
        for (int ea = threadIdx.x; ea < s * PA; ea += blockDim.x) {
            const int k = ea / PA, m = ea - k * PA;
            if (m >= P1) continue;
            const int e = k * P1 + m;
            const int j0 = D.k_start[k], j1 = D.k_start[k + 1];
            const int Mk = 2 * (j1 - j0), mm = m % Mk;
            const cpx<float> *rt = D.roots + 2 * j0;
            const float4 *vp = (m & 1) ? PIm : PRe;
            const float4 *vm = (m & 1) ? MIm : MRe;
            float bpx[kSets] = {0, 0, 0, 0}, bpy[kSets] = {0, 0, 0, 0};
            float bmx[kSets] = {0, 0, 0, 0}, bmy[kSets] = {0, 0, 0, 0};
            int idx = 0;
            for (int j = j0; j < j1; ++j) {
                const cpx<float> r = rt[idx];
                const float4 a = vp[j], c = vm[j];
                const float av[kSets] = {a.x, a.y, a.z, a.w}, cv[kSets] = {c.x, c.y, c.z, c.w};
#pragma unroll
                for (int st = 0; st < kSets; ++st) {
                    bpx[st] = fmaf(av[st], r.x, bpx[st]);
                    bpy[st] = fmaf(-av[st], r.y, bpy[st]);
                    bmx[st] = fmaf(cv[st], r.x, bmx[st]);
                    bmy[st] = fmaf(-cv[st], r.y, bmy[st]);
                }
                idx += mm;
                if (idx >= Mk) idx -= Mk;
            }
            Bs01[e] = make_float4(bpx[0] + bmx[0], bpy[0] + bmy[0], bpx[1] + bmx[1], bpy[1] + bmy[1]);
            Bs23[e] = make_float4(bpx[2] + bmx[2], bpy[2] + bmy[2], bpx[3] + bmx[3], bpy[3] + bmy[3]);
            Bd01[e] = make_float4(bpx[0] - bmx[0], bpy[0] - bmy[0], bpx[1] - bmx[1], bpy[1] - bmy[1]);
            Bd23[e] = make_float4(bpx[2] - bmx[2], bpy[2] - bmy[2], bpx[3] - bmx[3], bpy[3] - bmy[3]);
        }
        __syncthreads();
        // L_n^m = i^m sum_k (-lambda_k)^n / sqrt((n-m)!(n+m)!) b_k^m, the - direction reflected
        for (int i = threadIdx.x; i < nc; i += blockDim.x) {
            const int n = deg_of(i), m = i - tri(n, 0);
            const bool odd = (n + m) & 1;
            const float4 *B01 = odd ? Bd01 : Bs01, *B23 = odd ? Bd23 : Bs23;
            // sum over the quadrature nodes with compensated (Kahan) addition: the terms
            // (-lambda_k)^n b_k^m alternate in sign and cancel strongly at high degree
            float ax[kSets] = {0, 0, 0, 0}, ay[kSets] = {0, 0, 0, 0};
            float cx[kSets] = {0, 0, 0, 0}, cy[kSets] = {0, 0, 0, 0};
            auto kahan = [](float &sum, float &c, float v) {
                const float y = v - c, t = sum + y;
                c = (t - sum) - y;
                sum = t;
            };
            for (int k = 0; k < s; ++k) {
                const float c = D.x2l_c[size_t(k) * nc + i];
                const float4 b01 = B01[k * P1 + m], b23 = B23[k * P1 + m];
                kahan(ax[0], cx[0], c * b01.x);
                kahan(ay[0], cy[0], c * b01.y);
                kahan(ax[1], cx[1], c * b01.z);
                kahan(ay[1], cy[1], c * b01.w);
                kahan(ax[2], cx[2], c * b23.x);
                kahan(ay[2], cy[2], c * b23.y);
                kahan(ax[3], cx[3], c * b23.z);
                kahan(ay[3], cy[3], c * b23.w);
            }
#pragma unroll
            for (int st = 0; st < kSets; ++st) Lf[st * nc + i] = mul_ipow(mk(2 * ax[st], 2 * ay[st]), m + (m & 1));
        }
        __syncthreads();
        if (f == 0) {
            for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) Lw[i] += Lf[i];
        } else {
            rotate_sets_f<float, false, COL>(D.frot_bwd + size_t(f - 1) * D.frot_len, D.frot_off, p, Lf, Tm, Lr);
            __syncthreads();
            for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) Lw[i] += Lr[i];
        }
    }
    __syncthreads();
    cpx<float> *dst = L + size_t(b) * kSets * nc;
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) dst[i] += Lw[i];
}

static size_t smem_x2l4(int p, int s, int S) {
    const int nc = ncoef(p);
    return sizeof(float4) * 4 * size_t(S) + sizeof(cpx<float>) * (2 * kSets * s * (p + 1) + 4 * kSets * nc);
}

// ---------------------------------------------------------------- double-float plane waves, sets packed
// M2X, X2X and X2L of the FP64 form.  Every table value serves the four charge sets alike, so a thread
// carries two sets in the lanes of packed operations: half the FMA instructions of scalar double-floats,
// and one table load, index update and loop step for two sets (all four in one thread: 106 to 118
// registers and 12 to 14 warps per SM, M2X 6.2 and X2L 8.3 ms where this form takes 5.4 and 7.2, 1M-bead sphere
// at 6 digits).
// A quantity of a pair of sets stands as one float4 (h, h', l, l').
// Plane waves: Xo and Xi [box][direction][wave][4] float4: re {0,1}, re {2,3}, im {0,1}, im {2,3}.
// Neighbouring lanes carry the two pairs of one item: they share its table loads.
__device__ __forceinline__ df2 zero_df2() { return df2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ df2 operator+(df2 a, df2 b) { return renorm(sum_raw(a, b)); }
__device__ __forceinline__ df2 operator-(df2 a, df2 b) { return renorm(sum_raw(a, -b)); }
__device__ __forceinline__ df2 closed(df2 a) { return renorm(a); }
__device__ __forceinline__ void macc(df2 &acc, dfl s, df2 b) { macc(acc, dup(s), b); }
// a x + b y with scalar a, b
__device__ __forceinline__ df2 lin2(dfl a, df2 x, dfl b, df2 y) {
    return renorm(sum_raw(mul_df(dup(a), x), mul_df(dup(b), y)));
}

// n complex coefficients of four sets in shared memory: real parts [n][pair], then imaginary parts,
// 16 bytes each, so that consecutive threads touch consecutive banks.  pr: the pair of sets.
struct Planes {
    float4 *p;
    int n;
    __device__ __forceinline__ df2 x(int pr, int i) const { return as_df2(p[2 * i + pr]); }
    __device__ __forceinline__ df2 y(int pr, int i) const { return as_df2(p[2 * (n + i) + pr]); }
    __device__ __forceinline__ void set(int pr, int i, df2 a, df2 b) const {
        p[2 * i + pr] = as_float4(a);
        p[2 * (n + i) + pr] = as_float4(b);
    }
};
// coefficient i of the pair's sets in global memory ([set][nc] cpx<dfl>)
__device__ __forceinline__ void load_pair(const cpx<dfl> *g, int nc, int pr, int i, df2 &x, df2 &y) {
    const cpx<dfl> u = g[2 * pr * nc + i], v = g[(2 * pr + 1) * nc + i];
    x = df2{make_float2(u.x.h, v.x.h), make_float2(u.x.l, v.x.l)};
    y = df2{make_float2(u.y.h, v.y.h), make_float2(u.y.l, v.y.l)};
}

// The factored rotation of the four sets (rotate_sets_f): rotate_z forms tmp from a source of (x, y) per item,
// rotate_y the result in dst.  An item is (coefficient, pair of sets).
template <typename F>
__device__ __forceinline__ void rotate_z(const dfl *rf, const int *foff, int nc, Planes tmp, F source) {
    for (int e = threadIdx.x; e < 2 * nc; e += blockDim.x) {
        const int pr = e & 1, i = e >> 1, n = deg_of(i), m = i - tri(n, 0);
        const dfl *za = rf + foff[n];
        const dfl c = za[2 * m], sn = za[2 * m + 1];
        df2 x, y;
        source(pr, i, x, y);
        tmp.set(pr, i, lin2(c, x, -sn, y), lin2(sn, x, c, y));
    }
}
__device__ __forceinline__ void rotate_y(const dfl *rf, const int *foff, int nc, Planes tmp, Planes dst) {
    for (int e = threadIdx.x; e < 2 * nc; e += blockDim.x) {
        const int pr = e & 1, i = e >> 1, n = deg_of(i), m = i - tri(n, 0), q = n + 1, t0 = tri(n, 0);
        const dfl *o = rf + foff[n], *yre = o + 4 * q + m, *yim = yre + q * q;
        df2 re = zero_df2(), im = re;
        // the frame rotations' middle angle is pi/2: checkerboard y blocks, Im of m = 0 zero
        for (int k = (m + n) & 1; k < q; k += 2) macc(re, yre[k * q], tmp.x(pr, t0 + k));
        if (m > 0)
            for (int k = 1 + ((m + n) & 1); k < q; k += 2) macc(im, yim[k * q], tmp.y(pr, t0 + k));
        re = closed(re);
        im = closed(im);
        const dfl c = o[2 * q + 2 * m], sn = o[2 * q + 2 * m + 1];
        dst.set(pr, i, lin2(c, re, -sn, im), lin2(sn, re, c, im));
    }
}

// A_k^m rows of one node at an odd stride, so that neighbouring nodes fall on different banks
__host__ __device__ inline int a_stride(int p) { return (p + 1) | 1; }

// M2X: one box per block, kc quadrature nodes at a time.
__global__ void __launch_bounds__(256, 3)
    k_m2x_df(int b0, DevTables<dfl> D, const cpx<dfl> *M, float4 *Xo, int f0, int nf, int kc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p), s = D.s, S = D.S, NS = a_stride(p);
    const Planes Mu{reinterpret_cast<float4 *>(smem_raw), nc};
    const Planes AE{Mu.p + 4 * nc, kc * NS}, AO{AE.p + 4 * kc * NS, kc * NS};
    const Planes Tm{AE.p, nc};   // rotation scratch, before the A rows are formed (node_chunk leaves room)
    const cpx<dfl> *src = M + size_t(b) * kSets * nc;
    const int hP = harm_lanes(p);
    for (int f = f0; f < f0 + nf; ++f) {
        if (f > 0) {
            const dfl *rf = D.frot_fwd + size_t(f - 1) * D.frot_len;
            rotate_z(rf, D.frot_off, nc, Tm, [&](int pr, int i, df2 &x, df2 &y) { load_pair(src, nc, pr, i, x, y); });
            __syncthreads();
            rotate_y(rf, D.frot_off, nc, Tm, Mu);
        } else {
            for (int e = threadIdx.x; e < 2 * nc; e += blockDim.x) {
                df2 x, y;
                load_pair(src, nc, e & 1, e >> 1, x, y);
                Mu.set(e & 1, e >> 1, x, y);
            }
        }
        __syncthreads();
        float4 *out = Xo + (size_t(b) * (2 * nf) + 2 * (f - f0)) * 4 * S;   // + direction; - direction 4 S further
        for (int k0 = 0; k0 < s; k0 += kc) {
            const int kn = min(kc, s - k0);
            // A_k^m split by parity of n + m (the - direction is the reflection (-1)^{n+m}), stored as
            // 2 i^m A_k^m so that the wave sum needs no sign logic: even m feed the real part, odd m the
            // imaginary part.  One thread per (pair of sets, node, column pair (m, p - m)): p + 2 terms.
            for (int e = threadIdx.x; e < 2 * kn * hP; e += blockDim.x) {
                const int pr = e & 1, r = e >> 1, kk = r / hP, c = r - kk * hP;
                const dfl *cc = D.m2x_c + size_t(k0 + kk) * nc;
                for (int h = 0; h < 2; ++h) {
                    const int m = h ? p - c : c;
                    if (h && m == c) break;
                    df2 evx = zero_df2(), evy = evx, odx = evx, ody = evx;
                    int n = m, i = tri(m, m);
                    for (; n < p; n += 2) {   // degrees n and n + 1
                        const int i1 = i + n + 1;
                        const dfl c0 = cc[i], c1 = cc[i1];
                        macc(evx, c0, Mu.x(pr, i));
                        macc(evy, c0, Mu.y(pr, i));
                        macc(odx, c1, Mu.x(pr, i1));
                        macc(ody, c1, Mu.y(pr, i1));
                        i = i1 + n + 2;
                    }
                    if (n == p) {
                        const dfl c0 = cc[i];
                        macc(evx, c0, Mu.x(pr, i));
                        macc(evy, c0, Mu.y(pr, i));
                    }
                    const float sg = m == 0 ? 1.f : (((m >> 1) & 1) ? -2.f : 2.f);   // 2 i^m up to i for odd m
                    AE.set(pr, kk * NS + m, scale2(sg, closed(evx)), scale2(sg, closed(evy)));
                    AO.set(pr, kk * NS + m, scale2(sg, closed(odx)), scale2(sg, closed(ody)));
                }
            }
            __syncthreads();
            // W_j = (w_k/M_k) [A^0 + 2 sum_m i^m Re(A^m e^{i m a_j})], A = AE +- AO.  Waves t and
            // M_k/2 - t of a node have angles a and pi - a: e^{i m (pi - a)} = (-1)^m conj(e^{i m a}), so with
            // P = sum a.x z.x and Q = sum a.y z.y over even (or odd) m, Re(A z) = P - Q serves wave t and
            // (-1)^m Re(A conj z) = +-(P + Q) its partner: two multiply-adds per (m, set) for both waves.
            const int ub = D.u_start[k0], un = D.u_start[k0 + kn] - ub;
            for (int e = threadIdx.x; e < 2 * un; e += blockDim.x) {
                const int pr = e & 1, u = ub + (e >> 1);
                const int k = D.u_k[u], row = (k - k0) * NS;
                const int j0 = D.k_start[k], H = D.k_start[k + 1] - j0, t = u - D.u_start[k], Mk = 2 * H;
                const bool pair = t > 0 && 2 * t != H;
                const cpx<dfl> *rt = D.roots + 2 * j0;
                const dfl wm = D.e_wm[j0 + t];
                int step2 = 2 * t;
                if (step2 >= Mk) step2 -= Mk;
#pragma unroll 1
                for (int odd = 0; odd < 2; ++odd) {
                    df2 pe = zero_df2(), qe = pe, po = pe, qo = pe;
                    int idx = t, m = 1;
                    if (!odd) {
                        pe = AE.x(pr, row);
                        po = AO.x(pr, row);
                        idx = step2;
                        m = 2;
                    }
                    for (; m <= p; m += 2) {
                        const cpx<dfl> z = rt[idx];
                        const int i = row + m;
                        macc(pe, z.x, AE.x(pr, i));
                        macc(qe, z.y, AE.y(pr, i));
                        macc(po, z.x, AO.x(pr, i));
                        macc(qo, z.y, AO.y(pr, i));
                        idx += step2;
                        if (idx >= Mk) idx -= Mk;
                    }
                    // real (even m) or imaginary (odd m) parts: + direction A = AE + AO, - direction AE - AO
                    auto put = [&](int j, df2 a, df2 o) {
                        float4 *d = out + 4 * j + 2 * odd + pr;
                        const df2 W = dup(wm);
                        d[0] = as_float4(renorm(mul_df(W, a + o)));
                        d[4 * S] = as_float4(renorm(mul_df(W, a - o)));
                    };
                    put(j0 + t, pe - qe, po - qo);
                    if (pair) {   // the partner, with sign (-1)^m
                        const df2 eb = pe + qe, ob = po + qo;
                        put(j0 + H - t, odd ? -eb : eb, odd ? -ob : ob);
                    }
                }
            }
            __syncthreads();
        }
    }
}

// X2X merge-and-shift (k_x2x), one thread per (wave, pair of sets).  Plain loads, two sources in flight: staging
// each thread's sources through shared memory by asynchronous copies four steps ahead was slower
// (1M-bead sphere 4.17 -> 4.46 ms, 15M-bead cube 25.7 -> 29.4 ms: it adds shared-memory instructions and
// takes a third of the L1).
// Blocks of 128 threads at 96 registers (five per SM) on large grids; of 256 threads (two per SM) where the
// grid leaves the SMs room and a block's own length counts (1M-bead sphere 4.24 -> 3.71 ms and 15M-bead cube
// 26.1 -> 23.0 ms from 256 to 128; 20k-bead sphere 0.133 -> 0.191 ms, 4,096 beads 0.058 -> 0.094 ms).
constexpr int kX2XSmallGrid = 3000;   // blocks
template <int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS)
    k_x2x_df(const int *parents, DevTables<dfl> D, const int *coll, const int *child, const int *leaf,
             const float4 *Xo, float4 *Xi, int f0, int nf) {
    __shared__ int src[216];
    __shared__ int vsrc[216], vsh[216], vpre[217];   // the present sources, compacted in slot order
    __shared__ int vend[216];   // child mask of its group at the last present source of a group, else 0
    const int P = parents[blockIdx.x];
    const int dl = blockIdx.y, d = 2 * f0 + dl;   // direction, and its slot in this pass's buffers
    const int S = D.S;
    for (int sl = threadIdx.x; sl < 216; sl += blockDim.x) {
        const int q = sl >> 3, o = sl & 7;
        const int Q = coll[27 * P + q];
        src[sl] = (Q >= 0 && !leaf[Q]) ? child[8 * Q + o] : -1;
    }
    __syncthreads();
    const int ng = D.grp_n[d];
    const int *goff = D.grp_off + d * (kGroupMax + 1);
    const int *gmask = D.grp_mask + d * kGroupMax;
    const int *slots = D.slot_list + d * 216;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, nsl = goff[ng];
        int carry = 0;
        for (int z0 = 0; z0 < nsl; z0 += 32) {
            const int z = z0 + lane;
            int ent = 0, sb = -1;
            if (z < nsl) {
                ent = slots[z];
                sb = src[ent & 255];
            }
            const unsigned bal = __ballot_sync(0xffffffffu, sb >= 0);
            const int pos = carry + __popc(bal & ((1u << lane) - 1u));
            if (z < nsl) vpre[z] = pos;
            if (sb >= 0) {
                vsrc[pos] = sb;
                vsh[pos] = (ent >> 8) * S;
            }
            carry += __popc(bal);
        }
        if (lane == 0) vpre[nsl] = carry;
    }
    __syncthreads();
    const int nz = vpre[goff[ng]];
    for (int z = threadIdx.x; z < nz; z += blockDim.x) vend[z] = 0;
    __syncthreads();
    for (int g = threadIdx.x; g < ng; g += blockDim.x) {
        const int z1 = vpre[goff[g + 1]];
        if (z1 > vpre[goff[g]]) vend[z1 - 1] = gmask[g];
    }
    __syncthreads();
    const size_t dstride = size_t(2 * nf) * 4 * S;
    const float4 *Xd = Xo + size_t(dl) * 4 * S;
    for (int e = threadIdx.x; e < 2 * S; e += blockDim.x) {
        const int j = e >> 1, pr = e & 1;
        df2 ax[8], ay[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) ax[t] = ay[t] = zero_df2();
        df2 gx = zero_df2(), gy = gx;
#pragma unroll 2
        for (int z = 0; z < nz; ++z) {
            const float4 *xs = Xd + size_t(vsrc[z]) * dstride + 4 * j + pr;
            const df2 x = as_df2(xs[0]), y = as_df2(xs[2]);
            const cpx<dfl> sh = D.shift[vsh[z] + j];
            const df2 sx = dup(sh.x), sy = dup(sh.y);
            macc(gx, sx, x);
            macc(gx, -sy, y);
            macc(gy, sy, x);
            macc(gy, sx, y);
            const int mask = vend[z];   // block-uniform
            if (mask) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if ((mask >> t) & 1) {
                        ax[t] = sum_raw(ax[t], gx);
                        ay[t] = sum_raw(ay[t], gy);
                    }
                gx = gy = zero_df2();
            }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int ch = child[8 * P + t];
            if (ch < 0) continue;
            const cpx<dfl> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
            const df2 x = renorm(ax[t]), y = renorm(ay[t]);
            float4 *dst = Xi + (size_t(ch) * (2 * nf) + dl) * 4 * S + 4 * j + pr;
            dst[0] = as_float4(lin2(sh.x, x, -sh.y, y));
            dst[2] = as_float4(lin2(sh.y, x, sh.x, y));
        }
    }
}

// X2L: one box per block, kc quadrature nodes at a time (umax wave-pair units at most).
__global__ void __launch_bounds__(256, 3)
    k_x2l_df(int b0, DevTables<dfl> D, const float4 *Xi, cpx<dfl> *L, int f0, int nf, int kc, int umax) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p), s = D.s, S = D.S, P1 = p + 1, NS = a_stride(p);
    const Planes Lf{reinterpret_cast<float4 *>(smem_raw), nc};   // the frame's sums
    // b+ + b- and b+ - b- per (node, m)
    const Planes Bs{Lf.p + 4 * nc, kc * NS}, Bd{Bs.p + 4 * kc * NS, kc * NS};
    // per unit (waves t and M_k/2 - t of a node): sums and differences of the pair's real and imaginary
    // parts, UQ[direction][re +, re -, im +, im -][unit][pair of sets]
    float4 *UQ = Bd.p + 4 * kc * NS;
    const Planes Tm{Bs.p, nc};   // rotation scratch over the B rows and the units (node_chunk leaves room)
    cpx<dfl> *dst = L + size_t(b) * kSets * nc;
    for (int f = f0; f < f0 + nf; ++f) {
        const float4 *in = Xi + (size_t(b) * (2 * nf) + 2 * (f - f0)) * 4 * S;
        for (int k0 = 0; k0 < s; k0 += kc) {
            const int kn = min(kc, s - k0);
            const int ub = D.u_start[k0], un = D.u_start[k0 + kn] - ub;
            __syncthreads();
            for (int e = threadIdx.x; e < 4 * un; e += blockDim.x) {   // (unit, direction, pair of sets)
                const int u = e >> 2, dir = (e >> 1) & 1, pr = e & 1;
                const int k = D.u_k[ub + u], j0 = D.k_start[k], H = D.k_start[k + 1] - j0, t = ub + u - D.u_start[k];
                const bool pair = t > 0 && 2 * t != H;
                const float4 *w = in + dir * 4 * S + pr;
                const df2 ax = as_df2(w[4 * (j0 + t)]), ay = as_df2(w[4 * (j0 + t) + 2]);
                df2 bx = zero_df2(), by = bx;
                if (pair) {
                    bx = as_df2(w[4 * (j0 + H - t)]);
                    by = as_df2(w[4 * (j0 + H - t) + 2]);
                }
                float4 *q = UQ + 8 * dir * umax + 2 * u + pr;
                q[0] = as_float4(ax + bx);
                q[2 * umax] = as_float4(ax - bx);
                q[4 * umax] = as_float4(ay + by);
                q[6 * umax] = as_float4(ay - by);
            }
            __syncthreads();
            // b_k^m = sum_{j < M_k/2} (I_j + (-1)^m conj I_j) e^{-i m a_j}
            //       = 2 sum_j Re(I_j) e^{-i m a_j}      (m even)
            //       = 2i sum_j Im(I_j) e^{-i m a_j}     (m odd; the factor i is applied below)
            // With e^{-i m (pi - a)} = (-1)^m conj(e^{-i m a}), a wave pair adds
            // (v + (-1)^m v') cos(m a) - i (v - (-1)^m v') sin(m a): even m take the
            // sum and difference of the real parts, odd m those of the imaginary parts.
            // A thread takes node kk and its mirror kn - 1 - kk: the nodes' wave counts grow with k, so
            // the sums over two mirrored nodes are about equally long.
            const int items = ((kn + 1) >> 1) * P1;
            for (int e = threadIdx.x; e < 2 * items; e += blockDim.x) {
                const int pr = e & 1, r = e >> 1, ka = r / P1, m = r - ka * P1;
                for (int h = 0; h < 2; ++h) {
                    const int kk = h ? kn - 1 - ka : ka, k = k0 + kk;
                    if (h && kk == ka) break;
                    const int j0 = D.k_start[k], Mk = 2 * (D.k_start[k + 1] - j0);
                    const int u0 = D.u_start[k] - ub, u1 = D.u_start[k + 1] - ub;
                    const int mm = m % Mk;
                    const cpx<dfl> *rt = D.roots + 2 * j0;
                    const float4 *xp = UQ + ((m & 1) ? 6 : 0) * umax + pr, *yp = UQ + ((m & 1) ? 4 : 2) * umax + pr;
                    df2 bpx = zero_df2(), bpy = bpx, bmx = bpx, bmy = bpx;
                    int idx = 0;
                    for (int u = u0; u < u1; ++u) {
                        const cpx<dfl> z = rt[idx];
                        macc(bpx, z.x, as_df2(xp[2 * u]));
                        macc(bpy, -z.y, as_df2(yp[2 * u]));
                        macc(bmx, z.x, as_df2(xp[8 * umax + 2 * u]));
                        macc(bmy, -z.y, as_df2(yp[8 * umax + 2 * u]));
                        idx += mm;
                        if (idx >= Mk) idx -= Mk;
                    }
                    // the + direction and the reflected - direction enter L through
                    // b+ + b- (n + m even) and b+ - b- (n + m odd)
                    Bs.set(pr, kk * NS + m, bpx + bmx, bpy + bmy);
                    Bd.set(pr, kk * NS + m, bpx - bmx, bpy - bmy);
                }
            }
            __syncthreads();
            // L_n^m = i^m sum_k (-lambda_k)^n / sqrt((n-m)!(n+m)!) b_k^m, the - direction reflected
            for (int e = threadIdx.x; e < 2 * nc; e += blockDim.x) {
                const int pr = e & 1, i = e >> 1, n = deg_of(i), m = i - tri(n, 0);
                const Planes B = ((n + m) & 1) ? Bd : Bs;
                df2 x = zero_df2(), y = x;
                if (k0) {
                    x = Lf.x(pr, i);
                    y = Lf.y(pr, i);
                }
                const dfl *c = D.x2l_c + size_t(k0) * nc + i;
                for (int kk = 0; kk < kn; ++kk, c += nc) {
                    macc(x, *c, B.x(pr, kk * NS + m));
                    macc(y, *c, B.y(pr, kk * NS + m));
                }
                x = closed(x);
                y = closed(y);
                if (k0 + kc >= s) {   // the last nodes: times 2 i^(m + (m & 1))
                    const float sg = ((m + (m & 1)) & 2) ? -2.f : 2.f;
                    x = scale2(sg, x);
                    y = scale2(sg, y);
                }
                Lf.set(pr, i, x, y);
            }
        }
        __syncthreads();
        if (f > 0) {   // back to world axes; Lf is free once rotated about z
            const dfl *rf = D.frot_bwd + size_t(f - 1) * D.frot_len;
            rotate_z(rf, D.frot_off, nc, Tm, [&](int pr, int i, df2 &x, df2 &y) {
                x = Lf.x(pr, i);
                y = Lf.y(pr, i);
            });
            __syncthreads();
            rotate_y(rf, D.frot_off, nc, Tm, Lf);
            __syncthreads();
        }
        for (int e = threadIdx.x; e < 2 * nc; e += blockDim.x) {
            const int pr = e & 1, i = e >> 1;
            const df2 x = Lf.x(pr, i), y = Lf.y(pr, i);
            cpx<dfl> *d0 = dst + 2 * pr * nc + i, *d1 = d0 + nc;
            cpx<dfl> u = *d0, v = *d1;
            u += mk(dfl(x.h.x, x.l.x), dfl(y.h.x, y.l.x));
            v += mk(dfl(x.h.y, x.l.y), dfl(y.h.y, y.l.y));
            *d0 = u;
            *d1 = v;
        }
    }
}

// Four sets in one thread, for the box-origin form below.
struct df4 {
    df2 v[2];
};
__device__ __forceinline__ df4 zero_df4() { return df4{{zero_df2(), zero_df2()}}; }
__device__ __forceinline__ void macc(df4 &acc, dfl s, const df4 &b) {
    macc(acc.v[0], s, b.v[0]);
    macc(acc.v[1], s, b.v[1]);
}
__device__ __forceinline__ df4 operator+(const df4 &a, const df4 &b) { return df4{{a.v[0] + b.v[0], a.v[1] + b.v[1]}}; }
__device__ __forceinline__ df4 lin2(dfl a, const df4 &x, dfl b, const df4 &y) {
    return df4{{lin2(a, x.v[0], b, y.v[0]), lin2(a, x.v[1], b, y.v[1])}};
}

// X2X with the box origin of q4 (k_x2x4), one thread per wave, all four sets.
__global__ void __launch_bounds__(256, 1) k_x2x4_df(const int *parents, DevTables<dfl> D, const int *coll, const int *child, const int *leaf,
                          const double *side, const float4 *Xo, float4 *Xi, int f0, int nf) {
    __shared__ int src[216];
    const int P = parents[blockIdx.x];
    const int dl = blockIdx.y, d = 2 * f0 + dl;
    const int S = D.S;
    const double hc = 0.5 * side[P];   // side of P's children (and of the sources)
    for (int sl = threadIdx.x; sl < 216; sl += blockDim.x) {
        const int q = sl >> 3, o = sl & 7;
        const int Q = coll[27 * P + q];
        src[sl] = (Q >= 0 && !leaf[Q]) ? child[8 * Q + o] : -1;
    }
    __syncthreads();
    const int ng = D.grp_n[d];
    const int *goff = D.grp_off + d * (kGroupMax + 1);
    const int *gmask = D.grp_mask + d * kGroupMax;
    const int *slots = D.slot_list + d * 216;
    const size_t dstride = size_t(2 * nf) * 4 * S;
    const float4 *Xd = Xo + size_t(dl) * 4 * S;
    // set 3 += (dx, dy, dz) . sets 0..2 of one part (re or im)
    auto move = [](df4 &v, dfl dx, dfl dy, dfl dz) {
        dfl a(v.v[1].h.y, v.v[1].l.y);
        macc(a, dx, dfl(v.v[0].h.x, v.v[0].l.x));
        macc(a, dy, dfl(v.v[0].h.y, v.v[0].l.y));
        macc(a, dz, dfl(v.v[1].h.x, v.v[1].l.x));
        a = closed(a);
        v.v[1].h.y = a.h;
        v.v[1].l.y = a.l;
    };
    for (int j = threadIdx.x; j < S; j += blockDim.x) {
        df4 ax[8], ay[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) ax[t] = ay[t] = zero_df4();
        for (int g = 0; g < ng; ++g) {
            df4 gx = zero_df4(), gy = gx;
            bool any = false;
            for (int z = goff[g]; z < goff[g + 1]; ++z) {
                const int ent = slots[z], sl = ent & 255, sb = src[sl];
                if (sb < 0) continue;
                any = true;
                const float4 *xs = Xd + size_t(sb) * dstride + 4 * j;
                df4 x{{as_df2(xs[0]), as_df2(xs[1])}}, y{{as_df2(xs[2]), as_df2(xs[3])}};
                // slot = colleague (dx, dy, dz in -1..1, index 9 dz + 3 dy + dx + 13) x 8 + child octant:
                // source centre - P's centre = hc (2 d + bit - 1/2) per axis, in world axes
                const int q = sl >> 3, o = sl & 7;
                const dfl ex(hc * (2 * (q % 3 - 1) + (o & 1) - 0.5)), ey(hc * (2 * ((q / 3) % 3 - 1) + ((o >> 1) & 1) - 0.5)),
                    ez(hc * (2 * (q / 9 - 1) + ((o >> 2) & 1) - 0.5));
                move(x, ex, ey, ez);
                move(y, ex, ey, ez);
                const cpx<dfl> sh = D.shift[size_t(ent >> 8) * S + j];
                macc(gx, sh.x, x);
                macc(gx, -sh.y, y);
                macc(gy, sh.y, x);
                macc(gy, sh.x, y);
            }
            if (!any) continue;
            const int mask = gmask[g];
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if ((mask >> t) & 1) {
                    ax[t] = ax[t] + gx;
                    ay[t] = ay[t] + gy;
                }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int ch = child[8 * P + t];
            if (ch < 0) continue;
            // P's centre - child t's centre = -(hc / 2) (2 bit - 1) per axis
            const double h = 0.5 * hc;
            const dfl ex((t & 1) ? -h : h), ey((t & 2) ? -h : h), ez((t & 4) ? -h : h);
            move(ax[t], ex, ey, ez);
            move(ay[t], ex, ey, ez);
            const cpx<dfl> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
            const df4 x = lin2(sh.x, ax[t], -sh.y, ay[t]), y = lin2(sh.y, ax[t], sh.x, ay[t]);
            float4 *dst = Xi + (size_t(ch) * (2 * nf) + dl) * 4 * S + 4 * j;
            dst[0] = as_float4(x.v[0]);
            dst[1] = as_float4(x.v[1]);
            dst[2] = as_float4(y.v[0]);
            dst[3] = as_float4(y.v[1]);
        }
    }
}


// ---------------------------------------------------------------- far-field evaluation
constexpr int kNE = 18;   // evaluation expansions of Eq. (2.8) per box
constexpr int kNF = 12;   // evaluated per bead after the fold of k_eval_prep (per-potential form)
constexpr int kNF2 = 6;   // evaluated per bead in the one-expansion-per-component form

// Build the 18 evaluation expansions of Eq. (2.8) from 4 source expansions.
// IRREG = multipole source (degrees grow by one per derivative), else local.
template <typename T, bool IRREG>
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
        if (IRREG) d_multipole(src + k * ncoef(p), p, gx, gx + st, gx + 2 * st, P, G);
        else d_local(src + k * ncoef(p), p, gx, gx + st, gx + 2 * st, P, G);
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
    int pl = IRREG ? p + 1 : p - 1;
    if (IRREG) d_multipole(tmp + 3 * st, pl, EV + 15 * st, EV + 16 * st, EV + 17 * st, P, G);
    else d_local(tmp + 3 * st, pl, EV + 15 * st, EV + 16 * st, EV + 17 * st, P, G);
    __syncthreads();
}

// rb: the multipoles carry q4 about their own box centres (box origin), so the
// set-4 gradient is re-based from the source box's centre to the leaf's.
template <typename T>
__global__ void k_far_eval(const int *leaves, DevTables<T> D, const int *beg, const int *end, const double *ctr,
                           const double *side, const int *lvl, const int *bsys, const int *woff, const int *widx,
                           const double *pos, int64_t n, SysConst sc, const cpx<T> *L, const cpx<T> *M,
                           double *ufar, int rb) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int li = blockIdx.x;
    int b = leaves[li];
    const int p = D.p, nc = ncoef(p), P = p + 2, st = ncoef(P);
    T *smr = reinterpret_cast<T *>(smem_raw);
    Rec<T> R = load_rec(D, smr);
    Lad<T> G = load_lad(D, smr + rec_floats<T>(p));
    cpx<T> *EV = reinterpret_cast<cpx<T> *>(smr + tab_floats<T>(p));
    cpx<T> *tmp = EV + kNE * st;
    cpx<T> *srcs = tmp + 4 * st;
    int sy = bsys[b];
    const double C1 = sc.pc[sy].C1, C2 = sc.pc[sy].C2, icube = sc.pc[sy].icube;
    double c0x = sc.cube[4 * sy], c0y = sc.cube[4 * sy + 1], c0z = sc.cube[4 * sy + 2];
    double cbx = ctr[3 * b], cby = ctr[3 * b + 1], cbz = ctr[3 * b + 2];
    float c3b[9];
    if constexpr (kIsDf<T>)
        for (int k = 0; k < 9; ++k) c3b[k] = sc.c3[9 * size_t(b) + k];
    int j0 = beg[b], j1 = end[b];
    int nw = woff[li + 1] - woff[li];
    if (nw == 0) return;
    for (int jc = j0; jc < j1; jc += blockDim.x) {
        int j = jc + threadIdx.x;
        bool act = j < j1;
        double x = act ? pos[j] : cbx, y = act ? pos[n + j] : cby, z = act ? pos[2 * n + j] : cbz;
        double u[3] = {0, 0, 0};
        for (int w = 0; w < nw; ++w) {
            const int C = widx[woff[li] + w];
            const cpx<T> *E = M + size_t(C) * kSets * nc;
            __syncthreads();
            for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) srcs[i] = E[i];
            __syncthreads();
            // origin of the source expansion's q4: its own centre (box origin) or the cube centre
            T acc[kNE];
#pragma unroll
            for (int q = 0; q < kNE; ++q) acc[q] = T(0);
            if constexpr (kIsDf<T>) {
                // lengths in the split units; L4 and the C2 term carry their factors here
                T cb[3], v[3], xi[3];
                const double ihd = inv_side_u(sc.pc[sy], lvl[C]);
                const T ihs = T(ihd);
                for (int a = 0; a < 3; ++a) {
                    cb[a] = rb ? coord_diff(c3b, sc.c3 + 9 * size_t(C), a) : dfl3(c3b[3 * a], c3b[3 * a + 1], c3b[3 * a + 2]);
                    v[a] = act ? coord_diff(sc.p3, n, j, a, sc.c3 + 9 * size_t(C)) * ihs : T(1);
                    xi[a] = act ? coord_diff(sc.p3, n, j, a, c3b) * ihs : T(0);
                }
                build_eval_set<T, true>(srcs, p, P, EV, tmp, cb[0], cb[1], cb[2], G);
                eval_fields<T, kNE, true>(v[0], v[1], v[2], P, EV, st, R.a, R.b, R.c, acc);
                const T cc = T(double(sc.pc[sy].d_k23h) + double(sc.pc[sy].d_k23l)) * ihs;
                const double w1 = sc.pc[sy].C1 * sc.pc[sy].d_xs * force_unit(sc.fmax[sy]) * ihd;
                for (int d = 0; d < 3; ++d) {
                    T t = acc[d] + ihs * (acc[12 + d] - cc * acc[15 + d]);
                    for (int k = 0; k < 3; ++k) t -= xi[k] * acc[3 + 3 * k + d];
                    u[d] += w1 * double(t);
                }
            } else {
                const double ox = rb ? ctr[3 * C] : c0x, oy = rb ? ctr[3 * C + 1] : c0y, oz = rb ? ctr[3 * C + 2] : c0z;
                build_eval_set<T, true>(srcs, p, P, EV, tmp, T(cbx - ox), T(cby - oy), T(cbz - oz), G);
                double ih = icube * pow2i(lvl[C]);   // 1 / side[C], exactly
                T vx = T((x - ctr[3 * C]) * ih), vy = T((y - ctr[3 * C + 1]) * ih), vz = T((z - ctr[3 * C + 2]) * ih);
                eval_fields<T, kNE, true>(vx, vy, vz, P, EV, st, R.a, R.b, R.c, acc);
                double xi[3] = {(x - cbx) * ih, (y - cby) * ih, (z - cbz) * ih};
                for (int d = 0; d < 3; ++d) {
                    double v = double(acc[d]);
                    for (int k = 0; k < 3; ++k) v -= xi[k] * double(acc[3 + 3 * k + d]);
                    u[d] += C1 * ih * v + C1 * ih * ih * double(acc[12 + d]) - C2 * ih * ih * ih * double(acc[15 + d]);
                }
            }
        }
        if (act)
            for (int d = 0; d < 3; ++d) ufar[3 * size_t(j) + d] += u[d];
    }
}

// Per leaf at level >= 2: the 18 derived local expansions of Eq. (2.8),
// written to global memory for the bead-parallel evaluation.
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
    cpx<T> *srcs = reinterpret_cast<cpx<T> *>(smr + ((6 * ncoef(p + 2) + 1) & ~1));
    cpx<T> *tmp = srcs + kSets * nc;
    const cpx<T> *E = L + size_t(b) * kSets * nc;
    for (int i = threadIdx.x; i < kSets * nc; i += blockDim.x) srcs[i] = E[i];
    __syncthreads();
    int sy = bsys[b];
    cpx<T> *EV = EVg + size_t(li) * kNE * nc;
    if (rb) {
        build_eval_set<T, false>(srcs, p, p, EV, tmp, T(0), T(0), T(0), G);
    } else if constexpr (kIsDf<T>) {
        const float *c = sc.c3 + 9 * size_t(b);
        build_eval_set<T, false>(srcs, p, p, EV, tmp, dfl3(c[0], c[1], c[2]), dfl3(c[3], c[4], c[5]),
                                 dfl3(c[6], c[7], c[8]), G);
    } else {
        build_eval_set<T, false>(srcs, p, p, EV, tmp, T(ctr[3 * b] - sc.cube[4 * sy]),
                                 T(ctr[3 * b + 1] - sc.cube[4 * sy + 1]), T(ctr[3 * b + 2] - sc.cube[4 * sy + 2]), G);
    }
    // Fold the terms of Eq. (2.8) that are not multiplied by a coordinate into
    // fields 0..2 (in units of C1/h):  L_d + h^-1 dL4'_d - (C2/C1) h^-2 dL_C,d.
    // The bead evaluation then needs fields 0..11 only.
    const double ih = sc.pc[sy].icube * pow2i(lvl[b]);
    T c4 = T(ih), cc = T(sc.pc[sy].C2 / sc.pc[sy].C1 * ih * ih);
    if constexpr (kIsDf<T>) {   // lengths in the split units: C2 / C1 = 2a^2/3 there
        const double ihs = inv_side_u(sc.pc[sy], lvl[b]);
        c4 = T(ihs);
        cc = T((double(sc.pc[sy].d_k23h) + double(sc.pc[sy].d_k23l)) * ihs * ihs);
    }
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
    int nf = kNF;
    if (per_component) {
        // Approach 2 of Sec. 2: one expansion per velocity component.  With
        // G_kd = dL_k/dx_d (fields 3 + 3k + d, degree <= p - 1) and x the bead
        // offset in box units, sum_k x_k G_kd = A_d + |x|^2 B_d with A_d, B_d
        // harmonic: for each degree-n part h of G_kd, with g = h / (2n + 1),
        //   x_k h = [x_k h - |x|^2 d_k g] + |x|^2 d_k g,
        // where the bracket is -|x|^(2n+3) d_k(g / |x|^(2n+1)) (Kelvin transform:
        // the same coefficients read as a multipole expansion), so
        //   A_d = -sum_k [d_k of g as a multipole, read as a local expansion],
        //   B_d =  sum_k [d_k of g as a local expansion].
        // Fields become H_d = F_d - A_d (0..2, degree <= p) and B_d (3..5).
        __syncthreads();
        for (int i = threadIdx.x; i < 9 * nc; i += blockDim.x) {
            const int c = i % nc;
            const T w = T(1) / T(2 * deg_of(c) + 1);
            cpx<T> v = EV[3 * nc + i];
            EV[3 * nc + i] = mk(w * v.x, w * v.y);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 3 * nc; i += blockDim.x) {
            const int d = i / nc, c = i - d * nc;
            cpx<T> a = mk<T>(0, 0), bb = mk<T>(0, 0);
            for (int k = 0; k < 3; ++k) {
                const cpx<T> *g = EV + (3 + 3 * k + d) * nc;
                a += d_mul_one(g, p - 1, k, c, G);
                bb += d_loc_one(g, p - 1, k, c, G);
            }
            EV[d * nc + c] += a;
            EV[(12 + d) * nc + c] = bb;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 3 * nc; i += blockDim.x) EV[3 * nc + i] = EV[12 * nc + i];
        nf = kNF2;
    }
    __syncthreads();
    // the evaluated fields carry the factor 2 of the m > 0 terms of Re(sum E h)
    for (int i = threadIdx.x; i < nf * nc; i += blockDim.x) {
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
template <typename T, int NF>
__global__ void k_eval_apply(int64_t n, const int *bead_leaf, const int *leaves, DevTables<T> D, const double *ctr,
                             const double *side, const int *lvl, const int *bsys, const double *pos, SysConst sc,
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
            eval_fields<T, NF, false, true>(xi[0], xi[1], xi[2], p, EVg + size_t(li) * kNE * nc, nc, D.rec_a, D.rec_b,
                                            D.rec_c, acc);
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
        eval_fields<T, NF, false, true>(T(xi[0]), T(xi[1]), T(xi[2]), p, EVg + size_t(li) * kNE * nc, nc, D.rec_a,
                                        D.rec_b, D.rec_c, acc);
        if constexpr (NF == kNF2) {
            // fields 0..2: H_d; 3..5: B_d
            const double r2 = xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2];
            for (int d = 0; d < 3; ++d) u[d] = C1 * ih * (double(acc[d]) - r2 * double(acc[3 + d]));
        } else {
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

template <typename T>
static size_t smem_p2x(int p, int threads) {
    const int nc = ncoef(p), chunk = p2x_chunk(p, threads);
    return sizeof(T) * ((rec_floats<T>(p) + 1) & ~1) + sizeof(cpx<T>) * (chunk * nc + 2 * kSets * nc) +
           sizeof(T) * 4 * chunk + 64;
}
template <typename T>
static size_t smem_m2x(int p, int s) {
    int nc = ncoef(p);
    return sizeof(cpx<T>) * (3 * kSets * nc + 2 * s * (kSets * (p + 1) + 1));
}
template <typename T>
static size_t smem_far(int p) {
    int st = ncoef(p + 2);
    return sizeof(T) * tab_floats<T>(p) + sizeof(cpx<T>) * (kNE * st + 4 * st + kSets * ncoef(p)) + 64;
}
template <typename T>
static size_t smem_lap(int p) {
    int st = ncoef(p + 2);
    return sizeof(T) * tab_floats<T>(p) + sizeof(cpx<T>) * (13 * st + 3 * st + ncoef(p)) + 64;
}

// Raise a kernel's dynamic shared-memory limit once per device and kernel
// (never while a stream is being captured: the first, uncaptured matvec sets
// every limit it needs).
static std::mutex g_smem_mu;
static std::map<std::pair<int, const void *>, size_t> g_smem_done;

template <typename K>
static int set_smem(K kernel, size_t bytes) {
    if (bytes <= 40 * 1024) return RPY_OK;   // below the default limit, static shared memory included
    int dev = 0;
    RPY_CHECK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_smem_mu);
    size_t &d = g_smem_done[{dev, reinterpret_cast<const void *>(kernel)}];
    if (bytes > d) {
        RPY_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)));
        d = bytes;
    }
    return RPY_OK;
}

// Threads of an X2X block: each handles elements e, e + blockDim, ... of the
// 4 S merged plane waves; the fewest warps that keep the number of rounds of
// 256 threads, so that the last round is not left nearly empty.
static int even_threads(int items, int most = 256) {
    const int rounds = (items + most - 1) / most;
    return std::max(64, ((items + rounds - 1) / rounds + 31) / 32 * 32);
}
static int x2x_threads(int S) { return even_threads(kSets * S); }

// Node chunks of the double-float M2X and X2L (equal ones): one for all nodes, split until the block's
// shared memory (fixed bytes + per-node bytes + 256 bytes per wave-pair unit when units are staged) is at most
// 48 KB (56 KB with units), or until a chunk of X2L holds at most 200 (node, m) sums, below which its phases
// run out of threads.  Measured: X2L of the 1M-bead sphere (p = 16) 7.2 / 9.9 ms at 49 / 98 KB; of the 200k sphere at 9
// digits (p = 25) 13.9 / 8.5 / 7.5 ms at 56 / 72 / 100 KB; M2X there 11.4 / 5.3 / 5.5 ms at 30 / 48 / 60 KB.
struct NodeChunk {
    int kc, umax;
    size_t smem;
};
static NodeChunk node_chunk(const OpTables &h, bool stage_units) {
    const int nc = ncoef(h.p), NS = a_stride(h.p);
    NodeChunk c{};
    for (int nch = 1; nch <= h.s; ++nch) {   // equal chunks
        const int kc = (h.s + nch - 1) / nch;
        int um = 0;
        for (int k0 = 0; k0 < h.s; k0 += kc) um = std::max(um, h.u_start[std::min(h.s, k0 + kc)] - h.u_start[k0]);
        // the rotation scratch (4 nc float4) shares the memory of the rows and the staged units
        const size_t work = std::max(size_t(8) * kc * NS + (stage_units ? 16 * size_t(um) : 0), size_t(4) * nc);
        c = NodeChunk{kc, um, sizeof(float4) * (4 * size_t(nc) + work)};
        if (c.smem <= (stage_units ? 56u : 48u) * 1024 || (stage_units && kc * (h.p + 1) <= 200)) break;
    }
    return c;
}

static int run_waves_df(Tree &t, const DevTables<dfl> &D, const cpx<dfl> *M, cpx<dfl> *L, int rb, cudaStream_t st) {
    const int nf = t.x_frames, b2 = t.level_off[2], n2 = t.nbox - b2, p = D.p;
    float4 *Xo = static_cast<float4 *>(t.Xo), *Xi = static_cast<float4 *>(t.Xi);
    const NodeChunk cm = node_chunk(*t.tabs, false), cl = node_chunk(*t.tabs, true);
    RPY_TRY(set_smem(k_m2x_df, cm.smem));
    RPY_TRY(set_smem(k_x2l_df, cl.smem));
    for (int f0 = 0; f0 < 3; f0 += nf) {
        prof_mark(t, RPY_STAGE_M2X, st);
        k_m2x_df<<<n2, even_threads(2 * cm.umax), cm.smem, st>>>(b2, D, M, Xo, f0, nf, cm.kc);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
        prof_mark(t, RPY_STAGE_X2X, st);
        if (t.n_x2x_par > 0) {
            const dim3 g(t.n_x2x_par, 2 * nf);
            if (rb)
                k_x2x4_df<<<g, even_threads(D.S), 0, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf, t.side_u, Xo,
                                                           Xi, f0, nf);
            else if (t.n_x2x_par * 2 * nf < kX2XSmallGrid)
                k_x2x_df<256, 2><<<g, even_threads(2 * D.S), 0, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf, Xo,
                                                                      Xi, f0, nf);
            else
                k_x2x_df<128, 5><<<g, even_threads(2 * D.S, 128), 0, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf,
                                                                           Xo, Xi, f0, nf);
            RPY_LAUNCHED(1);
            RPY_CHECK(cudaGetLastError());
        }
        prof_mark(t, RPY_STAGE_X2L, st);
        k_x2l_df<<<n2, even_threads((cl.kc + 1) / 2 * (p + 1) * 2), cl.smem, st>>>(b2, D, Xi, L, f0, nf, cl.kc, cl.umax);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
    }
    return RPY_OK;
}

static int run_waves_f32(Tree &t, const DevTables<float> &D, const cpx<float> *M, cpx<float> *L, int rb,
                         cudaStream_t st) {
    const int nf = t.x_frames, b2 = t.level_off[2], n2 = t.nbox - b2, p = D.p;
    cpx<float> *Xo = static_cast<cpx<float> *>(t.Xo), *Xi = static_cast<cpx<float> *>(t.Xi);
    const size_t smx = smem_m2x<float>(p, D.s), sxl = smem_x2l4(p, D.s, D.S);
    const bool col = y_by_column(sizeof(float), p);
    auto m2x = col ? k_m2x<float, true> : k_m2x<float, false>;
    auto x2l = col ? k_x2l4<true> : k_x2l4<false>;
    RPY_TRY(set_smem(m2x, smx));
    RPY_TRY(set_smem(x2l, sxl));
    for (int f0 = 0; f0 < 3; f0 += nf) {
        prof_mark(t, RPY_STAGE_M2X, st);
        m2x<<<n2, even_threads(D.S), smx, st>>>(b2, n2, D, M, Xo, f0, nf);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
        prof_mark(t, RPY_STAGE_X2X, st);
        if (t.n_x2x_par > 0) {
            const dim3 g(t.n_x2x_par, 2 * nf);
            if (D.S > 256 && D.S <= 480) {
                // a producer warp stages the sources through shared memory by bulk copies
                // (measured faster than per-thread loads from 323 stored waves up; at 3 digits,
                // 134 waves, the per-thread loads below keep two to three blocks per SM and win)
                const size_t sxx = x2x_tma_smem(D.S);
                RPY_TRY(set_smem(k_x2x_tma, sxx));
                k_x2x_tma<<<g, (D.S + 31) / 32 * 32 + 32, sxx, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf,
                                                                     t.b_side, Xo, Xi, f0, nf, rb, t.dev_status);
            } else if (D.S <= 256) {
                // shifts from per-axis factors in shared memory (measured faster there; at more
                // waves the shared memory costs occupancy and the table is faster)
                const size_t sxx = sizeof(float) * ((6 * D.S + 3) & ~3) + 2 * sizeof(cpx<float>) * 6 * D.S;
                if (rb)
                    k_x2x4<float, true><<<g, even_threads(D.S), sxx, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf,
                                                                           t.b_side, Xo, Xi, f0, nf, rb);
                else   // cube origin, few plane waves: one set per thread
                    k_x2x<float, true><<<g, x2x_threads(D.S), sxx, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf,
                                                                         Xo, Xi, f0, nf);
            } else {
                k_x2x4<float, false><<<g, even_threads(D.S), 0, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf,
                                                                      t.b_side, Xo, Xi, f0, nf, rb);
            }
            RPY_LAUNCHED(1);
            RPY_CHECK(cudaGetLastError());
        }
        prof_mark(t, RPY_STAGE_X2L, st);
        // blocks sized to the (node, m) items of the widest phase at low order; at high order the
        // shared memory already limits the blocks per SM and 256 threads hide latency better
        const int tx = D.s * (p + 1) <= 256 ? even_threads(D.s * (p + 1)) : 256;
        x2l<<<n2, tx, sxl, st>>>(b2, n2, D, Xi, L, f0, nf);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
    }
    return RPY_OK;
}

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
    // origin of q4 (RPY charges only; the Laplace diagnostic takes its charges as given):
    // each expansion's own box centre by default in the FP32 form at 6 digits, the cube
    // centre otherwise (in the FP64 form, and at 3 digits, its rounding stays far below the setting)
    const int fl = t.params.flags;
    const int rb = lapq ? 0
                        : (fl & RPY_FLAG_BOX_ORIGIN) ? 1
                        : (fl & RPY_FLAG_CUBE_ORIGIN) ? 0
                        : (sizeof(T) == 4 && t.params.digits >= 6);
    // box sides in the units of the expansions' lengths
    const double *side = kIsDf<T> ? t.side_u : t.b_side;
    // upward pass
    size_t sp = smem_p2x<T>(p, 128);
    RPY_TRY(set_smem(k_p2x<T, 0>, sp));
    RPY_TRY(set_smem(k_p2x<T, 1>, sp));
    k_p2x<T, 0><<<n2, 128, sp, st>>>(b2, n2, D, t.b_begin, t.b_end, t.b_center, side, t.b_level, t.b_leaf,
                                     t.b_sys, t.x_off, t.x_idx, t.pos, fs, lapq, t.n, sc, M, rb);
    RPY_LAUNCHED(1);
    RPY_CHECK(cudaGetLastError());
    prof_mark(t, RPY_STAGE_M2M, st);
    // FP64 form: rotation-based M2M and L2L (fewer operations).  FP32: the dense
    // operators below p = 12, the rotation forms (one child per block) from there
    const bool rot_l = sizeof(T) == 8 || p >= 12;
    size_t smr2 = sizeof(cpx<T>) * 3 * kSets * nc;
    int Dd = 2 * nc, thr = ((Dd + 31) / 32) * 32;
    size_t smd = sizeof(T) * kSets * Dd;
    RPY_TRY(set_smem(k_l2l_rot<T>, smr2));
    RPY_TRY(set_smem(k_m2m_child<T>, smr2));
    if constexpr (sizeof(T) == 4) {
        RPY_TRY(set_smem(k_m2m<T>, smd));
        RPY_TRY(set_smem(k_l2l<T>, smd));
    }
    for (int l = t.nlevels - 2; l >= 2; --l) {
        int lb = t.level_off[l], ln = t.level_off[l + 1] - lb;
        if (ln > 0) {
            const int cb = t.level_off[l + 1], cn = t.level_off[l + 2] - cb;   // their children
            if (rot_l) {
                // the share slots exist whenever a level >= 2 does (tree_alloc_workspace)
                if (cn > 0) {
                    if (!t.m2m_scratch) return RPY_ERR_INTERNAL;
                    cpx<T> *Sc = static_cast<cpx<T> *>(t.m2m_scratch);
                    k_m2m_child<T><<<cn, 256, smr2, st>>>(cb, lb, D, t.b_parent, t.b_cell, side, rb, M, Sc);
                    k_m2m_sum<T><<<ln, 256, 0, st>>>(lb, kSets * nc, t.b_leaf, t.b_child, Sc, M);
                    RPY_LAUNCHED(2);
                }
            } else if constexpr (sizeof(T) == 4) {
                k_m2m<T><<<ln, thr, smd, st>>>(lb, ln, D, t.b_leaf, t.b_child, side, rb, M);
                RPY_LAUNCHED(1);
            }
        }
    }
    RPY_CHECK(cudaGetLastError());
    // plane-wave M2L: all three frames in one pass, or (large trees, where the
    // plane-wave buffers of six directions would not fit) one frame per pass,
    // each pass adding its frame's share into L (with profiling on, every pass's
    // M2X, X2X and X2L launches are timed under their own stages).
    if constexpr (kIsDf<T>) RPY_TRY(run_waves_df(t, D, M, L, rb, st));
    else RPY_TRY(run_waves_f32(t, D, M, L, rb, st));
    // X list
    prof_mark(t, RPY_STAGE_P2L, st);
    k_p2x<T, 1><<<n2, 128, sp, st>>>(b2, n2, D, t.b_begin, t.b_end, t.b_center, side, t.b_level, t.b_leaf,
                                     t.b_sys, t.x_off, t.x_idx, t.pos, fs, lapq, t.n, sc, L, rb);
    RPY_LAUNCHED(1);
    RPY_CHECK(cudaGetLastError());
    // downward pass
    prof_mark(t, RPY_STAGE_L2L, st);
    for (int l = 3; l < t.nlevels; ++l) {
        int lb = t.level_off[l], ln = t.level_off[l + 1] - lb;
        if (ln > 0) {
            if (rot_l) k_l2l_rot<T><<<ln, 256, smr2, st>>>(lb, ln, D, t.b_parent, t.b_cell, side, rb, L);
            else if constexpr (sizeof(T) == 4) k_l2l<T><<<ln, thr, smd, st>>>(lb, ln, D, t.b_parent, t.b_cell, side, rb, L);
            RPY_LAUNCHED(1);
        }
    }
    RPY_CHECK(cudaGetLastError());
    prof_mark(t, RPY_STAGE_EVAL, st);
    if (ufar) {
        cpx<T> *EVg = static_cast<cpx<T> *>(t.EVg);
        size_t sp2 = sizeof(T) * (((6 * ncoef(p + 2) + 1) & ~1)) + sizeof(cpx<T>) * 2 * kSets * nc + 64;
        RPY_TRY(set_smem(k_eval_prep<T>, sp2));
        // one expansion per velocity component unless the per-potential form is asked for
        const int per_comp = (t.params.flags & RPY_FLAG_EVAL_PER_POTENTIAL) ? 0 : 1;
        k_eval_prep<T><<<t.nleaf, 128, sp2, st>>>(t.leaves, D, t.b_center, t.b_level, t.b_sys, sc, L, EVg, per_comp,
                                                  rb);
        RPY_LAUNCHED(1);
        const int ga = int((t.n + 127) / 128);
        if (per_comp)
            k_eval_apply<T, kNF2><<<ga, 128, 0, st>>>(t.n, t.bead_leaf, t.leaves, D, t.b_center, side, t.b_level,
                                                      t.b_sys, t.pos, sc, EVg, ufar);
        else
            k_eval_apply<T, kNF><<<ga, 128, 0, st>>>(t.n, t.bead_leaf, t.leaves, D, t.b_center, side, t.b_level,
                                                     t.b_sys, t.pos, sc, EVg, ufar);
        RPY_LAUNCHED(1);
        size_t sf = smem_far<T>(p);
        RPY_TRY(set_smem(k_far_eval<T>, sf));
        k_far_eval<T><<<t.nleaf, 64, sf, st>>>(t.leaves, D, t.b_begin, t.b_end, t.b_center, side, t.b_level,
                                                t.b_sys, t.w_off, t.w_idx, t.pos, t.n, sc, L, M, ufar, rb);
        RPY_LAUNCHED(1);
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
