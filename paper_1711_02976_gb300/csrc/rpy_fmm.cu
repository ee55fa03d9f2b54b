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

#include "rpy_far.h"
#include "rpy_harmonics.h"

namespace rpy {

// ---------------------------------------------------------------- harmonics, several points per warp
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
    const int nc = ncoef(p), chunk = p2x_chunk(p, threads);
    return sizeof(T) * ((rec_floats<T>(p) + 1) & ~1) + sizeof(cpx<T>) * (chunk * nc + 2 * kSets * nc) +
           sizeof(T) * 4 * chunk + 64;
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
    RPY_TRY(run_m2m_t(t, D, M, rb, st));
    // plane-wave M2L: all three frames in one pass, or (large trees, where the
    // plane-wave buffers of six directions would not fit) one frame per pass,
    // each pass adding its frame's share into L (with profiling on, every pass's
    // M2X, X2X and X2L launches are timed under their own stages).
    RPY_TRY(run_waves_t(t, D, M, L, rb, st));
    // X list
    prof_mark(t, RPY_STAGE_P2L, st);
    k_p2x<T, 1><<<n2, 128, sp, st>>>(b2, n2, D, t.b_begin, t.b_end, t.b_center, side, t.b_level, t.b_leaf,
                                     t.b_sys, t.x_off, t.x_idx, t.pos, fs, lapq, t.n, sc, L, rb);
    RPY_LAUNCHED(1);
    RPY_CHECK(cudaGetLastError());
    // downward pass
    prof_mark(t, RPY_STAGE_L2L, st);
    RPY_TRY(run_l2l_t(t, D, L, rb, st));
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
