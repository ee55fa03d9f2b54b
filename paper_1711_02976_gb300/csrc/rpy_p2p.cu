// Near field: direct RPY tensor (Sec. 1) over the U list of every leaf, the
// self term, and the final combine / unpermute of the matvec.
//
// One CTA per work item: up to 256 target beads of one leaf (large leaves are
// split into several items, launched in decreasing order of cost).  The beads of
// the leaf's source boxes are staged through shared memory in chunks (coalesced
// SoA loads) and every thread sums its own targets.
//
// Pair blocks (R = r_i - r_j, s = kT/eta):
//   r >= 2a : s/(8 pi r) [ (1 + 2a^2/(3r^2)) F + (1 - 2a^2/r^2) (R.F)/r^2 R ]
//   0<r<2a  : s/(6 pi a) [ (1 - 9r/(32a)) F + (3/(32a)) (R.F)/r R ]   (standard overlap form)
//   r = 0   : s/(6 pi a) F                                           (r -> 0 limit)
// The self term s/(6 pi a) F_i is added once.
//
// FP64 form (k_p2p_df): every pair value and sum is a double-float, the unevaluated sum of two FP32
// numbers (about 48 significant bits; two-sum of Knuth, products by FMA as in Dekker 1971 /
// Ogita, Rump and Oishi 2005).  This part executes 2 FP64 operations per SM and clock but
// 128 FP32 ones: 24 FP64 operations per pair cost 12 cycles, the 200 FP32 operations of
// the double-float form under 2.  The running sums go to FP64 every kDfBlock pairs of sources.  Pairs closer
// than 2^-24 of the root cube's side, leaves below level 17 and systems whose
// lengths or forces lie outside the FP32 exponent range take every operation in FP64 (near64).
// FP32 form (precision setting, k_p2p32): positions relative to the target
// leaf centre in FP32; every thread carries one target and takes two staged sources in
// the two lanes of packed FP32x2 operations, four sources per iteration; an
// iteration whose pairs are all far (across the warp) evaluates the far branch
// alone, any other evaluates both branches with selects; accumulation is Kahan-compensated across blocks of kP32Block sources;
// pairs closer than 1e-3 a (where the FP32 difference of coordinates loses the
// direction) are recomputed in FP64 from the FP64 positions.
#include <cmath>

#include <mutex>
#include <set>

#include "rpy_internal.h"

namespace rpy {

constexpr int kP2PThreads = 256;

// Reciprocal square root for r2 > 0: an FP32 seed taken from the bit pattern
// of r2 (exponent rebased from 1023 to 127, mantissa truncated to 23 bits, by
// integer operations only), rsqrtf of it, and one Newton step in FP64,
//   e = 1 - r2 y0^2,  y = y0 + (y0/2) e      (relative error ~1.5 d^2 for a seed error d),
// with y0/2 formed by decrementing the exponent.  Returns false when r2 lies
// outside the normal FP32 range; the caller then takes 1/sqrt(r2).
__device__ __forceinline__ bool rsqrt_seeded(double r2, double &ri) {
    const unsigned hi = unsigned(__double2hiint(r2)), lo = unsigned(__double2loint(r2));
    const unsigned he = hi - (896u << 20);
    if (he - (1u << 20) >= (254u << 20)) return false;   // FP32 exponent outside [1, 254]
    const float y0f = rsqrtf(__uint_as_float(__funnelshift_l(lo, he, 3)));
    const unsigned yb = __float_as_uint(y0f);
    const double y0 = __hiloint2double(int((yb >> 3) + (896u << 20)), int(yb << 29));
    const double y0h = __hiloint2double(int((yb >> 3) + (895u << 20)), int(yb << 29));
    const double e = fma(-r2 * y0, y0, 1.0);
    ri = fma(y0h, e, y0);
    return true;
}

__device__ __forceinline__ void overlap_pair(double dx, double dy, double dz, double r2, double fx, double fy, double fz,
                                             double a, double co, double *acc) {
    if (r2 > 0.0) {
        double r = sqrt(r2);
        double RF = dx * fx + dy * fy + dz * fz;
        double t1 = co * (1.0 - 9.0 * r / (32.0 * a));
        double t2 = co * (3.0 / (32.0 * a)) * RF / r;
        acc[0] += t1 * fx + t2 * dx;
        acc[1] += t1 * fy + t2 * dy;
        acc[2] += t1 * fz + t2 * dz;
    } else {
        acc[0] += co * fx;
        acc[1] += co * fy;
        acc[2] += co * fz;
    }
}

// Hardware reciprocal square root, flushing subnormals (the argument here is at
// least 1e-6 a^2, kept normal by k_pair_const).
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Source staging: the beads of all source boxes of a leaf's list are streamed
// through shared memory in chunks of blockDim, across box boundaries.  Every
// thread locates its bead of the chunk by walking the list from a uniform
// cursor (lists hold a few dozen boxes).
struct SrcCursor {
    int u, off;   // list position and offset inside that box
};

__device__ __forceinline__ int cursor_locate(SrcCursor c, int u1, int t, const int *uidx, const int *beg,
                                             const int *end) {
    int u = c.u, off = c.off;
    while (u < u1) {
        int C = uidx[u];
        int avail = end[C] - beg[C] - off;
        if (t < avail) return beg[C] + off + t;
        t -= avail;
        ++u;
        off = 0;
    }
    return -1;
}

__device__ __forceinline__ SrcCursor cursor_advance(SrcCursor c, int u1, int t, const int *uidx, const int *beg,
                                                    const int *end) {
    while (c.u < u1) {
        int C = uidx[c.u];
        int avail = end[C] - beg[C] - c.off;
        if (t < avail) {
            c.off += t;
            return c;
        }
        t -= avail;
        ++c.u;
        c.off = 0;
    }
    return c;
}

// All pairs of one item in FP64: the general form, for what k_p2p_df cannot represent.  smem
// holds 9 x kP2PThreads doubles and kP2PThreads ints.
// Thread layout: R = min(T, blockDim) targets per pass and G = blockDim / R groups; group g takes
// every G-th bead of each staged chunk.  Far pairs accumulate in units of s/(8 pi) (applied
// once per target) with explicit FMAs: 24 FP64 operations per pair and no conversions; 1/r from a
// single-precision seed and one Newton step.
__device__ __noinline__ void near64(unsigned char *smem, int tb, int te, int u0, int u1, const int *beg,
                                    const int *end, const int *uidx, const double *pos, const double *fs, int64_t n,
                                    const PairConst &pc, int add_self, double *out) {
    double *sx = reinterpret_cast<double *>(smem), *sy = sx + kP2PThreads, *sz = sy + kP2PThreads;
    double *sfx = sz + kP2PThreads, *sfy = sfx + kP2PThreads, *sfz = sfy + kP2PThreads, *red = sfz + kP2PThreads;
    int *sj = reinterpret_cast<int *>(red + 3 * kP2PThreads);
    const double a = pc.a, co = pc.co, cf = pc.cf, k23 = pc.k23, nk2 = pc.nk2;
    const long long a2x4 = __double_as_longlong(pc.a2x4);   // r2 >= 4a^2 compared on the bit patterns
    const int nt = te - tb;
    const int Rn = nt < kP2PThreads ? nt : kP2PThreads;
    const int G = kP2PThreads / Rn;
    const int tl = threadIdx.x % Rn, g = threadIdx.x / Rn;
    for (int i0 = tb; i0 < te; i0 += Rn) {
        const int i = i0 + tl;
        const bool act = i < te && g < G;
        const double xi = act ? pos[i] : 0.0, yi = act ? pos[n + i] : 0.0, zi = act ? pos[2 * n + i] : 0.0;
        double ax = 0, ay = 0, az = 0;   // far pairs, units of s/(8 pi)
        double accd[3] = {0, 0, 0};      // overlapping pairs
        SrcCursor cur{u0, 0};
        while (cur.u < u1) {
            __syncthreads();
            int j = cursor_locate(cur, u1, threadIdx.x, uidx, beg, end);
            sj[threadIdx.x] = j;
            if (j >= 0) {
                sx[threadIdx.x] = pos[j];
                sy[threadIdx.x] = pos[n + j];
                sz[threadIdx.x] = pos[2 * n + j];
                sfx[threadIdx.x] = fs[j];
                sfy[threadIdx.x] = fs[n + j];
                sfz[threadIdx.x] = fs[2 * n + j];
            }
            cur = cursor_advance(cur, u1, kP2PThreads, uidx, beg, end);
            __syncthreads();
            if (!act) continue;
            for (int jj = g; jj < kP2PThreads; jj += G) {
                const int jg = sj[jj];
                if (jg < 0) break;
                const double dx = xi - sx[jj], dy = yi - sy[jj], dz = zi - sz[jj];
                const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
                const double fx = sfx[jj], fy = sfy[jj], fz = sfz[jj];
                if (__double_as_longlong(r2) >= a2x4) {
                    // [(1 + 2a^2/(3r^2)) F + (1 - 2a^2/r^2)(R.F)/r^2 R] / r = t1 F + t2 R,
                    //   t1 = ri + k23 ri^3,  t2 = ri^3 (1 - 2a^2 ri^2) R.F
                    double ri;
                    if (!rsqrt_seeded(r2, ri)) ri = 1.0 / sqrt(r2);
                    const double ri2 = ri * ri;
                    const double B = ri * ri2;
                    const double t1 = fma(k23, B, ri);
                    const double w = fma(nk2, ri2, 1.0);
                    const double RF = fma(dz, fz, fma(dy, fy, dx * fx));
                    const double t2 = (B * w) * RF;
                    ax = fma(t2, dx, fma(t1, fx, ax));
                    ay = fma(t2, dy, fma(t1, fy, ay));
                    az = fma(t2, dz, fma(t1, fz, az));
                } else if (jg != i) {
                    overlap_pair(dx, dy, dz, r2, fx, fy, fz, a, co, accd);
                }
            }
        }
        __syncthreads();
        red[threadIdx.x] = fma(cf, ax, accd[0]);
        red[kP2PThreads + threadIdx.x] = fma(cf, ay, accd[1]);
        red[2 * kP2PThreads + threadIdx.x] = fma(cf, az, accd[2]);
        __syncthreads();
        if (act && g == 0) {
            double v[3];
            for (int c = 0; c < 3; ++c) {
                v[c] = red[c * kP2PThreads + threadIdx.x];
                for (int gg = 1; gg < G; ++gg) v[c] += red[c * kP2PThreads + threadIdx.x + gg * Rn];
            }
            const double cs = add_self ? co : 0.0;
            out[3 * size_t(i)] = v[0] + cs * fs[i];
            out[3 * size_t(i) + 1] = v[1] + cs * fs[n + i];
            out[3 * size_t(i) + 2] = v[2] + cs * fs[2 * n + i];
        }
    }
}

// Thread layout of k_p2p_df: an item of T targets is taken in P parts of R = ceil(T / P) targets, G = threads / R
// groups of R threads each; every group takes its share of the staged sources for the thread's target of
// each part in turn.  T G / (P threads) of the lanes do work; another part must raise that by 6%, since each
// has its own block sums (T = 57: one part 89%, three 97%).  15M-bead cube: one part 155.4 ms, at most three 149.1, four
// 147.9; without the 6% small leaves lose (4,096 beads 0.024 -> 0.034 ms).
struct TargetParts {
    int P, R, G;
};
__device__ __forceinline__ TargetParts target_parts(int nt, int threads, int most) {
    TargetParts b{1, nt, threads / nt};
    for (int P = 2; P <= most; ++P) {
        const int R = (nt + P - 1) / P, G = threads / R;
        if (16 * G * b.P > 17 * b.G * P) b = TargetParts{P, R, G};
    }
    return b;
}

// ---------------------------------------------------------------- FP64 form in double-floats

// Positions of the FP64 form as three floats per coordinate, x' = h + m + l in units of 2^e with e the
// exponent of the root cube's side, relative to the cube's centre: h a multiple of 2^-23 and m of 2^-46, so
// that the differences of two h's and of two m's are exact in FP32, and l the rest, rounded
// at 2^-71: the difference of two FP64 coordinates is kept to its last bit.
__device__ __forceinline__ void split3(double x, double c, double xs, float &fh, float &fm, float &fl) {
    const double d = x - c, bb = d - x, err = (x - (d - bb)) + (-c - bb);   // d + err = x - c exactly
    const double v = d * xs;
    const double h = (v + 805306368.0) - 805306368.0;   // 1.5 * 2^29: ulp 2^-23
    const double r = v - h;
    const double m = (r + 96.0) - 96.0;                 // 1.5 * 2^6: ulp 2^-46
    fh = float(h);
    fm = float(m);
    fl = float((r - m) + err * xs);
}

// The beads [9][n] and the box centres [nbox][9], and the box sides in the same units.
__global__ void k_split3(const double *pos, const int *bead_sys, const double *cube, int64_t n, const double *ctr,
                         const double *side, const int *bsys, int nbox, float *p3, float *c3, double *side_u) {
    int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) {
        const double *c = cube + 4 * bead_sys[i];
        const double xs = near_unit(c[3]);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            split3(pos[a * n + i], c[a], xs, p3[3 * a * n + i], p3[(3 * a + 1) * n + i], p3[(3 * a + 2) * n + i]);
        return;
    }
    i -= n;
    if (i >= nbox) return;
    const double *c = cube + 4 * bsys[i];
    const double xs = near_unit(c[3]);
    side_u[i] = side[i] * xs;
    for (int a = 0; a < 3; ++a)
        split3(ctr[3 * i + a], c[a], xs, c3[9 * i + 3 * a], c3[9 * i + 3 * a + 1], c3[9 * i + 3 * a + 2]);
}

int split_positions_f64(Tree &t, cudaStream_t st) {
    k_split3<<<unsigned((t.n + t.nbox + 255) / 256), 256, 0, st>>>(t.pos, t.bead_sys, t.sys_cube, t.n, t.b_center,
                                                                   t.b_side, t.b_sys, t.nbox, t.p3, t.c3, t.side_u);
    RPY_LAUNCHED(1);
    RPY_CHECK(cudaGetLastError());
    return RPY_OK;
}

// Sorted forces as double-floats in units of 2^e, e the exponent of the system's largest component.
__global__ void k_split_force(const double *fs, const int *bead_sys, const int *fmax, int64_t n, float *f2) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double sc = force_scale(fmax[bead_sys[i]]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double v = fs[a * n + i] * sc;
        const float h = float(v);
        f2[(2 * a) * n + i] = h;
        f2[(2 * a + 1) * n + i] = float(v - double(h));
    }
}

int split_forces_f64(Tree &t, cudaStream_t st) {
    k_split_force<<<unsigned((t.n + 255) / 256), 256, 0, st>>>(t.fs, t.bead_sys, t.sys_fmax, t.n, t.f2);
    RPY_LAUNCHED(1);
    RPY_CHECK(cudaGetLastError());
    return RPY_OK;
}

// The difference of two coordinates held as three floats, normalised.
__device__ __forceinline__ df2 diff3(float2 xh, float2 xm, float2 xl, float2 sh, float2 sm, float2 sl) {
    const float2 dh = sub2(xh, sh), dm = sub2(xm, sm), dl = sub2(xl, sl);   // the first two exact
    df2 r;
    r.h = add2(dh, dm);                          // dh = 0 or |dh| >= |dm|
    r.l = add2(sub2(dm, sub2(r.h, dh)), dl);
    return r;
}

// What both branches of a pair share: r^2 (hi part r2), 1/r = ri and 1/r^2 = ri2 as
// double-floats, and R.F.
struct PairDf {
    df2 r2, ri, ri2, rf;
};

__device__ __forceinline__ void pair_r2(const df2 *D, df2 &r2) {
    const float2 px = mul2(D[0].h, D[0].h), py = mul2(D[1].h, D[1].h), pz = mul2(D[2].h, D[2].h);
    const float2 ex = fma2(D[0].h, D[0].h, neg2(px)), ey = fma2(D[1].h, D[1].h, neg2(py)),
                 ez = fma2(D[2].h, D[2].h, neg2(pz));
    const float2 ll = fma2(D[2].h, D[2].l, fma2(D[1].h, D[1].l, mul2(D[0].h, D[0].l)));
    float2 t1, t2;
    r2.h = two_sum2(two_sum2(px, py, t1), pz, t2);
    r2.l = fma2(dup(2.f), ll, add2(add2(ex, ey), add2(ez, add2(t1, t2))));
}

// 1/r from the hardware approximation y of 1/sqrt(r2): one Newton step with the residual r^2 y^2 - 1 from
// u = r^2 y brings y within half an ulp and a bit; then, with exact products, z = r^2 y^2 - 1 again and
// 1/r = y (1 - z/2 + 3 z^2/8).  (An FP32 residual in the first step leaves y, and with it the roundings of
// every low part below, 1.5 times as far off.)
__device__ __forceinline__ void pair_common(const df2 *D, const df2 *F, float2 r2clamped, PairDf &P) {
    float2 y = make_float2(rsqrt_ftz(r2clamped.x), rsqrt_ftz(r2clamped.y));
    const float2 u = mul2(P.r2.h, y), eu = fma2(P.r2.l, y, fma2(P.r2.h, y, neg2(u)));
    y = fma2(mul2(y, dup(-0.5f)), fma2(eu, y, fma2(u, y, dup(-1.f))), y);
    const float2 p2 = mul2(y, y), e2 = fma2(y, y, neg2(p2));
    const float2 z = add2(fma2(P.r2.h, p2, dup(-1.f)), fma2(P.r2.h, e2, mul2(P.r2.l, p2)));
    const float2 d = mul2(z, fma2(dup(0.375f), z, dup(-0.5f)));
    P.ri.h = y;
    P.ri.l = mul2(y, d);
    P.ri2.h = p2;
    P.ri2.l = fma2(p2, add2(d, d), e2);
    const float2 qx = mul2(D[0].h, F[0].h), qy = mul2(D[1].h, F[1].h), qz = mul2(D[2].h, F[2].h);
    const float2 ex = fma2(D[0].h, F[0].h, neg2(qx)), ey = fma2(D[1].h, F[1].h, neg2(qy)),
                 ez = fma2(D[2].h, F[2].h, neg2(qz));
    float2 cl = mul2(D[0].h, F[0].l);
    cl = fma2(D[0].l, F[0].h, cl);
    cl = fma2(D[1].h, F[1].l, cl);
    cl = fma2(D[1].l, F[1].h, cl);
    cl = fma2(D[2].h, F[2].l, cl);
    cl = fma2(D[2].l, F[2].h, cl);
    float2 t1, t2;
    P.rf.h = two_sum2(two_sum2(qx, qy, t1), qz, t2);
    P.rf.l = add2(add2(add2(ex, ey), add2(ez, add2(t1, t2))), cl);
}

// r >= 2a:  T1 = ri (1 + V),  T2 = ri^3 (1 - 3V) R.F,  V = (2a^2/3) ri^2 <= 1/6
__device__ __forceinline__ void pair_far(const PairDf &P, df2 k23, df2 &T1, df2 &T2) {
    const df2 V = mul_df(P.ri2, k23);
    df2 a1, a2;
    a1.h = add2(dup(1.f), V.h);
    a1.l = add2(sub2(V.h, sub2(a1.h, dup(1.f))), V.l);
    a2.h = fma2(dup(-3.f), V.h, dup(1.f));
    a2.l = fma2(dup(-3.f), V.l, fma2(dup(-3.f), V.h, sub2(dup(1.f), a2.h)));
    T1 = mul_df(P.ri, a1);
    T2 = mul_df(mul_df(mul_df(P.ri2, a2), P.rf), P.ri);
}

// 0 < r < 2a, in the same units:  T1 = 4/(3a) (1 - 9r/(32a)),  T2 = 1/(8 a^2) ri R.F
__device__ __forceinline__ void pair_overlap(const PairDf &P, const PairConst &pc, df2 &T1, df2 &T2) {
    const df2 c9{dup(pc.d_c9h), dup(pc.d_c9l)}, c43{dup(pc.d_c43h), dup(pc.d_c43l)}, c8{dup(pc.d_c8h), dup(pc.d_c8l)};
    const df2 v = mul_df(mul_df(P.r2, P.ri), c9);   // <= 9/16
    df2 b;
    b.h = sub2(dup(1.f), v.h);
    b.l = sub2(sub2(sub2(dup(1.f), b.h), v.h), v.l);
    T1 = mul_df(b, c43);
    T2 = mul_df(mul_df(P.ri, c8), P.rf);
}

// S + C += T1 F + T2 D, renormalised
__device__ __forceinline__ void accumulate_df(df2 T1, df2 F, df2 T2, df2 D, float2 &S, float2 &C) {
    const df2 q1 = mul_df(T1, F), q2 = mul_df(T2, D);
    float2 t1, t2;
    const float2 h = two_sum2(q1.h, q2.h, t1);
    const float2 lo = add2(add2(q1.l, q2.l), t1);
    const float2 s = two_sum2(S, h, t2);
    const float2 c = add2(t2, add2(C, lo));
    S = add2(s, c);
    C = sub2(c, sub2(S, s));
}

// A pair closer than 2^-24 of the root cube's side, from the FP64 positions.
__device__ __noinline__ void pair_tiny_f64(int j, int i, const PairConst &pc, const double *pos, const double *fs,
                                           int64_t n, double *acc) {
    const double dx = pos[i] - pos[j], dy = pos[n + i] - pos[n + j], dz = pos[2 * n + i] - pos[2 * n + j];
    const double fx = fs[j], fy = fs[n + j], fz = fs[2 * n + j], r2 = dx * dx + dy * dy + dz * dz;
    if (r2 >= pc.a2x4) {
        const double ri = 1.0 / sqrt(r2), ri2 = ri * ri;
        const double t1 = pc.cf * fma(pc.k23, ri2 * ri, ri);
        const double t2 = pc.cf * ri * ri2 * fma(pc.nk2, ri2, 1.0) * (dx * fx + dy * fy + dz * fz);
        acc[0] += t1 * fx + t2 * dx;
        acc[1] += t1 * fy + t2 * dy;
        acc[2] += t1 * fz + t2 * dz;
    } else {
        overlap_pair(dx, dy, dz, r2, fx, fy, fz, pc.a, pc.co, acc);
    }
}

constexpr int kDfThreads = kP2PThreads;
constexpr int kDfChunk = 512;    // sources staged per pass
constexpr int kDfList = 256;     // list boxes per prefix segment
constexpr int kDfStride = 9;     // float4 per staged pair of sources: 15 packed values, 2 indices, 1 of padding
constexpr int kDfBlock = 8;      // pairs of sources per double-float block between FP64 sums
constexpr int kDfMaxLevel = 17;  // deeper leaves hold pairs closer than the three-float split resolves
constexpr int kDfParts = 4;      // parts of an item's targets at most
constexpr size_t kDfSmem = sizeof(float4) * kDfStride * (kDfChunk / 2) + sizeof(double) * 6 * kDfParts * kDfThreads +
                           sizeof(int) * (2 * kDfList + 4);
static_assert(sizeof(float4) * kDfStride * (kDfChunk / 2) >= kP2PThreads * (9 * sizeof(double) + sizeof(int)),
              "near64 works in the staging buffer");

// The list's beads are staged in chunks as pairs (two sources in the two lanes of the packed operations), and
// group g takes every G-th pair for the thread's target of each part.  The list's boxes are prefix-summed in shared
// memory and each staged bead finds its box by binary search.  A pair of sources stands in 9 float4 (8 used): the
// groups of a warp then read different banks.
__global__ void __launch_bounds__(kDfThreads, 2)
    k_p2p_df(const int4 *items, const int *beg, const int *end, const int *bsys, const int *lvl,
             const int *uoff, const int *uidx, const float *p3, const float *f2, const int *fmax, const double *pos,
             const double *fs, int64_t n, SysConst sc, int add_self, double *out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *sS = reinterpret_cast<float4 *>(smem_raw);
    double *sU = reinterpret_cast<double *>(sS + kDfStride * (kDfChunk / 2));   // [part][3][threads] running sums
    double *sD = sU + 3 * kDfParts * kDfThreads;                                 // [part][threads][3] FP64 pairs
    int *lb = reinterpret_cast<int *>(sD + 3 * kDfParts * kDfThreads), *lpre = lb + kDfList;
    int *any64 = lpre + kDfList + 1;
    const int4 item = items[blockIdx.x];
    const int li = item.x, b = item.y, sys = bsys[b];
    const int tb = item.z, te = item.w, nt = te - tb;
    const int u0 = uoff[li], u1 = uoff[li + 1];
    const PairConst &pc = sc.pc[sys];
    const int fw = fmax[sys];
    if (!pc.d_ok || !near_range_ok(fw) || lvl[b] > kDfMaxLevel) {
        near64(smem_raw, tb, te, u0, u1, beg, end, uidx, pos, fs, n, pc, add_self, out);
        return;
    }
    const float lim = pc.d_lim, tiny = kDfTiny2;
    const df2 k23{dup(pc.d_k23h), dup(pc.d_k23l)};
    const TargetParts tp = target_parts(nt, kDfThreads, kDfParts);
    const int G = tp.G, tl = threadIdx.x % tp.R, g = threadIdx.x / tp.R;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int c = 0; c < 3 * tp.P; ++c) {
        sU[c * kDfThreads + threadIdx.x] = 0.0;
        sD[c * kDfThreads + threadIdx.x] = 0.0;
    }
    if (threadIdx.x == 0) *any64 = 0;
    for (int us = u0; us < u1; us += kDfList) {
        const int L = min(kDfList, u1 - us);
        __syncthreads();
        if (warp == 0) {   // prefix of the box sizes of this list segment
            int carry = 0;
            for (int q0 = 0; q0 < L; q0 += 32) {
                const int q = q0 + lane;
                int cnt = 0;
                if (q < L) {
                    const int C = uidx[us + q];
                    lb[q] = beg[C];
                    cnt = end[C] - beg[C];
                }
                int v = cnt;
                for (int o = 1; o < 32; o <<= 1) {
                    const int w = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += w;
                }
                if (q < L) lpre[q + 1] = carry + v;
                carry += __shfl_sync(0xffffffffu, v, 31);
            }
            if (lane == 0) lpre[0] = 0;
        }
        __syncthreads();
        const int Ns = lpre[L];
        for (int c0 = 0; c0 < Ns; c0 += kDfChunk) {
            const int nS = min(kDfChunk, Ns - c0), nP = (nS + 1) >> 1;
            // the barrier after the prefix or after the previous chunk's pairs orders these writes
            for (int e = threadIdx.x; e < 2 * nP; e += kDfThreads) {
                float *w = reinterpret_cast<float *>(sS + kDfStride * (e >> 1)) + (e & 1);
                if (e < nS) {
                    const int q = c0 + e;
                    int lo = 0, hi = L;   // box: lpre[lo] <= q < lpre[lo + 1]
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (lpre[mid] <= q) lo = mid;
                        else hi = mid;
                    }
                    const int j = lb[lo] + (q - lpre[lo]);
#pragma unroll
                    for (int k = 0; k < 9; ++k) w[2 * k] = p3[k * n + j];
#pragma unroll
                    for (int k = 0; k < 6; ++k) w[18 + 2 * k] = f2[k * n + j];
                    reinterpret_cast<int *>(w)[30] = j;
                } else {   // an odd last source gets a partner without force, 3.5 units from every bead or more
#pragma unroll
                    for (int k = 0; k < 15; ++k) w[2 * k] = k == 0 ? 4.f : 0.f;
                    reinterpret_cast<int *>(w)[30] = -1;
                }
            }
            __syncthreads();
            for (int part = 0; part < tp.P && g < G; ++part) {
                const int i = tb + part * tp.R + tl;
                if (i >= te) break;
                float2 X[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) X[k] = dup(p3[k * n + i]);
                double *const U = sU + 3 * part * kDfThreads + threadIdx.x;
                double *const tiny64 = sD + 3 * (part * kDfThreads + threadIdx.x);
                for (int e0 = g; e0 < nP; e0 += kDfBlock * G) {
                    float2 S[3], C[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) S[c] = C[c] = dup(0.f);
                    const int e1 = min(nP, e0 + kDfBlock * G);
                    for (int e = e0; e < e1; e += G) {
                        const float4 *s = sS + kDfStride * e;
                        const float4 v0 = s[0], v1 = s[1], v2 = s[2], v3 = s[3], v4 = s[4], v5 = s[5], v6 = s[6], v7 = s[7];
                        df2 D[3], F[3];
                        D[0] = diff3(X[0], X[1], X[2], make_float2(v0.x, v0.y), make_float2(v0.z, v0.w),
                                     make_float2(v1.x, v1.y));
                        D[1] = diff3(X[3], X[4], X[5], make_float2(v1.z, v1.w), make_float2(v2.x, v2.y),
                                     make_float2(v2.z, v2.w));
                        D[2] = diff3(X[6], X[7], X[8], make_float2(v3.x, v3.y), make_float2(v3.z, v3.w),
                                     make_float2(v4.x, v4.y));
                        F[0] = df2{make_float2(v4.z, v4.w), make_float2(v5.x, v5.y)};
                        F[1] = df2{make_float2(v5.z, v5.w), make_float2(v6.x, v6.y)};
                        F[2] = df2{make_float2(v6.z, v6.w), make_float2(v7.x, v7.y)};
                        PairDf P;
                        pair_r2(D, P.r2);
                        df2 T1, T2;
                        if (__all_sync(__activemask(), fminf(P.r2.h.x, P.r2.h.y) >= lim)) {
                            pair_common(D, F, P.r2.h, P);
                            pair_far(P, k23, T1, T2);
                        } else {
                            // some lane has an overlapping, very close or self pair: both branches with selects
                            pair_common(D, F, make_float2(fmaxf(P.r2.h.x, tiny), fmaxf(P.r2.h.y, tiny)), P);
                            df2 O1, O2;
                            pair_far(P, k23, T1, T2);
                            pair_overlap(P, pc, O1, O2);
                            // far, then overlapping, then FP64 (lim = tiny where 2a is below the split's resolution:
                            // a pair exactly there is far)
                            const bool fx = P.r2.h.x >= lim, fy = P.r2.h.y >= lim;
                            const bool ox = P.r2.h.x > tiny, oy = P.r2.h.y > tiny;
                            auto pick = [&](float2 far, float2 near) {
                                return make_float2(fx ? far.x : (ox ? near.x : 0.f), fy ? far.y : (oy ? near.y : 0.f));
                            };
                            T1.h = pick(T1.h, O1.h);
                            T1.l = pick(T1.l, O1.l);
                            T2.h = pick(T2.h, O2.h);
                            T2.l = pick(T2.l, O2.l);
                            const bool tx = !fx && !ox, ty = !fy && !oy;
                            if (tx || ty) {
                                const int jx = __float_as_int(v7.z), jy = __float_as_int(v7.w);
                                if (tx && jx != i) {
                                    pair_tiny_f64(jx, i, pc, pos, fs, n, tiny64);
                                    *any64 = 1;
                                }
                                if (ty && jy != i) {
                                    pair_tiny_f64(jy, i, pc, pos, fs, n, tiny64);
                                    *any64 = 1;
                                }
                            }
                        }
#pragma unroll
                        for (int c = 0; c < 3; ++c) accumulate_df(T1, F[c], T2, D[c], S[c], C[c]);
                    }
                    // the two lanes of the block into the FP64 sums
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const float s = S[c].x + S[c].y, bb = s - S[c].x;
                        const float e = (S[c].x - (s - bb)) + (S[c].y - bb);
                        U[c * kDfThreads] += double(s) + double((C[c].x + C[c].y) + e);
                    }
                }
            }
            __syncthreads();
        }
    }
    __syncthreads();
    // one thread per (component, target) adds the groups in order
    const double unit = pc.cf * pc.d_xs * force_unit(fw), co = pc.co;
    const bool any = *any64 != 0;
    for (int q = threadIdx.x; q < 3 * nt; q += kDfThreads) {
        const int c = q / nt, tt = q - c * nt, it = tb + tt, part = tt / tp.R, t0 = tt - part * tp.R;
        double v = 0.0;
        for (int gg = 0; gg < G; ++gg) v += sU[(3 * part + c) * kDfThreads + t0 + gg * tp.R];
        double u = unit * v;
        if (any)
            for (int gg = 0; gg < G; ++gg) u += sD[3 * (part * kDfThreads + t0 + gg * tp.R) + c];
        out[3 * size_t(it) + c] = u + (add_self ? co * fs[c * n + it] : 0.0);
    }
}

// ---------------------------------------------------------------- FP32 form
constexpr int kP32Threads = 256;
constexpr int kP32Chunk = 1024;    // sources staged per pass at most
constexpr int kP32List = 256;      // list boxes per prefix segment
constexpr int kP32Block = 32;      // source pairs per plain FP32 block (terms per lane) between Kahan merges

struct P32Const {
    float a2x4, tiny2, k23, nk2;
    float co_cf, nco_c9, co_c3;   // co_cf = (s/(6 pi a)) / (s/(8 pi)), c9 = 9/(32 a), c3 = 3/(32 a)
};

// Sorted positions as hi + lo floats (x = hi + lo to ~2^-48 relative), so that
// coordinates relative to a leaf centre are formed in FP32 as
// (x_hi - c_hi) + (x_lo - c_lo) with the accuracy of one FP32 rounding of the
// difference; no FP64 work remains in the near-field staging.
__global__ void k_split_f32(const double *pos, int64_t n3, float *p32) {
    int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n3) return;
    double x = pos[i];
    float hi = float(x);
    p32[i] = hi;
    p32[n3 + i] = float(x - double(hi));
}

int split_positions_f32(Tree &t, cudaStream_t st) {
    int64_t n3 = 3 * t.n;
    k_split_f32<<<unsigned((n3 + 255) / 256), 256, 0, st>>>(t.pos, n3, t.p32);
    RPY_LAUNCHED(1);
    RPY_CHECK(cudaGetLastError());
    return RPY_OK;
}

// FP64 pair for beads within 1e-3 a of each other (where the FP32 difference of
// coordinates loses the direction), from the FP64 positions.
__device__ __forceinline__ void pair_tiny64(int jg, int i, double a, double co, const double *pos, const double *fs,
                                            int64_t n, double *acc) {
    double ddx = pos[i] - pos[jg], ddy = pos[n + i] - pos[n + jg], ddz = pos[2 * n + i] - pos[2 * n + jg];
    overlap_pair(ddx, ddy, ddz, ddx * ddx + ddy * ddy + ddz * ddz, fs[jg], fs[n + jg], fs[2 * n + jg], a, co, acc);
}

// One pair, both branches without divergence, in units of s/(8 pi), with
// ri = 1/max(r, 1e-3 a):
//   r >= 2a          :  t1 = ri + k23 ri^3,      c = ri^3 (1 - 2a^2 ri^2)
//   1e-3 a < r < 2a  :  t1 = co_cf (1 - c9 r),   c = co_cf c3 ri
//   r <= 1e-3 a      :  t1 = c = 0  (the self pair; other such pairs are taken in FP64)
//   u += t1 F + c (R.F) R
__device__ __forceinline__ void pair32(float dx, float dy, float dz, float r2, float fx, float fy, float fz,
                                       const P32Const &k, float &px, float &py, float &pz) {
    const float ri = rsqrt_ftz(fmaxf(r2, k.tiny2));
    const float ri2 = ri * ri;
    const float B = ri * ri2;
    const bool far = r2 >= k.a2x4, on = r2 > k.tiny2;
    float t1 = far ? fmaf(k.k23, B, ri) : fmaf(k.nco_c9, r2 * ri, k.co_cf);
    float c = far ? B * fmaf(k.nk2, ri2, 1.0f) : k.co_c3 * ri;
    t1 = on ? t1 : 0.0f;
    c = on ? c : 0.0f;
    const float t2 = c * fmaf(dz, fz, fmaf(dy, fy, dx * fx));
    px = fmaf(t2, dx, fmaf(t1, fx, px));
    py = fmaf(t2, dy, fmaf(t1, fy, py));
    pz = fmaf(t2, dz, fmaf(t1, fz, pz));
}

// Packed forms over a pair of staged sources (lanes .x and .y) and the thread's target.
// x - x_j is formed as x + (-x_j), which rounds as the difference does.
__device__ __forceinline__ float2 packed_r2(float2 DX, float2 DY, float2 DZ) {
    return __ffma2_rn(DZ, DZ, __ffma2_rn(DY, DY, __fmul2_rn(DX, DX)));
}

// The r >= 2a branch of pair32 on both lanes, for pairs known to be far (the clamp and the selects of pair32
// are then the identity): the same operations in the same order, hence the same rounding lane by lane.
__device__ __forceinline__ void far_packed(float2 DX, float2 DY, float2 DZ, float2 RI, float2 FX, float2 FY,
                                           float2 FZ, float2 K23, float2 NK2, float2 &AX, float2 &AY, float2 &AZ) {
    const float2 RI2 = __fmul2_rn(RI, RI);
    const float2 B = __fmul2_rn(RI, RI2);
    const float2 T1 = __ffma2_rn(K23, B, RI);
    const float2 C = __fmul2_rn(B, __ffma2_rn(NK2, RI2, make_float2(1.f, 1.f)));
    const float2 T2 = __fmul2_rn(C, __ffma2_rn(DZ, FZ, __ffma2_rn(DY, FY, __fmul2_rn(DX, FX))));
    AX = __ffma2_rn(T2, DX, __ffma2_rn(T1, FX, AX));
    AY = __ffma2_rn(T2, DY, __ffma2_rn(T1, FY, AY));
    AZ = __ffma2_rn(T2, DZ, __ffma2_rn(T1, FZ, AZ));
}
__device__ __forceinline__ float2 rsqrt2(float2 r2) { return make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y)); }

__device__ __forceinline__ void kahan_merge(float &s, float &c, float v) {
    float y = v - c;
    float t = s + y;
    c = (t - s) - y;
    s = t;
}

// An item of T targets uses G = blockDim / T groups of T threads, one target each; the list's beads are staged
// as pairs and group g takes every G-th pair, two pairs (four sources) per iteration.  The list's boxes are
// prefix-summed in shared memory and each staged bead finds its box by binary search.  Chunks are of equal size.
// A vote picks the form of each iteration: all pairs of the warp far (the packed far branch alone), otherwise
// both branches with selects.
// Bound by the FP32 FMA pipe (63% busy) and the issue slots.  Sources rather than targets in the two lanes: half the
// staging memory per source, so chunks of 1,024 instead of 512, and half the running sums; 15M-bead cube
// 22.25 -> 22.1 ms, 256 systems 29.2 -> 28.5, noise 50k 0.071 -> 0.064.  Items that carry their box and target range: 22.0.  A third form for iterations that are far but for
// self pairs (1 in 27 on a uniform system, with 1/r = 0 there) was no faster: 22.2 and 29.2 ms.
constexpr int kP32Queue = 256;   // FP64 pairs of one staged chunk handled after its FP32 loop
constexpr size_t kP32Smem = sizeof(float4) * 3 * (kP32Chunk / 2) + sizeof(float2) * 3 * kP32Threads +
                            sizeof(double) * 3 * kP32Threads + sizeof(int) * kP32Chunk +
                            sizeof(int) * (2 * kP32List + 2) + sizeof(float) * 6 + sizeof(int) * (kP32Queue + 2);

__global__ void __launch_bounds__(kP32Threads, 4) k_p2p32(const int4 *items, const int *beg,
                                                         const int *end,
                                                         const int *bsys, const double *ctr, const int *uoff,
                                                         const int *uidx, const float *p32, const float *f32,
                                                         const double *pos, const double *fs, int64_t n, SysConst sc,
                                                         int add_self, double *out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // staged pair e, relative to the target leaf centre: sS[3e] = (-x, -x', -y, -y'),
    // sS[3e+1] = (-z, -z', fx, fx'), sS[3e+2] = (fy, fy', fz, fz')
    float4 *sS = reinterpret_cast<float4 *>(smem_raw);
    float2 *sK = reinterpret_cast<float2 *>(sS + 3 * (kP32Chunk / 2));   // [3][kP32Threads] Kahan states (S, C)
    double *sD = reinterpret_cast<double *>(sK + 3 * kP32Threads);       // [kP32Threads][3] FP64 pairs
    int *sJ = reinterpret_cast<int *>(sD + 3 * kP32Threads);
    int *lb = sJ + kP32Chunk, *lpre = lb + kP32List;
    float *sCtr = reinterpret_cast<float *>(lpre + kP32List + 2);   // target leaf centre, hi and lo floats
    int *sQn = reinterpret_cast<int *>(sCtr + 6);   // [0] queue length, [1] any FP64 pair of this item
    int *sQ = sQn + 2;                              // queued pairs: thread << 11 | source slot
    const int4 item = items[blockIdx.x];
    const int li = item.x, b = item.y, sys = bsys[b];
    const PairConst &pc = sc.pc[sys];
    const double a = pc.a, cf = pc.cf, co = pc.co;
    P32Const k;
    k.a2x4 = pc.f_a2x4;
    k.tiny2 = pc.f_tiny2;
    k.k23 = pc.f_k23;
    k.nk2 = pc.f_nk2;
    k.co_cf = pc.f_co_cf;
    k.nco_c9 = pc.f_nco_c9;
    k.co_c3 = pc.f_co_c3;
    if (threadIdx.x < 3) {
        const double c = ctr[3 * b + threadIdx.x];
        const float h = float(c);
        sCtr[threadIdx.x] = h;
        sCtr[3 + threadIdx.x] = float(c - double(h));
    }
    if (threadIdx.x == 0) sQn[0] = sQn[1] = 0;
    __syncthreads();
    const float chx = sCtr[0], chy = sCtr[1], chz = sCtr[2], clx = sCtr[3], cly = sCtr[4], clz = sCtr[5];
    const float *xh = p32, *yh = p32 + n, *zh = p32 + 2 * n, *xl = p32 + 3 * n, *yl = p32 + 4 * n, *zl = p32 + 5 * n;
    const float2 K23 = make_float2(k.k23, k.k23), NK2 = make_float2(k.nk2, k.nk2);
    const int u0 = uoff[li], u1 = uoff[li + 1];
    const int tb = item.z, te = item.w, nt = te - tb;
    const int G = kP32Threads / nt;
    const int tl = threadIdx.x % nt, g = threadIdx.x / nt;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = tb + tl;
    const bool act = g < G;
    const float xa = (xh[i] - chx) + (xl[i] - clx), ya = (yh[i] - chy) + (yl[i] - cly), za = (zh[i] - chz) + (zl[i] - clz);
    const float2 X = make_float2(xa, xa), Y = make_float2(ya, ya), Z = make_float2(za, za);
    for (int c = 0; c < 3; ++c) {
        sK[c * kP32Threads + threadIdx.x] = make_float2(0.f, 0.f);
        sD[3 * threadIdx.x + c] = 0.0;
    }
    for (int us = u0; us < u1; us += kP32List) {
        const int L = min(kP32List, u1 - us);
        __syncthreads();
        // prefix of the box sizes of this list segment (warp 0)
        if (warp == 0) {
            int carry = 0;
            for (int q0 = 0; q0 < L; q0 += 32) {
                int q = q0 + lane, cnt = 0;
                if (q < L) {
                    int C = uidx[us + q];
                    lb[q] = beg[C];
                    cnt = end[C] - beg[C];
                }
                int v = cnt;
                for (int o = 1; o < 32; o <<= 1) {
                    int w = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += w;
                }
                if (q < L) lpre[q + 1] = carry + v;
                carry += __shfl_sync(0xffffffffu, v, 31);
            }
            if (lane == 0) lpre[0] = 0;
        }
        __syncthreads();
        const int Ns = lpre[L];
        const int nch = (Ns + kP32Chunk - 1) / kP32Chunk;
        const int csz = nch ? ((Ns + nch - 1) / nch + 1) & ~1 : 2;   // equal chunks of whole pairs
        for (int c0 = 0; c0 < Ns; c0 += csz) {
            const int nS = min(csz, Ns - c0), nP = (nS + 1) >> 1;
            // no barrier here: the one after the prefix (first chunk) or after the
            // previous chunk's compute (and its FP64 queue pass) already orders
            // every read of sS and sJ before this chunk's writes
            for (int e = threadIdx.x; e < 2 * nP; e += kP32Threads) {
                float *w = reinterpret_cast<float *>(sS + 3 * (e >> 1)) + (e & 1);
                float px = 1e15f, py = 1e15f, pz = 1e15f, fx = 0.f, fy = 0.f, fz = 0.f;
                int j = -1;   // an odd last source gets a partner without force, not far at every scale of lengths
                if (e < nS) {
                    int q = c0 + e, lo = 0, hi = L;   // box: lpre[lo] <= q < lpre[lo + 1]
                    while (hi - lo > 1) {
                        int mid = (lo + hi) >> 1;
                        if (lpre[mid] <= q) lo = mid;
                        else hi = mid;
                    }
                    j = lb[lo] + (q - lpre[lo]);
                    px = (xh[j] - chx) + (xl[j] - clx);
                    py = (yh[j] - chy) + (yl[j] - cly);
                    pz = (zh[j] - chz) + (zl[j] - clz);
                    fx = f32[j];
                    fy = f32[n + j];
                    fz = f32[2 * n + j];
                }
                w[0] = -px;
                w[2] = -py;
                w[4] = -pz;
                w[6] = fx;
                w[8] = fy;
                w[10] = fz;
                sJ[e] = j;
            }
            __syncthreads();
            if (act) {
                for (int eb = g; eb < nP; eb += kP32Block * G) {
                    const int ee = min(nP, eb + kP32Block * G);
                    float2 AX = make_float2(0.f, 0.f), AY = AX, AZ = AX;   // lane sums of this block
                    // pairs at most 1e-3 a apart other than the self pair and the partner (j < 0): to FP64
                    auto close = [&](int e, float2 R2) {
                        for (int h = 0; h < 2; ++h) {
                            const int j = sJ[2 * e + h];
                            if (!((h ? R2.y : R2.x) > k.tiny2) && j >= 0 && j != i) {
                                const int q = atomicAdd(&sQn[0], 1);
                                if (q < kP32Queue) sQ[q] = (threadIdx.x << 11) | (2 * e + h);
                            }
                        }
                    };
                    // both branches with selects
                    auto slow = [&](int e, float2 DX, float2 DY, float2 DZ, float2 R2, float2 FX, float2 FY, float2 FZ) {
                        pair32(DX.x, DY.x, DZ.x, R2.x, FX.x, FY.x, FZ.x, k, AX.x, AY.x, AZ.x);
                        pair32(DX.y, DY.y, DZ.y, R2.y, FX.y, FY.y, FZ.y, k, AX.y, AY.y, AZ.y);
                        if (!(R2.x > k.tiny2) || !(R2.y > k.tiny2)) close(e, R2);
                    };
                    int e = eb;
                    for (; e + G < ee; e += 2 * G) {
                        const int e1 = e + G;
                        const float4 S0 = sS[3 * e], S1 = sS[3 * e + 1], S2 = sS[3 * e + 2];
                        const float4 U0 = sS[3 * e1], U1 = sS[3 * e1 + 1], U2 = sS[3 * e1 + 2];
                        const float2 DX = __fadd2_rn(X, make_float2(S0.x, S0.y)), DY = __fadd2_rn(Y, make_float2(S0.z, S0.w)),
                                     DZ = __fadd2_rn(Z, make_float2(S1.x, S1.y));
                        const float2 EX = __fadd2_rn(X, make_float2(U0.x, U0.y)), EY = __fadd2_rn(Y, make_float2(U0.z, U0.w)),
                                     EZ = __fadd2_rn(Z, make_float2(U1.x, U1.y));
                        const float2 R2 = packed_r2(DX, DY, DZ), Q2 = packed_r2(EX, EY, EZ);
                        const float2 FX = make_float2(S1.z, S1.w), FY = make_float2(S2.x, S2.y),
                                     FZ = make_float2(S2.z, S2.w);
                        const float2 GX = make_float2(U1.z, U1.w), GY = make_float2(U2.x, U2.y),
                                     GZ = make_float2(U2.z, U2.w);
                        if (__all_sync(__activemask(), fminf(fminf(R2.x, R2.y), fminf(Q2.x, Q2.y)) >= k.a2x4)) {
                            far_packed(DX, DY, DZ, rsqrt2(R2), FX, FY, FZ, K23, NK2, AX, AY, AZ);
                            far_packed(EX, EY, EZ, rsqrt2(Q2), GX, GY, GZ, K23, NK2, AX, AY, AZ);
                        } else {
                            slow(e, DX, DY, DZ, R2, FX, FY, FZ);
                            slow(e1, EX, EY, EZ, Q2, GX, GY, GZ);
                        }
                    }
                    if (e < ee) {
                        const float4 S0 = sS[3 * e], S1 = sS[3 * e + 1], S2 = sS[3 * e + 2];
                        const float2 DX = __fadd2_rn(X, make_float2(S0.x, S0.y)), DY = __fadd2_rn(Y, make_float2(S0.z, S0.w)),
                                     DZ = __fadd2_rn(Z, make_float2(S1.x, S1.y));
                        const float2 R2 = packed_r2(DX, DY, DZ);
                        const float2 FX = make_float2(S1.z, S1.w), FY = make_float2(S2.x, S2.y),
                                     FZ = make_float2(S2.z, S2.w);
                        if (__all_sync(__activemask(), fminf(R2.x, R2.y) >= k.a2x4))
                            far_packed(DX, DY, DZ, rsqrt2(R2), FX, FY, FZ, K23, NK2, AX, AY, AZ);
                        else
                            slow(e, DX, DY, DZ, R2, FX, FY, FZ);
                    }
                    const float Pv[3][2] = {{AX.x, AX.y}, {AY.x, AY.y}, {AZ.x, AZ.y}};
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        float2 kc = sK[c * kP32Threads + threadIdx.x];
                        kahan_merge(kc.x, kc.y, Pv[c][0]);
                        kahan_merge(kc.x, kc.y, Pv[c][1]);
                        sK[c * kP32Threads + threadIdx.x] = kc;
                    }
                }
            }
            __syncthreads();
            const int nq = sQn[0];
            if (nq > 0) {
                // FP64 pairs of this chunk: from the queue, or (queue overflow)
                // by every thread re-scanning its own sources
                if (nq <= kP32Queue) {
                    for (int e = threadIdx.x; e < nq; e += kP32Threads) {
                        const int v = sQ[e], t = v >> 11, jj = v & 2047;
                        double acc[3] = {0, 0, 0};
                        pair_tiny64(sJ[jj], tb + t % nt, a, co, pos, fs, n, acc);
                        for (int c = 0; c < 3; ++c) atomicAdd(&sD[3 * t + c], acc[c]);
                    }
                } else if (act) {
                    for (int e = g; e < nP; e += G) {
                        const float4 S0 = sS[3 * e], S1 = sS[3 * e + 1];
                        for (int h = 0; h < 2; ++h) {
                            const float dx = xa + (h ? S0.y : S0.x), dy = ya + (h ? S0.w : S0.z), dz = za + (h ? S1.y : S1.x);
                            const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                            const int jg = sJ[2 * e + h];
                            if (!(r2 > k.tiny2) && jg >= 0 && jg != i)
                                pair_tiny64(jg, i, a, co, pos, fs, n, &sD[3 * threadIdx.x]);
                        }
                    }
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    sQn[0] = 0;
                    sQn[1] = 1;
                }
            }
        }
    }
    // group reduction: one thread per (component, target) merges the Kahan
    // states (S, C) of the G groups in FP32 (Kahan over the S, plain sum of
    // the small C) and forms the FP64 result once
    __syncthreads();
    const bool tiny = sQn[1] != 0;
    for (int q = threadIdx.x; q < 3 * nt; q += kP32Threads) {
        const int c = q / nt, tt = q - c * nt, it = tb + tt;
        float S = 0.f, C = 0.f, Cs = 0.f;
        for (int gg = 0; gg < G; ++gg) {
            const float2 v = sK[c * kP32Threads + tt + gg * nt];
            kahan_merge(S, C, v.x);
            Cs += v.y;
        }
        double u = cf * (double(S) - (double(C) + double(Cs)));
        if (tiny)
            for (int gg = 0; gg < G; ++gg) u += sD[3 * (tt + gg * nt) + c];
        out[3 * size_t(it) + c] = u + (add_self ? co * fs[c * n + it] : 0.0);
    }
}

// The dynamic shared memory of both near-field kernels exceeds the default 48 KB: raise the
// limit once per device.
static cudaError_t set_near_smem() {
    static std::mutex mu;
    static std::set<int> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done.count(dev)) return cudaSuccess;
    e = cudaFuncSetAttribute(k_p2p32, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kP32Smem));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_p2p_df, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kDfSmem));
    if (e == cudaSuccess) done.insert(dev);
    return e;
}

// U lists (near field, self term added), the direct substitutes of small
// W / X interactions (no self term), or both in one pass (the full matvec).
int run_p2p(Tree &t, const double *fs, double *out, const SysConst &sc, cudaStream_t st, int list) {
    const bool direct_list = list == kListD, merged = list == kListM;
    const int *off = merged ? t.m_off : (direct_list ? t.d_off : t.u_off);
    const int *idx = merged ? t.m_idx : (direct_list ? t.d_idx : t.u_idx);
    int add_self = direct_list ? 0 : 1;
    const int4 *items = merged ? t.m_items : (direct_list ? t.d_items : t.u_items);
    if (t.n_items == 0) return RPY_OK;
    RPY_CHECK(set_near_smem());
    if (t.params.precision == RPY_FP32) {
        k_p2p32<<<t.n_items, kP32Threads, kP32Smem, st>>>(items, t.b_begin, t.b_end, t.b_sys, t.b_center,
                                                          off, idx, t.p32, t.f32, t.pos, fs, t.n, sc, add_self, out);
        RPY_LAUNCHED(1);
    } else {
        k_p2p_df<<<t.n_items, kDfThreads, kDfSmem, st>>>(items, t.b_begin, t.b_end, t.b_sys, t.b_level, off,
                                                         idx, t.p3, t.f2, t.sys_fmax, t.pos, fs, t.n, sc, add_self,
                                                         out);
        RPY_LAUNCHED(1);
    }
    RPY_CHECK(cudaGetLastError());
    return RPY_OK;
}

}  // namespace rpy
