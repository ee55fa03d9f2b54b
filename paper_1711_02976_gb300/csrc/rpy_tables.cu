// Host construction of the FMM operator tables for one (p, digits) setting.
//
// All expansions are stored in box units: for a box of side h and centre c,
//   multipole  phi(x) = (1/h) sum_{n,m} M_n^m z_n^m((x - c)/h),
//   local      phi(x) = (1/h) sum_{n,m} L_n^m y_n^m((x - c)/h),
// so every operator below is independent of the level (Sec. 2 expansion
// forms; the scaling is this library's choice).
//
// Tables:
//   M2M / L2L   rotations to the shift axis and z shifts; for the host tests also
//               dense real matrices per child octant, built from the
//               addition theorem of regular solid harmonics
//               R_n^m(u + v) = sum_{k,l} R_k^l(u) R_{n-k}^{m-l}(v),
//               R_n^m = r^n P_n^m e^{i m phi} / (n+m)!, which in the paper's
//               normalisation reads y_n^m(u+v) = sum G_{nm,kl}(v) y_k^l(u).
//   rotations   Y_n^m(A w) = sum_m' K_{m m'} Y_n^m'(w) for the two coordinate
//               frames whose z axis is world x or world y, computed by exact
//               quadrature on the sphere.
//   plane waves the quadrature of gen_exp_quadrature.py; M2X coefficients
//               lambda^n / sqrt((n-m)!(n+m)!), X2L coefficients
//               (-lambda)^n / sqrt((n-m)!(n+m)!), and the diagonal shift
//               factors e^{-lambda dz + i lambda (dx cos a + dy sin a)}.
//   groups      merge-and-shift bookkeeping: which children of a parent's
//               colleagues feed which children of the parent, per direction.
#include <cmath>
#include <mutex>
#include <complex>
#include <cstring>
#include <map>

#include "exp_quadrature.h"
#include "rpy_harmonics.h"

namespace rpy {

using cd = std::complex<double>;

static std::vector<double> g_fact;   // n! for n <= 4 kMaxP + 8

static double fact(int n) {
    if (g_fact.empty()) {
        g_fact.resize(4 * kMaxP + 9);
        g_fact[0] = 1.0;
        for (size_t i = 1; i < g_fact.size(); ++i) g_fact[i] = g_fact[i - 1] * double(i);
    }
    return g_fact[n];
}

static double Nnm(int n, int m) {   // sqrt((n+|m|)!(n-|m|)!)
    int am = m < 0 ? -m : m;
    return std::sqrt(fact(n + am) * fact(n - am));
}

static double sgn_m(int m) { return (m >= 0 || ((-m) % 2 == 0)) ? 1.0 : -1.0; }

// y_n^m(v) for all n <= p, m in [-n, n] (complex, full range).
static void regular_full(const double v[3], int p, std::vector<cd> &out) {
    HarmRec h = harm_rec(p);
    std::vector<cpx<double>> tmp(ncoef(p));
    regular_all<double>(v[0], v[1], v[2], p, h.a.data(), h.b.data(), h.c.data(), tmp.data());
    out.assign((p + 1) * (p + 1), cd(0, 0));
    for (int n = 0; n <= p; ++n)
        for (int m = 0; m <= n; ++m) {
            cd y(tmp[tri(n, m)].x, tmp[tri(n, m)].y);
            out[n * n + n + m] = y;
            out[n * n + n - m] = std::conj(y);
        }
}

// G_{nm,kl}(v): y_n^m(u + v) = sum_{k<=n,l} G y_k^l(u).
struct AddTheorem {
    int p;
    std::vector<cd> yv;   // y_j^q(v), full
    AddTheorem(int p_, const double v[3]) : p(p_) { regular_full(v, p_, yv); }
    cd R(int j, int q) const {   // R_j^q(v) = y_j^q / (s_q N_j^q)
        if (q > j || -q > j) return cd(0, 0);
        return yv[j * j + j + q] / (sgn_m(q) * Nnm(j, q));
    }
    cd G(int n, int m, int k, int l) const {
        if (k > n) return cd(0, 0);
        return (sgn_m(m) * Nnm(n, m) / (sgn_m(l) * Nnm(k, l))) * R(n - k, m - l);
    }
};

// Accumulate coefficient c * X^{(k,l)} into output (n, m>=0), real 2-layout.
// X^{(k,l)} = X_k^|l| for l >= 0, conj(X_k^|l|) for l < 0.
static void add_real(std::vector<double> &Tt, int D, int out_n, int out_m, int in_k, int in_l, cd c) {
    int ro = 2 * tri(out_n, out_m);
    int ci = 2 * tri(in_k, in_l < 0 ? -in_l : in_l);
    double cr = c.real(), cim = c.imag();
    double s = in_l < 0 ? -1.0 : 1.0;
    // out_re += cr xr - s ci xi ; out_im += ci xr + s cr xi   (stored transposed [in][out])
    Tt[size_t(ci) * D + ro] += cr;
    Tt[size_t(ci + 1) * D + ro] += -s * cim;
    Tt[size_t(ci) * D + ro + 1] += cim;
    Tt[size_t(ci + 1) * D + ro + 1] += s * cr;
}

static void octant_delta(int o, double d[3]) {
    for (int a = 0; a < 3; ++a) d[a] = ((o >> a) & 1) ? 0.25 : -0.25;
}

static void build_m2m(int p, std::vector<double> &out) {
    int nc = ncoef(p), D = 2 * nc;
    out.assign(size_t(8) * D * D, 0.0);
    for (int o = 0; o < 8; ++o) {
        double d[3];
        octant_delta(o, d);
        AddTheorem at(p, d);
        std::vector<double> Tt(size_t(D) * D, 0.0);
        // M^p_n^m = sum_{k<=n,l} conj(G_{nm,kl}(d)) 2^{-k} M^c_k^l
        for (int n = 0; n <= p; ++n)
            for (int m = 0; m <= n; ++m)
                for (int k = 0; k <= n; ++k)
                    for (int l = -k; l <= k; ++l) {
                        cd g = at.G(n, m, k, l);
                        if (g == cd(0, 0)) continue;
                        add_real(Tt, D, n, m, k, l, std::conj(g) * std::ldexp(1.0, -k));
                    }
        std::memcpy(&out[size_t(o) * D * D], Tt.data(), sizeof(double) * D * D);
    }
}

static void build_l2l(int p, std::vector<double> &out) {
    int nc = ncoef(p), D = 2 * nc;
    out.assign(size_t(8) * D * D, 0.0);
    for (int o = 0; o < 8; ++o) {
        double d[3];
        octant_delta(o, d);
        AddTheorem at(p, d);
        std::vector<double> Tt(size_t(D) * D, 0.0);
        // L^c_k^l = 2^{-k-1} sum_{n>=k, m} L^p_n^m G_{nm,kl}(d)
        for (int k = 0; k <= p; ++k)
            for (int l = 0; l <= k; ++l)
                for (int n = k; n <= p; ++n)
                    for (int m = -n; m <= n; ++m) {
                        cd g = at.G(n, m, k, l);
                        if (g == cd(0, 0)) continue;
                        add_real(Tt, D, k, l, n, m, g * std::ldexp(1.0, -k - 1));
                    }
        std::memcpy(&out[size_t(o) * D * D], Tt.data(), sizeof(double) * D * D);
    }
}

// Gauss-Legendre nodes on [-1, 1] (Newton on P_n).
static void legendre_pd(int n, double z, double &p, double &dp) {
    double p0 = 1.0, p1 = 0.0;
    for (int j = 1; j <= n; ++j) {
        double p2 = p1;
        p1 = p0;
        p0 = ((2.0 * j - 1.0) * z * p1 - (j - 1.0) * p2) / j;
    }
    p = p0;
    dp = n * (z * p0 - p1) / (z * z - 1.0);
}

static void gauss_legendre(int n, std::vector<double> &x, std::vector<double> &w) {
    x.resize(n);
    w.resize(n);
    for (int i = 0; i < n; ++i) {
        double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), p = 0.0, dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            legendre_pd(n, z, p, dp);
            double dz = p / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        legendre_pd(n, z, p, dp);
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// K_{m m'} with Y_n^m(A w) = sum_{m'} K_{m m'} Y_n^{m'}(w), all m, m' in [-n, n].
static std::vector<cd> rotmat(const double A[9], int n) {
    int dim = 2 * n + 1;
    std::vector<cd> K(size_t(dim) * dim, cd(0, 0));
    std::vector<double> gx, gw;
    gauss_legendre(n + 1, gx, gw);
    int nphi = 2 * n + 2;
    std::vector<cd> ya, yw;
    for (size_t i = 0; i < gx.size(); ++i) {
        double ct = gx[i], st = std::sqrt(std::max(0.0, 1.0 - ct * ct));
        for (int j = 0; j < nphi; ++j) {
            double ph = 2.0 * M_PI * j / nphi;
            double w[3] = {st * std::cos(ph), st * std::sin(ph), ct};
            double aw[3] = {A[0] * w[0] + A[1] * w[1] + A[2] * w[2], A[3] * w[0] + A[4] * w[1] + A[5] * w[2],
                            A[6] * w[0] + A[7] * w[1] + A[8] * w[2]};
            regular_full(aw, n, ya);
            regular_full(w, n, yw);
            double wt = gw[i] * 2.0 * M_PI / nphi * (2.0 * n + 1.0) / (4.0 * M_PI);
            for (int m = -n; m <= n; ++m)
                for (int mp = -n; mp <= n; ++mp)
                    K[size_t(m + n) * dim + (mp + n)] += wt * ya[n * n + n + m] * std::conj(yw[n * n + n + mp]);
        }
    }
    return K;
}

// Frame matrices (rows = frame axes in world coordinates).
static const double kQx[9] = {0, 1, 0, 0, 0, 1, 1, 0, 0};   // x'=y, y'=z, z'=x
static const double kQy[9] = {0, 0, 1, 1, 0, 0, 0, 1, 0};   // x'=z, y'=x, z'=y

static void transpose3(const double A[9], double B[9]) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) B[3 * i + j] = A[3 * j + i];
}

// Real per-degree blocks, layout [off_n + out*(2(n+1)) + in], 2-real local index 2m+part.
static void rotation_offsets(int p, std::vector<int> &off) {
    off.resize(p + 2);
    off[0] = 0;
    for (int n = 0; n <= p; ++n) off[n + 1] = off[n] + 4 * (n + 1) * (n + 1);
}
static void build_rotations(int p, std::vector<double> &fwd, std::vector<double> &bwd, std::vector<int> &off) {
    rotation_offsets(p, off);
    fwd.assign(size_t(2) * off[p + 1], 0.0);
    bwd.assign(size_t(2) * off[p + 1], 0.0);
    for (int f = 0; f < 2; ++f) {
        const double *Q = f == 0 ? kQx : kQy;
        double Qt[9];
        transpose3(Q, Qt);
        for (int n = 0; n <= p; ++n) {
            int B = 2 * (n + 1), dim = 2 * n + 1;
            std::vector<cd> D = rotmat(Qt, n);   // forward: M'_{m'} = sum_m M_m D_{m m'}
            std::vector<cd> K = rotmat(Q, n);    // backward: L_m = sum_{m'} L'_{m'} K_{m' m}
            double *F = &fwd[size_t(f) * off[p + 1] + off[n]];
            double *Bk = &bwd[size_t(f) * off[p + 1] + off[n]];
            for (int mo = 0; mo <= n; ++mo)
                for (int mi = -n; mi <= n; ++mi) {
                    cd cf = D[size_t(mi + n) * dim + (mo + n)];
                    cd cb = K[size_t(mi + n) * dim + (mo + n)];
                    int ro = 2 * mo, ci = 2 * (mi < 0 ? -mi : mi);
                    double s = mi < 0 ? -1.0 : 1.0;
                    F[ro * B + ci] += cf.real();
                    F[ro * B + ci + 1] += -s * cf.imag();
                    F[(ro + 1) * B + ci] += cf.imag();
                    F[(ro + 1) * B + ci + 1] += s * cf.real();
                    Bk[ro * B + ci] += cb.real();
                    Bk[ro * B + ci + 1] += -s * cb.imag();
                    Bk[(ro + 1) * B + ci] += cb.imag();
                    Bk[(ro + 1) * B + ci + 1] += s * cb.real();
                }
            // clean round-off of exact zeros / ones
            for (int i = 0; i < B * B; ++i) {
                if (std::fabs(F[i]) < 1e-15) F[i] = 0.0;
                if (std::fabs(Bk[i]) < 1e-15) Bk[i] = 0.0;
            }
        }
    }
}

// Per child octant: rotation whose third row (the frame's z axis) is the unit
// shift direction from the parent centre to the child centre.
static void octant_frame(int o, double Q[9]) {
    double sx = (o & 1) ? 1.0 : -1.0, sy = (o & 2) ? 1.0 : -1.0, sz = (o & 4) ? 1.0 : -1.0;
    double r3 = 1.0 / std::sqrt(3.0), r2 = 1.0 / std::sqrt(2.0);
    double z[3] = {sx * r3, sy * r3, sz * r3};
    double x[3] = {-sy * r2, sx * r2, 0.0};
    double y[3] = {z[1] * x[2] - z[2] * x[1], z[2] * x[0] - z[0] * x[2], z[0] * x[1] - z[1] * x[0]};
    for (int a = 0; a < 3; ++a) {
        Q[a] = x[a];
        Q[3 + a] = y[a];
        Q[6 + a] = z[a];
    }
}

// Real per-degree blocks for an arbitrary rotation Q (frame = Q world), written
// at fwd / bwd in the layout of build_rotations.
static void rotation_blocks(const double Q[9], int p, const std::vector<int> &off, double *F, double *Bk) {
    double Qt[9];
    transpose3(Q, Qt);
    for (int n = 0; n <= p; ++n) {
        int B = 2 * (n + 1), dim = 2 * n + 1;
        std::vector<cd> D = rotmat(Qt, n);
        std::vector<cd> K = rotmat(Q, n);
        double *f = F + off[n], *bk = Bk + off[n];
        for (int i = 0; i < B * B; ++i) f[i] = bk[i] = 0.0;
        for (int mo = 0; mo <= n; ++mo)
            for (int mi = -n; mi <= n; ++mi) {
                cd cf = D[size_t(mi + n) * dim + (mo + n)];
                cd cb = K[size_t(mi + n) * dim + (mo + n)];
                int ro = 2 * mo, ci = 2 * (mi < 0 ? -mi : mi);
                double s = mi < 0 ? -1.0 : 1.0;
                f[ro * B + ci] += cf.real();
                f[ro * B + ci + 1] += -s * cf.imag();
                f[(ro + 1) * B + ci] += cf.imag();
                f[(ro + 1) * B + ci + 1] += s * cf.real();
                bk[ro * B + ci] += cb.real();
                bk[ro * B + ci + 1] += -s * cb.imag();
                bk[(ro + 1) * B + ci] += cb.imag();
                bk[(ro + 1) * B + ci + 1] += s * cb.real();
            }
    }
}

// ---------------------------------------------------------------- factorized rotations
// A rotation of the expansion coefficients of degree n, in the real block form
// above (F[out][in], 2-real index 2m + part), factors through the z-y-z Euler
// angles of its 3x3 matrix X = Rz(a) Ry(b) Rz(c) as F(X) = F(Rz(c)) F(Ry(b)) F(Rz(a)):
// the two z rotations are one 2x2 rotation per m, and the y rotation maps real
// parts to real parts and imaginary parts to imaginary parts (its Wigner matrix is
// real), so applying F costs 2(n+1)^2 + 8(n+1) FMAs instead of 4(n+1)^2.
// Layout per degree n at foff[n]: [za: (c, s) per m][zc: (c, s) per m]
// [Yre: (n+1) x (n+1)][Yim: (n+1) x (n+1)], applied as za, then Y, then zc.

// F(X) for degree n, as rotation_blocks builds it from rotmat(X).
static std::vector<double> fold_block(const double X[9], int n) {
    const int B = 2 * (n + 1), dim = 2 * n + 1;
    std::vector<cd> D = rotmat(X, n);
    std::vector<double> F(size_t(B) * B, 0.0);
    for (int mo = 0; mo <= n; ++mo)
        for (int mi = -n; mi <= n; ++mi) {
            cd c = D[size_t(mi + n) * dim + (mo + n)];
            int ro = 2 * mo, ci = 2 * (mi < 0 ? -mi : mi);
            double sg = mi < 0 ? -1.0 : 1.0;
            F[ro * B + ci] += c.real();
            F[ro * B + ci + 1] += -sg * c.imag();
            F[(ro + 1) * B + ci] += c.imag();
            F[(ro + 1) * B + ci + 1] += sg * c.real();
        }
    return F;
}

static void rot_z(double a, double R[9]) {
    const double c = std::cos(a), s = std::sin(a);
    const double M[9] = {c, -s, 0, s, c, 0, 0, 0, 1};
    for (int i = 0; i < 9; ++i) R[i] = M[i];
}
static void rot_y(double b, double R[9]) {
    const double c = std::cos(b), s = std::sin(b);
    const double M[9] = {c, 0, s, 0, 1, 0, -s, 0, c};
    for (int i = 0; i < 9; ++i) R[i] = M[i];
}

int factor_len(int n) { return 4 * (n + 1) + 2 * (n + 1) * (n + 1); }

// Fills `out` (layout above) for the rotation X; false if a factor does not have the
// expected structure.  With `quarter` (the
// frame rotations, whose middle angle is pi/2) the y blocks must also have the
// checkerboard structure the kernels rely on: Yre[mo][mi] = 0 unless mo + mi + n
// is even, Yim[mo][mi] = 0 unless mo + mi + n is odd (rows and columns m >= 1;
// the m = 0 imaginary parts of real fields vanish).
static bool factor_rotation(const double X[9], int p, const std::vector<int> &foff, double *out,
                            bool quarter = false) {
    // X = Rz(a) Ry(b) Rz(c): X22 = cos b, X02 = cos a sin b, X12 = sin a sin b,
    // X20 = -sin b cos c, X21 = sin b sin c
    const double b = std::acos(std::max(-1.0, std::min(1.0, X[8])));
    double a, c;
    if (std::fabs(std::sin(b)) > 1e-12) {
        a = std::atan2(X[5], X[2]);
        c = std::atan2(X[7], -X[6]);
    } else {   // b = 0 or pi: only a +- c is defined
        a = std::atan2(X[3], X[0]);
        c = 0.0;
    }
    double Za[9], Yb[9], Zc[9];
    rot_z(a, Za);
    rot_y(b, Yb);
    rot_z(c, Zc);
    for (int n = 0; n <= p; ++n) {
        const int B = 2 * (n + 1), q = n + 1;
        std::vector<double> F = fold_block(X, n), FA = fold_block(Za, n), FY = fold_block(Yb, n),
                            FC = fold_block(Zc, n);
        // F must equal FC FY FA
        std::vector<double> T(size_t(B) * B, 0.0), U(size_t(B) * B, 0.0);
        for (int i = 0; i < B; ++i)
            for (int k = 0; k < B; ++k)
                for (int j = 0; j < B; ++j) T[i * B + j] += FY[i * B + k] * FA[k * B + j];
        for (int i = 0; i < B; ++i)
            for (int k = 0; k < B; ++k)
                for (int j = 0; j < B; ++j) U[i * B + j] += FC[i * B + k] * T[k * B + j];
        double err = 0.0;
        for (int i = 0; i < B * B; ++i) err = std::max(err, std::fabs(U[i] - F[i]));
        if (err > 1e-11) return false;
        double *o = out + foff[n];
        for (int m = 0; m <= n; ++m) {
            const int r = 2 * m;
            // z rotations: [[c, -s], [s, c]] on (Re, Im) of coefficient m, zero elsewhere
            if (std::fabs(FA[r * B + r] - FA[(r + 1) * B + r + 1]) > 1e-12 ||
                std::fabs(FA[r * B + r + 1] + FA[(r + 1) * B + r]) > 1e-12 ||
                std::fabs(FC[r * B + r] - FC[(r + 1) * B + r + 1]) > 1e-12 ||
                std::fabs(FC[r * B + r + 1] + FC[(r + 1) * B + r]) > 1e-12)
                return false;
            o[2 * m] = FA[r * B + r];
            o[2 * m + 1] = FA[(r + 1) * B + r];
            o[2 * q + 2 * m] = FC[r * B + r];
            o[2 * q + 2 * m + 1] = FC[(r + 1) * B + r];
        }
        double *yre = o + 4 * q, *yim = yre + q * q;
        for (int mo = 0; mo <= n; ++mo)
            for (int mi = 0; mi <= n; ++mi) {
                if (std::fabs(FY[(2 * mo) * B + 2 * mi + 1]) > 1e-12 || std::fabs(FY[(2 * mo + 1) * B + 2 * mi]) > 1e-12)
                    return false;
                yre[mo * q + mi] = FY[(2 * mo) * B + 2 * mi];
                yim[mo * q + mi] = FY[(2 * mo + 1) * B + 2 * mi + 1];
            }
        if (quarter)
            for (int mo = 0; mo <= n; ++mo)
                for (int mi = 0; mi <= n; ++mi) {
                    const bool even = ((mo + mi + n) & 1) == 0;
                    if (!even && std::fabs(yre[mo * q + mi]) > 1e-13) return false;
                    if (mo > 0 && mi > 0 && even && std::fabs(yim[mo * q + mi]) > 1e-13) return false;
                    if (mo == 0 && mi > 0 && std::fabs(yim[mi]) > 1e-13) return false;
                }
    }
    return true;
}

// signed-permutation frame matrices P_d for the six directions
static void frame_matrix(int d, int P[9]) {
    static const int Pz[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
    static const int Px[9] = {0, 1, 0, 0, 0, 1, 1, 0, 0};
    static const int Py[9] = {0, 0, 1, 1, 0, 0, 0, 1, 0};
    const int *B = d < 2 ? Pz : (d < 4 ? Px : Py);
    for (int i = 0; i < 9; ++i) P[i] = B[i];
    if (d & 1)
        for (int j = 0; j < 3; ++j) P[6 + j] = -P[6 + j];
}

// direction of a (target - source) centre offset in child units, or -1 if adjacent
static int classify(const int D2[3]) {   // D2 = 2 * offset (integers)
    if (D2[2] >= 4) return 0;
    if (D2[2] <= -4) return 1;
    if (D2[1] >= 4) return 4;
    if (D2[1] <= -4) return 5;
    if (D2[0] >= 4) return 2;
    if (D2[0] <= -4) return 3;
    return -1;
}

static int shift_index(const int v2[3]) {   // v2 = 2 * half-integer offset in [-5, 5]
    int ix = (v2[0] + 5) / 2, iy = (v2[1] + 5) / 2, iz = (v2[2] + 5) / 2;
    return ix + 6 * iy + 36 * iz;
}

static void build_groups(OpTables &t) {
    t.grp_off.assign(kDirs * (kGroupMax + 1), 0);
    t.grp_n.assign(kDirs, 0);
    t.grp_mask.assign(kDirs * kGroupMax, 0);
    t.slot_list.assign(kDirs * 216, -1);
    t.child_shift.assign(kDirs * 8, 0);
    for (int d = 0; d < kDirs; ++d) {
        int P[9];
        frame_matrix(d, P);
        std::map<int, std::vector<int>> by_mask;
        for (int q = 0; q < 27; ++q) {
            int dq[3] = {q % 3 - 1, (q / 3) % 3 - 1, q / 9 - 1};
            for (int o = 0; o < 8; ++o) {
                int s2[3];   // 2 * source centre relative to parent centre, child units
                for (int a = 0; a < 3; ++a) s2[a] = 4 * dq[a] + (((o >> a) & 1) ? 1 : -1);
                int mask = 0;
                for (int tt = 0; tt < 8; ++tt) {
                    int D2[3];
                    for (int a = 0; a < 3; ++a) D2[a] = (((tt >> a) & 1) ? 1 : -1) - s2[a];
                    if (classify(D2) == d) mask |= 1 << tt;
                }
                if (!mask) continue;
                int v2[3];   // frame offset parent - source = P (-s)
                for (int i = 0; i < 3; ++i) v2[i] = -(P[3 * i] * s2[0] + P[3 * i + 1] * s2[1] + P[3 * i + 2] * s2[2]);
                by_mask[mask].push_back((q * 8 + o) | (shift_index(v2) << 8));
            }
        }
        int g = 0, pos = 0;
        for (auto &kv : by_mask) {
            t.grp_mask[d * kGroupMax + g] = kv.first;
            t.grp_off[d * (kGroupMax + 1) + g] = pos;
            for (int e : kv.second) t.slot_list[d * 216 + pos++] = e;
            ++g;
        }
        t.grp_off[d * (kGroupMax + 1) + g] = pos;
        t.grp_n[d] = g;
        for (int tt = 0; tt < 8; ++tt) {
            int c2[3];
            for (int a = 0; a < 3; ++a) c2[a] = ((tt >> a) & 1) ? 1 : -1;
            int v2[3];
            for (int i = 0; i < 3; ++i) v2[i] = P[3 * i] * c2[0] + P[3 * i + 1] * c2[1] + P[3 * i + 2] * c2[2];
            t.child_shift[d * 8 + tt] = shift_index(v2);
        }
    }
}

// Plane-wave rule `qd` (3..6): the rule generated for that many digits.
const ExpQuad &exp_quadrature(int qd) {
    static ExpQuad q[5];
    static std::once_flag once;
    std::call_once(once, [] {
        auto set = [](ExpQuad &e, int s, const double *l, const double *w, const int *m) {
            e.s = s;
            e.lambda.assign(l, l + s);
            e.weight.assign(w, w + s);
            e.m.assign(m, m + s);
        };
        set(q[0], RPY_EXPQ_D3_S, rpy_expq_d3_lambda, rpy_expq_d3_weight, rpy_expq_d3_m);
        set(q[1], RPY_EXPQ_D4_S, rpy_expq_d4_lambda, rpy_expq_d4_weight, rpy_expq_d4_m);
        set(q[2], RPY_EXPQ_D5_S, rpy_expq_d5_lambda, rpy_expq_d5_weight, rpy_expq_d5_m);
        set(q[3], RPY_EXPQ_D6_S, rpy_expq_d6_lambda, rpy_expq_d6_weight, rpy_expq_d6_m);
        set(q[4], RPY_EXPQ_D9_S, rpy_expq_d9_lambda, rpy_expq_d9_weight, rpy_expq_d9_m);
    });
    return q[qd <= 3 ? 0 : (qd >= 9 ? 4 : (qd >= 6 ? 3 : qd - 3))];
}

// Expansion order per setting, chosen from measured rel-L2 against the oracle
// (1M-bead sphere and 4M-bead cube): p = 8 gives 5.5e-5 / 1.9e-5 at 3 digits,
// p = 18 gives 4.0e-8 at 6 digits, each with a far-field-only error at least
// 3x below the setting.
int default_order(int digits) { return digits <= 3 ? 8 : (digits <= 6 ? 18 : 26); }
int default_leaf_cap(int digits) { return digits <= 3 ? 40 : (digits <= 6 ? 100 : 120); }

int build_tables(int p, int qd, OpTables &t) {
    if (p < 2 || p > kMaxP) return RPY_ERR_INVALID;
    const ExpQuad &q = exp_quadrature(qd);
    t.p = p;
    t.nc = ncoef(p);
    t.digits = qd;
    t.s = q.s;
    t.S = q.half();
    t.m2x_c.assign(size_t(q.s) * t.nc, 0.0);
    t.x2l_c.assign(size_t(q.s) * t.nc, 0.0);
    for (int k = 0; k < q.s; ++k)
        for (int n = 0; n <= p; ++n)
            for (int m = 0; m <= n; ++m) {
                double inv = 1.0 / Nnm(n, m);
                t.m2x_c[size_t(k) * t.nc + tri(n, m)] = std::pow(q.lambda[k], n) * inv;
                t.x2l_c[size_t(k) * t.nc + tri(n, m)] = std::pow(-q.lambda[k], n) * inv;
            }
    t.e_k.clear(); t.e_cos.clear(); t.e_sin.clear(); t.e_wm.clear();
    t.k_start.assign(q.s + 1, 0);
    for (int k = 0; k < q.s; ++k) {
        t.k_start[k] = int(t.e_k.size());
        for (int j = 0; j < q.m[k] / 2; ++j) {
            double al = 2.0 * M_PI * j / q.m[k];
            t.e_k.push_back(k);
            t.e_cos.push_back(std::cos(al));
            t.e_sin.push_back(std::sin(al));
            t.e_wm.push_back(q.weight[k] / q.m[k]);
        }
    }
    t.k_start[q.s] = int(t.e_k.size());
    t.u_k.clear();
    t.u_start.assign(q.s + 1, 0);
    for (int k = 0; k < q.s; ++k) {
        t.u_start[k] = int(t.u_k.size());
        const int H = q.m[k] / 2;
        for (int u = 0; u < H / 2 + 1; ++u) t.u_k.push_back(k);
    }
    t.u_start[q.s] = int(t.u_k.size());
    t.shift.assign(size_t(216) * t.S * 2, 0.0);
    for (int off = 0; off < 216; ++off) {
        double dx = (off % 6) - 2.5, dy = ((off / 6) % 6) - 2.5, dz = (off / 36) - 2.5;
        for (int e = 0; e < t.S; ++e) {
            double lam = q.lambda[t.e_k[e]];
            double mag = std::exp(-lam * dz);
            double ph = lam * (dx * t.e_cos[e] + dy * t.e_sin[e]);
            t.shift[(size_t(off) * t.S + e) * 2] = mag * std::cos(ph);
            t.shift[(size_t(off) * t.S + e) * 2 + 1] = mag * std::sin(ph);
        }
    }
    build_groups(t);
    // factorized rotations: frames (x, y) and the eight child octants, forward and back
    {
        t.frot_off.resize(p + 2);
        t.frot_off[0] = 0;
        for (int n = 0; n <= p; ++n) t.frot_off[n + 1] = t.frot_off[n] + factor_len(n);
        const int FL = t.frot_off[p + 1];
        t.frot_fwd.assign(size_t(2) * FL, 0.0);
        t.frot_bwd.assign(size_t(2) * FL, 0.0);
        t.forot_fwd.assign(size_t(8) * FL, 0.0);
        t.forot_bwd.assign(size_t(8) * FL, 0.0);
        for (int f = 0; f < 2; ++f) {
            const double *Q = f == 0 ? kQx : kQy;
            double Qt[9];
            transpose3(Q, Qt);
            if (!factor_rotation(Qt, p, t.frot_off, &t.frot_fwd[size_t(f) * FL], true) ||
                !factor_rotation(Q, p, t.frot_off, &t.frot_bwd[size_t(f) * FL], true))
                return RPY_ERR_INTERNAL;
        }
        for (int o = 0; o < 8; ++o) {
            double Q[9], Qt[9];
            octant_frame(o, Q);
            transpose3(Q, Qt);
            if (!factor_rotation(Qt, p, t.frot_off, &t.forot_fwd[size_t(o) * FL]) ||
                !factor_rotation(Q, p, t.frot_off, &t.forot_bwd[size_t(o) * FL]))
                return RPY_ERR_INTERNAL;
        }
    }
    // z shifts of M2M / L2L
    {
        // along the frame z axis the shift is delta = sqrt(3)/4 parent sides:
        // M2M  M^p_n^m = sum_{k=m..n} (N_n^m / N_k^m) delta^{n-k} / (n-k)! 2^{-k} M^c_k^m
        // L2L  L^c_k^m = sum_{n=k..p} (N_n^m / N_k^m) delta^{n-k} / (n-k)! 2^{-k-1} L^p_n^m
        double delta = std::sqrt(3.0) / 4.0;
        t.zm2m.assign(size_t(t.nc) * (p + 1), 0.0);
        t.zl2l.assign(size_t(t.nc) * (p + 1), 0.0);
        for (int n = 0; n <= p; ++n)
            for (int m = 0; m <= n; ++m)
                for (int k = m; k <= p; ++k) {
                    if (k <= n)
                        t.zm2m[size_t(tri(n, m)) * (p + 1) + k] =
                            Nnm(n, m) / Nnm(k, m) * std::pow(delta, n - k) / fact(n - k) * std::ldexp(1.0, -k);
                    if (k >= n)   // output (n, m) of L2L takes inputs of degree k >= n
                        t.zl2l[size_t(tri(n, m)) * (p + 1) + k] =
                            Nnm(k, m) / Nnm(n, m) * std::pow(delta, k - n) / fact(k - n) * std::ldexp(1.0, -n - 1);
                }
    }
    t.roots.assign(size_t(2) * t.S * 2, 0.0);
    for (int k = 0; k < q.s; ++k)
        for (int r = 0; r < q.m[k]; ++r) {
            size_t idx = size_t(2) * t.k_start[k] + r;
            t.roots[2 * idx] = std::cos(2.0 * M_PI * r / q.m[k]);
            t.roots[2 * idx + 1] = std::sin(2.0 * M_PI * r / q.m[k]);
        }
    HarmRec h = harm_rec(p);
    t.rec_a = h.a;
    t.rec_b = h.b;
    t.rec_c = h.c;
    t.rec_cm.assign(h.c.size(), 1.0);
    for (size_t m = 1; m < h.c.size(); ++m) t.rec_cm[m] = t.rec_cm[m - 1] * h.c[m];
    int nl = ncoef(p + 2);
    t.lad.assign(size_t(6) * nl, 0.0);
    auto sq = [](long v) { return v > 0 ? std::sqrt(double(v)) : 0.0; };
    for (int k = 0; k <= p + 2; ++k)
        for (int m = 0; m <= k; ++m) {
            int i = tri(k, m);
            t.lad[0 * nl + i] = sq(long(k + 1 + m) * (k + 1 - m));
            t.lad[1 * nl + i] = sq(long(k - m + 1) * (k - m + 2));
            t.lad[2 * nl + i] = sq(long(k + m + 1) * (k + m + 2));
            t.lad[3 * nl + i] = sq(long(k + m) * (k - m));
            t.lad[4 * nl + i] = sq(long(k + m) * (k + m - 1));
            t.lad[5 * nl + i] = sq(long(k - m) * (k - m - 1));
        }
    return RPY_OK;
}

int build_reference_table(const OpTables &t, int which, std::vector<double> &v) {
    const int p = t.p;
    std::vector<double> other;
    std::vector<int> off;
    switch (which) {
        case 1: build_m2m(p, v); return RPY_OK;
        case 2: build_l2l(p, v); return RPY_OK;
        case 3: build_rotations(p, v, other, off); return RPY_OK;
        case 4: build_rotations(p, other, v, off); return RPY_OK;
        case 10:
            rotation_offsets(p, off);
            v.assign(off.begin(), off.end());
            return RPY_OK;
        case 12:
        case 13: {
            rotation_offsets(p, off);
            const size_t L = off.back();
            v.assign(8 * L, 0.0);
            other.assign(L, 0.0);
            for (int o = 0; o < 8; ++o) {
                double Q[9];
                octant_frame(o, Q);
                double *mine = &v[o * L], *rest = other.data();
                rotation_blocks(Q, p, off, which == 12 ? mine : rest, which == 12 ? rest : mine);
            }
            return RPY_OK;
        }
        case 16:
        case 17:
        case 18: {   // shift(off) = shz[iz] shx[ix] shy[iy], off = ix + 6 iy + 36 iz, offset d = index - 2.5 per axis
            const ExpQuad &q = exp_quadrature(t.digits);
            v.clear();
            for (int i = 0; i < 6; ++i)
                for (int e = 0; e < t.S; ++e) {
                    const double lam = q.lambda[t.e_k[e]], d = i - 2.5;
                    const double ph = lam * d * (which == 17 ? t.e_cos[e] : t.e_sin[e]);
                    if (which == 16) v.push_back(std::exp(-lam * d));
                    else v.insert(v.end(), {std::cos(ph), std::sin(ph)});
                }
            return RPY_OK;
        }
        default: return RPY_ERR_INVALID;
    }
}

}  // namespace rpy
