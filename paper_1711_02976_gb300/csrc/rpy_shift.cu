// Multipole-to-multipole and local-to-local shifts between a box and its children (M2M, L2L) of both
// precision forms: rotate into the frame whose z axis is the shift direction, apply the m-diagonal z
// shift, rotate back (O(p^3) per child instead of the O(p^4) of a dense operator).
//
// One block per parent, cb of its children at a time; an item is one coefficient of one child with four sets
// (FP32) or two (double-floats) in packed operations (rpy_quad.h).  The z rotation that follows the shift is applied
// as the shift is summed, and a parent's children are added in octant order (a fixed order).
// Measured, M2M and L2L in ms, from one child per block in scalar double-floats (FP64 form) and the dense
// operators (FP32 form below order 12): 15M-bead cube 3.0 and 2.95 -> 1.5 and 1.5; 1M-bead sphere and cube, 6 digits 2.1 and 1.9 ->
// 1.75 and 1.47, FP32 0.81 and 0.78 -> 0.42 and 0.41; 256 systems FP32 1.26 and 1.61 -> 0.96 and 1.12; 50k beads FP32 0.173 and
// 0.069 -> 0.034 and 0.035 (few parents: the dense form's serial chain of eight operators); 4,096 beads 0.026
// and 0.020 -> 0.016 and 0.014.
// rb (box origin of q4): set 4 moves its origin with the expansion, M4 += (c_child - c_parent) . M_F for a child's
// share, L4 += (c_parent - c_child) . L_F for a shifted local.
#include <cooperative_groups.h>

#include "rpy_quad.h"

namespace rpy {

// set 4 += (dx, dy, dz) . sets 1..3 of coefficient i; v: the sets of pr (the last), from the planes' first part
// (q = 0: real, 1: imaginary)
__device__ __forceinline__ void move_set4(const Planes<float> &, int, int, float dx, float dy, float dz, f4 &v) {
    v.b.y = fmaf(dz, v.b.x, fmaf(dy, v.a.y, fmaf(dx, v.a.x, v.b.y)));
}
__device__ __forceinline__ void move_set4(const Planes<dfl> &B, int q, int i, dfl dx, dfl dy, dfl dz, df2 &v) {
    const df2 f = q ? B.y(0, i) : B.x(0, i);
    dfl a(v.h.y, v.l.y);
    macc(a, dx, dfl(f.h.x, f.l.x));
    macc(a, dy, dfl(f.h.y, f.l.y));
    macc(a, dz, dfl(v.h.x, v.l.x));
    a = closed(a);
    v.h.y = a.h;
    v.l.y = a.l;
}

// The present children of box b in octant order; returns their number (all threads of the block).
__device__ __forceinline__ int children_of(const int *child, int b, int *ch, int *oct) {
    if (threadIdx.x == 0) {
        int k = 0;
        for (int o = 0; o < 8; ++o)
            if (child[8 * b + o] >= 0) {
                ch[k] = child[8 * b + o];
                oct[k++] = o;
            }
        ch[8] = k;
    }
    __syncthreads();
    return ch[8];
}

// CL: a cluster of eight blocks per parent, one child each (blockIdx.y its octant, cb = 1), which then add
// a slice of the coefficients each from all eight through distributed shared memory.
template <typename T, bool COL, bool CL>
__device__ __forceinline__ void m2m_body(int b0, const DevTables<T> &D, const int *leaf, const int *child,
                                         const double *side, int rb, int cb, cpx<T> *M) {
    using V = typename Quad<T>::V;
    constexpr int N = Quad<T>::N, SH = Quad<T>::SH;
    __shared__ int ch[9], oct[8];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    if (leaf[b]) return;
    const int nc = ncoef(D.p), per = N * nc;   // items of a child
    float4 *const pa = reinterpret_cast<float4 *>(smem_raw), *const pb = pa + cb * 2 * per;
    auto A = [&](int c) { return Planes<T>{pa + c * 2 * per, nc}; };
    auto B = [&](int c) { return Planes<T>{pb + c * 2 * per, nc}; };
    const Planes<T> sum{pb + cb * 2 * per, nc};   // where the children take several rounds
    int nch;
    if (CL) {
        const int c = child[8 * b + blockIdx.y];
        nch = c >= 0;
        if (threadIdx.x == 0) {
            ch[0] = c;
            oct[0] = blockIdx.y;
        }
        __syncthreads();
    } else {
        nch = children_of(child, b, ch, oct);
    }
    cpx<T> *dst = M + size_t(b) * kSets * nc;
    for (int g = 0; g < nch; g += cb) {
        const int cn = min(cb, nch - g), items = cn * per;
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH;
            V x, y;
            load_sets(M + size_t(ch[g + c]) * kSets * nc, nc, pr, i, x, y);
            rotate_z(D.forot_fwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, x, y, A(c));
        }
        __syncthreads();
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH;
            V x, y;
            rotate_y<false, COL>(D.forot_fwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, A(c), x, y);
            B(c).set(pr, i, x, y);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH, n = deg_of(i), m = i - tri(n, 0);
            const Planes<T> in = B(c);
            const T *z = D.zm2m + i;   // stored [k][coefficient]
            V x = zero<V>(), y = x;
            for (int k = m; k <= n; ++k) {
                macc(x, z[k * nc], in.x(pr, tri(k, m)));
                macc(y, z[k * nc], in.y(pr, tri(k, m)));
            }
            rotate_z(D.forot_bwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, closed(x), closed(y), A(c));
        }
        __syncthreads();
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH;
            V x, y;
            rotate_y<false, COL>(D.forot_bwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, A(c), x, y);
            B(c).set(pr, i, x, y);
        }
        __syncthreads();
        for (int e = threadIdx.x; !CL && e < per; e += blockDim.x) {
            const int pr = e & (N - 1), i = e >> SH;
            V x = zero<V>(), y = x;
            if (g) {
                x = sum.x(pr, i);
                y = sum.y(pr, i);
            }
            for (int c = 0; c < cn; ++c) {
                V vx = B(c).x(pr, i), vy = B(c).y(pr, i);
                if (rb && pr == N - 1) {
                    const int o = oct[g + c];
                    const double h = 0.5 * side[ch[g + c]];   // child centre - parent centre = h (2 bit - 1) per axis
                    const T dx((o & 1) ? h : -h), dy((o & 2) ? h : -h), dz((o & 4) ? h : -h);
                    move_set4(B(c), 0, i, dx, dy, dz, vx);
                    move_set4(B(c), 1, i, dx, dy, dz, vy);
                }
                x = x + vx;
                y = y + vy;
            }
            if (g + cb >= nch) store_sets(dst, nc, pr, i, x, y);
            else sum.set(pr, i, x, y);
        }
        // the next round's first writes go to A, which the last barrier freed; its second phase writes B
        // behind a barrier
    }
    if constexpr (CL) {
        auto cluster = cooperative_groups::this_cluster();
        cluster.sync();
        // this block's slice of the items, summed over the present children in octant order
        const int slice = (per + 7) / 8, e1 = min(per, (int(blockIdx.y) + 1) * slice);
        for (int e = blockIdx.y * slice + threadIdx.x; e < e1; e += blockDim.x) {
            const int pr = e & (N - 1), i = e >> SH;
            V x = zero<V>(), y = x;
            for (int o = 0; o < 8; ++o) {
                const int c = child[8 * b + o];
                if (c < 0) continue;
                const Planes<T> R{cluster.map_shared_rank(pb, o), nc};
                V vx = R.x(pr, i), vy = R.y(pr, i);
                if (rb && pr == N - 1) {
                    const double h = 0.5 * side[c];   // child centre - parent centre = h (2 bit - 1) per axis
                    const T dx((o & 1) ? h : -h), dy((o & 2) ? h : -h), dz((o & 4) ? h : -h);
                    move_set4(R, 0, i, dx, dy, dz, vx);
                    move_set4(R, 1, i, dx, dy, dz, vy);
                }
                x = x + vx;
                y = y + vy;
            }
            store_sets(dst, nc, pr, i, x, y);
        }
        cluster.sync();   // no block leaves while another reads its planes
    }
}
template <typename T, bool COL>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 3 : 5)
    k_m2m(int b0, DevTables<T> D, const int *leaf, const int *child, const double *side, int rb, int cb, cpx<T> *M) {
    m2m_body<T, COL, false>(b0, D, leaf, child, side, rb, cb, M);
}
template <typename T, bool COL>
__global__ void __cluster_dims__(1, 8, 1) __launch_bounds__(256, sizeof(T) == 8 ? 3 : 5)
    k_m2m_cluster(int b0, DevTables<T> D, const int *leaf, const int *child, const double *side, int rb, cpx<T> *M) {
    m2m_body<T, COL, true>(b0, D, leaf, child, side, rb, 1, M);
}

template <typename T, bool COL>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 3 : 5)
    k_l2l(int b0, DevTables<T> D, const int *leaf, const int *child, const double *side, int rb, int cb, cpx<T> *L) {
    using V = typename Quad<T>::V;
    constexpr int N = Quad<T>::N, SH = Quad<T>::SH;
    __shared__ int ch[9], oct[8];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    if (leaf[b]) return;
    const int p = D.p, nc = ncoef(p), per = N * nc;
    float4 *const pa = reinterpret_cast<float4 *>(smem_raw), *const pb = pa + cb * 2 * per;
    auto A = [&](int c) { return Planes<T>{pa + c * 2 * per, nc}; };
    auto B = [&](int c) { return Planes<T>{pb + c * 2 * per, nc}; };
    const int nch = children_of(child, b, ch, oct);
    const cpx<T> *src = L + size_t(b) * kSets * nc;
    // gridDim.y blocks share the parent's children
    for (int g = blockIdx.y * cb; g < nch; g += cb * gridDim.y) {
        const int items = min(cb, nch - g) * per;
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH;
            V x, y;
            load_sets(src, nc, pr, i, x, y);
            rotate_z(D.forot_fwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, x, y, A(c));
        }
        __syncthreads();
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH;
            V x, y;
            rotate_y<false, COL>(D.forot_fwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, A(c), x, y);
            B(c).set(pr, i, x, y);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH, n = deg_of(i), m = i - tri(n, 0);
            const Planes<T> in = B(c);
            const T *z = D.zl2l + i;   // stored [k][coefficient]
            V x = zero<V>(), y = x;
            for (int k = n; k <= p; ++k) {
                macc(x, z[k * nc], in.x(pr, tri(k, m)));
                macc(y, z[k * nc], in.y(pr, tri(k, m)));
            }
            rotate_z(D.forot_bwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, closed(x), closed(y), A(c));
        }
        __syncthreads();
        for (int e = threadIdx.x; e < items; e += blockDim.x) {
            const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH;
            V x, y;
            rotate_y<false, COL>(D.forot_bwd + oct[g + c] * D.frot_len, D.frot_off, i, pr, A(c), x, y);
            if (rb) B(c).set(pr, i, x, y);
            else add_sets(L + size_t(ch[g + c]) * kSets * nc, nc, pr, i, x, y);
        }
        __syncthreads();
        if (rb) {
            for (int e = threadIdx.x; e < items; e += blockDim.x) {
                const int c = e / per, r = e - c * per, pr = r & (N - 1), i = r >> SH, o = oct[g + c];
                V x = B(c).x(pr, i), y = B(c).y(pr, i);
                if (pr == N - 1) {
                    const double h = 0.5 * side[ch[g + c]];   // parent centre - child centre = -h (2 bit - 1) per axis
                    const T dx((o & 1) ? -h : h), dy((o & 2) ? -h : h), dz((o & 4) ? -h : h);
                    move_set4(B(c), 0, i, dx, dy, dz, x);
                    move_set4(B(c), 1, i, dx, dy, dz, y);
                }
                add_sets(L + size_t(ch[g + c]) * kSets * nc, nc, pr, i, x, y);
            }
            __syncthreads();
        }
    }
}

// M2M takes a cluster per parent (a block per child; 20k-bead sphere 0.32 -> 0.10 ms, but a 15M-bead cube
// 1.5 -> 4.0 ms if taken everywhere) where a level has few parents, so that its blocks are
// short, unless a child has too few items to fill one; L2L, which needs no sum, splits a parent's children
// over blocks there too, and always where one child fills a block.
constexpr int kClusterParents = 2500, kSplitParents = 600;

// Children at a time: all eight, halved until the planes take at most 40 KB (FP32 24).
template <typename T>
static int shift_children(int p, bool sum, size_t &smem) {
    const size_t per = sizeof(float4) * 2 * Quad<T>::N * ncoef(p);
    int cb = 8;
    for (;; cb >>= 1) {
        smem = per * (2 * cb + (sum && cb < 8 ? 1 : 0));
        if (cb == 1 || smem <= (kIsDf<T> ? 40 : 24) * 1024) return cb;
    }
}

template <typename T>
int run_m2m_t(Tree &t, const DevTables<T> &D, cpx<T> *M, int rb, cudaStream_t st) {
    const double *side = kIsDf<T> ? t.side_u : t.b_side;
    const bool col = y_by_column(sizeof(T), D.p);
    auto k = col ? k_m2m<T, true> : k_m2m<T, kIsDf<T>>;
    const int per = Quad<T>::N * ncoef(D.p);
    auto kc = col ? k_m2m_cluster<T, true> : k_m2m_cluster<T, kIsDf<T>>;
    const size_t smem1 = sizeof(float4) * 4 * Quad<T>::N * ncoef(D.p);
    const int thr1 = even_threads(per);
    RPY_TRY(set_smem(kc, smem1));
    size_t smem = 0;
    const int cb = shift_children<T>(D.p, true, smem), thr = even_threads(cb * per);
    RPY_TRY(set_smem(k, smem));
    for (int l = t.nlevels - 2; l >= 2; --l) {
        const int lb = t.level_off[l], ln = t.level_off[l + 1] - lb;
        if (ln <= 0) continue;
        if (per >= 64 && ln <= kClusterParents) kc<<<dim3(ln, 8), thr1, smem1, st>>>(lb, D, t.b_leaf, t.b_child, side, rb, M);
        else k<<<ln, thr, smem, st>>>(lb, D, t.b_leaf, t.b_child, side, rb, cb, M);
        RPY_LAUNCHED(1);
    }
    RPY_CHECK(cudaGetLastError());
    return RPY_OK;
}

template <typename T>
int run_l2l_t(Tree &t, const DevTables<T> &D, cpx<T> *L, int rb, cudaStream_t st) {
    const double *side = kIsDf<T> ? t.side_u : t.b_side;
    const bool col = y_by_column(sizeof(T), D.p);
    const int per = Quad<T>::N * ncoef(D.p);
    auto k = col ? k_l2l<T, true> : k_l2l<T, kIsDf<T>>;
    const size_t smem1 = sizeof(float4) * 4 * Quad<T>::N * ncoef(D.p);
    const int thr1 = even_threads(per);
    size_t smem = 0;
    const int cb = shift_children<T>(D.p, false, smem), thr = even_threads(cb * per);
    RPY_TRY(set_smem(k, smem));
    for (int l = 2; l + 1 < t.nlevels; ++l) {
        const int lb = t.level_off[l], ln = t.level_off[l + 1] - lb;
        if (ln <= 0) continue;
        if (per >= 128 || ln <= kSplitParents) k<<<dim3(ln, 8), thr1, smem1, st>>>(lb, D, t.b_leaf, t.b_child, side, rb, 1, L);
        else k<<<ln, thr, smem, st>>>(lb, D, t.b_leaf, t.b_child, side, rb, cb, L);
        RPY_LAUNCHED(1);
    }
    RPY_CHECK(cudaGetLastError());
    return RPY_OK;
}

template int run_m2m_t<dfl>(Tree &, const DevTables<dfl> &, cpx<dfl> *, int, cudaStream_t);
template int run_m2m_t<float>(Tree &, const DevTables<float> &, cpx<float> *, int, cudaStream_t);
template int run_l2l_t<dfl>(Tree &, const DevTables<dfl> &, cpx<dfl> *, int, cudaStream_t);
template int run_l2l_t<float>(Tree &, const DevTables<float> &, cpx<float> *, int, cudaStream_t);

}  // namespace rpy
