// Plane-wave multipole-to-local step (M2X, X2X merge-and-shift, X2L) of both precision forms.
//
// Every table value (node factors, roots of unity, shifts, rotations) serves the four charge sets alike, so a
// thread carries several sets of one item: all four in FP32 (two packed FP32x2 registers), a pair of them in
// double-floats (T = dfl, one packed double-float), and a pair in X2X of either.  One table load, index
// update and loop step then serves them all, and the packed operations halve the FMA instructions.
// Neighbouring lanes carry the pairs of one item: they share its table loads.
//
// Layouts: plane waves Xo and Xi [box][direction][wave][re of 4 sets, im of 4 sets] (Quad<T>: the sets of a
// part in one or two float4); M and L [box][set][coefficient] cpx<T> as elsewhere.
//
// Measured, ms (M2X, X2X, X2L).  FP64 form, from scalar double-floats: 1M-bead sphere and cube at 6 digits
// 8.8, 5.3, 9.0 -> 5.3, 3.6, 7.4; 15M-bead cube at 3 digits 16.6, 29.2, 21.7 -> 9.2, 22.0, 12.2; 200k beads at 9 digits
// 11.5, 3.3, 15.0 -> 5.2, 2.3, 7.4.  FP32 form, from one wave or set per operation: 1M beads at 6 digits
// 2.48, 2.03, 2.07 -> 1.50, 2.05, 1.66; 15M-bead cube 4.61, 10.9, 4.47 -> 2.87, 6.7, 4.6; 256 systems, 11.5M beads,
// 8.26, 9.8, 6.7 -> 4.4, 6.4, 6.4.
#include "rpy_far.h"
#include "rpy_quad.h"

namespace rpy {

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


// A_k^m rows of one node at an odd stride, so that neighbouring nodes fall on different banks
__host__ __device__ inline int a_stride(int p) { return (p + 1) | 1; }

// ---------------------------------------------------------------- M2X
// One box per block, kc quadrature nodes at a time.
template <typename T, bool COL>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 3 : 3)
    k_m2x(int b0, DevTables<T> D, const cpx<T> *M, float4 *Xo, int f0, int nf, int kc) {
    using V = typename Quad<T>::V;
    constexpr int N = Quad<T>::N, SH = Quad<T>::SH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p), s = D.s, S = D.S, NS = a_stride(p);
    const Planes<T> Mu{reinterpret_cast<float4 *>(smem_raw), nc};
    const Planes<T> AE{Mu.p + 2 * N * nc, kc * NS}, AO{AE.p + 2 * N * kc * NS, kc * NS};
    const Planes<T> Tm{AE.p, nc};   // rotation scratch, before the A rows are formed (node_chunk leaves room)
    const cpx<T> *src = M + size_t(b) * kSets * nc;
    const int hP = harm_lanes(p);
    for (int f = f0; f < f0 + nf; ++f) {
        if (f > 0) {
            const T *rf = D.frot_fwd + size_t(f - 1) * D.frot_len;
            for (int e = threadIdx.x; e < N * nc; e += blockDim.x) {
                V x, y;
                load_sets(src, nc, e & (N - 1), e >> SH, x, y);
                rotate_z(rf, D.frot_off, e >> SH, e & (N - 1), x, y, Tm);
            }
            __syncthreads();
            for (int e = threadIdx.x; e < N * nc; e += blockDim.x) {
                V x, y;
                rotate_y<true, COL>(rf, D.frot_off, e >> SH, e & (N - 1), Tm, x, y);
                Mu.set(e & (N - 1), e >> SH, x, y);
            }
        } else {
            for (int e = threadIdx.x; e < N * nc; e += blockDim.x) {
                V x, y;
                load_sets(src, nc, e & (N - 1), e >> SH, x, y);
                Mu.set(e & (N - 1), e >> SH, x, y);
            }
        }
        __syncthreads();
        // + direction; the - direction follows 2 N S float4 further
        float4 *out = Xo + (size_t(b) * (2 * nf) + 2 * (f - f0)) * 2 * N * S;
        for (int k0 = 0; k0 < s; k0 += kc) {
            const int kn = min(kc, s - k0);
            // A_k^m split by parity of n + m (the - direction is the reflection (-1)^{n+m}), stored as
            // 2 i^m A_k^m so that the wave sum needs no sign logic: even m feed the real part, odd m the
            // imaginary part.  One item per (node, column pair (m, p - m)): p + 2 terms.  (An item for each part:
            // twice the table loads, FP32 M2X of the 1M-bead sphere 1.52 -> 1.84 ms.)
            for (int e = threadIdx.x; e < N * kn * hP; e += blockDim.x) {
                const int pr = e & (N - 1), r = e >> SH, kk = r / hP, c = r - kk * hP;
                const T *cc = D.m2x_c + size_t(k0 + kk) * nc;
                for (int h = 0; h < 2; ++h) {
                    const int m = h ? p - c : c;
                    if (h && m == c) break;
                    V evx = zero<V>(), evy = evx, odx = evx, ody = evx;
                    int n = m, i = tri(m, m);
                    for (; n < p; n += 2) {   // degrees n and n + 1
                        const int i1 = i + n + 1;
                        const T c0 = cc[i], c1 = cc[i1];
                        macc(evx, c0, Mu.x(pr, i));
                        macc(evy, c0, Mu.y(pr, i));
                        macc(odx, c1, Mu.x(pr, i1));
                        macc(ody, c1, Mu.y(pr, i1));
                        i = i1 + n + 2;
                    }
                    if (n == p) {
                        const T c0 = cc[i];
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
            for (int e = threadIdx.x; e < N * un; e += blockDim.x) {
                const int pr = e & (N - 1), u = ub + (e >> SH);
                const int4 ui = D.u_info[u];
                const int row = (ui.x - k0) * NS, j0 = ui.y, H = ui.z, t = ui.w, Mk = 2 * H;
                const bool pair = t > 0 && 2 * t != H;
                const cpx<T> *rt = D.roots + 2 * j0;
                const T wm = D.e_wm[j0 + t];
                int step2 = 2 * t;
                if (step2 >= Mk) step2 -= Mk;
#pragma unroll 1
                for (int odd = 0; odd < 2; ++odd) {
                    V pe = zero<V>(), qe = pe, po = pe, qo = pe;
                    int idx = t, m = 1;
                    if (!odd) {
                        pe = AE.x(pr, row);
                        po = AO.x(pr, row);
                        idx = step2;
                        m = 2;
                    }
                    for (; m <= p; m += 2) {
                        const cpx<T> z = rt[idx];
                        const int i = row + m;
                        macc(pe, z.x, AE.x(pr, i));
                        macc(qe, z.y, AE.y(pr, i));
                        macc(po, z.x, AO.x(pr, i));
                        macc(qo, z.y, AO.y(pr, i));
                        idx += step2;
                        if (idx >= Mk) idx -= Mk;
                    }
                    // real (even m) or imaginary (odd m) parts: + direction A = AE + AO, - direction AE - AO
                    auto store = [&](int j, V a, V o) {
                        float4 *d = out + 2 * N * j + N * odd + pr;
                        d[0] = put(times(wm, a + o));
                        d[2 * N * S] = put(times(wm, a - o));
                    };
                    store(j0 + t, pe - qe, po - qo);
                    if (pair) {   // the partner, with sign (-1)^m
                        const V eb = pe + qe, ob = po + qo;
                        store(j0 + H - t, odd ? -eb : eb, odd ? -ob : ob);
                    }
                }
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------- X2X merge-and-shift
// Per parent and direction, the present sources (children of the parent's colleagues) are shifted to the
// parent's centre and summed per group of children they serve, then shifted once to each child.
struct X2XList {
    int src[216];
    int vsrc[216], vsh[216], vpre[217];   // the present sources and their shift rows (times S), in slot order
    int vend[216];                        // child mask of its group at the last present source of a group, else 0
};

// Fills the list (all threads of the block); returns the number of present sources.  place(position, slot)
// sees each of them once.
template <typename T, typename F>
__device__ __forceinline__ int x2x_sources(X2XList &W, const DevTables<T> &D, int P, int d, int row, const int *coll,
                                           const int *child, const int *leaf, F place) {
    for (int sl = threadIdx.x; sl < 216; sl += blockDim.x) {
        const int q = sl >> 3, o = sl & 7;
        const int Q = coll[27 * P + q];
        W.src[sl] = (Q >= 0 && !leaf[Q]) ? child[8 * Q + o] : -1;
    }
    __syncthreads();
    const int ng = D.grp_n[d];
    const int *goff = D.grp_off + d * (kGroupMax + 1);
    const int *gmask = D.grp_mask + d * kGroupMax;
    const int *slots = D.slot_list + d * 216;
    // warp 0 keeps the slots whose source box exists; vpre[z] = present slots before z, so group g covers
    // vsrc[vpre[goff[g]] .. vpre[goff[g + 1]])
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, nsl = goff[ng];
        int carry = 0;
        for (int z0 = 0; z0 < nsl; z0 += 32) {
            const int z = z0 + lane;
            int ent = 0, sb = -1;
            if (z < nsl) {
                ent = slots[z];
                sb = W.src[ent & 255];
            }
            const unsigned bal = __ballot_sync(0xffffffffu, sb >= 0);
            const int pos = carry + __popc(bal & ((1u << lane) - 1u));
            if (z < nsl) W.vpre[z] = pos;
            if (sb >= 0) {
                W.vsrc[pos] = sb;
                W.vsh[pos] = (ent >> 8) * row;
                place(pos, ent & 255);
            }
            carry += __popc(bal);
        }
        if (lane == 0) W.vpre[nsl] = carry;
    }
    __syncthreads();
    const int nz = W.vpre[goff[ng]];
    for (int z = threadIdx.x; z < nz; z += blockDim.x) W.vend[z] = 0;
    __syncthreads();
    for (int g = threadIdx.x; g < ng; g += blockDim.x) {
        const int z1 = W.vpre[goff[g + 1]];
        if (z1 > W.vpre[goff[g]]) W.vend[z1 - 1] = gmask[g];
    }
    __syncthreads();
    return nz;
}

// A pair of sets in one thread (PairOf).
__device__ __forceinline__ float2 get_pair(float2 m) { return m; }
__device__ __forceinline__ df2 get_pair(float4 m) { return as_df2(m); }
__device__ __forceinline__ float2 put_pair(float2 v) { return v; }
__device__ __forceinline__ float4 put_pair(df2 v) { return as_float4(v); }

// One thread per (wave, pair of sets).
// Plain loads, two sources in flight (double-floats): staging each thread's sources through shared memory by
// asynchronous copies four steps ahead was slower (1M-bead sphere 4.17 -> 4.46 ms, 15M-bead cube 25.7 ->
// 29.4 ms: it adds shared-memory instructions and takes a third of the L1).
// FP32: eight sources in flight at 72 registers (seven blocks of 128): 15M-bead cube 6.7 ms; four in flight at 64
// registers 8.4, twelve at 96 7.5.
// Blocks of 128 threads (96 registers in double-floats, five per SM) on large grids; of 256 threads where the
// grid leaves the SMs room and a block's own length counts (1M-bead sphere 4.24 -> 3.71 ms and 15M-bead cube
// 26.1 -> 23.0 ms from 256 to 128; 20k-bead sphere 0.133 -> 0.191 ms, 4,096 beads 0.058 -> 0.094 ms).
constexpr int kX2XSmallGrid = 3000;   // blocks
template <typename T, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS)
    k_x2x(const int *parents, DevTables<T> D, const int *coll, const int *child, const int *leaf,
          const typename PairOf<T>::Mem *Xo, typename PairOf<T>::Mem *Xi, int f0, int nf) {
    using V = typename PairOf<T>::V;
    __shared__ X2XList W;
    const int P = parents[blockIdx.x];
    const int dl = blockIdx.y, d = 2 * f0 + dl;   // direction, and its slot in this pass's buffers
    const int S = D.S;
    const int nz = x2x_sources(W, D, P, d, S, coll, child, leaf, [](int, int) {});
    const size_t dstride = size_t(2 * nf) * 4 * S;
    const auto *Xd = Xo + size_t(dl) * 4 * S;
    for (int e = threadIdx.x; e < 2 * S; e += blockDim.x) {
        const int j = e >> 1, pr = e & 1;
        V ax[8], ay[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) ax[t] = ay[t] = zero<V>();
        V gx = zero<V>(), gy = gx;
        constexpr int kUnroll = sizeof(T) == 8 ? 2 : 8;
#pragma unroll kUnroll
        for (int z = 0; z < nz; ++z) {
            const auto *xs = Xd + size_t(W.vsrc[z]) * dstride + 4 * j + pr;
            const V x = get_pair(xs[0]), y = get_pair(xs[2]);
            const cpx<T> sh = D.shift[W.vsh[z] + j];
            macc(gx, sh.x, x);
            macc(gx, neg1(sh.y), y);
            macc(gy, sh.y, x);
            macc(gy, sh.x, y);
            const int mask = W.vend[z];   // block-uniform
            if (mask) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if ((mask >> t) & 1) {
                        ax[t] = sum_raw(ax[t], gx);
                        ay[t] = sum_raw(ay[t], gy);
                    }
                gx = gy = zero<V>();
            }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int ch = child[8 * P + t];
            if (ch < 0) continue;
            const cpx<T> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
            const V x = closed(ax[t]), y = closed(ay[t]);
            auto *dst = Xi + (size_t(ch) * (2 * nf) + dl) * 4 * S + 4 * j + pr;
            dst[0] = put_pair(lin2(sh.x, x, neg1(sh.y), y));
            dst[2] = put_pair(lin2(sh.y, x, sh.x, y));
        }
    }
}

// Box origin of q4 = F . (r - o): set 4 travels with its origin at the centre of the box whose expansion it
// is.  Each source's set 4 moves to the parent centre as it is merged, X4 += (c_source - c_parent) . X_F, and
// each merged sum moves to the child as it is shifted there, X4 += (c_parent - c_child) . X_F, with X_F the
// force sets 1..3 of the same wave (rotations of the frames act on the plane-wave variables only, so the
// world offsets apply as they are).
struct Sets4f {
    f4 v;
};
struct Sets4d {
    df2 v[2];
};
__device__ __forceinline__ void macc(Sets4f &a, float s, const Sets4f &b) { macc(a.v, s, b.v); }
__device__ __forceinline__ void macc(Sets4d &a, dfl s, const Sets4d &b) {
    macc(a.v[0], s, b.v[0]);
    macc(a.v[1], s, b.v[1]);
}
__device__ __forceinline__ void accum(Sets4f &a, const Sets4f &b) { a.v = a.v + b.v; }
__device__ __forceinline__ void accum(Sets4d &a, const Sets4d &b) {
    a.v[0] = a.v[0] + b.v[0];
    a.v[1] = a.v[1] + b.v[1];
}
__device__ __forceinline__ Sets4f lin2(float a, const Sets4f &x, float b, const Sets4f &y) {
    return Sets4f{lin2(a, x.v, b, y.v)};
}
__device__ __forceinline__ Sets4d lin2(dfl a, const Sets4d &x, dfl b, const Sets4d &y) {
    return Sets4d{{lin2(a, x.v[0], b, y.v[0]), lin2(a, x.v[1], b, y.v[1])}};
}
__device__ __forceinline__ void load4(const float4 *m, Sets4f &v) { get(m[0], v.v); }
__device__ __forceinline__ void load4(const float4 *m, Sets4d &v) {
    get(m[0], v.v[0]);
    get(m[1], v.v[1]);
}
__device__ __forceinline__ void store4(float4 *m, const Sets4f &v) { m[0] = put(v.v); }
__device__ __forceinline__ void store4(float4 *m, const Sets4d &v) {
    m[0] = put(v.v[0]);
    m[1] = put(v.v[1]);
}
// set 4 += (dx, dy, dz) . sets 1..3 of one part (re or im)
__device__ __forceinline__ void move_origin(Sets4f &v, float dx, float dy, float dz) {
    v.v.b.y = fmaf(dz, v.v.b.x, fmaf(dy, v.v.a.y, fmaf(dx, v.v.a.x, v.v.b.y)));
}
__device__ __forceinline__ void move_origin(Sets4d &v, dfl dx, dfl dy, dfl dz) {
    dfl a(v.v[1].h.y, v.v[1].l.y);
    macc(a, dx, dfl(v.v[0].h.x, v.v[0].l.x));
    macc(a, dy, dfl(v.v[0].h.y, v.v[0].l.y));
    macc(a, dz, dfl(v.v[1].h.x, v.v[1].l.x));
    a = closed(a);
    v.v[1].h.y = a.h;
    v.v[1].l.y = a.l;
}
template <typename T> struct AllSets;
template <> struct AllSets<float> { using V = Sets4f; };
template <> struct AllSets<dfl> { using V = Sets4d; };

// slot = colleague (dx, dy, dz in -1..1, index 9 dz + 3 dy + dx + 13) x 8 + child octant:
// source centre - P's centre = hc (2 d + bit - 1/2) per axis, in world axes, hc the children's side
template <typename T>
__device__ __forceinline__ void source_offset(int sl, double hc, T &dx, T &dy, T &dz) {
    const int q = sl >> 3, o = sl & 7;
    dx = T(hc * (2 * (q % 3 - 1) + (o & 1) - 0.5));
    dy = T(hc * (2 * ((q / 3) % 3 - 1) + ((o >> 1) & 1) - 0.5));
    dz = T(hc * (2 * (q / 9 - 1) + ((o >> 2) & 1) - 0.5));
}

// One thread per wave, all four sets (box origin).
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 1 : 2)
    k_x2x4(const int *parents, DevTables<T> D, const int *coll, const int *child, const int *leaf, const double *side,
           const float4 *Xo, float4 *Xi, int f0, int nf) {
    using V = typename AllSets<T>::V;
    constexpr int N = Quad<T>::N;
    __shared__ X2XList W;
    __shared__ T vd[3][216];   // source centre - parent centre
    const int P = parents[blockIdx.x];
    const int dl = blockIdx.y, d = 2 * f0 + dl;
    const int S = D.S;
    const double hc = 0.5 * side[P];   // side of P's children (and of the sources)
    const int nz = x2x_sources(W, D, P, d, S, coll, child, leaf,
                               [&](int pos, int sl) { source_offset(sl, hc, vd[0][pos], vd[1][pos], vd[2][pos]); });
    const size_t dstride = size_t(2 * nf) * 2 * N * S;
    const float4 *Xd = Xo + size_t(dl) * 2 * N * S;
    for (int j = threadIdx.x; j < S; j += blockDim.x) {
        V ax[8] = {}, ay[8] = {}, gx = {}, gy = {};
#pragma unroll 2
        for (int z = 0; z < nz; ++z) {
            const float4 *xs = Xd + size_t(W.vsrc[z]) * dstride + 2 * N * j;
            V x, y;
            load4(xs, x);
            load4(xs + N, y);
            move_origin(x, vd[0][z], vd[1][z], vd[2][z]);
            move_origin(y, vd[0][z], vd[1][z], vd[2][z]);
            const cpx<T> sh = D.shift[W.vsh[z] + j];
            macc(gx, sh.x, x);
            macc(gx, neg1(sh.y), y);
            macc(gy, sh.y, x);
            macc(gy, sh.x, y);
            const int mask = W.vend[z];   // block-uniform
            if (mask) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if ((mask >> t) & 1) {
                        accum(ax[t], gx);
                        accum(ay[t], gy);
                    }
                gx = gy = V{};
            }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int ch = child[8 * P + t];
            if (ch < 0) continue;
            // P's centre - child t's centre = -(hc / 2) (2 bit - 1) per axis
            const double h = 0.5 * hc;
            const T ex((t & 1) ? -h : h), ey((t & 2) ? -h : h), ez((t & 4) ? -h : h);
            move_origin(ax[t], ex, ey, ez);
            move_origin(ay[t], ex, ey, ez);
            const cpx<T> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
            float4 *dst = Xi + (size_t(ch) * (2 * nf) + dl) * 2 * N * S + 2 * N * j;
            store4(dst, lin2(sh.x, ax[t], neg1(sh.y), ay[t]));
            store4(dst + N, lin2(sh.y, ax[t], sh.x, ay[t]));
        }
    }
}

// FP32 with more than 256 waves: the same sums fed by a producer warp, which stages the present sources
// through shared memory by bulk copies (TMA) into kX2XStages buffers, each holding one source's outgoing
// waves in one direction (8 S floats) and its shift row (S values, rows padded to an even length).
// Buffer q is "full" when its copies have landed (an mbarrier with the transaction count) and "empty" when
// every consumer warp has read it (an mbarrier with one arrival per consumer warp); the producer refills a
// buffer as soon as it is empty, so the consumers never wait on a global load and the block needs no
// barrier per source.
constexpr int kX2XStages = 4;
__host__ __device__ inline int x2x_tma_stage_elems(int S) { return 4 * S + ((S + 1) & ~1); }
__host__ inline size_t x2x_tma_smem(int S) { return sizeof(cpx<float>) * size_t(kX2XStages) * x2x_tma_stage_elems(S); }

__global__ void __launch_bounds__(512, 1)
    k_x2x_tma(const int *parents, DevTables<float> D, const int *coll, const int *child, const int *leaf,
              const double *side, const float4 *Xo, float4 *Xi, int f0, int nf, int rb, unsigned *status) {
    __shared__ X2XList W;
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
    if (threadIdx.x == 0) {
        bad = 0;
        issued = 0;
        for (int q = 0; q < kX2XStages; ++q) {
            mbar_init(&full[q], 1);
            mbar_init(&empty[q], unsigned(ncw));
        }
        mbar_init_fence();
    }
    const int nz = x2x_sources(W, D, P, d, Sp, coll, child, leaf,
                               [&](int pos, int sl) { source_offset(sl, hc, vd[0][pos], vd[1][pos], vd[2][pos]); });
    const int stage_elems = x2x_tma_stage_elems(S);
    cpx<float> *stage0 = reinterpret_cast<cpx<float> *>(smem_raw);
    if (warp == ncw) {
        // producer: one lane issues the copies, refilling each buffer once it is empty
        if (lane == 0) {
            const size_t dstride = size_t(2 * nf) * 2 * S;
            const float4 *Xd = Xo + size_t(dl) * 2 * S;
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
                bulk_load(buf, Xd + size_t(W.vsrc[z]) * dstride, src_bytes, &full[q]);
                bulk_load(buf + 4 * S, D.shiftp + W.vsh[z], sh_bytes, &full[q]);
                issued = z + 1;
            }
        }
    } else {
        const int j = threadIdx.x;
        const bool act = j < S;
        Sets4f ax[8] = {}, ay[8] = {}, gx = {}, gy = {};
        for (int z = 0; z < nz; ++z) {
            const int q = z % kX2XStages;
            if (!mbar_wait(&full[q], unsigned(z / kX2XStages) & 1u) || *(volatile int *)&bad) {
                bad = 1;
                break;
            }
            if (act) {
                const cpx<float> *buf = stage0 + size_t(q) * stage_elems;
                const float4 *xs = reinterpret_cast<const float4 *>(buf) + 2 * j;
                Sets4f x, y;
                load4(xs, x);
                load4(xs + 1, y);
                if (rb) {
                    move_origin(x, vd[0][z], vd[1][z], vd[2][z]);
                    move_origin(y, vd[0][z], vd[1][z], vd[2][z]);
                }
                const cpx<float> sh = buf[4 * S + j];
                macc(gx, sh.x, x);
                macc(gx, -sh.y, y);
                macc(gy, sh.y, x);
                macc(gy, sh.x, y);
                const int mask = W.vend[z];   // block-uniform
                if (mask) {
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if ((mask >> t) & 1) {
                            accum(ax[t], gx);
                            accum(ay[t], gy);
                        }
                    gx = gy = Sets4f{};
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[q]);   // this warp is done with buffer q
        }
        if (!*(volatile int *)&bad && act) {
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int ch = child[8 * P + t];
                if (ch < 0) continue;
                if (rb) {   // P's centre - child t's centre = -(hc / 2) (2 bit - 1) per axis
                    const float h = float(0.5 * hc);
                    const float ex = (t & 1) ? -h : h, ey = (t & 2) ? -h : h, ez = (t & 4) ? -h : h;
                    move_origin(ax[t], ex, ey, ez);
                    move_origin(ay[t], ex, ey, ez);
                }
                const cpx<float> sh = D.shift[size_t(D.child_shift[d * 8 + t]) * S + j];
                float4 *dst = Xi + (size_t(ch) * (2 * nf) + dl) * 2 * S + 2 * j;
                store4(dst, lin2(sh.x, ax[t], -sh.y, ay[t]));
                store4(dst + 1, lin2(sh.y, ax[t], sh.x, ay[t]));
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
// One term of the sum over the quadrature nodes.  FP32: compensated (Kahan) addition, since the terms
// (-lambda_k)^n b_k^m alternate in sign and cancel strongly at high degree; double-floats carry their own.
__device__ __forceinline__ void node_term(df2 &sum, df2 &, dfl c, df2 b) { macc(sum, c, b); }
__device__ __forceinline__ void node_term(float2 &sum, float2 &comp, float c, float2 b) {
    const float2 v = fma2(dup(c), b, neg2(comp)), t = add2(sum, v);
    comp = sub2(sub2(t, sum), v);
    sum = t;
}
__device__ __forceinline__ void node_term(f4 &sum, f4 &comp, float c, f4 b) {
    node_term(sum.a, comp.a, c, b.a);
    node_term(sum.b, comp.b, c, b.b);
}

// One box per block, kc quadrature nodes at a time (all of them in FP32), umax wave-pair units at most.
template <typename T, bool COL>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 3 : 5)
    k_x2l(int b0, DevTables<T> D, const float4 *Xi, cpx<T> *L, int f0, int nf, int kc, int umax, int mirror) {
    using V = typename Quad<T>::V;
    constexpr int N = Quad<T>::N, SH = Quad<T>::SH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p), s = D.s, S = D.S, P1 = p + 1, NS = a_stride(p);
    const Planes<T> Lf{reinterpret_cast<float4 *>(smem_raw), nc};   // the frame's sums
    // b+ + b- and b+ - b- per (node, m)
    const Planes<T> Bs{Lf.p + 2 * N * nc, kc * NS}, Bd{Bs.p + 2 * N * kc * NS, kc * NS};
    // per unit (waves t and M_k/2 - t of a node): sums and differences of the two waves' real and imaginary
    // parts, UQ[direction][re +, re -, im +, im -][unit][N]
    float4 *UQ = Bd.p + 2 * N * kc * NS;
    const int us = N * umax;
    const Planes<T> Tm{Bs.p, nc};   // rotation scratch over the B rows and the units (node_chunk leaves room)
    cpx<T> *dst = L + size_t(b) * kSets * nc;
    for (int f = f0; f < f0 + nf; ++f) {
        const float4 *in = Xi + (size_t(b) * (2 * nf) + 2 * (f - f0)) * 2 * N * S;
        for (int k0 = 0; k0 < s; k0 += kc) {
            const int kn = min(kc, s - k0);
            const int ub = D.u_start[k0], un = D.u_start[k0 + kn] - ub;
            __syncthreads();
            for (int e = threadIdx.x; e < 2 * N * un; e += blockDim.x) {   // (unit, direction, pr)
                const int pr = e & (N - 1), dir = (e >> SH) & 1, u = e >> (SH + 1);
                const int4 ui = D.u_info[ub + u];
                const int j0 = ui.y, H = ui.z, t = ui.w;
                const bool pair = t > 0 && 2 * t != H;
                const float4 *w = in + dir * 2 * N * S + pr;
                V ax, ay, bx = zero<V>(), by = bx;
                get(w[2 * N * (j0 + t)], ax);
                get(w[2 * N * (j0 + t) + N], ay);
                if (pair) {
                    get(w[2 * N * (j0 + H - t)], bx);
                    get(w[2 * N * (j0 + H - t) + N], by);
                }
                float4 *q = UQ + 4 * dir * us + N * u + pr;
                q[0] = put(ax + bx);
                q[us] = put(ax - bx);
                q[2 * us] = put(ay + by);
                q[3 * us] = put(ay - by);
            }
            __syncthreads();
            // b_k^m = sum_{j < M_k/2} (I_j + (-1)^m conj I_j) e^{-i m a_j}
            //       = 2 sum_j Re(I_j) e^{-i m a_j}      (m even)
            //       = 2i sum_j Im(I_j) e^{-i m a_j}     (m odd; the factor i is applied below)
            // With e^{-i m (pi - a)} = (-1)^m conj(e^{-i m a}), a wave pair adds
            // (v + (-1)^m v') cos(m a) - i (v - (-1)^m v') sin(m a): even m take the
            // sum and difference of the real parts, odd m those of the imaginary parts.
            // With `mirror` an item is node ka and its mirror kn - 1 - ka: the nodes' wave counts grow with k, so
            // the sums over two mirrored nodes are about equally long; otherwise one node (few items).
            const int items = (mirror ? (kn + 1) >> 1 : kn) * P1;
            for (int e = threadIdx.x; e < N * items; e += blockDim.x) {
                const int pr = e & (N - 1), r = e >> SH, ka = r / P1, m = r - ka * P1;
                for (int h = 0; h <= mirror; ++h) {
                    const int kk = h ? kn - 1 - ka : ka, k = k0 + kk;
                    if (h && kk == ka) break;
                    const int j0 = D.k_start[k], Mk = 2 * (D.k_start[k + 1] - j0);
                    const int u0 = D.u_start[k] - ub, u1 = D.u_start[k + 1] - ub;
                    const int mm = m % Mk;
                    const cpx<T> *rt = D.roots + 2 * j0;
                    const float4 *xp = UQ + ((m & 1) ? 3 : 0) * us + pr, *yp = UQ + ((m & 1) ? 2 : 1) * us + pr;
                    V bpx = zero<V>(), bpy = bpx, bmx = bpx, bmy = bpx;
                    int idx = 0;
                    for (int u = u0; u < u1; ++u) {
                        const cpx<T> z = rt[idx];
                        V a, c, a2, c2;
                        get(xp[N * u], a);
                        get(yp[N * u], c);
                        get(xp[4 * us + N * u], a2);
                        get(yp[4 * us + N * u], c2);
                        macc(bpx, z.x, a);
                        macc(bpy, neg1(z.y), c);
                        macc(bmx, z.x, a2);
                        macc(bmy, neg1(z.y), c2);
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
            for (int e = threadIdx.x; e < N * nc; e += blockDim.x) {
                const int pr = e & (N - 1), i = e >> SH, n = deg_of(i), m = i - tri(n, 0);
                const Planes<T> B = ((n + m) & 1) ? Bd : Bs;
                V x = zero<V>(), y = x, cx = x, cy = x;
                if (k0) {
                    x = Lf.x(pr, i);
                    y = Lf.y(pr, i);
                }
                const T *c = D.x2l_c + size_t(k0) * nc + i;
                for (int kk = 0; kk < kn; ++kk, c += nc) {
                    node_term(x, cx, *c, B.x(pr, kk * NS + m));
                    node_term(y, cy, *c, B.y(pr, kk * NS + m));
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
        if (f > 0) {   // back to world axes
            const T *rf = D.frot_bwd + size_t(f - 1) * D.frot_len;
            for (int e = threadIdx.x; e < N * nc; e += blockDim.x) {
                const int pr = e & (N - 1), i = e >> SH;
                rotate_z(rf, D.frot_off, i, pr, Lf.x(pr, i), Lf.y(pr, i), Tm);
            }
            __syncthreads();
        }
        for (int e = threadIdx.x; e < N * nc; e += blockDim.x) {
            const int pr = e & (N - 1), i = e >> SH;
            V x = Lf.x(pr, i), y = Lf.y(pr, i);
            if (f > 0) rotate_y<true, COL>(D.frot_bwd + size_t(f - 1) * D.frot_len, D.frot_off, i, pr, Tm, x, y);
            add_sets(dst, nc, pr, i, x, y);
        }
    }
}

// FP32 below order 12: single waves instead of wave pairs (no unit lookups and sums in the staging, which
// weigh more than the doubled angle sum when it has few orders), one set per item in the rotations, so that
// the 28 to 78 coefficients fill more lanes (15M-bead cube, p = 6: 4.6 ms against 5.4 for k_x2l, 256 systems,
// p = 8: 6.3 against 6.7).
__global__ void __launch_bounds__(256, 4)
    k_x2l_low(int b0, DevTables<float> D, const float4 *Xi, cpx<float> *L, int f0, int nf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = b0 + blockIdx.x;
    const int p = D.p, nc = ncoef(p), s = D.s, S = D.S, P1 = p + 1, SP = s * P1;
    float4 *PRe = reinterpret_cast<float4 *>(smem_raw);   // [S] + direction, real parts of sets 0..3
    float4 *PIm = PRe + S, *MRe = PIm + S, *MIm = MRe + S;
    // b+ + b- (Bs) and b+ - b- (Bd) per (node, m)
    const Planes<float> Bs{MIm + S, SP}, Bd{Bs.p + 2 * SP, SP};
    cpx<float> *Lf = reinterpret_cast<cpx<float> *>(Bd.p + 2 * SP);   // [4][nc]
    cpx<float> *Lw = Lf + kSets * nc, *Tm = Lw + kSets * nc;          // world sums, rotation scratch
    // (node, m) items at a stride of PA = 8 per node when p + 1 <= 8, so that a quarter-warp never
    // straddles two nodes (its wave loads are then broadcasts)
    const int PA = P1 <= 8 ? 8 : P1;
    for (int f = f0; f < f0 + nf; ++f) {
        __syncthreads();
        const float4 *sp = Xi + (size_t(b) * (2 * nf) + 2 * (f - f0)) * 2 * S, *sm = sp + 2 * S;
        for (int j = threadIdx.x; j < S; j += blockDim.x) {
            const float4 a = sp[2 * j], c = sp[2 * j + 1], d = sm[2 * j], e = sm[2 * j + 1];
            PRe[j] = a;
            PIm[j] = c;
            MRe[j] = d;
            MIm[j] = e;
        }
        __syncthreads();
        // b_k^m = 2 sum_j Re(I_j) e^{-i m a_j} (m even), 2i sum_j Im(I_j) e^{-i m a_j} (m odd)
        for (int ea = threadIdx.x; ea < s * PA; ea += blockDim.x) {
            const int k = ea / PA, m = ea - k * PA;
            if (m >= P1) continue;
            const int j0 = D.k_start[k], j1 = D.k_start[k + 1];
            const int Mk = 2 * (j1 - j0), mm = m % Mk;
            const cpx<float> *rt = D.roots + 2 * j0;
            const float4 *vp = (m & 1) ? PIm : PRe, *vm = (m & 1) ? MIm : MRe;
            f4 bpx = zero<f4>(), bpy = bpx, bmx = bpx, bmy = bpx;
            int idx = 0;
            for (int j = j0; j < j1; ++j) {
                const cpx<float> z = rt[idx];
                f4 a, c;
                get(vp[j], a);
                get(vm[j], c);
                macc(bpx, z.x, a);
                macc(bpy, -z.y, a);
                macc(bmx, z.x, c);
                macc(bmy, -z.y, c);
                idx += mm;
                if (idx >= Mk) idx -= Mk;
            }
            Bs.set(0, k * P1 + m, bpx + bmx, bpy + bmy);
            Bd.set(0, k * P1 + m, bpx - bmx, bpy - bmy);
        }
        __syncthreads();
        // L_n^m = i^m sum_k (-lambda_k)^n / sqrt((n-m)!(n+m)!) b_k^m, the - direction reflected
        for (int i = threadIdx.x; i < nc; i += blockDim.x) {
            const int n = deg_of(i), m = i - tri(n, 0);
            const Planes<float> B = ((n + m) & 1) ? Bd : Bs;
            f4 x = zero<f4>(), y = x, cx = x, cy = x;
            for (int k = 0; k < s; ++k) {
                const float c = D.x2l_c[size_t(k) * nc + i];
                node_term(x, cx, c, B.x(0, k * P1 + m));
                node_term(y, cy, c, B.y(0, k * P1 + m));
            }
            const float sg = ((m + (m & 1)) & 2) ? -2.f : 2.f;   // times 2 i^(m + (m & 1))
            x = scale2(sg, x);
            y = scale2(sg, y);
            Lf[i] = mk(x.a.x, y.a.x);
            Lf[nc + i] = mk(x.a.y, y.a.y);
            Lf[2 * nc + i] = mk(x.b.x, y.b.x);
            Lf[3 * nc + i] = mk(x.b.y, y.b.y);
        }
        __syncthreads();
        // back to world axes, added to the frames before
        if (f > 0) {
            const float *rf = D.frot_bwd + (f - 1) * D.frot_len;
            for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
                const int st = e / nc, i = e - st * nc, n = deg_of(i), m = i - tri(n, 0);
                const float *za = rf + D.frot_off[n];
                const float c = za[2 * m], sn = za[2 * m + 1];
                const cpx<float> v = Lf[e];
                Tm[e] = mk(mul_diff(c, v.x, sn, v.y), mul_diff(sn, v.x, -c, v.y));
            }
            __syncthreads();
            for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) {
                const int st = e / nc, i = e - st * nc, n = deg_of(i), m = i - tri(n, 0), q = n + 1;
                const float *o = rf + D.frot_off[n], *yre = o + 4 * q + m * q, *yim = yre + q * q;
                const cpx<float> *in = Tm + st * nc + tri(n, 0);
                float re = 0.f, im = 0.f;
                for (int k = (m + n) & 1; k < q; k += 2) re = fmaf(yre[k], in[k].x, re);
                if (m > 0)
                    for (int k = 1 + ((m + n) & 1); k < q; k += 2) im = fmaf(yim[k], in[k].y, im);
                const float c = o[2 * q + 2 * m], sn = o[2 * q + 2 * m + 1];
                const cpx<float> r = mk(mul_diff(c, re, sn, im), mul_diff(sn, re, -c, im));
                Lw[e] = f > f0 ? Lw[e] + r : r;
            }
        } else {
            for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) Lw[e] = Lf[e];
        }
    }
    // every thread adds the sums it formed
    cpx<float> *dst = L + size_t(b) * kSets * nc;
    for (int e = threadIdx.x; e < kSets * nc; e += blockDim.x) dst[e] += Lw[e];
}
static size_t smem_x2l_low(int p, int s, int S) {
    const int nc = ncoef(p);
    return sizeof(float4) * (4 * size_t(S) + 4 * size_t(s) * (p + 1)) + sizeof(cpx<float>) * 3 * kSets * nc;
}

// ---------------------------------------------------------------- driver
// Node chunks of M2X and X2L (equal ones): one for all nodes, split in double-floats until the block's shared
// memory (fixed bytes + per-node bytes + 256 bytes per wave-pair unit when units are staged) is at most
// 48 KB (56 KB with units), or until a chunk of X2L holds at most 200 (node, m) sums, below which its phases
// run out of threads.  Measured: X2L of the 1M-bead sphere (p = 16) 7.2 / 9.9 ms at 49 / 98 KB; of the 200k sphere at 9
// digits (p = 25) 13.9 / 8.5 / 7.5 ms at 56 / 72 / 100 KB; M2X there 11.4 / 5.3 / 5.5 ms at 30 / 48 / 60 KB.
// FP32 rows take half the bytes and its compensated node sum wants all nodes at once.
struct NodeChunk {
    int kc, umax;
    size_t smem;
};
template <typename T>
static NodeChunk node_chunk(const OpTables &h, bool stage_units) {
    constexpr int N = Quad<T>::N;
    const int nc = ncoef(h.p), NS = a_stride(h.p);
    NodeChunk c{};
    for (int nch = 1; nch <= h.s; ++nch) {
        const int kc = (h.s + nch - 1) / nch;
        int um = 0;
        for (int k0 = 0; k0 < h.s; k0 += kc) um = std::max(um, h.u_start[std::min(h.s, k0 + kc)] - h.u_start[k0]);
        // the rotation scratch (2 N nc float4) shares the memory of the rows and the staged units
        const size_t work = std::max(size_t(4 * N) * kc * NS + (stage_units ? size_t(8 * N) * um : 0), size_t(2 * N) * nc);
        c = NodeChunk{kc, um, sizeof(float4) * (size_t(2 * N) * nc + work)};
        if (!kIsDf<T> || c.smem <= (stage_units ? 56u : 48u) * 1024 || (stage_units && kc * (h.p + 1) <= 200)) break;
    }
    return c;
}

template <typename T>
int run_waves_t(Tree &t, const DevTables<T> &D, const cpx<T> *M, cpx<T> *L, int rb, cudaStream_t st) {
    using Mem = typename PairOf<T>::Mem;
    constexpr int N = Quad<T>::N;
    const int b2 = t.level_off[2], n2 = t.nbox - b2, p = D.p;
    const double *side = kIsDf<T> ? t.side_u : t.b_side;
    // all three frames in one pass, or (large trees, where the plane-wave buffers of six directions
    // would not fit) one frame per pass, each pass adding its frame's share into L (with profiling on, every
    // pass's launches are timed under their own stages)
    const int nf = t.x_frames;
    float4 *Xo = static_cast<float4 *>(t.Xo), *Xi = static_cast<float4 *>(t.Xi);
    const NodeChunk cm = node_chunk<T>(*t.tabs, false), cl = node_chunk<T>(*t.tabs, true);
    const bool col = y_by_column(sizeof(T), p);
    auto m2x = col ? k_m2x<T, true> : k_m2x<T, kIsDf<T>>;
    const bool low = !kIsDf<T> && p < 12;
    const size_t s_low = smem_x2l_low(p, D.s, D.S);
    if (low) RPY_TRY(set_smem(k_x2l_low, s_low));
    auto x2l = k_x2l<T, true>;
    const int one = N * cl.kc * (p + 1), mirror = kIsDf<T> && one > 160;
    const int xl_threads = even_threads(mirror ? N * ((cl.kc + 1) / 2) * (p + 1) : one);
    RPY_TRY(set_smem(m2x, cm.smem));
    RPY_TRY(set_smem(x2l, cl.smem));
    for (int f0 = 0; f0 < 3; f0 += nf) {
        prof_mark(t, RPY_STAGE_M2X, st);
        m2x<<<n2, even_threads(N * cm.umax), cm.smem, st>>>(b2, D, M, Xo, f0, nf, cm.kc);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
        prof_mark(t, RPY_STAGE_X2X, st);
        if (t.n_x2x_par > 0) {
            const dim3 g(t.n_x2x_par, 2 * nf);
            const Mem *xo = static_cast<const Mem *>(t.Xo);
            Mem *xi = static_cast<Mem *>(t.Xi);
            bool done = false;
            if constexpr (!kIsDf<T>) {
                // a producer warp stages the sources through shared memory by bulk copies
                if (D.S > 256 && D.S <= 480) {
                    const size_t sxx = x2x_tma_smem(D.S);
                    RPY_TRY(set_smem(k_x2x_tma, sxx));
                    k_x2x_tma<<<g, (D.S + 31) / 32 * 32 + 32, sxx, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf,
                                                                         side, Xo, Xi, f0, nf, rb, t.dev_status);
                    done = true;
                }
            }
            if (!done && rb)
                k_x2x4<T><<<g, even_threads(D.S), 0, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf, side, Xo, Xi,
                                                           f0, nf);
            else if (!done && t.n_x2x_par * 2 * nf < kX2XSmallGrid)
                k_x2x<T, 256, (sizeof(T) == 8 ? 2 : 4)><<<g, even_threads(2 * D.S), 0, st>>>(t.x2x_par, D, t.b_coll, t.b_child, t.b_leaf,
                                                                      xo, xi, f0, nf);
            else if (!done)
                k_x2x<T, 128, (sizeof(T) == 8 ? 5 : 7)><<<g, even_threads(2 * D.S, 128), 0, st>>>(t.x2x_par, D, t.b_coll, t.b_child,
                                                                           t.b_leaf, xo, xi, f0, nf);
            RPY_LAUNCHED(1);
            RPY_CHECK(cudaGetLastError());
        }
        prof_mark(t, RPY_STAGE_X2L, st);
        if constexpr (!kIsDf<T>) {
            if (low) k_x2l_low<<<n2, even_threads(D.s * (p + 1)), s_low, st>>>(b2, D, Xi, L, f0, nf);
        }
        if (!low) x2l<<<n2, xl_threads, cl.smem, st>>>(b2, D, Xi, L, f0, nf, cl.kc, cl.umax, mirror);
        RPY_LAUNCHED(1);
        RPY_CHECK(cudaGetLastError());
    }
    return RPY_OK;
}

template int run_waves_t<dfl>(Tree &, const DevTables<dfl> &, const cpx<dfl> *, cpx<dfl> *, int, cudaStream_t);
template int run_waves_t<float>(Tree &, const DevTables<float> &, const cpx<float> *, cpx<float> *, int, cudaStream_t);

}  // namespace rpy
