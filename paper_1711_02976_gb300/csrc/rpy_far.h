// Shared by the far field's translation units (rpy_fmm.cu: expansions and evaluation; rpy_waves.cu: plane waves).
#pragma once

#include <algorithm>

#include "rpy_internal.h"

namespace rpy {

__device__ __forceinline__ int deg_of(int idx) {
    int n = int((sqrtf(8.0f * idx + 1.0f) - 1.0f) * 0.5f);
    while (tri(n + 1, 0) <= idx) ++n;
    while (tri(n, 0) > idx) --n;
    return n;
}

// Lanes per point: columns m and P - m share a lane, so every lane runs P + 2
// recurrence steps (a column per lane would leave the lanes of high m idle
// while column 0 runs P + 1 steps, and lanes above P idle altogether; the
// arithmetic pipes are charged per warp instruction).
__host__ __device__ constexpr int harm_lanes(int P) { return P / 2 + 1; }

// Raises a kernel's dynamic shared-memory limit, once per device and kernel.
int raise_smem(const void *kernel, size_t bytes);
template <typename K>
inline int set_smem(K kernel, size_t bytes) {
    return raise_smem(reinterpret_cast<const void *>(kernel), bytes);
}

// The fewest warps that keep the number of rounds of `most` threads over the items, so that the last
// round is not left nearly empty.
inline int even_threads(int items, int most = 256) {
    const int rounds = (items + most - 1) / most;
    return std::max(64, ((items + rounds - 1) / rounds + 31) / 32 * 32);
}

// Two charge sets of one value in a packed operand (V), and in memory.
template <typename T> struct PairOf;
template <> struct PairOf<float> {
    using V = float2;
    using Mem = float2;
};
template <> struct PairOf<dfl> {
    using V = df2;
    using Mem = float4;
};

// M2X, X2X and X2L of one matvec: M -> L (added), through t.Xo and t.Xi
template <typename T>
int run_waves_t(Tree &t, const DevTables<T> &D, const cpx<T> *M, cpx<T> *L, int rb, cudaStream_t st);

// Upward and downward shifts, level by level
template <typename T>
int run_m2m_t(Tree &t, const DevTables<T> &D, cpx<T> *M, int rb, cudaStream_t st);
template <typename T>
int run_l2l_t(Tree &t, const DevTables<T> &D, cpx<T> *L, int rb, cudaStream_t st);

}  // namespace rpy
