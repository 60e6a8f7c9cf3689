// Row views of a system for the solve kernels: the forward solve reads L by
// rows (CSR), the transpose solve reads L by columns (CSC; the values from a
// copy gathered into CSC order before the solve, or through the map to L's
// own: entry_val).
#pragma once

#include "solve.cuh"

namespace spt {

// ------------------------------------------------------------- row views
template <class T, bool TR> struct RV;

// (chk_*: identity in the product build, bounds checks in SPTRSV_CHECKED)
template <class T> __device__ __forceinline__ int chk_row(const Sys<T> &A, int i)
{
    return chk_index(i, 0, A.n, A.chk);
}
template <class T> __device__ __forceinline__ int chk_pos(const Sys<T> &A, int p)
{
    return chk_index(p, 0, (int)A.nnz, A.chk);
}

template <class T> struct RV<T, false> {
    static __device__ __forceinline__ int beg(const Sys<T> &A, int i) { return ldro(A.rp + chk_row(A, i)); }
    static __device__ __forceinline__ int end(const Sys<T> &A, int i) { return ldro(A.rp + chk_row(A, i) + 1) - 1; }
    static __device__ __forceinline__ T diag(const Sys<T> &A, int, int e) { return ldro(A.v + chk_pos(A, e)); }
    static __device__ __forceinline__ int col(const Sys<T> &A, int p) { return chk_row(A, ldro(A.ci + chk_pos(A, p))); }
    static __device__ __forceinline__ T val(const Sys<T> &A, int p) { return ldro(A.v + chk_pos(A, p)); }
};

template <class T> struct RV<T, true> {
    static __device__ __forceinline__ int beg(const Sys<T> &A, int i) { return ldro(A.cp + chk_row(A, i)) + 1; }
    static __device__ __forceinline__ int end(const Sys<T> &A, int i) { return ldro(A.cp + chk_row(A, i) + 1); }
    static __device__ __forceinline__ T diag(const Sys<T> &A, int b, int) { return ldro(A.cv + chk_pos(A, b - 1)); }
    static __device__ __forceinline__ int col(const Sys<T> &A, int q) { return chk_row(A, ldro(A.crow + chk_pos(A, q))); }
    static __device__ __forceinline__ T val(const Sys<T> &A, int q) { return ldro(A.cv + chk_pos(A, q)); }
};

// Current value of entry p (the plan's CSC copy of the values is refreshed for
// other paths only).
template <class T, bool TR> __device__ __forceinline__ T entry_val(const Sys<T> &A, int p)
{
    return TR ? ldro(A.v + chk_pos(A, ldro(A.tmap + chk_pos(A, p)))) : RV<T, false>::val(A, p);
}

// Column of entry p of T (the rewritten right-hand side's extra terms).
template <class T> __device__ __forceinline__ int tcol(const Sys<T> &A, int p)
{
    return chk_row(A, ldro(A.tci + p));
}

template <class T>
__device__ __forceinline__ bool has_trow(const Sys<T> &A, int i)
{
    return A.tmask != nullptr && ((ldro(A.tmask + (i >> 5)) >> (i & 31)) & 1u);
}

// Position of a row in processing order (forward: i, transpose: n-1-i).
template <bool TR> __device__ __forceinline__ int order_pos(int n, int i) { return TR ? n - 1 - i : i; }

// Make a loaded value "used" here: the load must complete before this
// point, so that a warp waiting for its turn holds all of its operands
// instead of stalling on them after the turn comes.
__device__ __forceinline__ void consume(int v) { asm volatile("" ::"r"(v)); }
__device__ __forceinline__ void consume(float v) { asm volatile("" ::"f"(v)); }
__device__ __forceinline__ void consume(double v) { asm volatile("" ::"d"(v)); }

// Row of nonzero p inside a 32-row chunk whose lanes hold the chunk's row
// starts (s = row_ptr[r0 + lane], lanes >= nrows unused): the last lane l <
// nrows with s_l <= p, by a five-step binary search over the lanes.
__device__ __forceinline__ int row_in_chunk(int s, int nrows, int p)
{
    int lo = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        const int cand = lo + step;
        const int v = __shfl_sync(SPT_FULL_MASK, s, cand & 31);
        if (cand < nrows && v <= p) lo = cand;
    }
    return lo;
}

// Product of two rows of k elements, summed in order; V elements a load.
template <class T, int V> __device__ __forceinline__ T row_dot(const T *a, const T *b, int k)
{
    struct alignas(sizeof(T) * V) Vec { T v[V]; };
    T s = T(0);
    for (int q = 0; q < k; q += V) {
        const Vec x = *reinterpret_cast<const Vec *>(a + q), y = *reinterpret_cast<const Vec *>(b + q);
#pragma unroll
        for (int u = 0; u < V; ++u) s += x.v[u] * y.v[u];
    }
    return s;
}

// The most elements a load (16 bytes at most) that rows of k elements at
// multiples of ld elements from a and b allow.
template <class T> __host__ __device__ __forceinline__ int row_vec(const T *a, const T *b, int64_t ld, int k)
{
    const size_t bits = reinterpret_cast<size_t>(a) | reinterpret_cast<size_t>(b) |
                        (size_t)ld * sizeof(T) | (size_t)k * sizeof(T);
    int v = 16 / (int)sizeof(T);
    while (v > 1 && bits % ((size_t)v * sizeof(T)) != 0) v >>= 1;
    return v;
}

template <class T, int KT>
__device__ __forceinline__ void group_reduce(T (&acc)[KT], int lpr)
{
    for (int o = lpr >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < KT; ++r) acc[r] += shfl_xor(acc[r], o);
}

// Column sweep over the dependencies INSIDE a group of 32 rows (one row per
// lane, in processing order).  dmask: bit s is set when this lane's row
// depends on row s of the group; coef[s*32 + lane] holds that coefficient
// (per-warp table).  Steps visit only rows that some lane depends on: lane s
// forms its solution candidate (b - acc) / L_ii -- final, since all of its
// own in-group dependencies are earlier rows -- and broadcasts it (warp
// shuffles for up to 4 right-hand sides, a per-warp shared buffer for more);
// every lane that depends on row s adds coef * x_s.
template <class T, int KT>
__device__ __forceinline__ void group_sweep(unsigned dmask, const T *coef, T *xbuf, T (&acc)[KT],
                                            const T (&bv)[KT], T rinv)
{
    const int lane = threadIdx.x & 31;
    unsigned need = __reduce_or_sync(0xffffffffu, dmask);
    while (need) {
        const int s = __ffs(need) - 1;
        need &= need - 1;
        const bool hit = (dmask >> s) & 1u;
        const T c = hit ? coef[s * 32 + lane] : T(0);
        if (KT <= 4) {
#pragma unroll
            for (int r = 0; r < KT; ++r) {
                const T t = (bv[r] - acc[r]) * rinv;
                const T xs = __shfl_sync(0xffffffffu, t, s);
                if (hit) acc[r] += c * xs;
            }
        } else {
            if (lane == s) {
#pragma unroll
                for (int r = 0; r < KT; ++r) xbuf[r] = (bv[r] - acc[r]) * rinv;
            }
            __syncwarp();
            if (hit) {
#pragma unroll
                for (int r = 0; r < KT; ++r) acc[r] += c * xbuf[r];
            }
            __syncwarp();
        }
    }
}

}  // namespace spt
