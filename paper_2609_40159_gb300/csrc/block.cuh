// Thread-block-local synchronisation-free solve of one system with several
// lanes per row, and the level-ordered one, used by the single-system block
// mode (solve.cu) and by the batched solve (batch.cu).  (One lane per row:
// strip.cuh.)
#pragma once

#include "rows.cuh"

namespace spt {

// Shared-memory layout (dynamic): ring of `ring` rows x KT solution values,
// ring of row tags (position of the row held by the slot, -1 = empty), ring
// of chunk tags, counters {ticket, completed prefix}.
template <class T, int KT> struct BlockSmem {
    volatile T *xr;
    volatile int *tag;
    volatile int *cdone;
    int *ctr;
};

__device__ __forceinline__ void fence_cta() { asm volatile("fence.sc.cta;" ::: "memory"); }
__device__ __forceinline__ void fence_acq_rel_cta() { asm volatile("fence.acq_rel.cta;" ::: "memory"); }

__device__ __forceinline__ int ld_relaxed_cta_smem(const int *p)
{
    int v;
    asm volatile("ld.relaxed.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"(smem_addr(p)) : "memory");
    return v;
}

// Solve one system with the whole thread block.  Rows are handled in
// processing order by row groups of `rpw` rows taken from a shared ticket; a
// group may start only when every group at least P positions earlier is
// complete, so that (with kc >= 2P ring groups) a ring slot is never reused
// while a running group can still need it.  Dependencies from the same
// group resolve through the warp loop, those up to P groups back through the
// ring tags, older ones are read from global memory (complete by the
// throttle).  Returns false when a wait gave up.
// DIRECT: the values are read in L's own order (the plan's copy in CSC order
// may be old).
template <class T, int KT, bool TR, bool DIRECT = false>
__device__ bool block_solve(const Sys<T> &A, const Rhs<T> &R, int rpw, int kc, int P,
                            const BlockSmem<T, KT> &sm, const Waiter &w, int withhold)
{
    const int lane = threadIdx.x & 31;
    const int lpr = 32 / rpw;
    const int g = lane / lpr, sl = lane & (lpr - 1);
    const unsigned gm = lpr == 32 ? 0xffffffffu : ((1u << lpr) - 1u);
    const int n = A.n;
    const int ring = kc * rpw;
    const int nchunks = (n + rpw - 1) / rpw;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(sm.ctr, 1);
        c = __shfl_sync(SPT_FULL_MASK, c, 0);
        if (c >= nchunks) return true;
        int ok = 1;
        if (lane == 0 && c - P >= 0) {
            WaitClock clk;
            while (*(volatile int *)(sm.ctr + 1) <= c - P) {
                if (clk.expired(w)) { ok = 0; break; }
            }
        }
        ok = __shfl_sync(SPT_FULL_MASK, ok, 0);
        if (!ok) return false;
        fence_cta();
        const int base = c * rpw;
        const int pos = base + g;
        const bool valid = pos < n;
        const int i = valid ? (TR ? n - 1 - pos : pos) : 0;
        const int a = valid ? RV<T, TR>::beg(A, i) : 0;
        const int e = valid ? RV<T, TR>::end(A, i) : 0;
        const unsigned leaders = __ballot_sync(SPT_FULL_MASK, valid && sl == 0);
        const int kt = R.k;  // <= KT
        T acc[KT];
#pragma unroll
        for (int r = 0; r < KT; ++r) acc[r] = T(0);
        if (!TR && valid && has_trow(A, i)) {
            const int tb = A.trp[i], te = A.trp[i + 1];
            for (int p = tb + sl; p < te; p += lpr) {
                const T tv = ldro(A.tv + p);
                const T *bb = R.b + (int64_t)tcol(A, p) * R.ld;
#pragma unroll
                for (int r = 0; r < KT; ++r)
                    if (r < kt) acc[r] -= tv * bb[r];
            }
        }
        int p = a + sl;
        unsigned fin = 0;
        bool failed = false;
        for (;;) {
            const bool open = valid && !((fin >> (g * lpr)) & 1u);
            if (open) {
                while (p < e) {
                    const int j = RV<T, TR>::col(A, p);
                    const int pj = order_pos<TR>(n, j);
                    const int cj = pj / rpw;
                    const T vv = DIRECT ? entry_val<T, TR>(A, p) : RV<T, TR>::val(A, p);
                    if (cj == c) {
                        const int gj = pj - base;
                        if (!((fin >> (gj * lpr)) & 1u)) break;
                        const volatile T *xx = sm.xr + (pj % ring) * KT;
#pragma unroll
                        for (int r = 0; r < KT; ++r)
                            if (r < kt) acc[r] += vv * xx[r];
                    } else if (cj <= c - P) {
                        const T *xx = R.x + (int64_t)j * R.ld;
#pragma unroll
                        for (int r = 0; r < KT; ++r)
                            if (r < kt) acc[r] += vv * xx[r];
                    } else {
                        const int slot = pj % ring;
                        if (sm.tag[slot] != pj) {
                            WaitClock clk;
                            while (sm.tag[slot] != pj) {
                                if (clk.expired(w)) { failed = true; break; }
                            }
                            if (failed) break;
                        }
                        fence_cta();
                        const volatile T *xx = sm.xr + slot * KT;
#pragma unroll
                        for (int r = 0; r < KT; ++r)
                            if (r < kt) acc[r] += vv * xx[r];
                    }
                    p += lpr;
                }
            }
            const bool ready = !open || p >= e || failed;
            const unsigned bal = __ballot_sync(SPT_FULL_MASK, ready);
            if (__any_sync(SPT_FULL_MASK, failed)) return false;
            const bool grp_ready = ((bal >> (g * lpr)) & gm) == gm;
            const bool newly = open && grp_ready;
            if (__any_sync(SPT_FULL_MASK, newly)) {
                T red[KT];
#pragma unroll
                for (int r = 0; r < KT; ++r) red[r] = acc[r];
                group_reduce<T, KT>(red, lpr);
                if (newly && sl == 0) {
                    const T d = DIRECT ? entry_val<T, TR>(A, TR ? a - 1 : e) : RV<T, TR>::diag(A, a, e);
                    const T *bb = R.b + (int64_t)i * R.ld;
                    T *xx = R.x + (int64_t)i * R.ld;
                    volatile T *xrr = sm.xr + (pos % ring) * KT;
#pragma unroll
                    for (int r = 0; r < KT; ++r)
                        if (r < kt) {
                            const T xv = (bb[r] - red[r]) / d;
                            xrr[r] = xv;
                            xx[r] = xv;
                        }
                    fence_cta();
                    if (i != withhold) sm.tag[pos % ring] = pos;
                }
            }
            fin |= __ballot_sync(SPT_FULL_MASK, newly && sl == 0);
            __syncwarp();
            if ((fin & leaders) == leaders) break;
        }
        // group complete: publish it and advance the completed prefix
        if (lane == 0) {
            fence_cta();
            sm.cdone[c % kc] = c;
            fence_cta();
            for (;;) {
                const int pf = *(volatile int *)(sm.ctr + 1);
                if (pf >= nchunks || sm.cdone[pf % kc] != pf) break;
                atomicCAS(sm.ctr + 1, pf, pf + 1);
            }
        }
    }
}

constexpr int kPreload = 16;  // entries of a row loaded before a group's turn

// acc[r] += v * src[r] for r < KT, with 16-byte loads when the layout allows
// (src is KT-aligned and KT*sizeof(T) is a multiple of 16).
template <class T, int KT>
__device__ __forceinline__ void axpy_vec(T v, const T *src, T (&acc)[KT])
{
    if constexpr (sizeof(T) * KT % 16 == 0) {
        constexpr int V = 16 / sizeof(T);
#pragma unroll
        for (int q = 0; q < KT / V; ++q) {
            const float4 f = reinterpret_cast<const float4 *>(src)[q];
            const T *t = reinterpret_cast<const T *>(&f);
#pragma unroll
            for (int u = 0; u < V; ++u) acc[q * V + u] += v * t[u];
        }
    } else {
#pragma unroll
        for (int r = 0; r < KT; ++r) acc[r] += v * src[r];
    }
}

template <class T, int KT>
__device__ __forceinline__ void store_vec(T *dst, const T (&v)[KT])
{
    if constexpr (sizeof(T) * KT % 16 == 0) {
        constexpr int V = 16 / sizeof(T);
#pragma unroll
        for (int q = 0; q < KT / V; ++q)
            reinterpret_cast<float4 *>(dst)[q] = *reinterpret_cast<const float4 *>(&v[q * V]);
    } else {
#pragma unroll
        for (int r = 0; r < KT; ++r) dst[r] = v[r];
    }
}

// In-group dependencies of a 32-row group, solved in registers: lane L holds
// the scaled candidates t_L = (b_L - sum over earlier groups) / L_LL and the
// coefficients C_Ls = L_Ls / L_LL of its in-group dependencies s < L (bits of
// dmask, coefficient coef(s)); x_L = t_L - sum_s C_Ls x_s.  Every step, each
// lane that still waits takes one dependency that is solved by now; a row is
// solved when it waits for none.  The number of steps is the group's longest
// chain counted in multiply-adds (about 5 for a band of 256, 12 for 64), where
// a sweep over the rows takes 31.
template <class T, int KT, class Coef>
__device__ __forceinline__ void group_list(T (&t)[KT], unsigned dmask, Coef coef)
{
    unsigned rem = dmask;
    unsigned done = __ballot_sync(SPT_FULL_MASK, rem == 0);
    while (done != SPT_FULL_MASK) {
        // (the smallest unsolved row waits for solved rows only)
        const unsigned av = rem & done;
        const bool hit = av != 0;
        const int s = hit ? __ffs(av) - 1 : 0;
        const T cf = coef(s);
#pragma unroll
        for (int r = 0; r < KT; ++r) {
            const T xs = __shfl_sync(SPT_FULL_MASK, t[r], s);
            // a select, not a zero coefficient: an overflowed x_s must not
            // turn independent rows into NaN
            t[r] = hit ? fma(-cf, xs, t[r]) : t[r];
        }
        rem &= hit ? ~(1u << s) : ~0u;
        done = __ballot_sync(SPT_FULL_MASK, rem == 0);
    }
}

// Block-local level-scheduled solve: the rows in level order (transpose:
// its reverse), cut into groups of at most 32 rows of ONE level (`groups`,
// dealt to the warps round-robin, one lane per row).  The rows of a level
// do not depend on each other, so a group needs no in-group sweep, and the
// groups of one level run at the same time; a group waits only until every
// group of the earlier levels is complete (a shared counter of completed
// groups reaches its `wait`: before that count is reached, only groups of
// earlier levels can complete, as later ones are still waiting).  Progress:
// the smallest incomplete group waits for smaller groups only, and its
// warp has completed all of its earlier (smaller) groups.
// Dependencies live in a shared-memory ring addressed by processing
// position (slot = position mod ring).  While a group of level l runs, only
// groups of level l write the ring, at positions below the level's end
// `lend`; so every position q >= lend - ring still holds its own value, and
// entries at positions below base - win (win = ring - (lend - base)) are
// read from global memory instead.  Values, ring slots and global copies of
// a group are written before its completion is counted (release), and a
// waiter acquires the count, so both reads see complete values.
template <class T, int KT, bool TR>
__device__ bool block_solve_levels(const Sys<T> &A, const Rhs<T> &R, const int32_t *__restrict__ perm,
                                   const int32_t *__restrict__ iperm, const LevelGroup *__restrict__ groups,
                                   int ngroups, int kc, int nwarps, const BlockSmem<T, KT> &sm,
                                   const Waiter &w, int withhold)
{
    constexpr int NP = kPreload;
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    if (wid >= nwarps) return true;
    const int n = A.n;
    const int ring = kc * 32;  // a power of two
    const int rmask = ring - 1;
    const int kt = R.k;
    const T *ring0 = const_cast<const T *>(sm.xr);
    // row at processing position q; processing position of row j
    auto row_at = [&](int q) { return chk_row(A, ldro(perm + (TR ? n - 1 - q : q))); };
    auto pos_of = [&](int j) {
        const int p = chk_index(ldro(iperm + j), 0, n, A.chk);
        return TR ? n - 1 - p : p;
    };
    // a warp's next group, its rows and their extents are loaded one group
    // ahead, and the group after it one more ahead, so that a group's
    // entries are one dependent load away when it starts
    LevelGroup gn{0, 0, 0, 0}, gnn{0, 0, 0, 0};
    int i_nx = 0, a_nx = 0, e_nx = 0;
    if (wid < ngroups) {
        gn = groups[wid];
        i_nx = row_at(gn.base + (lane < gn.cnt ? lane : 0));
        a_nx = RV<T, TR>::beg(A, i_nx);
        e_nx = RV<T, TR>::end(A, i_nx);
    }
    if (wid + nwarps < ngroups) gnn = groups[wid + nwarps];
    for (int g = wid; g < ngroups; g += nwarps) {
        const LevelGroup G = gn;
        const int i = i_nx, a = a_nx, e = e_nx;
        if (g + nwarps < ngroups) {
            gn = gnn;
            i_nx = row_at(gn.base + (lane < gn.cnt ? lane : 0));
            a_nx = RV<T, TR>::beg(A, i_nx);
            e_nx = RV<T, TR>::end(A, i_nx);
            if (g + 2 * nwarps < ngroups) gnn = groups[g + 2 * nwarps];
        }
        const int base = G.base;
        const bool valid = lane < G.cnt;
        const int pos = base + (valid ? lane : 0);
        // ---- 1. independent of the solution
        const int safe = TR ? a - 1 : e;  // position of the diagonal entry
        const T rinv = valid ? T(1) / RV<T, TR>::diag(A, a, e) : T(0);
        T acc[KT], bv[KT];
#pragma unroll
        for (int r = 0; r < KT; ++r) {
            acc[r] = T(0);
            bv[r] = (valid && r < kt) ? R.b[(int64_t)i * R.ld + r] : T(0);
        }
        if (!TR && valid && has_trow(A, i)) {
            for (int p = A.trp[i]; p < A.trp[i + 1]; ++p) {
                const T tv = ldro(A.tv + p);
                const T *bb = R.b + (int64_t)tcol(A, p) * R.ld;
#pragma unroll
                for (int r = 0; r < KT; ++r)
                    if (r < kt) acc[r] -= tv * bb[r];
            }
        }
        int jj[NP];
        T vv[NP];
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int q = a + u < e ? a + u : safe;
            jj[u] = pos_of(RV<T, TR>::col(A, q));
            vv[u] = RV<T, TR>::val(A, q);
        }
        // ring window of this group (see above)
        const int win = max(0, ring - (G.lend - base));
        const int lo = base - win;
        bool any_glob = false;
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const bool in = valid && a + u < e;
            const bool use = in && jj[u] >= lo;
            any_glob |= in && !use;
            // ring pass decided now: an entry in the ring keeps its value and
            // becomes its slot's offset; any other entry reads slot 0 with
            // weight 0 (global ones are applied separately, once complete)
            vv[u] = use ? vv[u] : T(0);
            jj[u] = use ? (jj[u] & rmask) * KT : 0;
        }
        const bool longrow = valid && e - a > NP;
        consume(rinv);
#pragma unroll
        for (int r = 0; r < KT; ++r) consume(bv[r]);
        // ---- 2. wait for every group of the earlier levels
        bool ok = true;
        {
            WaitClock clk;
            int done;
            while ((done = ld_relaxed_cta_smem(sm.ctr + 1)) < G.wait) {
                if (G.wait - done > nwarps) __nanosleep(200);
                if (clk.expired(w)) { ok = false; break; }
            }
            fence_acq_rel_cta();
        }
        if (!__all_sync(SPT_FULL_MASK, ok)) return false;
        // ---- 3. dependencies: ring, then global memory, then long rows' tails
#pragma unroll
        for (int u = 0; u < NP; ++u) axpy_vec<T, KT>(vv[u], ring0 + jj[u], acc);
        if (__any_sync(SPT_FULL_MASK, any_glob)) {
            for (int p = a; any_glob && p < e && p < a + NP; ++p) {
                const int j = RV<T, TR>::col(A, p);
                if (pos_of(j) < lo) {
                    const T v = RV<T, TR>::val(A, p);
                    const T *xx = R.x + (int64_t)j * R.ld;
#pragma unroll
                    for (int r = 0; r < KT; ++r)
                        if (r < kt) acc[r] += v * xx[r];
                }
            }
        }
        if (__any_sync(SPT_FULL_MASK, longrow)) {
            for (int p = a + NP; longrow && p < e; ++p) {
                const int j = RV<T, TR>::col(A, p);
                const int pj = pos_of(j);
                const T v = RV<T, TR>::val(A, p);
                if (pj >= lo) {
                    axpy_vec<T, KT>(v, ring0 + (pj & rmask) * KT, acc);
                } else {
                    const T *xx = R.x + (int64_t)j * R.ld;
#pragma unroll
                    for (int r = 0; r < KT; ++r)
                        if (r < kt) acc[r] += v * xx[r];
                }
            }
        }
        T t[KT];
#pragma unroll
        for (int r = 0; r < KT; ++r) t[r] = (bv[r] - acc[r]) * rinv;
        // ---- 4. publish: ring slot and global copy, then (release) the count
        if (valid) {
            store_vec<T, KT>(const_cast<T *>(sm.xr) + (pos & rmask) * KT, t);
            T *xx = R.x + (int64_t)i * R.ld;
#pragma unroll
            for (int r = 0; r < KT; ++r)
                if (r < kt) xx[r] = t[r];
        }
        const bool hold = __any_sync(SPT_FULL_MASK, valid && i == withhold);
        __syncwarp();
        if (lane == 0 && !hold) {
            fence_acq_rel_cta();
            atomicAdd(sm.ctr + 1, 1);
        }
    }
    return true;
}

template <class T, int KT>
__device__ __forceinline__ BlockSmem<T, KT> carve_block_smem(unsigned char *raw, int ring, int kc)
{
    BlockSmem<T, KT> sm;
    T *xr = reinterpret_cast<T *>(raw);
    sm.xr = xr;
    int *tag = reinterpret_cast<int *>(xr + (size_t)ring * KT);
    sm.tag = tag;
    sm.cdone = tag + ring;
    sm.ctr = tag + ring + kc;
    return sm;
}

// Fresh state for one system.
template <class T, int KT>
__device__ __forceinline__ void reset_block_smem(const BlockSmem<T, KT> &sm, int ring, int kc)
{
    for (int t = threadIdx.x; t < ring * KT; t += blockDim.x) sm.xr[t] = T(0);
    for (int t = threadIdx.x; t < ring; t += blockDim.x) sm.tag[t] = -1;
    for (int t = threadIdx.x; t < kc; t += blockDim.x) sm.cdone[t] = -1;
    if (threadIdx.x == 0) { sm.ctr[0] = 0; sm.ctr[1] = 0; }
}

}  // namespace spt
