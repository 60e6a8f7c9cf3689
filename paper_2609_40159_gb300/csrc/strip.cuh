// Strips: a system cut into groups of 32 rows in processing order (row order;
// transpose: last row first), solved in order by the warps of one thread block
// in turn, one lane per row.
//
// What bounds such a solve is the dependent chain of groups, so everything of
// a group that does not depend on the solution is prepared before it, into one
// block of bytes: by the plan what each entry is to its group, before every
// solve by the whole GPU the values in the order they are read, reciprocal
// diagonals and the inverse of the group's triangle (strip.cu).  A warp holds
// all of that in registers when its turn comes.
// Measured on a band of 64 (60,001 rows, FP32, one column a block): 3,400
// cycles a group with the values gathered by the solve and a sweep over the 32
// rows, 1,540 with one warp walking all groups from a shared-memory pipeline
// (a lone warp issues an instruction in four cycles), 790 here, the refresh
// included; the sum of 28 + 16 coefficients a row, the triangle and the
// hand-over from warp to warp (two shared-memory round trips) are left.
#pragma once

#include <cfloat>

#include "block.cuh"

namespace spt {

// First 16 bytes of a block.
struct StripHead {
    uint32_t bits;   // staged older dependencies of the busiest row (5), on the previous group (5), kind (2),
                     // steps (5), tail (1), far (1)
    uint32_t dense;  // 1: no inverse, the triangle itself is staged (refreshed by every solve)
    uint32_t unused[2];
};
__host__ __device__ constexpr uint32_t strip_bits(int na, int nb, uint32_t kind, int steps, bool tail, bool far)
{
    return (uint32_t)na | (uint32_t)nb << 5 | kind << 10 | (uint32_t)steps << 12 | (uint32_t)tail << 17 |
           (uint32_t)far << 18;
}

// A block after its head.  A quad is four entries of each of the 32 rows.
//   codes   per quad of dependencies (older ones first), 8 bytes a row: rows of
//           the ring of solutions; `ring`: a row of zeros (no dependency, or one
//           too old for the ring)
//   far     if some are too old: per quad, 16 bytes a row: distances of those
//           before the group's first position, else 0
//   words   4 bytes a row each: steps: the rows that four steps take, 8 bits
//           each; inverse: mask of the group's rows that the row depends on;
//           tail: first entry that is not staged
//   rinv    reciprocal diagonals
//   values  per quad: of the dependencies, then of the triangle (four steps, or
//           four columns of the inverse; FP64: the first two values of all rows,
//           then the other two)
struct StripBits {
    int na, nb, qa, qb, steps;
    uint32_t kind;
    bool tail, far;
    __host__ __device__ __forceinline__ explicit StripBits(uint32_t b)
        : na(b & 31), nb((b >> 5) & 31), qa((na + 3) / 4), qb((nb + 3) / 4), steps((b >> 12) & 31),
          kind((b >> 10) & 3), tail((b >> 17) & 1), far((b >> 18) & 1)
    {
    }
    __host__ __device__ __forceinline__ int staged() const { return qa + qb; }
    __host__ __device__ __forceinline__ int tri_words() const
    {
        return kind == kTriSteps ? (steps + 3) / 4 : kind == kTriInverse ? 1 : 0;
    }
    __host__ __device__ __forceinline__ int tri_quads() const
    {
        return kind == kTriSteps ? (steps + 3) / 4 : kind == kTriInverse ? 8 : 0;
    }
    __host__ __device__ __forceinline__ int at_words() const { return 16 + (far ? 768 : 256) * staged(); }
    __host__ __device__ __forceinline__ int at_rinv() const { return at_words() + 128 * (tri_words() + (tail ? 1 : 0)); }
    __host__ __device__ __forceinline__ int at_values(int w) const { return at_rinv() + 32 * w; }
    __host__ __device__ __forceinline__ int bytes(int w) const
    {
        return at_values(w) + 128 * w * (staged() + tri_quads());
    }
};

// Plan-time tables of one direction of several systems, all groups in one list
// (a launch for each of many small systems costs more than its work).
struct StripSrc {
    const int32_t *ptr, *idx;  // CSR row pointers and columns, or CSC column pointers and rows
    int64_t g0, e0;            // its first group and entry in the lists
    int32_t n;
};
struct StripBuild {
    const StripSrc *src;  // device, nsrc entries, by g0
    int32_t nsrc;
    int64_t ng;           // groups of all
    int32_t ring_most;
    bool trans, f64;
    int32_t *far;         // by system: the farthest dependency, from which its ring follows
    uint32_t *bits;       // by group
    int32_t *units;       // by group: size of its block (16 bytes)
    uint32_t *ofs;        // the sizes' prefix sums (ng + 1)
    int64_t *total;
    int32_t *stage;       // the most shared memory that the refresh of a group takes
};
__host__ __device__ inline int32_t strip_ring(int32_t far, int32_t most)
{
    const int32_t want = (far + 31) / 32 * 32 + 32;  // (distances count from the group's first position)
    return want < kStripRingLeast ? kStripRingLeast : want > most ? most : want;
}
// Everything but the blocks, then these (ecode: by entry of the list).
cudaError_t strip_sizes(const StripBuild &B, cudaStream_t s, const Scratch *from);
cudaError_t strip_tables(const StripBuild &B, const uint32_t *ofs, unsigned char *blocks, uint16_t *ecode,
                         cudaStream_t s);

// The refresh before a solve: of one system, or of every group of a batch
// (chunks: (system, 32 * group); stage: the most of its systems' Strips).  Of a single system: resets the control block
// for the solve that follows too (small systems wait for the host's launches).
template <class T>
cudaError_t strip_stage(const Sys<T> &A, const Strips &V, PlanCtl *ctl, bool trans, cudaStream_t s);
template <class T>
cudaError_t strip_stage_batch(const BatchMat *mats, const RowChunk *chunks, int64_t nchunks, int stage, bool trans,
                              cudaStream_t s);

// The system again, every entry on its own: with an infinite or NaN solution
// coefficients of 0 and products with an inverse spread it to rows that do not
// depend on it.
template <class T, int KT, bool TR>
__device__ __noinline__ bool strip_again(const Sys<T> &A, const Rhs<T> &R, unsigned char *smem, const Waiter &w,
                                         int withhold)
{
    constexpr int kc = 16, rpw = 16;
    BlockSmem<T, KT> sm = carve_block_smem<T, KT>(smem, kc * rpw, kc);
    reset_block_smem<T, KT>(sm, kc * rpw, kc);
    __syncthreads();
    return (int)(threadIdx.x >> 5) < 4 ? block_solve<T, KT, TR, true>(A, R, rpw, kc, kc / 2, sm, w, withhold) : true;
}

// Shared-memory loads by 32-bit address.
__device__ __forceinline__ void lds(unsigned a, float (&v)[1])
{
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[0]) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds(unsigned a, float (&v)[2])
{
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds(unsigned a, float (&v)[4])
{
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void lds(unsigned a, double (&v)[1])
{
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v[0]) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds(unsigned a, double (&v)[2])
{
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds(unsigned a, double (&v)[4])
{
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a) : "memory");
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2+16];" : "=d"(v[2]), "=d"(v[3]) : "r"(a) : "memory");
}

// Shared memory of a block that solves KT columns: the ring and its row of
// zeros, a table of coefficients for each warp (FP64: and the rows that steps
// take), the count of solved groups.
constexpr int kStripWarps = 8;   // of a single system's block
template <class T> constexpr int kStripTable = sizeof(T) == 8 ? 1024 + 128 : 1024;
__host__ __device__ inline size_t strip_ring_bytes(int ring, int KT, int w) { return (size_t)(ring + 4) * KT * w; }
inline size_t strip_smem(int ring, int KT, bool f64, int warps)
{
    const int w = f64 ? 8 : 4;
    return strip_ring_bytes(ring, KT, w) + (size_t)warps * (f64 ? kStripTable<double> : kStripTable<float>) * w + 16;
}

// In-order solve over the strips: the groups are dealt to `nwarps` warps
// round-robin and completed in order.  Group c:
//   1. before any wait: loads its block (coalesced loads whose addresses depend
//      on the group's offset and head alone, loaded two and one groups ahead),
//      its right-hand sides, and applies the dependencies older than the ring
//      (global memory);
//   2. waits for the groups <= c-2 and applies their solutions from the ring
//      while group c-1 is being solved;
//   3. waits for group c-1, applies its solutions, resolves the dependencies
//      inside the group and publishes: ring, count of groups (release), global
//      copy.
// Raises *bad when a solution is not finite (products with a coefficient of 0
// then spread it to rows that do not depend on it: the caller solves the
// system again, entry by entry).
// Ring slot safety: with kc = ring / 32, the slot of group cj is rewritten by
// group cj + kc only after every group < cj + kc is complete, i.e. after every
// reader of cj finished.  Global reads: the warp that solved group g stores
// g's global x (after publishing g) before it publishes its next group, g +
// nwarps.  A warp starting group c has itself completed c - nwarps, after
// acquiring the completion of every group < c - nwarps, which covers the
// global x of every group <= c - 2 nwarps - 1; entries at least kc >= 2 nwarps
// + 1 groups back are therefore read from global memory before the warp waits.
template <class T, int KT, bool TR>
__device__ __forceinline__ bool strip_turns(const Sys<T> &A, const Strips &V, const Rhs<T> &R, int nwarps,
                                            unsigned char *smem, int *ctr, int *bad, const Waiter &w, int withhold)
{
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int NA = F64 ? 2 : 4, NB = 3;  // quads of dependencies held in registers
    constexpr int W = (int)sizeof(T);
    constexpr int NT = F64 ? 2 : 8;  // quads of the triangle held in registers
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = A.n, ng = (n + 31) / 32, ring = V.ring;
    const int lim = ring - 32;  // farthest distance that the ring holds
    const int kt = R.k;
    T *ring0 = reinterpret_cast<T *>(smem);
    const unsigned ringa = smem_addr(smem);
    T *tab = reinterpret_cast<T *>(smem + strip_ring_bytes(ring, KT, W)) + (size_t)wid * kStripTable<T>;
    uint32_t *tabid = reinterpret_cast<uint32_t *>(tab + 1024);
    const uint32_t zeros = (uint32_t)ring * 0x10001u;
    auto block_of = [&](uint32_t o) { return V.blocks + (size_t)o * 16u; };
    auto quad = [&](const T *vals, int q, T (&v)[4]) {
        if constexpr (F64) {
            const double2 p0 = __ldg(reinterpret_cast<const double2 *>(vals) + q * 64 + lane);
            const double2 p1 = __ldg(reinterpret_cast<const double2 *>(vals) + q * 64 + 32 + lane);
            v[0] = p0.x; v[1] = p0.y; v[2] = p1.x; v[3] = p1.y;
        } else {
            const float4 p = __ldg(reinterpret_cast<const float4 *>(vals) + q * 32 + lane);
            v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
        }
    };
    uint32_t o1 = 0, o2 = 0;  // offsets of this group's block and of the warp's next
    uint2 hw = make_uint2(0u, 0u);
    if (wid < ng) {
        o1 = ldro(V.ofs + wid);
        hw = __ldg(reinterpret_cast<const uint2 *>(block_of(o1)));
    }
    if (wid + nwarps < ng) o2 = ldro(V.ofs + wid + nwarps);
    for (int c = wid; c < ng; c += nwarps) {
        const unsigned char *blk = block_of(o1);
        const StripBits h(hw.x);
        const bool dense = hw.y != 0u;
        o1 = o2;
        if (c + nwarps < ng) hw = __ldg(reinterpret_cast<const uint2 *>(block_of(o1)));
        if (c + 2 * nwarps < ng) o2 = ldro(V.ofs + c + 2 * nwarps);
        const int staged = h.staged(), base = c * 32, pos = base + lane;
        const bool valid = pos < n;
        const int i = valid ? (TR ? n - 1 - pos : pos) : (TR ? n - 1 : 0);
        const int slot0 = base % ring;
        // ---- 1. independent of the solution
        const T *vals = reinterpret_cast<const T *>(blk + h.at_values(W));
        uint2 cd[NA + NB];  // byte offsets in the ring, 16 bits each
        T vv[NA + NB][4];
#pragma unroll
        for (int q = 0; q < NA + NB; ++q) {
            cd[q] = make_uint2(zeros, zeros);
#pragma unroll
            for (int u = 0; u < 4; ++u) vv[q][u] = T(0);
            if (q < NA ? q < h.qa : q - NA < h.qb) {
                const int at = q < NA ? q : h.qa + q - NA;
                cd[q] = __ldg(reinterpret_cast<const uint2 *>(blk + 16) + at * 32 + lane);
                quad(vals, at, vv[q]);
            }
        }
        T tri[NT][4];
        uint32_t ids[2] = {0u, 0u};
        const uint32_t *words = reinterpret_cast<const uint32_t *>(blk + h.at_words()) + lane;
#pragma unroll
        for (int q = 0; q < NT; ++q)
            if (q < h.tri_quads()) quad(vals, staged + q, tri[q]);
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (q < h.tri_words()) ids[q] = __ldg(words + 32 * q);
        const T rinv = __ldg(reinterpret_cast<const T *>(blk + h.at_rinv()) + lane);
        T acc[KT], bv[KT];
#pragma unroll
        for (int r = 0; r < KT; ++r) {
            acc[r] = T(0);
            bv[r] = (valid && r < kt) ? R.b[(int64_t)i * R.ld + r] : T(0);
        }
        if (__builtin_expect(A.tmask != nullptr, 0) && !TR && valid && has_trow(A, i)) {
            for (int p = A.trp[i]; p < A.trp[i + 1]; ++p) {
                const T tv = ldro(A.tv + p);
                const T *bb = R.b + (int64_t)tcol(A, p) * R.ld;
#pragma unroll
                for (int r = 0; r < KT; ++r)
                    if (r < kt) acc[r] -= tv * bb[r];
            }
        }
        auto add_global = [&](T v, int pj) {
            const T *xx = R.x + (int64_t)chk_row(A, TR ? n - 1 - pj : pj) * R.ld;
#pragma unroll
            for (int r = 0; r < KT; ++r)
                if (r < kt) acc[r] += v * xx[r];
        };
        if (__builtin_expect(h.far, 0)) {
            for (int q = 0; q < staged; ++q) {
                const int4 d = __ldg(reinterpret_cast<const int4 *>(blk + 16 + 256 * staged) + q * 32 + lane);
                T v[4];
                quad(vals, q, v);
                if (d.x) add_global(v[0], base - d.x);
                if (d.y) add_global(v[1], base - d.y);
                if (d.z) add_global(v[2], base - d.z);
                if (d.w) add_global(v[3], base - d.w);
            }
        }
        int ta = 0, te = 0;  // the row's entries that are not staged
        if (__builtin_expect(h.tail, 0)) {
            ta = (int)__ldg(words + 32 * h.tri_words());
            te = valid ? RV<T, TR>::end(A, i) : 0;
            for (int p = ta; p < te; ++p) {
                const int pj = order_pos<TR>(n, RV<T, TR>::col(A, p));
                if (base - pj > lim) add_global(entry_val<T, TR>(A, p), pj);
            }
        }
        auto tail_pass = [&](int near, int far) {  // distances [near, far]
            for (int p = ta; p < te; ++p) {
                const int d = base - order_pos<TR>(n, RV<T, TR>::col(A, p));
                if (d >= near && d <= far) {
                    const int r = slot0 - d;
                    axpy_vec<T, KT>(entry_val<T, TR>(A, p), ring0 + (r < 0 ? r + ring : r) * KT, acc);
                }
            }
        };
        // steps beyond those in registers (FP64), or the triangle itself: in
        // shared memory, [step or column][row]
        if ((F64 && h.kind == kTriSteps && h.steps > 4 * NT) || (h.kind == kTriInverse && dense)) {
            for (int q = 0; q < h.tri_quads(); ++q) {
                T v[4];
                quad(vals, staged + q, v);
#pragma unroll
                for (int u = 0; u < 4; ++u) tab[(4 * q + u) * 32 + lane] = v[u];
            }
            if (F64)
                for (int q = 2; q < h.tri_words(); ++q) tabid[32 * q + lane] = __ldg(words + 32 * q);
        }
        const bool hold = __any_sync(SPT_FULL_MASK, valid && i == withhold);
        // (everything is at hand before the wait: what the compiler moved
        // behind it would be on the chain)
        consume(rinv);
#pragma unroll
        for (int r = 0; r < KT; ++r) consume(bv[r]);
#pragma unroll
        for (int q = 0; q < NA + NB; ++q) {
            cd[q].x *= KT * W;
            cd[q].y *= KT * W;
            consume((int)cd[q].x);
            consume((int)cd[q].y);
#pragma unroll
            for (int u = 0; u < 4; ++u) consume(vv[q][u]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) consume((int)ids[q]);
        // every lane polls the count of solved groups; a warp two or more
        // groups from its turn sleeps between polls, so that waiting warps
        // leave the issue slots to the working ones
        auto wait_done = [&](int upto) {
            // (one load of a warp is not one moment: no vote inside the loop)
            WaitClock clk;
            int done;
            bool good = true;
            while ((done = ld_acquire_cta_smem(ctr)) < upto) {
                if (upto - done > 1) __nanosleep(64);
                if (clk.expired(w)) { good = false; break; }
            }
            return __all_sync(SPT_FULL_MASK, good) != 0;
        };
        auto ring_quad = [&](const uint2 cq, const T (&v)[4], int cnt) {
            const unsigned o[4] = {cq.x & 0xffffu, cq.x >> 16, cq.y & 0xffffu, cq.y >> 16};
            if constexpr (F64) {
                // one by one, as each multiply-add takes 64 cycles
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (u < cnt) axpy_vec<T, KT>(v[u], reinterpret_cast<const T *>(smem + o[u]), acc);
            } else {
                T f[4][KT];
#pragma unroll
                for (int u = 0; u < 4; ++u) lds(ringa + o[u], f[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int r = 0; r < KT; ++r) acc[r] = fma(v[u], f[u][r], acc[r]);
            }
        };
        // ---- 2. groups <= c-2
        if (!wait_done(c - 1)) return false;
#pragma unroll
        for (int q = 0; q < NA; ++q)
            if (q < h.qa) ring_quad(cd[q], vv[q], h.na - 4 * q);
        auto load_quad = [&](int at, int cnt) {
            T v[4];
            quad(vals, at, v);
            uint2 cq = __ldg(reinterpret_cast<const uint2 *>(blk + 16) + at * 32 + lane);
            cq.x *= KT * W;
            cq.y *= KT * W;
            ring_quad(cq, v, cnt);
        };
        if (h.qa > NA)
            for (int q = NA; q < h.qa; ++q) load_quad(q, h.na - 4 * q);
        if (__builtin_expect(h.tail, 0)) tail_pass(33, lim);
#pragma unroll
        for (int r = 0; r < KT; ++r) consume(acc[r]);
        // ---- 3. group c-1, then this group
        if (!wait_done(c)) return false;
        // (FP32: whole quads of zeros cost less than branches)
#pragma unroll
        for (int q = 0; q < NB; ++q)
            if (!F64 || q < h.qb) ring_quad(cd[NA + q], vv[NA + q], h.nb - 4 * q);
        if (__builtin_expect(h.qb > NB, 0))
            for (int q = NB; q < h.qb; ++q) load_quad(h.qa + q, h.nb - 4 * q);
        if (__builtin_expect(h.tail, 0)) tail_pass(1, 32);
        T t[KT];
#pragma unroll
        for (int r = 0; r < KT; ++r) t[r] = (bv[r] - acc[r]) * rinv;
        if (h.kind == kTriSteps) {
#pragma unroll
            for (int k = 0; k < (F64 ? 4 * NT : 8); ++k) {
                if ((F64 || k % 2 == 0) && k >= h.steps) break;
                const int s = ids[k / 4] >> (8 * (k % 4));  // (a shuffle takes the lane modulo 32)
#pragma unroll
                for (int r = 0; r < KT; ++r)
                    t[r] = fma(-tri[k / 4][k % 4], __shfl_sync(SPT_FULL_MASK, t[r], s), t[r]);
            }
            if constexpr (F64) {
                for (int k = 4 * NT; k < h.steps; ++k) {
                    const int s = tabid[(k / 4) * 32 + lane] >> (8 * (k % 4));
                    const T cf = tab[k * 32 + lane];
#pragma unroll
                    for (int r = 0; r < KT; ++r) t[r] = fma(-cf, __shfl_sync(SPT_FULL_MASK, t[r], s), t[r]);
                }
            }
        } else if (h.kind == kTriInverse) {
            if constexpr (!F64) {
                if (__builtin_expect(dense, 0)) {
                    group_list<T, KT>(t, ids[0], [&](int s) { return tab[s * 32 + lane]; });
                } else {
                    const unsigned slots = ringa + slot0 * KT * W;
                    store_vec<float, KT>(ring0 + (slot0 + lane) * KT, t);
                    __syncwarp();
                    if constexpr (KT == 1) {
                        float y[4] = {0.0f, 0.0f, 0.0f, 0.0f}, g[8][4];
#pragma unroll
                        for (int q = 0; q < 8; ++q) lds(slots + 16 * q, g[q]);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
#pragma unroll
                            for (int u = 0; u < 4; ++u) y[u] = fmaf(tri[q][u], g[q][u], y[u]);
                        t[0] += (y[0] + y[1]) + (y[2] + y[3]);
                    } else {
                        float y[2][KT];
#pragma unroll
                        for (int r = 0; r < KT; ++r) y[0][r] = y[1][r] = 0.0f;
#pragma unroll
                        for (int q = 0; q < 8; ++q)
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                float g[KT];
                                lds(slots + (4 * q + u) * KT * W, g);
#pragma unroll
                                for (int r = 0; r < KT; ++r) y[u & 1][r] = fmaf(tri[q][u], g[r], y[u & 1][r]);
                            }
#pragma unroll
                        for (int r = 0; r < KT; ++r) t[r] += y[0][r] + y[1][r];
                    }
                    __syncwarp();
                }
            }
        }
        store_vec<T, KT>(ring0 + (slot0 + lane) * KT, t);
        __syncwarp();
        if (lane == 0 && !hold) st_release_cta_smem(ctr, c + 1);
        if (valid) {
            T *xx = R.x + (int64_t)i * R.ld;
#pragma unroll
            for (int r = 0; r < KT; ++r)
                if (r < kt) xx[r] = t[r];
        }
        bool finite = true;
#pragma unroll
        for (int r = 0; r < KT; ++r) finite &= fabs(t[r]) <= (F64 ? T(DBL_MAX) : T(FLT_MAX));
        if (!finite) *bad = 1;
        __syncwarp();
    }
    return true;
}

// One system's KT columns by the whole thread block (`nwarps` of its warps
// work); s_bad: a word of shared memory.
template <class T, int KT, bool TR>
__device__ __forceinline__ bool strip_solve(const Sys<T> &A, const Strips &V, const Rhs<T> &R, int nwarps,
                                            unsigned char *smem, int warps_alloc, int *s_bad, const Waiter &w,
                                            int withhold)
{
    const int ring = V.ring;
    int *ctr = reinterpret_cast<int *>(smem + strip_ring_bytes(ring, KT, (int)sizeof(T)) +
                                       (size_t)warps_alloc * kStripTable<T> * sizeof(T));
    T *ring0 = reinterpret_cast<T *>(smem);
    for (int t = threadIdx.x; t < (ring + 4) * KT; t += blockDim.x) ring0[t] = T(0);
    if (threadIdx.x == 0) {
        *ctr = 0;
        *s_bad = 0;
    }
    __syncthreads();
    bool ok = true;
    if ((int)(threadIdx.x >> 5) < nwarps) ok = strip_turns<T, KT, TR>(A, V, R, nwarps, smem, ctr, s_bad, w, withhold);
    if (!__syncthreads_and(ok)) return false;
    if (*s_bad) ok = strip_again<T, KT, TR>(A, R, smem, w, withhold);
    return ok;
}

}  // namespace spt
