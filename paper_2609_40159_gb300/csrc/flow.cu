// Cluster flow solve: the hybrid schedule with every level thin -- rows in
// level order, each waiting for its own dependencies only -- on ONE
// thread-block cluster per right-hand side (k_flow), after a pass of the whole
// GPU that lays L's values out in the order the cluster reads them
// (k_flow_stage).
//
// What bounds it: the chain of levels.  One hop of a grid-wide kernel is a
// store to L2 and a poll that sees it (870 cycles measured between most SMs);
// a store into the shared memory of another SM of the cluster is seen after
// 280, one inside the SM after 160 (one lane polling), and FP64 adds 64 cycles
// for each dependent operation.  So
// the rows of a level are shared by the blocks of one cluster, every block
// keeps the recent solutions its rows depend on in a ring in shared memory,
// and a row's solution is stored into the ring of every block that needs it
// (which ones is known from the plan).  The loads of a group are issued one
// group of the warp ahead: with them on the chain the solve was bound by 16
// warps' worth of memory latency, 1.7x slower.
// Measured, one right-hand side, forward (2D Laplacian 1024^2, 2,047 levels;
// power-law DAG of 1M rows, 15,795 levels), grid-wide hybrid kernel -> this:
// FP64 3.16 -> 1.07 ms and 20.5 -> 12.8 ms, FP32 2.61 -> 0.68 ms and
// 19.2 -> 9.1 ms; four right-hand sides on 401^2 (FP32) 2.10 -> 0.25 ms.
#include <algorithm>
#include <atomic>
#include <climits>

#include "flow.cuh"
#include "rows.cuh"

namespace spt {

namespace {

// ------------------------------------------------------------ solution ring
// Code of position q: bit 31, its generation q / R + 1 and its slot q mod R of
// the shared-memory ring; a dependency too old for the ring has its row + 1 as
// its code (bit 31 clear), no dependency 0.  A slot holds a solution together
// with its position's code: FP32 {bits, code} in one 64-bit word; FP64 two words {low bits, code}
// and {high bits, code}, each checked on its own, so that only the single-copy
// atomicity of 64-bit accesses is relied on.
constexpr uint32_t kNear = 0x80000000u;
constexpr int kSlotBits = 15;
template <class T> struct Ring;
template <> struct Ring<float> {
    static constexpr int R = 27648;  // 216 KB
    static constexpr int kBytes = 8;
};
template <> struct Ring<double> {
    static constexpr int R = 13824;  // 216 KB
    static constexpr int kBytes = 16;
};
// Positions of an epoch.  During epoch e (a group belongs to the epoch of its
// first position; it may reach 31 positions further) the ring is written at
// positions [e H, e H + H + 31) and read at positions >= (e - 1) H: distinct
// slots, as 2 H + 31 < R.
__host__ __device__ constexpr int epoch_rows(int R) { return (R - 32) / 2; }

__device__ __forceinline__ uint32_t near_code(int q, int R)
{
    return kNear | ((uint32_t)(q / R + 1) << kSlotBits) | (uint32_t)(q % R);
}
// (code 0 -- no dependency -- is the slot after the ring: value 0, code 0)
template <class T> __device__ __forceinline__ unsigned slot_of(unsigned ring, uint32_t code)
{
    return ring + (code ? code & ((1u << kSlotBits) - 1u) : (unsigned)Ring<T>::R) * Ring<T>::kBytes;
}

// (Remote: another block's slot, a shared::cluster address)
template <bool Remote> __device__ __forceinline__ void slot_store(unsigned a, float x, uint32_t code)
{
    const unsigned long long v = ((unsigned long long)code << 32) | __float_as_uint(x);
    if (Remote) asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
    else asm volatile("st.relaxed.cluster.shared::cta.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
template <bool Remote> __device__ __forceinline__ void slot_store(unsigned a, double x, uint32_t code)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const unsigned long long lo = ((unsigned long long)code << 32) | (bits & 0xffffffffull);
    const unsigned long long hi = ((unsigned long long)code << 32) | (bits >> 32);
    if (Remote)
        asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(lo), "l"(hi) : "memory");
    else
        asm volatile("st.relaxed.cluster.shared::cta.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ bool slot_load(unsigned a, uint32_t code, float &x)
{
    unsigned long long v;
    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    x = __uint_as_float((uint32_t)v);
    return (uint32_t)(v >> 32) == code;
}
__device__ __forceinline__ bool slot_load(unsigned a, uint32_t code, double &x)
{
    unsigned long long lo, hi;
    asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "r"(a) : "memory");
    x = __longlong_as_double((long long)((hi << 32) | (lo & 0xffffffffull)));
    return (uint32_t)(lo >> 32) == code && (uint32_t)(hi >> 32) == code;
}
__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_arrive()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ float ld_x(const float *p)
{
    float v;
    asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double ld_x(const double *p)
{
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}

constexpr int kFlowThreads = 512;
constexpr int kFlowWarps = kFlowThreads / 32;

// Waits of one block.  A warp that gives up tells its cluster (the abort words
// in shared memory, looked at often) and the other right-hand sides' clusters
// (the plan's abort flag, read by a block when it starts and every 4,096
// polls): more clusters than the GPU holds run in waves, which would otherwise
// wait the whole limit one after another.
struct FlowWait {
    Waiter w;
    unsigned abort_at;  // shared address of the block's abort word
    int csize;
    __device__ __forceinline__ bool gave_up() const
    {
        return ld_relaxed_smem(abort_at) != 0;
    }
    static __device__ __forceinline__ int ld_relaxed_smem(unsigned a)
    {
        int v;
        asm volatile("ld.relaxed.cluster.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
        return v;
    }
    __device__ __forceinline__ void give_up() const
    {
        spt::give_up(w);
        for (int c = 0; c < csize; ++c)
            asm volatile("st.relaxed.cluster.shared::cluster.s32 [%0], %1;" ::"r"(map_rank(abort_at, c)), "r"(1)
                         : "memory");
    }
};

// Bound of a polling loop that a whole warp runs together: false once the
// wait limit has passed or another warp gave up.
struct FlowClock {
    long long start = 0;
    unsigned polls = 0;
    __device__ __forceinline__ bool go_on(const FlowWait &fw)
    {
        if ((++polls & 63u) != 0) return true;
        if (__any_sync(SPT_FULL_MASK, fw.gave_up())) return false;
        if ((polls & 4095u) == 0 && __any_sync(SPT_FULL_MASK, aborted(fw.w))) return false;
        const long long t = clock64();
        if (start == 0) start = t;
        if (__any_sync(SPT_FULL_MASK, (double)(t - start) > 2.2 * (double)fw.w.limit_ns)) {
            fw.give_up();
            return false;
        }
        return true;
    }
};

// Waits, all lanes together, until code[u] has come to its slot for u < N in
// every lane (code 0: the slot that is always ready, value 0); false when the
// cluster gave up.  While nothing has come, the warp reads one slot, that of
// `first` (the same in every lane): the polls of all warps of a block share
// the shared-memory port with the stores that they wait for.
template <class T, int N>
__device__ __forceinline__ bool slots_wait(uint32_t first, const uint32_t *code, unsigned ring, const FlowWait &fw,
                                           T *xv)
{
    FlowClock clk;
    {
        const unsigned a = slot_of<T>(ring, first);
        // (one load of a warp is not one moment: two lanes may read the slot
        // before and after it is written, hence the vote)
        T ignored;
        while (!__all_sync(SPT_FULL_MASK, slot_load(a, first, ignored)))
            if (!clk.go_on(fw)) return false;
    }
    unsigned a[N];
#pragma unroll
    for (int u = 0; u < N; ++u) a[u] = slot_of<T>(ring, code[u]);
    for (;;) {
        bool got = true;
#pragma unroll
        for (int u = 0; u < N; ++u) got &= slot_load(a[u], code[u], xv[u]);
        if (__all_sync(SPT_FULL_MASK, got)) return true;
        if (!clk.go_on(fw)) return false;
    }
}

// Values of one lane's first four entries as they are staged.
template <class T> struct Four;
template <> struct Four<float> {
    float4 a;
    __device__ __forceinline__ void load(const void *p, int64_t t) { a = __ldg((const float4 *)p + t); }
    __device__ __forceinline__ void store(void *p, int64_t t) const { ((float4 *)p)[t] = a; }
    __device__ __forceinline__ void get(float (&v)[4]) const { v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; }
    __device__ __forceinline__ void set(const float (&v)[4]) { a = make_float4(v[0], v[1], v[2], v[3]); }
};
template <> struct Four<double> {
    double2 a, b;
    __device__ __forceinline__ void load(const void *p, int64_t t)
    {
        a = __ldg((const double2 *)p + 2 * t);
        b = __ldg((const double2 *)p + 2 * t + 1);
    }
    __device__ __forceinline__ void store(void *p, int64_t t) const
    {
        ((double2 *)p)[2 * t] = a;
        ((double2 *)p)[2 * t + 1] = b;
    }
    __device__ __forceinline__ void get(double (&v)[4]) const { v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y; }
    __device__ __forceinline__ void set(const double (&v)[4])
    {
        a = make_double2(v[0], v[1]);
        b = make_double2(v[2], v[3]);
    }
};

__device__ __forceinline__ int meta_llpr(uint32_t m) { return (m >> 16) & 15; }
__device__ __forceinline__ int meta_most(uint32_t m) { return (m >> 20) & 15; }

// The values in the order that the solve reads them (every solve: L's values
// may have changed since the last).
template <class T, bool TR> __global__ void __launch_bounds__(256) k_flow_stage(Sys<T> A, FlowSched F, Waiter w)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) st_relaxed(w.abort_flag, 0);  // for the solve that follows
    const int64_t nslots = (int64_t)F.ngroups * 32;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nslots; t += (int64_t)gridDim.x * blockDim.x) {
        const FlowLane ln = F.lanes[t];
        if (ln.row < 0) continue;
        const int2 s = F.src[t];
        const int llpr = meta_llpr(ln.meta);
        T v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = s.x + (u << llpr) < s.y ? entry_val<T, TR>(A, s.x + (u << llpr)) : T(0);
        Four<T> f;
        f.set(v);
        f.store(F.vals, t);
        if ((t & ((1 << llpr) - 1)) == 0)
            static_cast<T *>(F.inv)[t] = T(1) / entry_val<T, TR>(A, TR ? s.x - 1 : s.y);
    }
}

template <class T, bool TR>
__global__ void __launch_bounds__(kFlowThreads, 1)
k_flow(Sys<T> A, FlowSched F, Rhs<T> R, int32_t withhold, Waiter w)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_abort;
    constexpr int NR = Ring<T>::R, SB = Ring<T>::kBytes, H = epoch_rows(NR);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned rank = cluster_rank();
    const int col = blockIdx.x / F.csize;  // one cluster per right-hand side
    const T *b = R.b + col;
    T *x = R.x + col;
    const unsigned ring = smem_addr(smraw);
    for (int t = threadIdx.x; t < NR * SB / 16 + 1; t += kFlowThreads)
        reinterpret_cast<uint4 *>(smraw)[t] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) s_abort = aborted(w) ? 1 : 0;
    const FlowWait fw{w, smem_addr(&s_abort), F.csize};
    cluster_arrive();
    const int nepochs = (F.n + H - 1) / H;
    const int g1 = F.gptr[rank + 1];
    int gi = F.gptr[rank] + wid;
    // right-hand side of a row (b, or b + T b of a rewritten system)
    auto rhs = [&](const FlowLane &ln) {
        if (ln.row < 0 || (lane & ((1 << meta_llpr(ln.meta)) - 1)) != 0) return T(0);
        const int i = chk_row(A, ln.row);
        T s = b[(int64_t)i * R.ld];
        if (!TR && has_trow(A, i))
            for (int p = A.trp[i]; p < A.trp[i + 1]; ++p)
                s += ldro(A.tv + p) * b[(int64_t)tcol(A, p) * R.ld];
        return s;
    };
    // everything a group needs is loaded one group of the warp ahead (its
    // rows two ahead)
    const FlowLane none{-1, 0u, 0u, 0};
    FlowLane ln = none, ln_nx = none;
    uint4 cd_nx = make_uint4(0u, 0u, 0u, 0u);
    Four<T> fv_nx;
    T bv_nx = T(0), inv_nx = T(0);
    auto fetch = [&](int g, const FlowLane &l) {
        const int64_t t = (int64_t)g * 32 + lane;
        cd_nx = __ldg(F.codes + t);
        fv_nx.load(F.vals, t);
        inv_nx = ldro(static_cast<const T *>(F.inv) + t);
        bv_nx = rhs(l);
    };
    if (gi < g1) {
        ln = F.lanes[(int64_t)gi * 32 + lane];
        fetch(gi, ln);
    }
    if (gi + kFlowWarps < g1) ln_nx = F.lanes[(int64_t)(gi + kFlowWarps) * 32 + lane];
    cluster_wait();
    int epoch = 0;
    for (; gi < g1; gi += kFlowWarps) {
        const FlowLane me = ln;
        uint32_t code[4] = {cd_nx.x, cd_nx.y, cd_nx.z, cd_nx.w};
        T v[4];
        fv_nx.get(v);
        const T bv = bv_nx, rinv = inv_nx;
        ln = ln_nx;
        const int gn = gi + kFlowWarps;
        if (gn < g1) fetch(gn, ln);
        if (gn + kFlowWarps < g1) ln_nx = F.lanes[(int64_t)(gn + kFlowWarps) * 32 + lane];
        const int llpr = meta_llpr(me.meta), most = meta_most(me.meta);
        const int lpr = 1 << llpr;
        const bool lead = me.row >= 0 && (lane & (lpr - 1)) == 0;
        // where the row's solution goes: its own block, another one, more
        const unsigned own = slot_of<T>(ring, me.code);
        unsigned mask = lead && me.row != withhold ? me.meta & 0xffffu : 0u;
        const bool here = (mask >> rank) & 1u;
        mask &= ~(1u << rank);
        const bool there = mask != 0;
        const unsigned other = map_rank(own, there ? __ffs(mask) - 1 : rank);
        mask &= mask - 1;
        const bool anythere = __any_sync(SPT_FULL_MASK, there), anymore = __any_sync(SPT_FULL_MASK, mask != 0);
        // ---- the group's epoch: the rows of every epoch before the last are in x
        __syncwarp();
        for (; epoch < me.epoch; ++epoch) {
            cluster_arrive();
            cluster_wait();
        }
        // dependencies too old for the ring; what is left waits for its slot
        T acc = T(0);
        bool far = false;
#pragma unroll
        for (int u = 0; u < 4; ++u) far |= code[u] != 0u && !(code[u] & kNear);
        if (__any_sync(SPT_FULL_MASK, far)) {
            T xf[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                xf[u] = T(0);
                if (code[u] != 0u && !(code[u] & kNear)) xf[u] = ld_x(x + (int64_t)chk_row(A, (int)code[u] - 1) * R.ld);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (code[u] != 0u && !(code[u] & kNear)) {
                    acc = fma(v[u], xf[u], acc);
                    code[u] = 0u;
                    v[u] = T(0);
                }
        }
        uint32_t newest = 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) newest = code[u] ? code[u] : newest;
        const unsigned waiting = __ballot_sync(SPT_FULL_MASK, newest != 0u);
        const uint32_t first = waiting ? __shfl_sync(SPT_FULL_MASK, newest, 31 - __clz(waiting)) : 0u;
        consume(acc);
        consume(bv);
        consume(rinv);
        // ---- the row's turn
        T xv[4];
        bool ok;
        if (most <= 2) {
            ok = slots_wait<T, 2>(first, code, ring, fw, xv);
            acc = fma(v[0], xv[0], acc);
            acc = fma(v[1], xv[1], acc);
        } else {
            ok = slots_wait<T, 4>(first, code, ring, fw, xv);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc = fma(v[u], xv[u], acc);
        }
        if (llpr != 0) {
            if (llpr == 5 && ok) {
                // entries beyond the staged ones (a row of the longest class),
                // the next 32 loaded while these are waited for
                const int2 s = F.src[(int64_t)gi * 32 + lane];
                int p = s.x + 128;
                uint32_t cn = p < s.y ? ldro(F.ecode + p) : 0u;
                T vn = p < s.y ? entry_val<T, TR>(A, p) : T(0);
                for (; ok && __any_sync(SPT_FULL_MASK, p < s.y); p += 32) {
                    uint32_t c1 = cn;
                    const T v1 = vn;
                    const int pn = p + 32;
                    cn = pn < s.y ? ldro(F.ecode + pn) : 0u;
                    vn = pn < s.y ? entry_val<T, TR>(A, pn) : T(0);
                    T xf = T(0), x1;
                    const bool old = c1 != 0u && !(c1 & kNear);
                    if (old) {
                        xf = ld_x(x + (int64_t)chk_row(A, (int)c1 - 1) * R.ld);
                        c1 = 0u;
                    }
                    const unsigned wt = __ballot_sync(SPT_FULL_MASK, c1 != 0u);
                    const uint32_t f1 = wt ? __shfl_sync(SPT_FULL_MASK, c1, 31 - __clz(wt)) : 0u;
                    ok = slots_wait<T, 1>(f1, &c1, ring, fw, &x1);
                    acc = fma(v1, old ? xf : x1, acc);
                }
            }
            for (int o = lpr >> 1; o > 0; o >>= 1) acc += shfl_xor(acc, o);
        }
        const T xi = (bv - acc) * rinv;
        if (ok) {  // (a break here instead costs 1 % of every solve)
            if (anythere) {
                if (there) slot_store<true>(other, xi, me.code);
                if (anymore)
                    for (unsigned m = mask; m; m &= m - 1) slot_store<true>(map_rank(own, __ffs(m) - 1), xi, me.code);
            }
            if (here) slot_store<false>(own, xi, me.code);
        }
        if (lead) x[(int64_t)me.row * R.ld] = xi;
        __syncwarp();
    }
    for (; epoch < nepochs; ++epoch) {  // the last one: no block leaves while others may store to it
        cluster_arrive();
        cluster_wait();
    }
}

// ------------------------------------------------------------ plan tables
// Length class of a row: 1, 4, 16 or 32 lanes, so that all but the longest
// rows have their entries loaded before their turn.
__device__ __forceinline__ int flow_class(int len) { return len <= 4 ? 0 : len <= 16 ? 1 : len <= 64 ? 2 : 3; }

__global__ void k_flow_keys(const int32_t *__restrict__ ptr, const int32_t *__restrict__ lev, int32_t n, int32_t L,
                            bool trans, uint32_t *keys, int32_t *rows, int32_t *counts)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int len = ldro(ptr + i + 1) - ldro(ptr + i) - 1;
        const int l = ldro(lev + i);
        const uint32_t k = (uint32_t)(trans ? L - 1 - l : l) * kFlowClasses + flow_class(len);
        keys[i] = k;
        rows[i] = (int32_t)i;
        atomicAdd(counts + k, 1);
    }
}

__global__ void k_flow_inverse(const int32_t *__restrict__ order, int32_t n, int32_t *iperm)
{
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        iperm[order[q]] = (int32_t)q;
}

// Block (5 bits) and epoch of every position, one warp per group.
__global__ void k_flow_meta(const FlowGroup *__restrict__ groups, const int32_t *__restrict__ gptr, int32_t ngroups,
                            int32_t csize, int32_t H, uint32_t *meta, uint32_t *mask)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < ngroups; g += nw) {
        int c = 0;
        while (c + 1 < csize && gptr[c + 1] <= g) ++c;
        const FlowGroup G = groups[g];
        if (lane < G.cnt) {
            meta[G.base + lane] = (uint32_t)(G.base / H) << 5 | (uint32_t)c;
            mask[G.base + lane] = 0u;
        }
    }
}

// Code of every entry, and the blocks that each solution goes to: 8 lanes per
// position.
__global__ void k_flow_codes(const int32_t *__restrict__ ptr, const int32_t *__restrict__ idx, int32_t n, bool trans,
                             int32_t NR, const int32_t *__restrict__ order, const int32_t *__restrict__ iperm,
                             const uint32_t *__restrict__ meta, uint32_t *mask, uint32_t *ecode)
{
    const int sl = threadIdx.x & 7, H = epoch_rows(NR);
    const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 3;
    for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3; q < n; q += step) {
        const int i = order[q];
        const int a = ldro(ptr + i) + (trans ? 1 : 0), e = ldro(ptr + i + 1) - (trans ? 0 : 1);
        const uint32_t m = meta[q];
        const int64_t lo = ((int64_t)(m >> 5) - 1) * H;
        const unsigned bit = 1u << (m & 31);
        for (int p = a + sl; p < e; p += 8) {
            const int j = ldro(idx + p), d = ldro(iperm + j);
            const bool near = d >= lo;
            ecode[p] = near ? near_code(d, NR) : (uint32_t)j + 1u;
            if (near) atomicOr(mask + d, bit);
        }
    }
}

// One thread per lane of every group.
__global__ void k_flow_lanes(const int32_t *__restrict__ ptr, bool trans, int32_t NR,
                             const int32_t *__restrict__ order, const FlowGroup *__restrict__ groups, int32_t ngroups,
                             const uint32_t *__restrict__ mask, const uint32_t *__restrict__ ecode, FlowLane *lanes,
                             uint4 *codes, int2 *src)
{
    const int64_t nslots = (int64_t)ngroups * 32;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nslots; t += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(t & 31);
        const FlowGroup G = groups[t >> 5];
        const int r = lane >> G.llpr, sl = lane & ((1 << G.llpr) - 1), q = G.base + r;
        FlowLane ln{-1, 0u, 0u, G.base / epoch_rows(NR)};
        uint32_t c[4] = {0u, 0u, 0u, 0u};
        int a = 0, e = 0;
        if (r < G.cnt) {
            const int i = order[q];
            a = ldro(ptr + i) + (trans ? 1 : 0) + sl;
            e = ldro(ptr + i + 1) - (trans ? 0 : 1);
            ln.row = i;
            ln.code = near_code(q, NR);
            ln.meta = mask[q];
            for (int u = 0; u < 4; ++u)
                if (a + (u << G.llpr) < e) c[u] = ecode[a + (u << G.llpr)];
        }
        // (32 consecutive threads hold one group)
        const int mine = e > a ? min(4, (e - a + (1 << G.llpr) - 1) >> G.llpr) : 0;
        ln.meta |= (uint32_t)G.llpr << 16 | (uint32_t)__reduce_max_sync(SPT_FULL_MASK, mine) << 20;
        lanes[t] = ln;
        codes[t] = make_uint4(c[0], c[1], c[2], c[3]);
        src[t] = make_int2(a, e);
    }
}

int flow_grid(int64_t work) { return (int)std::min<int64_t>(std::max<int64_t>((work + 255) / 256, 1), 152 * 16); }

template <class T, bool TR> cudaError_t flow_config(cudaLaunchConfig_t &c, cudaLaunchAttribute *at, int csize)
{
    static DeviceOnce once;  // one per kernel instantiation
    constexpr int smem = Ring<T>::R * Ring<T>::kBytes + 16;  // the ring and the slot that is always ready
    int device = -1;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess)
        e = (cudaError_t)once.run(device, [] {
            cudaError_t q = cudaFuncSetAttribute(k_flow<T, TR>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (q == cudaSuccess)
                q = cudaFuncSetAttribute(k_flow<T, TR>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            return (int)q;
        });
    if (e != cudaSuccess) return e;
    c.blockDim = dim3(kFlowThreads);
    c.dynamicSmemBytes = smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)csize;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaSuccess;
}

template <class T> bool flow_fits(int csize)
{
    int n = 0;
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at[1];
    c.gridDim = dim3((unsigned)csize);
    bool ok = flow_config<T, false>(c, at, csize) == cudaSuccess &&
              cudaOccupancyMaxActiveClusters(&n, k_flow<T, false>, &c) == cudaSuccess && n >= 1;
    ok = ok && flow_config<T, true>(c, at, csize) == cudaSuccess &&
         cudaOccupancyMaxActiveClusters(&n, k_flow<T, true>, &c) == cudaSuccess && n >= 1;
    if (!ok) cudaGetLastError();
    return ok;
}

}  // namespace

// (a property of the device: asked once for each device, type and size)
bool flow_cluster_fits(int csize, bool f64)
{
    static std::atomic<int> known[64][2][5];  // 0: not asked, 1: no, 2: yes
    int device = -1, l = 0;
    while ((1 << l) < csize) ++l;
    const bool keep = cudaGetDevice(&device) == cudaSuccess && device >= 0 && device < 64 && l < 5;
    const int k = keep ? known[device][f64][l].load() : 0;
    if (k) return k == 2;
    const bool fits = f64 ? flow_fits<double>(csize) : flow_fits<float>(csize);
    if (keep) known[device][f64][l] = fits ? 2 : 1;
    return fits;
}

cudaError_t flow_order(const int32_t *ptr, const int32_t *lev, int32_t n, int32_t L, bool trans, int32_t *order,
                       int32_t *iperm, int32_t *counts, cudaStream_t s, const Scratch *from)
{
    uint32_t *keys = nullptr;  // keys, sorted keys, rows
    cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int32_t) * (size_t)L * kFlowClasses, s);
    Scratch tmp(s, from);
    if (e == cudaSuccess) e = tmp.take(&keys, 3 * (size_t)n);
    if (e != cudaSuccess) return e;
    int32_t *rows = reinterpret_cast<int32_t *>(keys + 2 * (size_t)n);
    k_flow_keys<<<flow_grid(n), 256, 0, s>>>(ptr, lev, n, L, trans, keys, rows, counts);
    int bits = 0;
    while (bits < 32 && (((uint32_t)L * kFlowClasses - 1) >> bits) != 0) ++bits;
    e = radix_sort_pairs(keys, rows, keys + n, order, n, bits, s, &tmp);
    if (e == cudaSuccess) {
        k_flow_inverse<<<flow_grid(n), 256, 0, s>>>(order, n, iperm);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t flow_tables(const int32_t *ptr, const int32_t *idx, int32_t n, bool trans, bool f64, const int32_t *order,
                        const int32_t *iperm, const FlowGroup *groups, const int32_t *gptr, int32_t ngroups,
                        int32_t csize, uint32_t *meta, uint32_t *mask, FlowLane *lanes, uint4 *codes, int2 *src,
                        uint32_t *ecode, cudaStream_t s)
{
    const int NR = f64 ? Ring<double>::R : Ring<float>::R;
    k_flow_meta<<<flow_grid((int64_t)ngroups * 32), 256, 0, s>>>(groups, gptr, ngroups, csize, epoch_rows(NR), meta,
                                                                 mask);
    k_flow_codes<<<flow_grid((int64_t)n * 8), 256, 0, s>>>(ptr, idx, n, trans, NR, order, iperm, meta, mask, ecode);
    k_flow_lanes<<<flow_grid((int64_t)ngroups * 32), 256, 0, s>>>(ptr, trans, NR, order, groups, ngroups, mask, ecode,
                                                                  lanes, codes, src);
    return cudaGetLastError();
}

template <class T>
cudaError_t solve_flow(const Sys<T> &A, const FlowSched &F, const Rhs<T> &R, bool trans, int32_t withhold,
                       const Waiter &w, cudaStream_t s)
{
    if (A.n <= 0) return cudaSuccess;
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at[1];
    cudaError_t e = trans ? flow_config<T, true>(c, at, F.csize) : flow_config<T, false>(c, at, F.csize);
    if (e != cudaSuccess) return e;
    c.gridDim = dim3((unsigned)(F.csize * R.k));
    c.stream = s;
    const int sg = flow_grid((int64_t)F.ngroups * 32);
    if (trans) k_flow_stage<T, true><<<sg, 256, 0, s>>>(A, F, w);
    else k_flow_stage<T, false><<<sg, 256, 0, s>>>(A, F, w);
    return trans ? cudaLaunchKernelEx(&c, k_flow<T, true>, A, F, R, withhold, w)
                 : cudaLaunchKernelEx(&c, k_flow<T, false>, A, F, R, withhold, w);
}

template cudaError_t solve_flow<double>(const Sys<double> &, const FlowSched &, const Rhs<double> &, bool, int32_t,
                                        const Waiter &, cudaStream_t);
template cudaError_t solve_flow<float>(const Sys<float> &, const FlowSched &, const Rhs<float> &, bool, int32_t,
                                       const Waiter &, cudaStream_t);

}  // namespace spt
