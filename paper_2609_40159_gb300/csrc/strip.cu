// Strips (strip.cuh): plan-time tables and the refresh before a solve.
#include <algorithm>

#include "strip.cuh"

namespace spt {

namespace {

// Where an entry's value goes: bit 15: C[row][column] of the group's triangle
// (row << 5 | column); bit 14: the row's diagonal; bit 13: nowhere (read by the
// solve itself); else slot (row << 7 | slot) of the group's quads, bit 12: scaled
// by the row's reciprocal diagonal.
constexpr uint16_t kToTri = 0x8000, kToDiag = 0x4000, kNowhere = 0x2000, kScaled = 0x1000;

constexpr int kStageWarps = 4;
constexpr int kStageEntries = 12;  // (11 a row in the mean fit a group in one go)
constexpr int kTri = 36;       // row stride of a triangle in shared memory
constexpr float kMaxInverse = 16.0f;
constexpr int kMaxSteps = 8;   // FP32: longer schedules become an inverse
// Shared memory that the refresh of a group takes (values of w bytes): the
// diagonals, the quads put together (of dependencies, and of steps), and the
// triangle where it becomes an inverse.
__host__ __device__ __forceinline__ int stage_bytes(const StripBits &h, int w)
{
    const int inv = h.kind == kTriInverse;
    return 32 * w + 128 * w * (h.staged() + (inv ? 0 : h.tri_quads())) + (inv ? 32 * kTri * w : 0);
}

// What a row's entries are to its group: dependencies of the group itself
// (mask), of the previous group (nb), older ones (na); entries from `ptail` on
// that are not of the group are not staged.
struct RowScan {
    int na = 0, nb = 0, ptail = 0, reach = 0;
    unsigned mask = 0;
    bool tail = false;
};

__device__ __forceinline__ RowScan scan_row(const int32_t *idx, int a, int e, int n, bool trans, int base)
{
    RowScan r;
    for (int p = a; p < e; ++p) {
        const int j = ldro(idx + p);
        const int d = base - (trans ? n - 1 - j : j);
        if (d <= 0) {
            r.mask |= 1u << -d;
            continue;
        }
        r.reach = max(r.reach, d);
        if (r.tail) continue;
        int &c = d <= 32 ? r.nb : r.na;
        if (c == (d <= 32 ? kStripNear : kStripOld)) {
            r.tail = true;
            r.ptail = p;
        } else {
            ++c;
        }
    }
    return r;
}

// Schedule of a group's in-group dependencies (every lane with its row's mask):
// every step, each row that still waits takes its first dependency that is
// solved by then; a row is solved when it waits for none (row r after r steps
// at most).  Returns the number of steps; take(step, row) for each.
template <class F> __device__ __forceinline__ int schedule_steps(unsigned mask, F take)
{
    unsigned rem = mask;
    unsigned done = __ballot_sync(SPT_FULL_MASK, rem == 0);
    int step = 0;
    for (; done != SPT_FULL_MASK; ++step) {
        const unsigned av = rem & done;
        if (av) {
            take(step, __ffs(av) - 1);
            rem &= ~(av & (0u - av));
        }
        done = __ballot_sync(SPT_FULL_MASK, rem == 0);
    }
    return step;
}

// System of a group of the list.
__device__ __forceinline__ int src_of(const StripBuild &B, int64_t g)
{
    int lo = 0, hi = B.nsrc;  // the last that does not start after g
    while (hi - lo > 1) {
        const int m = (lo + hi) / 2;
        if (B.src[m].g0 <= g) lo = m;
        else hi = m;
    }
    return lo;
}

// Warp per group: the farthest dependency.
__global__ void __launch_bounds__(256) k_strip_reach(StripBuild B)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < B.ng; g += nw) {
        const int m = src_of(B, g);
        const StripSrc S = B.src[m];
        const int i = (int)((g - S.g0) * 32) + lane;
        int far = 0;
        if (i < S.n) {
            // (the first entry of a row, the last of a column, is the farthest)
            const int a = ldro(S.ptr + i), e = ldro(S.ptr + i + 1);
            if (e - a > 1) far = B.trans ? ldro(S.idx + e - 1) - i : i - ldro(S.idx + a);
        }
        far = __reduce_max_sync(SPT_FULL_MASK, far);
        if (lane == 0 && far > B.far[m]) atomicMax(B.far + m, far);
    }
}

// Warp per group: what its block holds, and its size.
__global__ void __launch_bounds__(256) k_strip_sizes(StripBuild B)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < B.ng; g += nw) {
        const int m = src_of(B, g);
        const StripSrc S = B.src[m];
        const int ring = strip_ring(B.far[m], B.ring_most);
        const int base = (int)((g - S.g0) * 32), pos = base + lane;
        RowScan r;
        if (pos < S.n) {
            const int i = B.trans ? S.n - 1 - pos : pos;
            r = scan_row(S.idx, ldro(S.ptr + i) + (B.trans ? 1 : 0), ldro(S.ptr + i + 1) - (B.trans ? 0 : 1), S.n,
                         B.trans, base);
        }
        const int na = __reduce_max_sync(SPT_FULL_MASK, r.na), nb = __reduce_max_sync(SPT_FULL_MASK, r.nb);
        const int far = __reduce_max_sync(SPT_FULL_MASK, r.reach);
        const bool tail = __any_sync(SPT_FULL_MASK, r.tail);
        const int steps = schedule_steps(r.mask, [](int, int) {});
        // a step costs a shuffle and a multiply-add (30 cycles, FP64 90), the
        // inverse (FP32) about 250 whatever the triangle
        const uint32_t kind = steps == 0 ? kTriNone : !B.f64 && steps > kMaxSteps ? kTriInverse : kTriSteps;
        if (lane == 0) {
            B.bits[g] = strip_bits(na, nb, kind, steps, tail, far > ring - 32);
            const StripBits h(B.bits[g]);
            B.units[g] = h.bytes(B.f64 ? 8 : 4) / 16;
            const int need = stage_bytes(h, B.f64 ? 8 : 4);
            if (need > *B.stage) atomicMax(B.stage, need);
        }
    }
}

__global__ void __launch_bounds__(256)
k_strip_tables(StripBuild B, const uint32_t *__restrict__ ofs, unsigned char *blocks, uint16_t *ecodes)
{
    const int lane = threadIdx.x & 31;
    const bool trans = B.trans;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < B.ng; g += nw) {
        const int m = src_of(B, g);
        const StripSrc S = B.src[m];
        const int32_t *ptr = S.ptr, *idx = S.idx;
        const int n = S.n, ring = strip_ring(B.far[m], B.ring_most);
        uint16_t *ecode = ecodes + S.e0;
        const int base = (int)((g - S.g0) * 32), pos = base + lane;
        const StripBits h(B.bits[g]);
        unsigned char *blk = blocks + (size_t)ofs[g] * 16u;
        const int staged = h.staged();
        uint16_t *code = reinterpret_cast<uint16_t *>(blk + 16) + 4 * lane;  // slot s at code[128 (s / 4) + s % 4]
        int32_t *dist = reinterpret_cast<int32_t *>(blk + 16 + 256 * staged) + 4 * lane;  // as code
        uint32_t *word = reinterpret_cast<uint32_t *>(blk + h.at_words()) + lane;
        if (lane == 0) *reinterpret_cast<uint4 *>(blk) = make_uint4(B.bits[g], 0u, 0u, 0u);
        const uint32_t zeros = (uint32_t)ring * 0x10001u;
        for (int q = 0; q < staged; ++q) {
            *reinterpret_cast<uint2 *>(code + 128 * q) = make_uint2(zeros, zeros);
            if (h.far) *reinterpret_cast<int4 *>(dist + 128 * q) = make_int4(0, 0, 0, 0);
        }
        // (a step that takes nothing: the row itself, times 0)
        if (h.kind == kTriSteps)
            for (int q = 0; q < h.tri_words(); ++q) word[32 * q] = (uint32_t)lane * 0x01010101u;
        RowScan r;
        int first = 0, last = 0;
        if (pos < n) {
            const int i = trans ? n - 1 - pos : pos;
            const int a = ldro(ptr + i), e = ldro(ptr + i + 1);
            first = trans ? a + 1 : a;
            last = trans ? e : e - 1;
            r = scan_row(idx, first, last, n, trans, base);
            ecode[trans ? a : e - 1] = (uint16_t)(kToDiag | lane);
        }
        const int tp = r.tail ? r.ptail : last;
        uint8_t step_of[32];
        schedule_steps(r.mask, [&](int k, int s) {
            step_of[s] = (uint8_t)k;
            if (h.kind == kTriSteps) {
                uint32_t &wd = word[32 * (k >> 2)];
                wd = (wd & ~(0xffu << (8 * (k & 3)))) | (uint32_t)s << (8 * (k & 3));
            }
        });
        if (h.kind == kTriInverse) word[0] = r.mask;
        if (h.tail) word[32 * h.tri_words()] = (uint32_t)tp;
        int ka = 0, kb = 0;
        for (int p = first; p < last; ++p) {
            const int j = ldro(idx + p);
            const int d = base - (trans ? n - 1 - j : j);
            uint16_t c;
            if (d <= 0) {
                c = h.kind == kTriInverse ? (uint16_t)(kToTri | lane << 5 | -d)
                                          : (uint16_t)(kScaled | lane << 7 | (4 * staged + step_of[-d]));
            } else if (p >= tp) {
                c = kNowhere;
            } else {
                const int slot = d <= 32 ? 4 * h.qa + kb++ : ka++;
                const int at = 128 * (slot >> 2) + (slot & 3);
                if (d <= ring - 32) code[at] = (uint16_t)((base - d) % ring);
                else dist[at] = d;
                c = (uint16_t)(lane << 7 | slot);
            }
            ecode[p] = c;
        }
    }
}

// Inverse of a group's unit triangle I + C in place: C row-major in shared
// memory (stride kTri, zeros where there is no entry and on the diagonal)
// becomes W = (I + C)^-1 - I.  W (I + C) = I, solved from the last column by
// lane L for row L in registers; C is read with broadcast 16-byte loads.
// Returns the largest magnitude in the lane's row.
__device__ __forceinline__ float invert_triangle(float *c, int lane)
{
    float wr[32];
#pragma unroll
    for (int s = 0; s < 32; ++s) wr[s] = s == lane ? 1.0f : 0.0f;
#pragma unroll
    for (int s = 31; s >= 1; --s) {
        const float ws = wr[s];
#pragma unroll
        for (int q = 0; q < 32; q += 4) {
            if (q >= s) continue;
            const float4 f = *reinterpret_cast<const float4 *>(c + s * kTri + q);
            const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q + u < s) wr[q + u] = fmaf(-ws, v[u], wr[q + u]);
        }
    }
    float big = 0.0f;
#pragma unroll
    for (int s = 0; s < 32; ++s) {
        wr[s] = s == lane ? 0.0f : wr[s];
        big = fabsf(wr[s]) <= big ? big : fabsf(wr[s]);  // (a NaN becomes the result)
    }
    __syncwarp();
    if (__all_sync(SPT_FULL_MASK, big <= kMaxInverse)) {
#pragma unroll
        for (int q = 0; q < 32; q += 4)
            *reinterpret_cast<float4 *>(c + lane * kTri + q) = make_float4(wr[q], wr[q + 1], wr[q + 2], wr[q + 3]);
    }
    return big;
}

// Where a group's block and entries are.  Loaded while the group before is
// staged: what a group's entries wait for would otherwise be three loads from
// memory one after another.
struct StageAt {
    unsigned char *blk;
    uint32_t bits;
    int p0, p1;
    __device__ __forceinline__ StageAt() : blk(nullptr), bits(0u), p0(0), p1(0) {}
    template <class T> __device__ __forceinline__ StageAt(const Sys<T> &A, const Strips &V, int g, bool trans)
    {
        blk = V.blocks + (size_t)ldro(V.ofs + g) * 16u;
        bits = *reinterpret_cast<const uint32_t *>(blk);
        const int base = g * 32, rows = min(32, A.n - base), lo = trans ? A.n - base - rows : base;
        const int32_t *ptr = trans ? A.cp : A.rp;
        p0 = ldro(ptr + lo);
        p1 = ldro(ptr + lo + rows);
    }
};

// The groups of a warp: a block takes consecutive ones, its warps in turn, as
// neighbours share the lines of the tables and, transposed, of the values that
// they gather.
struct StageShare {
    int64_t first, end;
    __device__ __forceinline__ explicit StageShare(int64_t groups)
    {
        const int64_t per = (groups + (int64_t)gridDim.x * kStageWarps - 1) / ((int64_t)gridDim.x * kStageWarps);
        const int64_t start = blockIdx.x * per * kStageWarps;
        first = start + (threadIdx.x >> 5);
        end = min(groups, start + per * kStageWarps);
    }
};

// One group's values into its block, by one warp.  The entries of the group's
// rows are contiguous (CSR forward, CSC transpose), so everything is read and
// written along lanes; the quads are put together in shared memory.
template <class T, bool TR>
__device__ __forceinline__ void stage_group(const Sys<T> &A, const Strips &V, int g, const StageAt &at,
                                            unsigned char *raw)
{
    constexpr int HV = 16 / (int)sizeof(T);  // values of 16 bytes
    const int lane = threadIdx.x & 31;
    T *diag = reinterpret_cast<T *>(raw);
    T *quads = diag + 32;  // as in the block: FP32 [quad][row][4], FP64 [quad][half][row][2]
    unsigned char *blk = at.blk;
    const StripBits h(at.bits);
    const int rows = min(32, A.n - g * 32);
    const int staged = h.staged(), qv = staged + (h.kind == kTriInverse ? 0 : h.tri_quads());
    float *tri = reinterpret_cast<float *>(quads + qv * 128);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 *q4 = reinterpret_cast<float4 *>(quads);
    constexpr int P = 4 / HV;  // 16-byte planes of a quad
    for (int q = 0; q < qv * P; ++q) q4[q * 32 + lane] = zero;
    diag[lane] = T(1);
    if constexpr (sizeof(T) == 4) {
        if (h.kind == kTriInverse)
#pragma unroll
            for (int q = 0; q < 32; q += 4) *reinterpret_cast<float4 *>(tri + lane * kTri + q) = zero;
    }
    __syncwarp();
    // several entries a lane at a time: the loads of all are in flight together
    // (one at a time: 2.4x)
    const int p1 = at.p1;
    for (int pa = at.p0 + lane; pa - lane < p1; pa += 32 * kStageEntries) {
        unsigned c[kStageEntries];
        T v[kStageEntries];
#pragma unroll
        for (int u = 0; u < kStageEntries; ++u) {
            const int p = pa + 32 * u;
            c[u] = p < p1 ? ldro(V.ecode + p) : kNowhere;
            v[u] = p < p1 ? entry_val<T, TR>(A, p) : T(0);
        }
        // (all of them: left to itself the compiler moves each value's load to its
        // store, behind the store before)
#pragma unroll
        for (int u = 0; u < kStageEntries; ++u) {
            consume((int)c[u]);
            consume(v[u]);
        }
#pragma unroll
        for (int u = 0; u < kStageEntries; ++u) {
            const int row = (c[u] & (kToTri | kToDiag)) ? (c[u] >> 5) & 31 : (c[u] >> 7) & 31, slot = c[u] & 127;
            T *to = quads + ((slot / HV) * 32 + row) * HV + slot % HV;
            if (sizeof(T) == 4) to = c[u] & kToTri ? reinterpret_cast<T *>(tri + row * kTri + (c[u] & 31)) : to;
            to = c[u] & kToDiag ? diag + (c[u] & 31) : to;
            if (!(c[u] & kNowhere)) *to = v[u];
        }
    }
    __syncwarp();
    const T rinv = lane < rows ? T(1) / diag[lane] : T(0);
    reinterpret_cast<T *>(blk + h.at_rinv())[lane] = rinv;
    float4 *out = reinterpret_cast<float4 *>(blk + h.at_values(sizeof(T)));
    for (int q = 0; q < qv * P; ++q) {
        float4 f = q4[q * 32 + lane];
        if (q >= staged * P) {
            T *v = reinterpret_cast<T *>(&f);
#pragma unroll
            for (int u = 0; u < HV; ++u) v[u] *= rinv;
        }
        out[q * 32 + lane] = f;
    }
    if constexpr (sizeof(T) == 4) {
        if (h.kind == kTriInverse) {
            float *row = tri + lane * kTri;
#pragma unroll
            for (int q = 0; q < 32; q += 4) {
                float4 f = *reinterpret_cast<float4 *>(row + q);
                f.x *= rinv; f.y *= rinv; f.z *= rinv; f.w *= rinv;
                *reinterpret_cast<float4 *>(row + q) = f;
            }
            __syncwarp();
            // a large inverse would lose accuracy to the substitution: then
            // the triangle itself is staged
            const float big = invert_triangle(tri, lane);
            const bool kept = __all_sync(SPT_FULL_MASK, big <= kMaxInverse);
#pragma unroll
            for (int q = 0; q < 8; ++q) out[(staged + q) * 32 + lane] = *reinterpret_cast<float4 *>(row + 4 * q);
            if (lane == 0) reinterpret_cast<StripHead *>(blk)->dense = kept ? 0u : 1u;
        }
    }
    __syncwarp();
}

template <class T, bool TR>
__global__ void __launch_bounds__(32 * kStageWarps) k_strip_stage(Sys<T> A, Strips V, PlanCtl *ctl)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) reset_ctl(ctl);
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned char *raw = smraw + (threadIdx.x >> 5) * V.stage;
    const int64_t ng = ((int64_t)A.n + 31) / 32;
    const StageShare sh(ng);
    StageAt next;
    if (sh.first < sh.end) next = StageAt(A, V, (int)sh.first, TR);
    for (int64_t g = sh.first; g < sh.end; g += kStageWarps) {
        const StageAt at = next;
        if (g + kStageWarps < sh.end) next = StageAt(A, V, (int)g + kStageWarps, TR);
        stage_group<T, TR>(A, V, (int)g, at, raw);
    }
}

template <class T, bool TR>
__global__ void __launch_bounds__(32 * kStageWarps)
k_strip_stage_batch(const BatchMat *__restrict__ mats, const RowChunk *__restrict__ chunks, int64_t nchunks, int stage)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned char *raw = smraw + (threadIdx.x >> 5) * stage;
    const StageShare sh(nchunks);
    auto sys = [&](const BatchMat &M) {
        Sys<T> A{};
        A.n = M.n;
        A.nnz = M.nnz;
        A.rp = M.rp; A.v = (const T *)M.v;
        A.cp = M.cp; A.tmap = M.tmap;
        return A;
    };
    auto look = [&](int64_t c) {
        const RowChunk ch = chunks[c];
        const BatchMat &M = mats[ch.mat];
        const Strips V = M.strips[TR ? 1 : 0];
        return V.blocks ? StageAt(sys(M), V, ch.r0 >> 5, TR) : StageAt();
    };
    StageAt next;
    if (sh.first < sh.end) next = look(sh.first);
    for (int64_t c = sh.first; c < sh.end; c += kStageWarps) {
        const StageAt at = next;
        if (c + kStageWarps < sh.end) next = look(c + kStageWarps);
        if (at.blk == nullptr) continue;
        const RowChunk ch = chunks[c];
        const BatchMat &M = mats[ch.mat];
        stage_group<T, TR>(sys(M), M.strips[TR ? 1 : 0], ch.r0 >> 5, at, raw);
    }
}

int warp_grid(int64_t groups) { return (int)std::min<int64_t>(std::max<int64_t>((groups + 7) / 8, 1), 152 * 16); }
// (many blocks: groups cost unequally, and four or five blocks are resident on
// an SM; 512 systems, forward solve, 8 / 32 / 128 blocks an SM: 7.43 / 7.07 /
// 6.91 ms)
int stage_grid(int64_t groups)
{
    return (int)std::min<int64_t>(std::max<int64_t>((groups + kStageWarps - 1) / kStageWarps, 1), 152 * 128);
}

}  // namespace

cudaError_t strip_sizes(const StripBuild &B, cudaStream_t s, const Scratch *from)
{
    k_strip_reach<<<warp_grid(B.ng), 256, 0, s>>>(B);
    k_strip_sizes<<<warp_grid(B.ng), 256, 0, s>>>(B);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = exclusive_scan_i32(B.units, reinterpret_cast<int32_t *>(B.ofs), B.ng, B.total, s, from);
    return e;
}

cudaError_t strip_tables(const StripBuild &B, const uint32_t *ofs, unsigned char *blocks, uint16_t *ecode,
                         cudaStream_t s)
{
    k_strip_tables<<<warp_grid(B.ng), 256, 0, s>>>(B, ofs, blocks, ecode);
    return cudaGetLastError();
}

template <class T>
cudaError_t strip_stage(const Sys<T> &A, const Strips &V, PlanCtl *ctl, bool trans, cudaStream_t s)
{
    if (A.n <= 0) return cudaSuccess;
    const int smem = kStageWarps * V.stage, most = (int)kBlockSmemBudget;
    const int grid = stage_grid(((int64_t)A.n + 31) / 32);
    const cudaError_t e = trans ? allow_smem<k_strip_stage<T, true>>(most) : allow_smem<k_strip_stage<T, false>>(most);
    if (e != cudaSuccess) return e;
    if (trans) k_strip_stage<T, true><<<grid, 32 * kStageWarps, smem, s>>>(A, V, ctl);
    else k_strip_stage<T, false><<<grid, 32 * kStageWarps, smem, s>>>(A, V, ctl);
    return cudaGetLastError();
}

template <class T>
cudaError_t strip_stage_batch(const BatchMat *mats, const RowChunk *chunks, int64_t nchunks, int stage, bool trans,
                              cudaStream_t s)
{
    const int smem = kStageWarps * stage, most = (int)kBlockSmemBudget;
    // (both, also without chunks: a plan calls this once outside any capture)
    cudaError_t e = allow_smem<k_strip_stage_batch<T, true>>(most);
    if (e == cudaSuccess) e = allow_smem<k_strip_stage_batch<T, false>>(most);
    if (e != cudaSuccess || nchunks <= 0) return e;
    const int grid = stage_grid(nchunks);
    if (trans) k_strip_stage_batch<T, true><<<grid, 32 * kStageWarps, smem, s>>>(mats, chunks, nchunks, stage);
    else k_strip_stage_batch<T, false><<<grid, 32 * kStageWarps, smem, s>>>(mats, chunks, nchunks, stage);
    return cudaGetLastError();
}

#define SPT_INST(T)                                                                                   \
    template cudaError_t strip_stage<T>(const Sys<T> &, const Strips &, PlanCtl *, bool, cudaStream_t); \
    template cudaError_t strip_stage_batch<T>(const BatchMat *, const RowChunk *, int64_t, int, bool, \
                                              cudaStream_t);
SPT_INST(double)
SPT_INST(float)
#undef SPT_INST

}  // namespace spt
