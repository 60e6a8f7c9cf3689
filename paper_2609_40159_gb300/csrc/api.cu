// C ABI of the SpTRSV library (declared in include/sptrsv.h): handles, plans,
// level analysis, rewriting, single and batched solves, adjoints.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <climits>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "flow.cuh"
#include "solve.cuh"
#include "strip.cuh"

using namespace spt;

namespace {

// Device memory for the length of a call.
template <class T> struct DeviceArray {
    T *p = nullptr;
    cudaError_t get(size_t count) { return cudaMalloc(&p, sizeof(T) * count); }
    ~DeviceArray() { cudaFree(p); }
};

// Named NVTX range for a profiler timeline (no cost without a tool attached).
struct Range {
    explicit Range(const char *name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
};
constexpr long long kDefaultWaitNs = 10ll * 1000 * 1000 * 1000;  // 10 s
constexpr int kUpdateRounds = 32;  // fixpoint rounds of an incremental analysis before the full pass

bool debug_mode()
{
    static int on = -1;
    if (on < 0) {
        const char *v = getenv("SPTRSV_DEBUG");
        on = (v && v[0] && v[0] != '0') ? 1 : 0;
    }
    return on == 1;
}

sptrsv_status from_cuda(cudaError_t e)
{
    if (e == cudaSuccess) return SPTRSV_OK;
    if (debug_mode()) fprintf(stderr, "[sptrsv] CUDA error: %s\n", cudaGetErrorString(e));
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? SPTRSV_ENOMEM : SPTRSV_ECUDA;
}

// With SPTRSV_DEBUG set, every asynchronous entry point synchronises so that
// a failing kernel is reported by the call that launched it.
sptrsv_status debug_sync(sptrsv_status st, cudaStream_t s, const char *what)
{
    if (st != SPTRSV_OK || !debug_mode()) return st;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) fprintf(stderr, "[sptrsv] %s: %s\n", what, cudaGetErrorString(e));
    return from_cuda(e);
}

// Rows per warp from the mean row length; a heavy tail of long rows (more
// than 0.5 % of the rows with over 32 off-diagonals: one lane would walk
// each of them alone, on the dependency chain) takes a warp per row.
int default_rpw(int32_t n, int64_t nnz, int64_t long_rows = 0)
{
    if (n > 0 && long_rows * 200 > n) return 1;
    const double avg = n > 0 ? (double)nnz / n : 1.0;
    if (avg <= 12) return 32;
    if (avg <= 24) return 16;
    if (avg <= 48) return 8;
    if (avg <= 96) return 4;
    return 1;
}

// The same for block-local solves, which stage up to 16 dependencies a row on
// the previous group and 28 older ones: one lane per row for longer rows too.
int block_rpw(int32_t n, int64_t nnz, int64_t long_rows = 0)
{
    const int r = default_rpw(n, nnz, long_rows);
    return r == 16 && (double)nnz / n <= 20.0 ? 32 : r;
}

int default_kt(int k)
{
    int kt = 1;
    while (kt < k && kt < 16) kt <<= 1;
    return kt;
}

bool valid_rpw(int r) { return r == 1 || r == 2 || r == 4 || r == 8 || r == 16 || r == 32; }
bool valid_kt(int k) { return k == 1 || k == 2 || k == 4 || k == 8 || k == 16; }
}  // namespace

struct sptrsv_handle_st {
    cudaStream_t stream = nullptr;
    DeviceInfo di;
    int *d_status = nullptr;
    PlanCtl *d_ctl = nullptr;
    long long *d_scratch = nullptr;  // validation result, max level, stats
    // test hook of the level analysis (sptrsv_debug_withhold_level)
    int32_t dbg_withhold = -1;
    long long dbg_wait_ns = 0;
    int64_t dbg_table_limit = -1;  // (sptrsv_debug_limit_tables)
};

struct PlanMat {
    // one system of a (possibly batched) plan
    sptrsv_csr L{};
    sptrsv_csr T{};
    bool hasT = false;
    int32_t nlevels = 0;
    int32_t *d_lev = nullptr, *d_perm = nullptr, *d_level_ptr = nullptr;
    std::vector<int32_t> h_level_ptr;
    int32_t *d_cp = nullptr, *d_crow = nullptr, *d_tmap = nullptr;
    void *d_cv = nullptr;  // L's values in CSC order (transpose solves)
    uint32_t *d_tmask = nullptr;
    // CSC of T (the adjoint's T^T gathers by column), its column mask
    int32_t *d_tcp = nullptr, *d_trow = nullptr, *d_ttmap = nullptr;
    uint32_t *d_tcmask = nullptr;
    // level-ordered batched schedule (built when first used): inverse of
    // d_perm, row groups of each direction
    int32_t *d_iperm = nullptr;
    LevelGroup *d_lgroups[2] = {nullptr, nullptr};
    int32_t n_lgroups[2] = {0, 0};
    // strips of each direction (block-local in-order solves)
    Strips strips[2]{};
};

struct sptrsv_plan_st {
    sptrsv_handle h = nullptr;
    bool batched = false;
    sptrsv_dtype dtype = SPTRSV_F64;
    long long spin = kDefaultWaitNs;  // bounded-wait limit, nanoseconds
    int32_t withhold = -1;
    bool have_csc = false;
    std::vector<void *> owned;
    PlanCtl *d_ctl = nullptr;
    // single system
    PlanMat M;
    int mode = SPTRSV_MODE_SYNCFREE, rpw = 32, kt = 1;
    int32_t *d_chunk_fwd = nullptr, *d_chunk_tr = nullptr;
    int chunk_rpw = 0;
    uint32_t *d_flags = nullptr;
    // value-carrying ready flags of single-right-hand-side solves (16 bytes
    // per row: the solution bits and the epoch)
    unsigned long long *d_vflags = nullptr;
    int grid_level = 0, grid_sf = 0;
    int grid_level_max = 0;  // grid_level at the occupancy maximum
    int32_t max_width = 0;
    // hybrid schedule: thin-level threshold (0 = automatic) and, per
    // direction, the first level of the thin run holding every level
    int32_t thin_rows = 0, seg_rows = -1;
    int32_t *d_seg[2] = {nullptr, nullptr};
    // cluster flow schedule of each direction ([0] forward, [1] transpose),
    // built when the hybrid mode is chosen; off: could not be built
    FlowSched flow[2];
    bool flow_ready[2] = {false, false}, flow_off[2] = {false, false};
    // row-major copies of a column-major right-hand-side block and its
    // solution (sptrsv_solve_layout), grown on demand
    void *d_lay = nullptr;
    size_t lay_bytes = 0;
    // batched
    std::vector<PlanMat> mats;
    std::vector<int64_t> rhs_off, vals_off, row_off;
    BatchMat *d_mats = nullptr;
    std::vector<BatchMat> h_mats;
    // work items of each direction ([0] forward, [1] transpose): per system
    // rows per warp and rhs columns per work item, the items (system, rhs
    // column tile, geometry), their launch order, shared memory and grid
    struct Geom {
        std::vector<int32_t> rpw, tile, sched;  // (tile 0: automatic)
        bool csc_vals = false;  // some item reads L's values in CSC order
        bool strips = false;    // some item is solved over strips
        int stage = 0;          // shared memory of a group's refresh
        BatchItem *d_items = nullptr;
        int32_t *d_order = nullptr;
        int32_t nitems = 0;
        size_t smem = 0;
        int grid = 0;
    } geo[2];
    int32_t max_items = 0;
    // Columns an item: the plan's option, else two, four level by level in FP32
    // (on 256 training systems of 1,000-40,000 rows over strips, FP32, 3.43 /
    // 3.03 / 3.40 ms a step with 1 / 2 / 4; on 32 small FP64 ones 0.41 / 0.42 /
    // 0.63 ms; 64 systems level by level, forward, FP32 0.62 / 0.60 ms with 2 /
    // 4, FP64 2.9 / 5.3 ms)
    int tile_of(int d, size_t m) const
    {
        if (geo[d].tile[m]) return geo[d].tile[m];
        return geo[d].sched[m] == kSchedLevel && dtype == SPTRSV_F32 ? 4 : 2;
    }
    bool takes_strips(int d, size_t m) const
    {
        return geo[d].rpw[m] == 32 && geo[d].sched[m] == kSchedInOrder && mats[m].L.n > 0;
    }
    void strips_to_build(int d, std::vector<PlanMat *> *need)
    {
        if (d == 1 && !have_csc) return;
        for (size_t m = 0; m < mats.size(); ++m)
            if (takes_strips(d, m) && !mats[m].strips[d].blocks) need->push_back(&mats[m]);
    }
    int last_dir = 0;  // direction of the last batched solve (for the trace)
    RowChunk *d_gchunks = nullptr, *d_tchunks = nullptr;  // all 32-row chunks; chunks with T rows
    int64_t n_gchunks = 0, n_tchunks = 0;
    RowChunk *d_ctiles = nullptr;   // tiles of the CSC value gather: (system, first entry)
    int64_t n_ctiles = 0;
    RowChunk *d_fchunks = nullptr;  // every 32-row chunk of the rewritten systems
    int64_t n_fchunks = 0;
    void *d_bt = nullptr;           // b + T b of the rewritten systems (packed like b)
    long long *d_trace = nullptr;  // per work item: start ns, end ns, SM of the last batch solve
    // steps from host buffers (sptrsv_batch_step_host): two device buffer
    // sets used alternately, a stream for the copies in and one for the
    // copies out (the solves run on the handle's stream)
    struct HostSet {
        void *b = nullptr, *w = nullptr, *x = nullptr, *gbp = nullptr, *gb = nullptr, *gv = nullptr;
        cudaEvent_t h2d = nullptr, comp = nullptr, d2h = nullptr;
        bool used = false;
    } hset[2];
    cudaStream_t s_h2d = nullptr, s_d2h = nullptr;
    int64_t nsteps = 0;

    // One allocation that the plan's arrays of known size are carved from (one
    // of more than 1 MB takes 50 us, and 36 us to give back).
    char *arena = nullptr;
    size_t arena_left = 0;
    static size_t padded(size_t bytes) { return (std::max<size_t>(bytes, 1) + 255) / 256 * 256; }
    void reserve(size_t bytes)
    {
        if (alloc(&arena, bytes) == cudaSuccess) arena_left = bytes;
        else cudaGetLastError();  // (then one by one)
    }
    template <class P> cudaError_t alloc(P **p, size_t bytes)
    {
        if (padded(bytes) <= arena_left) {
            *p = reinterpret_cast<P *>(arena);
            arena += padded(bytes);
            arena_left -= padded(bytes);
            return cudaSuccess;
        }
        void *q = nullptr;
        cudaError_t e = cudaMalloc(&q, bytes > 0 ? bytes : 16);
        if (e == cudaSuccess) { owned.push_back(q); *p = static_cast<P *>(q); }
        return e;
    }
    // Tables of a schedule that the plan can do without.
    template <class P> cudaError_t alloc_tables(P **p, size_t bytes)
    {
        if (h->dbg_table_limit >= 0 && bytes > (size_t)h->dbg_table_limit) return cudaErrorMemoryAllocation;
        void *q = nullptr;  // (not of the arena: it may be released)
        cudaError_t e = cudaMalloc(&q, bytes);
        if (e == cudaSuccess) { owned.push_back(q); *p = static_cast<P *>(q); }
        return e;
    }
    void release(void *q)
    {
        owned.erase(std::remove(owned.begin(), owned.end(), q), owned.end());
        cudaFree(q);
    }
};

// ------------------------------------------------------------------ handle
extern "C" sptrsv_status sptrsv_create(sptrsv_handle *handle, void *stream)
{
    if (!handle) return SPTRSV_EINVAL;
    *handle = nullptr;
    sptrsv_handle h = new (std::nothrow) sptrsv_handle_st;
    if (!h) return SPTRSV_ENOMEM;
    h->stream = (cudaStream_t)stream;
    cudaError_t e = cudaGetDevice(&h->di.device);
    int sms = 0, smem = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->di.device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->di.device);
    h->di.num_sms = sms;
    h->di.max_smem_optin = (size_t)smem;
    if (e == cudaSuccess) e = cudaMalloc(&h->d_status, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&h->d_ctl, sizeof(PlanCtl));
    if (e == cudaSuccess) e = cudaMalloc(&h->d_scratch, 16 * sizeof(long long));
    if (e == cudaSuccess) e = cudaMemset(h->d_status, 0, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(h->d_ctl, 0, sizeof(PlanCtl));
    if (e != cudaSuccess) {
        cudaFree(h->d_status); cudaFree(h->d_ctl); cudaFree(h->d_scratch);
        delete h;
        return from_cuda(e);
    }
    *handle = h;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_destroy(sptrsv_handle h)
{
    if (!h) return SPTRSV_EINVAL;
    cudaStreamSynchronize(h->stream);
    cudaFree(h->d_status);
    cudaFree(h->d_ctl);
    cudaFree(h->d_scratch);
    delete h;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_set_stream(sptrsv_handle h, void *stream)
{
    if (!h) return SPTRSV_EINVAL;
    h->stream = (cudaStream_t)stream;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_get_status(sptrsv_handle h)
{
    if (!h) return SPTRSV_EINVAL;
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return from_cuda(e);
    int st = 0;
    e = cudaMemcpy(&st, h->d_status, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return from_cuda(e);
    if (st != 0) cudaMemset(h->d_status, 0, sizeof(int));
    return (sptrsv_status)st;
}

extern "C" const char *sptrsv_status_string(sptrsv_status s)
{
    switch (s) {
    case SPTRSV_OK: return "ok";
    case SPTRSV_EINVAL: return "invalid argument";
    case SPTRSV_ENOTLOWER: return "matrix is not lower triangular";
    case SPTRSV_EDIAG: return "diagonal missing, not last or zero";
    case SPTRSV_EUNSORTED: return "columns of a row are not strictly increasing";
    case SPTRSV_ETARGET: return "rewrite target outside [0, lev(i))";
    case SPTRSV_ENOMEM: return "out of device memory";
    case SPTRSV_ETIMEOUT: return "a bounded device wait gave up";
    case SPTRSV_ECUDA: return "CUDA error";
    case SPTRSV_ENOTSUP: return "not supported";
    case SPTRSV_ERANGE: return "index out of range (bounds-checked build)";
    }
    return "unknown status";
}

// -------------------------------------------------------------- internals
namespace {

sptrsv_status check_csr(const sptrsv_csr *L)
{
    if (!L || L->n < 0 || L->nnz < 0 || L->nnz >= INT_MAX) return SPTRSV_EINVAL;
    if (L->dtype != SPTRSV_F64 && L->dtype != SPTRSV_F32) return SPTRSV_EINVAL;
    if (L->n > 0 && (!L->row_ptr || !L->col_idx || !L->vals)) return SPTRSV_EINVAL;
    return SPTRSV_OK;
}

sptrsv_status validate_impl(sptrsv_handle h, const sptrsv_csr &L, int32_t *bad_row)
{
    if (bad_row) *bad_row = -1;
    if (L.n == 0) return SPTRSV_OK;
    cudaError_t e = launch_validate(L, h->d_scratch, h->stream);
    long long r = LLONG_MAX;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&r, h->d_scratch, sizeof(r), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return from_cuda(e);
    if (r == LLONG_MAX) return SPTRSV_OK;
    if (bad_row) *bad_row = (int32_t)(r / 16);
    return (sptrsv_status)(r % 16);
}

// Levels of L into lev (device, n) and their count.  Validates first.
// Levels of L; rows before 32 * (first_row / 32) keep the levels already in
// `lev` (incremental recompute after a rewrite that left them unchanged).
sptrsv_status levels_impl(sptrsv_handle h, const sptrsv_csr &L, int32_t *lev, int32_t *nlevels,
                          long long spin, int32_t first_row = 0)
{
    *nlevels = 0;
    sptrsv_status st = validate_impl(h, L, nullptr);
    if (st != SPTRSV_OK || L.n == 0) return st;
    cudaStream_t s = h->stream;
    cudaError_t e = cudaMemsetAsync(&h->d_ctl->abort_flag, 0, sizeof(int), s);
    Ctl ctl{h->d_status, &h->d_ctl->abort_flag, &h->d_ctl->ticket};
    if (h->dbg_withhold >= 0 && h->dbg_wait_ns > 0) spin = h->dbg_wait_ns;
    int32_t restart = 0;  // rows from here on are (re)computed by the sync-free pass
    if (first_row > 0 && e == cudaSuccess) {
        // after a change confined to rows >= first_row: fixpoint rounds from
        // the previous levels; a change that propagates through more than
        // kUpdateRounds rounds (a level collapse renumbers every later level)
        // or moves many rows at once is finished by the sync-free pass from
        // the first unsettled row
        bool converged = false;
        e = launch_levels_update(L, first_row, lev, ctl, spin, h->di, s, kUpdateRounds, h->dbg_withhold,
                                 &converged, &restart);
        int hab0 = 0;
        if (e == cudaSuccess) e = cudaMemcpy(&hab0, &h->d_ctl->abort_flag, sizeof(int), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return from_cuda(e);
        if (hab0) return SPTRSV_ETIMEOUT;
        if (converged) restart = L.n;
    }
    const int64_t c0 = restart / 32;
    if (e == cudaSuccess && 32 * c0 < L.n) {
        e = cudaMemsetAsync(lev + 32 * c0, 0xFF, sizeof(int32_t) * (size_t)(L.n - 32 * c0), s);
        if (e == cudaSuccess) e = launch_levels(L, lev, ctl, spin, h->di, s, c0, h->dbg_withhold);
    }
    int32_t *dmax = reinterpret_cast<int32_t *>(h->d_scratch + 1);
    if (e == cudaSuccess) e = launch_max(lev, L.n, dmax, s);
    int32_t hm = -1;
    int hab = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hm, dmax, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hab, &h->d_ctl->abort_flag, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return from_cuda(e);
    if (hab) return SPTRSV_ETIMEOUT;
    *nlevels = hm + 1;
    return SPTRSV_OK;
}

sptrsv_status analyze_into(sptrsv_handle h, const sptrsv_csr &L, int32_t *lev, int32_t *perm,
                           int32_t *level_ptr, int64_t *cost, int32_t *nlevels, double *stats,
                           long long spin, int32_t first_row = 0, const Scratch *from = nullptr)
{
    sptrsv_status st = levels_impl(h, L, lev, nlevels, spin, first_row);
    if (st != SPTRSV_OK) return st;
    cudaStream_t s = h->stream;
    cudaError_t e = level_partition(L, lev, *nlevels, perm, level_ptr, cost, s, from);
    if (e == cudaSuccess && stats) {
        double *dst = reinterpret_cast<double *>(h->d_scratch + 2);
        e = launch_level_stats(L.n, L.nnz, *nlevels, level_ptr, cost, dst, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(stats, dst, 6 * sizeof(double), cudaMemcpyDeviceToHost, s);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return from_cuda(e);
}

template <class T> Sys<T> sys_of(const PlanMat &M, int *chk)
{
    Sys<T> A;
    A.nnz = M.L.nnz;
    A.chk = chk;
    A.n = M.L.n;
    A.rp = M.L.row_ptr; A.ci = M.L.col_idx; A.v = (const T *)M.L.vals;
    A.cp = M.d_cp; A.crow = M.d_crow; A.tmap = M.d_tmap; A.cv = (const T *)M.d_cv;
    A.trp = M.hasT ? M.T.row_ptr : nullptr;
    A.tci = M.hasT ? M.T.col_idx : nullptr;
    A.tv = M.hasT ? (const T *)M.T.vals : nullptr;
    A.tmask = M.hasT ? M.d_tmask : nullptr;
    A.tcp = M.d_tcp; A.trow = M.d_trow; A.ttmap = M.d_ttmap;
    return A;
}

// Bytes of the arrays that prepare_mat allocates.
size_t mat_bytes(const sptrsv_csr &L, const sptrsv_csr *T, bool want_csc)
{
    auto b = [](int64_t count, size_t w) { return sptrsv_plan_st::padded(w * (size_t)std::max<int64_t>(count, 1)); };
    const int64_t n = std::max(L.n, 1);
    size_t all = 2 * b(n, 4) + b(n + 1, 4);
    if (T && T->n > 0) all += 2 * b((n + 31) / 32, 4) + b(n + 1, 4) + 2 * b(T->nnz, 4);
    if (want_csc) all += b(n + 1, 4) + 2 * b(L.nnz, 4) + b(L.nnz, L.dtype == SPTRSV_F64 ? 8 : 4);
    return all;
}

// Scratch of a plan's steps (a system of n rows and nnz entries): the sort by
// level, the sort by column, and both directions' orders of the cluster flow.
size_t plan_scratch(int32_t n, int64_t nnz, bool want_csc)
{
    auto b = [](int64_t count) { return Scratch::padded(4 * (size_t)std::max<int64_t>(count, 1)); };
    const size_t rows = 3 * b(n) + b(3 * (int64_t)n) + radix_sort_scratch(n);
    const size_t csc = want_csc ? b(n) + 3 * b(nnz) + radix_sort_scratch(nnz) : 0;
    const size_t flow = b((want_csc ? 2 : 1) * (int64_t)n * 5) + b(3 * (int64_t)n) + radix_sort_scratch(n);
    return std::max({rows, csc, flow});
}

// Analysis + schedule data + optional CSC for one system of a plan; cost:
// scratch for the level costs (n entries).  The caller synchronises.
sptrsv_status prepare_mat(sptrsv_plan p, PlanMat &M, const sptrsv_csr &L, const sptrsv_csr *T,
                          bool want_csc, int64_t *cost, const Scratch *from)
{
    sptrsv_handle h = p->h;
    cudaStream_t s = h->stream;
    M.L = L;
    const int32_t n = L.n;
    const size_t nn = (size_t)(n > 0 ? n : 1);
    if (T && T->n > 0) {
        if (T->n != n || T->dtype != L.dtype || !T->row_ptr || (T->nnz > 0 && (!T->col_idx || !T->vals)))
            return SPTRSV_EINVAL;
        M.T = *T;
        M.hasT = true;
    }
    cudaError_t e = p->alloc(&M.d_lev, sizeof(int32_t) * nn);
    if (e == cudaSuccess) e = p->alloc(&M.d_perm, sizeof(int32_t) * nn);
    if (e == cudaSuccess) e = p->alloc(&M.d_level_ptr, sizeof(int32_t) * (nn + 1));
    if (e != cudaSuccess) return from_cuda(e);
    sptrsv_status st = analyze_into(h, L, M.d_lev, M.d_perm, M.d_level_ptr, cost, &M.nlevels, nullptr, p->spin, 0, from);
    if (st != SPTRSV_OK) return st;
    M.h_level_ptr.assign((size_t)M.nlevels + 1, 0);
    if (n > 0) {
        e = cudaMemcpy(M.h_level_ptr.data(), M.d_level_ptr, sizeof(int32_t) * (M.nlevels + 1), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return from_cuda(e);
    }
    if (M.hasT) {
        const size_t tnz = (size_t)(M.T.nnz > 0 ? M.T.nnz : 1);
        e = p->alloc(&M.d_tmask, sizeof(uint32_t) * ((nn + 31) / 32));
        if (e == cudaSuccess) e = build_tmask(M.T.row_ptr, n, M.d_tmask, s);
        if (e == cudaSuccess) e = p->alloc(&M.d_tcp, sizeof(int32_t) * (nn + 1));
        if (e == cudaSuccess) e = p->alloc(&M.d_trow, sizeof(int32_t) * tnz);
        if (e == cudaSuccess) e = p->alloc(&M.d_ttmap, sizeof(int32_t) * tnz);
        if (e == cudaSuccess) e = p->alloc(&M.d_tcmask, sizeof(uint32_t) * ((nn + 31) / 32));
        if (e == cudaSuccess)
            e = M.T.nnz > 0 ? build_csc(M.T.row_ptr, M.T.col_idx, n, M.T.nnz, M.d_tcp, M.d_trow, M.d_ttmap, s, from)
                            : cudaMemsetAsync(M.d_tcp, 0, sizeof(int32_t) * (nn + 1), s);
        if (e == cudaSuccess) e = build_tmask(M.d_tcp, n, M.d_tcmask, s);
        if (e != cudaSuccess) return from_cuda(e);
    }
    if (want_csc) {
        e = p->alloc(&M.d_cp, sizeof(int32_t) * (nn + 1));
        if (e == cudaSuccess) e = p->alloc(&M.d_crow, sizeof(int32_t) * (size_t)(L.nnz > 0 ? L.nnz : 1));
        if (e == cudaSuccess) e = p->alloc(&M.d_tmap, sizeof(int32_t) * (size_t)(L.nnz > 0 ? L.nnz : 1));
        if (e == cudaSuccess)
            e = p->alloc(&M.d_cv, (L.dtype == SPTRSV_F64 ? 8 : 4) * (size_t)(L.nnz > 0 ? L.nnz : 1));
        if (e == cudaSuccess) e = build_csc(L.row_ptr, L.col_idx, n, L.nnz, M.d_cp, M.d_crow, M.d_tmap, s, from);
        if (e != cudaSuccess) return from_cuda(e);
    }
    return SPTRSV_OK;
}

sptrsv_status ensure_chunks(sptrsv_plan p)
{
    if (p->chunk_rpw == p->rpw) return SPTRSV_OK;
    const int32_t n = p->M.L.n;
    const int64_t nch = ((int64_t)n + p->rpw - 1) / p->rpw;
    cudaError_t e = cudaSuccess;
    // chunk tables are owned; reallocate at the largest size ever needed
    if (!p->d_chunk_fwd) {
        const int64_t maxch = n > 0 ? n : 1;  // rpw = 1
        e = p->alloc(&p->d_chunk_fwd, sizeof(int32_t) * (size_t)maxch);
        if (e == cudaSuccess) e = p->alloc(&p->d_chunk_tr, sizeof(int32_t) * (size_t)maxch);
        if (e != cudaSuccess) return from_cuda(e);
    }
    if (nch > 0 && p->M.nlevels > 0) {
        e = build_chunk_levels(p->M.d_level_ptr, p->M.nlevels, n, p->rpw, false, p->d_chunk_fwd, p->h->stream);
        if (e == cudaSuccess)
            e = build_chunk_levels(p->M.d_level_ptr, p->M.nlevels, n, p->rpw, true, p->d_chunk_tr, p->h->stream);
        if (e != cudaSuccess) return from_cuda(e);
    }
    p->chunk_rpw = p->rpw;
    return SPTRSV_OK;
}

// Thin-run heads of the hybrid schedule, per direction (processing order:
// forward = level order, transpose = reverse level order): seg[l] = l for a
// thick level, the run's first level for a level of a run of consecutive
// thin levels.
sptrsv_status ensure_hybrid(sptrsv_plan p)
{
    const PlanMat &M = p->M;
    const int32_t L = M.nlevels;
    // automatic: every level thin (one synchronisation-free run in level
    // order); barriers before thick levels measured slower on every
    // workload tried (2D/3D Laplacians, power-law DAG, banded)
    const int32_t thr = p->thin_rows > 0 ? p->thin_rows : INT32_MAX;
    if (p->seg_rows == thr && p->d_seg[0]) return SPTRSV_OK;
    cudaError_t e = cudaSuccess;
    for (int d = 0; d < 2 && e == cudaSuccess; ++d)
        if (!p->d_seg[d]) e = p->alloc(&p->d_seg[d], sizeof(int32_t) * (size_t)std::max(L, 1));
    if (e != cudaSuccess) return from_cuda(e);
    std::vector<int32_t> seg((size_t)std::max(L, 1));
    for (int d = 0; d < 2 && e == cudaSuccess; ++d) {
        for (int32_t k = 0; k < L; ++k) {
            const int32_t l = d == 0 ? k : L - 1 - k;  // level of processing index k
            const bool thin = M.h_level_ptr[l + 1] - M.h_level_ptr[l] < thr;
            const int32_t l_prev = d == 0 ? k - 1 : L - k;
            const bool prev_thin = k > 0 && M.h_level_ptr[l_prev + 1] - M.h_level_ptr[l_prev] < thr;
            seg[k] = thin && prev_thin ? seg[k - 1] : k;
        }
        if (L > 0) e = cudaMemcpy(p->d_seg[d], seg.data(), sizeof(int32_t) * L, cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) return from_cuda(e);
    p->seg_rows = thr;
    return SPTRSV_OK;
}

// Strips (strip.cuh) of the systems of each direction that have none; left out
// when their memory cannot be had (then the solves take several lanes per row).
// Both directions in one go, as of a small system the allocations and
// synchronisations are what this takes.  The caller synchronises.
void build_strips(sptrsv_plan p, const std::vector<PlanMat *> (&mats)[2], const Scratch *from = nullptr)
{
    const size_t nm[2] = {mats[0].size(), mats[1].size()}, all = nm[0] + nm[1];
    if (all == 0) return;
    std::vector<StripSrc> src(all);
    int64_t ng[2] = {0, 0}, nnz[2] = {0, 0};
    for (int d = 0; d < 2; ++d)
        for (size_t m = 0; m < nm[d]; ++m) {
            const PlanMat &M = *mats[d][m];
            src[d * nm[0] + m] = StripSrc{d ? M.d_cp : M.L.row_ptr, d ? M.d_crow : M.L.col_idx, ng[d], nnz[d], M.L.n};
            ng[d] += ((int64_t)M.L.n + 31) / 32;
            nnz[d] += M.L.nnz;
        }
    cudaStream_t s = p->h->stream;
    // scratch: the systems; totals, refresh memory and reaches (read back); then by direction
    // and group offsets (copied to the tables), sizes and contents
    char *tmp = nullptr, *tab = nullptr;
    const size_t b_src = sizeof(StripSrc) * all, b_ofs[2] = {4 * ((size_t)ng[0] + 1), 4 * ((size_t)ng[1] + 1)};
    const size_t b_back = 24 + 4 * all, at_ofs = (b_src + b_back + 15) / 16 * 16;
    Scratch scratch(s, from);
    cudaError_t e = scratch.take(&tmp, at_ofs + b_ofs[0] + b_ofs[1] + 8 * (size_t)(ng[0] + ng[1]));
    if (e != cudaSuccess) { cudaGetLastError(); return; }
    StripBuild B[2]{};
    uint32_t *u = reinterpret_cast<uint32_t *>(tmp + at_ofs + b_ofs[0] + b_ofs[1]);
    for (int d = 0; d < 2; ++d) {
        B[d].total = reinterpret_cast<int64_t *>(tmp + b_src) + d;
        B[d].src = reinterpret_cast<StripSrc *>(tmp) + d * nm[0];
        B[d].stage = reinterpret_cast<int32_t *>(tmp + b_src + 16) + d;
        B[d].far = reinterpret_cast<int32_t *>(tmp + b_src + 24) + d * nm[0];
        B[d].ofs = reinterpret_cast<uint32_t *>(tmp + at_ofs + (d ? b_ofs[0] : 0));
        B[d].units = reinterpret_cast<int32_t *>(u);
        B[d].bits = u + ng[d];
        u += 2 * ng[d];
        B[d].nsrc = (int32_t)nm[d];
        B[d].ng = ng[d];
        B[d].trans = d != 0;
        B[d].f64 = p->dtype == SPTRSV_F64;
        B[d].ring_most = strip_ring_most(B[d].f64, p->batched);
    }
    std::vector<char> back(b_back);
    int64_t total[2];
    e = cudaMemcpyAsync(tmp, src.data(), b_src, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(tmp + b_src, 0, b_back, s);
    for (int d = 0; d < 2 && e == cudaSuccess; ++d)
        if (nm[d]) e = strip_sizes(B[d], s, &scratch);
    if (e == cudaSuccess) e = cudaMemcpyAsync(back.data(), tmp + b_src, b_back, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    std::memcpy(total, back.data(), sizeof(total));
    if (e == cudaSuccess && (total[0] > INT32_MAX || total[1] > INT32_MAX)) e = cudaErrorMemoryAllocation;  // (32 GB)
    // one allocation: blocks, offsets and entry codes of both
    const size_t b_blocks = 16 * (size_t)(total[0] + total[1]);
    if (e == cudaSuccess)
        e = p->alloc_tables(&tab, b_blocks + b_ofs[0] + b_ofs[1] + 2 * (size_t)(nnz[0] + nnz[1]));
    if (e == cudaSuccess) e = cudaMemcpyAsync(tab + b_blocks, tmp + at_ofs, b_ofs[0] + b_ofs[1], cudaMemcpyDeviceToDevice, s);
    for (int d = 0; d < 2 && e == cudaSuccess; ++d) {
        if (!nm[d]) continue;
        unsigned char *blocks = reinterpret_cast<unsigned char *>(tab) + (d ? 16 * (size_t)total[0] : 0);
        uint32_t *ofs = reinterpret_cast<uint32_t *>(tab + b_blocks + (d ? b_ofs[0] : 0));
        uint16_t *ecode = reinterpret_cast<uint16_t *>(tab + b_blocks + b_ofs[0] + b_ofs[1]) + (d ? nnz[0] : 0);
        const int32_t *far = reinterpret_cast<const int32_t *>(back.data() + 24) + d * nm[0];
        const int32_t stage = reinterpret_cast<const int32_t *>(back.data() + 16)[d];
        e = strip_tables(B[d], ofs, blocks, ecode, s);
        for (size_t m = 0; m < nm[d] && e == cudaSuccess; ++m)
            mats[d][m]->strips[d] = Strips{blocks, ofs + src[d * nm[0] + m].g0, ecode + src[d * nm[0] + m].e0,
                                           strip_ring(far[m], B[d].ring_most), stage};
    }
    if (e != cudaSuccess && tab) {
        for (int d = 0; d < 2; ++d)
            for (PlanMat *M : mats[d]) M->strips[d] = Strips{};
        p->release(tab);
    }
    if (e != cudaSuccess) cudaGetLastError();
}

// Tables of the cluster flow schedule (flow.cuh).  One block
// of the cluster per 24 rows of the mean level: below that another block does
// not shorten a level (power-law DAG, 63 rows a level: 2 blocks 10.4 ms, 4
// 9.6 ms, 16 9.2 ms transpose).  Beyond 8 blocks only for very wide levels:
// with 16 the 2D Laplacian (512 rows a level) gains 6 % at one right-hand
// side, but the GPU holds too few such clusters for eight (5.0 against 3.5 ms).
// The directions [d0, d1) in one go and into one allocation (as the strips).
// The caller synchronises.
sptrsv_status build_flow(sptrsv_plan p, int d0, int d1, const Scratch *from)
{
    const PlanMat &M = p->M;
    const int32_t n = M.L.n, L = M.nlevels;
    const size_t nn = (size_t)n, nc = (size_t)L * kFlowClasses, nd = (size_t)(d1 - d0);
    cudaStream_t s = p->h->stream;
    const bool f64 = p->dtype == SPTRSV_F64;
    if (n > kFlowMaxRows) return SPTRSV_ENOTSUP;
    int csize = 1;
    const double width = (double)n / L;
    while (csize < (width >= 768.0 ? kFlowMaxCluster : 8) && width > 24.0 * csize) csize <<= 1;
    while (csize > 1 && !flow_cluster_fits(csize, f64)) csize >>= 1;
    if (!flow_cluster_fits(csize, f64)) return SPTRSV_ENOTSUP;
    // scratch: counts of all directions (read back), then by direction order,
    // its inverse, and the positions' blocks and masks
    int32_t *counts = nullptr;
    Scratch scratch(s, from);
    cudaError_t e = scratch.take(&counts, nd * (4 * nn + nc));
    if (e != cudaSuccess) return from_cuda(e);
    struct Dir {
        const int32_t *ptr, *idx;
        int32_t *order, *iperm;
        uint32_t *meta, *mask;
        int32_t g0, ng;  // its groups in the list of all
    } D[2];
    for (int d = d0; d < d1 && e == cudaSuccess; ++d) {
        Dir &Q = D[d - d0];
        Q.ptr = d ? M.d_cp : M.L.row_ptr;
        Q.idx = d ? M.d_crow : M.L.col_idx;
        Q.order = counts + nd * nc + (size_t)(d - d0) * 4 * nn;
        Q.iperm = Q.order + nn;
        Q.meta = reinterpret_cast<uint32_t *>(Q.iperm + nn);
        Q.mask = Q.meta + nn;
        e = flow_order(Q.ptr, M.d_lev, n, L, d != 0, Q.order, Q.iperm, counts + (size_t)(d - d0) * nc, s, &scratch);
    }
    std::vector<int32_t> cnt(nd * nc);
    if (e == cudaSuccess) e = cudaMemcpyAsync(cnt.data(), counts, sizeof(int32_t) * nd * nc, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    // groups of one level and class, an equal share of every level's groups,
    // in order, to each block of the cluster
    std::vector<FlowGroup> all;
    std::vector<int32_t> gptr;  // csize + 1 of each direction
    static const int llpr[kFlowClasses] = {0, 2, 4, 5};
    for (size_t d = 0; d < nd && e == cudaSuccess; ++d) {
        std::vector<std::vector<FlowGroup>> by((size_t)csize);
        std::vector<FlowGroup> lev;
        int32_t q = 0;
        for (int32_t l = 0; l < L; ++l) {
            lev.clear();
            for (int c = 0; c < kFlowClasses; ++c) {
                int32_t left = cnt[d * nc + (size_t)l * kFlowClasses + c];
                for (const int32_t most = 32 >> llpr[c]; left > 0;) {
                    const int32_t take = std::min(most, left);
                    lev.push_back(FlowGroup{q, take, llpr[c]});
                    q += take;
                    left -= take;
                }
            }
            const int64_t G = (int64_t)lev.size();
            for (int64_t g = 0; g < G; ++g) by[(size_t)(g * csize / G)].push_back(lev[(size_t)g]);
        }
        D[d].g0 = (int32_t)all.size();
        gptr.push_back(0);
        for (const auto &v : by) {
            all.insert(all.end(), v.begin(), v.end());
            gptr.push_back((int32_t)all.size() - D[d].g0);
        }
        D[d].ng = gptr.back();
    }
    // one allocation, so that nothing is left of tables that cannot be had
    const size_t ns = 32 * std::max<size_t>(all.size(), 1), w = f64 ? 8 : 4;
    const size_t at_codes = sizeof(FlowLane) * ns, at_vals = at_codes + sizeof(uint4) * ns;
    const size_t at_inv = at_vals + 4 * w * ns, at_src = at_inv + w * ns, at_ecode = at_src + sizeof(int2) * ns;
    const size_t at_gptr = at_ecode + sizeof(uint32_t) * (size_t)M.L.nnz * nd;
    char *tab = nullptr;
    FlowGroup *groups = nullptr;
    if (e == cudaSuccess) e = p->alloc_tables(&tab, at_gptr + sizeof(int32_t) * gptr.size());
    if (e == cudaSuccess) e = scratch.take(&groups, all.size());
    if (e == cudaSuccess) e = cudaMemcpyAsync(groups, all.data(), sizeof(FlowGroup) * all.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(tab + at_gptr, gptr.data(), sizeof(int32_t) * gptr.size(), cudaMemcpyHostToDevice, s);
    for (int d = d0; d < d1 && e == cudaSuccess; ++d) {
        const Dir &Q = D[d - d0];
        const size_t s0 = 32 * (size_t)Q.g0;
        FlowLane *lanes = reinterpret_cast<FlowLane *>(tab) + s0;
        uint4 *codes = reinterpret_cast<uint4 *>(tab + at_codes) + s0;
        int2 *src = reinterpret_cast<int2 *>(tab + at_src) + s0;
        uint32_t *ecode = reinterpret_cast<uint32_t *>(tab + at_ecode) + (size_t)(d - d0) * (size_t)M.L.nnz;
        const int32_t *d_gptr = reinterpret_cast<int32_t *>(tab + at_gptr) + (size_t)(d - d0) * ((size_t)csize + 1);
        e = flow_tables(Q.ptr, Q.idx, n, d != 0, f64, Q.order, Q.iperm, groups + Q.g0, d_gptr, Q.ng, csize, Q.meta,
                        Q.mask, lanes, codes, src, ecode, s);
        FlowSched F{};
        F.lanes = lanes;
        F.codes = codes;
        F.src = src;
        F.ecode = ecode;
        F.gptr = d_gptr;
        F.vals = tab + at_vals + 4 * w * s0;
        F.inv = tab + at_inv + w * s0;
        F.n = n;
        F.csize = csize;
        F.ngroups = Q.ng;
        p->flow[d] = F;
    }
    if (e != cudaSuccess) {
        if (tab) p->release(tab);
        return from_cuda(e);
    }
    for (int d = d0; d < d1; ++d) p->flow_ready[d] = true;
    return SPTRSV_OK;
}

// Whether the plan's settings call for the cluster flow schedule: the hybrid
// mode with its automatic threshold (one synchronisation-free run in level
// order) and grid.
bool flow_wanted(const sptrsv_plan_st *p)
{
    return p->mode == SPTRSV_MODE_HYBRID && p->thin_rows == 0 && p->grid_level == p->grid_level_max && p->M.L.n > 0;
}

// Builds the tables of the plan's mode and settings, so that a solve launches
// kernels only: called by whatever changes them.  Where the flow's tables
// cannot be had, the grid-wide hybrid kernel runs.
sptrsv_status prepare_schedules(sptrsv_plan p, const Scratch *from = nullptr)
{
    const int dirs = p->have_csc ? 2 : 1;
    auto open = [&](int d) { return flow_wanted(p) && d < dirs && !p->flow_ready[d] && !p->flow_off[d]; };
    bool built = open(0) || open(1);
    // (where there is no room for both directions, for one)
    if (!(open(0) && open(1)) || build_flow(p, 0, 2, from) != SPTRSV_OK)
        for (int d = 0; d < dirs; ++d)
            if (open(d)) p->flow_off[d] = build_flow(p, d, d + 1, from) != SPTRSV_OK;
    std::vector<PlanMat *> need[2];
    for (int d = 0; d < dirs; ++d)
        if (p->mode == SPTRSV_MODE_BLOCK && p->rpw == 32 && p->M.L.n > 0 && !p->M.strips[d].blocks)
            need[d].push_back(&p->M);
    build_strips(p, need, from);
    built = built || !need[0].empty() || !need[1].empty();
    sptrsv_status st = SPTRSV_OK;
    if (p->mode == SPTRSV_MODE_HYBRID && !(flow_wanted(p) && p->flow_ready[0] && p->flow_ready[dirs - 1]))
        st = ensure_hybrid(p);
    const cudaError_t e = built ? cudaStreamSynchronize(p->h->stream) : cudaSuccess;
    return st == SPTRSV_OK ? from_cuda(e) : st;
}

// Mode from the mean level width: narrow (deep) systems stay on one SM, very
// wide levels go level by level over the whole chip (row-order sync-free
// solving keeps only the rows in flight near the wavefront: 9x slower than
// level order on the 3D Laplacian), the rest takes the hybrid schedule on a
// cluster.  The upper line: 3D Laplacian, FP32, one column, level order against
// cluster at 1,744 rows a level 197 / 137 us, at 2,720 253 / 248, at 5,500 395 /
// 1,000 (eight columns cross at about 900: 130 / 156 us at 1,058).
int auto_mode(const PlanMat &M)
{
    if (M.L.n == 0 || M.nlevels == 0) return SPTRSV_MODE_SYNCFREE;
    const double width = (double)M.L.n / M.nlevels;
    if (width < 48.0) return SPTRSV_MODE_BLOCK;
    if (width >= 2048.0) return SPTRSV_MODE_LEVEL_PERSISTENT;
    return SPTRSV_MODE_HYBRID;
}

// Whether two [n x k] blocks of one leading dimension (elements of w bytes)
// share an element: their spans meet, and x is not made of other columns of
// b's rows.
bool share_elements(const void *b, const void *x, int32_t n, int32_t k, int64_t ld, size_t w)
{
    const int64_t span = ((int64_t)(n - 1) * ld + k) * (int64_t)w;
    const int64_t d = (const char *)x - (const char *)b;
    if (d >= span || -d >= span) return false;
    const int64_t row = ld * (int64_t)w, width = k * (int64_t)w;
    const int64_t at = ((d % row) + row) % row;  // x's first column, from the start of a row of b
    return at < width || at + width > row;
}

// The solves over strips read b a second time where a solution is not finite
// (strip.cuh), after x has been written: where the two share elements they
// read this copy of b, which has the same leading dimension.
struct OwnRhs {
    void *copy = nullptr;
    cudaStream_t s = nullptr;
    cudaError_t take(const void **b, int64_t n, int64_t k, int64_t ld, size_t w, cudaStream_t stream)
    {
        s = stream;
        const size_t span = ((size_t)(n - 1) * (size_t)ld + (size_t)k) * w, row = (size_t)ld * w;
        cudaError_t e = cudaMallocAsync(&copy, span, s);
        if (e != cudaSuccess) { copy = nullptr; return e; }
        if (n == 1 || k == ld)
            e = cudaMemcpyAsync(copy, *b, span, cudaMemcpyDeviceToDevice, s);
        else
            e = cudaMemcpy2DAsync(copy, row, *b, row, (size_t)k * w, (size_t)n, cudaMemcpyDeviceToDevice, s);
        *b = copy;
        return e;
    }
    ~OwnRhs()
    {
        if (copy) cudaFreeAsync(copy, s);
    }
};

template <class T>
sptrsv_status solve_impl(sptrsv_plan p, const void *b, void *x, int32_t nrhs, int64_t ld, bool trans)
{
    const PlanMat &M = p->M;
    if (M.L.n == 0) return SPTRSV_OK;
    if (!b || !x || nrhs < 1 || ld < nrhs) return SPTRSV_EINVAL;
    if (trans && !p->have_csc) return SPTRSV_ENOTSUP;
    cudaStream_t s = p->h->stream;
    Sys<T> A = sys_of<T>(M, p->h->d_status);
    int mode = p->mode;
    if (mode == SPTRSV_MODE_BLOCK && !block_mode_supported(nrhs, sizeof(T) == 8)) mode = SPTRSV_MODE_SYNCFREE;
    const int dir = trans ? 1 : 0;
    // schedules that lay the values out themselves
    const bool strips = mode == SPTRSV_MODE_BLOCK && p->rpw == 32 && M.strips[dir].blocks != nullptr;
    const bool flow = flow_wanted(p) && p->flow_ready[dir];
    OwnRhs own;
    if (strips && share_elements(b, x, M.L.n, nrhs, ld, sizeof(T))) {
        cudaError_t eo = own.take(&b, M.L.n, nrhs, ld, sizeof(T), s);
        if (eo != cudaSuccess) return from_cuda(eo);
    }
    Rhs<T> R{(const T *)b, (T *)x, ld, nrhs};
    // (k_level_cols fills x before it reads b)
    const size_t span = ((size_t)(M.L.n - 1) * (size_t)ld + (size_t)nrhs) * sizeof(T);
    const bool apart = (const char *)b + span <= (const char *)x || (const char *)x + span <= (const char *)b;
    const bool cols = mode == SPTRSV_MODE_LEVEL_PERSISTENT && p->rpw == 32 && apart;
    if (trans && !strips && !flow && !cols) {
        cudaError_t eg = csc_values<T>(M.d_tmap, (const T *)M.L.vals, (T *)M.d_cv, M.L.nnz, s);
        if (eg != cudaSuccess) return from_cuda(eg);
    }
    SyncArgs sy{p->d_flags, p->d_ctl, p->withhold, Waiter{p->h->d_status, &p->d_ctl->abort_flag, p->spin}};
    // one right-hand side: the synchronisation-free waits read the values
    // from the flags themselves
    if (nrhs == 1) sy.vflags = p->d_vflags;
    const int kt = std::min(p->kt, default_kt(nrhs));
    cudaError_t e = cudaSuccess;
    switch (mode) {
    case SPTRSV_MODE_LEVEL_LAUNCH:
        e = solve_level_launch<T>(A, M.d_perm, M.h_level_ptr, R, trans, s);
        break;
    case SPTRSV_MODE_LEVEL_PERSISTENT: {
        sptrsv_status st = ensure_chunks(p);
        if (st != SPTRSV_OK) return st;
        Sched S{M.d_perm, M.d_level_ptr, M.nlevels, trans ? p->d_chunk_tr : p->d_chunk_fwd,
                ((int64_t)M.L.n + p->rpw - 1) / p->rpw};
        if (cols) {
            e = solve_level_cols<T>(A, S, R, kt, trans, sy, p->grid_level, s);
            break;
        }
        const int64_t want = (2 * (int64_t)p->max_width / p->rpw + 7) / 8;  // blocks of 8 warps
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(p->grid_level, want));
        e = solve_level_persistent<T>(A, S, R, p->rpw, kt, trans, sy, grid, s);
        break;
    }
    case SPTRSV_MODE_HYBRID: {
        if (flow) {
            e = solve_flow<T>(A, p->flow[dir], R, trans, p->withhold, sy.w, s);
            break;
        }
        sptrsv_status st = ensure_chunks(p);
        if (st == SPTRSV_OK) st = ensure_hybrid(p);
        if (st != SPTRSV_OK) return st;
        Sched S{M.d_perm, M.d_level_ptr, M.nlevels, trans ? p->d_chunk_tr : p->d_chunk_fwd,
                ((int64_t)M.L.n + p->rpw - 1) / p->rpw, p->d_seg[trans ? 1 : 0], M.d_lev};
        e = solve_level_persistent<T>(A, S, R, p->rpw, kt, trans, sy, p->grid_level, s);
        break;
    }
    case SPTRSV_MODE_BLOCK: {
        const double width = M.nlevels > 0 ? (double)M.L.n / M.nlevels : 1.0;
        const int rpw = p->rpw == 32 && !strips ? 16 : p->rpw;
        e = solve_block<T>(A, M.strips[dir], R, rpw, trans, sy, block_warps_for(width, rpw), s);
        break;
    }
    default:
        e = solve_syncfree<T>(A, R, p->rpw, kt, trans, sy, p->grid_sf, s);
        break;
    }
    return debug_sync(from_cuda(e), s, trans ? "solve_transpose" : "solve");
}

}  // namespace

// --------------------------------------------------------------- validate
extern "C" sptrsv_status sptrsv_validate(sptrsv_handle h, const sptrsv_csr *L, int32_t *bad_row)
{
    if (!h) return SPTRSV_EINVAL;
    sptrsv_status st = check_csr(L);
    if (st != SPTRSV_OK) return st;
    return validate_impl(h, *L, bad_row);
}

// ---------------------------------------------------------------- analyze
extern "C" sptrsv_status sptrsv_analyze(sptrsv_handle h, const sptrsv_csr *L, int32_t *lev,
                                        int32_t *perm, int32_t *level_ptr, int64_t *level_cost,
                                        int32_t *nlevels, double stats[6])
{
    Range range("sptrsv_analyze");
    if (!h || !nlevels) return SPTRSV_EINVAL;
    sptrsv_status st = check_csr(L);
    if (st != SPTRSV_OK) return st;
    if (L->n > 0 && (!lev || !perm || !level_ptr || !level_cost)) return SPTRSV_EINVAL;
    if (L->n == 0) {
        *nlevels = 0;
        if (stats) for (int q = 0; q < 6; ++q) stats[q] = 0.0;
        if (level_ptr) cudaMemsetAsync(level_ptr, 0, sizeof(int32_t), h->stream);
        return from_cuda(cudaStreamSynchronize(h->stream));
    }
    double tmp[6];
    return analyze_into(h, *L, lev, perm, level_ptr, level_cost, nlevels, stats ? stats : tmp, kDefaultWaitNs);
}

extern "C" sptrsv_status sptrsv_analyze_incremental(sptrsv_handle h, const sptrsv_csr *L, int32_t first_row,
                                                    int32_t *lev, int32_t *perm, int32_t *level_ptr,
                                                    int64_t *level_cost, int32_t *nlevels, double stats[6])
{
    Range range("sptrsv_analyze_incremental");
    if (!h || !nlevels) return SPTRSV_EINVAL;
    sptrsv_status st = check_csr(L);
    if (st != SPTRSV_OK) return st;
    if (first_row < 0 || first_row > L->n) return SPTRSV_EINVAL;
    if (L->n == 0) return sptrsv_analyze(h, L, lev, perm, level_ptr, level_cost, nlevels, stats);
    if (!lev || !perm || !level_ptr || !level_cost) return SPTRSV_EINVAL;
    double tmp[6];
    return analyze_into(h, *L, lev, perm, level_ptr, level_cost, nlevels, stats ? stats : tmp, kDefaultWaitNs,
                        first_row);
}

extern "C" sptrsv_status sptrsv_level_summary(sptrsv_handle h, const sptrsv_csr *L, const int32_t *perm,
                                              const int32_t *level_ptr, const int64_t *level_cost,
                                              int32_t nlevels, double threshold, uint8_t *thin,
                                              int32_t *pick, int64_t summary[3])
{
    Range range("sptrsv_level_summary");
    if (!h || !L || !summary || nlevels < 0) return SPTRSV_EINVAL;
    if (nlevels > 0 && (!L->row_ptr || !perm || !level_ptr || !level_cost || !thin || !pick)) return SPTRSV_EINVAL;
    unsigned long long *d = reinterpret_cast<unsigned long long *>(h->d_scratch + 9);
    unsigned long long host[3] = {0, 0, 0};
    cudaError_t e = launch_level_summary(L->row_ptr, perm, level_ptr, level_cost, nlevels, threshold, thin, pick,
                                         d, h->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(host, d, sizeof(host), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return from_cuda(e);
    for (int q = 0; q < 3; ++q) summary[q] = (int64_t)host[q];
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_transpose(sptrsv_handle h, const sptrsv_csr *A, sptrsv_csr_out *At)
{
    Range range("sptrsv_transpose");
    if (!h || !A || !At || A->n < 0 || A->nnz < 0) return SPTRSV_EINVAL;
    if (A->dtype != SPTRSV_F64 && A->dtype != SPTRSV_F32) return SPTRSV_EINVAL;
    if (!At->row_ptr || (A->n > 0 && !A->row_ptr)) return SPTRSV_EINVAL;
    if (A->nnz > 0 && (!A->col_idx || !A->vals || !At->col_idx || !At->vals)) return SPTRSV_EINVAL;
    cudaStream_t s = h->stream;
    int32_t *tmap = nullptr;
    cudaError_t e = cudaMallocAsync(&tmap, sizeof(int32_t) * (size_t)(A->nnz > 0 ? A->nnz : 1), s);
    if (e == cudaSuccess) e = build_csc(A->row_ptr, A->col_idx, A->n, A->nnz, At->row_ptr, At->col_idx, tmap, s);
    if (e == cudaSuccess && A->nnz > 0)
        e = A->dtype == SPTRSV_F64
                ? csc_values<double>(tmap, (const double *)A->vals, (double *)At->vals, A->nnz, s)
                : csc_values<float>(tmap, (const float *)A->vals, (float *)At->vals, A->nnz, s);
    if (tmap) cudaFreeAsync(tmap, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return from_cuda(e);
}

// ---------------------------------------------------------------- rewrite
extern "C" sptrsv_status sptrsv_rewrite(sptrsv_handle h, const sptrsv_csr *L, const int32_t *lev,
                                        const int32_t *rows, const int32_t *targets, int32_t nrows,
                                        int64_t *nnz_Lp, int64_t *nnz_T, sptrsv_csr_out *Lp_out,
                                        sptrsv_csr_out *T_out)
{
    Range range("sptrsv_rewrite");
    if (!h || nrows < 0) return SPTRSV_EINVAL;
    sptrsv_status st = check_csr(L);
    if (st != SPTRSV_OK) return st;
    if (L->n > 0 && !lev) return SPTRSV_EINVAL;
    if (nrows > 0 && !rows) return SPTRSV_EINVAL;
    return (sptrsv_status)rewrite_run(*L, lev, rows, targets, nrows, nnz_Lp, nnz_T, Lp_out, T_out,
                                      h->di, h->stream);
}

// ------------------------------------------------------------------ plans
extern "C" sptrsv_status sptrsv_plan_create(sptrsv_handle h, const sptrsv_csr *L, const sptrsv_csr *T,
                                            const sptrsv_plan_opts *opts, sptrsv_plan *plan)
{
    Range range("sptrsv_plan_create");
    if (!h || !plan) return SPTRSV_EINVAL;
    *plan = nullptr;
    sptrsv_status st = check_csr(L);
    if (st != SPTRSV_OK) return st;
    sptrsv_plan p = new (std::nothrow) sptrsv_plan_st;
    if (!p) return SPTRSV_ENOMEM;
    p->h = h;
    p->dtype = L->dtype;
    sptrsv_plan_opts o{};
    if (opts) o = *opts;
    if (o.wait_limit_us > 0) p->spin = o.wait_limit_us * 1000;
    const size_t nn = (size_t)(L->n > 0 ? L->n : 1);
    p->reserve(p->padded(sizeof(PlanCtl)) + 3 * p->padded(4 * nn) + p->padded(16 * nn) + mat_bytes(*L, T, o.build_transpose != 0));
    cudaError_t e = p->alloc(&p->d_ctl, sizeof(PlanCtl));
    if (e == cudaSuccess) e = cudaMemset(p->d_ctl, 0, sizeof(PlanCtl));
    if (e == cudaSuccess) e = p->alloc(&p->d_flags, sizeof(uint32_t) * nn);
    if (e == cudaSuccess) e = cudaMemset(p->d_flags, 0, sizeof(uint32_t) * nn);
    if (e == cudaSuccess) e = p->alloc(&p->d_vflags, 16 * nn);
    if (e != cudaSuccess) { sptrsv_plan_destroy(p); return from_cuda(e); }
    unsigned long long nlong = 0;
    if (!valid_rpw(o.rows_per_warp)) {
        // (read back by the analysis' synchronisation)
        unsigned long long *d = reinterpret_cast<unsigned long long *>(h->d_scratch + 8);
        e = launch_count_long(L->row_ptr, L->n, 32, d, h->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&nlong, d, sizeof(nlong), cudaMemcpyDeviceToHost, h->stream);
        if (e == cudaSuccess && L->n == 0) e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) { sptrsv_plan_destroy(p); return from_cuda(e); }
    }
    DeviceArray<char> buffer;
    const size_t bytes = plan_scratch(L->n, L->nnz, o.build_transpose != 0);
    if (buffer.get(bytes) != cudaSuccess) cudaGetLastError();  // (then from the pool)
    const Scratch scratch(h->stream, buffer.p, bytes);
    // (the level costs go where the flags will be)
    st = prepare_mat(p, p->M, *L, T, o.build_transpose != 0, reinterpret_cast<int64_t *>(p->d_vflags), &scratch);
    if (st == SPTRSV_OK) st = from_cuda(cudaMemsetAsync(p->d_vflags, 0, 16 * nn, h->stream));
    if (st != SPTRSV_OK) { sptrsv_plan_destroy(p); return st; }
    p->have_csc = o.build_transpose != 0;
    p->mode = o.mode != SPTRSV_MODE_AUTO ? o.mode : auto_mode(p->M);
    if (valid_rpw(o.rows_per_warp)) {
        p->rpw = o.rows_per_warp;
    } else {
        p->rpw = p->mode == SPTRSV_MODE_BLOCK ? block_rpw(L->n, L->nnz, (int64_t)nlong)
                                              : default_rpw(L->n, L->nnz, (int64_t)nlong);
    }
    // the hybrid schedule waits row by row on flags: 4 rows per warp (8
    // lanes a row; on the 2D Laplacian 3.2 ms against 4.2 ms with one row
    // per warp), one row per warp where long rows call for a whole warp
    // (heavy tail or long mean row: the row-length rule above gave 1)
    if (p->mode == SPTRSV_MODE_HYBRID && !valid_rpw(o.rows_per_warp)) p->rpw = p->rpw == 1 ? 1 : 4;
    p->kt = valid_kt(o.rhs_tile) ? o.rhs_tile : 16;
    if (p->mode < SPTRSV_MODE_LEVEL_LAUNCH || p->mode > SPTRSV_MODE_HYBRID) { sptrsv_plan_destroy(p); return SPTRSV_EINVAL; }
    p->grid_level = persistent_grid_level(1, p->dtype == SPTRSV_F64, h->di);
    p->grid_level_max = p->grid_level;
    {
        // warps beyond about twice the widest level only poll the progress
        // counter: cap the level-persistent grid accordingly
        int32_t maxw = 0;
        for (int32_t l = 0; l < p->M.nlevels; ++l)
            maxw = std::max(maxw, p->M.h_level_ptr[l + 1] - p->M.h_level_ptr[l]);
        p->max_width = maxw;
    }
    p->grid_sf = persistent_grid_syncfree(1, p->dtype == SPTRSV_F64, h->di);
    st = ensure_chunks(p);
    // (what the solves cannot do without they ask for again)
    if (st == SPTRSV_OK) prepare_schedules(p, &scratch);
    if (st == SPTRSV_OK) st = from_cuda(cudaStreamSynchronize(h->stream));
    if (st != SPTRSV_OK) { sptrsv_plan_destroy(p); return st; }
    *plan = p;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_plan_destroy(sptrsv_plan p)
{
    if (!p) return SPTRSV_EINVAL;
    if (p->h) cudaStreamSynchronize(p->h->stream);
    for (auto &S : p->hset)
        for (cudaEvent_t ev : {S.h2d, S.comp, S.d2h})
            if (ev) cudaEventDestroy(ev);
    for (cudaStream_t st : {p->s_h2d, p->s_d2h})
        if (st) {
            cudaStreamSynchronize(st);
            cudaStreamDestroy(st);
        }
    if (p->d_lay) cudaFree(p->d_lay);
    for (void *q : p->owned) cudaFree(q);
    delete p;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_plan_set_thin_rows(sptrsv_plan p, int32_t thin_rows)
{
    if (!p || p->batched || thin_rows < 0) return SPTRSV_EINVAL;
    p->thin_rows = thin_rows;
    return prepare_schedules(p);
}

extern "C" sptrsv_status sptrsv_plan_set_blocks_per_sm(sptrsv_plan p, int32_t blocks_per_sm)
{
    if (!p || p->batched || blocks_per_sm < 0) return SPTRSV_EINVAL;
    const int sms = std::max(1, p->h->di.num_sms);
    const int cap = (int)std::min<int64_t>(p->grid_level_max, (int64_t)blocks_per_sm * sms);
    p->grid_level = blocks_per_sm == 0 ? p->grid_level_max : std::max(1, cap);
    return prepare_schedules(p);
}

extern "C" sptrsv_status sptrsv_plan_info(sptrsv_plan p, int32_t *nlevels, int32_t *mode,
                                          int32_t *rows_per_warp, int32_t *rhs_tile)
{
    if (!p) return SPTRSV_EINVAL;
    if (nlevels) {
        if (p->batched) {
            int32_t mx = 0;
            for (const PlanMat &M : p->mats) mx = std::max(mx, M.nlevels);
            *nlevels = mx;
        } else {
            *nlevels = p->M.nlevels;
        }
    }
    if (mode) *mode = p->batched ? SPTRSV_MODE_BLOCK : p->mode;
    if (rows_per_warp) *rows_per_warp = p->batched ? (p->geo[0].rpw.empty() ? 32 : p->geo[0].rpw[0]) : p->rpw;
    if (rhs_tile) *rhs_tile = p->batched ? (p->geo[0].tile.empty() ? 4 : p->tile_of(0, 0)) : p->kt;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_plan_set(sptrsv_plan p, int32_t mode, int32_t rows_per_warp, int32_t rhs_tile)
{
    if (!p || p->batched) return SPTRSV_EINVAL;
    if (mode < SPTRSV_MODE_AUTO || mode > SPTRSV_MODE_HYBRID) return SPTRSV_EINVAL;
    if (rows_per_warp != 0 && !valid_rpw(rows_per_warp)) return SPTRSV_EINVAL;
    if (rhs_tile != 0 && !valid_kt(rhs_tile)) return SPTRSV_EINVAL;
    p->mode = mode == SPTRSV_MODE_AUTO ? auto_mode(p->M) : mode;
    if (rows_per_warp) p->rpw = rows_per_warp;
    if (rhs_tile) p->kt = rhs_tile;
    sptrsv_status st = ensure_chunks(p);
    if (st != SPTRSV_OK) return st;
    prepare_schedules(p);
    return from_cuda(cudaStreamSynchronize(p->h->stream));
}

extern "C" sptrsv_status sptrsv_solve(sptrsv_plan p, const void *b, void *x, int32_t nrhs, int64_t ld)
{
    Range range("sptrsv_solve");
    if (!p || p->batched) return SPTRSV_EINVAL;
    return p->dtype == SPTRSV_F64 ? solve_impl<double>(p, b, x, nrhs, ld, false)
                                  : solve_impl<float>(p, b, x, nrhs, ld, false);
}

extern "C" sptrsv_status sptrsv_solve_transpose(sptrsv_plan p, const void *gx, void *gb, int32_t nrhs, int64_t ld)
{
    Range range("sptrsv_solve_transpose");
    if (!p || p->batched) return SPTRSV_EINVAL;
    return p->dtype == SPTRSV_F64 ? solve_impl<double>(p, gx, gb, nrhs, ld, true)
                                  : solve_impl<float>(p, gx, gb, nrhs, ld, true);
}

namespace {
template <class T>
sptrsv_status solve_colmajor(sptrsv_plan p, const void *b, void *x, int32_t nrhs, int64_t ld, bool trans)
{
    const int64_t n = p->M.L.n;
    const size_t need = 2 * sizeof(T) * (size_t)n * (size_t)nrhs;
    cudaStream_t s = p->h->stream;
    if (need > p->lay_bytes) {
        cudaError_t e = cudaStreamSynchronize(s);  // the old buffer may still be in use
        if (e == cudaSuccess && p->d_lay) e = cudaFree(p->d_lay);
        p->d_lay = nullptr;
        p->lay_bytes = 0;
        if (e == cudaSuccess) e = cudaMalloc(&p->d_lay, need);
        if (e != cudaSuccess) return from_cuda(e);
        p->lay_bytes = need;
    }
    T *rb = static_cast<T *>(p->d_lay);
    T *rx = rb + (size_t)n * nrhs;
    // column r of b (element (i, r) at r * ld + i) -> row-major [n x nrhs]
    cudaError_t e = transpose_dense<T>(static_cast<const T *>(b), ld, rb, nrhs, nrhs, n, s);
    if (e != cudaSuccess) return from_cuda(e);
    sptrsv_status st = solve_impl<T>(p, rb, rx, nrhs, nrhs, trans);
    if (st != SPTRSV_OK) return st;
    return from_cuda(transpose_dense<T>(rx, nrhs, static_cast<T *>(x), ld, n, nrhs, s));
}
}  // namespace

extern "C" sptrsv_status sptrsv_solve_layout(sptrsv_plan p, const void *b, void *x, int32_t nrhs, int64_t ld,
                                             int32_t layout, int32_t transpose)
{
    Range range("sptrsv_solve_layout");
    if (!p || p->batched || (layout != SPTRSV_ROW_MAJOR && layout != SPTRSV_COL_MAJOR)) return SPTRSV_EINVAL;
    const bool tr = transpose != 0;
    if (layout == SPTRSV_ROW_MAJOR || nrhs == 1) {
        // one column: both layouts are the same vector
        const int64_t ldr = layout == SPTRSV_ROW_MAJOR ? ld : 1;
        if (layout == SPTRSV_COL_MAJOR && ld < p->M.L.n) return SPTRSV_EINVAL;
        return p->dtype == SPTRSV_F64 ? solve_impl<double>(p, b, x, nrhs, ldr, tr)
                                      : solve_impl<float>(p, b, x, nrhs, ldr, tr);
    }
    if (p->M.L.n == 0) return SPTRSV_OK;
    if (!b || !x || nrhs < 1 || ld < p->M.L.n) return SPTRSV_EINVAL;
    if (tr && !p->have_csc) return SPTRSV_ENOTSUP;
    return p->dtype == SPTRSV_F64 ? solve_colmajor<double>(p, b, x, nrhs, ld, tr)
                                  : solve_colmajor<float>(p, b, x, nrhs, ld, tr);
}

extern "C" sptrsv_status sptrsv_grad_vals(sptrsv_plan p, const void *gb, const void *x, int32_t nrhs,
                                          int64_t ld, void *gvals)
{
    Range range("sptrsv_grad_vals");
    if (!p || p->batched) return SPTRSV_EINVAL;
    if (p->M.L.n == 0) return SPTRSV_OK;
    if (!gb || !x || !gvals || nrhs < 1 || ld < nrhs) return SPTRSV_EINVAL;
    cudaError_t e;
    if (p->dtype == SPTRSV_F64)
        e = grad_vals<double>(sys_of<double>(p->M, p->h->d_status), (const double *)gb, (const double *)x, ld, nrhs, (double *)gvals, p->h->stream);
    else
        e = grad_vals<float>(sys_of<float>(p->M, p->h->d_status), (const float *)gb, (const float *)x, ld, nrhs, (float *)gvals, p->h->stream);
    return from_cuda(e);
}

extern "C" sptrsv_status sptrsv_tt_apply(sptrsv_plan p, const void *gbp, void *gb, int32_t nrhs, int64_t ld)
{
    Range range("sptrsv_tt_apply");
    if (!p || p->batched) return SPTRSV_EINVAL;
    if (p->M.L.n == 0) return SPTRSV_OK;
    if (!gbp || !gb || nrhs < 1 || ld < nrhs) return SPTRSV_EINVAL;
    cudaError_t e;
    if (p->dtype == SPTRSV_F64)
        e = tt_apply<double>(sys_of<double>(p->M, p->h->d_status), (const double *)gbp, (double *)gb, ld, nrhs, p->h->stream);
    else
        e = tt_apply<float>(sys_of<float>(p->M, p->h->d_status), (const float *)gbp, (float *)gb, ld, nrhs, p->h->stream);
    return from_cuda(e);
}

extern "C" sptrsv_status sptrsv_debug_withhold_row(sptrsv_plan p, int32_t row)
{
    if (!p) return SPTRSV_EINVAL;
    p->withhold = row;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_debug_withhold_level(sptrsv_handle h, int32_t row, int64_t wait_limit_us)
{
    if (!h || (row >= 0 && wait_limit_us <= 0)) return SPTRSV_EINVAL;
    h->dbg_withhold = row < 0 ? -1 : row;
    h->dbg_wait_ns = row < 0 ? 0 : wait_limit_us * 1000;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_debug_limit_tables(sptrsv_handle h, int64_t bytes)
{
    if (!h) return SPTRSV_EINVAL;
    h->dbg_table_limit = bytes < 0 ? -1 : bytes;
    return SPTRSV_OK;
}

// ----------------------------------------------------------------- batched
namespace {
bool valid_tile(int t) { return t == 1 || t == 2 || t == 4 || t == 8; }

int pow2_at_least(int v)
{
    int k = 1;
    while (k < v) k <<= 1;
    return k;
}

// Work items of one direction of a batch: every system is split into tiles
// of at most `tile` right-hand-side columns, each an independent in-order
// chain solved by one thread block.  Builds the items with their geometry,
// orders them longest estimated chain first (LPT), and sizes shared memory
// and the grid.
sptrsv_status rebuild_items(sptrsv_plan p, int dir)
{
    sptrsv_plan_st::Geom &G = p->geo[dir];
    const int32_t nmat = (int32_t)p->mats.size();
    const bool f64 = p->dtype == SPTRSV_F64;
    std::vector<BatchItem> items;
    std::vector<double> est;
    size_t smem = 16;
    G.csc_vals = G.strips = false;
    G.stage = 0;
    auto takes_strips = [&](int m) { return p->takes_strips(dir, m); };
    std::vector<PlanMat *> need[2];
    p->strips_to_build(dir, &need[dir]);
    build_strips(p, need);
    // (only systems solved over them: the others' values need not be laid out
    // before every solve)
    bool changed = false;
    for (int m = 0; m < nmat; ++m) {
        Strips &V = p->h_mats[m].strips[dir];
        const Strips use = takes_strips(m) ? p->mats[m].strips[dir] : Strips{};
        changed = changed || V.blocks != use.blocks;
        V = use;
    }
    if (changed) {
        cudaError_t e = cudaStreamSynchronize(p->h->stream);
        if (e == cudaSuccess)
            e = cudaMemcpy(p->d_mats, p->h_mats.data(), sizeof(BatchMat) * nmat, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return from_cuda(e);
    }
    for (int m = 0; m < nmat; ++m) {
        PlanMat &M = p->mats[m];
        const int k = p->h_mats[m].k;
        int tile = p->tile_of(dir, (size_t)m);
        // one lane per row, over the strips
        const bool one_lane = G.rpw[m] == 32 && (!takes_strips(m) || M.strips[dir].blocks || (dir == 1 && !p->have_csc));
        G.csc_vals = G.csc_vals || G.sched[m] == kSchedLevel || !one_lane;
        if (G.sched[m] == kSchedInOrder && one_lane) tile = std::min(tile, 4);
        for (int r0 = 0; r0 < k; r0 += tile) {
            BatchItem I{};
            I.mat = m;
            I.r0 = r0;
            I.kt = std::min(tile, k - r0);
            I.KT = pow2_at_least(I.kt);
            I.sched = G.sched[m];
            I.rpw = I.sched == kSchedLevel ? 32 : G.rpw[m] == 32 && !one_lane ? 16 : G.rpw[m];
            if (I.sched == kSchedInOrder && I.rpw == 32) {
                G.strips = true;
                G.stage = std::max(G.stage, (int)M.strips[dir].stage);
                I.nw = kBatchWarps;
                smem = std::max(smem, strip_smem(M.strips[dir].ring, I.KT, f64, kBatchWarps));
            } else {
                I.nw = I.sched == kSchedLevel
                           ? kBatchWarps
                           : std::min(kBatchWarps,
                                      block_warps_for(M.nlevels > 0 ? (double)M.L.n / M.nlevels : 1.0, I.rpw));
                block_geometry(I.rpw, I.KT, f64, I.nw, &I.kc, &I.P, kBatchSmemGrow);
                smem = std::max(smem, block_smem_bytes(I.rpw, I.KT, I.kc, f64));
            }
            items.push_back(I);
            // in order: a chain of n / 32 row groups whose cost grows with
            // the tile width; level-ordered: a chain of one or more groups per
            // level (each about a third of an in-order group); plus the
            // streamed matrix
            const double chain = I.sched == kSchedLevel ? 12.0 * (double)M.nlevels + 0.1 * (double)M.L.n
                                                        : (double)M.L.n;
            est.push_back(chain * (1.0 + 0.1 * I.KT) + 0.01 * (double)M.L.nnz);
        }
    }
    if (smem > kBlockSmemBudget) return SPTRSV_ENOTSUP;
    const int32_t ni = (int32_t)items.size();
    if (ni > p->max_items) return SPTRSV_EINVAL;
    std::vector<int32_t> order((size_t)ni);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return est[x] > est[y]; });
    cudaError_t e = cudaStreamSynchronize(p->h->stream);
    if (e == cudaSuccess && ni > 0)
        e = cudaMemcpy(G.d_items, items.data(), sizeof(BatchItem) * ni, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && ni > 0)
        e = cudaMemcpy(G.d_order, order.data(), sizeof(int32_t) * ni, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return from_cuda(e);
    G.nitems = ni;
    G.smem = smem;
    G.grid = std::min(batch_grid(smem, p->h->di), std::max(ni, 1));
    return SPTRSV_OK;
}

// Tables of the level-ordered schedule of system m in direction dir: the
// inverse permutation (once per system) and the row groups: every level's
// positions cut into groups of at most 32, in level order (forward) or in
// reverse level order (transpose), each with the number of groups of the
// levels before it in that order.
sptrsv_status ensure_level_tables(sptrsv_plan p, int m, int dir)
{
    PlanMat &M = p->mats[m];
    const int32_t n = M.L.n;
    cudaError_t e = cudaSuccess;
    if (!M.d_iperm) {
        e = p->alloc(&M.d_iperm, sizeof(int32_t) * (size_t)std::max(n, 1));
        if (e == cudaSuccess) e = inverse_perm(M.d_perm, M.d_iperm, n, p->h->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(p->h->stream);
        if (e != cudaSuccess) return from_cuda(e);
    }
    if (!M.d_lgroups[dir]) {
        std::vector<LevelGroup> g;
        const int32_t L = M.nlevels;
        const std::vector<int32_t> &lp = M.h_level_ptr;
        for (int32_t k = 0; k < L; ++k) {
            const int32_t l = dir == 0 ? k : L - 1 - k;
            // positions of level l in this direction's order
            const int32_t s = dir == 0 ? lp[l] : n - lp[l + 1];
            const int32_t t = dir == 0 ? lp[l + 1] : n - lp[l];
            const int32_t first = (int32_t)g.size();
            for (int32_t q = s; q < t; q += 32) g.push_back(LevelGroup{q, std::min(32, t - q), t, first});
        }
        e = p->alloc(&M.d_lgroups[dir], sizeof(LevelGroup) * std::max<size_t>(g.size(), 1));
        if (e == cudaSuccess && !g.empty())
            e = cudaMemcpy(M.d_lgroups[dir], g.data(), sizeof(LevelGroup) * g.size(), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return from_cuda(e);
        M.n_lgroups[dir] = (int32_t)g.size();
    }
    BatchMat &B = p->h_mats[m];
    B.perm = M.d_perm;
    B.iperm = M.d_iperm;
    B.lgroups[dir] = M.d_lgroups[dir];
    B.nlgroups[dir] = M.n_lgroups[dir];
    e = cudaStreamSynchronize(p->h->stream);
    if (e == cudaSuccess) e = cudaMemcpy(p->d_mats + m, &B, sizeof(BatchMat), cudaMemcpyHostToDevice);
    return from_cuda(e);
}

// New per-system schedules (SPTRSV_BATCH_INORDER / _LEVEL; 0 keeps) for the
// directions in `dirs`.
sptrsv_status set_schedule(sptrsv_plan p, int dirs, const int32_t *schedule)
{
    const int32_t nmat = (int32_t)p->h_mats.size();
    for (int m = 0; m < nmat; ++m)
        if (schedule[m] != 0 && schedule[m] != SPTRSV_BATCH_INORDER && schedule[m] != SPTRSV_BATCH_LEVEL)
            return SPTRSV_EINVAL;
    for (int d = 0; d < 2; ++d) {
        if (!((dirs >> d) & 1)) continue;
        sptrsv_plan_st::Geom &G = p->geo[d];
        const std::vector<int32_t> old = G.sched;
        for (int m = 0; m < nmat; ++m) {
            if (schedule[m] == SPTRSV_BATCH_LEVEL) {
                sptrsv_status st = ensure_level_tables(p, m, d);
                if (st != SPTRSV_OK) return st;
                G.sched[m] = kSchedLevel;
            } else if (schedule[m] == SPTRSV_BATCH_INORDER) {
                G.sched[m] = kSchedInOrder;
            }
        }
        sptrsv_status st = rebuild_items(p, d);
        if (st == SPTRSV_ENOTSUP) {
            G.sched = old;
            if (rebuild_items(p, d) != SPTRSV_OK) return SPTRSV_ECUDA;
        }
        if (st != SPTRSV_OK) return st;
    }
    return SPTRSV_OK;
}

// New per-system geometry for the directions in `dirs` (bit 0 forward, bit
// 1 transpose); values 0 keep the current one.  A geometry that does not fit
// in shared memory is refused and the previous one kept.
sptrsv_status set_geometry(sptrsv_plan p, int dirs, const int32_t *rows_per_warp, const int32_t *rhs_tile)
{
    const int32_t nmat = (int32_t)p->h_mats.size();
    for (int m = 0; m < nmat; ++m) {
        if (rows_per_warp && rows_per_warp[m] != 0 && !valid_rpw(rows_per_warp[m])) return SPTRSV_EINVAL;
        if (rhs_tile && rhs_tile[m] != 0 && !valid_tile(rhs_tile[m])) return SPTRSV_EINVAL;
    }
    for (int d = 0; d < 2; ++d) {
        if (!((dirs >> d) & 1)) continue;
        sptrsv_plan_st::Geom &G = p->geo[d];
        const std::vector<int32_t> old_rpw = G.rpw, old_tile = G.tile;
        for (int m = 0; m < nmat; ++m) {
            if (rows_per_warp && rows_per_warp[m]) G.rpw[m] = rows_per_warp[m];
            if (rhs_tile && rhs_tile[m]) G.tile[m] = rhs_tile[m];
        }
        sptrsv_status st = rebuild_items(p, d);
        if (st == SPTRSV_ENOTSUP) {
            G.rpw = old_rpw;
            G.tile = old_tile;
            if (rebuild_items(p, d) != SPTRSV_OK) return SPTRSV_ECUDA;
        }
        if (st != SPTRSV_OK) return st;
    }
    return SPTRSV_OK;
}
}  // namespace

extern "C" sptrsv_status sptrsv_batch_plan_create(sptrsv_handle h, int32_t nmat, const sptrsv_csr *Ls,
                                                  const sptrsv_csr *Ts, const int32_t *nrhs,
                                                  const sptrsv_plan_opts *opts, sptrsv_plan *plan)
{
    Range range("sptrsv_batch_plan_create");
    if (!h || !plan || nmat < 0 || (nmat > 0 && (!Ls || !nrhs))) return SPTRSV_EINVAL;
    *plan = nullptr;
    sptrsv_plan p = new (std::nothrow) sptrsv_plan_st;
    if (!p) return SPTRSV_ENOMEM;
    p->h = h;
    p->batched = true;
    p->dtype = nmat > 0 ? Ls[0].dtype : SPTRSV_F32;
    p->have_csc = false;
    bool want_csc = false;
    for (int m = 0; m < nmat && opts; ++m) want_csc = want_csc || opts[m].build_transpose;
    if (opts && opts[0].wait_limit_us > 0) p->spin = opts[0].wait_limit_us * 1000;
    size_t mats_bytes = 0, bytes = 0;
    int32_t n_most = 1;
    for (int m = 0; m < nmat; ++m) {
        if (check_csr(&Ls[m]) != SPTRSV_OK) continue;  // (refused below)
        mats_bytes += mat_bytes(Ls[m], Ts ? &Ts[m] : nullptr, want_csc);
        n_most = std::max(n_most, Ls[m].n);
        bytes = std::max(bytes, plan_scratch(Ls[m].n, Ls[m].nnz, want_csc));
    }
    p->reserve(p->padded(sizeof(PlanCtl)) + mats_bytes);
    cudaError_t e = p->alloc(&p->d_ctl, sizeof(PlanCtl));
    if (e == cudaSuccess) e = cudaMemset(p->d_ctl, 0, sizeof(PlanCtl));
    if (e != cudaSuccess) { sptrsv_plan_destroy(p); return from_cuda(e); }
    // scratch of every system in turn, its level costs first
    DeviceArray<char> buffer;
    bytes += Scratch::padded(sizeof(int64_t) * (size_t)n_most);
    if (buffer.get(bytes) != cudaSuccess) cudaGetLastError();  // (then from the pool)
    Scratch scratch(h->stream, buffer.p, bytes);
    int64_t *cost = nullptr;
    e = scratch.take(&cost, (size_t)n_most);
    if (e != cudaSuccess) { sptrsv_plan_destroy(p); return from_cuda(e); }
    p->mats.resize((size_t)nmat);
    p->rhs_off.assign((size_t)nmat + 1, 0);
    p->vals_off.assign((size_t)nmat + 1, 0);
    p->row_off.assign((size_t)nmat + 1, 0);
    p->h_mats.resize((size_t)nmat);
    for (int d = 0; d < 2; ++d) {
        p->geo[d].rpw.assign((size_t)nmat, 32);
        p->geo[d].tile.assign((size_t)nmat, 0);
        p->geo[d].sched.assign((size_t)nmat, kSchedInOrder);
    }
    int64_t ktot = 0;
    for (int m = 0; m < nmat; ++m) {
        sptrsv_status st = check_csr(&Ls[m]);
        if (st == SPTRSV_OK && (Ls[m].dtype != p->dtype || nrhs[m] < 1)) st = SPTRSV_EINVAL;
        if (st == SPTRSV_OK && opts && opts[m].rows_per_warp != 0 && !valid_rpw(opts[m].rows_per_warp))
            st = SPTRSV_EINVAL;
        if (st == SPTRSV_OK && opts && opts[m].rhs_tile != 0 && !valid_tile(opts[m].rhs_tile))
            st = SPTRSV_EINVAL;
        if (st == SPTRSV_OK) st = prepare_mat(p, p->mats[m], Ls[m], Ts ? &Ts[m] : nullptr, want_csc, cost, &scratch);
        if (st != SPTRSV_OK) { sptrsv_plan_destroy(p); return st; }
        const PlanMat &M = p->mats[m];
        BatchMat &B = p->h_mats[m];
        B.n = M.L.n;
        B.k = nrhs[m];
        B.nnz = M.L.nnz;
        B.rp = M.L.row_ptr; B.ci = M.L.col_idx; B.v = M.L.vals;
        B.cp = M.d_cp; B.crow = M.d_crow; B.tmap = M.d_tmap; B.cv = M.d_cv;
        B.trp = M.hasT ? M.T.row_ptr : nullptr;
        B.tci = M.hasT ? M.T.col_idx : nullptr;
        B.tv = M.hasT ? M.T.vals : nullptr;
        B.tmask = M.hasT ? M.d_tmask : nullptr;
        B.tcp = M.d_tcp; B.trow = M.d_trow; B.ttmap = M.d_ttmap;
        B.rhs_off = p->rhs_off[m];
        B.vals_off = p->vals_off[m];
        B.row_off = p->row_off[m];
        p->rhs_off[m + 1] = p->rhs_off[m] + (int64_t)M.L.n * B.k;
        p->vals_off[m + 1] = p->vals_off[m] + M.L.nnz;
        p->row_off[m + 1] = p->row_off[m] + M.L.n;
        for (int d = 0; d < 2; ++d) {
            p->geo[d].rpw[m] = opts && opts[m].rows_per_warp ? opts[m].rows_per_warp : block_rpw(M.L.n, M.L.nnz);
            if (opts && opts[m].rhs_tile) p->geo[d].tile[m] = opts[m].rhs_tile;
        }
        ktot += B.k;
    }
    p->have_csc = want_csc;
    p->max_items = (int32_t)std::max<int64_t>(ktot, 1);  // tiles of one column at most
    e = p->alloc(&p->d_mats, sizeof(BatchMat) * (size_t)(nmat > 0 ? nmat : 1));
    for (int d = 0; d < 2; ++d) {
        if (e == cudaSuccess) e = p->alloc(&p->geo[d].d_items, sizeof(BatchItem) * (size_t)p->max_items);
        if (e == cudaSuccess) e = p->alloc(&p->geo[d].d_order, sizeof(int32_t) * (size_t)p->max_items);
    }
    if (e == cudaSuccess) e = p->alloc(&p->d_trace, sizeof(long long) * 3 * (size_t)p->max_items);
    if (e == cudaSuccess && nmat > 0)
        e = cudaMemcpy(p->d_mats, p->h_mats.data(), sizeof(BatchMat) * nmat, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { sptrsv_plan_destroy(p); return from_cuda(e); }
    {
        // chunk tables of the elementwise adjoint kernels: every 32-row chunk,
        // and the chunks whose T-column mask word is non-zero
        std::vector<RowChunk> g, t, f;
        std::vector<uint32_t> mask;
        e = cudaStreamSynchronize(p->h->stream);  // T-row masks are built on the handle's stream
        for (int m = 0; m < nmat && e == cudaSuccess; ++m) {
            const PlanMat &M = p->mats[m];
            const int32_t nw = (M.L.n + 31) / 32;
            for (int32_t c = 0; c < nw; ++c) g.push_back(RowChunk{m, 32 * c});
            if (!M.hasT || nw == 0) continue;
            for (int32_t c = 0; c < nw; ++c) f.push_back(RowChunk{m, 32 * c});
            mask.resize((size_t)nw);
            e = cudaMemcpy(mask.data(), M.d_tcmask, sizeof(uint32_t) * nw, cudaMemcpyDeviceToHost);
            for (int32_t c = 0; c < nw && e == cudaSuccess; ++c)
                if (mask[c]) t.push_back(RowChunk{m, 32 * c});
        }
        p->n_gchunks = (int64_t)g.size();
        p->n_tchunks = (int64_t)t.size();
        p->n_fchunks = (int64_t)f.size();
        if (e == cudaSuccess && want_csc) {
            std::vector<RowChunk> ct;
            for (int m = 0; m < nmat; ++m)
                for (int64_t q = 0; q < p->mats[m].L.nnz; q += kCscTile) ct.push_back(RowChunk{m, (int32_t)q});
            p->n_ctiles = (int64_t)ct.size();
            if (!ct.empty()) {
                e = p->alloc(&p->d_ctiles, sizeof(RowChunk) * ct.size());
                if (e == cudaSuccess)
                    e = cudaMemcpy(p->d_ctiles, ct.data(), sizeof(RowChunk) * ct.size(), cudaMemcpyHostToDevice);
            }
        }
        if (e == cudaSuccess && !f.empty()) {
            e = p->alloc(&p->d_fchunks, sizeof(RowChunk) * f.size());
            if (e == cudaSuccess)
                e = cudaMemcpy(p->d_fchunks, f.data(), sizeof(RowChunk) * f.size(), cudaMemcpyHostToDevice);
            if (e == cudaSuccess)
                e = p->alloc(&p->d_bt, (p->dtype == SPTRSV_F64 ? 8 : 4) * (size_t)std::max<int64_t>(p->rhs_off[nmat], 1));
        }
        if (e == cudaSuccess) e = p->alloc(&p->d_gchunks, sizeof(RowChunk) * std::max<size_t>(g.size(), 1));
        if (e == cudaSuccess) e = p->alloc(&p->d_tchunks, sizeof(RowChunk) * std::max<size_t>(t.size(), 1));
        if (e == cudaSuccess && !g.empty())
            e = cudaMemcpy(p->d_gchunks, g.data(), sizeof(RowChunk) * g.size(), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && !t.empty())
            e = cudaMemcpy(p->d_tchunks, t.data(), sizeof(RowChunk) * t.size(), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) { sptrsv_plan_destroy(p); return from_cuda(e); }
    }
    std::vector<PlanMat *> need[2];
    for (int d = 0; d < 2; ++d) p->strips_to_build(d, &need[d]);
    build_strips(p, need, &scratch);
    sptrsv_status st = rebuild_items(p, 0);
    if (st == SPTRSV_OK) st = rebuild_items(p, 1);
    if (st != SPTRSV_OK) { sptrsv_plan_destroy(p); return st; }
    *plan = p;
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_batch_plan_set(sptrsv_plan p, const int32_t *rows_per_warp,
                                               const int32_t *rhs_tile)
{
    if (!p || !p->batched) return SPTRSV_EINVAL;
    return set_geometry(p, 3, rows_per_warp, rhs_tile);
}

extern "C" sptrsv_status sptrsv_batch_plan_set_direction(sptrsv_plan p, int32_t direction,
                                                         const int32_t *rows_per_warp, const int32_t *rhs_tile)
{
    if (!p || !p->batched || direction < 0 || direction > 2) return SPTRSV_EINVAL;
    return set_geometry(p, direction == 0 ? 3 : direction, rows_per_warp, rhs_tile);
}

extern "C" sptrsv_status sptrsv_batch_plan_set_schedule(sptrsv_plan p, int32_t direction, const int32_t *schedule)
{
    Range range("sptrsv_batch_plan_set_schedule");
    if (!p || !p->batched || !schedule || direction < 0 || direction > 2) return SPTRSV_EINVAL;
    return set_schedule(p, direction == 0 ? 3 : direction, schedule);
}

extern "C" sptrsv_status sptrsv_batch_offsets(sptrsv_plan p, int64_t *rhs_offset, int64_t *vals_offset)
{
    if (!p || !p->batched) return SPTRSV_EINVAL;
    if (rhs_offset) std::copy(p->rhs_off.begin(), p->rhs_off.end(), rhs_offset);
    if (vals_offset) std::copy(p->vals_off.begin(), p->vals_off.end(), vals_offset);
    return SPTRSV_OK;
}

namespace {
sptrsv_status batch_solve_impl(sptrsv_plan p, const void *b, void *x, bool trans)
{
    if (!p || !p->batched) return SPTRSV_EINVAL;
    const sptrsv_plan_st::Geom &G = p->geo[trans ? 1 : 0];
    if (G.nitems == 0) return SPTRSV_OK;
    if (!b || !x) return SPTRSV_EINVAL;
    if (trans && !p->have_csc) return SPTRSV_ENOTSUP;
    p->last_dir = trans ? 1 : 0;
    OwnRhs own;
    const int64_t total = p->rhs_off.back();
    const size_t wb = p->dtype == SPTRSV_F64 ? 8 : 4;
    if (G.strips && (const char *)x < (const char *)b + total * wb && (const char *)b < (const char *)x + total * wb) {
        cudaError_t eo = own.take(&b, 1, total, total, wb, p->h->stream);
        if (eo != cudaSuccess) return from_cuda(eo);
    }
    Waiter w{p->h->d_status, &p->d_ctl->abort_flag, p->spin};
    cudaError_t e = cudaSuccess;
    if (trans && G.csc_vals)
        e = p->dtype == SPTRSV_F64 ? batch_csc_values<double>(p->d_mats, p->d_ctiles, p->n_ctiles, p->h->stream)
                                   : batch_csc_values<float>(p->d_mats, p->d_ctiles, p->n_ctiles, p->h->stream);
    if (e == cudaSuccess && G.strips)
        e = p->dtype == SPTRSV_F64
                ? strip_stage_batch<double>(p->d_mats, p->d_gchunks, p->n_gchunks, G.stage, trans, p->h->stream)
                : strip_stage_batch<float>(p->d_mats, p->d_gchunks, p->n_gchunks, G.stage, trans, p->h->stream);
    if (e != cudaSuccess) return from_cuda(e);
    if (p->dtype == SPTRSV_F64)
        e = batch_solve<double>(p->d_mats, G.d_items, G.nitems, G.d_order, (const double *)b, (double *)x,
                                trans, p->d_ctl, w, G.grid, G.smem, p->d_trace, p->withhold,
                                p->d_fchunks, p->n_fchunks, (double *)p->d_bt, p->h->stream);
    else
        e = batch_solve<float>(p->d_mats, G.d_items, G.nitems, G.d_order, (const float *)b, (float *)x,
                               trans, p->d_ctl, w, G.grid, G.smem, p->d_trace, p->withhold,
                               p->d_fchunks, p->n_fchunks, (float *)p->d_bt, p->h->stream);
    return debug_sync(from_cuda(e), p->h->stream, "batch_solve");
}
}  // namespace

extern "C" sptrsv_status sptrsv_batch_solve(sptrsv_plan p, const void *b, void *x)
{
    Range range("sptrsv_batch_solve");
    return batch_solve_impl(p, b, x, false);
}

extern "C" sptrsv_status sptrsv_batch_solve_transpose(sptrsv_plan p, const void *gx, void *gb)
{
    Range range("sptrsv_batch_solve_transpose");
    return batch_solve_impl(p, gx, gb, true);
}

extern "C" sptrsv_status sptrsv_batch_trace(sptrsv_plan p, int64_t *trace)
{
    if (!p || !p->batched || !trace) return SPTRSV_EINVAL;
    const size_t nmat = p->mats.size();
    if (nmat == 0) return SPTRSV_OK;
    const sptrsv_plan_st::Geom &G = p->geo[p->last_dir];
    std::vector<long long> t(3 * (size_t)G.nitems);
    std::vector<BatchItem> items((size_t)G.nitems);
    cudaError_t e = cudaStreamSynchronize(p->h->stream);
    if (e == cudaSuccess && G.nitems > 0)
        e = cudaMemcpy(t.data(), p->d_trace, sizeof(long long) * t.size(), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && G.nitems > 0)
        e = cudaMemcpy(items.data(), G.d_items, sizeof(BatchItem) * items.size(), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return from_cuda(e);
    // per system: earliest start and latest end over its work items, and the
    // SM that started first
    for (size_t m = 0; m < nmat; ++m) {
        trace[3 * m] = INT64_MAX;
        trace[3 * m + 1] = 0;
        trace[3 * m + 2] = -1;
    }
    for (int32_t it = 0; it < G.nitems; ++it) {
        const int m = items[(size_t)it].mat;
        if (t[3 * (size_t)it] < trace[3 * m]) {
            trace[3 * m] = t[3 * (size_t)it];
            trace[3 * m + 2] = t[3 * (size_t)it + 2];
        }
        trace[3 * m + 1] = std::max<int64_t>(trace[3 * m + 1], t[3 * (size_t)it + 1]);
    }
    return SPTRSV_OK;
}

extern "C" sptrsv_status sptrsv_batch_grad_vals(sptrsv_plan p, const void *gb, const void *x, void *gvals)
{
    Range range("sptrsv_batch_grad_vals");
    if (!p || !p->batched) return SPTRSV_EINVAL;
    const int32_t nmat = (int32_t)p->mats.size();
    if (nmat == 0) return SPTRSV_OK;
    if (!gb || !x || !gvals) return SPTRSV_EINVAL;
    cudaError_t e;
    if (p->dtype == SPTRSV_F64)
        e = batch_grad_vals<double>(p->d_mats, p->d_gchunks, p->n_gchunks, (const double *)gb, (const double *)x,
                                    (double *)gvals, p->h->stream);
    else
        e = batch_grad_vals<float>(p->d_mats, p->d_gchunks, p->n_gchunks, (const float *)gb, (const float *)x,
                                   (float *)gvals, p->h->stream);
    return from_cuda(e);
}

extern "C" sptrsv_status sptrsv_batch_tt_apply(sptrsv_plan p, const void *gbp, void *gb)
{
    Range range("sptrsv_batch_tt_apply");
    if (!p || !p->batched) return SPTRSV_EINVAL;
    const int32_t nmat = (int32_t)p->mats.size();
    if (nmat == 0) return SPTRSV_OK;
    if (!gbp || !gb) return SPTRSV_EINVAL;
    cudaError_t e;
    if (p->dtype == SPTRSV_F64)
        e = batch_tt_apply<double>(p->d_mats, p->d_tchunks, p->n_tchunks, p->rhs_off[nmat], (const double *)gbp,
                                   (double *)gb, p->h->stream);
    else
        e = batch_tt_apply<float>(p->d_mats, p->d_tchunks, p->n_tchunks, p->rhs_off[nmat], (const float *)gbp,
                                  (float *)gb, p->h->stream);
    return from_cuda(e);
}

// ------------------------------------------------------ steps from host buffers
namespace {
sptrsv_status ensure_host_sets(sptrsv_plan p)
{
    if (p->s_h2d) return SPTRSV_OK;
    const int32_t nmat = (int32_t)p->mats.size();
    const size_t w = p->dtype == SPTRSV_F64 ? 8 : 4;
    const size_t rhs = w * (size_t)std::max<int64_t>(p->rhs_off[nmat], 1);
    const size_t nz = w * (size_t)std::max<int64_t>(p->vals_off[nmat], 1);
    cudaError_t e = cudaSuccess;
    for (auto &S : p->hset) {
        for (void **q : {&S.b, &S.w, &S.x, &S.gbp, &S.gb})
            if (e == cudaSuccess) e = p->alloc(q, rhs);
        if (e == cudaSuccess) e = p->alloc(&S.gv, nz);
        for (cudaEvent_t *ev : {&S.h2d, &S.comp, &S.d2h})
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->s_h2d, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->s_d2h, cudaStreamNonBlocking);
    return from_cuda(e);
}
}  // namespace

extern "C" sptrsv_status sptrsv_batch_step_host(sptrsv_plan p, const void *b, const void *w, void *x, void *gb,
                                                void *gvals)
{
    Range range("sptrsv_batch_step_host");
    if (!p || !p->batched || !b || !w || !x || !gb || !gvals) return SPTRSV_EINVAL;
    if (!p->have_csc) return SPTRSV_ENOTSUP;
    const int32_t nmat = (int32_t)p->mats.size();
    if (nmat == 0 || p->rhs_off[nmat] == 0) return SPTRSV_OK;
    sptrsv_status st = ensure_host_sets(p);
    if (st != SPTRSV_OK) return st;
    const size_t wb = p->dtype == SPTRSV_F64 ? 8 : 4;
    const size_t rhs = wb * (size_t)p->rhs_off[nmat];
    const size_t nz = wb * (size_t)p->vals_off[nmat];
    sptrsv_plan_st::HostSet &S = p->hset[p->nsteps & 1];
    cudaStream_t hs = p->h->stream;
    // copies in, once the previous step on this set no longer reads b and w
    cudaError_t e = S.used ? cudaStreamWaitEvent(p->s_h2d, S.comp, 0) : cudaSuccess;
    if (e == cudaSuccess) e = cudaMemcpyAsync(S.b, b, rhs, cudaMemcpyHostToDevice, p->s_h2d);
    if (e == cudaSuccess) e = cudaMemcpyAsync(S.w, w, rhs, cudaMemcpyHostToDevice, p->s_h2d);
    if (e == cudaSuccess) e = cudaEventRecord(S.h2d, p->s_h2d);
    // the step, once its inputs are in and the previous results of the set are out
    if (e == cudaSuccess) e = cudaStreamWaitEvent(hs, S.h2d, 0);
    if (e == cudaSuccess && S.used) e = cudaStreamWaitEvent(hs, S.d2h, 0);
    if (e != cudaSuccess) return from_cuda(e);
    st = sptrsv_batch_solve(p, S.b, S.x);
    if (st == SPTRSV_OK) st = sptrsv_batch_solve_transpose(p, S.w, S.gbp);
    if (st == SPTRSV_OK) st = sptrsv_batch_tt_apply(p, S.gbp, S.gb);
    if (st == SPTRSV_OK) st = sptrsv_batch_grad_vals(p, S.gbp, S.x, S.gv);
    if (st != SPTRSV_OK) return st;
    e = cudaEventRecord(S.comp, hs);
    // copies out
    if (e == cudaSuccess) e = cudaStreamWaitEvent(p->s_d2h, S.comp, 0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(x, S.x, rhs, cudaMemcpyDeviceToHost, p->s_d2h);
    if (e == cudaSuccess) e = cudaMemcpyAsync(gb, S.gb, rhs, cudaMemcpyDeviceToHost, p->s_d2h);
    if (e == cudaSuccess) e = cudaMemcpyAsync(gvals, S.gv, nz, cudaMemcpyDeviceToHost, p->s_d2h);
    if (e == cudaSuccess) e = cudaEventRecord(S.d2h, p->s_d2h);
    S.used = true;
    ++p->nsteps;
    return from_cuda(e);
}

extern "C" sptrsv_status sptrsv_batch_step_wait(sptrsv_plan p)
{
    Range range("sptrsv_batch_step_wait");
    if (!p || !p->batched) return SPTRSV_EINVAL;
    cudaError_t e = cudaStreamSynchronize(p->h->stream);
    if (e == cudaSuccess && p->s_h2d) e = cudaStreamSynchronize(p->s_h2d);
    if (e == cudaSuccess && p->s_d2h) e = cudaStreamSynchronize(p->s_d2h);
    if (e != cudaSuccess) return from_cuda(e);
    int status = 0;
    e = cudaMemcpy(&status, p->h->d_status, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return from_cuda(e);
    return (sptrsv_status)status;
}

// ------------------------------------------------------------ bounds checks
namespace {
__global__ void k_debug_check_index(int32_t index, int32_t n, int *status, int *out)
{
    const int v = chk_index(index, 0, n, status);
    if (v >= 0 && v < n) out[0] = v;  // the access a checked index feeds
}
}  // namespace

extern "C" int32_t sptrsv_checked_build(void)
{
#ifdef SPTRSV_CHECKED
    return 1;
#else
    return 0;
#endif
}

extern "C" sptrsv_status sptrsv_debug_check_index(sptrsv_handle h, int32_t index, int32_t n)
{
    if (!h || n < 1 || n > 32) return SPTRSV_EINVAL;
    k_debug_check_index<<<1, 1, 0, h->stream>>>(index, n, h->d_status, reinterpret_cast<int *>(h->d_scratch));
    return from_cuda(cudaGetLastError());
}
