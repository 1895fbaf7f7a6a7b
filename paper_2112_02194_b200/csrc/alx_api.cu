// C ABI of the library (declared in include/alx.h): context, argument checks, device memory,
// and the order in which the kernels of one half-epoch are launched.  No arithmetic of the method
// happens on the host.
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "../../include/alx.h"
#include "alx_common.cuh"
#include <nvtx3/nvToolsExt.h>      // header-only: ranges show up in a profiler's timeline, and cost nothing without one

using namespace alx;

// Device memory that a context keeps from call to call (grown as needed, given back when it is large, freed with the context)
enum Kept { kKeptRows, kKeptOrder, kKeptScratch, kKeptSums, kKeptTable, kKeptFallback, kKeptOut, kKeptUpload, kKeptWork, kKeptCount };
constexpr size_t kKeepMost = 256ull << 20;
// Page-locked staging of small transfers: the status word and small results come back together behind one wait, the arrays of
// a small call go up in one copy
constexpr size_t kBoxBytes = 64 << 10, kBoxSmall = 1 << 10;

struct alx_ctx {
    alx_options opt{};
    int device = 0;
    cudaStream_t stream = nullptr;
    int bf16 = 0;
    size_t elem = 4;
    int64_t n[2] = {0, 0};         // n[ALX_ROWS] = n_rows, n[ALX_COLS] = n_cols
    int64_t nnz = -1;
    int64_t split = ALX_DEFAULT_SPLIT;
    bool has_values = false;
    bool have_table[2] = {false, false};
    bool have_gram[2] = {false, false};

    // per orientation: [ALX_ROWS] = CSR (rows of the matrix), [ALX_COLS] = CSC
    int64_t *ptr[2] = {nullptr, nullptr};
    int32_t *idx[2] = {nullptr, nullptr};
    float *val[2] = {nullptr, nullptr};
    int32_t *order[2] = {nullptr, nullptr};
    int64_t *class_offs_dev[2] = {nullptr, nullptr};
    int64_t class_offs[2][ALX_N_CLASSES + 1] = {};
    int64_t *chunk_desc[2] = {nullptr, nullptr};
    int64_t *split_first[2] = {nullptr, nullptr};
    int64_t n_chunks[2] = {0, 0};
    int64_t n_split_rows[2] = {0, 0};
    // tensor path with the dual form: the rows of 1 .. 16 entries once more per orientation, those with at most 8 entries first
    int32_t *order16[2] = {nullptr, nullptr};
    int64_t n4[2] = {0, 0}, n8[2] = {0, 0};      // ... and those with at most 4 before them

    void *table[2] = {nullptr, nullptr};
    void *parts = nullptr;        // fp32 tables of 64 features: bfloat16 parts of the fixed table, [larger side][3][64], rewritten every half-epoch
    double *G64[2] = {nullptr, nullptr};   // Gramian of table [side]
    float *Bmat = nullptr;
    float *gram_partials = nullptr;
    float *split_partials = nullptr;
    void *dual_ws = nullptr;      // tensor path: B^-1 operand tiles and the flag of the dual form
    int64_t dual_candidates = 0;  // rows of classes 1 and 2 of the last half-epoch (solved in the dual form if the flag is set)
    int64_t dual_candidates32 = 0; // of them, the rows of 17 .. 32 observations (which the whole-rows kernel may have taken instead)
    // The launches of a whole epoch on this matrix, for small matrices: captured behind the second alx_epoch, replayed from the third on
    cudaGraphExec_t epoch_graph = nullptr;
    int epochs_run = 0;            // alx_epoch calls since the matrix was set
    int64_t epoch_launches = 0;    // kernels in the graph
    bool capturing = false;
    bool by_stamps = false;        // the last half-epoch's times are in `stamps`, not in the events
    unsigned long long *stamps = nullptr;          // device, [kStampSlots]
    int last_side = 0;             // side of the last half-epoch: its flag and policy record stay on the device until alx_get_stats asks
    double *loss_partials_buf = nullptr;
    unsigned *loss_counter = nullptr;              // zero between calls
    DevStatus *status = nullptr;
    unsigned long long *cg_counters = nullptr;   // tensor path, last half-epoch: rows solved by conjugate gradients, products, fall-backs; dual-form rows polished, their products
    int32_t *cg_fallback_list = nullptr;         // tensor path with conjugate gradients: the rows left to the Cholesky solve
    CgPolicy *cg_policy = nullptr;               // [2]: per side, what the solver choice of its next half-epoch rests on

    // second stream for the host copies that alx_load_host / alx_epoch_to_host overlap with kernels
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t copy_ev = nullptr;
    const void *upload_after_csr[2] = {nullptr, nullptr};   // alx_load_host: tables to upload behind the upload of S

    unsigned char *box = nullptr;                  // kBoxBytes, page-locked: DevStatus, then small results, payload from kBoxSmall on
    struct { void *p; size_t bytes; } kept[kKeptCount] = {};
    alx_ctx *fold = nullptr;                       // alx_fold_in's context for the new rows, made at the first call
    std::mutex calls;                              // alx_fold_in, alx_topk and alx_recall_at_k, which use what is kept

    cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    bool main_timed = false;
    alx_stats stats{};
    int64_t launches = 0;
    int64_t bytes_held = 0;
    std::vector<std::pair<void *, size_t>> owned;
    std::string err;
};

namespace {

alx_status fail(alx_ctx *c, alx_status code, const char *fmt, ...)
{
    if (c) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        c->err = buf;
    }
    return code;
}

#define ALX_CUDA(c, expr)                                                                          \
    do {                                                                                           \
        cudaError_t e_ = (expr);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return fail((c), e_ == cudaErrorMemoryAllocation ? ALX_ERR_OOM : ALX_ERR_CUDA,         \
                        "%s failed: %s", #expr, cudaGetErrorString(e_));                           \
    } while (0)

// a named range on the profiler's timeline for as long as the object lives
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) { cudaGetDevice(&prev); if (prev != dev) cudaSetDevice(dev); else prev = -1; }
    ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

void *dev_alloc(alx_ctx *c, size_t bytes)
{
    if (bytes == 0) bytes = 256;
    void *p = nullptr;
    if (c->opt.alloc) {
        p = c->opt.alloc(bytes, c->opt.alloc_user);
    } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
    }
    if (p) {
        c->owned.emplace_back(p, bytes);
        c->bytes_held += (int64_t)bytes;
    }
    return p;
}

void dev_free(alx_ctx *c, void *p)
{
    if (!p) return;
    for (size_t k = 0; k < c->owned.size(); ++k)
        if (c->owned[k].first == p) {
            c->bytes_held -= (int64_t)c->owned[k].second;
            c->owned.erase(c->owned.begin() + k);
            break;
        }
    if (c->opt.free) c->opt.free(p, c->opt.alloc_user); else cudaFree(p);
}

template <typename T> bool alloc_into(alx_ctx *c, T *&dst, size_t count)
{
    dst = static_cast<T *>(dev_alloc(c, count * sizeof(T)));
    return dst != nullptr;
}

#define ALX_ALLOC(c, dst, count)                                                                   \
    do {                                                                                           \
        if (!alloc_into((c), (dst), (size_t)(count)))                                              \
            return fail((c), ALX_ERR_OOM, "device allocation of %zu bytes failed",                 \
                        (size_t)(count) * sizeof(*(dst)));                                         \
    } while (0)

// Temporaries of one call: whatever is still registered when the call returns, on any path, goes back to the allocator
// (after the stream has drained, since kernels in flight may still use it).
struct Scratch {
    alx_ctx *c;
    std::vector<void *> held;
    explicit Scratch(alx_ctx *ctx) : c(ctx) {}
    Scratch(const Scratch &) = delete;
    Scratch &operator=(const Scratch &) = delete;
    template <typename T> T *keep(T *p) { if (p) held.push_back(p); return p; }
    void release(void *p)
    {
        for (size_t k = 0; k < held.size(); ++k)
            if (held[k] == p) { held.erase(held.begin() + k); dev_free(c, p); return; }
    }
    ~Scratch()
    {
        if (held.empty()) return;
        cudaStreamSynchronize(c->stream);
        for (void *p : held) dev_free(c, p);
    }
};

#define ALX_TMP(c, scratch, dst, count)                                                            \
    do {                                                                                           \
        ALX_ALLOC(c, dst, count);                                                                  \
        (scratch).keep(dst);                                                                       \
    } while (0)

alx_status ensure_box(alx_ctx *c)
{
    if (!c->box) ALX_CUDA(c, cudaHostAlloc(reinterpret_cast<void **>(&c->box), kBoxBytes, cudaHostAllocDefault));
    return ALX_OK;
}

// device memory of a slot, at least `bytes`; its old contents are gone when it had to grow.  The calls that use the slots wait
// for the stream before they return, so nothing in flight uses an old one.
alx_status keep(alx_ctx *c, Kept slot, size_t bytes, void **out)
{
    auto &k = c->kept[slot];
    if (k.bytes < bytes) {
        dev_free(c, k.p);
        k.p = nullptr;
        k.bytes = 0;
        const size_t want = bytes > kKeepMost ? bytes : bytes + bytes / 4;
        k.p = dev_alloc(c, want);
        if (!k.p) return fail(c, ALX_ERR_OOM, "device allocation of %zu bytes failed", want);
        k.bytes = want;
    }
    *out = k.p;
    return ALX_OK;
}
void give_back_large(alx_ctx *c)
{
    for (auto &k : c->kept)
        if (k.bytes > kKeepMost) { dev_free(c, k.p); k.p = nullptr; k.bytes = 0; }
}
constexpr size_t aligned(size_t bytes) { return (bytes + 255) / 256 * 256; }

// A host call's arrays, laid out one behind the other in a slot of device memory; small ones go up in one copy through the box.
struct Upload {
    alx_ctx *c;
    struct { const void *src; size_t bytes, at; } part[4];
    int n = 0;
    size_t total = 0;
    explicit Upload(alx_ctx *ctx) : c(ctx) {}
    int add(const void *src, size_t bytes)      // number of the part
    {
        part[n] = {src, bytes, total};
        total += aligned(bytes > 0 ? bytes : 1);
        return n++;
    }
    alx_status send(Kept slot, void *(&dev)[4])
    {
        void *base = nullptr;
        alx_status st = keep(c, slot, total, &base);
        if (st != ALX_OK) return st;
        for (int k = 0; k < n; ++k) dev[k] = static_cast<unsigned char *>(base) + part[k].at;
        if (total <= kBoxBytes - kBoxSmall) {
            if ((st = ensure_box(c)) != ALX_OK) return st;
            for (int k = 0; k < n; ++k)
                if (part[k].bytes) memcpy(c->box + kBoxSmall + part[k].at, part[k].src, part[k].bytes);
            ALX_CUDA(c, cudaMemcpyAsync(base, c->box + kBoxSmall, total, cudaMemcpyHostToDevice, c->stream));
        } else {
            for (int k = 0; k < n; ++k)
                if (part[k].bytes) ALX_CUDA(c, cudaMemcpyAsync(dev[k], part[k].src, part[k].bytes, cudaMemcpyHostToDevice, c->stream));
        }
        return ALX_OK;
    }
};

// Results on their way back to the host with the status word: small ones through the box (`take` hands them out after the wait).
// The box's payload is free by then: the upload that used it has been read.
struct Download {
    alx_ctx *c;
    struct { void *dst; size_t bytes, at; } part[4];
    int n = 0;
    size_t used = kBoxSmall;
    explicit Download(alx_ctx *ctx) : c(ctx) {}
    alx_status add(void *dst, const void *dev, size_t bytes)
    {
        alx_status st = ensure_box(c);
        if (st != ALX_OK) return st;
        if (used + aligned(bytes) <= kBoxBytes) {
            part[n++] = {dst, bytes, used};
            ALX_CUDA(c, cudaMemcpyAsync(c->box + used, dev, bytes, cudaMemcpyDeviceToHost, c->stream));
            used += aligned(bytes);
        } else {
            ALX_CUDA(c, cudaMemcpyAsync(dst, dev, bytes, cudaMemcpyDeviceToHost, c->stream));
        }
        return ALX_OK;
    }
    void take()
    {
        for (int k = 0; k < n; ++k) memcpy(part[k].dst, c->box + part[k].at, part[k].bytes);
    }
};

// the status word that a copy or a kernel has put into the box and the stream has been waited for: report and clear it
alx_status report_status(alx_ctx *c)
{
    DevStatus h;
    memcpy(&h, c->box, sizeof h);
    c->stats.not_spd += (int64_t)h.not_spd;
    if (h.flags == 0) return ALX_OK;
    ALX_CUDA(c, cudaMemsetAsync(c->status, 0, sizeof(DevStatus), c->stream));
    if (h.flags & kFlagBadRowptr) return fail(c, ALX_ERR_BAD_CSR, "rowptr is not a monotone offset array (near row %lld)", h.first_bad);
    if (h.flags & kFlagBadCol) return fail(c, ALX_ERR_BAD_CSR, "column index out of range at entry %lld", h.first_bad);
    if (h.flags & kFlagUnsorted) return fail(c, ALX_ERR_BAD_CSR, "column indices not strictly ascending inside a row at entry %lld", h.first_bad);
    // a wait that ran out leaves rows unsolved, which matters more than rows set to zero: report it first
    if (h.flags & kFlagTimeout)
        return fail(c, ALX_ERR_CUDA, "a bounded wait inside a kernel ran out (wait site %lld, block %lld)%s", h.first_bad / 1000000,
                    h.first_bad % 1000000, (h.flags & kFlagNotSpd) ? "; rows also met non-positive pivots" : "");
    if (h.flags & kFlagNotSpd) return fail(c, ALX_ERR_NOT_SPD, "%llu rows met a non-positive pivot (first: row %lld); they were set to zero", h.not_spd, h.first_bad);
    return fail(c, ALX_ERR_CUDA, "device status flags 0x%x", h.flags);
}

// wait for the stream, read and clear the device status word
alx_status check_device_status(alx_ctx *c)
{
    alx_status st = ensure_box(c);
    if (st != ALX_OK) return st;
    ALX_CUDA(c, cudaMemcpyAsync(c->box, c->status, sizeof(DevStatus), cudaMemcpyDeviceToHost, c->stream));
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    return report_status(c);
}

SideView side_view(const alx_ctx *c, int side)
{
    SideView v;
    v.ptr = c->ptr[side];
    v.idx = c->idx[side];
    v.val = c->val[side];
    v.order = c->order[side];
    v.chunk_desc = c->chunk_desc[side];
    v.split_first = c->split_first[side];
    v.n = c->n[side];
    v.nnz = c->nnz;
    return v;
}

// chunk descriptors of the rows longer than `split` of one orientation, from its class offsets
alx_status build_chunks(alx_ctx *c, int side, int64_t *scan_scratch, int64_t scan_elems)
{
    const int64_t *offs = c->class_offs[side];
    const int64_t n_split = offs[ALX_N_CLASSES] - offs[ALX_N_CLASSES - 1];
    c->n_split_rows[side] = n_split;
    c->n_chunks[side] = 0;
    if (n_split > 0) {
        Scratch tmp(c);
        int64_t *counts = nullptr;
        ALX_TMP(c, tmp, counts, n_split);
        ALX_ALLOC(c, c->split_first[side], n_split + 1);
        const int32_t *split_rows = c->order[side] + offs[ALX_N_CLASSES - 1];
        ALX_CUDA(c, launch_chunk_counts(c->ptr[side], split_rows, n_split, c->split, counts, c->stream, &c->launches));
        ALX_CUDA(c, scan_exclusive(counts, true, c->split_first[side], n_split, scan_scratch, scan_elems, c->stream,
                                   &c->launches));
        int64_t total = 0;
        ALX_CUDA(c, cudaMemcpyAsync(&total, c->split_first[side] + n_split, sizeof total, cudaMemcpyDeviceToHost, c->stream));
        ALX_CUDA(c, cudaStreamSynchronize(c->stream));
        c->n_chunks[side] = total;
        ALX_ALLOC(c, c->chunk_desc[side], 4 * total);
        ALX_CUDA(c, launch_chunk_fill(c->ptr[side], split_rows, n_split, c->split, c->split_first[side],
                                      c->chunk_desc[side], c->stream, &c->launches));
        ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    return ALX_OK;
}

// degree classes, order and chunk descriptors of one orientation
alx_status build_buckets(alx_ctx *c, int side, int64_t *scratch_a, int64_t *scratch_b, int64_t *scan_scratch,
                         int64_t scan_elems)
{
    const int64_t n = c->n[side];
    ALX_CUDA(c, launch_bucket(c->ptr[side], n, c->split, scratch_a, scratch_b, scan_scratch, scan_elems,
                              c->order[side], c->class_offs_dev[side], c->stream, &c->launches));
    ALX_CUDA(c, cudaMemcpyAsync(c->class_offs[side], c->class_offs_dev[side], sizeof(int64_t) * (ALX_N_CLASSES + 1),
                                cudaMemcpyDeviceToHost, c->stream));
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    alx_status st = build_chunks(c, side, scan_scratch, scan_elems);
    if (st != ALX_OK) return st;
    const int64_t *offs = c->class_offs[side];
    for (int k = 0; k < ALX_N_CLASSES; ++k) c->stats.rows_in_class[side][k] = offs[k + 1] - offs[k];
    c->stats.n_chunks[side] = c->n_chunks[side];
    return ALX_OK;
}

void drop_epoch_graph(alx_ctx *c)
{
    if (c->epoch_graph) cudaGraphExecDestroy(c->epoch_graph);
    c->epoch_graph = nullptr;
    c->epochs_run = 0;
}

void release_matrix(alx_ctx *c)
{
    drop_epoch_graph(c);
    for (int s = 0; s < 2; ++s) {
        dev_free(c, c->ptr[s]); c->ptr[s] = nullptr;
        dev_free(c, c->idx[s]); c->idx[s] = nullptr;
        dev_free(c, c->val[s]); c->val[s] = nullptr;
        dev_free(c, c->order[s]); c->order[s] = nullptr;
        dev_free(c, c->chunk_desc[s]); c->chunk_desc[s] = nullptr;
        dev_free(c, c->split_first[s]); c->split_first[s] = nullptr;
    }
    for (int s = 0; s < 2; ++s) { dev_free(c, c->order16[s]); c->order16[s] = nullptr; c->n4[s] = c->n8[s] = 0; }
    dev_free(c, c->split_partials); c->split_partials = nullptr;
    dev_free(c, c->loss_partials_buf); c->loss_partials_buf = nullptr;
    c->nnz = -1;
}

bool tensor_path(const alx_ctx *c) { return c->bf16 && c->opt.d == 128 && c->opt.kernels != 1; }
// d <= 64: a warp per row (alx_rows_warp.cu)
bool warp_path(const alx_ctx *c) { return c->opt.d <= 64 && c->opt.kernels != 1; }
// fp32 tables of 128 features: four warps per row (alx_rows_team.cu)
bool team_path(const alx_ctx *c) { return c->opt.d == 128 && !c->bf16 && c->opt.kernels != 1; }
// of the warp path, fp32 tables of 64 features: conjugate gradients
bool cg64(const alx_ctx *c) { return warp_path(c) && !c->bf16 && c->opt.d == 64; }
// rows of at most 16 observations in the dual form, by a warp each: on the FP32 ALUs (alx_dual64.cu) or by mma (alx_dual_warp.cu)
bool dual64(const alx_ctx *c) { return cg64(c) && c->opt.kernels == 0; }
bool dual_warp(const alx_ctx *c) { return c->opt.kernels == 0 && (team_path(c) || (warp_path(c) && c->bf16 && c->opt.d == 64)); }
// Fewer rows than this are not worth the inverse of the base matrix that the dual form starts with (25 us and more, against
// a few ns per row): they take the d x d solve with the others
constexpr int64_t kDualLeastRows = 256;
bool dual_form(const alx_ctx *c) { return tensor_path(c) && c->opt.kernels == 0; }
const int *dual_flag_of(const alx_ctx *c)
{
    return dual_form(c) ? dual_flag_ptr(c->dual_ws) : dual64(c) ? dual64_flag_ptr(c->dual_ws) : dual_warp_flag_ptr(c->dual_ws, c->opt.d);
}
float dual_cond_limit(const alx_ctx *c) { return c->opt.dual_cond_limit > 0.f ? c->opt.dual_cond_limit : ALX_DEFAULT_DUAL_COND_LIMIT; }
CgOptions cg_options(const alx_ctx *c, int solved_side)
{
    CgOptions o;
    // the start vector of a row is its stored embedding once that table holds something (set by the caller or solved)
    o.warm_start = c->opt.cg_start == ALX_CG_START_STORED && c->have_table[solved_side];
    o.enabled = c->opt.solver == ALX_SOLVER_AUTO;
    o.max_iter = c->opt.cg_max_iter > 0 ? c->opt.cg_max_iter : ALX_DEFAULT_CG_MAX_ITER;
    o.tol = c->opt.cg_tol > 0.f ? c->opt.cg_tol : (c->bf16 ? ALX_DEFAULT_CG_TOL_BF16 : ALX_DEFAULT_CG_TOL);
    o.counters = c->cg_counters;
    o.fallback_list = c->cg_fallback_list;
    o.policy = c->cg_policy ? c->cg_policy + solved_side : nullptr;
    o.switch_products = c->opt.cg_switch_products > 0.f ? c->opt.cg_switch_products : ALX_DEFAULT_CG_SWITCH_PRODUCTS;
    return o;
}

// floats of workspace that the sums of a side's chunks and long rows need
int64_t sums_floats(const alx_ctx *c, int side)
{
    const int64_t *offs = c->class_offs[side];
    const int64_t d = c->opt.d;
    if (team_path(c)) return team_sums_floats(offs, c->n_chunks[side]);
    const int64_t n_long = tensor_path(c) ? offs[kNClasses - 1] - offs[long_class_begin(offs)]
                           : cg64(c)      ? offs[kNClasses - 1] - offs[parts64_long_class(offs)] : 0;
    return (c->n_chunks[side] + n_long) * (d * d + d);
}

// rows of a side that the dual form is offered (class 1, and class 2 for d = 128); 0: none, or too few
int64_t dual_rows_of(const alx_ctx *c, int side)
{
    const int64_t *offs = c->class_offs[side];
    const int64_t n = dual_form(c) ? offs[3] - offs[1] : dual_warp(c) || dual64(c) ? offs[2] - offs[1] : 0;
    return n >= kDualLeastRows ? n : 0;
}

// the Gramian and the base matrix of a table; `solve`: also what the rows' dual form needs of the base matrix
alx_status gramian_of(alx_ctx *c, int table_side, bool solve, unsigned long long *stamps = nullptr, cudaStream_t aside = nullptr)
{
    const cudaStream_t s = aside ? aside : c->stream;
    if (tensor_path(c)) {
        ALX_CUDA(c, launch_gramian_umma(c->table[table_side], c->n[table_side], c->gram_partials, s, &c->launches));
        ALX_CUDA(c, launch_gramian_reduce(c->gram_partials, gramian_umma_partials(), c->opt.d, c->G64[table_side], c->Bmat,
                                          c->opt.alpha0, c->opt.lambda, s, &c->launches));
        if (solve && dual_form(c)) ALX_CUDA(c, launch_dual_prepare(c->Bmat, c->dual_ws, dual_cond_limit(c), c->opt.solver == ALX_SOLVER_AUTO, s,
                                                         &c->launches));
        c->have_gram[table_side] = true;
        return ALX_OK;
    }
    ALX_CUDA(c, launch_gramian(c->table[table_side], c->bf16, c->n[table_side], c->opt.d, c->gram_partials,
                               c->G64[table_side], c->Bmat, c->opt.alpha0, c->opt.lambda, stamps, s, &c->launches));
    if (solve && dual64(c)) ALX_CUDA(c, launch_dual64_prepare(c->Bmat, c->dual_ws, dual_cond_limit(c), s, &c->launches));
    if (solve && dual_warp(c)) {
        const float most = c->bf16 ? kDualWarpLimitBf16 : kDualWarpLimitF32;
        ALX_CUDA(c, launch_dual_warp_prepare(c->Bmat, c->dual_ws, c->opt.d, dual_cond_limit(c) < most ? dual_cond_limit(c) : most, s,
                                             &c->launches));
    }
    c->have_gram[table_side] = true;
    return ALX_OK;
}

// what the statistics say of a half-epoch
void note_half_epoch(alx_ctx *c, int side)
{
    c->last_side = side;
    c->dual_candidates = dual_rows_of(c, side);
    c->dual_candidates32 = dual_form(c) && c->dual_candidates > 0 ? c->class_offs[side][3] - c->class_offs[side][2] : 0;
    c->main_timed = tensor_path(c) || cg64(c);
    c->stats.kernel_path[side] = warp_path(c) || tensor_path(c) || team_path(c) ? 1 : 0;
}

// gramian_aside: the Gramian was launched on the second stream, copy_ev follows it
alx_status half_epoch_impl(alx_ctx *c, int side, const int32_t *cap_slot, float *cap_out, bool gramian_aside = false)
{
    if (c->nnz < 0) return fail(c, ALX_ERR_BAD_STATE, "alx_half_epoch before alx_set_csr");
    const int fixed = 1 - side;
    if (!c->have_table[fixed]) return fail(c, ALX_ERR_BAD_STATE, "the fixed table has not been set");
    NvtxRange range(side == ALX_ROWS ? "alx half-epoch: rows" : "alx half-epoch: columns");
    // (the launches of the d <= 64 kernels without conjugate gradients are the ones short enough to mind events in a graph)
    unsigned long long *stamps = c->capturing && warp_path(c) && !cg64(c) ? c->stamps : nullptr;
    if (!stamps) ALX_CUDA(c, record_event(c->ev[0], c->stream, c->capturing));
    alx_status st;
    {
        NvtxRange r("alx Gramian + base matrix");
        if (gramian_aside) ALX_CUDA(c, cudaStreamWaitEvent(c->stream, c->copy_ev, 0));
        else if ((st = gramian_of(c, fixed, dual_rows_of(c, side) > 0, stamps)) != ALX_OK) return st;
    }
    if (!stamps) ALX_CUDA(c, record_event(c->ev[1], c->stream, c->capturing));
    NvtxRange rows_range("alx rows: gather, sums, solve, store");
    RowOut out{c->table[side], cap_slot, cap_out};
    note_half_epoch(c, side);
    const int64_t n_dual = c->dual_candidates;
    if (warp_path(c)) {
        if (cg64(c)) ALX_CUDA(c, cudaMemsetAsync(c->cg_counters, 0, 5 * sizeof(unsigned long long), c->stream));
        if (n_dual > 0)
            ALX_CUDA(c, dual64(c) ? launch_rows_dual64(side_view(c, side), c->class_offs[side][1], n_dual, c->table[fixed], c->dual_ws, out,
                                                       c->stream, &c->launches)
                                  : launch_rows_dual_warp(side_view(c, side), c->class_offs[side][1], n_dual, c->table[fixed], c->bf16,
                                                          c->opt.d, c->dual_ws, out, c->status, c->stream, &c->launches));
        if (cg64(c)) ALX_CUDA(c, record_event(c->ev[3], c->stream, c->capturing));
        ALX_CUDA(c, launch_rows_warp(side_view(c, side), c->class_offs[side], c->n_chunks[side], c->n_split_rows[side], c->table[fixed],
                                     c->n[fixed], c->parts, c->bf16, c->opt.d, c->Bmat, c->split_partials, out, c->status, cg_options(c, side),
                                     n_dual > 0 ? dual_flag_of(c) : nullptr, stamps, c->stream, &c->launches));
        if (cg64(c)) ALX_CUDA(c, record_event(c->ev[4], c->stream, c->capturing));
    } else if (tensor_path(c)) {
        ALX_CUDA(c, cudaMemsetAsync(c->cg_counters, 0, 5 * sizeof(unsigned long long), c->stream));
        ALX_CUDA(c, launch_rows_umma(side_view(c, side), c->class_offs[side], c->n_chunks[side], c->n_split_rows[side],
                                     c->table[fixed], c->Bmat, c->split_partials, out, c->status, c->stream,
                                     &c->launches, c->ev[3], c->ev[4], c->capturing, n_dual > 0 ? c->dual_ws : nullptr, c->n[fixed],
                                     cg_options(c, side), c->order16[side], c->n4[side], c->n8[side]));
    } else if (team_path(c)) {
        if (n_dual > 0)
            ALX_CUDA(c, launch_rows_dual_warp(side_view(c, side), c->class_offs[side][1], n_dual, c->table[fixed], 0, c->opt.d, c->dual_ws, out,
                                              c->status, c->stream, &c->launches));
        ALX_CUDA(c, launch_rows_team(side_view(c, side), c->class_offs[side], c->n_chunks[side], c->n_split_rows[side],
                                     static_cast<const float *>(c->table[fixed]), c->Bmat, c->split_partials, out, c->status,
                                     n_dual > 0 ? dual_flag_of(c) : nullptr, c->stream, &c->launches));
    } else {
        ALX_CUDA(c, launch_rows_simple(side_view(c, side), c->class_offs[side], c->n_chunks[side], c->n_split_rows[side], c->table[fixed],
                                       c->bf16, c->opt.d, c->Bmat, c->split_partials, out, c->status, c->stream, &c->launches));
    }
    if (!stamps) ALX_CUDA(c, record_event(c->ev[2], c->stream, c->capturing));
    c->by_stamps = false;
    c->have_table[side] = true;
    c->have_gram[side] = false;
    return ALX_OK;
}

}  // namespace

extern "C" {

const char *alx_version(void) { return "alx-b200 0.1 (sm_100a)"; }

const char *alx_last_error(const alx_ctx *ctx) { return ctx ? ctx->err.c_str() : "null context"; }

alx_status alx_create(int64_t n_rows, int64_t n_cols, int32_t d, float lambda, float alpha0, alx_ctx **out)
{
    alx_options o;
    memset(&o, 0, sizeof o);
    o.n_rows = n_rows; o.n_cols = n_cols; o.d = d; o.lambda = lambda; o.alpha0 = alpha0;
    o.storage = ALX_F32; o.device = -1;
    return alx_create_ex(&o, out);   /* solver, cg_max_iter, cg_tol = 0: the defaults */
}

namespace {
alx_status create_impl(const alx_options *opt, const alx_ctx *parent, alx_ctx **out);
}

alx_status alx_create_ex(const alx_options *opt, alx_ctx **out) { return create_impl(opt, nullptr, out); }

namespace {
// parent: the new context borrows the parent's column table (alx_fold_in) and gets its rows' buffers call by call
alx_status create_impl(const alx_options *opt, const alx_ctx *parent, alx_ctx **out)
{
    if (!opt || !out) return ALX_ERR_INVALID_ARG;
    if (opt->n_rows < 1 || opt->n_cols < 1 || opt->n_rows >= (1ll << 31) || opt->n_cols >= (1ll << 31))
        return ALX_ERR_INVALID_ARG;
    if (opt->d != 16 && opt->d != 32 && opt->d != 64 && opt->d != 128) return ALX_ERR_UNSUPPORTED;
    if (!(opt->lambda > 0.f)) return ALX_ERR_UNSUPPORTED;   // lambda = 0: minimiser not unique
    if (!(opt->alpha0 >= 0.f)) return ALX_ERR_INVALID_ARG;
    if (opt->storage != ALX_F32 && opt->storage != ALX_BF16) return ALX_ERR_INVALID_ARG;
    if ((opt->alloc == nullptr) != (opt->free == nullptr)) return ALX_ERR_INVALID_ARG;
    if (opt->split != 0 && opt->split < 16) return ALX_ERR_INVALID_ARG;
    if (opt->solver != ALX_SOLVER_AUTO && opt->solver != ALX_SOLVER_CHOLESKY) return ALX_ERR_INVALID_ARG;
    if (opt->cg_start != ALX_CG_START_STORED && opt->cg_start != ALX_CG_START_ZERO) return ALX_ERR_INVALID_ARG;
    if (!(opt->cg_switch_products >= 0.f) || !(opt->dual_cond_limit >= 0.f)) return ALX_ERR_INVALID_ARG;
    if (opt->cg_max_iter < 0 || opt->cg_max_iter > 1024 || !(opt->cg_tol >= 0.f) || opt->cg_tol > 1e-2f) return ALX_ERR_INVALID_ARG;
    int dev = opt->device;
    if (dev < 0 && cudaGetDevice(&dev) != cudaSuccess) return ALX_ERR_CUDA;
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || dev >= count) return ALX_ERR_CUDA;

    alx_ctx *c = new (std::nothrow) alx_ctx();
    if (!c) return ALX_ERR_OOM;
    c->opt = *opt;
    c->device = dev;
    c->stream = static_cast<cudaStream_t>(opt->stream);
    c->bf16 = opt->storage == ALX_BF16;
    c->elem = c->bf16 ? 2 : 4;
    c->n[ALX_ROWS] = opt->n_rows;
    c->n[ALX_COLS] = opt->n_cols;
    c->split = opt->split ? opt->split : ALX_DEFAULT_SPLIT;
    DeviceGuard guard(dev);
    auto body = [&]() -> alx_status {
        const int d = opt->d;
        for (int s = 0; s < 2; ++s) {
            void *t = parent ? (s == ALX_COLS ? parent->table[s] : nullptr) : dev_alloc(c, (size_t)c->n[s] * d * c->elem);
            if (!t && !(parent && s == ALX_ROWS)) return fail(c, ALX_ERR_OOM, "device allocation of a %lld x %d table failed", (long long)c->n[s], d);
            c->table[s] = t;
            ALX_ALLOC(c, c->G64[s], d * d);
            ALX_ALLOC(c, c->class_offs_dev[s], ALX_N_CLASSES + 1);
        }
        ALX_ALLOC(c, c->Bmat, d * d);
        if (dual_form(c) || dual_warp(c) || dual64(c)) {
            c->dual_ws = dev_alloc(c, dual_form(c) ? dual_workspace_bytes() : dual64(c) ? dual64_workspace_bytes() : dual_warp_workspace_bytes(opt->d));
            if (!c->dual_ws) return fail(c, ALX_ERR_OOM, "device allocation of the dual-form workspace failed");
        }
        const int64_t nmax = c->n[0] > c->n[1] ? c->n[0] : c->n[1];
        if (cg64(c)) {
            c->parts = parent ? parent->parts : dev_alloc(c, (size_t)nmax * 384);
            if (!c->parts) return fail(c, ALX_ERR_OOM, "device allocation of the table of bfloat16 parts failed");
        }
        int64_t n_part = gramian_partials(nmax);
        if (gramian_umma_partials() > n_part) n_part = gramian_umma_partials();
        ALX_ALLOC(c, c->gram_partials, n_part * d * d);
        ALX_ALLOC(c, c->stamps, kStampSlots);
        ALX_CUDA(c, cudaMemsetAsync(c->stamps, 0, kStampSlots * sizeof(unsigned long long), c->stream));
        ALX_ALLOC(c, c->loss_counter, 1);
        ALX_CUDA(c, cudaMemsetAsync(c->loss_counter, 0, sizeof(unsigned), c->stream));
        ALX_ALLOC(c, c->status, 1);
        ALX_CUDA(c, cudaMemsetAsync(c->status, 0, sizeof(DevStatus), c->stream));
        ALX_ALLOC(c, c->cg_counters, 5);
        if ((tensor_path(c) || cg64(c)) && c->opt.solver == ALX_SOLVER_AUTO && !parent) ALX_ALLOC(c, c->cg_fallback_list, nmax);
        if (tensor_path(c) && c->opt.solver == ALX_SOLVER_AUTO) {
            ALX_ALLOC(c, c->cg_policy, 2);
            ALX_CUDA(c, cudaMemsetAsync(c->cg_policy, 0, 2 * sizeof(CgPolicy), c->stream));
        }
        ALX_CUDA(c, cudaMemsetAsync(c->cg_counters, 0, 5 * sizeof(unsigned long long), c->stream));
        for (auto &e : c->ev) ALX_CUDA(c, cudaEventCreate(&e));
        ALX_CUDA(c, cudaStreamSynchronize(c->stream));
        return ALX_OK;
    };
    alx_status st = body();
    if (st != ALX_OK) {
        alx_destroy(c);
        return st;
    }
    *out = c;
    return ALX_OK;
}
}  // namespace

alx_status alx_destroy(alx_ctx *c)
{
    if (!c) return ALX_OK;
    DeviceGuard guard(c->device);
    cudaStreamSynchronize(c->stream);
    if (c->fold) alx_destroy(c->fold);
    drop_epoch_graph(c);
    if (c->box) cudaFreeHost(c->box);
    for (auto &e : c->ev) if (e) cudaEventDestroy(e);
    if (c->copy_stream) { cudaStreamSynchronize(c->copy_stream); cudaStreamDestroy(c->copy_stream); }
    if (c->copy_ev) cudaEventDestroy(c->copy_ev);
    std::vector<std::pair<void *, size_t>> owned = c->owned;
    for (auto &p : owned) dev_free(c, p.first);
    delete c;
    return ALX_OK;
}

alx_status alx_set_csr(alx_ctx *c, const int64_t *rowptr, const int32_t *colidx, const float *values, int64_t nnz,
                       int on_device)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!rowptr || nnz < 0 || (nnz > 0 && !colidx)) return fail(c, ALX_ERR_INVALID_ARG, "null array or negative nnz");
    DeviceGuard guard(c->device);
    NvtxRange range("alx_set_csr: validate, transpose, degree classes");
    release_matrix(c);
    const int64_t n_rows = c->n[ALX_ROWS], n_cols = c->n[ALX_COLS];
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    const size_t nz = (size_t)(nnz > 0 ? nnz : 1);
    c->has_values = values != nullptr;
    ALX_ALLOC(c, c->ptr[0], n_rows + 1);
    ALX_ALLOC(c, c->idx[0], nz);
    ALX_CUDA(c, cudaMemcpyAsync(c->ptr[0], rowptr, sizeof(int64_t) * (n_rows + 1), kind, c->stream));
    if (nnz > 0) ALX_CUDA(c, cudaMemcpyAsync(c->idx[0], colidx, sizeof(int32_t) * nnz, kind, c->stream));
    if (values) {
        ALX_ALLOC(c, c->val[0], nz);
        if (nnz > 0) ALX_CUDA(c, cudaMemcpyAsync(c->val[0], values, sizeof(float) * nnz, kind, c->stream));
    }
    if (c->upload_after_csr[0] || c->upload_after_csr[1]) {
        // alx_load_host: the tables follow S over the bus on the second stream, while the kernels below run
        ALX_CUDA(c, cudaEventRecord(c->copy_ev, c->stream));
        ALX_CUDA(c, cudaStreamWaitEvent(c->copy_stream, c->copy_ev, 0));
        for (int sd = 0; sd < 2; ++sd)
            if (c->upload_after_csr[sd])
                ALX_CUDA(c, cudaMemcpyAsync(c->table[sd], c->upload_after_csr[sd], (size_t)c->n[sd] * c->opt.d * c->elem,
                                            cudaMemcpyHostToDevice, c->copy_stream));
    }
    // validate before anything indexes with these arrays
    ALX_CUDA(c, launch_validate(c->ptr[0], c->idx[0], n_rows, n_cols, nnz, c->status, c->stream, &c->launches));
    alx_status st = check_device_status(c);
    if (st != ALX_OK) { release_matrix(c); return st; }
    c->nnz = nnz;

    // scratch shared by the scans and the bucket passes
    const int64_t nmax = n_rows > n_cols ? n_rows : n_cols;
    const int64_t nb = bucket_blocks(nmax);
    const int64_t scan_elems = scan_scratch_elems(nb * kNClasses > nmax ? nb * kNClasses : nmax) + 16;
    Scratch tmp(c);
    int64_t *scan_scratch = nullptr, *blk_counts = nullptr, *blk_offs = nullptr, *class_entries = nullptr;
    int32_t *counts = nullptr;
    ALX_TMP(c, tmp, scan_scratch, scan_elems);
    ALX_TMP(c, tmp, blk_counts, nb * kNClasses);
    ALX_TMP(c, tmp, blk_offs, nb * kNClasses + 1);
    ALX_TMP(c, tmp, counts, n_cols);
    ALX_TMP(c, tmp, class_entries, 2 * kNClasses);

    // transpose: count, prefix sum, degree classes of the columns, fill, sort each column, labels
    ALX_ALLOC(c, c->ptr[1], n_cols + 1);
    ALX_ALLOC(c, c->idx[1], nz);
    ALX_CUDA(c, cudaMemsetAsync(counts, 0, sizeof(int32_t) * n_cols, c->stream));
    ALX_CUDA(c, launch_count_cols(c->idx[0], nnz, counts, c->stream, &c->launches));
    ALX_CUDA(c, scan_exclusive(counts, false, c->ptr[1], n_cols, scan_scratch, scan_elems, c->stream, &c->launches));
    for (int s = 0; s < 2; ++s) ALX_ALLOC(c, c->order[s], c->n[s]);
    st = build_buckets(c, ALX_COLS, blk_counts, blk_offs, scan_scratch, scan_elems);
    if (st != ALX_OK) return st;
    ALX_CUDA(c, cudaMemsetAsync(counts, 0, sizeof(int32_t) * n_cols, c->stream));
    ALX_CUDA(c, launch_fill_transpose(c->ptr[0], c->idx[0], n_rows, nnz, c->ptr[1], counts, c->idx[1], c->stream,
                                      &c->launches));
    ALX_CUDA(c, launch_sort_segments(c->ptr[1], c->idx[1], c->order[1], c->class_offs[1], c->stream, &c->launches));
    if (values) {
        ALX_ALLOC(c, c->val[1], nz);
        ALX_CUDA(c, launch_values_transpose(c->ptr[0], c->idx[0], c->val[0], c->ptr[1], c->idx[1], n_cols, nnz,
                                            c->val[1], c->stream, &c->launches));
    }
    st = build_buckets(c, ALX_ROWS, blk_counts, blk_offs, scan_scratch, scan_elems);
    if (st != ALX_OK) return st;
    if (dual_form(c)) {
        // the rows of 1 .. 16 entries, ordered by length class (at most 4, 5 .. 8, 9 .. 16): kernel instances with four and
        // eight observations per row take the first two parts at a quarter and half of the cost per row
        for (int s = 0; s < 2; ++s) {
            const int64_t n16 = c->class_offs[s][2] - c->class_offs[s][1];
            if (n16 <= 0) continue;
            const int64_t nb = (n16 + 1023) / 1024;
            int64_t *pc = nullptr, *po = nullptr;
            ALX_TMP(c, tmp, pc, nb + 2);
            ALX_TMP(c, tmp, po, nb + 2);
            ALX_ALLOC(c, c->order16[s], n16);
            ALX_CUDA(c, launch_partition_by_length(c->ptr[s], c->order[s] + c->class_offs[s][1], n16, 4, c->order16[s], pc, po,
                                                   class_entries + s, scan_scratch, scan_elems, c->stream, &c->launches));
            ALX_CUDA(c, cudaMemcpyAsync(&c->n4[s], class_entries + s, sizeof(int64_t), cudaMemcpyDeviceToHost, c->stream));
            ALX_CUDA(c, cudaStreamSynchronize(c->stream));
            const int64_t rest = n16 - c->n4[s];
            c->n8[s] = c->n4[s];
            if (rest > 0) {
                int32_t *part = nullptr;
                ALX_TMP(c, tmp, part, rest);
                ALX_CUDA(c, launch_partition_by_length(c->ptr[s], c->order16[s] + c->n4[s], rest, 8, part, pc, po, class_entries + s,
                                                       scan_scratch, scan_elems, c->stream, &c->launches));
                int64_t n58 = 0;
                ALX_CUDA(c, cudaMemcpyAsync(&n58, class_entries + s, sizeof(int64_t), cudaMemcpyDeviceToHost, c->stream));
                ALX_CUDA(c, cudaMemcpyAsync(c->order16[s] + c->n4[s], part, sizeof(int32_t) * rest, cudaMemcpyDeviceToDevice, c->stream));
                ALX_CUDA(c, cudaStreamSynchronize(c->stream));
                c->n8[s] += n58;
                tmp.release(part);
            }
            tmp.release(pc);
            tmp.release(po);
        }
    }
    for (int s = 0; s < 2; ++s)
        ALX_CUDA(c, launch_class_entries(c->ptr[s], c->order[s], c->class_offs_dev[s], c->n[s], class_entries + s * kNClasses,
                                         c->stream, &c->launches));
    ALX_CUDA(c, cudaMemcpyAsync(c->stats.entries_in_class, class_entries, 2 * kNClasses * sizeof(int64_t),
                                cudaMemcpyDeviceToHost, c->stream));
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    tmp.release(counts);
    tmp.release(blk_offs);
    tmp.release(blk_counts);
    tmp.release(scan_scratch);
    tmp.release(class_entries);

    for (int s = 0; s < 2; ++s) c->stats.long_rows[s] = c->stats.long_entries[s] = 0;
    if (tensor_path(c) || warp_path(c)) {
        int64_t *total = nullptr;
        ALX_TMP(c, tmp, total, 2);
        for (int s = 0; s < 2; ++s) {
            const int64_t *offs = c->class_offs[s];
            const int64_t first = offs[tensor_path(c) ? long_class_begin(offs) : cg64(c) ? parts64_long_class(offs) : warp_long_class(offs)];
            const int64_t n_long = offs[kNClasses - 1] - first;
            c->stats.long_rows[s] = n_long;
            ALX_CUDA(c, launch_sum_row_lengths(c->ptr[s], c->order[s] + first, n_long, total + s, c->stream, &c->launches));
        }
        ALX_CUDA(c, cudaMemcpyAsync(c->stats.long_entries, total, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, c->stream));
        ALX_CUDA(c, cudaStreamSynchronize(c->stream));
        tmp.release(total);
    }
    const int64_t sums = sums_floats(c, 0) > sums_floats(c, 1) ? sums_floats(c, 0) : sums_floats(c, 1);
    if (sums > 0) ALX_ALLOC(c, c->split_partials, sums);
    ALX_ALLOC(c, c->loss_partials_buf, loss_partials(nnz));
    c->stats.nnz = nnz;
    return ALX_OK;
}

alx_status alx_set_embeddings(alx_ctx *c, alx_side side, const void *src, alx_dtype src_dtype, int on_device)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!src || (side != ALX_ROWS && side != ALX_COLS) || (src_dtype != ALX_F32 && src_dtype != ALX_BF16))
        return fail(c, ALX_ERR_INVALID_ARG, "bad argument to alx_set_embeddings");
    DeviceGuard guard(c->device);
    const int64_t count = c->n[side] * c->opt.d;
    const size_t src_bytes = (size_t)count * (src_dtype == ALX_BF16 ? 2 : 4);
    const void *dev_src = src;
    Scratch tmp(c);
    void *staging = nullptr;
    if (!on_device) {
        if ((src_dtype == ALX_BF16) == (c->bf16 != 0)) {
            ALX_CUDA(c, cudaMemcpyAsync(c->table[side], src, src_bytes, cudaMemcpyHostToDevice, c->stream));
            ALX_CUDA(c, cudaStreamSynchronize(c->stream));
            c->have_table[side] = true;
            c->have_gram[side] = false;
            return ALX_OK;
        }
        staging = tmp.keep(dev_alloc(c, src_bytes));
        if (!staging) return fail(c, ALX_ERR_OOM, "staging allocation failed");
        ALX_CUDA(c, cudaMemcpyAsync(staging, src, src_bytes, cudaMemcpyHostToDevice, c->stream));
        dev_src = staging;
    }
    ALX_CUDA(c, launch_convert(dev_src, src_dtype == ALX_BF16, c->table[side], c->bf16, count, c->stream, &c->launches));
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    c->have_table[side] = true;
    c->have_gram[side] = false;
    return ALX_OK;
}

alx_status alx_set_embedding_rows(alx_ctx *c, alx_side side, int64_t row_begin, int64_t row_count, const void *src,
                                  alx_dtype src_dtype, int on_device)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!src || (side != ALX_ROWS && side != ALX_COLS) || (src_dtype != ALX_F32 && src_dtype != ALX_BF16) ||
        row_begin < 0 || row_count < 0 || row_begin + row_count > c->n[side])
        return fail(c, ALX_ERR_INVALID_ARG, "bad argument to alx_set_embedding_rows");
    if (row_count == 0) return ALX_OK;
    DeviceGuard guard(c->device);
    const int64_t count = row_count * c->opt.d;
    const size_t src_bytes = (size_t)count * (src_dtype == ALX_BF16 ? 2 : 4);
    char *dst = static_cast<char *>(c->table[side]) + (size_t)row_begin * c->opt.d * c->elem;
    const void *dev_src = src;
    Scratch tmp(c);
    void *staging = nullptr;
    const bool same = (src_dtype == ALX_BF16) == (c->bf16 != 0);
    if (same) {
        ALX_CUDA(c, cudaMemcpyAsync(dst, src, src_bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, c->stream));
    } else {
        if (!on_device) {
            staging = tmp.keep(dev_alloc(c, src_bytes));
            if (!staging) return fail(c, ALX_ERR_OOM, "staging allocation failed");
            ALX_CUDA(c, cudaMemcpyAsync(staging, src, src_bytes, cudaMemcpyHostToDevice, c->stream));
            dev_src = staging;
        }
        ALX_CUDA(c, launch_convert(dev_src, src_dtype == ALX_BF16, dst, c->bf16, count, c->stream, &c->launches));
    }
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    c->have_table[side] = true;
    c->have_gram[side] = false;
    return ALX_OK;
}

alx_status alx_get_embeddings(alx_ctx *c, alx_side side, void *dst, alx_dtype dst_dtype, int64_t row_begin,
                              int64_t row_count, int on_device)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!dst || (side != ALX_ROWS && side != ALX_COLS) || (dst_dtype != ALX_F32 && dst_dtype != ALX_BF16) ||
        row_begin < 0 || row_count < 0 || row_begin + row_count > c->n[side])
        return fail(c, ALX_ERR_INVALID_ARG, "bad argument to alx_get_embeddings");
    if (!c->have_table[side]) return fail(c, ALX_ERR_BAD_STATE, "table has not been set or solved yet");
    DeviceGuard guard(c->device);
    const int d = c->opt.d;
    const int64_t count = row_count * d;
    const char *src = static_cast<const char *>(c->table[side]) + (size_t)row_begin * d * c->elem;
    const size_t dst_bytes = (size_t)count * (dst_dtype == ALX_BF16 ? 2 : 4);
    const bool same = (dst_dtype == ALX_BF16) == (c->bf16 != 0);
    if (on_device) {
        ALX_CUDA(c, launch_convert(src, c->bf16, dst, dst_dtype == ALX_BF16, count, c->stream, &c->launches));
    } else if (same) {
        ALX_CUDA(c, cudaMemcpyAsync(dst, src, dst_bytes, cudaMemcpyDeviceToHost, c->stream));
    } else {
        Scratch tmp(c);
        void *staging = tmp.keep(dev_alloc(c, dst_bytes));
        if (!staging) return fail(c, ALX_ERR_OOM, "staging allocation failed");
        ALX_CUDA(c, launch_convert(src, c->bf16, staging, dst_dtype == ALX_BF16, count, c->stream, &c->launches));
        ALX_CUDA(c, cudaMemcpyAsync(dst, staging, dst_bytes, cudaMemcpyDeviceToHost, c->stream));
        ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    return check_device_status(c);
}

alx_status alx_half_epoch(alx_ctx *c, alx_side side)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (side != ALX_ROWS && side != ALX_COLS) return fail(c, ALX_ERR_INVALID_ARG, "bad side");
    DeviceGuard guard(c->device);
    return half_epoch_impl(c, side, nullptr, nullptr);
}

namespace {
alx_status ensure_copy_stream(alx_ctx *c)
{
    if (!c->copy_stream) ALX_CUDA(c, cudaStreamCreateWithFlags(&c->copy_stream, cudaStreamNonBlocking));
    if (!c->copy_ev) ALX_CUDA(c, cudaEventCreateWithFlags(&c->copy_ev, cudaEventDisableTiming));
    return ALX_OK;
}

// Matrices of at most this many entries replay their epochs as a graph: a half-epoch is five to ten launches and three events,
// 20 us of host time, which the GPU outruns up to some million entries; beyond, it makes no difference
constexpr int64_t kGraphEntries = 1ll << 24;

// Captures the launches of one epoch (on the library's second stream, whatever stream the context works on).  The state the
// launches depend on -- tables and matrix in place, both tables set -- is that of every later epoch on this matrix.  Where
// capturing fails, epochs go on as single launches.
void capture_epoch(alx_ctx *c)
{
    if (ensure_copy_stream(c) != ALX_OK) return;
    cudaStream_t user = c->stream;
    const int64_t launches = c->launches;
    if (cudaStreamBeginCapture(c->copy_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) { cudaGetLastError(); return; }
    c->stream = c->copy_stream;
    c->capturing = true;
    alx_status st = half_epoch_impl(c, ALX_ROWS, nullptr, nullptr);
    if (st == ALX_OK) st = half_epoch_impl(c, ALX_COLS, nullptr, nullptr);
    c->capturing = false;
    c->stream = user;
    c->epoch_launches = c->launches - launches;
    c->launches = launches;
    cudaGraph_t graph = nullptr;
    if (cudaStreamEndCapture(c->copy_stream, &graph) != cudaSuccess || !graph) { cudaGetLastError(); return; }
    if (st == ALX_OK && cudaGraphInstantiate(&c->epoch_graph, graph, 0) != cudaSuccess) {
        cudaGetLastError();
        c->epoch_graph = nullptr;
    }
    cudaGraphDestroy(graph);
}
}  // namespace

alx_status alx_epoch(alx_ctx *c)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    if (c->epoch_graph && c->have_table[0] && c->have_table[1]) {
        NvtxRange range("alx epoch (graph)");
        ALX_CUDA(c, cudaGraphLaunch(c->epoch_graph, c->stream));
        c->launches += c->epoch_launches;
        // (the host-side state of a half-epoch is what the capture of the columns' half left)
        c->have_gram[ALX_ROWS] = true;
        c->have_gram[ALX_COLS] = false;
        note_half_epoch(c, ALX_COLS);
        c->by_stamps = warp_path(c) && !cg64(c);
        return ALX_OK;
    }
    alx_status st = half_epoch_impl(c, ALX_ROWS, nullptr, nullptr);
    if (st == ALX_OK) st = half_epoch_impl(c, ALX_COLS, nullptr, nullptr);
    if (st != ALX_OK) return st;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (++c->epochs_run == 2 && c->nnz <= kGraphEntries && cudaStreamIsCapturing(c->stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone)
        capture_epoch(c);
    return ALX_OK;
}


alx_status alx_load_host(alx_ctx *c, const int64_t *rowptr, const int32_t *colidx, const float *values, int64_t nnz,
                         const void *W, const void *H)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!W || !H) return fail(c, ALX_ERR_INVALID_ARG, "null table");
    DeviceGuard guard(c->device);
    alx_status st = ensure_copy_stream(c);
    if (st != ALX_OK) return st;
    c->upload_after_csr[ALX_ROWS] = W;
    c->upload_after_csr[ALX_COLS] = H;
    st = alx_set_csr(c, rowptr, colidx, values, nnz, 0);
    c->upload_after_csr[0] = c->upload_after_csr[1] = nullptr;
    const cudaError_t e = cudaStreamSynchronize(c->copy_stream);     // whatever alx_set_csr returned, the copies have ended
    if (st != ALX_OK) return st;
    ALX_CUDA(c, e);
    for (int sd = 0; sd < 2; ++sd) {
        c->have_table[sd] = true;
        c->have_gram[sd] = false;
    }
    return ALX_OK;
}

alx_status alx_epoch_to_host(alx_ctx *c, void *W_dst, void *H_dst)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!W_dst || !H_dst) return fail(c, ALX_ERR_INVALID_ARG, "null destination");
    DeviceGuard guard(c->device);
    alx_status st = ensure_copy_stream(c);
    if (st != ALX_OK) return st;
    st = half_epoch_impl(c, ALX_ROWS, nullptr, nullptr);
    if (st != ALX_OK) return st;
    // the new W goes to the host on the second stream while the column pass (which only reads it) runs
    ALX_CUDA(c, cudaEventRecord(c->copy_ev, c->stream));
    ALX_CUDA(c, cudaStreamWaitEvent(c->copy_stream, c->copy_ev, 0));
    ALX_CUDA(c, cudaMemcpyAsync(W_dst, c->table[ALX_ROWS], (size_t)c->n[ALX_ROWS] * c->opt.d * c->elem, cudaMemcpyDeviceToHost,
                                c->copy_stream));
    st = half_epoch_impl(c, ALX_COLS, nullptr, nullptr);
    if (st == ALX_OK)
        ALX_CUDA(c, cudaMemcpyAsync(H_dst, c->table[ALX_COLS], (size_t)c->n[ALX_COLS] * c->opt.d * c->elem,
                                    cudaMemcpyDeviceToHost, c->stream));
    const cudaError_t e = cudaStreamSynchronize(c->copy_stream);
    if (st != ALX_OK) return st;
    ALX_CUDA(c, e);
    return check_device_status(c);
}

alx_status alx_half_epoch_capture(alx_ctx *c, alx_side side, const int64_t *row_ids, int64_t k, float *x_out)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if ((side != ALX_ROWS && side != ALX_COLS) || k < 0 || (k > 0 && (!row_ids || !x_out)))
        return fail(c, ALX_ERR_INVALID_ARG, "bad argument to alx_half_epoch_capture");
    for (int64_t j = 0; j < k; ++j)
        if (row_ids[j] < 0 || row_ids[j] >= c->n[side]) return fail(c, ALX_ERR_INVALID_ARG, "row id out of range");
    DeviceGuard guard(c->device);
    const int64_t n = c->n[side];
    const int d = c->opt.d;
    Scratch tmp(c);
    int32_t *slot = nullptr;
    float *cap = nullptr;
    ALX_TMP(c, tmp, slot, n);
    ALX_TMP(c, tmp, cap, (k > 0 ? k : 1) * d);
    std::vector<int32_t> h(n, -1);
    for (int64_t j = 0; j < k; ++j) h[row_ids[j]] = (int32_t)j;   // a repeated id keeps its last slot
    ALX_CUDA(c, cudaMemcpyAsync(slot, h.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, c->stream));
    alx_status st = half_epoch_impl(c, side, slot, cap);
    if (st == ALX_OK) {
        std::vector<float> tmp((size_t)(k > 0 ? k : 1) * d);
        ALX_CUDA(c, cudaMemcpyAsync(tmp.data(), cap, sizeof(float) * k * d, cudaMemcpyDeviceToHost, c->stream));
        ALX_CUDA(c, cudaStreamSynchronize(c->stream));
        for (int64_t j = 0; j < k; ++j)
            memcpy(x_out + j * d, tmp.data() + (size_t)h[row_ids[j]] * d, sizeof(float) * d);
        st = check_device_status(c);
    } else {
        cudaStreamSynchronize(c->stream);
    }
    return st;
}

alx_status alx_gramian(alx_ctx *c, alx_side table, double *dst)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!dst || (table != ALX_ROWS && table != ALX_COLS)) return fail(c, ALX_ERR_INVALID_ARG, "bad argument");
    if (!c->have_table[table]) return fail(c, ALX_ERR_BAD_STATE, "table has not been set");
    DeviceGuard guard(c->device);
    alx_status st = gramian_of(c, table, false);
    if (st != ALX_OK) return st;
    return alx_get_gramian(c, table, dst);
}

alx_status alx_get_gramian(alx_ctx *c, alx_side side, double *dst)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!dst || (side != ALX_ROWS && side != ALX_COLS)) return fail(c, ALX_ERR_INVALID_ARG, "bad argument");
    if (!c->have_gram[side]) return fail(c, ALX_ERR_BAD_STATE, "no Gramian of that table is current");
    DeviceGuard guard(c->device);
    const int d = c->opt.d;
    ALX_CUDA(c, cudaMemcpyAsync(dst, c->G64[side], sizeof(double) * d * d, cudaMemcpyDeviceToHost, c->stream));
    return check_device_status(c);
}

alx_status alx_loss(alx_ctx *c, double *total, double *components)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (!total) return fail(c, ALX_ERR_INVALID_ARG, "null output");
    if (c->nnz < 0) return fail(c, ALX_ERR_BAD_STATE, "alx_loss before alx_set_csr");
    if (!c->have_table[0] || !c->have_table[1]) return fail(c, ALX_ERR_BAD_STATE, "both tables must be set");
    DeviceGuard guard(c->device);
    alx_status st = ensure_box(c);
    if (st != ALX_OK) return st;
    const bool beside_gramian = !tensor_path(c) && !(c->have_gram[0] && c->have_gram[1]);
    for (int s = 0; s < 2; ++s)
        if (!c->have_gram[s] && (st = gramian_of(c, s, false)) != ALX_OK) return st;
    double *h = reinterpret_cast<double *>(c->box + 64);
    ALX_CUDA(c, launch_loss(c->ptr[0], c->idx[0], c->val[0], c->n[0], c->nnz, c->table[0], c->table[1], c->bf16, c->opt.d, c->G64[0],
                            c->G64[1], (double)c->opt.alpha0, (double)c->opt.lambda, c->loss_partials_buf, c->loss_counter, c->status,
                            reinterpret_cast<DevStatus *>(c->box), h, beside_gramian, c->stream, &c->launches));
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    st = report_status(c);
    if (st != ALX_OK) return st;
    *total = h[0] + h[1] + h[2];
    if (components) { components[0] = h[0]; components[1] = h[1]; components[2] = h[2]; }
    return ALX_OK;
}

alx_status alx_get_transpose(alx_ctx *c, int64_t *colptr, int32_t *rowidx, float *values_t)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (c->nnz < 0) return fail(c, ALX_ERR_BAD_STATE, "alx_get_transpose before alx_set_csr");
    DeviceGuard guard(c->device);
    if (colptr) ALX_CUDA(c, cudaMemcpyAsync(colptr, c->ptr[1], sizeof(int64_t) * (c->n[1] + 1), cudaMemcpyDeviceToHost, c->stream));
    if (rowidx && c->nnz > 0) ALX_CUDA(c, cudaMemcpyAsync(rowidx, c->idx[1], sizeof(int32_t) * c->nnz, cudaMemcpyDeviceToHost, c->stream));
    if (values_t) {
        if (!c->has_values) return fail(c, ALX_ERR_BAD_STATE, "the matrix was set without labels");
        if (c->nnz > 0) ALX_CUDA(c, cudaMemcpyAsync(values_t, c->val[1], sizeof(float) * c->nnz, cudaMemcpyDeviceToHost, c->stream));
    }
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    return ALX_OK;
}

alx_status alx_get_buckets(alx_ctx *c, alx_side side, int32_t *order, int64_t *class_offsets, int64_t *chunk_desc,
                           int64_t *n_chunks)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (side != ALX_ROWS && side != ALX_COLS) return fail(c, ALX_ERR_INVALID_ARG, "bad side");
    if (c->nnz < 0) return fail(c, ALX_ERR_BAD_STATE, "alx_get_buckets before alx_set_csr");
    DeviceGuard guard(c->device);
    if (order) ALX_CUDA(c, cudaMemcpyAsync(order, c->order[side], sizeof(int32_t) * c->n[side], cudaMemcpyDeviceToHost, c->stream));
    if (class_offsets) memcpy(class_offsets, c->class_offs[side], sizeof(int64_t) * (ALX_N_CLASSES + 1));
    if (n_chunks) *n_chunks = c->n_chunks[side];
    if (chunk_desc && c->n_chunks[side] > 0)
        ALX_CUDA(c, cudaMemcpyAsync(chunk_desc, c->chunk_desc[side], sizeof(int64_t) * 4 * c->n_chunks[side], cudaMemcpyDeviceToHost, c->stream));
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    return ALX_OK;
}

namespace {
// The rows half-step of Eq. 4 on new rows, in a context that borrows the column table.  What alx_set_csr does for the rows'
// side and nothing of its columns' (the transpose and the degree classes of a million columns were most of the time of a
// call with a few rows); buffers are kept from call to call, the solver's history is not.
alx_status fold_in_impl(alx_ctx *k, const int64_t *rowptr, const int32_t *colidx, const float *values, int64_t n, int64_t nnz, int on_device,
                        float *x_out)
{
    const int d = k->opt.d;
    alx_status st = ensure_box(k);
    if (st != ALX_OK) return st;
    // The Gramian of the column table needs nothing of the new rows: it runs beside their upload, checks and classes, on the
    // second stream (a request for a few rows waited 75 us for it after 60 us of those).  B^-1 too where the rows could have use for it.
    if ((st = ensure_copy_stream(k)) != ALX_OK) return st;
    ALX_CUDA(k, cudaEventRecord(k->copy_ev, k->stream));
    ALX_CUDA(k, cudaStreamWaitEvent(k->copy_stream, k->copy_ev, 0));
    if ((st = gramian_of(k, ALX_COLS, n >= kDualLeastRows, nullptr, k->copy_stream)) != ALX_OK) return st;
    ALX_CUDA(k, cudaEventRecord(k->copy_ev, k->copy_stream));
    // what the last call left
    dev_free(k, k->chunk_desc[0]); k->chunk_desc[0] = nullptr;
    dev_free(k, k->split_first[0]); k->split_first[0] = nullptr;
    k->nnz = -1;
    k->n[ALX_ROWS] = n;
    k->has_values = values != nullptr;
    k->have_table[ALX_ROWS] = false;
    // upload (or take the caller's device arrays as they are: they are only read, and not after the call)
    if (on_device) {
        k->ptr[0] = const_cast<int64_t *>(rowptr);
        k->idx[0] = const_cast<int32_t *>(colidx);
        k->val[0] = const_cast<float *>(values);
    } else {
        Upload up(k);
        void *dev[4];
        up.add(rowptr, sizeof(int64_t) * (n + 1));
        up.add(colidx, sizeof(int32_t) * nnz);
        if (values) up.add(values, sizeof(float) * nnz);
        if ((st = up.send(kKeptRows, dev)) != ALX_OK) return st;
        k->ptr[0] = static_cast<int64_t *>(dev[0]);
        k->idx[0] = static_cast<int32_t *>(dev[1]);
        k->val[0] = values ? static_cast<float *>(dev[2]) : nullptr;
    }
    void *order = nullptr, *scratch = nullptr, *table = nullptr, *list = nullptr, *sums = nullptr;
    const int64_t nb = bucket_blocks(n);
    const int64_t scan_elems = scan_scratch_elems(nb * kNClasses > n ? nb * kNClasses : n) + 16;
    if ((st = keep(k, kKeptOrder, sizeof(int32_t) * n, &order)) != ALX_OK) return st;
    if ((st = keep(k, kKeptScratch, sizeof(int64_t) * (2 * nb * kNClasses + 1 + scan_elems), &scratch)) != ALX_OK) return st;
    if ((st = keep(k, kKeptTable, (size_t)n * d * k->elem, &table)) != ALX_OK) return st;
    k->order[0] = static_cast<int32_t *>(order);
    k->table[0] = table;
    if (k->opt.solver == ALX_SOLVER_AUTO && (tensor_path(k) || cg64(k))) {
        if ((st = keep(k, kKeptFallback, sizeof(int32_t) * n, &list)) != ALX_OK) return st;
        k->cg_fallback_list = static_cast<int32_t *>(list);
    }
    if (k->cg_policy) ALX_CUDA(k, cudaMemsetAsync(k->cg_policy, 0, 2 * sizeof(CgPolicy), k->stream));
    int64_t *blk_counts = static_cast<int64_t *>(scratch), *blk_offs = blk_counts + nb * kNClasses, *scan = blk_offs + nb * kNClasses + 1;
    ALX_CUDA(k, launch_validate(k->ptr[0], k->idx[0], n, k->n[1], nnz, k->status, k->stream, &k->launches));
    // (the degree classes only look at the offsets' differences: nothing is indexed with them before the check below)
    ALX_CUDA(k, launch_bucket(k->ptr[0], n, k->split, blk_counts, blk_offs, scan, scan_elems, k->order[0], k->class_offs_dev[0], k->stream,
                              &k->launches));
    {
        Download down(k);
        if ((st = down.add(k->class_offs[0], k->class_offs_dev[0], sizeof(int64_t) * (ALX_N_CLASSES + 1))) != ALX_OK) return st;
        if ((st = check_device_status(k)) != ALX_OK) return st;
        down.take();
    }
    if ((st = build_chunks(k, 0, scan, scan_elems)) != ALX_OK) return st;
    if (sums_floats(k, 0) > 0) {
        if ((st = keep(k, kKeptSums, sizeof(float) * sums_floats(k, 0), &sums)) != ALX_OK) return st;
        k->split_partials = static_cast<float *>(sums);
    }
    k->nnz = nnz;
    if ((st = half_epoch_impl(k, ALX_ROWS, nullptr, nullptr, true)) != ALX_OK) return st;
    const size_t bytes = sizeof(float) * n * d;
    if (on_device) {
        ALX_CUDA(k, launch_convert(k->table[0], k->bf16, x_out, 0, n * d, k->stream, &k->launches));
        return check_device_status(k);
    }
    const void *x = k->table[0];
    if (k->bf16) {
        void *wide = nullptr;
        if ((st = keep(k, kKeptOut, bytes, &wide)) != ALX_OK) return st;
        ALX_CUDA(k, launch_convert(k->table[0], 1, wide, 0, n * d, k->stream, &k->launches));
        x = wide;
    }
    Download down(k);
    if ((st = down.add(x_out, x, bytes)) != ALX_OK) return st;
    st = check_device_status(k);
    if (st == ALX_OK) down.take();
    return st;
}
}  // namespace

alx_status alx_fold_in(alx_ctx *c, const int64_t *rowptr, const int32_t *colidx, const float *values, int64_t n_new,
                       int64_t nnz, int on_device, float *x_out)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (n_new < 0 || nnz < 0 || n_new >= (1ll << 31) || (n_new > 0 && (!rowptr || !x_out)) || (nnz > 0 && !colidx))
        return fail(c, ALX_ERR_INVALID_ARG, "bad argument to alx_fold_in");
    if (!c->have_table[ALX_COLS]) return fail(c, ALX_ERR_BAD_STATE, "the column table has not been set or solved yet");
    if (n_new == 0) return ALX_OK;
    DeviceGuard guard(c->device);
    std::lock_guard<std::mutex> lock(c->calls);
    if (!c->fold) {
        // a context of its own for the new rows: same options, the column table borrowed
        alx_options o = c->opt;
        o.n_rows = 1;
        o.device = c->device;
        alx_status st = create_impl(&o, c, &c->fold);
        if (st != ALX_OK) return fail(c, st, "alx_fold_in: the context for the new rows could not be created");
        c->fold->have_table[ALX_COLS] = true;
    }
    alx_ctx *k = c->fold;
    const int64_t before = k->launches;
    alx_status st = fold_in_impl(k, rowptr, colidx, values, n_new, nnz, on_device, x_out);
    c->launches += k->launches - before;
    if (st != ALX_OK) {
        cudaStreamSynchronize(k->stream);
        if (k->copy_stream) cudaStreamSynchronize(k->copy_stream);
        c->err = "alx_fold_in: " + k->err;
    }
    give_back_large(k);
    return st;
}

alx_status alx_topk(alx_ctx *c, alx_side items, const float *queries, int64_t m, int32_t k, const int64_t *exclude_ptr,
                    const int32_t *exclude_idx, int on_device, int32_t *ids_out, float *scores_out)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if ((items != ALX_ROWS && items != ALX_COLS) || m < 0 || k < 1 || k > ALX_MAX_TOPK || (m > 0 && (!queries || !ids_out)) ||
        (exclude_ptr && !exclude_idx && m > 0))
        return fail(c, ALX_ERR_INVALID_ARG, "bad argument to alx_topk");
    if (!c->have_table[items]) return fail(c, ALX_ERR_BAD_STATE, "the table has not been set or solved yet");
    if (m == 0) return ALX_OK;
    DeviceGuard guard(c->device);
    NvtxRange range("alx_topk");
    const int d = c->opt.d;
    const int64_t n_items = c->n[items];
    std::lock_guard<std::mutex> lock(c->calls);
    const float *Q = queries;
    const int64_t *ex_ptr = exclude_ptr;
    const int32_t *ex_idx = exclude_idx;
    int32_t *ids_dev = ids_out;
    float *scores_dev = scores_out;
    alx_status st;
    if (!on_device) {
        Upload up(c);
        void *dev[4];
        up.add(queries, sizeof(float) * m * d);
        if (exclude_ptr) {
            if (exclude_ptr[m] < 0) return fail(c, ALX_ERR_INVALID_ARG, "alx_topk: negative length of the exclusion lists");
            up.add(exclude_ptr, sizeof(int64_t) * (m + 1));
            up.add(exclude_idx, sizeof(int32_t) * exclude_ptr[m]);
        }
        if ((st = up.send(kKeptUpload, dev)) != ALX_OK) return st;
        Q = static_cast<const float *>(dev[0]);
        if (exclude_ptr) {
            ex_ptr = static_cast<const int64_t *>(dev[1]);
            ex_idx = static_cast<const int32_t *>(dev[2]);
        }
        void *out = nullptr;
        const size_t list = aligned(sizeof(int32_t) * m * k);
        if ((st = keep(c, kKeptOut, 2 * list, &out)) != ALX_OK) return st;
        ids_dev = static_cast<int32_t *>(out);
        scores_dev = scores_out ? reinterpret_cast<float *>(static_cast<unsigned char *>(out) + list) : nullptr;
    }
    const TopkPlan plan = topk_plan(n_items, m, k, c->opt.kernels != 1 && c->bf16 && d == 128);
    void *work = nullptr;
    if ((st = keep(c, kKeptWork, plan.workspace_bytes(), &work)) != ALX_OK) return st;
    const cudaError_t e = launch_topk(plan, c->table[items], c->bf16 != 0, n_items, d, Q, m, k, ex_ptr, ex_idx, work, ids_dev, scores_dev,
                                      c->status, c->stream, &c->launches);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(c->stream);
        return fail(c, ALX_ERR_CUDA, "alx_topk: %s", cudaGetErrorString(e));
    }
    Download down(c);
    if (!on_device) {
        if ((st = down.add(ids_out, ids_dev, sizeof(int32_t) * m * k)) != ALX_OK) return st;
        if (scores_out && (st = down.add(scores_out, scores_dev, sizeof(float) * m * k)) != ALX_OK) return st;
    }
    st = check_device_status(c);
    if (st == ALX_OK) down.take();
    give_back_large(c);
    return st;
}

alx_status alx_recall_at_k(alx_ctx *c, const int32_t *ids, int64_t m, int32_t k_stride, int32_t k, const int64_t *truth_ptr,
                           const int32_t *truth_idx, int on_device, double *recall, int64_t *n_counted)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    if (m < 0 || k < 1 || k > k_stride || !recall || (m > 0 && (!ids || !truth_ptr)))
        return fail(c, ALX_ERR_INVALID_ARG, "bad argument to alx_recall_at_k");
    DeviceGuard guard(c->device);
    std::lock_guard<std::mutex> lock(c->calls);
    const int32_t *ids_dev = ids;
    const int64_t *tp = truth_ptr;
    const int32_t *ti = truth_idx;
    alx_status st;
    if (!on_device && m > 0) {
        const int64_t nt = truth_ptr[m];
        if (nt < 0 || (nt > 0 && !truth_idx)) return fail(c, ALX_ERR_INVALID_ARG, "alx_recall_at_k: bad ground-truth lists");
        Upload up(c);
        void *dev[4];
        up.add(ids, sizeof(int32_t) * m * k_stride);
        up.add(truth_ptr, sizeof(int64_t) * (m + 1));
        up.add(truth_idx, sizeof(int32_t) * nt);
        if ((st = up.send(kKeptUpload, dev)) != ALX_OK) return st;
        ids_dev = static_cast<const int32_t *>(dev[0]);
        tp = static_cast<const int64_t *>(dev[1]);
        ti = static_cast<const int32_t *>(dev[2]);
    }
    void *work = nullptr;
    if ((st = keep(c, kKeptWork, sizeof(double) * (2 + (m > 0 ? m : 1)), &work)) != ALX_OK) return st;
    double *out2 = static_cast<double *>(work), *per_query = out2 + 2;
    ALX_CUDA(c, launch_recall(ids_dev, m, k_stride, k, tp, ti, per_query, out2, c->stream, &c->launches));
    double h[2] = {0.0, 0.0};
    Download down(c);
    if ((st = down.add(h, out2, sizeof h)) != ALX_OK) return st;
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    down.take();
    give_back_large(c);
    *recall = h[1] > 0.0 ? h[0] / h[1] : 0.0;
    if (n_counted) *n_counted = (int64_t)h[1];
    return ALX_OK;
}

alx_status alx_get_stats(alx_ctx *c, alx_stats *out)
{
    if (!c || !out) return ALX_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    float ms = 0.f;
    if (c->by_stamps) {
        unsigned long long t[kStampSlots];
        ALX_CUDA(c, cudaMemcpy(t, c->stamps, sizeof t, cudaMemcpyDeviceToHost));
        c->stats.ms_gramian = 1e-6 * (double)(t[kStampGramian] - t[kStampBegin]);
        c->stats.ms_rows = t[kStampEnd] > t[kStampGramian] ? 1e-6 * (double)(t[kStampEnd] - t[kStampGramian]) : 0.0;
        c->stats.ms_half_epoch = c->stats.ms_gramian + c->stats.ms_rows;
    } else {
        if (cudaEventElapsedTime(&ms, c->ev[0], c->ev[1]) == cudaSuccess) c->stats.ms_gramian = ms; else cudaGetLastError();
        if (cudaEventElapsedTime(&ms, c->ev[1], c->ev[2]) == cudaSuccess) c->stats.ms_rows = ms; else cudaGetLastError();
        if (cudaEventElapsedTime(&ms, c->ev[0], c->ev[2]) == cudaSuccess) c->stats.ms_half_epoch = ms; else cudaGetLastError();
    }
    c->stats.ms_main_kernel = 0.0;
    if (c->main_timed) {
        if (cudaEventElapsedTime(&ms, c->ev[3], c->ev[4]) == cudaSuccess) c->stats.ms_main_kernel = ms; else cudaGetLastError();
    }
    // (the flag and the record are rewritten by half-epochs only)
    c->stats.dual_rows = 0;
    if (c->dual_candidates > 0) {
        int flag = 0;
        CgPolicy pol{};
        ALX_CUDA(c, cudaMemcpy(&flag, dual_flag_of(c), sizeof flag, cudaMemcpyDeviceToHost));
        if (c->cg_policy) ALX_CUDA(c, cudaMemcpy(&pol, c->cg_policy + c->last_side, sizeof pol, cudaMemcpyDeviceToHost));
        if (flag) c->stats.dual_rows = c->dual_candidates - (pol.short_rows_by_cg ? c->dual_candidates32 : 0);
    }
    {
        unsigned long long h[5] = {0, 0, 0, 0, 0};
        ALX_CUDA(c, cudaMemcpy(h, c->cg_counters, sizeof h, cudaMemcpyDeviceToHost));
        c->stats.cg_rows = (int64_t)h[0];
        c->stats.cg_products = (int64_t)h[1];
        c->stats.cg_fallbacks = (int64_t)h[2];
        c->stats.dual_polished_rows = (int64_t)h[3];
        c->stats.dual_polish_products = (int64_t)h[4];
        c->stats.cholesky_by_policy[0] = c->stats.cholesky_by_policy[1] = 0;
        if (c->cg_policy) {
            CgPolicy pol[2];
            ALX_CUDA(c, cudaMemcpy(pol, c->cg_policy, sizeof pol, cudaMemcpyDeviceToHost));
            for (int sd = 0; sd < 2; ++sd) c->stats.cholesky_by_policy[sd] = pol[sd].use_cholesky;
        }
    }
    c->stats.kernel_launches = c->launches;
    c->stats.workspace_bytes = c->bytes_held;
    *out = c->stats;
    return ALX_OK;
}

alx_status alx_fp32_peak_tflops(alx_ctx *c, double *tflops)
{
    if (!c || !tflops) return ALX_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    ALX_CUDA(c, cudaStreamSynchronize(c->stream));
    double v = 0.0;
    ALX_CUDA(c, measure_fp32_peak(&v, c->stream));
    *tflops = v;
    return ALX_OK;
}

alx_status alx_synchronize(alx_ctx *c)
{
    if (!c) return ALX_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    return check_device_status(c);
}

}  // extern "C"
