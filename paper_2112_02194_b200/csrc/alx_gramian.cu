// Gramian of the fixed table, G = X^T X over all of its rows (Alg. 1 line 2; the remark under Eq. 4
// that sum_i h_i (x) h_i does not depend on the row being solved), and the base matrix
// alpha0 G + lambda I that every row's normal matrix starts from (Alg. 1 line 5).
//
// FP32-ALU version: blocks (a function of the table size only) each sum a range of rows; a block's groups of threads sum at
// most kFlushRows rows each in fp32 and hand those sums over to fp64 accumulators; the blocks' results are added in a fixed
// order in fp64.  So the result does not depend on how blocks are scheduled.
#include <mutex>
#include <string>

#include "../../include/alx.h"
#include "alx_common.cuh"
#include "alx_ptx.cuh"

namespace alx {

namespace {

constexpr int kGramBlocks = 148;      // one block per SM
constexpr int kStageGroupRows = 8;    // rows of a staged tile per group
constexpr int kFlushRows = 128;       // rows a group sums in fp32

// A thread owns a TILE x TILE tile of the lower triangle, TILES threads form a group, the groups of a block take different
// rows.  (One block per 4096 rows with full tiles left most of the chip idle on small tables and did twice the products:
// 2000 x 16 40 us, 60k x 128 fp32 0.62 ms.)
template <int D, typename T> struct GramGeo {
    static constexpr int TILE = D >= 32 ? 8 : 4, TG = D / TILE, TILES = TG * (TG + 1) / 2, TT = TILE * TILE;
    static constexpr int GROUPS = D == 128 ? 3 : D == 64 ? 12 : 40;
    static constexpr int THREADS = (TILES * GROUPS + 31) / 32 * 32;
    static constexpr int STAGE_ROWS = GROUPS * kStageGroupRows;
    static constexpr int STAGE = STAGE_ROWS * D * (int)sizeof(T);
    static constexpr int ELEMS = TILES * TT;
    static constexpr int PER = (ELEMS + THREADS - 1) / THREADS;
    static constexpr size_t SMEM = 2 * (size_t)STAGE + sizeof(float) * GROUPS * ELEMS;
    // feature number r of tile row or column I.  fp32: 16-byte chunks TG apart, so that the reads of neighbouring tiles meet
    // different banks; bfloat16: one chunk
    __host__ __device__ static constexpr int feature(int I, int r) { return sizeof(T) == 4 ? 4 * (I + (r / 4) * TG) + r % 4 : TILE * I + r; }
};

template <int D> __device__ __forceinline__ void load_tile(const float *row, int I, float (&v)[D >= 32 ? 8 : 4])
{
#pragma unroll
    for (int c = 0; c < (D >= 32 ? 2 : 1); ++c) {
        const float4 q = *reinterpret_cast<const float4 *>(row + 4 * (I + c * (D / 8)));
        v[4 * c] = q.x; v[4 * c + 1] = q.y; v[4 * c + 2] = q.z; v[4 * c + 3] = q.w;
    }
}
template <int D> __device__ __forceinline__ void load_tile(const __nv_bfloat16 *row, int I, float (&v)[D >= 32 ? 8 : 4])
{
    uint32_t w[D >= 32 ? 4 : 2];
    if constexpr (D >= 32) {
        const uint4 q = *reinterpret_cast<const uint4 *>(row + 8 * I);
        w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
    } else {
        const uint2 q = *reinterpret_cast<const uint2 *>(row + 4 * I);
        w[0] = q.x; w[1] = q.y;
    }
#pragma unroll
    for (int c = 0; c < (D >= 32 ? 4 : 2); ++c) {
        v[2 * c] = __uint_as_float(w[c] << 16);
        v[2 * c + 1] = __uint_as_float(w[c] & 0xFFFF0000u);
    }
}

template <int D, typename T>
__global__ void __launch_bounds__(GramGeo<D, T>::THREADS, 1) k_gramian_tiles(const T *__restrict__ X, int64_t n, int64_t rows_per_block,
                                                                            float *__restrict__ partials, unsigned long long *begin)
{
    if (blockIdx.x == 0) stamp(begin);
    let_next_start();
    using G = GramGeo<D, T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *red = reinterpret_cast<float *>(smem_raw + 2 * G::STAGE);
    const int tid = threadIdx.x, group = tid / G::TILES, tile = tid % G::TILES;
    const bool live = group < G::GROUPS;
    int I = 0;
    while ((I + 1) * (I + 2) / 2 <= tile) ++I;
    const int J = tile - I * (I + 1) / 2;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
    const int64_t r1 = r0 + rows_per_block < n ? r0 + rows_per_block : n;
    const int stages = (int)((r1 - r0 + G::STAGE_ROWS - 1) / G::STAGE_ROWS);

    auto load = [&](int s) {
        const int64_t base = r0 + (int64_t)s * G::STAGE_ROWS;
        const int64_t bytes = (r1 - base < G::STAGE_ROWS ? r1 - base : G::STAGE_ROWS) * D * (int)sizeof(T);
        const unsigned char *src = reinterpret_cast<const unsigned char *>(X + base * D);
        const uint32_t dst = ptx::smem_u32(smem_raw) + (s & 1) * G::STAGE;
        for (int p = tid * 16; p < bytes; p += G::THREADS * 16) ptx::cp_async16(dst + p, src + p);
    };
    float acc[G::TILE][G::TILE];
    double sum[G::PER];
#pragma unroll
    for (int a = 0; a < G::TILE; ++a)
#pragma unroll
        for (int b = 0; b < G::TILE; ++b) acc[a][b] = 0.f;
#pragma unroll
    for (int e = 0; e < G::PER; ++e) sum[e] = 0.0;
    if (stages > 0) load(0);
    ptx::cp_async_commit();
    for (int s = 0; s < stages; ++s) {
        if (s + 1 < stages) load(s + 1);
        ptx::cp_async_commit();
        ptx::cp_async_wait<1>();
        __syncthreads();
        const T *stage = reinterpret_cast<const T *>(smem_raw + (s & 1) * G::STAGE);
        const int64_t left = r1 - r0 - (int64_t)s * G::STAGE_ROWS;
        if (live) {
#pragma unroll 2
            for (int k = 0; k < kStageGroupRows; ++k) {
                const int r = k * G::GROUPS + group;
                if (r >= left) break;
                float x[G::TILE], y[G::TILE];
                load_tile<D>(stage + r * D, I, x);
                load_tile<D>(stage + r * D, J, y);
#pragma unroll
                for (int a = 0; a < G::TILE; ++a)
#pragma unroll
                    for (int b = 0; b < G::TILE; ++b) acc[a][b] = fmaf(x[a], y[b], acc[a][b]);
            }
        }
        if ((s + 1) % (kFlushRows / kStageGroupRows) == 0 || s + 1 == stages) {
            // the groups' fp32 sums to the fp64 accumulators
            if (live) {
#pragma unroll
                for (int a = 0; a < G::TILE; ++a)
#pragma unroll
                    for (int b = 0; b < G::TILE; ++b) {
                        red[(group * G::TT + a * G::TILE + b) * G::TILES + tile] = acc[a][b];
                        acc[a][b] = 0.f;
                    }
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < G::PER; ++e) {
                const int at = tid + e * G::THREADS;
                if (at < G::ELEMS)
#pragma unroll 4
                    for (int g = 0; g < G::GROUPS; ++g) sum[e] += (double)red[g * G::ELEMS + at];
            }
        }
        __syncthreads();
    }
    float *out = partials + (int64_t)blockIdx.x * G::ELEMS;
#pragma unroll
    for (int e = 0; e < G::PER; ++e)
        if (tid + e * G::THREADS < G::ELEMS) out[tid + e * G::THREADS] = (float)sum[e];
}

// Partial sums added in fp64 in a fixed order (eight interleaved sums, then those in order), and alpha0 G + lambda I in fp32.
// where(e, i, l): element e of a partial is G[i][l].  MIRROR: the partials hold a triangle, (l, i) is written too (tiles on the
// diagonal hold both: the same products in the same order, so equal bits).
template <bool MIRROR, typename Where>
__device__ __forceinline__ void reduce_partials(const float *__restrict__ partials, int64_t n_partials, int elems, int d, double *__restrict__ G64,
                                                float *__restrict__ Bmat, float alpha0, float lambda, Where where)
{
    __shared__ double part[8][32];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (e < elems) {
#pragma unroll 8
        for (int64_t p = slice; p < n_partials; p += 8) s += (double)partials[p * elems + e];
    }
    part[slice][lane] = s;
    __syncthreads();
    if (slice != 0 || e >= elems) return;
#pragma unroll
    for (int k = 1; k < 8; ++k) s += part[k][lane];
    int i, l;
    where(e, i, l);
    const float v = (float)((double)alpha0 * s + (i == l ? (double)lambda : 0.0));
    G64[i * d + l] = s;
    Bmat[i * d + l] = v;
    if (MIRROR) {
        G64[l * d + i] = s;
        Bmat[l * d + i] = v;
    }
}

template <int D, typename T>
__global__ void __launch_bounds__(256) k_gramian_reduce_tiles(const float *__restrict__ partials, int64_t n_partials, double *__restrict__ G64,
                                                              float *__restrict__ Bmat, float alpha0, float lambda,
                                                              unsigned long long *done)
{
    using G = GramGeo<D, T>;
    let_next_start();
    wait_for_previous();
    reduce_partials<true>(partials, n_partials, G::ELEMS, D, G64, Bmat, alpha0, lambda, [](int e, int &i, int &l) {
        const int tile = e % G::TILES, ab = e / G::TILES;
        int I = 0;
        while ((I + 1) * (I + 2) / 2 <= tile) ++I;
        i = G::feature(I, ab / G::TILE);
        l = G::feature(tile - I * (I + 1) / 2, ab % G::TILE);
    });
    stamp(done);
}

// full d x d partials (the tensor-core Gramian)
__global__ void __launch_bounds__(256) k_gramian_reduce(const float *__restrict__ partials, int64_t n_partials, int d,
                                                        double *__restrict__ G64, float *__restrict__ Bmat, float alpha0, float lambda)
{
    reduce_partials<false>(partials, n_partials, d * d, d, G64, Bmat, alpha0, lambda, [d](int e, int &i, int &l) { i = e / d; l = e % d; });
}

template <int D, typename T>
cudaError_t gramian_tiles_dt(const void *X, int64_t n, float *partials, double *G64, float *Bmat, float alpha0, float lambda,
                             unsigned long long *stamps, cudaStream_t s)
{
    using G = GramGeo<D, T>;
    static_assert(G::ELEMS <= D * D && G::SMEM <= 232448, "sizes");
    static SmemOnce allow;
    const cudaError_t e = allow(k_gramian_tiles<D, T>, G::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t blocks = gramian_partials(n), per = (n + blocks - 1) / blocks;
    k_gramian_tiles<D, T><<<(unsigned)blocks, G::THREADS, G::SMEM, s>>>(static_cast<const T *>(X), n, per, partials, stamps ? stamps + kStampBegin : nullptr);
    return launch_early(true, k_gramian_reduce_tiles<D, T>, (G::ELEMS + 31) / 32, 256, 0, s, partials, blocks, G64, Bmat, alpha0, lambda,
                        stamps ? stamps + kStampGramian : nullptr);
}

template <int D>
cudaError_t gramian_tiles_d(const void *X, int bf16, int64_t n, float *partials, double *G64, float *Bmat, float alpha0, float lambda,
                            unsigned long long *stamps, cudaStream_t s)
{
    return bf16 ? gramian_tiles_dt<D, __nv_bfloat16>(X, n, partials, G64, Bmat, alpha0, lambda, stamps, s)
                : gramian_tiles_dt<D, float>(X, n, partials, G64, Bmat, alpha0, lambda, stamps, s);
}

cudaError_t gramian_tiles(const void *X, int bf16, int64_t n, int d, float *partials, double *G64, float *Bmat, float alpha0, float lambda,
                          unsigned long long *stamps, cudaStream_t s)
{
    switch (d) {
    case 16: return gramian_tiles_d<16>(X, bf16, n, partials, G64, Bmat, alpha0, lambda, stamps, s);
    case 32: return gramian_tiles_d<32>(X, bf16, n, partials, G64, Bmat, alpha0, lambda, stamps, s);
    case 64: return gramian_tiles_d<64>(X, bf16, n, partials, G64, Bmat, alpha0, lambda, stamps, s);
    case 128: return gramian_tiles_d<128>(X, bf16, n, partials, G64, Bmat, alpha0, lambda, stamps, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// blocks of the FP32-ALU Gramian: at least 64 rows each, at most one per SM
int64_t gramian_partials(int64_t n)
{
    const int64_t b = (n + 63) / 64;
    return b < kGramBlocks ? (b > 0 ? b : 1) : kGramBlocks;
}

cudaError_t launch_gramian_reduce(const float *partials, int64_t n_partials, int d, double *G64, float *Bmat,
                                  float alpha0, float lambda, cudaStream_t s, int64_t *launches)
{
    k_gramian_reduce<<<(d * d + 31) / 32, 256, 0, s>>>(partials, n_partials, d, G64, Bmat, alpha0, lambda);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_gramian(const void *X, int bf16, int64_t n, int d, float *partials, double *G64, float *Bmat,
                           float alpha0, float lambda, unsigned long long *stamps, cudaStream_t s, int64_t *launches)
{
    *launches += 2;
    return gramian_tiles(X, bf16, n, d, partials, G64, Bmat, alpha0, lambda, stamps, s);
}

}  // namespace alx

// ---- FP32 FMA throughput probe (diagnostic; gives the denominator of the ALU roofline) ------------
namespace alx {
namespace {
__global__ void __launch_bounds__(256) k_ffma_probe(float *out, int iters)
{
    float a[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) a[k] = 1.0f + 1e-3f * (float)(threadIdx.x + k);
    const float m = 0.999999f, c = 1e-7f;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int k = 0; k < 16; ++k) a[k] = fmaf(a[k], m, c);
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) s += a[k];
    if (s == 12345.678f) out[0] = s;   // keeps the loop alive; practically never taken
}
}  // namespace

cudaError_t measure_fp32_peak(double *tflops, cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    float *out = nullptr;
    cudaError_t e = cudaMalloc(&out, 256);
    if (e != cudaSuccess) return e;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int iters = 1 << 16, grid = sms * 8;
    double best = 0.0;
    for (int rep = 0; rep < 4; ++rep) {
        cudaEventRecord(e0, s);
        k_ffma_probe<<<grid, 256, 0, s>>>(out, iters);
        cudaEventRecord(e1, s);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        const double fl = 2.0 * 16.0 * (double)iters * 256.0 * (double)grid;
        if (rep > 0 && ms > 0.f && fl / (ms * 1e-3) * 1e-12 > best) best = fl / (ms * 1e-3) * 1e-12;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    *tflops = best;
    return cudaGetLastError();
}
}  // namespace alx

// ---- Gramian without any allocation ---------------------------------------------------------------
// For callers that must not allocate device memory at the time of the call: code running inside a
// memory pool that has been frozen, a host thread that may not take the allocator's lock, a service
// whose memory budget was fixed at start-up.  The piece sums that the context-based path keeps in a
// buffer it allocates live here in a fixed array that is part of the library image, so every GPU that
// loads the library carries kNoAllocScratchFloats * 4 bytes (16 MiB + 64 KiB) until the process exits.
namespace alx {
namespace {

constexpr int64_t kNoAllocPieceFloats = 4ll << 20;                       // room for the piece sums
constexpr int64_t kNoAllocRowsPerPiece = 4096;                           // the limit on n: this many rows per d x d piece that fits
constexpr int64_t kNoAllocScratchFloats = kNoAllocPieceFloats + 128 * 128;  // + one d x d fp32 by-product
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocScratchFloats];

constexpr int kNoAllocMaxDevices = 64;
float *g_noalloc_ptr[kNoAllocMaxDevices] = {};   // device address of the array, per device ordinal
std::mutex g_noalloc_mutex;
thread_local std::string g_noalloc_error;

alx_status noalloc_fail(alx_status code, const std::string &msg)
{
    g_noalloc_error = msg;
    return code;
}

}  // namespace
}  // namespace alx

extern "C" {

int64_t alx_gramian_noalloc_max_rows(int32_t d)
{
    if (d != 16 && d != 32 && d != 64 && d != 128) return 0;
    return (alx::kNoAllocPieceFloats / ((int64_t)d * d)) * alx::kNoAllocRowsPerPiece;
}

const char *alx_noalloc_last_error(void) { return alx::g_noalloc_error.c_str(); }

alx_status alx_gramian_noalloc(const void *table, alx_dtype dtype, int64_t n, int32_t d, double *gramian,
                               void *stream)
{
    using namespace alx;
    if (!table || !gramian || n < 1 || (dtype != ALX_F32 && dtype != ALX_BF16))
        return noalloc_fail(ALX_ERR_INVALID_ARG, "alx_gramian_noalloc: null pointer, n < 1 or unknown dtype");
    if (d != 16 && d != 32 && d != 64 && d != 128)
        return noalloc_fail(ALX_ERR_UNSUPPORTED, "alx_gramian_noalloc: d must be 16, 32, 64 or 128");
    // the kernels read the table in 16-byte pieces and write doubles: a pointer that is not aligned for that would
    // fault on the device instead of being refused here
    if ((reinterpret_cast<uintptr_t>(table) & 15u) != 0 || (reinterpret_cast<uintptr_t>(gramian) & 7u) != 0)
        return noalloc_fail(ALX_ERR_INVALID_ARG,
                            "alx_gramian_noalloc: table must be 16-byte aligned and gramian 8-byte aligned");
    const int64_t max_rows = alx_gramian_noalloc_max_rows(d);
    if (n > max_rows)
        return noalloc_fail(ALX_ERR_UNSUPPORTED,
                            "alx_gramian_noalloc: " + std::to_string(n) + " rows exceed the fixed scratch array (at most " +
                                std::to_string(max_rows) + " rows for d = " + std::to_string(d) +
                                "); use a context and alx_gramian instead");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices)
        return noalloc_fail(ALX_ERR_CUDA, "alx_gramian_noalloc: no current CUDA device");
    float *scratch = nullptr;
    {
        // set-up, once per device, with that device current: the array's name is only a handle in host
        // code; the kernels need its device address
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_ptr[dev]) {
            void *p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || !p)
                return noalloc_fail(ALX_ERR_CUDA, std::string("alx_gramian_noalloc: cudaGetSymbolAddress failed: ") +
                                                      cudaGetErrorString(e));
            g_noalloc_ptr[dev] = static_cast<float *>(p);
        }
        scratch = g_noalloc_ptr[dev];
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    float *pieces = scratch, *base_out = scratch + kNoAllocPieceFloats;
    // every piece the reduction reads is written in full by the launch before it: nothing has to start at zero
    const cudaError_t e = gramian_tiles(table, dtype == ALX_BF16, n, d, pieces, gramian, base_out, 0.f, 0.f, nullptr, s);
    if (e != cudaSuccess)
        return noalloc_fail(ALX_ERR_CUDA, std::string("alx_gramian_noalloc: launch failed: ") + cudaGetErrorString(e));
    g_noalloc_error.clear();
    return ALX_OK;
}

}  // extern "C"
