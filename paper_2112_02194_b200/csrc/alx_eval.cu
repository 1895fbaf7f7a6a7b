// Recall@K (the metric of Table 2) of retrieved ids against held-out ground truth.
#include "alx_common.cuh"

namespace alx {

namespace {

// Recall@K of one query: hits among its first k ids / number of ground-truth ids (ascending, unique); queries without
// ground truth get -1 and are left out of the mean.  A warp per query, a lane per id: the bisections are chains of
// dependent loads, 32 of which run side by side (a thread per query took 41 us for 2048 x 50 ids).
__global__ void __launch_bounds__(256) k_recall_rows(const int32_t *__restrict__ ids, int64_t m, int k_stride, int k,
                                                     const int64_t *__restrict__ tptr, const int32_t *__restrict__ tidx,
                                                     double *__restrict__ per_query)
{
    const int64_t q = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= m) return;
    const int64_t t0 = tptr[q], t1 = tptr[q + 1];
    int hits = 0;
    if (t1 > t0)
        for (int r = lane; r < k; r += 32) {
            const int32_t id = ids[q * k_stride + r];
            if (id < 0) continue;
            int64_t lo = t0, hi = t1;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                const int32_t v = tidx[mid];
                if (v == id) { ++hits; break; }
                if (v < id) lo = mid + 1; else hi = mid;
            }
        }
    hits = __reduce_add_sync(0xFFFFFFFFu, hits);
    if (lane == 0) per_query[q] = t1 > t0 ? (double)hits / (double)(t1 - t0) : -1.0;
}

// sum and count of the non-negative entries, in an order that depends on m only (one block)
__global__ void __launch_bounds__(1024) k_recall_mean(const double *__restrict__ per_query, int64_t m, double *__restrict__ out)
{
    __shared__ double ssum[1024];
    __shared__ long long scnt[1024];
    double s = 0.0;
    long long c = 0;
    for (int64_t q = threadIdx.x; q < m; q += 1024) {
        const double v = per_query[q];
        if (v >= 0.0) { s += v; ++c; }
    }
    ssum[threadIdx.x] = s;
    scnt[threadIdx.x] = c;
    __syncthreads();
    for (int h = 512; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) { ssum[threadIdx.x] += ssum[threadIdx.x + h]; scnt[threadIdx.x] += scnt[threadIdx.x + h]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) { out[0] = ssum[0]; out[1] = (double)scnt[0]; }
}

}  // namespace

cudaError_t launch_recall(const int32_t *ids, int64_t m, int k_stride, int k, const int64_t *tptr, const int32_t *tidx,
                          double *per_query, double *out2, cudaStream_t s, int64_t *launches)
{
    if (m > 0) {
        k_recall_rows<<<(unsigned)((m + 7) / 8), 256, 0, s>>>(ids, m, k_stride, k, tptr, tidx, per_query);
        ++*launches;
    }
    k_recall_mean<<<1, 1024, 0, s>>>(per_query, m, out2);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace alx
