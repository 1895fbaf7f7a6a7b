// Selection shared by the Top-K scoring kernels (alx_topk.cu, alx_topk_umma.cu).
//
// The order is total: score descending, then id ascending.  A candidate is one 64-bit key, larger = better:
// the score's bits made monotone in the upper half, the complement of the id in the lower half.
//
// The items are taken in phases (topk_plan): a first one of a few thousand items sets every query's k-th best so far, which is
// the threshold of the next, longer phase, and so on.  In a phase a scoring block scans a slab of items in ascending id and
// appends, per query, every item that reaches the threshold to a list of its own in global memory; k_topk_merge cuts the lists
// of a phase to the k best that are not excluded.  A phase is so long that a list is expected to get about kTopkExpect
// items; a list that could overflow all the same (items in an unlucky order) is cut back where it stands, by one warp
// (warp_keep_best).  Sorted lists kept while scanning used to cost one shifting insertion per improvement, up to 1700 cycles
// each with an exclusion list; an append is a store, and exclusion lists are looked at only where lists are cut.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "alx_common.cuh"

namespace alx {

constexpr int kTopkQueries = 128;      // queries per block of the tensor-core scoring kernel
constexpr int kTopkTile = 256;         // no scoring kernel takes more items per step
constexpr int kTopkSlack = 128;        // appends beyond that before a buffer is cut back again
constexpr int kTopkMaxLaneKeys = 20;   // (256 + kTopkTile + kTopkSlack) / 32

// elements of one query's candidate buffer
__host__ __device__ inline int topk_cap(int k) { return (k + 31) / 32 * 32 + kTopkTile + kTopkSlack; }
constexpr int kTopkExpect = 96;        // appends per list a phase is planned for

constexpr int kTopkMostSlabs = 512;
constexpr int64_t kTopkTotal = 2304;       // candidates per query a phase is planned for (k_topk_merge takes 4096 keys at once)
constexpr int64_t kTopkOnePhase = 16384;   // up to this many items one phase does: its lists are short enough to merge

// the tensor-core scoring kernel (alx_topk_umma.cu; d = 128, bfloat16 table): operands of one batch of queries, then one
// launch per phase; a block keeps two lists per query and slab
constexpr int kTopkListsPerSlab = 2;
struct TopkUmma {
    CUtensorMap items, queries;
    int64_t m_pad;
};
int64_t topk_query_scratch_bytes(int64_t m);      // for the queries' bfloat16 parts
cudaError_t topk_umma_prepare(const void *H, int64_t n_items, const float *Q, int64_t m, void *scratch_q, TopkUmma *out, cudaStream_t s,
                              int64_t *launches);
cudaError_t launch_topk_umma(const TopkUmma &u, int64_t i_begin, int64_t i_end, int64_t m, int k, int cap, const int64_t *ex_ptr,
                             const int32_t *ex_idx, int slabs, int64_t slab, uint64_t *lists, int32_t *list_cnt, const unsigned *gtau,
                             DevStatus *st, cudaStream_t s);

__device__ __forceinline__ uint32_t score_order(float v)
{
    const uint32_t b = __float_as_uint(v + 0.f);      // (-0 becomes +0: they are equal scores)
    return b ^ ((b >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
__device__ __forceinline__ float order_score(uint32_t u)
{
    return __uint_as_float(u ^ ((u >> 31) ? 0x80000000u : 0xFFFFFFFFu));
}
__device__ __forceinline__ uint64_t topk_key(float v, int32_t id) { return ((uint64_t)score_order(v) << 32) | (uint32_t)~id; }
__device__ __forceinline__ int32_t key_id(uint64_t key) { return (int32_t)~(uint32_t)key; }
// the smallest score above v (v itself if there is none)
__device__ __forceinline__ float next_above(float v) { return v < INFINITY ? order_score(score_order(v) + 1u) : v; }

__device__ __forceinline__ bool excluded(const int64_t *__restrict__ ex_ptr, const int32_t *__restrict__ ex_idx, int64_t q,
                                         int32_t id)
{
    if (!ex_ptr) return false;
    int64_t lo = ex_ptr[q], hi = ex_ptr[q + 1];
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        const int32_t v = ex_idx[mid];
        if (v == id) return true;
        if (v < id) lo = mid + 1; else hi = mid;
    }
    return false;
}

// A point of (lo, hi], lo < hi: halfway between the scores at first, halfway between their bit patterns later (which ends any
// bisection within 32 further steps; halving the scores gets close in a handful of steps, the bit patterns of small scores of
// both signs are far apart)
__device__ __forceinline__ uint32_t bisect_at(uint32_t lo, uint32_t hi, int step)
{
    if (step < 12) {
        const float a = order_score(lo), b = order_score(hi);
        const uint32_t mid = score_order(a + 0.5f * (b - a));
        if (mid > lo && mid <= hi) return mid;      // (not so for infinite scores, or where rounding leaves the range)
    }
    return lo + (hi - lo) / 2 + 1;
}

// A cut keeps at least the k best and at most this many
__host__ __device__ inline int topk_kept_most(int k) { return k + k / 4 + 8; }

// One warp cuts a list of cnt keys, `stride` apart (cnt <= 32 * kTopkMaxLaneKeys) back to k .. topk_kept_most(k) of its best that are not
// excluded, in any order (all of them if there are fewer); the first `checked` keys are known not to be excluded.  Returns the
// new count (to every lane); where that is at least k, *tau_order receives the least score kept.  The bar is found by
// bisection between the least and the largest score (per-lane compares and one warp sum per step), which stops as soon as
// the count is in the range; scores equal to the k-th beyond the range are told apart by their ids.
__device__ __forceinline__ int warp_keep_best(uint64_t *buf, int stride, int cnt, int k, int checked, const int64_t *__restrict__ ex_ptr,
                                              const int32_t *__restrict__ ex_idx, int64_t q, uint32_t *tau_order)
{
    const int lane = threadIdx.x & 31;
    const int most = topk_kept_most(k);
    uint64_t e[kTopkMaxLaneKeys];
#pragma unroll
    for (int j = 0; j < kTopkMaxLaneKeys; ++j) {
        const int p = 32 * j + lane;
        e[j] = p < cnt ? buf[(int64_t)p * stride] : 0;
    }
    if (ex_ptr) {      // the lane's bisections in lockstep: their loads are independent
        const int64_t x0 = ex_ptr[q];
        const int len = (int)(ex_ptr[q + 1] - x0);
        const int32_t *x = ex_idx + x0;
        if (len > 0) {
            int at[kTopkMaxLaneKeys];      // last position whose id is <= the key's (or 0)
#pragma unroll
            for (int j = 0; j < kTopkMaxLaneKeys; ++j) at[j] = 0;
            for (int step = 1 << (31 - __clz(len)); step > 0; step >>= 1) {
#pragma unroll
                for (int j = 0; j < kTopkMaxLaneKeys; ++j) {
                    const int p = at[j] + step;
                    if (32 * j < cnt && p < len && x[p] <= key_id(e[j])) at[j] = p;
                }
            }
#pragma unroll
            for (int j = 0; j < kTopkMaxLaneKeys; ++j)
                if (32 * j < cnt && 32 * j + lane >= checked && x[at[j]] == key_id(e[j])) e[j] = 0;
        }
    }
    int mine = 0;
    uint32_t lo = 0xFFFFFFFFu, hi = 0;
#pragma unroll
    for (int j = 0; j < kTopkMaxLaneKeys; ++j) {
        const uint32_t s = (uint32_t)(e[j] >> 32);
        if (e[j]) { ++mine; lo = s < lo ? s : lo; hi = s > hi ? s : hi; }
    }
    const int n = __reduce_add_sync(0xFFFFFFFFu, mine);
    uint64_t bar = 1;      // keep keys >= bar
    if (n > most) {
        lo = __reduce_min_sync(0xFFFFFFFFu, lo);      // n keys reach lo: at least k
        hi = __reduce_max_sync(0xFFFFFFFFu, hi);      // fewer than k exceed hi: none does
        int at_lo = n;
        for (int step = 0; at_lo > most && lo < hi; ++step) {
            const uint32_t mid = bisect_at(lo, hi, step);
            int c = 0;
#pragma unroll
            for (int j = 0; j < kTopkMaxLaneKeys; ++j)
                if (32 * j < cnt) c += (uint32_t)(e[j] >> 32) >= mid;
            c = __reduce_add_sync(0xFFFFFFFFu, c);
            if (c >= k) { lo = mid; at_lo = c; } else hi = mid - 1;
        }
        bar = (uint64_t)lo << 32;
        if (at_lo > most) {      // lo is the k-th's own score, and too many equal it: the smaller ids of those
            uint32_t u = 0;
            for (int bit = 31; bit >= 0 && at_lo > most; --bit) {
                const uint64_t cand = bar | u | (1u << bit);
                int c = 0;
#pragma unroll
                for (int j = 0; j < kTopkMaxLaneKeys; ++j)
                    if (32 * j < cnt) c += e[j] >= cand;
                c = __reduce_add_sync(0xFFFFFFFFu, c);
                if (c >= k) { u |= 1u << bit; at_lo = c; }
            }
            bar |= u;
        }
    }
    // every lane holds its keys: write the survivors back to the front
    int kept = 0;
    uint32_t least = 0xFFFFFFFFu;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kTopkMaxLaneKeys; ++j) {
        if (32 * j >= cnt) break;
        const bool keep = e[j] >= bar;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, keep);
        if (keep) {
            buf[(int64_t)(kept + __popc(m & ((1u << lane) - 1u))) * stride] = e[j];
            const uint32_t s = (uint32_t)(e[j] >> 32);
            least = s < least ? s : least;
        }
        kept += __popc(m);
    }
    if (kept >= k) *tau_order = __reduce_min_sync(0xFFFFFFFFu, least);
    __syncwarp();
    return kept;
}

}  // namespace alx
