// Exact Top-K scoring on the tensor cores (Sec. 4.6) for d = 128 and bfloat16 tables.
//
// A block takes 128 queries and a slab of items.  The fp32 queries are split beforehand into three bfloat16 parts
// (q = q1 + q2 + q3 to 2^-24), so that every product is an exact product of bfloat16 values and the fp32 sums carry
// the query to fp32 accuracy.  Per tile of 256 items the MMA thread issues 3 parts x 8 K-steps of tcgen05.mma
// (128 x 256 x 16) into one of two tensor-memory accumulators (all 512 columns); the eight selection warps read the other
// one, a thread per query (= accumulator lane) and half of the columns, and append the scores that reach the query's threshold
// to one of its two lists (alx_topk.cuh).
//
//   warp 9     TMA: the three query tiles once, then the item tiles through a two-stage ring
//              (2D tile loads, 128-byte swizzle, K-major: a row of the table is a row of the operand)
//   warp 8     MMA issue (one thread)
//   warps 0-7  selection; an accumulator is handed back when all of them have read it.  Each reads 32 columns ahead of the
//              ones it looks at: with four warps and no read-ahead the selection took 7400 cycles a tile, twice the products
//
// Bound: the tensor pipe (24 x 128 cycles of products per tile; operand reads from shared memory: 12 KB per product, which
// is why the tile is 256 items wide -- at 128 the reads, 8 KB per 64 cycles of products, were the limit).  2048 queries x 1M
// items, k = 50, exclusion lists of 30: 1.06 ms over the phases (22 ms with lists kept sorted in shared memory).
//
// Every wait is bounded; a wait that gives up sets the block's abort flag, the roles leave their loops and the
// status word reports a timeout.
#include "alx_common.cuh"
#include "alx_ptx.cuh"
#include "alx_topk.cuh"

#include <cuda.h>
#include <cuda_bf16.h>

namespace alx {

using namespace ptx;

namespace {

constexpr int kD = 128;
constexpr int kTileItems = 256;
constexpr int kStages = 2;
constexpr int kQueryHalfBytes = kTopkQueries * 128;      // 128 rows x 64 bfloat16
constexpr int kItemHalfBytes = kTileItems * 128;
constexpr int kSelWarps = 8;
constexpr int kThreads = (kSelWarps + 2) * 32;
static_assert(kTileItems <= kTopkTile, "a tile's items fit a candidate buffer");

struct __align__(1024) TopkSmem {
    unsigned char q[3][2][kQueryHalfBytes];            // [part][feature half]: 128 queries x 64 features, swizzled
    unsigned char h[kStages][2][kItemHalfBytes];       // item tiles
    uint64_t q_full, full[kStages], empty[kStages], acc_full[2], acc_empty[2];
    uint32_t tmem_base;
    int abort_flag;
};

static_assert(sizeof(TopkSmem) + 1024 <= 232448, "shared memory of the Top-K kernel");

// 32 lanes x 32 consecutive columns, thread t of the warp gets lane (base lane + t): the load, and the wait for it, through which
// the registers are passed so that no use of them can be scheduled before it
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, float (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
          "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]),
          "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]), "=f"(v[24]),
          "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld32_wait(float (&v)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]),
                   "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]), "+f"(v[16]),
                   "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]), "+f"(v[23]), "+f"(v[24]),
                   "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28])
                 :
                 : "memory");
    asm volatile("" : "+f"(v[29]), "+f"(v[30]), "+f"(v[31])::"memory");
}

// one column of 32 lanes
__device__ __forceinline__ float tmem_ld1(uint32_t taddr)
{
    float v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;" : "=f"(v) : "r"(taddr) : "memory");
    return v;
}

// bf16 operands, fp32 accumulator, both operands K-major: D (+)= A * B^T
__host__ __device__ constexpr uint32_t idesc_bf16_k_major(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// fp32 queries -> three bfloat16 parts, [part][m_pad][128]; rows m .. m_pad - 1 are zero
__global__ void __launch_bounds__(256) k_split_queries(const float *__restrict__ Q, int64_t m, int64_t m_pad,
                                                       __nv_bfloat16 *__restrict__ P)
{
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= m_pad * kD) return;
    const float x = e < m * kD ? Q[e] : 0.f;
    const __nv_bfloat16 p1 = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(p1);
    const __nv_bfloat16 p2 = __float2bfloat16_rn(r1);
    const __nv_bfloat16 p3 = __float2bfloat16_rn(r1 - __bfloat162float(p2));
    P[e] = p1;
    P[m_pad * kD + e] = p2;
    P[2 * m_pad * kD + e] = p3;
}

__global__ void __launch_bounds__(kThreads, 1)
k_topk_umma(const __grid_constant__ CUtensorMap tmap_h, const __grid_constant__ CUtensorMap tmap_q, int64_t i_begin, int64_t i_end,
            int64_t m, int64_t m_pad, int k, int cap, const int64_t *__restrict__ ex_ptr, const int32_t *__restrict__ ex_idx, int64_t slab,
            uint64_t *lists, int32_t *__restrict__ list_cnt, const unsigned *__restrict__ gtau, DevStatus *st)
{
    extern __shared__ unsigned char smem_raw[];
    TopkSmem &sm = *reinterpret_cast<TopkSmem *>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t i0 = i_begin + (int64_t)blockIdx.y * slab;
    const int64_t i1 = i0 + slab < i_end ? i0 + slab : i_end;
    const int n_tiles = i1 > i0 ? (int)((i1 - i0 + kTileItems - 1) / kTileItems) : 0;
    if (tid == 0) {
        mbar_init(&sm.q_full, 1);
        for (int s = 0; s < kStages; ++s) { mbar_init(&sm.full[s], 1); mbar_init(&sm.empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&sm.acc_full[a], 1); mbar_init(&sm.acc_empty[a], kSelWarps); }
        sm.abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == kSelWarps) {
        tmem_alloc(&sm.tmem_base, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (warp == kSelWarps + 1) {
        if (lane == 0 && n_tiles > 0) {
            mbar_arrive_expect_tx(&sm.q_full, 3 * 2 * kQueryHalfBytes);
            for (int part = 0; part < 3; ++part)
                for (int half = 0; half < 2; ++half)
                    tma_tile_2d(smem_u32(&sm.q[part][half][0]), &tmap_q, 64 * half,
                                (int)(part * m_pad + (int64_t)blockIdx.x * kTopkQueries), &sm.q_full);
            for (int t = 0; t < n_tiles; ++t) {
                const int s = t % kStages;
                if (t >= kStages && !mbar_wait_parked(&sm.empty[s], (uint32_t)((t / kStages - 1) & 1), &sm.abort_flag, 71)) break;
                mbar_arrive_expect_tx(&sm.full[s], 2 * kItemHalfBytes);
                for (int half = 0; half < 2; ++half)
                    tma_tile_2d(smem_u32(&sm.h[s][half][0]), &tmap_h, 64 * half, (int)(i0 + (int64_t)t * kTileItems), &sm.full[s]);
            }
        }
    } else if (warp == kSelWarps) {
        if (lane == 0 && n_tiles > 0) {
            constexpr uint32_t kIdesc = idesc_bf16_k_major(128, kTileItems);
            bool ok = mbar_wait_parked(&sm.q_full, 0, &sm.abort_flag, 72);
            for (int t = 0; ok && t < n_tiles; ++t) {
                const int s = t % kStages, a = t & 1;
                ok = mbar_wait_parked(&sm.full[s], (uint32_t)((t / kStages) & 1), &sm.abort_flag, 73);
                if (ok && t >= 2) ok = mbar_wait_parked(&sm.acc_empty[a], (uint32_t)((t / 2 - 1) & 1), &sm.abort_flag, 74);
                if (!ok) break;
                tc_fence_after();
                const uint32_t dcol = sm.tmem_base + (uint32_t)(a * kTileItems);
                bool first = true;
                for (int half = 0; half < 2; ++half)
                    for (int ks = 0; ks < 4; ++ks) {
                        // K-major, 128-byte swizzle: 8-row groups 1024 bytes apart; a K step is 32 bytes along the row
                        const uint64_t bdesc = smem_desc(smem_u32(&sm.h[s][half][0]) + ks * 32, 16, 1024, 2);
                        for (int part = 0; part < 3; ++part) {
                            const uint64_t adesc = smem_desc(smem_u32(&sm.q[part][half][0]) + ks * 32, 16, 1024, 2);
                            umma_f16(dcol, adesc, bdesc, kIdesc, !first);
                            first = false;
                        }
                    }
                umma_commit(&sm.empty[s]);        // the stage may be refilled once these MMAs have read it
                umma_commit(&sm.acc_full[a]);
            }
        }
    } else {
        // selection: thread = query = accumulator lane and half of the columns, whose items it meets in ascending id
        const int sub = warp & 3, half = warp >> 2;
        const int64_t q = (int64_t)blockIdx.x * kTopkQueries + sub * 32 + lane;
        const bool live = q < m;
        const int64_t list = (int64_t)blockIdx.y * kTopkListsPerSlab + half;
        // lists of a block's queries are interleaved: entry p of query r at p * 128 + r
        uint64_t *block_lists = lists + (list * gridDim.x + blockIdx.x) * cap * kTopkQueries;
        uint64_t *mine = block_lists + sub * 32 + lane;
        uint64_t *next = mine;      // where the next entry goes
        int checked = 0;
        const unsigned g = live ? gtau[q] : 0u;
        float thr = !live ? INFINITY : g ? order_score(g) : -INFINITY;
        // 32 columns of the accumulator.  The usual case ends at the vote; a column that some query of the warp wants is read
        // again by itself.  (Appending from the 32 registers takes 32 copies of the append: with those the warps waited for
        // instructions three quarters of the time.)
        auto look = [&](const float (&v)[32], uint32_t taddr, int left, int64_t base) {
            float top = v[0];
#pragma unroll
            for (int j = 1; j < 32; ++j) top = fmaxf(top, v[j]);
            if (!__any_sync(0xFFFFFFFFu, top >= thr)) return;
            unsigned want = 0;
#pragma unroll
            for (int j = 0; j < 32; ++j) want |= v[j] >= thr ? 1u << j : 0u;
            if (left < 32) want &= left > 0 ? (1u << left) - 1u : 0u;
            unsigned any = __reduce_or_sync(0xFFFFFFFFu, want);
            while (any) {
                const int j = __ffs(any) - 1;
                any &= any - 1;
                const float x = tmem_ld1(taddr + j);
                if (want >> j & 1u) {
                    *next = topk_key(x, (int32_t)(base + j));
                    next += kTopkQueries;
                }
            }
        };
        for (int t = 0; t < n_tiles; ++t) {
            const int a = t & 1;
            if (!mbar_wait_parked_warp(&sm.acc_full[a], (uint32_t)((t / 2) & 1), &sm.abort_flag, 75)) break;
            tc_fence_after();
            const int c0 = half * (kTileItems / 2);
            const uint32_t trow = sm.tmem_base + ((uint32_t)(sub * 32) << 16) + (uint32_t)(a * kTileItems + c0);
            const int64_t base = i0 + (int64_t)t * kTileItems + c0;
            const int lim = i1 - base < kTileItems ? (int)(i1 - base) : kTileItems;
            float v0[32], v1[32];
            tmem_ld32_issue(trow, v0);
#pragma unroll 1
            for (int c = 0; c < kTileItems / 2; c += 64) {
                tmem_ld32_wait(v0);
                tmem_ld32_issue(trow + c + 32, v1);
                look(v0, trow + c, lim - c, base + c);
                tmem_ld32_wait(v1);
                if (c + 64 < kTileItems / 2) tmem_ld32_issue(trow + c + 64, v0);
                look(v1, trow + c + 32, lim - c - 32, base + c + 32);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.acc_empty[a]);
            const int cnt = (int)(next - mine) / kTopkQueries;
            // lists that could overflow in the next tile: the warp works on one at a time
            unsigned todo = __ballot_sync(0xFFFFFFFFu, cnt > cap - kTileItems / 2);
            while (todo) {
                const int owner = __ffs(todo) - 1;
                todo &= todo - 1;
                uint32_t tau = 0;
                const int kept = warp_keep_best(block_lists + sub * 32 + owner, kTopkQueries, __shfl_sync(0xFFFFFFFFu, cnt, owner), k,
                                                __shfl_sync(0xFFFFFFFFu, checked, owner), ex_ptr, ex_idx,
                                                (int64_t)blockIdx.x * kTopkQueries + sub * 32 + owner, &tau);
                if (lane == owner) {
                    checked = kept;      // later items have larger ids: strictly better ones only
                    next = mine + (int64_t)kept * kTopkQueries;
                    if (kept >= k) thr = fmaxf(thr, next_above(order_score(tau)));
                }
            }
        }
        if (live) list_cnt[list * m + q] = (int)(next - mine) / kTopkQueries;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kSelWarps) {
        tc_fence_after();
        tmem_dealloc(sm.tmem_base, 512);
    }
    if (tid == 0 && sm.abort_flag) raise_flag(st, kFlagTimeout, (long long)sm.abort_flag * 1000000 + blockIdx.x);
}

// 2D bfloat16 tensor [rows x 128], box 64 features x box_rows rows, 128-byte swizzle; rows past the extent read as zeros
cudaError_t tile_tensor_map(const void *X, int64_t rows, int box_rows, CUtensorMap *tm)
{
    typedef CUresult (*Encode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                               const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static Encode encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult qr;
        cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qr);
        if (e != cudaSuccess) return e;
        if (qr != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<Encode>(fn);
    }
    const cuuint64_t dims[2] = {(cuuint64_t)kD, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)kD * sizeof(__nv_bfloat16)};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(X), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int64_t padded_queries(int64_t m) { return (m + kTopkQueries - 1) / kTopkQueries * kTopkQueries; }

}  // namespace

int64_t topk_query_scratch_bytes(int64_t m) { return 3 * padded_queries(m) * kD * (int64_t)sizeof(__nv_bfloat16); }

cudaError_t topk_umma_prepare(const void *H, int64_t n_items, const float *Q, int64_t m, void *scratch_q, TopkUmma *out, cudaStream_t s,
                              int64_t *launches)
{
    out->m_pad = padded_queries(m);
    __nv_bfloat16 *P = static_cast<__nv_bfloat16 *>(scratch_q);
    k_split_queries<<<(unsigned)((out->m_pad * kD + 255) / 256), 256, 0, s>>>(Q, m, out->m_pad, P);
    ++*launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if ((e = tile_tensor_map(H, n_items, kTileItems, &out->items)) != cudaSuccess) return e;
    return tile_tensor_map(P, 3 * out->m_pad, kTopkQueries, &out->queries);
}

cudaError_t launch_topk_umma(const TopkUmma &u, int64_t i_begin, int64_t i_end, int64_t m, int k, int cap, const int64_t *ex_ptr,
                             const int32_t *ex_idx, int slabs, int64_t slab, uint64_t *lists, int32_t *list_cnt, const unsigned *gtau,
                             DevStatus *st, cudaStream_t s)
{
    const size_t smem = sizeof(TopkSmem) + 1024;
    static SmemOnce allow;
    const cudaError_t e = allow(k_topk_umma, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)(u.m_pad / kTopkQueries), (unsigned)slabs);
    k_topk_umma<<<grid, kThreads, smem, s>>>(u.items, u.queries, i_begin, i_end, m, u.m_pad, k, cap, ex_ptr, ex_idx, slab, lists,
                                             list_cnt, gtau, st);
    return cudaGetLastError();
}

}  // namespace alx
