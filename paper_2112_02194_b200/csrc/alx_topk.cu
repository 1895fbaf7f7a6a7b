// Exact Top-K of <q, h_i> over every row of a table (Sec. 4.6; the protocol of Sec. 5).  Every item is scored and every score
// is looked at; the order is total (score descending, then id ascending), so the result does not depend on how the items
// are divided among thread blocks.  The selection is described in alx_topk.cuh.
//
// Scoring kernels:
//   k_topk_fma     any d, either storage type: fp32 FMAs on tiles of items and queries staged in shared memory
//   k_topk_umma    d = 128, bfloat16 tables, more than kFmaQueries queries (alx_topk_umma.cu): tcgen05
// and k_topk_merge, a block per query, over the slabs' candidates.
#include "alx_common.cuh"
#include "alx_ptx.cuh"
#include "alx_topk.cuh"

namespace alx {

namespace {

constexpr int kFmaThreads = 256;
constexpr int kFmaStages = 3;

// Up to this many queries the FMA kernel is the faster one on bfloat16 tables of 128 features too: it is bound by reading
// the table (1M items: 256 MB), the tensor-core kernel by the 24 products of a tile, which cost the same for 1 query and 128.
constexpr int kFmaQueries = 16;

// Tile geometry for QT queries per block.  A thread owns 4 queries x TI items; the queries of a thread are QG apart and its
// items IG apart, so that the 16-byte reads of a warp touch every bank once (rows are padded by 16 bytes).
template <int D, typename T, int QT> struct FmaGeo {
    static constexpr int TQ = 4, QG = QT / TQ, IG = kFmaThreads / QG;
    static constexpr int TI = QT >= 64 ? 8 : QT / 4;
    static constexpr int WQ = QG < 4 ? QG : 4, WI = 32 / WQ;     // a warp's lanes: WI item groups x WQ query groups
    static constexpr int ITEMS = IG * TI;                        // items per tile
    static constexpr int FC = D * (int)sizeof(T) < 128 ? D : 128 / (int)sizeof(T);      // features per pipeline step: whole lines
    static constexpr int NC = D / FC;
    static constexpr int ROW = FC * (int)sizeof(T) + 16;         // bytes between the rows of a staged tile
    static constexpr int PIECES = FC * (int)sizeof(T) / 16;      // 16-byte pieces per row
    static constexpr int STAGE = ITEMS * ROW;
    static constexpr int QROW = D + 4;
    static constexpr size_t SMEM = (size_t)kFmaStages * STAGE + sizeof(float) * QT * QROW;
};

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// Grid (query tiles, slabs).  Pipeline of (tile, 128-byte piece of the rows) steps through three stages of cp.async; two features share
// a packed FMA (even and odd features in separate sums).  Bound: reading the table for few queries, the FMA pipe otherwise.
// 300 queries x 300k fp32 items of 64 features, k = 50: 0.37 ms over the phases (31 TFLOP/s; a thread per query with the query
// in registers and a sorted list in global memory took 9.6 ms); 3 queries x 1M bfloat16 items of 128: 5 TB/s in the last phase.
template <int D, typename T, int QT>
__global__ void __launch_bounds__(kFmaThreads, 2)
k_topk_fma(const T *__restrict__ H, int64_t i_begin, int64_t i_end, const float *__restrict__ Q, int64_t m, int k, int cap,
           const int64_t *__restrict__ ex_ptr, const int32_t *__restrict__ ex_idx, int64_t slab, uint64_t *lists,
           int32_t *__restrict__ list_cnt, const unsigned *__restrict__ gtau)
{
    using G = FmaGeo<D, T, QT>;
    constexpr int EL = 16 / (int)sizeof(T);      // features per 16-byte piece
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *qs = reinterpret_cast<float *>(smem_raw + kFmaStages * G::STAGE);
    __shared__ float thr_s[QT];
    __shared__ int cnt_s[QT], checked_s[QT];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ig = warp % (G::IG / G::WI) * G::WI + lane % G::WI, qg = warp / (G::IG / G::WI) * G::WQ + lane / G::WI;
    const int64_t q0 = (int64_t)blockIdx.x * QT;
    const int64_t i0 = i_begin + (int64_t)blockIdx.y * slab;
    const int64_t i1 = i0 + slab < i_end ? i0 + slab : i_end;
    const int n_tiles = i1 > i0 ? (int)((i1 - i0 + G::ITEMS - 1) / G::ITEMS) : 0;
    const int n_steps = n_tiles * G::NC;
    uint64_t *lists_q = lists + ((int64_t)blockIdx.y * m + q0) * cap;

    auto load_step = [&](int step) {
        const int64_t base = i0 + (int64_t)(step / G::NC) * G::ITEMS;
        const int f0 = (step % G::NC) * G::FC;
        const uint32_t dst = ptx::smem_u32(smem_raw) + (uint32_t)(step % kFmaStages) * G::STAGE;
#pragma unroll
        for (int p = tid; p < G::ITEMS * G::PIECES; p += kFmaThreads) {
            const int r = p / G::PIECES, c = p % G::PIECES;
            const bool in = base + r < i1;
            cp_async16_zfill(dst + r * G::ROW + c * 16, H + (in ? base + r : i0) * D + f0 + c * EL, in);
        }
    };
#pragma unroll
    for (int s = 0; s < kFmaStages - 1; ++s) {
        if (s < n_steps) load_step(s);
        ptx::cp_async_commit();
    }
    for (int e = tid; e < QT * D; e += kFmaThreads) {
        const int r = e / D;
        qs[r * G::QROW + e % D] = q0 + r < m ? Q[(q0 + r) * D + e % D] : 0.f;
    }
    if (tid < QT) {
        const unsigned g = q0 + tid < m ? gtau[q0 + tid] : 0u;
        thr_s[tid] = q0 + tid >= m ? INFINITY : g ? order_score(g) : -INFINITY;
        cnt_s[tid] = checked_s[tid] = 0;
    }

    float2 acc[G::TI][G::TQ];
#pragma unroll
    for (int i = 0; i < G::TI; ++i)
#pragma unroll
        for (int a = 0; a < G::TQ; ++a) acc[i][a] = make_float2(0.f, 0.f);

    auto cut_back = [&]() {      // every warp takes queries in turn
        for (int q = warp; q < QT; q += kFmaThreads / 32) {
            const int cnt = cnt_s[q];
            if (cnt <= cap - G::ITEMS) continue;
            uint32_t tau = 0;
            const int kept = warp_keep_best(lists_q + (int64_t)q * cap, 1, cnt, k, checked_s[q], ex_ptr, ex_idx, q0 + q, &tau);
            if (lane == 0) {
                cnt_s[q] = checked_s[q] = kept;      // later items have larger ids: strictly better ones only
                if (kept >= k) thr_s[q] = fmaxf(thr_s[q], next_above(order_score(tau)));
            }
        }
    };

    for (int step = 0; step < n_steps; ++step) {
        ptx::cp_async_wait<kFmaStages - 2>();
        __syncthreads();
        if (step + kFmaStages - 1 < n_steps) load_step(step + kFmaStages - 1);
        ptx::cp_async_commit();
        const unsigned char *tile = smem_raw + (step % kFmaStages) * G::STAGE + ig * G::ROW;
        const int chunk = step % G::NC;
        const float *qp = qs + qg * G::QROW + chunk * G::FC;
#pragma unroll
        for (int c = 0; c < G::PIECES; ++c) {
            float2 qv[G::TQ][EL / 2];
#pragma unroll
            for (int a = 0; a < G::TQ; ++a)
#pragma unroll
                for (int h = 0; h < EL / 4; ++h) {
                    const float4 v = *reinterpret_cast<const float4 *>(qp + a * G::QG * G::QROW + c * EL + 4 * h);
                    qv[a][2 * h] = make_float2(v.x, v.y);
                    qv[a][2 * h + 1] = make_float2(v.z, v.w);
                }
#pragma unroll
            for (int i = 0; i < G::TI; ++i) {
                const uint4 w = *reinterpret_cast<const uint4 *>(tile + i * G::IG * G::ROW + c * 16);
                const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
                float2 h[EL / 2];
                if constexpr (EL == 4) {
                    h[0] = make_float2(__uint_as_float(ww[0]), __uint_as_float(ww[1]));
                    h[1] = make_float2(__uint_as_float(ww[2]), __uint_as_float(ww[3]));
                } else {
#pragma unroll
                    for (int j = 0; j < EL / 2; ++j)
                        h[j] = make_float2(__uint_as_float(ww[j & 3] << 16), __uint_as_float(ww[j & 3] & 0xFFFF0000u));
                }
#pragma unroll
                for (int j = 0; j < EL / 2; ++j)
#pragma unroll
                    for (int a = 0; a < G::TQ; ++a) acc[i][a] = __ffma2_rn(h[j], qv[a][j], acc[i][a]);
            }
        }
        if (chunk == G::NC - 1) {
            const int t = step / G::NC;
            const int64_t base = i0 + (int64_t)t * G::ITEMS + ig;
#pragma unroll
            for (int a = 0; a < G::TQ; ++a) {
                const int q = qg + G::QG * a;
                const float thr = thr_s[q];
                float v[G::TI], vmax = -INFINITY;
#pragma unroll
                for (int i = 0; i < G::TI; ++i) {
                    v[i] = acc[i][a].x + acc[i][a].y;
                    vmax = fmaxf(vmax, v[i]);
                    acc[i][a] = make_float2(0.f, 0.f);
                }
                if (vmax >= thr) {
#pragma unroll
                    for (int i = 0; i < G::TI; ++i) {
                        const int64_t item = base + i * G::IG;
                        if (v[i] >= thr && item < i1)
                            lists_q[(int64_t)q * cap + atomicAdd(&cnt_s[q], 1)] = topk_key(v[i], (int32_t)item);
                    }
                }
            }
            __syncthreads();
            if (__syncthreads_or(tid < QT && cnt_s[tid] > cap - G::ITEMS)) {
                cut_back();
                __syncthreads();
            }
        }
    }
    ptx::cp_async_wait<0>();
    __syncthreads();
    if (tid < QT && q0 + tid < m) list_cnt[(int64_t)blockIdx.y * m + q0 + tid] = cnt_s[tid];
}

// ---- merge -------------------------------------------------------------------------------------------------------------
constexpr int kMergeThreads = 512;
constexpr int kMergeExcluded = 1024;      // exclusion lists up to this length are searched in shared memory
constexpr int kMergeKeys = 4096;
constexpr int kMergePer = kMergeKeys / kMergeThreads;
constexpr int kMergeBins = 2048;
constexpr int kMergeLists = kTopkMostSlabs * kTopkListsPerSlab;      // no phase has more lists per query

// A block per query, after each phase: the phase's candidates and the k best of the phases before (carry), without the
// excluded ids and those below the threshold the phase started from, are cut to the k best -- a histogram of the scores finds
// the bin of the k-th, then bisection as in warp_keep_best (here with block-wide counts) has the few steps within it left.  `last`: they are ranked by counting and written out; otherwise they are
// carried on and the k-th score becomes the next phase's threshold.  Lists in groups, so that any number of candidates fits.
// (The lists of query q: entry p of list l at ((l * query blocks + q / qb) * cap + p) * qb + q % qb, qb queries interleaved.)
// Bound: latency.  The counts of all lists are one load, scanned; then every candidate of the group has a thread's register,
// whose loads are all in flight together (a warp per list, list after list, took 23 us for 3 queries and now 7 to 11,
// 71 us for 2048 and now 52 to 71: there it is bound by the 32-byte sectors of the interleaved lists).
__global__ void __launch_bounds__(kMergeThreads, 3) k_topk_merge(const uint64_t *__restrict__ lists, const int32_t *__restrict__ list_cnt,
                                                              unsigned *gtau, uint64_t *carry, int first, int last, int64_t m, int k,
                                                              int cap, int n_lists, int qb, const int64_t *__restrict__ ex_ptr,
                                                              const int32_t *__restrict__ ex_idx, int32_t *__restrict__ ids_out,
                                                              float *__restrict__ scores_out)
{
    __shared__ uint64_t best[kMergeThreads];          // the k best so far, in any order (0: none)
    __shared__ int start_s[kMergeLists + 1];          // candidates of the lists before
    __shared__ uint16_t list_s[kMergeKeys];           // the list that a candidate of the group is on
    __shared__ int n_s, cnt_s[2][kMergeThreads / 32], max_s[2][kMergeThreads / 32];
    __shared__ int32_t ex_s[kMergeExcluded];
    __shared__ int hist[kMergeBins], bin_s, bin_above;
    __shared__ uint32_t bin_lo, bin_hi;
    __shared__ uint32_t ex_bits[kMergeThreads];       // a bit per excluded id (by its low bits): most candidates need no search
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t q = blockIdx.x;
    const uint64_t thr = (uint64_t)gtau[q] << 32;
    const int64_t q_blocks = (m + qb - 1) / qb;
    int flip = 0;
    auto block_sum = [&](int c) {
        flip ^= 1;
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (lane == 0) cnt_s[flip][warp] = c;
        __syncthreads();
        c = 0;
#pragma unroll
        for (int w = 0; w < kMergeThreads / 32; ++w) c += cnt_s[flip][w];
        return c;
    };
    const int64_t ex0 = ex_ptr ? ex_ptr[q] : 0;
    const int64_t ex_n = ex_ptr ? ex_ptr[q + 1] - ex0 : 0;
    const bool ex_here = ex_n <= kMergeExcluded;
    if (ex_here)
        for (int p = tid; p < (int)ex_n; p += kMergeThreads) ex_s[p] = ex_idx[ex0 + p];
    ex_bits[tid] = 0;
    auto left_out = [&](int32_t id) {
        if (!ex_here) return excluded(ex_ptr, ex_idx, q, id);
        if (!(ex_bits[(uint32_t)id / 32 % kMergeThreads] >> ((uint32_t)id % 32) & 1u)) return false;
        int lo = 0, hi = (int)ex_n;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (ex_s[mid] < id) lo = mid + 1; else hi = mid;
        }
        return lo < (int)ex_n && ex_s[lo] == id;
    };
    if (tid < k) best[tid] = first ? 0 : carry[q * k + tid];
    // where every list's candidates begin: thread t has lists kScan t .. kScan t + kScan - 1
    constexpr int kScan = kMergeLists / kMergeThreads;
    int cl[kScan], mine = 0, longest = 1;
#pragma unroll
    for (int j = 0; j < kScan; ++j) {
        const int l = tid * kScan + j;
        cl[j] = l < n_lists ? list_cnt[(int64_t)l * m + q] : 0;
        mine += cl[j];
        longest = max(longest, cl[j]);
    }
    int upto = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, upto, o);
        if (lane >= o) upto += v;
    }
    longest = __reduce_max_sync(0xFFFFFFFFu, longest);
    if (lane == 31) { cnt_s[0][warp] = upto; max_s[0][warp] = longest; }
    __syncthreads();
    int at = upto - mine;
#pragma unroll
    for (int w = 0; w < kMergeThreads / 32; ++w) {
        if (w < warp) at += cnt_s[0][w];
        longest = max(longest, max_s[0][w]);
    }
#pragma unroll
    for (int j = 0; j < kScan; ++j) {
        start_s[tid * kScan + j] = at;
        at += cl[j];
    }
    if (tid == kMergeThreads - 1) start_s[kMergeLists] = at;
    if (ex_here)
        for (int p = tid; p < (int)ex_n; p += kMergeThreads) atomicOr(&ex_bits[(uint32_t)ex_s[p] / 32 % kMergeThreads], 1u << ((uint32_t)ex_s[p] % 32));
    __syncthreads();
    const int total = start_s[kMergeLists];
    const int group = total <= kMergeKeys - k ? n_lists : (kMergeKeys - k) / longest;
    int n_best = first ? 0 : k;
    for (int s0 = 0; s0 < n_lists; s0 += group) {
        const int s1 = s0 + group < n_lists ? s0 + group : n_lists;
        const int base = start_s[s0], n_new = start_s[s1] - base, n_in = n_new + n_best;
        for (int l = s0 + tid / 8; l < s1; l += kMergeThreads / 8)      // eight threads per list: few long lists or many short ones
            for (int p = start_s[l] - base + tid % 8, e = start_s[l + 1] - base; p < e; p += 8) list_s[p] = (uint16_t)l;
#pragma unroll
        for (int b = 0; b < kMergeBins / kMergeThreads; ++b) hist[tid + kMergeThreads * b] = 0;
        if (tid == 0) { bin_lo = 0xFFFFFFFFu; bin_hi = 0; }
        __syncthreads();
        uint64_t e[kMergePer];
#pragma unroll
        for (int j = 0; j < kMergePer; ++j) {
            const int p = tid + kMergeThreads * j;
            e[j] = 0;
            if (p < n_new) {
                const int l = list_s[p];
                e[j] = lists[(((int64_t)l * q_blocks + q / qb) * cap + (p + base - start_s[l])) * qb + q % qb];
            } else if (p < n_in) {
                e[j] = best[p - n_new];
            }
        }
        int have = 0;
        uint32_t lo = 0xFFFFFFFFu, hi = 0;
#pragma unroll
        for (int j = 0; j < kMergePer; ++j) {
            if (kMergeThreads * j >= n_in) break;
            if (tid + kMergeThreads * j < n_new && e[j] != 0 && (e[j] < thr || (ex_n && left_out(key_id(e[j]))))) e[j] = 0;
            if (e[j]) {
                ++have;
                lo = min(lo, (uint32_t)(e[j] >> 32));
                hi = max(hi, (uint32_t)(e[j] >> 32));
            }
        }
        lo = __reduce_min_sync(0xFFFFFFFFu, lo);
        hi = __reduce_max_sync(0xFFFFFFFFu, hi);
        if (lane == 0) { max_s[0][warp] = (int)lo; max_s[1][warp] = (int)hi; }
        const int n = block_sum(have);
        uint64_t bar = 1;      // keep keys >= bar
        if (n > k) {
#pragma unroll
            for (int w = 0; w < kMergeThreads / 32; ++w) {
                lo = min(lo, (uint32_t)max_s[0][w]);
                hi = max(hi, (uint32_t)max_s[1][w]);
            }
            // (a bin never falls as the score rises: every step of its formula is monotone.  One bin for all where the scores'
            // range is zero, infinite or not a number.)
            const float least = order_score(lo), range = order_score(hi) - least;
            float per_score = (float)(kMergeBins - 1) / range;
            if (!(range > 0.f && range < INFINITY && per_score < INFINITY)) per_score = 0.f;
            auto bin_of = [&](uint64_t key) {
                return per_score > 0.f ? min((int)((order_score((uint32_t)(key >> 32)) - least) * per_score), kMergeBins - 1) : 0;
            };
#pragma unroll
            for (int j = 0; j < kMergePer; ++j)
                if (e[j]) atomicAdd(&hist[bin_of(e[j])], 1);
            __syncthreads();
            constexpr int kBins = kMergeBins / kMergeThreads;
            int c[kBins], from = 0;
#pragma unroll
            for (int b = 0; b < kBins; ++b) {
                c[b] = hist[tid * kBins + b];
                from += c[b];
            }
            int incl = from;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_down_sync(0xFFFFFFFFu, incl, o);
                if (lane + o < 32) incl += v;
            }
            if (lane == 0) max_s[0][warp] = incl;
            __syncthreads();
            int above = incl - from;
            for (int w = warp + 1; w < kMergeThreads / 32; ++w) above += max_s[0][w];
#pragma unroll
            for (int b = kBins - 1; b >= 0; --b) {
                if (above < k && above + c[b] >= k) { bin_s = tid * kBins + b; bin_above = above + c[b]; }
                above += c[b];
            }
            __syncthreads();
            const int bin = bin_s;
            int at_lo = bin_above;
            if (at_lo > k)
#pragma unroll
                for (int j = 0; j < kMergePer; ++j)
                    if (e[j] && bin_of(e[j]) == bin) {
                        atomicMin(&bin_lo, (uint32_t)(e[j] >> 32));
                        atomicMax(&bin_hi, (uint32_t)(e[j] >> 32));
                    }
            if (at_lo == k) {
                uint32_t kth = 0xFFFFFFFFu;
#pragma unroll
                for (int j = 0; j < kMergePer; ++j)
                    if (e[j] && bin_of(e[j]) >= bin) kth = min(kth, (uint32_t)(e[j] >> 32));
                kth = __reduce_min_sync(0xFFFFFFFFu, kth);
                if (lane == 0) atomicMin(&bin_lo, kth);
            }
            __syncthreads();
            lo = bin_lo;
            hi = at_lo > k ? bin_hi : lo;
            for (int step = 0; at_lo > k && lo < hi; ++step) {
                const uint32_t mid = bisect_at(lo, hi, step);
                int cc = 0;
#pragma unroll
                for (int j = 0; j < kMergePer; ++j)
                    if (kMergeThreads * j < n_in) cc += (uint32_t)(e[j] >> 32) >= mid;
                cc = block_sum(cc);
                if (cc >= k) { lo = mid; at_lo = cc; } else hi = mid - 1;
            }
            bar = (uint64_t)lo << 32;
            for (int bit = 31; bit >= 0 && at_lo > k; --bit) {      // scores equal to the k-th: the smaller ids
                const uint64_t cand = bar | (1u << bit);
                int cc = 0;
#pragma unroll
                for (int j = 0; j < kMergePer; ++j)
                    if (kMergeThreads * j < n_in) cc += e[j] >= cand;
                cc = block_sum(cc);
                if (cc >= k) { bar = cand; at_lo = cc; }
            }
        }
        if (tid == 0) n_s = 0;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kMergePer; ++j)
            if (e[j] != 0 && e[j] >= bar) best[atomicAdd(&n_s, 1)] = e[j];
        __syncthreads();
        n_best = n_s;
    }
    const int n = n_best;
    if (!last) {
        const uint64_t key = tid < n ? best[tid] : 0;
        if (tid < k) carry[q * k + tid] = key;
        if (n == k) {
            const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, tid < k ? (uint32_t)(key >> 32) : 0xFFFFFFFFu);
            if (lane == 0) cnt_s[0][warp] = (int)least;
            __syncthreads();
            if (tid == 0) {
                uint32_t all = least;
                for (int w = 1; w < kMergeThreads / 32; ++w) all = min(all, (uint32_t)cnt_s[0][w]);
                gtau[q] = all;
            }
        }
        return;
    }
    if (tid < k) {
        if (tid < n) {
            const uint64_t mine = best[tid];
            int rank = 0;
#pragma unroll 8
            for (int p = 0; p < n; ++p) rank += best[p] > mine;
            ids_out[q * k + rank] = key_id(mine);
            if (scores_out) scores_out[q * k + rank] = order_score((uint32_t)(mine >> 32));
        } else {      // fewer than k candidates: the rest of the row says so
            ids_out[q * k + tid] = -1;
            if (scores_out) scores_out[q * k + tid] = -INFINITY;
        }
    }
}

struct FmaArgs {
    const void *H;
    int64_t i_begin, i_end;
    const float *Q;
    int64_t m;
    int k, cap;
    const int64_t *ex_ptr;
    const int32_t *ex_idx;
    int slabs;
    int64_t slab;
    uint64_t *lists;
    int32_t *cnt;
    const unsigned *gtau;
    cudaStream_t s;
};

template <int D, typename T, int QT> cudaError_t launch_fma(const FmaArgs &a)
{
    using G = FmaGeo<D, T, QT>;
    static_assert(G::ITEMS <= kTopkTile, "a tile's items fit a candidate buffer");
    static SmemOnce allow;
    const cudaError_t e = allow(k_topk_fma<D, T, QT>, G::SMEM);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((a.m + QT - 1) / QT), (unsigned)a.slabs);
    k_topk_fma<D, T, QT><<<grid, kFmaThreads, G::SMEM, a.s>>>(static_cast<const T *>(a.H), a.i_begin, a.i_end, a.Q, a.m, a.k, a.cap,
                                                              a.ex_ptr, a.ex_idx, a.slab, a.lists, a.cnt, a.gtau);
    return cudaGetLastError();
}

template <int D, typename T> cudaError_t launch_fma_q(int qt, const FmaArgs &a)
{
    switch (qt) {
    case 4: return launch_fma<D, T, 4>(a);
    case 8: return launch_fma<D, T, 8>(a);
    case 16: return launch_fma<D, T, 16>(a);
    default: return launch_fma<D, T, 64>(a);
    }
}

template <int D> cudaError_t launch_fma_t(bool bf16, int qt, const FmaArgs &a)
{
    return bf16 ? launch_fma_q<D, __nv_bfloat16>(qt, a) : launch_fma_q<D, float>(qt, a);
}

constexpr int64_t kTopkWorkspace = 256ll << 20;      // candidate lists of one batch of queries

// slabs for a phase of `items` items: minimises (waves of blocks) x (items per slab + what a block costs beside them, in items)
int phase_slabs(int64_t items, int64_t tiles, int tile_items, int64_t resident, int64_t start)
{
    const int64_t most = (items + tile_items - 1) / tile_items < kTopkMostSlabs ? (items + tile_items - 1) / tile_items : kTopkMostSlabs;
    int64_t best = INT64_MAX;
    int slabs = 1;
    for (int64_t s = 1; s <= most && tiles * s <= 4 * resident + tiles; ++s) {
        const int64_t cost = (tiles * s + resident - 1) / resident * ((items + s - 1) / s + start);
        if (cost < best) { best = cost; slabs = (int)s; }
    }
    return slabs;
}

}  // namespace

// How a call is cut up: batches of queries whose candidate lists fit the workspace limit, phases and slabs of items.
TopkPlan topk_plan(int64_t n_items, int64_t m, int k, bool tensor_cores)
{
    TopkPlan p;
    p.tensor_cores = tensor_cores && m > kFmaQueries;
    p.cap = topk_cap(k);
    p.qt = p.tensor_cores ? kTopkQueries : m <= 4 ? 4 : m <= 8 ? 8 : m <= 16 ? 16 : 64;
    p.tile_items = p.tensor_cores || p.qt < 64 ? 256 : 128;
    const int64_t resident = p.tensor_cores ? 148 : 2 * 148, start = p.tensor_cores ? 1500 : 500;
    const int per_slab = p.tensor_cores ? kTopkListsPerSlab : 1;      // lists a slab keeps per query
    for (p.m_batch = m;; p.m_batch = (p.m_batch / 2 + p.qt - 1) / p.qt * p.qt) {
        const int64_t tiles = (p.m_batch + p.qt - 1) / p.qt;
        p.phases = 0;
        int lists = 0;
        int64_t seen = 0;
        while (seen < n_items) {
            int64_t len = n_items - seen;
            if (p.phases == 0) {
                // a tile per block, unless one phase does for all
                int64_t pilot = (int64_t)p.tile_items * ((resident + tiles - 1) / tiles);
                if (pilot > kTopkTotal) pilot = kTopkTotal / p.tile_items * p.tile_items;
                if (n_items > kTopkOnePhase) len = pilot;
            } else if (p.phases + 1 < TopkPlan::kMostPhases) {
                const int64_t slabs = phase_slabs(len, tiles, p.tile_items, resident, start);
                int64_t fit = seen / k * slabs * per_slab * kTopkExpect;
                if (fit > seen / k * kTopkTotal) fit = seen / k * kTopkTotal;
                if (fit + fit / 2 < len) len = fit / p.tile_items * p.tile_items;
                if (len < p.tile_items) len = p.tile_items < n_items - seen ? p.tile_items : n_items - seen;
            }
            TopkPlan::Phase &ph = p.phase[p.phases++];
            ph.begin = seen;
            ph.end = seen + len;
            ph.slabs = phase_slabs(len, tiles, p.tile_items, resident, start);
            ph.slab = ((len + ph.slabs - 1) / ph.slabs + p.tile_items - 1) / p.tile_items * p.tile_items;
            ph.slabs = (int)((len + ph.slab - 1) / ph.slab);
            lists = ph.slabs * per_slab > lists ? ph.slabs * per_slab : lists;
            seen += len;
        }
        const int64_t mp = tiles * p.qt;
        p.list_bytes = (int64_t)lists * mp * p.cap * (int64_t)sizeof(uint64_t);
        p.cnt_bytes = ((int64_t)lists * p.m_batch * 4 + 255) / 256 * 256;
        if (p.list_bytes <= kTopkWorkspace || p.m_batch <= p.qt) break;
    }
    p.tau_bytes = (p.m_batch * 4 + 255) / 256 * 256;
    p.carry_bytes = p.phases > 1 ? (p.m_batch * k * 8 + 255) / 256 * 256 : 0;
    p.query_bytes = p.tensor_cores ? topk_query_scratch_bytes(p.m_batch) : 0;
    return p;
}

cudaError_t launch_topk(const TopkPlan &p, const void *H, bool bf16, int64_t n_items, int d, const float *Q, int64_t m, int k,
                        const int64_t *ex_ptr, const int32_t *ex_idx, void *workspace, int32_t *ids_out, float *scores_out,
                        DevStatus *st, cudaStream_t s, int64_t *launches)
{
    unsigned char *w = static_cast<unsigned char *>(workspace);
    uint64_t *lists = reinterpret_cast<uint64_t *>(w);
    int32_t *cnt = reinterpret_cast<int32_t *>(w += p.list_bytes);
    unsigned *gtau = reinterpret_cast<unsigned *>(w += p.cnt_bytes);
    uint64_t *carry = reinterpret_cast<uint64_t *>(w += p.tau_bytes);
    void *parts = w + p.carry_bytes;
    for (int64_t q0 = 0; q0 < m; q0 += p.m_batch) {
        const int64_t mb = m - q0 < p.m_batch ? m - q0 : p.m_batch;
        const float *Qb = Q + q0 * d;
        const int64_t *exb = ex_ptr ? ex_ptr + q0 : nullptr;
        cudaError_t e = cudaMemsetAsync(gtau, 0, sizeof(unsigned) * mb, s);
        if (e != cudaSuccess) return e;
        TopkUmma u;
        if (p.tensor_cores && (e = topk_umma_prepare(H, n_items, Qb, mb, parts, &u, s, launches)) != cudaSuccess) return e;
        for (int f = 0; f < p.phases; ++f) {
            const TopkPlan::Phase &ph = p.phase[f];
            if (p.tensor_cores) {
                e = launch_topk_umma(u, ph.begin, ph.end, mb, k, p.cap, exb, ex_idx, ph.slabs, ph.slab, lists, cnt, gtau, st, s);
            } else {
                const FmaArgs a{H, ph.begin, ph.end, Qb, mb, k, p.cap, exb, ex_idx, ph.slabs, ph.slab, lists, cnt, gtau, s};
                switch (d) {
                case 16: e = launch_fma_t<16>(bf16, p.qt, a); break;
                case 32: e = launch_fma_t<32>(bf16, p.qt, a); break;
                case 64: e = launch_fma_t<64>(bf16, p.qt, a); break;
                case 128: e = launch_fma_t<128>(bf16, p.qt, a); break;
                default: return cudaErrorInvalidValue;
                }
            }
            if (e != cudaSuccess) return e;
            k_topk_merge<<<(unsigned)mb, kMergeThreads, 0, s>>>(lists, cnt, gtau, carry, f == 0, f == p.phases - 1, mb, k, p.cap,
                                                                ph.slabs * (p.tensor_cores ? kTopkListsPerSlab : 1),
                                                                p.tensor_cores ? kTopkQueries : 1, exb, ex_idx, ids_out + q0 * k,
                                                                scores_out ? scores_out + q0 * k : nullptr);
            *launches += 2;
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace alx
