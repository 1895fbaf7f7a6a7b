// The objective of Eq. 3 at the current tables.  The observed term is summed entry by entry
// (products and the length-d dot product in fp32, everything across entries in fp64, fixed order);
// the all-pairs term uses sum_u sum_i <w_u, h_i>^2 = <W^T W, H^T H>_F, the Gramian identity the paper
// states under Eq. 4 applied to the objective; the regulariser is the trace of the two Gramians.
#include "alx_common.cuh"
#include "alx_mma.cuh"

namespace alx {

namespace {

constexpr int kWarps = 8;
constexpr int kBlocksPerSm = 3;
// bfloat16 tables of 128 features: products by mma where rows hold 16 entries or more on average (shorter rows need the second set
// of products and another load of W rows in most steps: 12 a row 488 us against 471 for 1.2e7 entries, 24 a row 412 against 460,
// 120 a row 315 against 444; 64 features: 164 against 134 us at 20 a row).  Two blocks per SM: 16 loads of 16 bytes a lane are in flight
constexpr int64_t kMmaLeastRow = 16;
constexpr int64_t kMostBlocksMma = 148 * 2;
constexpr int64_t kMostBlocks = 148 * kBlocksPerSm;
// Entries a warp takes at a time; the warps then go on together to the next stretch of the matrix, so that at any time they
// read neighbouring rows of W, and of H where the matrix is local (one long range per warp spread them over the whole table:
// 70 ms instead of 35 ms for 1e9 entries within 1 % of the diagonal)
constexpr int kMostSpan = 512;

// entries per span: as many as give every SM something to do, a multiple of 32
int span_of(int64_t nnz)
{
    const int64_t s = nnz / (kMostBlocks * kWarps) / 32 * 32;
    return s < 32 ? 32 : s < kMostSpan ? (int)s : kMostSpan;
}

// largest u in [0, n) with ptr[u] <= e, by the whole warp: 32 probes a round
__device__ __forceinline__ int64_t warp_row_of(const int64_t *__restrict__ ptr, int64_t n, int64_t e, int lane)
{
    int64_t lo = 0, hi = n;      // ptr[lo] <= e, and ptr[hi] > e or hi = n
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t at = lo + (lane + 1) * step;
        const bool le = at < hi && ptr[at] <= e;
        const int below = __popc(__ballot_sync(0xFFFFFFFFu, le));      // probes are ascending: the first `below` hold
        const int64_t l = lo + below * step;
        hi = l + step < hi ? l + step : hi;
        lo = l;
    }
    return lo;
}

// 16 bytes of a table row as floats
__device__ __forceinline__ void unpack16(const uint4 &a, float (&v)[4])
{
    v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y); v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
}
__device__ __forceinline__ void unpack16(const uint4 &a, float (&v)[8])
{
    const uint32_t x[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[2 * k] = __uint_as_float(x[k] << 16);
        v[2 * k + 1] = __uint_as_float(x[k] & 0xFFFF0000u);
    }
}

// sums over the LANES lanes of a group of each of U values (U = 4, or 2 for LANES = 2): lane `part` of a group with
// t0 <= part < t0 + U receives the sum of v[part - t0].  The values are halved with the lanes: U - 1 shuffles, then one value's
// butterfly, then one shuffle to the lane that wants it.
template <int LANES, int U> __device__ __forceinline__ float group_sums(float (&v)[U], int t0, int lane)
{
    int o = LANES / 2;
#pragma unroll
    for (int n = U / 2; n > 0; n /= 2, o /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const float send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
            v[k] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
        }
    }
#pragma unroll
    for (; o > 0; o /= 2) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
    return __shfl_sync(0xFFFFFFFFu, v[0], (lane & ~(LANES - 1)) + (((lane & (LANES - 1)) - t0) & (U - 1)) * (LANES / U));
}

__device__ __forceinline__ double block_sum(double v, double *buf)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
    for (int w = 0; w < kWarps; ++w) r += buf[w];
    __syncthreads();
    return r;
}

// The 16 entries from `half` on of the batch by mma.sync m16n8k16: A = their H rows (lane (g, q) = (lane / 4, lane % 4) has the 16-byte
// pieces q + 4j of rows g and g + 8), B = the W rows of every second entry as columns (pieces alike, so that the features of A
// and B go by the same permutation), C[e][e / 2] the dot products.  Entries whose row is not the one of the entry before them
// and have an odd number need their own B: a second set of products, only where there is one.  The products start from zero
// and are added by FADD, as the instruction truncates its accumulator.  Returns the dot product of entry half + g + 8 (q / 2)
// to the lanes with q % 2 = g / 4.
// 27 instructions an entry became about 7, and the gather through L2 is the bound: 1e9 entries 42 -> 31 ms.
template <int CH> struct HRows {
    uint4 a[CH], b[CH];
};
template <int CH> __device__ __forceinline__ void load_h(HRows<CH> &h, const __nv_bfloat16 *__restrict__ H, int c, int half, int lane)
{
    const int64_t ca = __shfl_sync(0xFFFFFFFFu, c, half + (lane >> 2)), cb = __shfl_sync(0xFFFFFFFFu, c, half + (lane >> 2) + 8);
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        h.a[j] = __ldg(reinterpret_cast<const uint4 *>(H + ca * (32 * CH)) + (lane & 3) + 4 * j);
        h.b[j] = __ldg(reinterpret_cast<const uint4 *>(H + cb * (32 * CH)) + (lane & 3) + 4 * j);
    }
}
template <int CH> __device__ __forceinline__ void products(const HRows<CH> &h, const uint4 (&w)[CH], float (&d)[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = 0.f;
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        const uint32_t lo[4] = {h.a[j].x, h.b[j].x, h.a[j].y, h.b[j].y}, hi[4] = {h.a[j].z, h.b[j].z, h.a[j].w, h.b[j].w};
        float p[4] = {0.f, 0.f, 0.f, 0.f}, r[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(p, lo, w[j].x, w[j].y);
        mma_bf16(r, hi, w[j].z, w[j].w);
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] += p[k] + r[k];
    }
}
template <int CH>
__device__ __forceinline__ float dots(const HRows<CH> &h, const __nv_bfloat16 *__restrict__ W, int row, int half, int &w_row, uint4 (&w)[CH], int lane)
{
    const int g = lane >> 2, q = lane & 3;
    const int even = __shfl_sync(0xFFFFFFFFu, row, half + 2 * g), odd = __shfl_sync(0xFFFFFFFFu, row, half + 2 * g + 1);
    if (__any_sync(0xFFFFFFFFu, even != w_row)) {
        w_row = even;
#pragma unroll
        for (int j = 0; j < CH; ++j) w[j] = __ldg(reinterpret_cast<const uint4 *>(W + (int64_t)even * (32 * CH)) + q + 4 * j);
    }
    float d[4];
    products(h, w, d);
    const bool second = (g >> 1) & 1;      // (entry g: column g / 2, entry g + 8: column 4 + g / 2, columns 2q and 2q + 1 are here)
    float v = q < 2 ? (second ? d[1] : d[0]) : (second ? d[3] : d[2]);
    if (__any_sync(0xFFFFFFFFu, odd != even)) {
        w_row = odd;
#pragma unroll
        for (int j = 0; j < CH; ++j) w[j] = __ldg(reinterpret_cast<const uint4 *>(W + (int64_t)odd * (32 * CH)) + q + 4 * j);
        products(h, w, d);
        if (g & 1) v = q < 2 ? (second ? d[1] : d[0]) : (second ? d[3] : d[2]);
    }
    return v;
}

// A warp takes spans of entries, 32 at a time: every lane looks up its entry's column, label and row (a window of the row offsets,
// searched by shuffles).  A group of LANES lanes then works through LANES of the entries in turn, 16 bytes of a row a lane, so
// that the W row stays in registers while the row goes on; four entries' loads are in flight and their sums share a
// butterfly (with MMA: dots, above).  Bound without MMA: the latency of the H rows' gather (two rounds in flight, 24 warps per SM), and the 16 instructions an entry of 128 bfloat16 features takes.  The last
// block to finish adds the blocks' sums in order and the two Gramian terms.
template <int D, typename T, bool MMA>
__global__ void __launch_bounds__(kWarps * 32, MMA ? 2 : kBlocksPerSm) k_loss(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                                                      const float *__restrict__ values, int64_t n_rows, int64_t nnz, int span,
                                                      const T *__restrict__ W, const T *__restrict__ H, const double *__restrict__ GW,
                                                      const double *__restrict__ GH, double alpha0, double lambda, double *partials,
                                                      unsigned *counter, const DevStatus *st, DevStatus *host_status, double *host_result)
{
    constexpr int EL = 16 / (int)sizeof(T), LANES = D / EL, U = LANES < 4 ? LANES : 4;
    __shared__ double buf[kWarps];
    __shared__ int last_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = lane % LANES, first = lane - part;      // first lane of the group
    double acc = 0.0;
    for (int64_t e0 = ((int64_t)blockIdx.x * kWarps + warp) * span; e0 < nnz; e0 += (int64_t)gridDim.x * kWarps * span) {
        const int64_t e1 = e0 + span < nnz ? e0 + span : nnz;
        int64_t u = warp_row_of(rowptr, n_rows, e0, lane);
        int w_row = -1;
        float w[EL];
        [[maybe_unused]] uint4 wm[D >= 32 ? D / 32 : 1];
        // MMA: columns two batches ahead, labels one; the first 16 H rows of a batch are fetched while the batch before it is multiplied
        [[maybe_unused]] int32_t c0 = 0, c1 = 0;
        [[maybe_unused]] float y0 = 1.f;
        [[maybe_unused]] HRows<(D >= 32 ? D / 32 : 1)> h[2];
        if constexpr (MMA) {
            c0 = e0 + lane < e1 ? colidx[e0 + lane] : 0;
            c1 = e0 + 32 + lane < e1 ? colidx[e0 + 32 + lane] : 0;
            if (values && e0 + lane < e1) y0 = values[e0 + lane];
            load_h(h[0], H, c0, 0, lane);
        }
        for (int64_t base = e0; base < e1; base += 32) {
            const int64_t e = base + lane;
            const int64_t last = e1 - 1 < base + 31 ? e1 - 1 : base + 31;
            const int32_t c = MMA ? c0 : e < e1 ? colidx[e] : 0;
            const float y = MMA ? y0 : values && e < e1 ? values[e] : 1.f;
            if constexpr (MMA) {
                load_h(h[1], H, c, 16, lane);
                c0 = c1;
                c1 = e + 64 < e1 ? colidx[e + 64] : 0;
                y0 = values && e + 32 < e1 ? values[e + 32] : 1.f;
            }
            // row of this lane's entry: count the offsets ptr[u + 1 ..] that are <= e
            int64_t row = u, at = u + 1;
            while (true) {
                const int64_t p = at + lane < n_rows ? rowptr[at + lane] : INT64_MAX;
                int lo = 0;      // how many of the 32 offsets are <= e (they ascend)
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int64_t q = __shfl_sync(0xFFFFFFFFu, p, lo + step - 1);
                    if (q <= e) lo += step;
                }
                const int64_t q = __shfl_sync(0xFFFFFFFFu, p, 31);
                if (lo == 31 && q <= e) lo = 32;
                row += lo;
                if (q > last) break;      // (warp-uniform: the 32nd offset lies beyond the batch)
                at += 32;
            }
            u = __shfl_sync(0xFFFFFFFFu, row, (int)(last - base));
            if constexpr (MMA) {
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const float v = dots(h[t], W, (int)row, 16 * t, w_row, wm, lane);
                    if (t == 0 && base + 32 < e1) load_h(h[0], H, c0, 0, lane);
                    const int k = 16 * t + (lane >> 2) + ((lane & 2) << 2);
                    const double r = (double)__shfl_sync(0xFFFFFFFFu, y, k) - (double)v;
                    if ((lane & 1) == lane >> 4 && base + k < e1) acc = fma(r, r, acc);
                }
                continue;
            } else {
            float dot = 0.f;
            uint4 hr[2][U];
            auto load = [&](int t0, uint4(&to)[U]) {
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const int64_t hc = __shfl_sync(0xFFFFFFFFu, c, first + t0 + k);
                    to[k] = __ldg(reinterpret_cast<const uint4 *>(H + hc * D) + part);
                }
            };
            load(0, hr[0]);
#pragma unroll
            for (int t0 = 0; t0 < LANES; t0 += U) {
                if (t0 + U < LANES) load(t0 + U, hr[(t0 / U + 1) & 1]);      // one round ahead
                float s[U];
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const int wr = __shfl_sync(0xFFFFFFFFu, (int)row, first + t0 + k);
                    if (wr != w_row) {
                        w_row = wr;
                        unpack16(__ldg(reinterpret_cast<const uint4 *>(W + (int64_t)w_row * D) + part), w);
                    }
                    float hv[EL];
                    unpack16(hr[(t0 / U) & 1][k], hv);
                    s[k] = w[0] * hv[0];
#pragma unroll
                    for (int j = 1; j < EL; ++j) s[k] = fmaf(w[j], hv[j], s[k]);
                }
                const float d = group_sums<LANES, U>(s, t0, lane);
                if (part - t0 >= 0 && part - t0 < U) dot = d;
            }
            const double r = (double)y - (double)dot;
            if (e < e1) acc = fma(r, r, acc);
            }
        }
    }
    const double mine = block_sum(acc, buf);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = mine;
        __threadfence();
        last_s = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    wait_for_previous();      // the Gramians (the entries need none of them)
    double s = 0.0, f = 0.0, t = 0.0;
    for (unsigned p = threadIdx.x; p < gridDim.x; p += kWarps * 32) s += __ldcg(partials + p);
#pragma unroll 8
    for (int e = threadIdx.x; e < D * D; e += kWarps * 32) {
        const double a = GW[e], b = GH[e];
        f = fma(a, b, f);
        if (e / D == e % D) t += a + b;
    }
    s = block_sum(s, buf);
    f = block_sum(f, buf);
    t = block_sum(t, buf);
    if (threadIdx.x == 0) {
        // straight to the host, with the status word: one wait and no copies
        host_result[0] = nnz > 0 ? s : 0.0;
        host_result[1] = alpha0 * f;
        host_result[2] = lambda * t;
        *host_status = *st;
        *counter = 0;
    }
}

}  // namespace

int64_t loss_partials(int64_t nnz)
{
    const int64_t per = (int64_t)span_of(nnz) * kWarps, b = (nnz + per - 1) / per;
    return b < kMostBlocks ? (b > 0 ? b : 1) : kMostBlocks;
}

cudaError_t launch_loss(const int64_t *rowptr, const int32_t *colidx, const float *values, int64_t n_rows, int64_t nnz, const void *W,
                        const void *H, int bf16, int d, const double *GW, const double *GH, double alpha0, double lambda, double *partials,
                        unsigned *counter, const DevStatus *st, DevStatus *host_status, double *host_result, bool beside_gramian, cudaStream_t s, int64_t *launches)
{
    const int64_t sums = loss_partials(nnz);
    // beside_gramian: the launch before this one is the reduction of a Gramian, which starts when the tables are complete and which
    // this kernel waits for at its end
    const bool early = beside_gramian && nnz <= kEarlyEntries;
#define ALX_LOSS(DD, T, MMA)                                                                                                         \
    {                                                                                                                                \
        const int64_t blocks = MMA && sums > kMostBlocksMma ? kMostBlocksMma : sums;                                                 \
        const cudaError_t e = launch_early(early, k_loss<DD, T, MMA>, blocks, kWarps * 32, 0, s, rowptr, colidx, values, n_rows, nnz, \
                                           span_of(nnz), (const T *)W, (const T *)H, GW, GH, alpha0, lambda, partials, counter, st,  \
                                           host_status, host_result);                                                                \
        if (e != cudaSuccess) return e;                                                                                              \
    }
#define ALX_CASE(DD)                                                       \
    case DD:                                                               \
        if (!bf16) ALX_LOSS(DD, float, false)                              \
        else if (DD == 128 && nnz >= kMmaLeastRow * n_rows) ALX_LOSS(DD, __nv_bfloat16, (DD == 128)) \
        else ALX_LOSS(DD, __nv_bfloat16, false)                            \
        break;
    switch (d) {
        ALX_CASE(16)
        ALX_CASE(32)
        ALX_CASE(64)
        ALX_CASE(128)
    default: return cudaErrorInvalidValue;
    }
#undef ALX_CASE
#undef ALX_LOSS
    ++*launches;
    return cudaGetLastError();
}

}  // namespace alx
