// Row kernels of one half-epoch for fp32 tables of 128 features: a team of four warps per row.
//
// The same plan as the warp-per-row kernels (alx_rows_warp.cu), with the 128 x 128 matrix spread over four warps: the sums are
// mma.sync products of the three bfloat16 parts of the gathered rows (the six products down to 2^-24), the matrix stays in
// the mma fragments of the warps (warp w: the 16-row blocks w and 7 - w of the lower triangle, 18 blocks of 16 x 8 each, so the
// warps have equal shares of the sums and nearly equal ones of every trailing update), and is factored 16 columns at a time.
// For a panel every warp factors the diagonal block itself, redundantly, beside its own 32 rows below it (lane = row), so that
// the column steps need shuffles only; the block meets at a barrier before and after a panel.
//
// The FP32-ALU kernels (alx_rows.cu) gave such a row 256 threads that met at a barrier three times per 16 columns and did the
// trailing update with FMAs from shared memory: 60k x 25k, 2e6 entries, one epoch 17.4 ms; here 6.8 ms
// with the dual form for the rows of at most 16 entries (this kernel 5.1, the sums of long rows 0.7).
// Bound: the chain of 64 double column steps and the 128 steps of the back substitution (three teams per SM hide what they can).
#include "alx_common.cuh"
#include "alx_mma.cuh"
#include "alx_ptx.cuh"

namespace alx {

namespace {

constexpr int D = 128;
constexpr int kWarps = 4, kTeam = kWarps * 32;
constexpr int kTeamsPerSm = 3;
constexpr int kEntries = 16;                      // entries per stage = the K of one mma
constexpr int kStage = kEntries * D * 4;
constexpr int kRow = D * 2 + 16;                  // bytes between the rows of a bfloat16 tile (ldmatrix without conflicts)
constexpr int kTile = 3 * kEntries * kRow;
constexpr int kBlocks = 8;                        // 16-row blocks of the matrix
constexpr int kLo = 8, kHi = 16;                  // 16 x 8 blocks of block rows w (at most 8) and 7 - w (at most 16)
constexpr int kSums = 72 * 128 + D;               // floats of a row's sums in the workspace: fragments, then b
constexpr int kMostSlices = 8;

// panel k of L: rows 16 k .. 127, 16 columns; its bfloat16 parts lie where the later panels will (see alx_rows_warp.cu)
__host__ __device__ constexpr int panel_at(int k) { return 16 * (16 * kBlocks * k - 8 * k * (k - 1)); }
constexpr int kLFloats = panel_at(kBlocks) + 128;

struct __align__(16) TeamSmem {
    unsigned char ring[2][kStage];
    union {
        float L[kLFloats];
        unsigned char tile[kTile];
    };
    float b[D], z[D], dinv[D];      // right-hand side, then the solution; L^-1 b; reciprocal pivots
    float exchange[kWarps][64];
    float part[kWarps][16];
    float y[2][kEntries];
};
static_assert(kTeamsPerSm * (sizeof(TeamSmem) + 1024) <= 233472, "shared memory");

struct Acc {
    float lo[kLo][4], hi[kHi][4];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int n = 0; n < kLo; ++n)
#pragma unroll
            for (int j = 0; j < 4; ++j) lo[n][j] = 0.f;
#pragma unroll
        for (int n = 0; n < kHi; ++n)
#pragma unroll
            for (int j = 0; j < 4; ++j) hi[n][j] = 0.f;
    }
};

struct Feed {
    const float *X;
    const int32_t *idx;
    const float *val;
    int64_t at, end;      // the entries after the stages whose ids have been loaded
    int g;                // next stage to be consumed; stage g lives in slot g % 2
    int id, id_first;     // (lane < 16) ids of the stage after the one in flight; of a row's first stage
    float y, y_first;

    __device__ __forceinline__ void load_ids(int lane)
    {
        id = -1;
        y = 0.f;
        if (lane < kEntries && at + lane < end) {
            id = __ldg(idx + at + lane);
            y = val ? __ldg(val + at + lane) : 1.f;
        }
        at += kEntries;
    }
    // copies of a stage: every warp knows the ids; warp w brings entries w, w + 4, ...
    __device__ __forceinline__ void issue(TeamSmem &sm, int stage, int ids, float labels, int warp, int lane)
    {
        const uint32_t dst = ptx::smem_u32(&sm.ring[stage & 1][0]);
#pragma unroll
        for (int k = 0; k < kEntries / kWarps; ++k) {
            const int r = warp + kWarps * k;
            const int row = __shfl_sync(0xFFFFFFFFu, ids, r);
            cp_async16_zfill(dst + r * (D * 4) + lane * 16, X + (int64_t)(row < 0 ? 0 : row) * D + lane * 4, row >= 0);
        }
        if (warp == 0 && lane < kEntries) sm.y[stage & 1][lane] = labels;
        ptx::cp_async_commit();
    }
    __device__ __forceinline__ void start_ids(int64_t beg, int64_t e, int lane)
    {
        at = beg;
        end = e;
        load_ids(lane);
        id_first = id;
        y_first = y;
        load_ids(lane);
    }
    __device__ __forceinline__ void start_copies(TeamSmem &sm, int warp, int lane) { issue(sm, g, id_first, y_first, warp, lane); }
};

// c0, c1 (two blocks of 8 columns) += or -= A B^T, the six products of the parts from the smallest up
template <bool SUB>
__device__ __forceinline__ void add_products(float (&c0)[4], float (&c1)[4], const uint32_t (&a)[3][4], const uint32_t (&b)[3][4])
{
    constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
    float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        mma_bf16(t0, a[pa[q]], b[pb[q]][0], b[pb[q]][2]);
        mma_bf16(t1, a[pa[q]], b[pb[q]][1], b[pb[q]][3]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        c0[e] += SUB ? -t0[e] : t0[e];
        c1[e] += SUB ? -t1[e] : t1[e];
    }
}

// sums over `len` entries of the row that the feed was started on; b: this thread's feature of the right-hand side
__device__ __forceinline__ void sum_entries(Feed &feed, int64_t len, TeamSmem &sm, Acc &acc, float &b, int warp, int lane)
{
    const int tid = warp * 32 + lane;
    const int stages = (int)((len + kEntries - 1) / kEntries);
    const int ilo = warp, ihi = kBlocks - 1 - warp;
    for (int s = 0; s < stages; ++s, ++feed.g) {
        if (s + 1 < stages) {
            feed.issue(sm, feed.g + 1, feed.id, feed.y, warp, lane);
            feed.load_ids(lane);
            ptx::cp_async_wait<1>();
        } else {
            ptx::cp_async_wait<0>();
        }
        __syncthreads();      // the stage is here, and the tile's last readers are done
        const float *raw = reinterpret_cast<const float *>(&sm.ring[feed.g & 1][0]);
        const float *y = sm.y[feed.g & 1];
#pragma unroll
        for (int e = 0; e < kEntries; ++e) b = fmaf(y[e], raw[e * D + tid], b);      // (entries past the end are zeros)
        // the stage's bfloat16 parts: a thread per 4 features of every fourth entry
#pragma unroll
        for (int k = 0; k < kEntries / kWarps; ++k) {
            const int e = warp + kWarps * k;
            const float4 x = *reinterpret_cast<const float4 *>(raw + e * D + 4 * lane);
            uint32_t p[3][2];
            split_bf16(x.x, x.y, p[0][0], p[1][0], p[2][0]);
            split_bf16(x.z, x.w, p[0][1], p[1][1], p[2][1]);
#pragma unroll
            for (int q = 0; q < 3; ++q)
                *reinterpret_cast<uint2 *>(sm.tile + (q * kEntries + e) * kRow + lane * 8) = make_uint2(p[q][0], p[q][1]);
        }
        __syncthreads();
        const uint32_t src = ptx::smem_u32(sm.tile) + ((lane & 7) + 8 * (lane >> 4)) * kRow + 16 * ((lane >> 3) & 1);
        uint32_t al[3][4], ah[3][4];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            ldmatrix_x4_trans(src + q * kEntries * kRow + 32 * ilo, al[q]);
            ldmatrix_x4_trans(src + q * kEntries * kRow + 32 * ihi, ah[q]);
        }
#pragma unroll
        for (int j = 0; j < kBlocks; ++j) {
            if (j > ihi) break;
            uint32_t bf[3][4];
#pragma unroll
            for (int q = 0; q < 3; ++q) ldmatrix_x4_trans(src + q * kEntries * kRow + 32 * j, bf[q]);
            // (from zero in every stage, the sums by FADD: the accumulator of an mma truncates)
            add_products<false>(acc.hi[2 * j], acc.hi[2 * j + 1], ah, bf);
            if (j < kLo / 2 && j <= ilo) add_products<false>(acc.lo[2 * (j < kLo / 2 ? j : 0)], acc.lo[2 * (j < kLo / 2 ? j : 0) + 1], al, bf);
        }
    }
}

// element (r, c) .. of the fragment of block (i, n): rows 16 i + lane / 4 (+ 8), columns 8 n + 2 (lane % 4) (+ 1)
__device__ __forceinline__ void add_base(float (&c)[4], const float *__restrict__ Bmat, int i, int n, int lane)
{
    const float *p = Bmat + (16 * i + lane / 4) * D + 8 * n + 2 * (lane % 4);
    const float2 u = __ldg(reinterpret_cast<const float2 *>(p)), v = __ldg(reinterpret_cast<const float2 *>(p + 8 * D));
    c[0] += u.x; c[1] += u.y; c[2] += v.x; c[3] += v.y;
}

// Factor and solve; the solution replaces sm.b.  Returns (to every thread) whether every pivot was positive.
__device__ __forceinline__ bool factor_solve(Acc &acc, TeamSmem &sm, const float *__restrict__ Bmat, int warp, int lane)
{
    const int ilo = warp, ihi = kBlocks - 1 - warp, tid = warp * 32 + lane;
#pragma unroll
    for (int n = 0; n < kLo; ++n)
        if (n < 2 * (ilo + 1)) add_base(acc.lo[n], Bmat, ilo, n, lane);
#pragma unroll
    for (int n = 0; n < kHi; ++n)
        if (n < 2 * (ihi + 1)) add_base(acc.hi[n], Bmat, ihi, n, lane);
    auto put_block = [&](float *P, const float(&c)[4], int i, int n) {      // block (16 i .., 8 n ..) of the panel
        const int r = 16 * i + lane / 4, q = 2 * n + (lane % 4) / 2, o = 2 * (lane & 1);
        *reinterpret_cast<float2 *>(P + panel_chunk(r, q) + o) = make_float2(c[0], c[1]);
        *reinterpret_cast<float2 *>(P + panel_chunk(r + 8, q) + o) = make_float2(c[2], c[3]);
    };
    __syncthreads();      // (the tile, which L overlays, has been read)
#pragma unroll 1
    for (int k = 0; k < kBlocks; ++k) {
        float *P = sm.L + panel_at(k);
        const int rows = D - 16 * k;
#pragma unroll
        for (int kk = 0; kk < kBlocks; ++kk)
            if (kk == k) {
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    if (kk < kLo / 2 && ilo >= kk) put_block(P, acc.lo[2 * (kk < kLo / 2 ? kk : 0) + n], ilo - kk, n);
                    if (ihi >= kk) put_block(P, acc.hi[2 * kk + n], ihi - kk, n);
                }
            }
        __syncthreads();
        const int dl = lane & 15, own = 16 + tid;      // this lane's row of the diagonal block (lanes 16 .. 31: again), and its own row
        const bool mine = own < rows;
        float a0[16], a1[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float4 v = *reinterpret_cast<const float4 *>(P + panel_chunk(dl, c));
            a0[4 * c] = v.x; a0[4 * c + 1] = v.y; a0[4 * c + 2] = v.z; a0[4 * c + 3] = v.w;
            const float4 w = *reinterpret_cast<const float4 *>(P + panel_chunk(mine ? own : 0, c));
            a1[4 * c] = w.x; a1[4 * c + 1] = w.y; a1[4 * c + 2] = w.z; a1[4 * c + 3] = w.w;
        }
        float b0 = sm.b[16 * k + dl], b1 = mine ? sm.b[16 * k + own] : 0.f;
        // (the first write to the diagonal block's rows and to b comes after the barrier below)
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            const float p = __shfl_sync(0xFFFFFFFFu, a0[j], j), q = __shfl_sync(0xFFFFFFFFu, a0[j], j + 1);
            const float s = __shfl_sync(0xFFFFFFFFu, a0[j + 1], j + 1);
            float z0 = __shfl_sync(0xFFFFFFFFu, b0, j), z1 = __shfl_sync(0xFFFFFFFFu, b0, j + 1);
            // (a pivot that is not positive makes its reciprocal root a NaN, and is reported for that at the end)
            const float i0 = rsqrt_full(p), l10 = q * i0, dd = fmaf(-l10, l10, s), i1 = rsqrt_full(dd);
            z0 *= i0;
            z1 = fmaf(-z0, l10, z1) * i1;
            if (tid == 0) {
                *reinterpret_cast<float2 *>(sm.z + 16 * k + j) = make_float2(z0, z1);
                *reinterpret_cast<float2 *>(sm.dinv + 16 * k + j) = make_float2(i0, i1);
            }
            const float x0 = a0[j] * i0, x1 = fmaf(-x0, l10, a0[j + 1]) * i1;
            const float y0 = a1[j] * i0, y1 = fmaf(-y0, l10, a1[j + 1]) * i1;
            a0[j] = x0;
            a0[j + 1] = x1;
            a1[j] = y0;
            a1[j + 1] = y1;
            b0 = fmaf(-x1, z1, fmaf(-x0, z0, b0));      // (what it becomes in the rows up to j + 1 is not used)
            b1 = fmaf(-y1, z1, fmaf(-y0, z0, b1));
            if (j < 14) {
                float *ex = sm.exchange[warp] + 32 * ((j / 2) & 1);
                if (lane < 16) { ex[lane] = -x0; ex[16 + lane] = -x1; }
                __syncwarp();
#pragma unroll
                for (int c = (j + 2) & ~3; c < 16; c += 4) {
                    const float4 u = *reinterpret_cast<const float4 *>(ex + c), v = *reinterpret_cast<const float4 *>(ex + 16 + c);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int cc = c + 2 * h;
                        if (cc < j + 2) continue;
                        const float2 uu = h ? make_float2(u.z, u.w) : make_float2(u.x, u.y), vv = h ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
                        float2 t = make_float2(a0[cc], a0[cc + 1]), w = make_float2(a1[cc], a1[cc + 1]);
                        t = __ffma2_rn(make_float2(x1, x1), vv, __ffma2_rn(make_float2(x0, x0), uu, t));
                        w = __ffma2_rn(make_float2(y1, y1), vv, __ffma2_rn(make_float2(y0, y0), uu, w));
                        a0[cc] = t.x;
                        a0[cc + 1] = t.y;
                        a1[cc] = w.x;
                        a1[cc + 1] = w.y;
                    }
                }
            }
        }
        __syncthreads();      // every warp has read the panel and b
        if (warp == 0 && lane < 16) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                *reinterpret_cast<float4 *>(P + panel_chunk(lane, c)) = make_float4(a0[4 * c], a0[4 * c + 1], a0[4 * c + 2], a0[4 * c + 3]);
        }
        if (mine) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                *reinterpret_cast<float4 *>(P + panel_chunk(own, c)) = make_float4(a1[4 * c], a1[4 * c + 1], a1[4 * c + 2], a1[4 * c + 3]);
            sm.b[16 * k + own] = b1;
        }
        if (k + 1 < kBlocks) {
            // the rows below as bfloat16 parts, [part][row][16 columns], chunks exchanged in every other group of four rows
            unsigned char *tile = reinterpret_cast<unsigned char *>(sm.L + panel_at(k + 1));
            const int below = rows - 16;
            if (mine) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t p[3][4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) split_bf16(a1[8 * c + 2 * e], a1[8 * c + 2 * e + 1], p[0][e], p[1][e], p[2][e]);
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        *reinterpret_cast<uint4 *>(tile + (q * below + tid) * 32 + 16 * (c ^ ((tid >> 2) & 1))) =
                            make_uint4(p[q][0], p[q][1], p[q][2], p[q][3]);
                }
            }
            __syncthreads();
            // trailing update of the warp's blocks (i, n), i > k, n >= 2 (k + 1)
            const int lr = (lane & 7) + 8 * ((lane >> 3) & 1);
            const uint32_t src = ptx::smem_u32(tile) + lr * 32 + 16 * ((lane >> 4) ^ ((lr >> 2) & 1));
            if (ihi > k) {
                uint32_t al[3][4], ah[3][4];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    ldmatrix_x4(src + (q * below + 16 * (ihi - k - 1)) * 32, ah[q]);
                    if (ilo > k) ldmatrix_x4(src + (q * below + 16 * (ilo - k - 1)) * 32, al[q]);
                }
#pragma unroll
                for (int j = 1; j < kBlocks; ++j) {
                    if (j <= k || j > ihi) continue;
                    uint32_t bf[3][4];
#pragma unroll
                    for (int q = 0; q < 3; ++q) ldmatrix_x4(src + (q * below + 16 * (j - k - 1)) * 32, bf[q]);
                    add_products<true>(acc.hi[2 * j], acc.hi[2 * j + 1], ah, bf);
                    if (j < kLo / 2 && j <= ilo) add_products<true>(acc.lo[2 * (j < kLo / 2 ? j : 0)], acc.lo[2 * (j < kLo / 2 ? j : 0) + 1], al, bf);
                }
            }
            __syncthreads();      // the parts have been read: the next panel takes their place
        }
    }
    __syncthreads();
    // back substitution, panel by panel from the last: what the solved rows below take off (column c = tid % 16, every eighth
    // row a thread), then the 16 x 16 triangle by the first warp
    const int c = lane & 15;
    int at[4];      // column c of a row r of a panel: r * 16 + at[(r / 2) % 4]
#pragma unroll
    for (int v = 0; v < 4; ++v) at[v] = 4 * ((c >> 2) ^ v) + (c & 3);
    const int at_mine = 4 * ((c >> 2) ^ warp) + (c & 3);      // ... of this thread's rows 16 + 2 warp + lane / 16 (+ 8, ...)
#pragma unroll 1
    for (int k = kBlocks - 1; k >= 0; --k) {
        const float *P = sm.L + panel_at(k);
        float s = 0.f;
#pragma unroll 4
        for (int r = 16 + (tid >> 4); r < D - 16 * k; r += 8) s = fmaf(P[r * 16 + at_mine], sm.b[16 * k + r], s);
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 16);
        if (lane < 16) sm.part[warp][lane] = s;
        __syncthreads();
        if (warp == 0) {
            float x = sm.z[16 * k + c] - ((sm.part[0][c] + sm.part[1][c]) + (sm.part[2][c] + sm.part[3][c]));
            const float d = sm.dinv[16 * k + c];
#pragma unroll
            for (int j = 15; j >= 0; --j) {
                const float xj = __shfl_sync(0xFFFFFFFFu, x * d, j);
                if (lane == 0) sm.b[16 * k + j] = xj;
                x = fmaf(-P[j * 16 + at[(j >> 1) & 3]], xj, x);      // (columns from j on are done with)
            }
        }
        __syncthreads();
    }
    return !__syncthreads_or(!(sm.dinv[tid] == sm.dinv[tid]));
}

__device__ __forceinline__ void store_row(const TeamSmem &sm, bool ok, int64_t u, const RowOut &out, DevStatus *st, int tid)
{
    const float v = ok ? sm.b[tid] : 0.f;
    reinterpret_cast<float *>(out.table)[u * D + tid] = v;
    if (out.cap_slot) {
        const int slot = out.cap_slot[u];
        if (slot >= 0) out.cap_out[(int64_t)slot * D + tid] = v;
    }
    if (!ok && tid == 0) {
        atomicAdd(&st->not_spd, 1ull);
        raise_flag(st, kFlagNotSpd, u);
    }
}

// ---- whole rows: a team each, items dealt round-robin, item 0 the last of the order (the longest class)
__global__ void __launch_bounds__(kTeam, kTeamsPerSm) k_rows_team(SideView sv, int64_t last, int64_t count, const int *dual_flag,
                                                                  int64_t primal_count, const float *__restrict__ X,
                                                                  const float *__restrict__ Bmat, RowOut out, DevStatus *st)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TeamSmem &sm = *reinterpret_cast<TeamSmem *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (dual_flag && *dual_flag) count = primal_count;      // the rows behind them have been solved in the dual form
    int64_t item = blockIdx.x;
    if (item >= count) return;
    Feed feed;
    feed.X = X;
    feed.idx = sv.idx;
    feed.val = sv.val;
    feed.g = 0;
    int64_t u = sv.order[last - item];
    int64_t len = sv.ptr[u + 1] - sv.ptr[u];
    feed.start_ids(sv.ptr[u], sv.ptr[u + 1], lane);
    feed.start_copies(sm, warp, lane);
    int64_t un = item + gridDim.x < count ? sv.order[last - item - gridDim.x] : -1;
    while (true) {
        const int64_t after = item + 2 * (int64_t)gridDim.x;
        const int64_t bn = un < 0 ? 0 : sv.ptr[un], en = un < 0 ? 0 : sv.ptr[un + 1];
        const int64_t ua = after < count ? sv.order[last - after] : -1;
        Acc acc;
        acc.zero();
        float b = 0.f;
        sum_entries(feed, len, sm, acc, b, warp, lane);
        // the next row's first entries travel while this one is solved
        if (un >= 0) feed.start_ids(bn, en, lane);
        sm.b[threadIdx.x] = b;
        if (un >= 0) feed.start_copies(sm, warp, lane);      // (its slot was last read a stage and a barrier ago)
        const bool ok = factor_solve(acc, sm, Bmat, warp, lane);
        store_row(sm, ok, u, out, st, threadIdx.x);
        if (un < 0) return;
        __syncthreads();
        item += gridDim.x;
        u = un;
        un = ua;
        len = en - bn;
    }
}

// ---- long rows and chunks of split rows: `slices` teams per row, their sums to the workspace in fragment order
__global__ void __launch_bounds__(kTeam, kTeamsPerSm) k_sums_team(SideView sv, int64_t last, int chunks, int slices, const float *__restrict__ X,
                                                                  float *__restrict__ sums)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TeamSmem &sm = *reinterpret_cast<TeamSmem *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t item = blockIdx.x / slices;
    const int slice = blockIdx.x % slices;
    int64_t beg, end;
    if (chunks) {
        beg = sv.chunk_desc[4 * item + 1];
        end = sv.chunk_desc[4 * item + 2];
    } else {
        const int64_t u = sv.order[last - item];
        beg = sv.ptr[u];
        end = sv.ptr[u + 1];
    }
    const int64_t per = (end - beg + (int64_t)slices * kEntries - 1) / ((int64_t)slices * kEntries) * kEntries;
    beg += slice * per;
    end = beg + per < end ? beg + per : end;
    Acc acc;
    acc.zero();
    float b = 0.f;
    if (beg < end) {
        Feed feed;
        feed.X = X;
        feed.idx = sv.idx;
        feed.val = sv.val;
        feed.g = 0;
        feed.start_ids(beg, end, lane);
        feed.start_copies(sm, warp, lane);
        sum_entries(feed, end - beg, sm, acc, b, warp, lane);
    }
    float *dst = sums + (int64_t)blockIdx.x * kSums;
    float4 *f = reinterpret_cast<float4 *>(dst) + warp * 18 * 32 + lane;      // 18 blocks a warp: row w's, then row 7 - w's
#pragma unroll
    for (int n = 0; n < kLo; ++n)
        if (n < 2 * (warp + 1)) f[n * 32] = make_float4(acc.lo[n][0], acc.lo[n][1], acc.lo[n][2], acc.lo[n][3]);
    f += 2 * (warp + 1) * 32;
#pragma unroll
    for (int n = 0; n < kHi; ++n)
        if (n < 2 * (kBlocks - warp)) f[n * 32] = make_float4(acc.hi[n][0], acc.hi[n][1], acc.hi[n][2], acc.hi[n][3]);
    dst[72 * 128 + threadIdx.x] = b;
}

// a team per row: its slices' sums (of its chunks, for a split row) in ascending order, then the solve
__global__ void __launch_bounds__(kTeam, kTeamsPerSm) k_solve_sums_team(SideView sv, int64_t first, int chunks, int slices,
                                                                        const float *__restrict__ sums, const float *__restrict__ Bmat,
                                                                        RowOut out, DevStatus *st)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TeamSmem &sm = *reinterpret_cast<TeamSmem *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t item = blockIdx.x;
    const int64_t u = chunks ? sv.order[first + item] : sv.order[first - item];
    const int64_t s0 = chunks ? sv.split_first[item] * slices : item * slices;
    const int64_t s1 = chunks ? sv.split_first[item + 1] * slices : s0 + slices;
    Acc acc;
    acc.zero();
    float b = 0.f;
    for (int64_t s = s0; s < s1; ++s) {
        const float *src = sums + s * kSums;
        const float4 *f = reinterpret_cast<const float4 *>(src) + warp * 18 * 32 + lane;
        auto add = [](float(&c)[4], const float4 &v) { c[0] += v.x; c[1] += v.y; c[2] += v.z; c[3] += v.w; };
#pragma unroll
        for (int n = 0; n < kLo; ++n)
            if (n < 2 * (warp + 1)) add(acc.lo[n], f[n * 32]);
        f += 2 * (warp + 1) * 32;
#pragma unroll
        for (int n = 0; n < kHi; ++n)
            if (n < 2 * (kBlocks - warp)) add(acc.hi[n], f[n * 32]);
        b += src[72 * 128 + threadIdx.x];
    }
    sm.b[threadIdx.x] = b;
    __syncthreads();
    const bool ok = factor_solve(acc, sm, Bmat, warp, lane);
    store_row(sm, ok, u, out, st, threadIdx.x);
}

__global__ void k_zero_rows_team(const int32_t *__restrict__ rows, int64_t count, RowOut out)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count * D) return;
    const int64_t u = rows[t / D];
    const int c = (int)(t % D);
    reinterpret_cast<float *>(out.table)[u * D + c] = 0.f;
    if (out.cap_slot) {
        const int slot = out.cap_slot[u];
        if (slot >= 0) out.cap_out[(int64_t)slot * D + c] = 0.f;
    }
}

// Rows of more than 1024 entries (classes 8 up) and chunks are cut into slices as long as that gives the chip no more than a
// block per team: a team alone takes 0.25 ms for 8192 entries.  1: not cut (long rows then go with the others).
int team_slices(int64_t items) { return items <= 0 ? 1 : items >= 148 * kTeamsPerSm / 2 ? 1 : (int)(148 * kTeamsPerSm / items < kMostSlices ? 148 * kTeamsPerSm / items : kMostSlices); }

}  // namespace

int64_t team_sums_floats(const int64_t *offs, int64_t n_chunks)
{
    const int64_t n_long = offs[kNClasses - 1] - offs[8];
    const int ls = team_slices(n_long);
    const int64_t a = n_chunks * team_slices(n_chunks), b = ls > 1 ? n_long * ls : 0;
    return (a > b ? a : b) * kSums;
}

cudaError_t launch_rows_team(const SideView &sv, const int64_t *offs, int64_t n_chunks, int64_t n_split_rows, const float *X, const float *Bmat,
                             float *sums, RowOut out, DevStatus *st, const int *dual_flag, cudaStream_t s, int64_t *launches)
{
    const size_t smem = sizeof(TeamSmem);
    cudaError_t e;
    static SmemOnce allow_rows, allow_sums, allow_solve;
    if ((e = allow_rows(k_rows_team, smem)) != cudaSuccess) return e;
    if ((e = allow_sums(k_sums_team, smem)) != cudaSuccess) return e;
    if ((e = allow_solve(k_solve_sums_team, smem)) != cudaSuccess) return e;
    if (n_chunks > 0) {
        const int slices = team_slices(n_chunks);
        k_sums_team<<<(unsigned)(n_chunks * slices), kTeam, smem, s>>>(sv, 0, 1, slices, X, sums);
        k_solve_sums_team<<<(unsigned)n_split_rows, kTeam, smem, s>>>(sv, offs[kNClasses - 1], 1, slices, sums, Bmat, out, st);
        *launches += 2;
    }
    const int64_t n_long = offs[kNClasses - 1] - offs[8];
    int64_t end = offs[kNClasses - 1];
    const int slices = team_slices(n_long);
    if (n_long > 0 && slices > 1) {
        k_sums_team<<<(unsigned)(n_long * slices), kTeam, smem, s>>>(sv, end - 1, 0, slices, X, sums);
        k_solve_sums_team<<<(unsigned)n_long, kTeam, smem, s>>>(sv, end - 1, 0, slices, sums, Bmat, out, st);
        *launches += 2;
        end = offs[8];
    }
    const int64_t n = end - offs[1];
    if (n > 0) {
        k_rows_team<<<(unsigned)(n < 148 * kTeamsPerSm ? n : 148 * kTeamsPerSm), kTeam, smem, s>>>(sv, end - 1, n, dual_flag, end - offs[2], X,
                                                                                                           Bmat, out, st);
        ++*launches;
    }
    const int64_t n_zero = offs[1] - offs[0];
    if (n_zero > 0) {
        k_zero_rows_team<<<(unsigned)((n_zero * D + 255) / 256), 256, 0, s>>>(sv.order + offs[0], n_zero, out);
        ++*launches;
    }
    return cudaGetLastError();
}

}  // namespace alx
