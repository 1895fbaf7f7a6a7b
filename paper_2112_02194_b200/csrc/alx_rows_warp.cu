// Row kernels of one half-epoch for d = 16, 32 and 64, either storage type: a warp per row, the matrix in registers.
//
// For each row u of the solved side (Alg. 1 lines 3-10, Eq. 4): gather, A = sum x (x) x and b = sum y x, add the base
// matrix, Cholesky, solve, round, store.  The FP32-ALU kernels (alx_rows.cu) give a row a block of 256 threads that meets at a
// barrier several times per 16 columns; at these d a row is a few thousand operations and the barriers were the run time
// (d = 64, bfloat16: 25 ns of the chip per row of 20 entries).  Here
//   - 16 entries at a time come through a two-stage cp.async ring of the warp's own; the next row's first entries are on their
//     way while the warp solves this one;
//   - the sums are mma.sync m16n8k16 products on the lower triangle's 16 x 8 blocks.  A gathered tile is both operands: one
//     ldmatrix.trans per 16 features gives the A fragment, and its registers are the B fragments of the same features.
//     bfloat16 tables: products exact, sums in fp32.  fp32 tables: x = x1 + x2 + x3 in bfloat16 parts, the six products down to
//     2^-24 (the scheme of the d = 64 tcgen05 path).  The warp-level instruction because a row's matrix is a fraction of a
//     tcgen05 tile: m16n8k16 runs at 1024 FMA per cycle and SM (measured, 550 TFLOP/s), which at these d leaves the sums
//     behind the solve, and the result is where the solve wants it, in the warp's registers;
//   - Cholesky with lane = row (d = 64: rows l and l + 32; d = 16: two matrices per warp), two columns per step, the finished
//     columns of L in shared memory: their broadcast reads drive the trailing update (packed FMAs), and the back
//     substitution reads them across.
// Rows of more than 256 entries, and the chunks of rows longer than `split`, are summed by a block of eight warps, each a
// slice of the entries; the slices are added in a fixed order.
//
// Bound: issue slots of the solve (d = 64: about 3400 per row) and, for long rows, the mma rate.
#include "alx_common.cuh"
#include "alx_ptx.cuh"

namespace alx {

namespace {

constexpr int kEntries = 16;       // entries per stage = the K of one mma
constexpr int kBlockWarps = 8;     // warps per row in the long-row kernels
constexpr int kLongClass = 6;      // degree classes from here on (more than 256 entries) go to the long-row kernel

template <int D, typename T> struct WGeo {
    static constexpr bool kF32 = sizeof(T) == 4;
    static constexpr int MB = D / 16;                       // 16-feature blocks
    static constexpr int NB = MB * (MB + 1);                // 16 x 8 blocks of the lower triangle: 2 (i + 1) per block row i
    static constexpr int PARTS = kF32 ? 3 : 1;
    static constexpr int PIECES = D * (int)sizeof(T) / 16;  // 16-byte pieces of a table row
    static constexpr int ROW = D * 2 + 16;                  // bytes between the rows of a bfloat16 tile (ldmatrix without conflicts)
    static constexpr int RAW = kF32 ? D * 4 : ROW;          // ... of a gathered stage
    static constexpr int STAGE = kEntries * RAW;
    static constexpr int TILE = kF32 ? 3 * kEntries * ROW : 0;      // bfloat16 parts of a stage
    static constexpr int ROWS = D == 16 ? 2 : 1;            // matrices a warp solves at a time
    // columns of L, four at a time from the diagonal block down; the stride of a group's columns is 4 mod 8 floats
    static constexpr int group_stride(int g) { return D - 4 * g + ((D / 4 - g) % 2 == 0 ? 4 : 0); }
    __host__ __device__ static constexpr int group_base(int g)
    {
        // sum of 4 * group_stride over the groups before g (D / 4 is even: the even ones are padded)
        return 4 * (D * g - 2 * g * (g - 1) + 4 * ((g + 1) / 2));
    }
    static constexpr int L_FLOATS = group_base(D / 4);
    static constexpr int T_FLOATS = (D < 32 ? D : 32) * ((D < 32 ? D : 32) + 4);      // transposition buffer of one matrix
    static constexpr int SOLVE = 4 * (ROWS * (L_FLOATS > T_FLOATS ? L_FLOATS : T_FLOATS) + ROWS * D);
    static constexpr int B_AT = ROWS * (L_FLOATS > T_FLOATS ? L_FLOATS : T_FLOATS);      // right-hand sides, behind the factor
    static constexpr int WORK = SOLVE;                      // the parts share the factor's place
    static_assert(TILE <= 4 * B_AT, "the parts leave the right-hand sides alone");
    static constexpr int WARP = 2 * STAGE + (WORK + 15) / 16 * 16;
    static constexpr int BASE = NB * 32 * 16;               // the base matrix in fragment order, per block
    static constexpr int REGS_WARPS = D == 64 ? 12 : 20;      // warps per SM
};

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// the sums of one row as the warp holds them: block (i, n), n < 2 (i + 1), is number i (i + 1) + n
template <int D, typename T> struct Sums {
    float c[WGeo<D, T>::NB][4];
    float b[2];      // features 2 f and 2 f + 1 of the right-hand side, f = lane % (D / 2)
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int n = 0; n < WGeo<D, T>::NB; ++n)
#pragma unroll
            for (int j = 0; j < 4; ++j) c[n][j] = 0.f;
        b[0] = b[1] = 0.f;
    }
};

// The warp's gather ring.  Stages are numbered through all rows; stage g lives in slot g % 2.
template <int D, typename T> struct Feed {
    using G = WGeo<D, T>;
    const T *X;
    const int32_t *idx;
    const float *val;
    uint32_t ring;      // shared address
    int g;              // next stage to be consumed
    // the row being fed: the stage after the one in flight has its ids in `id`, the one in flight its labels in y[]
    int64_t at, end;
    int id;
    float y, y_next;

    __device__ __forceinline__ void load_ids(int lane)
    {
        id = -1;
        y_next = 0.f;
        if (lane < kEntries && at + lane < end) {
            id = __ldg(idx + at + lane);
            y_next = val ? __ldg(val + at + lane) : 1.f;
        }
        at += kEntries;
    }
    __device__ __forceinline__ void issue(int slot, int lane)
    {
        const uint32_t dst = ring + (uint32_t)slot * G::STAGE;
#pragma unroll
        for (int k = 0; k < kEntries * G::PIECES / 32; ++k) {
            const int p = lane + 32 * k, r = p / G::PIECES, c = p % G::PIECES;
            const int row = __shfl_sync(0xFFFFFFFFu, id, r);
            cp_async16_zfill(dst + r * G::RAW + c * 16, X + (int64_t)(row < 0 ? 0 : row) * D + c * (16 / (int)sizeof(T)), row >= 0);
        }
        ptx::cp_async_commit();
    }
    // first stage of a row's entries [beg, e): ids, then its copies, then the ids of the second stage
    __device__ __forceinline__ void start(int64_t beg, int64_t e, int lane)
    {
        at = beg;
        end = e;
        load_ids(lane);
        y = y_next;
        issue(g & 1, lane);
        load_ids(lane);
    }
};

// Sums over the entries of the row that `feed` was started on.
template <int D, typename T>
__device__ __forceinline__ void sum_entries(Feed<D, T> &feed, int64_t len, unsigned char *smem_ring, unsigned char *tile, Sums<D, T> &acc, int lane)
{
    using G = WGeo<D, T>;
    constexpr int LP = D / 2, EP = 32 / LP;      // lanes per entry and entries side by side in the right-hand side's sums
    const int stages = (int)((len + kEntries - 1) / kEntries);
    for (int s = 0; s < stages; ++s) {
        const float y = feed.y;
        if (s + 1 < stages) {
            feed.y = feed.y_next;
            feed.issue((feed.g + 1) & 1, lane);
            feed.load_ids(lane);
            ptx::cp_async_wait<1>();
        } else {
            ptx::cp_async_wait<0>();
        }
        __syncwarp();
        const unsigned char *raw = smem_ring + (feed.g & 1) * G::STAGE;
        // right-hand side, and for fp32 tables the bfloat16 parts of the stage
#pragma unroll
        for (int e0 = 0; e0 < kEntries; e0 += EP) {
            const int e = e0 + lane / LP, f = lane % LP;
            const float ye = feed.val ? __shfl_sync(0xFFFFFFFFu, y, e) : 1.f;      // (entries past the end are zeros)
            if constexpr (G::kF32) {
                const float2 x = *reinterpret_cast<const float2 *>(raw + e * G::RAW + f * 8);
                acc.b[0] = fmaf(ye, x.x, acc.b[0]);
                acc.b[1] = fmaf(ye, x.y, acc.b[1]);
                const uint32_t p1 = pack_bf16(x.x, x.y);
                const float r0 = x.x - bf16_lo(p1), r1 = x.y - bf16_hi(p1);
                const uint32_t p2 = pack_bf16(r0, r1);
                const uint32_t p3 = pack_bf16(r0 - bf16_lo(p2), r1 - bf16_hi(p2));
                *reinterpret_cast<uint32_t *>(tile + e * G::ROW + f * 4) = p1;
                *reinterpret_cast<uint32_t *>(tile + (kEntries + e) * G::ROW + f * 4) = p2;
                *reinterpret_cast<uint32_t *>(tile + (2 * kEntries + e) * G::ROW + f * 4) = p3;
            } else {
                const uint32_t w = *reinterpret_cast<const uint32_t *>(raw + e * G::RAW + f * 4);
                acc.b[0] = fmaf(ye, bf16_lo(w), acc.b[0]);
                acc.b[1] = fmaf(ye, bf16_hi(w), acc.b[1]);
            }
        }
        if constexpr (G::kF32) __syncwarp();
        const uint32_t src = ptx::smem_u32(G::kF32 ? tile : raw) + ((lane & 7) + 8 * (lane >> 4)) * G::ROW + 16 * ((lane >> 3) & 1);
        uint32_t a[G::PARTS][G::MB][4];
#pragma unroll
        for (int p = 0; p < G::PARTS; ++p)
#pragma unroll
            for (int i = 0; i < G::MB; ++i) ldmatrix_x4_trans(src + p * kEntries * G::ROW + 32 * i, a[p][i]);
        // the parts' products from the smallest up
        constexpr int kPairs = G::kF32 ? 6 : 1;
        constexpr int pa[6] = {G::kF32 ? 2 : 0, 0, 1, 1, 0, 0}, pb[6] = {0, G::kF32 ? 2 : 0, 1, 0, 1, 0};
#pragma unroll
        for (int q = 0; q < kPairs; ++q)
#pragma unroll
            for (int i = 0; i < G::MB; ++i)
#pragma unroll
                for (int n = 0; n < 2 * (i + 1); ++n) {
                    const uint32_t(&bf)[4] = a[G::kF32 ? pb[q] : 0][n / 2];
                    mma_bf16(acc.c[i * (i + 1) + n], a[G::kF32 ? pa[q] : 0][i], bf[n % 2], bf[2 + n % 2]);
                }
        __syncwarp();      // the slot and the parts may be overwritten
        ++feed.g;
    }
#pragma unroll
    for (int o = LP; o < 32; o <<= 1) {
        acc.b[0] += __shfl_xor_sync(0xFFFFFFFFu, acc.b[0], o);
        acc.b[1] += __shfl_xor_sync(0xFFFFFFFFu, acc.b[1], o);
    }
}

__device__ __forceinline__ float rsqrt_full(float p)
{
    float inv = rsqrtf(p);
    return inv * fmaf(-0.5f * p * inv, inv, 1.5f);      // one Newton step: full fp32 accuracy
}

// Cholesky, forward and back substitution of the warp's matrix (two for d = 16, one per half-warp).  Lane: row r = lane % 32
// (% 16) in a0, row r + 32 in a1 for d = 64; b likewise.  L: the warp's columns in shared memory.  The solution replaces b.
// Returns whether every pivot was positive.
template <int D, typename T>
__device__ __forceinline__ bool factor_solve(float (&a0)[D < 32 ? D : 32], float (&a1)[D == 64 ? 64 : 1], float &b0, float &b1, float *L,
                                             int lane)
{
    using G = WGeo<D, T>;
    constexpr int H = D < 32 ? D : 32;
    const int r = lane & (H - 1);
    const int half = lane & ~(H - 1);      // first lane of this matrix
    bool ok = true;
    float d0 = 0.f, d1 = 0.f;              // reciprocal pivots of the lane's rows
#pragma unroll
    for (int j = 0; j < D; j += 2) {
        const int src = half + (j & (H - 1));
        float p, q, s, z0, z1;
        if (j < 32) {
            p = __shfl_sync(0xFFFFFFFFu, a0[j & (H - 1)], src);
            q = __shfl_sync(0xFFFFFFFFu, a0[j & (H - 1)], src + 1);
            s = __shfl_sync(0xFFFFFFFFu, a0[(j + 1) & (H - 1)], src + 1);
            z0 = __shfl_sync(0xFFFFFFFFu, b0, src);
            z1 = __shfl_sync(0xFFFFFFFFu, b0, src + 1);
        } else {
            p = __shfl_sync(0xFFFFFFFFu, a1[D == 64 ? j : 0], src);
            q = __shfl_sync(0xFFFFFFFFu, a1[D == 64 ? j : 0], src + 1);
            s = __shfl_sync(0xFFFFFFFFu, a1[D == 64 ? j + 1 : 0], src + 1);
            z0 = __shfl_sync(0xFFFFFFFFu, b1, src);
            z1 = __shfl_sync(0xFFFFFFFFu, b1, src + 1);
        }
        const float i0 = rsqrt_full(p), l10 = q * i0, dd = fmaf(-l10, l10, s), i1 = rsqrt_full(dd);
        ok = ok && p > 0.f && dd > 0.f;
        z0 *= i0;
        z1 = fmaf(-z0, l10, z1) * i1;
        float *c0 = L + G::group_base(j / 4) + (j % 4) * G::group_stride(j / 4) - 4 * (j / 4);
        float *c1 = c0 + G::group_stride(j / 4);
        float x00 = 0.f, x01 = 0.f, x10 = 0.f, x11 = 0.f;
        if (j < 32) {
            x00 = a0[j & (H - 1)] * i0;
            x01 = fmaf(-x00, l10, a0[(j + 1) & (H - 1)]) * i1;
            if (r >= 4 * (j / 4)) { c0[r] = x00; c1[r] = x01; }
            const float nb = fmaf(-x01, z1, fmaf(-x00, z0, b0));
            b0 = r > j + 1 ? nb : r == j ? z0 : r == j + 1 ? z1 : b0;
            d0 = r == j ? i0 : r == j + 1 ? i1 : d0;
        }
        if constexpr (D == 64) {
            x10 = a1[j] * i0;
            x11 = fmaf(-x10, l10, a1[j + 1]) * i1;
            if (j < 32 || r + 32 >= 4 * (j / 4)) { c0[r + 32] = x10; c1[r + 32] = x11; }
            const float nb = fmaf(-x11, z1, fmaf(-x10, z0, b1));
            b1 = r + 32 > j + 1 ? nb : r + 32 == j ? z0 : r + 32 == j + 1 ? z1 : b1;
            d1 = r + 32 == j ? i0 : r + 32 == j + 1 ? i1 : d1;
        }
        __syncwarp();
#pragma unroll
        for (int c = (j + 2) & ~3; c < D; c += 4) {
            const float4 u = *reinterpret_cast<const float4 *>(c0 + c), v = *reinterpret_cast<const float4 *>(c1 + c);
            const float2 m00 = make_float2(-x00, -x00), m01 = make_float2(-x01, -x01);
            const float2 m10 = make_float2(-x10, -x10), m11 = make_float2(-x11, -x11);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int cc = c + 2 * h;
                if (cc < j + 2) continue;
                const float2 uu = h ? make_float2(u.z, u.w) : make_float2(u.x, u.y), vv = h ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
                if (cc < 32) {
                    float2 t = make_float2(a0[cc & (H - 1)], a0[(cc + 1) & (H - 1)]);
                    t = __ffma2_rn(m01, vv, __ffma2_rn(m00, uu, t));
                    a0[cc & (H - 1)] = t.x;
                    a0[(cc + 1) & (H - 1)] = t.y;
                }
                if constexpr (D == 64) {
                    float2 t = make_float2(a1[cc], a1[cc + 1]);
                    t = __ffma2_rn(m11, vv, __ffma2_rn(m10, uu, t));
                    a1[cc] = t.x;
                    a1[cc + 1] = t.y;
                }
            }
        }
    }
    // back substitution, from the last column: x_j to everybody, then row i < j takes L[j][i] x_j off
    const int g0 = r / 4;
    const float *l0 = L + G::group_base(g0) + (r % 4) * (D - 4 * g0 + ((D / 4 - g0) % 2 == 0 ? 4 : 0)) - 4 * g0;
    if constexpr (D == 64) {
        const int g1 = (r + 32) / 4;
        const float *l1 = L + G::group_base(g1) + (r % 4) * (D - 4 * g1 + ((D / 4 - g1) % 2 == 0 ? 4 : 0)) - 4 * g1;
#pragma unroll 8
        for (int j = 63; j >= 32; --j) {
            const float x = __shfl_sync(0xFFFFFFFFu, b1 * d1, j - 32);
            const float m0 = l0[j], m1 = l1[j];
            b0 = fmaf(-m0, x, b0);
            b1 = r + 32 < j ? fmaf(-m1, x, b1) : r + 32 == j ? x : b1;
        }
    }
#pragma unroll 8
    for (int j = H - 1; j >= 0; --j) {
        const float x = __shfl_sync(0xFFFFFFFFu, b0 * d0, half + j);
        const float m0 = l0[j];
        b0 = r < j ? fmaf(-m0, x, b0) : r == j ? x : b0;
    }
    const unsigned bad = __ballot_sync(0xFFFFFFFFu, !ok);
    return D == 16 ? (bad >> half & 0xFFFFu) == 0 : bad == 0;
}

template <int D, typename T> __device__ __forceinline__ void put_b(const Sums<D, T> &acc, float *b_s, int lane)
{
    if (lane < D / 2) *reinterpret_cast<float2 *>(b_s + 2 * lane) = make_float2(acc.b[0], acc.b[1]);
    __syncwarp();
}

// adds the base matrix to the sums and hands the rows to their lanes through shared memory; matrix `which` of a d = 16 pair
template <int D, typename T>
__device__ __forceinline__ void place_rows(const Sums<D, T> &acc, const float4 *base, float *work, float (&a0)[D < 32 ? D : 32],
                                           float (&a1)[D == 64 ? 64 : 1], int which, int lane)
{
    using G = WGeo<D, T>;
    constexpr int H = D < 32 ? D : 32, S = H + 4;
    float *t = work + which * G::T_FLOATS;
    // passes of H rows x H columns: (rows 0..31), and for d = 64 (rows 32..63) x two halves of the columns
#pragma unroll
    for (int pass = 0; pass < (D == 64 ? 3 : 1); ++pass) {
        const int i0 = pass == 0 ? 0 : 2, n0 = pass == 2 ? 4 : 0;
#pragma unroll
        for (int i = i0; i < (D == 16 ? 1 : i0 + 2); ++i)
#pragma unroll
            for (int n = n0; n < n0 + H / 8; ++n)
                if (n < 2 * (i + 1)) {
                    const int blk = i * (i + 1) + n;
                    const float4 v = base[blk * 32 + lane];
                    float *dst = t + (16 * (i - i0) + lane / 4) * S + 8 * (n - n0) + 2 * (lane % 4);
                    *reinterpret_cast<float2 *>(dst) = make_float2(acc.c[blk][0] + v.x, acc.c[blk][1] + v.y);
                    *reinterpret_cast<float2 *>(dst + 8 * S) = make_float2(acc.c[blk][2] + v.z, acc.c[blk][3] + v.w);
                }
        __syncwarp();
        if (D != 16 || (lane >> 4) == which) {
            const float *row = t + (lane & (H - 1)) * S;
#pragma unroll
            for (int c = 0; c < H; c += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(row + c);
                if (pass == 0) {
                    a0[c] = v.x; a0[c + 1] = v.y; a0[c + 2] = v.z; a0[c + 3] = v.w;
                } else if constexpr (D == 64) {
                    const int o = 32 * (pass - 1) + c;
                    a1[o] = v.x; a1[o + 1] = v.y; a1[o + 2] = v.z; a1[o + 3] = v.w;
                }
            }
        }
        __syncwarp();
    }
}

template <int D, typename T>
__device__ __forceinline__ void store_row(float b0, float b1, bool ok, int64_t u, const RowOut &out, DevStatus *st, int lane)
{
    constexpr int H = D < 32 ? D : 32;
    const int r = lane & (H - 1);
    T *row = reinterpret_cast<T *>(out.table) + u * D;
    const float v0 = ok ? b0 : 0.f, v1 = ok ? b1 : 0.f;
    store_elem(row + r, v0);
    if (D == 64) store_elem(row + 32 + r, v1);
    if (out.cap_slot) {
        const int slot = out.cap_slot[u];
        if (slot >= 0) {
            out.cap_out[(int64_t)slot * D + r] = v0;
            if (D == 64) out.cap_out[(int64_t)slot * D + 32 + r] = v1;
        }
    }
    if (!ok && r == 0) {
        atomicAdd(&st->not_spd, 1ull);
        raise_flag(st, kFlagNotSpd, u);
    }
}

// the base matrix in the order of the mma fragments (block-wide)
template <int D, typename T> __device__ __forceinline__ void load_base(const float *__restrict__ Bmat, float4 *base)
{
    for (int e = threadIdx.x; e < WGeo<D, T>::NB * 32; e += blockDim.x) {
        const int blk = e / 32, lane = e % 32;
        int i = 0;
        while ((i + 1) * (i + 2) <= blk) ++i;
        const int row = 16 * i + lane / 4, col = 8 * (blk - i * (i + 1)) + 2 * (lane % 4);
        base[e] = make_float4(Bmat[row * D + col], Bmat[row * D + col + 1], Bmat[(row + 8) * D + col], Bmat[(row + 8) * D + col + 1]);
    }
}

// ---- rows of at most 256 entries: a warp each, items dealt round-robin (they are sorted by length class, so a warp's items
// are of all lengths); item 0 is the last of the order, i.e. of the longest class
template <int D, typename T>
__global__ void __launch_bounds__(WGeo<D, T>::REGS_WARPS * 32, 1)
k_rows_warp(SideView sv, int64_t last, int64_t count, const T *__restrict__ X, const float *__restrict__ Bmat, RowOut out, DevStatus *st)
{
    using G = WGeo<D, T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *base = reinterpret_cast<float4 *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *mine = smem_raw + G::BASE + warp * G::WARP;
    unsigned char *work = mine + 2 * G::STAGE;
    load_base<D, T>(Bmat, base);
    __syncthreads();
    const int64_t warps = (int64_t)gridDim.x * G::REGS_WARPS;
    int64_t item = ((int64_t)warp * gridDim.x + blockIdx.x) * G::ROWS;
    if (item >= count) return;
    Feed<D, T> feed;
    feed.X = X;
    feed.idx = sv.idx;
    feed.val = sv.val;
    feed.ring = ptx::smem_u32(mine);
    feed.g = 0;
    int64_t u = sv.order[last - item];
    int64_t beg = sv.ptr[u], end = sv.ptr[u + 1];
    feed.start(beg, end, lane);
    float *b_s = reinterpret_cast<float *>(work) + G::B_AT;
    while (true) {
        float a0[D < 32 ? D : 32], a1[D == 64 ? 64 : 1], b0 = 0.f, b1 = 0.f;
        int64_t u_pair = -1;
        const int64_t next = item + warps * G::ROWS;
        int64_t un = next < count ? sv.order[last - next] : -1, bn = 0, en = 0;
        {
            Sums<D, T> acc;
            acc.zero();
            sum_entries<D, T>(feed, end - beg, mine, work, acc, lane);
            if constexpr (D == 16) {
                put_b<D, T>(acc, b_s, lane);
                place_rows<D, T>(acc, base, reinterpret_cast<float *>(work), a0, a1, 0, lane);
                if (item + 1 < count) {
                    u_pair = sv.order[last - item - 1];
                    const int64_t b2 = sv.ptr[u_pair], e2 = sv.ptr[u_pair + 1];
                    feed.start(b2, e2, lane);
                    acc.zero();
                    sum_entries<D, T>(feed, e2 - b2, mine, work, acc, lane);
                }      // (a lone last row: the second matrix is the first one again, and is not stored)
                put_b<D, T>(acc, b_s + D, lane);
                place_rows<D, T>(acc, base, reinterpret_cast<float *>(work), a0, a1, 1, lane);
                b0 = b_s[lane];
            } else {
                put_b<D, T>(acc, b_s, lane);
                place_rows<D, T>(acc, base, reinterpret_cast<float *>(work), a0, a1, 0, lane);
                b0 = b_s[lane];
                if (D == 64) b1 = b_s[lane + 32];
            }
        }
        __syncwarp();
        // the next row's first entries travel while this one is solved
        if (un >= 0) {
            bn = sv.ptr[un];
            en = sv.ptr[un + 1];
            feed.start(bn, en, lane);
        }
        const bool ok = factor_solve<D, T>(a0, a1, b0, b1, reinterpret_cast<float *>(work) + (D == 16 ? (lane >> 4) * G::L_FLOATS : 0), lane);
        if (D != 16 || lane < 16) store_row<D, T>(b0, b1, ok, u, out, st, lane);
        else if (u_pair >= 0) store_row<D, T>(b0, b1, ok, u_pair, out, st, lane);
        if (un < 0) return;
        __syncwarp();
        item = next;
        u = un;
        beg = bn;
        end = en;
    }
}

// ---- longer rows and chunks of split rows: a block of eight warps, each a slice of the entries; the slices' sums are added in
// warp order.  A chunk's sums go to the workspace in fragment order ([NB x 128] and b); a row is solved by the first warp.
template <int D, typename T> struct BGeo {
    using G = WGeo<D, T>;
    static constexpr int SUMS = G::NB * 128 + D;      // floats
    static constexpr int FEED = kBlockWarps * (2 * G::STAGE + G::TILE);
    static constexpr int RED = kBlockWarps * SUMS * 4;
    static constexpr int SHARED = FEED > RED ? FEED : RED;
    static constexpr size_t SMEM = (size_t)G::BASE + G::WORK + SHARED + 16;
};

template <int D, typename T>
__device__ __forceinline__ void solve_sums(const float *sums, const float4 *base, float *work, int64_t u, const RowOut &out, DevStatus *st, int lane)
{
    using G = WGeo<D, T>;
    Sums<D, T> acc;
#pragma unroll
    for (int n = 0; n < G::NB; ++n) {
        const float4 v = *reinterpret_cast<const float4 *>(sums + (n * 32 + lane) * 4);
        acc.c[n][0] = v.x; acc.c[n][1] = v.y; acc.c[n][2] = v.z; acc.c[n][3] = v.w;
    }
    float a0[D < 32 ? D : 32], a1[D == 64 ? 64 : 1], b0, b1 = 0.f;
    for (int w = 0; w < G::ROWS; ++w) place_rows<D, T>(acc, base, work, a0, a1, w, lane);
    b0 = sums[G::NB * 128 + (lane & (D < 32 ? D - 1 : 31))];
    if (D == 64) b1 = sums[G::NB * 128 + 32 + lane];
    const bool ok = factor_solve<D, T>(a0, a1, b0, b1, work + (D == 16 ? (lane >> 4) * G::L_FLOATS : 0), lane);
    if (D != 16 || lane < 16) store_row<D, T>(b0, b1, ok, u, out, st, lane);
}

template <int D, typename T, bool CHUNK>
__global__ void __launch_bounds__(kBlockWarps * 32, 1)
k_rows_block(SideView sv, int64_t last, const T *__restrict__ X, const float *__restrict__ Bmat, float *__restrict__ partials, RowOut out,
             DevStatus *st)
{
    using G = WGeo<D, T>;
    using B = BGeo<D, T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *base = reinterpret_cast<float4 *>(smem_raw);
    float *work = reinterpret_cast<float *>(smem_raw + G::BASE);
    unsigned char *shared = smem_raw + G::BASE + G::WORK;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t u = 0, beg, end, slot = 0;
    if (CHUNK) {
        const int64_t *desc = sv.chunk_desc + (int64_t)blockIdx.x * 4;
        beg = desc[1]; end = desc[2]; slot = desc[3];
    } else {
        u = sv.order[last - blockIdx.x];
        beg = sv.ptr[u]; end = sv.ptr[u + 1];
        load_base<D, T>(Bmat, base);
    }
    const int64_t slice = (end - beg + kBlockWarps * kEntries - 1) / (kBlockWarps * kEntries) * kEntries;
    const int64_t my_beg = beg + warp * slice, my_end = my_beg + slice < end ? my_beg + slice : end;
    Sums<D, T> acc;
    acc.zero();
    if (my_beg < my_end) {
        unsigned char *mine = shared + warp * (2 * G::STAGE + G::TILE);
        Feed<D, T> feed;
        feed.X = X;
        feed.idx = sv.idx;
        feed.val = sv.val;
        feed.ring = ptx::smem_u32(mine);
        feed.g = 0;
        feed.start(my_beg, my_end, lane);
        sum_entries<D, T>(feed, my_end - my_beg, mine, mine + 2 * G::STAGE, acc, lane);
    }
    __syncthreads();
    float *red = reinterpret_cast<float *>(shared);
#pragma unroll
    for (int n = 0; n < G::NB; ++n)
        *reinterpret_cast<float4 *>(red + warp * B::SUMS + (n * 32 + lane) * 4) = make_float4(acc.c[n][0], acc.c[n][1], acc.c[n][2], acc.c[n][3]);
    if (lane < D / 2) {
        red[warp * B::SUMS + G::NB * 128 + 2 * lane] = acc.b[0];
        red[warp * B::SUMS + G::NB * 128 + 2 * lane + 1] = acc.b[1];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < B::SUMS; e += kBlockWarps * 32) {
        float s = red[e];
#pragma unroll
        for (int w = 1; w < kBlockWarps; ++w) s += red[w * B::SUMS + e];
        if (CHUNK) partials[slot * B::SUMS + e] = s;
        else red[e] = s;
    }
    if (CHUNK) return;
    __syncthreads();
    if (warp == 0) solve_sums<D, T>(red, base, work, u, out, st, lane);
}

// one warp per split row: its chunks' sums in ascending order, then the solve
template <int D, typename T>
__global__ void __launch_bounds__(32) k_split_solve_warp(SideView sv, int64_t split_begin, const float *__restrict__ partials,
                                                         const float *__restrict__ Bmat, RowOut out, DevStatus *st)
{
    using G = WGeo<D, T>;
    using B = BGeo<D, T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *base = reinterpret_cast<float4 *>(smem_raw);
    float *work = reinterpret_cast<float *>(smem_raw + G::BASE);
    float *sums = reinterpret_cast<float *>(smem_raw + G::BASE + G::WORK);
    const int lane = threadIdx.x;
    load_base<D, T>(Bmat, base);
    const int64_t u = sv.order[split_begin + blockIdx.x];
    const int64_t c0 = sv.split_first[blockIdx.x], c1 = sv.split_first[blockIdx.x + 1];
    for (int e = 4 * lane; e < B::SUMS; e += 128) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int64_t c = c0; c < c1; ++c) {
            const float4 v = *reinterpret_cast<const float4 *>(partials + c * B::SUMS + e);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *reinterpret_cast<float4 *>(sums + e) = s;
    }
    __syncwarp();
    solve_sums<D, T>(sums, base, work, u, out, st, lane);
}

// rows without observations: A^-1 0 = 0
template <typename T>
__global__ void k_zero_rows_warp(const int32_t *__restrict__ rows, int64_t count, int d, RowOut out)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count * d) return;
    const int64_t u = rows[t / d];
    const int c = (int)(t % d);
    store_elem(reinterpret_cast<T *>(out.table) + u * d + c, 0.f);
    if (out.cap_slot) {
        const int slot = out.cap_slot[u];
        if (slot >= 0) out.cap_out[(int64_t)slot * d + c] = 0.f;
    }
}

template <int D, typename T>
cudaError_t rows_warp_dt(const SideView &sv, const int64_t *offs, int64_t n_chunks, int64_t n_split_rows, const void *Xv, const float *Bmat,
                         float *partials, RowOut out, DevStatus *st, cudaStream_t s, int64_t *launches)
{
    using G = WGeo<D, T>;
    using B = BGeo<D, T>;
    static_assert(B::SUMS <= D * D + D, "a chunk's sums fit its place in the workspace");
    static_assert(B::SMEM <= 232448 && (size_t)G::BASE + G::REGS_WARPS * G::WARP <= 232448, "shared memory");
    const T *X = reinterpret_cast<const T *>(Xv);
    const size_t smem_warp = (size_t)G::BASE + G::REGS_WARPS * G::WARP;
    const size_t smem_split = (size_t)G::BASE + G::WORK + 4 * B::SUMS;
    cudaError_t e;
    // longest work first
    if (n_chunks > 0) {
        if ((e = cudaFuncSetAttribute(k_rows_block<D, T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)B::SMEM)) != cudaSuccess) return e;
        k_rows_block<D, T, true><<<(unsigned)n_chunks, kBlockWarps * 32, B::SMEM, s>>>(sv, 0, X, Bmat, partials, out, st);
        k_split_solve_warp<D, T><<<(unsigned)n_split_rows, 32, smem_split, s>>>(sv, offs[kNClasses - 1], partials, Bmat, out, st);
        *launches += 2;
    }
    const int64_t n_long = offs[kNClasses - 1] - offs[kLongClass];
    if (n_long > 0) {
        if ((e = cudaFuncSetAttribute(k_rows_block<D, T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)B::SMEM)) != cudaSuccess) return e;
        k_rows_block<D, T, false><<<(unsigned)n_long, kBlockWarps * 32, B::SMEM, s>>>(sv, offs[kNClasses - 1] - 1, X, Bmat, partials, out, st);
        ++*launches;
    }
    const int64_t n_warp = offs[kLongClass] - offs[1];
    if (n_warp > 0) {
        if ((e = cudaFuncSetAttribute(k_rows_warp<D, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_warp)) != cudaSuccess) return e;
        const int64_t per_warp = G::ROWS, blocks = (n_warp + per_warp - 1) / per_warp;      // few rows: one per SM before two
        k_rows_warp<D, T><<<(unsigned)(blocks < 148 ? blocks : 148), G::REGS_WARPS * 32, smem_warp, s>>>(sv, offs[kLongClass] - 1, n_warp, X,
                                                                                                       Bmat, out, st);
        ++*launches;
    }
    const int64_t n_zero = offs[1] - offs[0];
    if (n_zero > 0) {
        k_zero_rows_warp<T><<<(unsigned)((n_zero * D + 255) / 256), 256, 0, s>>>(sv.order + offs[0], n_zero, D, out);
        ++*launches;
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rows_warp(const SideView &sv, const int64_t *offs, int64_t n_chunks, int64_t n_split_rows, const void *X, int bf16, int d,
                             const float *Bmat, float *partials, RowOut out, DevStatus *st, cudaStream_t s, int64_t *launches)
{
#define ALX_CASE(DD)                                                                                                                      case DD:                                                                                                                                  return bf16 ? rows_warp_dt<DD, __nv_bfloat16>(sv, offs, n_chunks, n_split_rows, X, Bmat, partials, out, st, s, launches)                          : rows_warp_dt<DD, float>(sv, offs, n_chunks, n_split_rows, X, Bmat, partials, out, st, s, launches);
    switch (d) {
        ALX_CASE(16)
        ALX_CASE(32)
        ALX_CASE(64)
    default: return cudaErrorInvalidValue;
    }
#undef ALX_CASE
}

}  // namespace alx
