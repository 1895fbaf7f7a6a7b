// Row kernels of one half-epoch for d = 16, 32 and 64, either storage type: a warp per row, the matrix in registers.
//
// For each row u of the solved side (Alg. 1 lines 3-10, Eq. 4): gather, A = sum x (x) x and b = sum y x, add the base
// matrix, Cholesky, solve, round, store.  The FP32-ALU kernels (alx_rows.cu) give a row a block of 256 threads that meets at a
// barrier several times per 16 columns; at these d a row is a few thousand operations and the barriers were the run time
// (d = 64, bfloat16: 25 ns of the chip per row of 20 entries, here 6).  Here
//   - 16 entries at a time come through a two-stage cp.async ring of the warp's own; the next row's first entries are on their
//     way while the warp solves this one;
//   - the sums are mma.sync m16n8k16 products on the lower triangle's 16 x 8 blocks.  A gathered tile is both operands: one
//     ldmatrix.trans per 16 features gives the A fragment, and its registers are the B fragments of the same features.
//     bfloat16 tables: products exact, sums in fp32.  fp32 tables: x = x1 + x2 + x3 in bfloat16 parts, the six products down to
//     2^-24.  The warp-level instruction because a row's matrix is a fraction of a
//     tcgen05 tile: m16n8k16 runs at 1024 FMA per cycle and SM (measured, 550 TFLOP/s), which at these d leaves the sums
//     behind the solve, and the result is where the solve wants it, in the warp's registers;
//   - Cholesky with lane = row (d = 64: rows l and l + 32; d = 16: two matrices per warp), two columns per step, the finished
//     columns of L in shared memory: their broadcast reads drive the trailing update (packed FMAs), and the back
//     substitution reads them across.
// Long rows (warp_long_class), and the chunks of rows longer than `split`, are summed by a block of warps, each a slice of the
// entries; the slices are added in a fixed order.
//
// fp32 tables of 64 features with conjugate gradients: k_rows_cg64, the same over a table of the bfloat16 parts.
//
// Bound: issue slots of the solve (d = 64: about 3000 per row) and, for long rows, the mma rate.
#include "alx_common.cuh"
#include "alx_mma.cuh"
#include "alx_ptx.cuh"

namespace alx {

namespace {

constexpr int kEntries = 16;       // entries per stage = the K of one mma

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
    // panel k of L: rows 16 k .. D - 1, 16 columns, 64 bytes a row.  The bfloat16 parts of a panel lie where later panels
    // will: 3 x (rows below the diagonal block) x 32 bytes, which only the last but one panel has too little room for
    __host__ __device__ static constexpr int panel_at(int k) { return 16 * (16 * MB * k - 8 * k * (k - 1)); }      // floats
    static constexpr int L_FLOATS = panel_at(MB) + (MB > 1 ? 128 : 0);
    static constexpr int B_AT = 4 * ROWS * L_FLOATS > TILE ? ROWS * L_FLOATS : TILE / 4;      // right-hand sides, reciprocal pivots
    static constexpr int SOLVE = 4 * (B_AT + 2 * ROWS * D);
    static constexpr int WORK = SOLVE;                      // the parts of a gathered stage share the factor's place
    static constexpr int WARP = 2 * STAGE + (WORK + 15) / 16 * 16;
    static constexpr int BASE = NB * 32 * 16;               // the base matrix in fragment order, per block
    static constexpr int REGS_WARPS = D == 64 ? (kF32 ? 11 : 12) : 20;      // warps per SM
};

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
    // a row's entries [beg, e): the loads of the ids of its first two stages ...
    int id_first;
    __device__ __forceinline__ void start_ids(int64_t beg, int64_t e, int lane)
    {
        at = beg;
        end = e;
        load_ids(lane);
        y = y_next;
        id_first = id;
        load_ids(lane);
    }
    // ... and, later, the copies of the first stage
    __device__ __forceinline__ void start_copies(int lane)
    {
        const int second = id;
        id = id_first;
        issue(g & 1, lane);
        id = second;
    }
    __device__ __forceinline__ void start(int64_t beg, int64_t e, int lane)
    {
        start_ids(beg, e, lane);
        start_copies(lane);
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
        // the parts' products from the smallest up, each stage's from zero: the accumulator of an mma truncates, and adding up a
        // whole row in it biases long rows by 1e-5 (the final sums are ordinary FADDs)
        constexpr int kPairs = G::kF32 ? 6 : 1;
        constexpr int pa[6] = {G::kF32 ? 2 : 0, 0, 1, 1, 0, 0}, pb[6] = {0, G::kF32 ? 2 : 0, 1, 0, 1, 0};
#pragma unroll
        for (int i = 0; i < G::MB; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                float t[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                for (int q = 0; q < kPairs; ++q) {
                    const uint32_t(&bf)[4] = a[G::kF32 ? pb[q] : 0][j];
                    mma_bf16(t[0], a[G::kF32 ? pa[q] : 0][i], bf[0], bf[2]);
                    mma_bf16(t[1], a[G::kF32 ? pa[q] : 0][i], bf[1], bf[3]);
                }
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc.c[i * (i + 1) + 2 * j + n][e] += t[n][e];
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

// Cholesky, forward and back substitution of the warp's matrix: the sums in acc (lower triangle, base matrix added), the
// right-hand side in b_s; the solution replaces b_s.  Blocked, 16 columns per panel: the panel goes through shared memory to
// lane = row (rows l and l + 32 below the diagonal block's first), is factored there two columns per step, stays in shared
// memory as part of L and, in three bfloat16 parts, is both operands of the trailing update: the blocks of the matrix never
// leave the mma fragments.  (With the whole matrix in lane = row, every column of L had to be read by every lane: 2200
// shared-memory wavefronts per 64 x 64 matrix, 85 % of that pipe.)  d = 16: two matrices, one per half-warp, `acc2` the second.
template <int D, typename T>
__device__ __forceinline__ bool factor_solve(Sums<D, T> &acc, Sums<D, T> &acc2, float *L, float *b_s, int lane)
{
    using G = WGeo<D, T>;
    constexpr int MB = G::MB;
    float *dinv_s = b_s + G::ROWS * D;
    const int half = D == 16 ? lane & 16 : 0;      // first lane of this lane's matrix
    const int rl = D == 16 ? lane & 15 : lane;
    float *b_m = b_s + half;                       // d = 16: 16 floats a matrix
    float *dinv_m = dinv_s + half;
    const bool first = rl == 0;                    // the lane that writes down what all lanes of the matrix know
    auto put_block = [&](float *P, const float(&c)[4], int i, int n) {      // block (16 i .., 8 n ..) of the panel
        const int r = 16 * i + lane / 4, q = 2 * n + (lane % 4) / 2, o = 2 * (lane & 1);
        *reinterpret_cast<float2 *>(P + panel_chunk(r, q) + o) = make_float2(c[0], c[1]);
        *reinterpret_cast<float2 *>(P + panel_chunk(r + 8, q) + o) = make_float2(c[2], c[3]);
    };
#pragma unroll 1
    for (int k = 0; k < MB; ++k) {
        float *P = L + G::panel_at(k);
        const int rows = D - 16 * k;
        // the panel's blocks to shared memory
#pragma unroll
        for (int kk = 0; kk < MB; ++kk)
            if (kk == k) {
#pragma unroll
                for (int i = kk; i < MB; ++i)
#pragma unroll
                    for (int n = 0; n < 2; ++n) put_block(P, acc.c[i * (i + 1) + 2 * kk + n], i - kk, n);
            }
        if (D == 16) {
            put_block(L + G::L_FLOATS, acc2.c[0], 0, 0);
            put_block(L + G::L_FLOATS, acc2.c[1], 0, 1);
        }
        __syncwarp();
        float *Pm = D == 16 ? L + (half ? G::L_FLOATS : 0) : P;
        const bool two = D == 64 && lane + 32 < rows;
        float a0[16], a1[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float4 v = *reinterpret_cast<const float4 *>(Pm + panel_chunk(rl < rows ? rl : 0, c));
            a0[4 * c] = v.x; a0[4 * c + 1] = v.y; a0[4 * c + 2] = v.z; a0[4 * c + 3] = v.w;
            if (D == 64) {
                const float4 w = *reinterpret_cast<const float4 *>(Pm + panel_chunk(two ? rl + 32 : 0, c));
                a1[4 * c] = w.x; a1[4 * c + 1] = w.y; a1[4 * c + 2] = w.z; a1[4 * c + 3] = w.w;
            }
        }
        float b0 = rl < rows ? b_m[16 * k + rl] : 0.f, b1 = two ? b_m[16 * k + 32 + rl] : 0.f;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            const float p = __shfl_sync(0xFFFFFFFFu, a0[j], half + j), q = __shfl_sync(0xFFFFFFFFu, a0[j], half + j + 1);
            const float s = __shfl_sync(0xFFFFFFFFu, a0[j + 1], half + j + 1);
            float z0 = __shfl_sync(0xFFFFFFFFu, b0, half + j), z1 = __shfl_sync(0xFFFFFFFFu, b0, half + j + 1);
            // (a pivot that is not positive makes its reciprocal root a NaN, and is reported for that at the end)
            const float i0 = rsqrt_full(p), l10 = q * i0, dd = fmaf(-l10, l10, s), i1 = rsqrt_full(dd);
            z0 *= i0;
            z1 = fmaf(-z0, l10, z1) * i1;
            if (first) {
                *reinterpret_cast<float2 *>(b_m + 16 * k + j) = make_float2(z0, z1);
                *reinterpret_cast<float2 *>(dinv_m + 16 * k + j) = make_float2(i0, i1);
            }
            const float x0 = a0[j] * i0, x1 = fmaf(-x0, l10, a0[j + 1]) * i1;
            a0[j] = x0;
            a0[j + 1] = x1;
            b0 = fmaf(-x1, z1, fmaf(-x0, z0, b0));      // (what it becomes in the rows up to j + 1 is not used)
            float y0 = 0.f, y1 = 0.f;
            if (D == 64) {
                y0 = a1[j] * i0;
                y1 = fmaf(-y0, l10, a1[j + 1]) * i1;
                a1[j] = y0;
                a1[j + 1] = y1;
                b1 = fmaf(-y1, z1, fmaf(-y0, z0, b1));
            }
            if (j < 14) {
                // the two columns of the diagonal block's rows to everybody: the place of the panel's first two rows serves
                // as the exchange (its rows are in registers)
                float *ex = Pm + 32 * ((j / 2) & 1);
                if (rl < 16) { ex[rl] = -x0; ex[16 + rl] = -x1; }
                __syncwarp();
#pragma unroll
                for (int c = (j + 2) & ~3; c < 16; c += 4) {
                    const float4 u = *reinterpret_cast<const float4 *>(ex + c), v = *reinterpret_cast<const float4 *>(ex + 16 + c);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int cc = c + 2 * h;
                        if (cc < j + 2) continue;
                        const float2 uu = h ? make_float2(u.z, u.w) : make_float2(u.x, u.y), vv = h ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
                        float2 t = make_float2(a0[cc], a0[cc + 1]);
                        t = __ffma2_rn(make_float2(x1, x1), vv, __ffma2_rn(make_float2(x0, x0), uu, t));
                        a0[cc] = t.x;
                        a0[cc + 1] = t.y;
                        if (D == 64) {
                            float2 w = make_float2(a1[cc], a1[cc + 1]);
                            w = __ffma2_rn(make_float2(y1, y1), vv, __ffma2_rn(make_float2(y0, y0), uu, w));
                            a1[cc] = w.x;
                            a1[cc + 1] = w.y;
                        }
                    }
                }
            }
        }
        __syncwarp();
        // L's rows back, and the right-hand side of the rows below the diagonal block
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (rl < rows) *reinterpret_cast<float4 *>(Pm + panel_chunk(rl, c)) = make_float4(a0[4 * c], a0[4 * c + 1], a0[4 * c + 2], a0[4 * c + 3]);
            if (two) *reinterpret_cast<float4 *>(Pm + panel_chunk(rl + 32, c)) = make_float4(a1[4 * c], a1[4 * c + 1], a1[4 * c + 2], a1[4 * c + 3]);
        }
        if (rl >= 16 && rl < rows) b_m[16 * k + rl] = b0;
        if (two) b_m[16 * k + 32 + rl] = b1;
        if (D > 16 && k + 1 < MB) {
            // the rows below the diagonal block as bfloat16 parts, [part][row][16 columns]: 32-byte rows, the two 16-byte
            // chunks exchanged in every other group of four rows (ldmatrix without conflicts)
            unsigned char *tile = reinterpret_cast<unsigned char *>(L + G::panel_at(k + 1));
            const int below = rows - 16;
            auto put_parts = [&](const float(&x)[16], int r) {      // r: row below the diagonal block
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t p[3][4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float u = x[8 * c + 2 * e], v = x[8 * c + 2 * e + 1];
                        p[0][e] = pack_bf16(u, v);
                        const float u1 = u - bf16_lo(p[0][e]), v1 = v - bf16_hi(p[0][e]);
                        p[1][e] = pack_bf16(u1, v1);
                        p[2][e] = pack_bf16(u1 - bf16_lo(p[1][e]), v1 - bf16_hi(p[1][e]));
                    }
#pragma unroll
                    for (int part = 0; part < 3; ++part)
                        *reinterpret_cast<uint4 *>(tile + (part * below + r) * 32 + 16 * (c ^ ((r >> 2) & 1))) =
                            make_uint4(p[part][0], p[part][1], p[part][2], p[part][3]);
                }
            };
            if (rl >= 16 && rl < rows) put_parts(a0, rl - 16);
            if (two) put_parts(a1, rl + 16);
            __syncwarp();
            // trailing update of the blocks (i, n), i > k, n >= 2 (k + 1)
            const int lr = (lane & 7) + 8 * ((lane >> 3) & 1);
            const uint32_t src = ptx::smem_u32(tile) + lr * 32 + 16 * ((lane >> 4) ^ ((lr >> 2) & 1));
#pragma unroll
            for (int kk = 0; kk + 1 < MB; ++kk)
                if (kk == k) {
                    constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
                    uint32_t f[3][MB][4];
#pragma unroll
                    for (int part = 0; part < 3; ++part)
#pragma unroll
                        for (int i = kk + 1; i < MB; ++i) ldmatrix_x4(src + (part * (D - 16 * (kk + 1)) + 16 * (i - kk - 1)) * 32, f[part][i]);
#pragma unroll
                    for (int i = kk + 1; i < MB; ++i)
#pragma unroll
                        for (int j = kk + 1; j <= i; ++j) {
                            float t[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                            for (int q = 0; q < 6; ++q) {
                                mma_bf16(t[0], f[pa[q]][i], f[pb[q]][j][0], f[pb[q]][j][2]);
                                mma_bf16(t[1], f[pa[q]][i], f[pb[q]][j][1], f[pb[q]][j][3]);
                            }
#pragma unroll
                            for (int n = 0; n < 2; ++n)
#pragma unroll
                                for (int e = 0; e < 4; ++e) acc.c[i * (i + 1) + 2 * j + n][e] -= t[n][e];
                        }
                }
        }
        __syncwarp();
    }
    // back substitution, panel by panel from the last: what the solved rows below take off (lanes: column c, rows of one
    // parity), then the 16 x 16 triangle
    const int c = lane & 15;
    int at[4];      // column c of a row r of a panel: r * 16 + at[(r / 2) % 4]
#pragma unroll
    for (int v = 0; v < 4; ++v) at[v] = 4 * ((c >> 2) ^ v) + (c & 3);
    bool bad = false;
#pragma unroll 1
    for (int k = MB - 1; k >= 0; --k) {
        const float *Pm = D == 16 ? L + (half ? G::L_FLOATS : 0) : L + G::panel_at(k);
        float s = 0.f;
        if (D > 16) {
            const float *row = Pm + (16 + (lane >> 4)) * 16, *xs = b_s + 16 * k + 16 + (lane >> 4);
#pragma unroll 1
            for (int r = 16; r < D - 16 * k; r += 8, row += 128, xs += 8)
#pragma unroll
                for (int v = 0; v < 4; ++v) s = fmaf(row[32 * v + at[v]], xs[2 * v], s);
            s += __shfl_xor_sync(0xFFFFFFFFu, s, 16);
        }
        float x = b_m[16 * k + c] - s;
        const float d = dinv_m[16 * k + c];
        bad |= !(d == d);
        __syncwarp();
#pragma unroll
        for (int j = 15; j >= 0; --j) {
            const float xj = __shfl_sync(0xFFFFFFFFu, x * d, half + j);
            if (first) b_m[16 * k + j] = xj;
            x = fmaf(-Pm[j * 16 + at[(j >> 1) & 3]], xj, x);      // (columns from j on are done with)
        }
        __syncwarp();
    }
    const unsigned who = __ballot_sync(0xFFFFFFFFu, bad);
    return D == 16 ? (who >> half & 0xFFFFu) == 0 : who == 0;
}

template <int D, typename T> __device__ __forceinline__ void put_b(const Sums<D, T> &acc, float *b_s, int lane)
{
    if (lane < D / 2) *reinterpret_cast<float2 *>(b_s + 2 * lane) = make_float2(acc.b[0], acc.b[1]);
    __syncwarp();
}

template <int D, typename T> __device__ __forceinline__ void add_base(Sums<D, T> &acc, const float4 *base, int lane)
{
#pragma unroll
    for (int n = 0; n < WGeo<D, T>::NB; ++n) {
        const float4 v = base[n * 32 + lane];
        acc.c[n][0] += v.x; acc.c[n][1] += v.y; acc.c[n][2] += v.z; acc.c[n][3] += v.w;
    }
}

// ---- conjugate gradients (Sec. 4.5): fp32 tables of 64 features with ALX_SOLVER_AUTO
struct WarpCg {
    int max_iter, warm;                // step limit; start from the stored embedding
    float tol2;
    unsigned long long *counters;      // rows, products, rows left to the Cholesky kernel (nullptr: Cholesky for every row)
    int32_t *fallback_list;
};
constexpr int kCgVerifyProducts = 24;

// sums over the warp of two values, to every lane: six shuffles
__device__ __forceinline__ void warp_sums(float &a, float &b, int lane)
{
    const bool up = (lane & 16) != 0;
    float t = (up ? b : a) + __shfl_xor_sync(0xFFFFFFFFu, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    const float other = __shfl_xor_sync(0xFFFFFFFFu, t, 16);
    a = up ? other : t;
    b = up ? t : other;
}

// the warp's 64 x 64 matrix (lower triangle in mma fragments) to lane = rows l and l + 32, whole rows, quadrant by quadrant
// through shared memory (t: 32 x 36 floats)
__device__ __forceinline__ void symmetric_rows(const Sums<64, float> &acc, float *t, float (&a0)[64], float (&a1)[64], int lane)
{
    constexpr int S = 36;
    const int r = lane / 4, q = 2 * (lane % 4);
#pragma unroll
    for (int pass = 0; pass < 3; ++pass) {      // rows 0..31 x columns 0..31; rows 32..63 x columns 0..31; rows and columns 32..63
        const int i0 = pass == 0 ? 0 : 2, n0 = pass == 2 ? 4 : 0;
#pragma unroll
        for (int i = i0; i < i0 + 2; ++i)
#pragma unroll
            for (int n = n0; n < n0 + 4; ++n)
                if (n < 2 * (i + 1)) {
                    const float(&c)[4] = acc.c[i * (i + 1) + n];
                    const int row = 16 * (i - i0) + r, col = 8 * (n - n0) + q;
                    *reinterpret_cast<float2 *>(t + row * S + col) = make_float2(c[0], c[1]);
                    *reinterpret_cast<float2 *>(t + (row + 8) * S + col) = make_float2(c[2], c[3]);
                    if (pass != 1 && i == i0 + 1 && n < n0 + 2) {      // the block above the diagonal is this one's transpose
                        t[col * S + row] = c[0];
                        t[(col + 1) * S + row] = c[1];
                        t[col * S + row + 8] = c[2];
                        t[(col + 1) * S + row + 8] = c[3];
                    }
                }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(t + lane * S + c);
            float *a = pass == 0 ? a0 + c : pass == 1 ? a1 + c : a1 + 32 + c;
            a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w;
        }
        if (pass == 1) {
#pragma unroll
            for (int c = 0; c < 32; ++c) a0[32 + c] = t[c * S + lane];
        }
        __syncwarp();
    }
}

// Single-reduction conjugate gradients (Chronopoulos-Gear): one product w = A r and one pair of sums (r.r, r.w) per step.
// x: the lane's two components of the start vector, then of the solution.  vec: 64 floats of shared memory.  Returns whether
// |r| <= tol |b| was reached; after many products the true residual is looked at once (the recurrence's can drift).
__device__ __forceinline__ bool conjugate_gradients(const WarpCg &cg, const float (&a0)[64], const float (&a1)[64], float *vec, float b0, float b1,
                                                    float &x0, float &x1, int &products, int lane)
{
    auto product = [&](float v0, float v1, float &w0, float &w1) {
        __syncwarp();
        vec[lane] = v0;
        vec[lane + 32] = v1;
        __syncwarp();
        float2 s0 = make_float2(0.f, 0.f), s1 = s0, t0 = s0, t1 = s0;
#pragma unroll
        for (int c = 0; c < 64; c += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(vec + c);
            const float2 lo = make_float2(v.x, v.y), hi = make_float2(v.z, v.w);
            s0 = __ffma2_rn(make_float2(a0[c], a0[c + 1]), lo, s0);
            s1 = __ffma2_rn(make_float2(a0[c + 2], a0[c + 3]), hi, s1);
            t0 = __ffma2_rn(make_float2(a1[c], a1[c + 1]), lo, t0);
            t1 = __ffma2_rn(make_float2(a1[c + 2], a1[c + 3]), hi, t1);
        }
        w0 = (s0.x + s0.y) + (s1.x + s1.y);
        w1 = (t0.x + t0.y) + (t1.x + t1.y);
        ++products;
    };
    bool warm = cg.warm != 0;
    float w0, w1, r0 = b0, r1 = b1, p0 = 0.f, p1 = 0.f, s0 = 0.f, s1 = 0.f;
    float bb = b0 * b0 + b1 * b1, unused = 0.f;
    warp_sums(bb, unused, lane);
    if (warm) {                 // r = b - A x0
        product(x0, x1, w0, w1);
        r0 = b0 - w0;
        r1 = b1 - w1;
    } else {
        x0 = x1 = 0.f;
    }
    float rg_old = 0.f, inv_alpha_old = 0.f;
    bool ok = false;
    for (int it = 0;; ++it) {
        product(r0, r1, w0, w1);
        float g = r0 * r0 + r1 * r1, dl = r0 * w0 + r1 * w1;
        warp_sums(g, dl, lane);
        if (it == 0 && warm && !(g <= bb)) {
            // the start vector is further from the solution than zero is: start again from zero
            warm = false;
            x0 = x1 = 0.f;
            r0 = b0;
            r1 = b1;
            it = -1;
            continue;
        }
        if (g <= cg.tol2 * bb) { ok = true; break; }        // (also b = 0: x = 0)
        if (it >= cg.max_iter) break;
        const float rg = __fdividef(1.f, g);
        const float beta = g * rg_old;                           // 0 at the first step
        const float inv_alpha = dl * rg - beta * inv_alpha_old;  // p.A p / |r|^2
        if (!(inv_alpha > 0.f) || !(inv_alpha <= 3.0e38f)) break;
        const float alpha = __fdividef(1.f, inv_alpha);
        p0 = fmaf(beta, p0, r0);
        p1 = fmaf(beta, p1, r1);
        s0 = fmaf(beta, s0, w0);
        s1 = fmaf(beta, s1, w1);
        x0 = fmaf(alpha, p0, x0);
        x1 = fmaf(alpha, p1, x1);
        r0 = fmaf(-alpha, s0, r0);
        r1 = fmaf(-alpha, s1, r1);
        rg_old = rg;
        inv_alpha_old = inv_alpha;
    }
    if (ok && products >= kCgVerifyProducts) {
        product(x0, x1, w0, w1);
        float t = (b0 - w0) * (b0 - w0) + (b1 - w1) * (b1 - w1);
        unused = 0.f;
        warp_sums(t, unused, lane);
        ok = t <= 4.f * cg.tol2 * bb;
    }
    return ok;
}

template <int D, typename T>
__device__ __forceinline__ void store_row(const float *x, bool ok, int64_t u, const RowOut &out, DevStatus *st, int lane)
{
    constexpr int H = D < 32 ? D : 32;
    const int r = lane & (H - 1);
    T *row = reinterpret_cast<T *>(out.table) + u * D;
    const float v0 = ok ? x[r] : 0.f, v1 = D == 64 && ok ? x[D == 64 ? r + 32 : 0] : 0.f;
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

// rows without observations: A^-1 0 = 0 (grid-wide)
struct ZeroRows {
    const int32_t *rows;
    int64_t count;
};
template <int D, typename T> __device__ __forceinline__ void store_zeros(const ZeroRows &zero, const RowOut &out)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < zero.count * D; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = zero.rows[t / D];
        const int c = (int)(t % D);
        store_elem(reinterpret_cast<T *>(out.table) + u * D + c, 0.f);
        if (out.cap_slot) {
            const int slot = out.cap_slot[u];
            if (slot >= 0) out.cap_out[(int64_t)slot * D + c] = 0.f;
        }
    }
}

// The launch before this one may still run (programmatic dependent launch: it solves other rows).  The last thing a block does
// is wait for it, so that whatever follows this grid follows both; then the time is noted.
__device__ __forceinline__ void finish_after_previous(unsigned long long *done)
{
    wait_for_previous();
    stamp(done);
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

// ---- rows up to the long ones: a warp each, items dealt round-robin (they are sorted by length class, so a warp's items
// are of all lengths); item 0 is the last of the order, i.e. of the longest class
// `primal_count`, where *dual_flag is set: the items before the rows that the dual form has solved.  `list`: the rows to solve
// instead of the order's, *list_count of them (negative entries are skipped).
template <int D, typename T>
__global__ void __launch_bounds__(WGeo<D, T>::REGS_WARPS * 32, 1)
k_rows_warp(SideView sv, int64_t last, int64_t count, const int *dual_flag, int64_t primal_count, const int32_t *list,
            const unsigned long long *list_count, const T *__restrict__ X, const float *__restrict__ Bmat, RowOut out, ZeroRows zero, int wait_first, unsigned long long *done, DevStatus *st)
{
    using G = WGeo<D, T>;
    if (wait_first) wait_for_previous();
    store_zeros<D, T>(zero, out);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *base = reinterpret_cast<float4 *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *mine = smem_raw + G::BASE + warp * G::WARP;
    unsigned char *work = mine + 2 * G::STAGE;
    if (dual_flag && *dual_flag) count = primal_count;
    if (list_count) count = (int64_t)*list_count;
    if ((int64_t)blockIdx.x * G::ROWS >= count) {
        finish_after_previous(done);
        return;
    }
    load_base<D, T>(Bmat, base);
    __syncthreads();
    const int64_t warps = (int64_t)gridDim.x * G::REGS_WARPS;
    auto row_at = [&](int64_t k) -> int64_t { return list ? list[k] : sv.order[last - k]; };
    int64_t item = ((int64_t)warp * gridDim.x + blockIdx.x) * G::ROWS;
    if (item >= count) return;      // (never a block's first warp)
    Feed<D, T> feed;
    feed.X = X;
    feed.idx = sv.idx;
    feed.val = sv.val;
    feed.ring = ptx::smem_u32(mine);
    feed.g = 0;
    int64_t u = row_at(item);
    int64_t beg = u < 0 ? 0 : sv.ptr[u], end = u < 0 ? 0 : sv.ptr[u + 1];
    feed.start(beg, end, lane);
    float *b_s = reinterpret_cast<float *>(work) + G::B_AT;
    // the row after this one is looked up while this one is summed: its id a row ahead, its range now
    int64_t un = item + warps * G::ROWS < count ? row_at(item + warps * G::ROWS) : -1;
    while (true) {
        int64_t u_pair = -1;
        const int64_t next = item + warps * G::ROWS, after = next + warps * G::ROWS;
        const bool more = next < count;
        const int64_t bn = un < 0 ? 0 : sv.ptr[un], en = un < 0 ? 0 : sv.ptr[un + 1];
        const int64_t ua = after < count ? row_at(after) : -1;
        Sums<D, T> acc, acc2;
        acc.zero();
        sum_entries<D, T>(feed, u < 0 ? 1 : end - beg, mine, work, acc, lane);      // (a skipped row: one stage of zeros)
        put_b<D, T>(acc, b_s, lane);
        if constexpr (D == 16) {      // a second matrix; a lone last row goes without
            acc2.zero();
            if (item + 1 < count) {
                u_pair = row_at(item + 1);
                const int64_t b2 = u_pair < 0 ? 0 : sv.ptr[u_pair], e2 = u_pair < 0 ? 0 : sv.ptr[u_pair + 1];
                feed.start(b2, e2, lane);
                sum_entries<D, T>(feed, u_pair < 0 ? 1 : e2 - b2, mine, work, acc2, lane);
            }
            put_b<D, T>(acc2, b_s + D, lane);
            add_base<D, T>(acc2, base, lane);
        }
        // the next row's first entries travel while this one is solved
        if (more) feed.start_ids(bn, en, lane);
        add_base<D, T>(acc, base, lane);
        if (more) feed.start_copies(lane);
        const bool ok = factor_solve<D, T>(acc, acc2, reinterpret_cast<float *>(work), b_s, lane);
        if (D != 16 || lane < 16) {
            if (u >= 0) store_row<D, T>(b_s, ok, u, out, st, lane);
        } else if (u_pair >= 0) {
            store_row<D, T>(b_s + D, ok, u_pair, out, st, lane);
        }
        if (!more) break;
        __syncwarp();
        item = next;
        u = un;
        un = ua;
        beg = bn;
        end = en;
    }
    if (warp == 0) finish_after_previous(done);
}

// ---- long rows and chunks of split rows: a block of warps, each a slice of the entries; the slices' sums are added in warp
// order.  A chunk's sums go to the workspace in fragment order ([NB x 128] and b); a row is solved by the first warp.
template <int D, typename T> struct BGeo {
    using G = WGeo<D, T>;
    static constexpr int kBlockWarps = D == 64 ? 12 : 8;                 // warps per row, and blocks per SM: the registers of the sums
    static constexpr int kBlocks = D == 64 ? 1 : D == 32 ? 3 : 4;
    static constexpr int SUMS = G::NB * 128 + D;      // floats
    static constexpr int FEED = kBlockWarps * (2 * G::STAGE + G::TILE);
    static constexpr int RED = kBlockWarps * SUMS * 4;
    static constexpr int SHARED = FEED > RED ? FEED : RED;
    static constexpr size_t SMEM = (size_t)G::BASE + G::WORK + SHARED + 16;
};

template <int D, typename T> __device__ __forceinline__ void load_sums(const float *sums, Sums<D, T> &acc, int lane)
{
#pragma unroll
    for (int n = 0; n < WGeo<D, T>::NB; ++n) {
        const float4 v = *reinterpret_cast<const float4 *>(sums + (n * 32 + lane) * 4);
        acc.c[n][0] = v.x; acc.c[n][1] = v.y; acc.c[n][2] = v.z; acc.c[n][3] = v.w;
    }
}

template <int D, typename T, bool CG>
__device__ __forceinline__ void solve_sums(const float *sums, const float4 *base, float *work, int64_t u, const RowOut &out, const WarpCg &cg,
                                           DevStatus *st, int lane)
{
    using G = WGeo<D, T>;
    float *b_s = work + G::B_AT;
    if constexpr (CG) {
        Sums<D, T> acc;
        load_sums<D, T>(sums, acc, lane);
        add_base<D, T>(acc, base, lane);
        const float b0 = sums[G::NB * 128 + lane], b1 = sums[G::NB * 128 + 32 + lane];
        const float *stored = reinterpret_cast<const float *>(out.table) + u * D;
        float x0 = cg.warm ? stored[lane] : 0.f, x1 = cg.warm ? stored[lane + 32] : 0.f;
        float a0[64], a1[64];
        symmetric_rows(acc, work, a0, a1, lane);
        int products = 0;
        const bool ok = conjugate_gradients(cg, a0, a1, b_s, b0, b1, x0, x1, products, lane);
        if (lane == 0) {
            atomicAdd(&cg.counters[0], 1ull);
            atomicAdd(&cg.counters[1], (unsigned long long)products);
            if (!ok) cg.fallback_list[atomicAdd(&cg.counters[2], 1ull)] = -1;      // solved below: nothing for the list's kernel
        }
        if (ok) {
            __syncwarp();
            b_s[lane] = x0;
            b_s[lane + 32] = x1;
            __syncwarp();
            store_row<D, T>(b_s, true, u, out, st, lane);
            return;
        }
    }
    Sums<D, T> acc, acc2;
    load_sums<D, T>(sums, acc, lane);
    for (int e = lane; e < G::ROWS * D; e += 32) b_s[e] = sums[G::NB * 128 + (e & (D - 1))];
    add_base<D, T>(acc, base, lane);
    if constexpr (D == 16) acc2 = acc;
    __syncwarp();
    const bool ok = factor_solve<D, T>(acc, acc2, work, b_s, lane);
    if (D != 16 || lane < 16) store_row<D, T>(b_s, ok, u, out, st, lane);
}

template <int D, typename T, bool CHUNK>
__global__ void __launch_bounds__(BGeo<D, T>::kBlockWarps * 32, BGeo<D, T>::kBlocks)
k_rows_block(SideView sv, int64_t last, const T *__restrict__ X, const float *__restrict__ Bmat, float *__restrict__ partials, RowOut out,
             DevStatus *st)
{
    using G = WGeo<D, T>;
    using B = BGeo<D, T>;
    constexpr int kBlockWarps = B::kBlockWarps;
    wait_for_previous();
    let_next_start();      // the rows of a warp each may start beside these
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
    if (warp == 0) solve_sums<D, T, false>(red, base, work, u, out, WarpCg{}, st, lane);
}

// one warp per row whose sums are in the workspace: split rows first (their chunks' sums are added in ascending order), then
// n_long whole rows of one sum each, behind the n_chunks of the others
template <int D, typename T, bool CG>
__global__ void __launch_bounds__(32) k_solve_sums_warp(SideView sv, int64_t split_begin, int64_t n_split, int64_t n_chunks,
                                                        const float *__restrict__ partials, const float *__restrict__ Bmat, RowOut out,
                                                        WarpCg cg, DevStatus *st)
{
    using G = WGeo<D, T>;
    using B = BGeo<D, T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *base = reinterpret_cast<float4 *>(smem_raw);
    float *work = reinterpret_cast<float *>(smem_raw + G::BASE);
    float *sums = reinterpret_cast<float *>(smem_raw + G::BASE + G::WORK);
    const int lane = threadIdx.x;
    load_base<D, T>(Bmat, base);
    const int64_t k = blockIdx.x, whole = k - n_split;      // whole rows: from the end of their classes, as k_sums64 takes them
    const int64_t u = sv.order[whole < 0 ? split_begin + k : split_begin - 1 - whole];
    const int64_t c0 = whole < 0 ? sv.split_first[k] : n_chunks + whole, c1 = whole < 0 ? sv.split_first[k + 1] : c0 + 1;
    for (int e = 4 * lane; e < B::SUMS; e += 128) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int64_t c = c0; c < c1; ++c) {
            const float4 v = *reinterpret_cast<const float4 *>(partials + c * B::SUMS + e);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *reinterpret_cast<float4 *>(sums + e) = s;
    }
    __syncwarp();
    solve_sums<D, T, CG>(sums, base, work, u, out, cg, st, lane);
}

// ---- fp32 tables of 64 features over a table of their bfloat16 parts: [row][x1 | x2 | x3][64], x = x1 + x2 + x3 to 2^-24, written once
// per half-epoch, so that a gathered row is an mma operand as it lands (converting every gathered entry was a third of the
// instructions of the sums).  The right-hand side is a product too, with the labels' three parts as columns.
__global__ void __launch_bounds__(256) k_parts64(const float *__restrict__ X, int64_t n, uint32_t *__restrict__ P)
{
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;      // four features of a row
    if (e >= n * 16) return;
    const float4 x = reinterpret_cast<const float4 *>(X)[e];
    uint32_t p[3][2];
    split_bf16(x.x, x.y, p[0][0], p[1][0], p[2][0]);
    split_bf16(x.z, x.w, p[0][1], p[1][1], p[2][1]);
    uint32_t *row = P + (e / 16) * 96 + 2 * (e % 16);
#pragma unroll
    for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2 *>(row + 32 * q) = make_uint2(p[q][0], p[q][1]);
}

struct PGeo {
    using G = WGeo<64, float>;
    static constexpr int ROW = 144;                       // bytes between the rows of a staged part
    static constexpr int PART = kEntries * ROW, STAGE = 3 * PART;
    static constexpr int PIECES = 24;                     // 16-byte pieces of a table row
    static constexpr int WARPS = 12;                      // per SM: registers
    static constexpr int WARP = 2 * STAGE + 512;          // ring, vector, right-hand side
    static constexpr int SUMS = G::NB * 128 + 64;
    static constexpr int RING = 4;                        // stages of the long-row kernel
};
static_assert(PGeo::G::BASE + PGeo::WARPS * PGeo::WARP <= 232448 && 32 * 36 * 4 <= PGeo::STAGE, "shared memory");

// labels of a stage as an mma B operand: column 0, 1, 2 = their bfloat16 parts; y0 .. y3 = labels of entries 2 q, 2 q + 1, 2 q + 8,
// 2 q + 9, q = lane % 4
__device__ __forceinline__ void label_operand(float y0, float y1, float y2, float y3, uint32_t &b0, uint32_t &b1, int lane)
{
    uint32_t p[2][3];
    split_bf16(y0, y1, p[0][0], p[0][1], p[0][2]);
    split_bf16(y2, y3, p[1][0], p[1][1], p[1][2]);
    const int n = lane >> 2;
    b0 = n == 0 ? p[0][0] : n == 1 ? p[0][1] : n == 2 ? p[0][2] : 0u;
    b1 = n == 0 ? p[1][0] : n == 1 ? p[1][1] : n == 2 ? p[1][2] : 0u;
}

// Whole rows by a warp each: conjugate gradients, the matrix in registers.
struct PartsFeed {
    const uint4 *P;
    const int32_t *idx;
    const float *val;
    uint32_t ring;
    int g;                          // next stage to be consumed; stage g lives in slot g % 2
    int64_t at, end;
    int id, id_first;               // (lane < 16) ids of the stage after the one in flight; of a row's first stage
    float y, y_next;                // labels of the stage in flight, of the one after it

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
    __device__ __forceinline__ void issue(int slot, int ids, int lane)
    {
        const uint32_t dst = ring + (uint32_t)slot * PGeo::STAGE;
#pragma unroll 1
        for (int k = 0; k < kEntries; k += 4) {      // eight lanes per part of a row (unrolled in full it does not fit the registers)
            const int r = k + (lane >> 3), c = lane & 7;
            const int row = __shfl_sync(0xFFFFFFFFu, ids, r);
            const uint4 *src = P + (int64_t)(row < 0 ? 0 : row) * PGeo::PIECES + c;
#pragma unroll
            for (int p = 0; p < 3; ++p) cp_async16_zfill(dst + p * PGeo::PART + r * PGeo::ROW + c * 16, src + 8 * p, row >= 0);
        }
        ptx::cp_async_commit();
    }
    __device__ __forceinline__ void start_ids(int64_t beg, int64_t e, int lane)
    {
        at = beg;
        end = e;
        load_ids(lane);
        y = y_next;
        id_first = id;
        load_ids(lane);
    }
    __device__ __forceinline__ void start_copies(int lane) { issue(g & 1, id_first, lane); }
};

__device__ __forceinline__ void sum_parts(PartsFeed &feed, int64_t len, Sums<64, float> &acc, float *b_s, int lane)
{
    const int stages = (int)((len + kEntries - 1) / kEntries);
    float bacc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) bacc[i][e] = 0.f;
    const uint32_t lane_at = ((lane & 7) + 8 * (lane >> 4)) * PGeo::ROW + 16 * ((lane >> 3) & 1);
#pragma unroll 1
    for (int s = 0; s < stages; ++s) {
        const float y = feed.y;
        if (s + 1 < stages) {
            feed.y = feed.y_next;
            feed.issue((feed.g + 1) & 1, feed.id, lane);
            feed.load_ids(lane);
            ptx::cp_async_wait<1>();
        } else {
            ptx::cp_async_wait<0>();
        }
        __syncwarp();
        uint32_t yb0 = lane < 4 ? 0x3F803F80u : 0u, yb1 = yb0;      // (labels of 1; entries past the end are zeros)
        if (feed.val) {
            const int q = 2 * (lane & 3);
            label_operand(__shfl_sync(0xFFFFFFFFu, y, q), __shfl_sync(0xFFFFFFFFu, y, q + 1), __shfl_sync(0xFFFFFFFFu, y, q + 8),
                          __shfl_sync(0xFFFFFFFFu, y, q + 9), yb0, yb1, lane);
        }
        const uint32_t src = feed.ring + (feed.g & 1) * PGeo::STAGE + lane_at;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t a[3][4];
#pragma unroll
            for (int p = 0; p < 3; ++p) ldmatrix_x4_trans(src + p * PGeo::PART + 32 * i, a[p]);
            float tb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int p = 2; p >= 0; --p) mma_bf16(tb, a[p], yb0, yb1);
            // the parts' products from the smallest up, each stage's from zero: the accumulator of an mma truncates.  (The other
            // operand is loaded again for every block: four blocks' fragments at once do not fit the registers.)
            constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                uint32_t b[3][4];
#pragma unroll
                for (int p = 0; p < 3; ++p) ldmatrix_x4_trans(src + p * PGeo::PART + 32 * j, b[p]);
                float t[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    mma_bf16(t[0], a[pa[q]], b[pb[q]][0], b[pb[q]][2]);
                    mma_bf16(t[1], a[pa[q]], b[pb[q]][1], b[pb[q]][3]);
                }
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc.c[i * (i + 1) + 2 * j + n][e] += t[n][e];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) bacc[i][e] += tb[e];
        }
        __syncwarp();      // the slot may be overwritten
        ++feed.g;
    }
    // columns 0, 1 are in the quad's first lane, 2 in its second
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float u = bacc[i][0] + bacc[i][1], v = bacc[i][2] + bacc[i][3];
        const float u1 = __shfl_down_sync(0xFFFFFFFFu, u, 1), v1 = __shfl_down_sync(0xFFFFFFFFu, v, 1);
        if ((lane & 3) == 0) {
            b_s[16 * i + lane / 4] = u + u1;
            b_s[16 * i + 8 + lane / 4] = v + v1;
        }
    }
    __syncwarp();
}

__global__ void __launch_bounds__(PGeo::WARPS * 32, 1)
k_rows_cg64(SideView sv, int64_t last, int64_t count, const int *dual_flag, int64_t primal_count, const uint4 *__restrict__ P,
            const float *__restrict__ Bmat, RowOut out, ZeroRows zero, WarpCg cg, DevStatus *st)
{
    using G = WGeo<64, float>;
    store_zeros<64, float>(zero, out);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *base = reinterpret_cast<float4 *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *mine = smem_raw + G::BASE + warp * PGeo::WARP;
    float *vec = reinterpret_cast<float *>(mine + 2 * PGeo::STAGE), *b_s = vec + 64;
    if (dual_flag && *dual_flag) count = primal_count;      // the rows behind them have been solved in the dual form
    if ((int64_t)blockIdx.x >= count) return;
    load_base<64, float>(Bmat, base);
    __syncthreads();
    const int64_t warps = (int64_t)gridDim.x * PGeo::WARPS;
    unsigned rows = 0, products = 0;
    const int64_t item = (int64_t)warp * gridDim.x + blockIdx.x;
    if (item >= count) return;
    PartsFeed feed;
    feed.P = P;
    feed.idx = sv.idx;
    feed.val = sv.val;
    feed.ring = ptx::smem_u32(mine);
    feed.g = 0;
    // the walk: rows are looked up two ahead (id), one ahead (range); 32-bit ids and lengths, for the registers
    const int32_t *walk = sv.order + (last - item);
    int left = (int)((count - item - 1) / warps);      // rows after the current one
    int u = *walk, un = left > 0 ? *(walk - warps) : -1;
    int len = (int)(sv.ptr[u + 1] - sv.ptr[u]);
    feed.start_ids(sv.ptr[u], sv.ptr[u + 1], lane);
    feed.start_copies(lane);
    while (true) {
        float a0[64], a1[64];
        const int ua = left > 1 ? *(walk - 2 * warps) : -1;
        {
            const int64_t bn = left > 0 ? sv.ptr[un] : 0;
            const int len_next = left > 0 ? (int)(sv.ptr[un + 1] - bn) : 0;
            Sums<64, float> acc;
            acc.zero();
            sum_parts(feed, len, acc, b_s, lane);
            len = len_next;
            if (left > 0) feed.start_ids(bn, bn + len, lane);
            add_base<64, float>(acc, base, lane);
            // (through the slot that the next row's first stage will not take)
            symmetric_rows(acc, reinterpret_cast<float *>(mine + ((feed.g + 1) & 1) * PGeo::STAGE), a0, a1, lane);
        }
        if (left > 0) feed.start_copies(lane);      // they travel while this row is solved
        float *row = reinterpret_cast<float *>(out.table) + (int64_t)u * 64;
        float x0 = cg.warm ? row[lane] : 0.f, x1 = cg.warm ? row[lane + 32] : 0.f;
        int spent = 0;
        const bool ok = conjugate_gradients(cg, a0, a1, vec, b_s[lane], b_s[lane + 32], x0, x1, spent, lane);
        ++rows;
        products += spent;
        if (ok) {
            row[lane] = x0;
            row[lane + 32] = x1;
            if (out.cap_slot) {
                const int slot = out.cap_slot[u];
                if (slot >= 0) {
                    out.cap_out[(int64_t)slot * 64 + lane] = x0;
                    out.cap_out[(int64_t)slot * 64 + 32 + lane] = x1;
                }
            }
        } else if (lane == 0) {
            cg.fallback_list[atomicAdd(&cg.counters[2], 1ull)] = u;
        }
        if (left == 0) break;
        __syncwarp();
        --left;
        walk -= warps;
        u = un;
        un = ua;
    }
    if (lane == 0) {
        atomicAdd(&cg.counters[0], (unsigned long long)rows);
        atomicAdd(&cg.counters[1], (unsigned long long)products);
    }
}

// Sums of long rows and of the chunks of split rows: a block of four warps per item.  The warps share the gathered stages and have
// the matrix's 16 x 16 blocks among them, three (or two) each, so that every accumulator sees all of an item's entries; the large
// products and the five small ones have accumulators of their own, and the large sums are truncated once per 16 entries.
template <int W> struct Blocks64 {      // blocks (i, j) of warp W: (3, 0 .. 2); (2, 0 .. 2); (1, 0), (1, 1); (0, 0), (3, 3)
    static constexpr int N = W < 2 ? 3 : 2;
    __host__ __device__ static constexpr int i(int k) { return W < 3 ? 3 - W : 3 * k; }
    __host__ __device__ static constexpr int j(int k) { return W < 3 ? k : 3 * k; }
};

struct Sums64 {
    float big[3][2][4], small[3][2][4], b[4];
};

template <int W> __device__ __forceinline__ void products64(uint32_t src, uint32_t yb0, uint32_t yb1, Sums64 &acc)
{
    using K = Blocks64<W>;
    uint32_t f[3][4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool used = W == 0 || (W == 1 && i < 3) || (W == 2 && i < 2) || (W == 3 && (i == 0 || i == 3));
        if (used)
#pragma unroll
            for (int p = 0; p < 3; ++p) ldmatrix_x4_trans(src + p * PGeo::PART + 32 * i, f[p][i]);
    }
    constexpr int pa[5] = {2, 0, 1, 1, 0}, pb[5] = {0, 2, 1, 0, 1};
#pragma unroll
    for (int k = 0; k < K::N; ++k) {
        const int i = K::i(k), j = K::j(k);
#pragma unroll
        for (int n = 0; n < 2; ++n) mma_bf16(acc.big[k][n], f[0][i], f[0][j][n], f[0][j][2 + n]);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q)
#pragma unroll
        for (int k = 0; k < K::N; ++k)
#pragma unroll
            for (int n = 0; n < 2; ++n) mma_bf16(acc.small[k][n], f[pa[q]][K::i(k)], f[pb[q]][K::j(k)][n], f[pb[q]][K::j(k)][2 + n]);
    constexpr int ib = W == 3 ? 0 : 3 - W;      // the warp's features of the right-hand side
#pragma unroll
    for (int p = 2; p >= 0; --p) mma_bf16(acc.b, f[p][ib], yb0, yb1);
}

template <int W> __device__ __forceinline__ void write64(const Sums64 &acc, float *dst, int lane)
{
    using K = Blocks64<W>;
#pragma unroll
    for (int k = 0; k < K::N; ++k)
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const float *x = acc.big[k][n], *y = acc.small[k][n];
            *reinterpret_cast<float4 *>(dst + ((K::i(k) * (K::i(k) + 1) + 2 * K::j(k) + n) * 32 + lane) * 4) =
                make_float4(x[0] + y[0], x[1] + y[1], x[2] + y[2], x[3] + y[3]);
        }
    const float u = acc.b[0] + acc.b[1], v = acc.b[2] + acc.b[3];
    const float u1 = __shfl_down_sync(0xFFFFFFFFu, u, 1), v1 = __shfl_down_sync(0xFFFFFFFFu, v, 1);
    constexpr int ib = W == 3 ? 0 : 3 - W;
    if ((lane & 3) == 0) {
        dst[PGeo::G::NB * 128 + 16 * ib + lane / 4] = u + u1;
        dst[PGeo::G::NB * 128 + 16 * ib + 8 + lane / 4] = v + v1;
    }
}

__global__ void __launch_bounds__(128, 4) k_sums64(SideView sv, int64_t n_chunks, int64_t last_long, const uint4 *__restrict__ P, float *__restrict__ sums)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float y_s[PGeo::RING][kEntries];
    constexpr int R = PGeo::RING;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int64_t beg, end;
    if ((int64_t)blockIdx.x < n_chunks) {
        beg = sv.chunk_desc[4 * (int64_t)blockIdx.x + 1];
        end = sv.chunk_desc[4 * (int64_t)blockIdx.x + 2];
    } else {
        const int64_t u = sv.order[last_long - ((int64_t)blockIdx.x - n_chunks)];
        beg = sv.ptr[u];
        end = sv.ptr[u + 1];
    }
    const int stages = (int)((end - beg + kEntries - 1) / kEntries);
    // a thread brings three 16-byte pieces of a stage; their rows' ids are looked up two stages before
    const int r0 = tid / PGeo::PIECES, c0 = tid % PGeo::PIECES, r1 = (tid + 128) / PGeo::PIECES, c1 = (tid + 128) % PGeo::PIECES;
    const int r2 = (tid + 256) / PGeo::PIECES, c2 = (tid + 256) % PGeo::PIECES;
    int id[3];
    float y = 0.f;
    auto load_ids = [&](int s) {
        const int64_t at = beg + (int64_t)s * kEntries;
        id[0] = at + r0 < end ? __ldg(sv.idx + at + r0) : -1;
        id[1] = at + r1 < end ? __ldg(sv.idx + at + r1) : -1;
        id[2] = at + r2 < end ? __ldg(sv.idx + at + r2) : -1;
        if (tid < kEntries) y = at + tid < end ? (sv.val ? __ldg(sv.val + at + tid) : 1.f) : 0.f;
    };
    const uint32_t ring = ptx::smem_u32(smem_raw);
    auto issue = [&](int s) {
        const uint32_t dst = ring + (uint32_t)(s % R) * PGeo::STAGE;
        cp_async16_zfill(dst + (c0 / 8) * PGeo::PART + r0 * PGeo::ROW + (c0 % 8) * 16, P + (int64_t)(id[0] < 0 ? 0 : id[0]) * PGeo::PIECES + c0, id[0] >= 0);
        cp_async16_zfill(dst + (c1 / 8) * PGeo::PART + r1 * PGeo::ROW + (c1 % 8) * 16, P + (int64_t)(id[1] < 0 ? 0 : id[1]) * PGeo::PIECES + c1, id[1] >= 0);
        cp_async16_zfill(dst + (c2 / 8) * PGeo::PART + r2 * PGeo::ROW + (c2 % 8) * 16, P + (int64_t)(id[2] < 0 ? 0 : id[2]) * PGeo::PIECES + c2, id[2] >= 0);
        if (tid < kEntries) y_s[s % R][tid] = y;
    };
#pragma unroll
    for (int s = 0; s < R - 1; ++s) {
        if (s < stages) {
            load_ids(s);
            issue(s);
        }
        ptx::cp_async_commit();
    }
    if (R - 1 < stages) load_ids(R - 1);
    Sums64 acc;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int n = 0; n < 2; ++n) acc.big[k][n][e] = acc.small[k][n][e] = 0.f;
        acc.b[e] = 0.f;
    }
    const uint32_t lane_at = ((lane & 7) + 8 * (lane >> 4)) * PGeo::ROW + 16 * ((lane >> 3) & 1);
#pragma unroll 1
    for (int s = 0; s < stages; ++s) {
        ptx::cp_async_wait<R - 2>();
        __syncthreads();      // the stage is here for all, and the slot of the one before it is free
        if (s + R - 1 < stages) {
            issue(s + R - 1);
            if (s + R < stages) load_ids(s + R);
        }
        ptx::cp_async_commit();
        uint32_t yb0, yb1;
        const float *ys = y_s[s % R] + 2 * (lane & 3);
        label_operand(ys[0], ys[1], ys[8], ys[9], yb0, yb1, lane);
        const uint32_t src = ring + (uint32_t)(s % R) * PGeo::STAGE + lane_at;
        if (warp == 0) products64<0>(src, yb0, yb1, acc);
        else if (warp == 1) products64<1>(src, yb0, yb1, acc);
        else if (warp == 2) products64<2>(src, yb0, yb1, acc);
        else products64<3>(src, yb0, yb1, acc);
    }
    float *dst = sums + (int64_t)blockIdx.x * PGeo::SUMS;
    if (warp == 0) write64<0>(acc, dst, lane);
    else if (warp == 1) write64<1>(acc, dst, lane);
    else if (warp == 2) write64<2>(acc, dst, lane);
    else write64<3>(acc, dst, lane);
}

template <int D, typename T> __global__ void __launch_bounds__(256) k_zero_rows_warp(ZeroRows zero, RowOut out) { store_zeros<D, T>(zero, out); }

struct WarpRows {
    SideView sv;
    const int64_t *offs;
    int64_t n_chunks, n_split_rows;
    const void *X;
    void *parts;               // fp32 tables of 64 features: room for the table's bfloat16 parts
    const float *Bmat;
    float *partials;
    RowOut out;
    DevStatus *st;
    WarpCg cg;
    const int *dual_flag;      // set on the device when the rows of class 1 have been solved in the dual form
    unsigned long long *stamps;      // time stamps of the half-epoch, or null
    bool early;                      // few entries: the kernels may start while the one before them ends
    cudaStream_t s;
    int64_t *launches;
};

// The rows without observations: with the launch of the others (`blocks` of `threads`) where that has a thread for every 32 values,
// else by a launch of their own, now.
template <int D, typename T> ZeroRows zero_rows(const WarpRows &a, int64_t blocks, int64_t threads)
{
    const ZeroRows z{a.sv.order + a.offs[0], a.offs[1] - a.offs[0]};
    if (z.count * D <= blocks * threads * 32) return z;
    const int64_t grid = (z.count * D + 255) / 256;
    k_zero_rows_warp<D, T><<<(unsigned)(grid < (1 << 20) ? grid : 1 << 20), 256, 0, a.s>>>(z, a.out);
    ++*a.launches;
    return ZeroRows{nullptr, 0};
}

// rows order[end - 1], order[end - 2] .. by a warp each, down to class `first`; `list` (with its device-side count) instead
template <int D, typename T>
cudaError_t whole_rows(const WarpRows &a, int64_t end, const int32_t *list, const unsigned long long *list_count, bool after_block_rows)
{
    using G = WGeo<D, T>;
    static_assert((size_t)G::BASE + G::REGS_WARPS * G::WARP <= 232448, "shared memory");
    const size_t smem = (size_t)G::BASE + G::REGS_WARPS * G::WARP;
    const int64_t n = list ? 0 : end - a.offs[1];
    if (!list && n <= 0) {
        zero_rows<D, T>(a, 0, 0);
        return cudaGetLastError();
    }
    static SmemOnce allow;
    const cudaError_t e = allow(k_rows_warp<D, T>, smem);
    if (e != cudaSuccess) return e;
    int64_t blocks = list ? 148 : (n + G::ROWS - 1) / G::ROWS;      // few rows: one per SM before two
    if (blocks > 148) blocks = 148;
    const ZeroRows zero = list ? ZeroRows{nullptr, 0} : zero_rows<D, T>(a, blocks, G::REGS_WARPS * 32);
    // where k_rows_block is the launch before this one (a launch of the rows without observations may be between) the two run
    // side by side: everything this one reads was complete before k_rows_block let it start
    const bool beside = after_block_rows && zero.rows;
    const cudaError_t el = launch_early(beside || (!list && a.early), k_rows_warp<D, T>, blocks, G::REGS_WARPS * 32, smem, a.s, a.sv, end - 1, n, list ? nullptr : a.dual_flag,
                                        end - a.offs[2], list, list_count, reinterpret_cast<const T *>(a.X), a.Bmat, a.out, zero, beside ? 0 : 1,
                                        a.stamps ? a.stamps + kStampEnd : nullptr, a.st);
    if (el != cudaSuccess) return el;
    ++*a.launches;
    return cudaGetLastError();
}

template <int D, typename T, bool CG> cudaError_t solve_rows(const WarpRows &a, int64_t n_long)
{
    if (a.n_split_rows + n_long <= 0) return cudaSuccess;
    const size_t smem = (size_t)WGeo<D, T>::BASE + WGeo<D, T>::WORK + 4 * BGeo<D, T>::SUMS;
    k_solve_sums_warp<D, T, CG><<<(unsigned)(a.n_split_rows + n_long), 32, smem, a.s>>>(a.sv, a.offs[kNClasses - 1], a.n_split_rows, a.n_chunks,
                                                                                      a.partials, a.Bmat, a.out, a.cg, a.st);
    ++*a.launches;
    return cudaGetLastError();
}

template <int D, typename T> cudaError_t rows_warp_dt(const WarpRows &a)
{
    using B = BGeo<D, T>;
    static_assert(B::SUMS <= D * D + D, "a chunk's sums fit its place in the workspace");
    static_assert(B::SMEM <= 232448, "shared memory");
    const T *X = reinterpret_cast<const T *>(a.X);
    const int64_t *offs = a.offs, end_long = offs[kNClasses - 1], begin_long = offs[warp_long_class(offs)];
    cudaError_t e;
    // longest work first
    if (a.n_chunks > 0) {
        static SmemOnce allow;
        if ((e = allow(k_rows_block<D, T, true>, B::SMEM)) != cudaSuccess) return e;
        e = launch_early(a.early, k_rows_block<D, T, true>, a.n_chunks, B::kBlockWarps * 32, B::SMEM, a.s, a.sv, 0, X, a.Bmat, a.partials, a.out, a.st);
        if (e != cudaSuccess) return e;
        ++*a.launches;
        if ((e = solve_rows<D, T, false>(a, 0)) != cudaSuccess) return e;
    }
    if (end_long > begin_long) {
        static SmemOnce allow;
        if ((e = allow(k_rows_block<D, T, false>, B::SMEM)) != cudaSuccess) return e;
        e = launch_early(a.early, k_rows_block<D, T, false>, end_long - begin_long, B::kBlockWarps * 32, B::SMEM, a.s, a.sv, end_long - 1, X, a.Bmat,
                         a.partials, a.out, a.st);
        if (e != cudaSuccess) return e;
        ++*a.launches;
    }
    return whole_rows<D, T>(a, begin_long, nullptr, nullptr, end_long > begin_long);
}

// fp32 tables of 64 features: long rows and chunks over the parts whatever the solver, the other rows too with conjugate gradients
cudaError_t rows_parts64(const WarpRows &a, bool use_cg, int64_t n_table)
{
    const int64_t *offs = a.offs, end_long = offs[kNClasses - 1], begin_long = offs[parts64_long_class(offs)];
    const int64_t n_long = end_long - begin_long, n = begin_long - offs[1];
    const uint4 *P = static_cast<const uint4 *>(a.parts);
    cudaError_t e;
    if (a.n_chunks + n_long > 0 || (use_cg && n > 0)) {
        k_parts64<<<(unsigned)((n_table * 16 + 255) / 256), 256, 0, a.s>>>(static_cast<const float *>(a.X), n_table, static_cast<uint32_t *>(a.parts));
        ++*a.launches;
    }
    if (a.n_chunks + n_long > 0) {
        const size_t smem = PGeo::RING * PGeo::STAGE;
        k_sums64<<<(unsigned)(a.n_chunks + n_long), 128, smem, a.s>>>(a.sv, a.n_chunks, end_long - 1, P, a.partials);
        ++*a.launches;
        e = use_cg ? solve_rows<64, float, true>(a, n_long) : solve_rows<64, float, false>(a, n_long);
        if (e != cudaSuccess) return e;
    }
    if (use_cg) {
        if (n > 0) {
            const size_t smem = PGeo::G::BASE + PGeo::WARPS * PGeo::WARP;
            static SmemOnce allow;
            if ((e = allow(k_rows_cg64, smem)) != cudaSuccess) return e;
            const int64_t blocks = n < 148 ? n : 148;
            k_rows_cg64<<<(unsigned)blocks, PGeo::WARPS * 32, smem, a.s>>>(a.sv, begin_long - 1, n, a.dual_flag, begin_long - offs[2], P, a.Bmat, a.out,
                                                                          zero_rows<64, float>(a, blocks, PGeo::WARPS * 32), a.cg, a.st);
            ++*a.launches;
            // the rows conjugate gradients did not finish (none, as a rule: its blocks then return at once)
            if ((e = whole_rows<64, float>(a, begin_long, a.cg.fallback_list, a.cg.counters + 2, false)) != cudaSuccess) return e;
        }
        else zero_rows<64, float>(a, 0, 0);
        return cudaGetLastError();
    }
    return whole_rows<64, float>(a, begin_long, nullptr, nullptr, false);
}

}  // namespace

cudaError_t launch_rows_warp(const SideView &sv, const int64_t *offs, int64_t n_chunks, int64_t n_split_rows, const void *X, int64_t n_table,
                             void *parts, int bf16, int d, const float *Bmat, float *partials, RowOut out, DevStatus *st, const CgOptions &cg,
                             const int *dual_flag, unsigned long long *stamps, cudaStream_t s, int64_t *launches)
{
    const WarpRows a{sv, offs, n_chunks, n_split_rows, X, parts, Bmat, partials, out, st,
                     WarpCg{cg.max_iter, cg.warm_start ? 1 : 0, cg.tol * cg.tol, cg.counters, cg.fallback_list}, dual_flag, stamps, sv.nnz <= kEarlyEntries, s, launches};
    switch (d) {
    case 16: return bf16 ? rows_warp_dt<16, __nv_bfloat16>(a) : rows_warp_dt<16, float>(a);
    case 32: return bf16 ? rows_warp_dt<32, __nv_bfloat16>(a) : rows_warp_dt<32, float>(a);
    case 64: return bf16 ? rows_warp_dt<64, __nv_bfloat16>(a) : rows_parts64(a, cg.enabled, n_table);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace alx
