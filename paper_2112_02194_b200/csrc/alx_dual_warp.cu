// Rows with at most 16 observations in the dual form of Eq. 4, a warp per row, on warp-level mma:
//   w = B^-1 H^T (I + H B^-1 H^T)^-1 y,   B = alpha0 G + lambda I   (the push-through identity: an exact restatement),
// a 16 x 16 system instead of a d x d one, for bfloat16 tables of 64 features and fp32 tables of 128.
//   gather the k <= 16 rows of H (the rest are zeros), as bfloat16 parts: x = x1 + x2 + x3 for fp32 tables, x for bfloat16;
//   Z = H B^-1 by mma m16n8k16, B^-1 in three bfloat16 parts that wait in shared memory in fragment order (the products down to
//   2^-24), Z in the accumulators; S = I + Z H^T by mma again, Z's accumulators split into parts in place -- an accumulator pair
//   is an A fragment; Cholesky of S in the warp; w = Z^T t from the accumulators.
// The next row's H rows are in registers on their way while a row is worked on.
//
// The form is used only while B is well conditioned (its error grows with cond(B)): k_binv_fragments sets a flag from
// ||B||_F ||B^-1||_F; with the flag clear this kernel does nothing and the d x d kernels take these rows as well.
//
// Bound: the chain of a row (the 16 x 16 factorisation and substitution are half of it) over 8 to 16 warps per SM: 2.7 ns of the
// chip per row for d = 64 bfloat16, 11 ns for d = 128 fp32, where the d x d solves take 9 and 90.  (fp32 tables of 64 features
// keep the FP32-ALU kernel of alx_dual64.cu: 3.7 ns against 4.0 here, and it holds its residual up to higher conditions.)
#include "alx_common.cuh"
#include "alx_inverse.cuh"
#include "alx_mma.cuh"
#include "alx_ptx.cuh"

namespace alx {

namespace {

constexpr int kObs = 16;

template <int D, typename T> struct DGeo {
    static constexpr bool kF32 = sizeof(T) == 4;
    static constexpr int KS = D / 16, NB = D / 8;               // K steps and 8-column blocks of Z
    static constexpr int PARTS = kF32 ? 3 : 1;
    static constexpr int ROW = 2 * D + 16;                      // bytes between the rows of a bfloat16 tile (ldmatrix without conflicts)
    static constexpr int TILE = PARTS * kObs * ROW;
    static constexpr int ROW_PIECES = D * (int)sizeof(T) / 16;  // 16-byte pieces of a table row
    static constexpr int PIECES = kObs * ROW_PIECES / 32;       // ... of all rows, per lane
    static constexpr int SCRATCH = 4 * (256 + 64 + 32);         // S / L, exchange, t, reciprocal pivots
    static constexpr int WARP = TILE + SCRATCH;
    static constexpr int WARPS = D == 128 ? 8 : 16;             // per SM: registers
    static constexpr int BINV = 3 * D * D * 2;                  // bytes of B^-1 in fragment order
    static constexpr size_t SMEM = (size_t)BINV + WARPS * WARP;
};

// Element (k, n) of part q of B^-1 as an mma B operand: two adjacent 8-column blocks of a K step make one 16-byte read per lane
template <int D> __host__ __device__ constexpr int binv_at(int k, int n, int q)
{
    return (((((k >> 4) * (D / 16) + (n >> 4)) * 3 + q) * 32) + (n & 7) * 4 + ((k & 7) >> 1)) * 8 + ((n >> 3) & 1) * 4 + ((k >> 3) & 1) * 2 + (k & 1);
}

// B^-1 in fp64 (alx_inverse.cuh), written as three bfloat16 parts in fragment order; flag = 1 if B is positive definite and
// ||B||_F ||B^-1||_F <= cond_limit
template <int D>
__global__ void __launch_bounds__(SweepGeo<D>::THREADS, 1) k_binv_fragments(const float *__restrict__ Bmat, __nv_bfloat16 *__restrict__ frag,
                                                                           int *__restrict__ flag, double cond_limit)
{
    __shared__ SweepSmem<D> sm;
    double cond;
    const bool ok = sweep_inverse<D>(Bmat, sm, &cond, [&](int i, int c, double s) {
        float v = (float)s;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const __nv_bfloat16 p = __float2bfloat16_rn(v);
            frag[binv_at<D>(i, c, q)] = p;
            v -= __bfloat162float(p);
        }
    });
    if (threadIdx.x == 0) *flag = (ok && cond <= cond_limit) ? 1 : 0;
}

template <int D, typename T>
__global__ void __launch_bounds__(DGeo<D, T>::WARPS * 32, 1)
k_dual_warp(SideView sv, int64_t first, int64_t count, const T *__restrict__ X, const uint4 *__restrict__ binv, const int *__restrict__ flag,
            RowOut out, DevStatus *st)
{
    using G = DGeo<D, T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (*flag == 0) return;
    const uint4 *bf = reinterpret_cast<const uint4 *>(smem_raw);
    for (int e = threadIdx.x; e < G::BINV / 16; e += G::WARPS * 32) reinterpret_cast<uint4 *>(smem_raw)[e] = binv[e];
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *tile = smem_raw + G::BINV + warp * G::WARP;
    float *S = reinterpret_cast<float *>(tile + G::TILE), *ex = S + 256, *t_s = ex + 64, *dinv_s = t_s + 16;
    const int64_t warps = (int64_t)gridDim.x * G::WARPS;
    int64_t item = (int64_t)warp * gridDim.x + blockIdx.x;
    if (item >= count) return;

    // a row's lookup, two rows ahead: its range; one row ahead: its ids and labels (lane = observation), then its H rows
    uint4 raw[G::PIECES];
    auto load_range = [&](int64_t k, int64_t &u, int64_t &beg, int &len) {
        u = k < count ? sv.order[first + k] : -1;
        beg = u < 0 ? 0 : sv.ptr[u];
        len = u < 0 ? 0 : (int)(sv.ptr[u + 1] - beg);
    };
    auto load_ids = [&](int64_t beg, int len, int &id, float &y) {
        id = lane < len ? __ldg(sv.idx + beg + lane) : -1;
        y = lane < len ? (sv.val ? __ldg(sv.val + beg + lane) : 1.f) : 0.f;
    };
    auto load_rows = [&](int id) {
#pragma unroll
        for (int j = 0; j < G::PIECES; ++j) {
            const int p = lane + 32 * j, r = p / G::ROW_PIECES, c = p % G::ROW_PIECES;
            const int row = __shfl_sync(0xFFFFFFFFu, id, r);
            raw[j] = row < 0 ? make_uint4(0u, 0u, 0u, 0u) : __ldg(reinterpret_cast<const uint4 *>(X + (int64_t)row * D) + c);
        }
    };
    int64_t u, beg, un, bn;
    int len, ln, id;
    float y, y_next;
    load_range(item, u, beg, len);
    load_range(item + warps, un, bn, ln);
    load_ids(beg, len, id, y);
    load_rows(id);
    load_ids(bn, ln, id, y_next);
    while (true) {
        // the H rows as bfloat16 parts, [part][observation][feature]
        __syncwarp();
#pragma unroll
        for (int j = 0; j < G::PIECES; ++j) {
            const int p = lane + 32 * j, r = p / G::ROW_PIECES, c = p % G::ROW_PIECES;
            if constexpr (G::kF32) {
                uint32_t q[3][2];
                split_bf16(__uint_as_float(raw[j].x), __uint_as_float(raw[j].y), q[0][0], q[1][0], q[2][0]);
                split_bf16(__uint_as_float(raw[j].z), __uint_as_float(raw[j].w), q[0][1], q[1][1], q[2][1]);
#pragma unroll
                for (int k = 0; k < 3; ++k) *reinterpret_cast<uint2 *>(tile + (k * kObs + r) * G::ROW + c * 8) = make_uint2(q[k][0], q[k][1]);
            } else {
                *reinterpret_cast<uint4 *>(tile + r * G::ROW + c * 16) = raw[j];
            }
        }
        __syncwarp();
        int64_t ua, ba;
        int la;
        load_range(item + 2 * warps, ua, ba, la);
        if (un >= 0) load_rows(id);
        // Z = H B^-1: A = H (observations x features), B = B^-1; the parts' products from the smallest up
        constexpr int pa[6] = {G::kF32 ? 2 : 0, 0, G::kF32 ? 1 : 0, G::kF32 ? 1 : 0, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
        float z[G::NB][4];
#pragma unroll
        for (int n = 0; n < G::NB; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) z[n][e] = 0.f;
        const uint32_t src = ptx::smem_u32(tile) + ((lane & 7) + 8 * ((lane >> 3) & 1)) * G::ROW + 16 * (lane >> 4);
#pragma unroll 1
        for (int ks = 0; ks < G::KS; ++ks) {
            uint32_t a[G::PARTS][4];
#pragma unroll
            for (int q = 0; q < G::PARTS; ++q) ldmatrix_x4(src + q * kObs * G::ROW + 32 * ks, a[q]);
#pragma unroll
            for (int n2 = 0; n2 < G::NB / 2; ++n2) {
                uint4 b[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) b[q] = bf[((ks * (G::NB / 2) + n2) * 3 + q) * 32 + lane];
                if constexpr (G::kF32) {
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        mma_bf16(z[2 * n2], a[pa[q]], b[pb[q]].x, b[pb[q]].y);
                        mma_bf16(z[2 * n2 + 1], a[pa[q]], b[pb[q]].z, b[pb[q]].w);
                    }
                } else {
#pragma unroll
                    for (int q = 2; q >= 0; --q) {
                        mma_bf16(z[2 * n2], a[0], b[q].x, b[q].y);
                        mma_bf16(z[2 * n2 + 1], a[0], b[q].z, b[q].w);
                    }
                }
            }
        }
        // S = Z H^T: accumulator blocks 2 ks and 2 ks + 1 are the A fragment of K step ks; B = the observations' rows
        float s[2][4];
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[n][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < G::KS; ++ks) {
            uint32_t a[3][4], h[G::PARTS][4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                split_bf16(z[2 * ks + e / 2][2 * (e % 2)], z[2 * ks + e / 2][2 * (e % 2) + 1], a[0][e], a[1][e], a[2][e]);
#pragma unroll
            for (int q = 0; q < G::PARTS; ++q) ldmatrix_x4(src + q * kObs * G::ROW + 32 * ks, h[q]);
            if constexpr (G::kF32) {
#pragma unroll
                for (int q = 0; q < 6; ++q)
#pragma unroll
                    for (int n = 0; n < 2; ++n) mma_bf16(s[n], a[pa[q]], h[pb[q]][n], h[pb[q]][2 + n]);
            } else {
#pragma unroll
                for (int q = 2; q >= 0; --q)
#pragma unroll
                    for (int n = 0; n < 2; ++n) mma_bf16(s[n], a[q], h[0][n], h[0][2 + n]);
            }
        }
        // I + S, rows to lanes; S t = y
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int r = lane / 4, col = 8 * n + 2 * (lane % 4), q = col / 4, o = col & 3;
            *reinterpret_cast<float2 *>(S + panel_chunk(r, q) + o) = make_float2(s[n][0] + (r == col), s[n][1] + (r == col + 1));
            *reinterpret_cast<float2 *>(S + panel_chunk(r + 8, q) + o) = make_float2(s[n][2] + (r + 8 == col), s[n][3] + (r + 8 == col + 1));
        }
        __syncwarp();
        const bool ok = solve16(S, ex, __shfl_sync(0xFFFFFFFFu, y, lane & 15), t_s, dinv_s, lane);
        // w = Z^T t: this lane's rows lane / 4 and + 8 of every column pair, then the sum over the eight lanes with the same columns,
        // blocks halved with the lanes
        {
            const float t0 = t_s[lane / 4], t1 = t_s[lane / 4 + 8];
            float v[G::NB][2];
#pragma unroll
            for (int n = 0; n < G::NB; ++n) {
                v[n][0] = fmaf(z[n][2], t1, z[n][0] * t0);
                v[n][1] = fmaf(z[n][3], t1, z[n][1] * t0);
            }
#pragma unroll
            for (int h = G::NB / 2, o = 16; o >= 4; h /= 2, o /= 2) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int n = 0; n < G::NB / 2; ++n)
                    if (n < h)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float send = up ? v[n][e] : v[n + h][e], keep = up ? v[n + h][e] : v[n][e];
                            v[n][e] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
                        }
            }
            constexpr int LEFT = G::NB / 8;
            const int n0 = (((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)) * LEFT;
            T *row = reinterpret_cast<T *>(out.table) + u * D;
            const int slot = out.cap_slot ? out.cap_slot[u] : -1;
#pragma unroll
            for (int n = 0; n < LEFT; ++n) {
                const int f = 8 * (n0 + n) + 2 * (lane % 4);
                const float w0 = ok ? v[n][0] : 0.f, w1 = ok ? v[n][1] : 0.f;
                if constexpr (G::kF32) *reinterpret_cast<float2 *>(row + f) = make_float2(w0, w1);
                else *reinterpret_cast<uint32_t *>(row + f) = pack_bf16(w0, w1);
                if (slot >= 0) *reinterpret_cast<float2 *>(out.cap_out + (int64_t)slot * D + f) = make_float2(w0, w1);
            }
            if (!ok && lane == 0) {
                atomicAdd(&st->not_spd, 1ull);
                raise_flag(st, kFlagNotSpd, u);
            }
        }
        if (un < 0) return;
        y = y_next;
        load_ids(ba, la, id, y_next);
        item += warps;
        u = un;
        un = ua;
    }
}

template <int D, typename T>
cudaError_t launch_dt(const SideView &sv, int64_t first, int64_t count, const void *X, const void *ws, RowOut out, DevStatus *st, cudaStream_t s)
{
    using G = DGeo<D, T>;
    static_assert(G::SMEM <= 232448, "shared memory");
    static SmemOnce allow;
    const cudaError_t e = allow(k_dual_warp<D, T>, G::SMEM);
    if (e != cudaSuccess) return e;
    k_dual_warp<D, T><<<(unsigned)(count < 148 ? count : 148), G::WARPS * 32, G::SMEM, s>>>(
        sv, first, count, static_cast<const T *>(X), static_cast<const uint4 *>(ws), dual_warp_flag_ptr(ws, D), out, st);
    return cudaGetLastError();
}

}  // namespace

size_t dual_warp_workspace_bytes(int d) { return (size_t)3 * d * d * 2 + 256; }
const int *dual_warp_flag_ptr(const void *ws, int d) { return reinterpret_cast<const int *>(static_cast<const unsigned char *>(ws) + (size_t)3 * d * d * 2); }

cudaError_t launch_dual_warp_prepare(const float *Bmat, void *ws, int d, float cond_limit, cudaStream_t s, int64_t *launches)
{
    int *flag = const_cast<int *>(dual_warp_flag_ptr(ws, d));
    __nv_bfloat16 *frag = static_cast<__nv_bfloat16 *>(ws);
    if (d == 64) k_binv_fragments<64><<<1, SweepGeo<64>::THREADS, 0, s>>>(Bmat, frag, flag, (double)cond_limit);
    else if (d == 128) k_binv_fragments<128><<<1, SweepGeo<128>::THREADS, 0, s>>>(Bmat, frag, flag, (double)cond_limit);
    else return cudaErrorInvalidValue;
    ++*launches;
    return cudaGetLastError();
}

// rows sv.order[first .. first + count): rows of 1 .. 16 observations (degree class 1)
cudaError_t launch_rows_dual_warp(const SideView &sv, int64_t first, int64_t count, const void *X, int bf16, int d, const void *ws, RowOut out,
                                  DevStatus *st, cudaStream_t s, int64_t *launches)
{
    if (count <= 0) return cudaSuccess;
    ++*launches;
    if (d == 64 && bf16) return launch_dt<64, __nv_bfloat16>(sv, first, count, X, ws, out, st, s);
    if (d == 128 && !bf16) return launch_dt<128, float>(sv, first, count, X, ws, out, st, s);
    return cudaErrorInvalidValue;
}

}  // namespace alx
