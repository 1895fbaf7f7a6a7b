// Inverse of the D x D base matrix B = alpha0 G + lambda I in fp64, by one block (both dual-form kernels need it once per
// half-epoch, and everything waits for it).
#pragma once
#include "alx_common.cuh"

namespace alx {

// Symmetric sweep (Gauss-Jordan on a positive definite matrix): pivot j turns a_ic into a_ic - a_ij a_jc / a_jj, the pivot's
// row and column into a_ij / a_jj and the pivot into -1 / a_jj; after all D pivots the matrix is -B^-1.  A thread keeps a
// 4 x 4 tile of the lower triangle in registers; a step hands on one column through shared memory (two buffers, one barrier).
// Bound: D dependent steps of barrier, shared-memory read, 16 FMAs a thread and the reciprocal of the next pivot, all in fp64 on
// one SM: about 1300 cycles each at d = 128, 680 at 64.  d = 128: 475 -> 92 us, d = 64: 137 -> 23 us (the Cholesky it replaces gave a row to a thread, with a division,
// a square root and three barriers per column, and then two triangular products as chains of shared-memory reads).
template <int D> struct SweepGeo {
    static constexpr int T = D / 4, TILES = T * (T + 1) / 2, THREADS = (TILES + 31) / 32 * 32;
};

template <int D> struct SweepSmem {
    double col[2][D];
    double inv[2];
    double red[2][SweepGeo<D>::THREADS / 32];
    int ok;
};

__device__ __forceinline__ double reciprocal(double p)
{
    // single-precision start, two Newton steps (relative error 2^-24 -> 2^-48 -> below fp64 rounding)
    double r = (double)(1.f / (float)p);
    r = r * fma(-p, r, 2.0);
    return r * fma(-p, r, 2.0);
}

// All SweepGeo<D>::THREADS threads.  emit(i, c, value): element (i, c) of B^-1, called once for every element.  Returns, to
// every thread, whether every pivot was positive; *cond = ||B||_F ||B^-1||_F.
template <int D, typename Emit>
__device__ bool sweep_inverse(const float *__restrict__ Bmat, SweepSmem<D> &sm, double *cond, Emit emit)
{
    using G = SweepGeo<D>;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const bool live = t < G::TILES;
    int I = 0;
    if (live) {
        I = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
        while ((I + 1) * (I + 2) / 2 <= t) ++I;
        while (I * (I + 1) / 2 > t) --I;
    }
    const int J = live ? t - I * (I + 1) / 2 : 0;
    const double twice = I == J ? 1.0 : 2.0;
    double a[4][4], fro = 0.0;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            a[r][c] = live ? (double)Bmat[(4 * I + r) * D + 4 * J + c] : 0.0;
            fro += a[r][c] * a[r][c];
        }
    fro *= live ? twice : 0.0;
    if (t == 0) sm.ok = 1;
    // hands on column j (rows from its own tile column, and the tile row's entries for the rows above it)
    auto publish = [&](int j) {
        const int jt = j >> 2, buf = j & 1;
        if (!live) return;
        if (J == jt) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c == (j & 3)) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) sm.col[buf][4 * I + r] = a[r][c];
                    if (I == jt) {
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            if (r == c) {
                                if (!(a[r][c] > 0.0)) sm.ok = 0;
                                sm.inv[buf] = reciprocal(a[r][c]);
                            }
                    }
                }
        } else if (I == jt) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (r == (j & 3)) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) sm.col[buf][4 * J + c] = a[r][c];
                }
        }
    };
    __syncthreads();
    publish(0);
    __syncthreads();
#pragma unroll 1
    for (int j4 = 0; j4 < D; j4 += 4) {
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const int j = j4 + jj, jt = j >> 2, buf = j & 1;
            const double inv = sm.inv[buf];
            double vr[4], vc[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                vr[e] = sm.col[buf][4 * I + e];
                vc[e] = sm.col[buf][4 * J + e] * inv;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) a[r][c] = fma(-vr[r], vc[c], a[r][c]);
            if (I == jt) {      // the pivot's row
#pragma unroll
                for (int c = 0; c < 4; ++c) a[jj][c] = vc[c];
            }
            if (J == jt) {      // ... and column
#pragma unroll
                for (int r = 0; r < 4; ++r) a[r][jj] = vr[r] * inv;
                if (I == jt) a[jj][jj] = -inv;
            }
            if (j + 1 < D) publish(j + 1);
            __syncthreads();
        }
    }
    double fro_inv = 0.0;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (live) {
                fro_inv += a[r][c] * a[r][c];
                emit(4 * I + r, 4 * J + c, -a[r][c]);
                if (I != J) emit(4 * J + c, 4 * I + r, -a[r][c]);
            }
    fro_inv *= twice;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fro += __shfl_xor_sync(0xFFFFFFFFu, fro, o);
        fro_inv += __shfl_xor_sync(0xFFFFFFFFu, fro_inv, o);
    }
    if (lane == 0) { sm.red[0][warp] = fro; sm.red[1][warp] = fro_inv; }
    __syncthreads();
    double f = 0.0, g = 0.0;
    for (int w = 0; w < G::THREADS / 32; ++w) { f += sm.red[0][w]; g += sm.red[1][w]; }
    *cond = sqrt(f) * sqrt(g);
    return sm.ok != 0;
}

}  // namespace alx
