// Warp-level matrix instructions and the small pieces that the row kernels built on them share (alx_rows_warp.cu,
// alx_rows_team.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace alx {

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
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
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

__device__ __forceinline__ float rsqrt_full(float p)
{
    float inv = rsqrtf(p);
    return inv * fmaf(-0.5f * p * inv, inv, 1.5f);      // one Newton step: full fp32 accuracy
}

// address (floats) of 16-byte chunk c of row r of a panel, swizzled so that eight lanes reading rows in a row meet every bank once
__device__ __forceinline__ int panel_chunk(int r, int c) { return r * 16 + 4 * (c ^ ((r >> 1) & 3)); }

// The bfloat16 parts p1, p2, p3 of (u, v), each the nearest to what the parts before it leave
__device__ __forceinline__ void split_bf16(float u, float v, uint32_t &p1, uint32_t &p2, uint32_t &p3)
{
    p1 = pack_bf16(u, v);
    const float u1 = u - bf16_lo(p1), v1 = v - bf16_hi(p1);
    p2 = pack_bf16(u1, v1);
    p3 = pack_bf16(u1 - bf16_lo(p2), v1 - bf16_hi(p2));
}

// S t = y for the warp's 16 x 16 matrix S (panel layout, both triangles; overwritten by L): lane l (and l + 16) = row l % 16, y its
// label.  Cholesky two columns per step, the new columns through `ex` (64 floats); t to t_s, reciprocal pivots to dinv_s (16
// floats each).  Returns whether every pivot was positive (one that is not makes its reciprocal root a NaN).
__device__ __forceinline__ bool solve16(float *S, float *ex, float y, float *t_s, float *dinv_s, int lane)
{
    const int rl = lane & 15;
    float a[16], b = y;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float4 v = *reinterpret_cast<const float4 *>(S + panel_chunk(rl, c));
        a[4 * c] = v.x; a[4 * c + 1] = v.y; a[4 * c + 2] = v.z; a[4 * c + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        const float p = __shfl_sync(0xFFFFFFFFu, a[j], j), q = __shfl_sync(0xFFFFFFFFu, a[j], j + 1), s = __shfl_sync(0xFFFFFFFFu, a[j + 1], j + 1);
        float z0 = __shfl_sync(0xFFFFFFFFu, b, j), z1 = __shfl_sync(0xFFFFFFFFu, b, j + 1);
        const float i0 = rsqrt_full(p), l10 = q * i0, i1 = rsqrt_full(fmaf(-l10, l10, s));
        z0 *= i0;
        z1 = fmaf(-z0, l10, z1) * i1;
        if (lane == 0) {
            *reinterpret_cast<float2 *>(t_s + j) = make_float2(z0, z1);
            *reinterpret_cast<float2 *>(dinv_s + j) = make_float2(i0, i1);
        }
        const float x0 = a[j] * i0, x1 = fmaf(-x0, l10, a[j + 1]) * i1;
        a[j] = x0;
        a[j + 1] = x1;
        b = fmaf(-x1, z1, fmaf(-x0, z0, b));
        if (j < 14) {
            float *e = ex + 32 * ((j / 2) & 1);
            if (lane < 16) { e[lane] = -x0; e[16 + lane] = -x1; }
            __syncwarp();
#pragma unroll
            for (int c = (j + 2) & ~3; c < 16; c += 4) {
                const float4 u = *reinterpret_cast<const float4 *>(e + c), v = *reinterpret_cast<const float4 *>(e + 16 + c);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int cc = c + 2 * h;
                    if (cc < j + 2) continue;
                    float2 t = make_float2(a[cc], a[cc + 1]);
                    t = __ffma2_rn(make_float2(x0, x0), h ? make_float2(u.z, u.w) : make_float2(u.x, u.y), t);
                    t = __ffma2_rn(make_float2(x1, x1), h ? make_float2(v.z, v.w) : make_float2(v.x, v.y), t);
                    a[cc] = t.x;
                    a[cc + 1] = t.y;
                }
            }
        }
    }
    __syncwarp();
    if (lane < 16)
#pragma unroll
        for (int c = 0; c < 4; ++c) *reinterpret_cast<float4 *>(S + panel_chunk(lane, c)) = make_float4(a[4 * c], a[4 * c + 1], a[4 * c + 2], a[4 * c + 3]);
    __syncwarp();
    int at[4];      // column rl of row r: r * 16 + at[(r / 2) % 4]
#pragma unroll
    for (int v = 0; v < 4; ++v) at[v] = 4 * ((rl >> 2) ^ v) + (rl & 3);
    float x = t_s[rl];
    const float d = dinv_s[rl];
    __syncwarp();
#pragma unroll
    for (int j = 15; j >= 0; --j) {
        const float xj = __shfl_sync(0xFFFFFFFFu, x * d, j);
        if (lane == 0) t_s[j] = xj;
        x = fmaf(-S[j * 16 + at[(j >> 1) & 3]], xj, x);      // (columns from j on are done with)
    }
    __syncwarp();
    return __ballot_sync(0xFFFFFFFFu, !(d == d)) == 0;
}

}  // namespace alx
