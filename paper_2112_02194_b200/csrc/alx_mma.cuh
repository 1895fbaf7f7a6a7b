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

}  // namespace alx
