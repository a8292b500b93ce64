#pragma once
// Exact products of fixed-point numbers on the tensor cores: 55 bits and sign in seven signed
// digits of base 256, each exact in bfloat16 (the scheme: large_digits.cu).
#include <stdint.h>

namespace mbe {

constexpr int DIGITS = 7;  // of base 256

// Signed base-256 digits of f (|f| <= 2^55), the most significant first, as bfloat16.
__device__ __forceinline__ void to_digits(long long f, uint16_t (&d)[DIGITS])
{
#pragma unroll
    for (int i = DIGITS - 1; i >= 0; --i) {
        const int v = i == 0 ? (int)f : (int)((f + 128) & 255) - 128;
        f = (f - v) >> 8;
        d[i] = (uint16_t)(__float_as_uint((float)v) >> 16);  // (exact: at most 8 significant bits)
    }
}

__device__ __forceinline__ uint32_t shared_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_trans(uint32_t (&r)[2], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, "
        "%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The seven sums of an element, joined (in units of 256^7).
__device__ __forceinline__ long long join_digits(const float (&acc)[DIGITS][4], int e)
{
    long long s = (long long)__float2int_rn(acc[0][e]);
#pragma unroll
    for (int d = 1; d < DIGITS - 1; ++d) s = s * 256 + __float2int_rn(acc[d][e]);
    return s + ((__float2int_rn(acc[DIGITS - 1][e]) + 128) >> 8);
}

}  // namespace mbe
