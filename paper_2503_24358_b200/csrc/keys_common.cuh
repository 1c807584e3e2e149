// What the key kernels that apply W through the tensor cores (keys.cu, keys_block.cu) share: the image of the update matrix
// that pack_w_kernel writes, the instructions they issue, and the quantizer's small pieces.
#pragma once
#include "device_helpers.cuh"
#include <cuda_fp16.h>

constexpr int D = SQUAT_D;
constexpr float kMagic = 12582912.0f;     // 1.5 * 2^23: adding it rounds to an integer (ties to even)

// One head's image (see pack_w_kernel), blocks of 16 channels: diagonal blocks doubled | hi panels | lo panels.  Panel b holds the
// entries that lead from block b to the later channels, N = 112 - 16 b of them, K-major: float index (k / 4) * 4 N + 4 n + k % 4.
constexpr int KEY_BLK = 16, KEY_NBLK = D / KEY_BLK;
constexpr int KEY_DIAG_FLOATS = 2 * KEY_NBLK * KEY_BLK * KEY_BLK;
__host__ __device__ constexpr int key_panel_off(int b) { return KEY_BLK * (b * (D - KEY_BLK) - KEY_BLK * (b * (b - 1) / 2)); }   // sum of 16 (112 - 16 i), i < b
constexpr int KEY_PANEL_FLOATS = key_panel_off(KEY_NBLK - 1);
constexpr int KEY_IMG_FLOATS = SQUAT_KEY_IMG_FLOATS;
static_assert(KEY_IMG_FLOATS == KEY_DIAG_FLOATS + 2 * KEY_PANEL_FLOATS, "what the handle allocates per head");
// instruction descriptor: fp32 accumulator, tf32 A and B, both K-major, N = n, M = 128
__host__ __device__ constexpr unsigned tc_idesc(int n) { return (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(n >> 3) << 17) | ((128u >> 4) << 24); }

__device__ __forceinline__ float min3_nan(float a, float b, float c)
{
    float r;
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Correctly rounded  rng / L  for L = 3 or 15 (q' = q + (rng - L q) * RN(1/L); checked against
// true division over full mantissa ranges on the host).
template <int BITS>
__device__ __forceinline__ float div_by_levels(float rng)
{
    constexpr float L = float((1 << BITS) - 1);
    constexpr float invL = 1.0f / L;
    const float q = __fmul_rn(rng, invL);
    const float r = __fmaf_rn(-L, q, rng);
    return __fmaf_rn(r, invL, q);
}

// shared-memory matrix descriptor, no swizzle, K-major: 8 x 16-byte core matrices, lbo bytes between the two
// halves of a K step, sbo bytes between groups of 8 rows
__device__ __forceinline__ u64 umma_desc(unsigned addr, unsigned lbo, unsigned sbo)
{
    return (u64)((addr & 0x3FFFF) >> 4) | ((u64)(lbo >> 4) << 16) | ((u64)(sbo >> 4) << 32) | (1ull << 46);
}
// D[128 x N] (+)= A[128 x 8] * B[N x 8]^T, tf32 operands from shared memory, fp32 accumulation in tensor memory
__device__ __forceinline__ void umma_tf32_ss(unsigned d_taddr, u64 a_desc, u64 b_desc, unsigned idesc, unsigned accumulate)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d_taddr), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// umma_tf32_ss with A from tensor memory (rows = lanes, 8 consecutive 32-bit columns)
__device__ __forceinline__ void umma_tf32_ts(unsigned d_taddr, unsigned a_taddr, u64 b_desc, unsigned idesc, unsigned accumulate)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}"
                 ::"r"(d_taddr), "r"(a_taddr), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ unsigned tf32_of(float x)             // round to nearest tf32 (10 mantissa bits)
{
    unsigned r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
