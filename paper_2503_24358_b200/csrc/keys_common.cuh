// What the key kernels that apply W through the tensor cores (keys.cu, keys_lane.cu, keys_block.cu) share: the image of the update matrix
// that pack_w_kernel writes, the instructions they issue, and the quantizer's small pieces.
#pragma once
#include "device_helpers.cuh"
#include <cuda_fp16.h>

constexpr int D = SQUAT_D;
constexpr float kMagic = 12582912.0f;     // 1.5 * 2^23: adding it rounds to an integer (ties to even)

// One head's image (see pack_w_kernel), blocks of 32 channels: diagonal blocks | hi panels | lo panels | the diagonal blocks once more, for
// the kernel that sweeps them in halves of 16.  Panel b holds the entries that lead from block b to the later channels, N = 96 - 32 b of them,
// K-major: float index (k / 4) * 4 N + 4 n + k % 4.
constexpr int KEY_BLK = 32, KEY_HALF = 16, KEY_NBLK = D / KEY_BLK;
constexpr int KEY_PLAIN_FLOATS = KEY_NBLK * KEY_BLK * KEY_BLK;
// a block in halves: first half onto itself (every entry twice) | first onto second | second onto itself (every entry twice)
constexpr int KEY_OWN_FLOATS = 2 * KEY_HALF * KEY_HALF, KEY_ACROSS_FLOATS = KEY_HALF * KEY_HALF;
constexpr int KEY_DIAG_BLK_FLOATS = 2 * KEY_OWN_FLOATS + KEY_ACROSS_FLOATS, KEY_DIAG_FLOATS = KEY_NBLK * KEY_DIAG_BLK_FLOATS;
__host__ __device__ constexpr int key_panel_off(int b) { return KEY_BLK * (b * (D - KEY_BLK) - KEY_BLK * (b * (b - 1) / 2)); }   // sum of 32 (96 - 32 i), i < b
constexpr int KEY_PANEL_FLOATS = key_panel_off(KEY_NBLK - 1);
constexpr int KEY_IMG_FLOATS = SQUAT_KEY_IMG_FLOATS;
static_assert(KEY_IMG_FLOATS == KEY_PLAIN_FLOATS + 2 * KEY_PANEL_FLOATS + KEY_DIAG_FLOATS, "what the handle allocates per head");
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
// 32 consecutive columns of the warp's lanes into registers (lane l gets row l)
__device__ __forceinline__ void tmem_ld32(unsigned taddr, unsigned (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// barrier `id` of nthreads threads
__device__ __forceinline__ void team_barrier(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
