// What the key kernels that apply W through the tensor cores (keys.cu, keys_block.cu) share: the image of the update matrix
// that pack_w_kernel writes, the instructions they issue, and the quantizer's small pieces.
#pragma once
#include "device_helpers.cuh"
#include <cuda_fp16.h>

constexpr int D = SQUAT_D;
constexpr int BLK = 32;                   // channels per block of the image
constexpr int NBLK = D / BLK;             // 4
constexpr float kMagic = 12582912.0f;     // 1.5 * 2^23: adding it rounds to an integer (ties to even)

// One head's image (see pack_w_kernel): diagonal blocks | hi panels | lo panels
constexpr int TC_DIAG_FLOATS = NBLK * BLK * BLK;     // four 32 x 32 diagonal blocks of W^T
constexpr int TC_PANEL_FLOATS = BLK * (3 * BLK + 2 * BLK + BLK);     // panels of source blocks 0..2: (96 - 32 b) x 32
constexpr int TC_IMG_FLOATS = TC_DIAG_FLOATS + 2 * TC_PANEL_FLOATS;  // = d * d: diag | hi panels | lo panels
static_assert(TC_IMG_FLOATS == D * D, "the staged image of W has the size of W");
__host__ __device__ constexpr int tc_panel_off(int b) { return b == 0 ? 0 : (b == 1 ? 3 * BLK * BLK : 5 * BLK * BLK); }
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
__device__ __forceinline__ void team_barrier(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
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
