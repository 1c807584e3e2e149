// What the reader's kernels share (attention.cu, attention_mma.cuh).
#pragma once
#include <cuda_fp16.h>
#include "squat_internal.cuh"

struct AttnParams {
    const void *q;             // [B, Hq, D]
    int q_bf16;
    int B, Hq, H, T;           // T: quantized tokens per (batch, head)
    const unsigned char *kc, *vc;
    const void *ks, *kz, *vs, *vz;   // float32, or binary16 in the M16 instances
    long long csb, csh;        // cache strides in tokens
    int G;
    const void *k_res, *v_res; // [B, H, R, D]
    int res_bf16, R;
    float scale;
    float *part;               // [B, Hq, parts, D], parts = nchunk and, if R > 0, the residual buffer
    float *ml;                 // [B, Hq, parts, 2]
    int nchunk, chunk;         // chunk: tokens per CTA, a power of two, 256 .. 1024
    float *out;                // [B, Hq, D]
    // rotary tables (pre-embedding key storage only): cos/sin of (32 a theta_i) [blocks][64] and of (l theta_i) [32][64]
    const float2 *rope_a, *rope_b;
    long long first_pos;       // position of cached token 0; a multiple of 32
    int meta16;                // the cache's scales and zero-points are binary16
    unsigned *status;          // device status word
};

__device__ __forceinline__ float attn_warp_sum(float v)
{
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    return v;
}

__device__ __forceinline__ float attn_load_elem(const void *p, long long idx, int bf16)
{
    if (bf16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(p)[idx]);
    return reinterpret_cast<const float *>(p)[idx];
}

constexpr int ATTN_MMA_TILE = 128;            // tokens per product
constexpr int ATTN_MMA_MAX_TILES = 8;         // tiles per CTA: chunks of at most 1024 tokens
// resident CTAs per SM the kernel is built for, by query heads per pass (96 or 128 registers: six CTAs of 80 were slower)
constexpr int ATTN_CTAS_PER_SM(int nq, bool rope) { return nq >= 4 || rope ? 4 : 5; }
int squat_launch_attn_mma(const AttnParams &p, int bits, cudaStream_t st);     // keys stored after the rotary embedding
int squat_launch_attn_rope(const AttnParams &p, int bits, cudaStream_t st);    // before it
