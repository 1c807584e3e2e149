// Reader of the packed cache: scores and weighted values of a chunk of tokens on the integer tensor cores
// (tcgen05.mma.kind::i8, 32-bit integer accumulators in tensor memory).  Keys stored before the rotary embedding (ROPE): the
// values only; every token then sees another query, so the scores are no contraction and stay on the CUDA cores.
//
// A 2- or 4-bit code is an exact byte after one shift and one mask per FOUR (two) codes, and sums of byte products are
// exact, so the only rounding left is the one that puts the other operand in fixed point:
//   scores   <q, k_t> = sum_c (q_c scale_c) code_tc + sum_c q_c zero_c.  q_c scale_c, scaled by a power of two to 31 bits of
//            the group's largest one, is four signed base-256 digits; the product of the codes of 128 tokens (A: 128 x 128
//            bytes) with the digits (B: one column per token group, head and digit) gives four integers per token and
//            head, which are put together in float32.  31 bits of the largest term are more than a float32 sum keeps.
//   values   sum_t (w_t scale_tg) code_tc + sum_t w_t zero_tg.  The same with the roles turned: A = the codes transposed (the
//            same bytes in shared memory, described as M-major), B = the digits of w_t scale_tg, one column per channel
//            group, head and digit.  Accumulated over the chunk's tiles in tensor memory.  31 bits (28 at least) of the
//            largest product of the channel group and head in the chunk, however far the scales lie apart.
// A lane owns a token (its row of key codes, its weight, its value metadata); a warp makes the digits of the query for one
// token group.  Key codes are A in tensor memory (row = lane), so they never cross shared memory, whose wavefronts were the
// tightest pipe with both operands there (78 % busy); value codes, which must be read transposed, go through it.  The digits
// of four heads are one 16-byte store: an int's bytes ARE its base-256 digits, and B is described as N-major, so nothing is
// transposed.  Within a 32-bit word of codes the unpacking leaves the channels interleaved (byte i of piece j is channel
// (8 / BITS) i + j of the word); the same order is used for the other operand.
//
// Bound: HBM (bits / 8 + metadata bytes per cached element) for long caches.  The CUDA-core form that this replaces spent
// two instructions per code and head and was bound by them.  Whole call, 64 x 32 heads x 4096 tokens (1.07 GB): 374 -> 257 to 274
// us by box, 58 % of DRAM throughput in a capture of this kernel; 16 x 8 KV heads x 8160 tokens with four query heads each: 149 -> 60
// us.
#pragma once
#include <type_traits>
#include "attention.cuh"
#include "device_helpers.cuh"

namespace {

constexpr int D = SQUAT_D;
constexpr int THREADS = 128, WARPS = 4;
constexpr int TILE = ATTN_MMA_TILE, MAX_TILES = ATTN_MMA_MAX_TILES;


// Shared-memory matrix descriptors.  Codes: 128-byte rows (token), 128-byte swizzle, groups of 8 rows 1024 bytes apart;
// K-major for the scores (K = channel), M-major for the values (K = token).  Digits: no swizzle, N-major: 16 bytes of
// columns x 8 rows of K are one 128-byte piece, the next 8 rows follow 160 bytes on (leading offset; 160, so that the
// lanes' 16-byte stores fall on distinct banks), the next 16 columns come after all 128 rows (stride offset).
constexpr unsigned DIG_PIECE = 160, DIG_CHUNK = DIG_PIECE * (D / 8);
__device__ __forceinline__ u64 codes_desc(unsigned addr)
{
    return (u64)((addr & 0x3FFFF) >> 4) | ((u64)1 << 16) | ((u64)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ u64 digits_desc(unsigned addr)
{
    return (u64)((addr & 0x3FFFF) >> 4) | ((u64)(DIG_PIECE >> 4) << 16) | ((u64)(DIG_CHUNK >> 4) << 32) | (1ull << 46);
}
// instruction descriptor: int32 accumulator, A unsigned bytes, B signed bytes, M = 128, N = n, B N-major, A K-major (scores) or M-major (values)
__host__ __device__ constexpr unsigned idesc_i8(int n, bool a_m_major)
{
    return (2u << 4) | (1u << 10) | ((a_m_major ? 1u : 0u) << 15) | (1u << 16) | ((unsigned)(n >> 3) << 17) | ((128u >> 4) << 24);
}
// the same with A in tensor memory (row = lane, four bytes a column)
__device__ __forceinline__ void mma_i8_ta(unsigned d_taddr, unsigned a_taddr, u64 b_desc, unsigned idesc, unsigned accumulate)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n}"
                 ::"r"(d_taddr), "r"(a_taddr), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st16(unsigned taddr, const uint32_t (&r)[16])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_ld4(unsigned taddr, int (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}

// N scales or zero-points as they were loaded (float32 or binary16); they become floats where they are used, so that nothing
// waits for a load where it is issued
template <int N, bool M16>
struct Meta {
    using raw_t = typename std::conditional<M16, typename std::conditional<N == 4, uint2, typename std::conditional<N == 2, uint32_t, unsigned short>::type>::type,
                                            typename std::conditional<N == 4, float4, typename std::conditional<N == 2, float2, float>::type>::type>::type;
    raw_t raw;
    __device__ __forceinline__ void load(const void *p, long long i) { raw = __ldg(reinterpret_cast<const raw_t *>(p) + i); }   // i: in units of N
    __device__ __forceinline__ void get(float (&out)[N]) const
    {
        if constexpr (M16) {
            uint32_t w[2] = {0, 0};
            if constexpr (N == 4) { w[0] = raw.x; w[1] = raw.y; }
            else w[0] = raw;
#pragma unroll
            for (int g = 0; g < N; ++g) out[g] = __half2float(__ushort_as_half((unsigned short)(w[g / 2] >> (16 * (g & 1)))));
        } else if constexpr (N == 4) {
            out[0] = raw.x; out[1] = raw.y; out[2] = raw.z; out[3] = raw.w;
        } else if constexpr (N == 2) {
            out[0] = raw.x; out[1] = raw.y;
        } else {
            out[0] = raw;
        }
    }
};

// element by element, two at a time (N is 1 or even)
template <int N>
__device__ __forceinline__ void fma_n(float (&d)[N], const float (&a)[N], const float (&b)[N], const float (&c)[N])
{
    if constexpr (N == 1) d[0] = fmaf(a[0], b[0], c[0]);
    else {
#pragma unroll
        for (int i = 0; i < N; i += 2) unpack2(ffma2(pack2(a[i], a[i + 1]), pack2(b[i], b[i + 1]), pack2(c[i], c[i + 1])), d[i], d[i + 1]);
    }
}
template <int N>
__device__ __forceinline__ void mul_n(float (&d)[N], const float (&a)[N], const float (&b)[N])
{
    if constexpr (N == 1) d[0] = a[0] * b[0];
    else {
#pragma unroll
        for (int i = 0; i < N; i += 2) unpack2(fmul2(pack2(a[i], a[i + 1]), pack2(b[i], b[i + 1])), d[i], d[i + 1]);
    }
}

// Power of two that takes values up to mx (>= 0) to at most 2^30, and its inverse (NaN for a non-finite mx)
__device__ __forceinline__ float fixed_scale(float mx, float &inv)
{
    const int e = max((int)(__float_as_uint(mx) >> 23) & 0xff, 30);
    inv = e == 255 ? __uint_as_float(0x7fc00000u) : __uint_as_float((unsigned)(e - 29) << 23);
    return __uint_as_float((unsigned)(283 - e) << 23);
}
// round(x) as four signed base-256 digits, lowest in the lowest byte
__device__ __forceinline__ unsigned digits_of(float x)
{
    return ((unsigned)__float2int_rn(x) + 0x00808080u) ^ 0x00808080u;
}
// the number whose digits were multiplied, times inv
__device__ __forceinline__ float from_digits(const int (&d)[4], float inv)
{
    return fmaf((float)(d[3] * 256 + d[2]), 65536.0f, (float)(d[1] * 256 + d[0])) * inv;
}

// Unpacking leaves every code where it is in its byte: piece j of a word is (x >> 0) & (mask << BITS j), four bytes that
// hold 2^(BITS j) times a code.  The factor is a power of two: the query's digits take it out before they are rounded (31
// bits of the largest term, at least 25 for the last piece), the values' sums afterwards.
// the same for sums over a whole chunk, whose digits may not be joined in 32 bits
__device__ __forceinline__ float from_long_digits(const int (&d)[4], float inv)
{
    return fmaf(fmaf((float)d[3], 256.0f, (float)d[2]), 65536.0f, fmaf((float)d[1], 256.0f, (float)d[0])) * inv;
}

// byte k of an unpacked row holds this channel, 2^(BITS piece_at(k)) times its code
template <int BITS>
__device__ __forceinline__ int channel_at(int k)
{
    constexpr int PIECES = 8 / BITS, PER_WORD = 32 / BITS;     // pieces of four bytes per word of codes
    return k / PER_WORD * PER_WORD + (k & 3) * PIECES + (k % PER_WORD >> 2);
}
template <int BITS>
__device__ __forceinline__ int piece_at(int k) { return k % (32 / BITS) >> 2; }

template <int BITS, int NQ, int NG, bool ROPE>
struct Shape {
    static constexpr int N = NG * NQ * 4 < 16 ? 16 : NG * NQ * 4;
    static constexpr int TMEM_COLS = 32 + N > 64 ? 128 : 64;    // the keys' bytes, the accumulator of the scores, then of the values
    static constexpr int DIG_BYTES = N / 16 * (int)DIG_CHUNK;
    static constexpr size_t SMEM = 1024 + TILE * D + 2 * DIG_BYTES + sizeof(float) * MAX_TILES * TILE * NQ +
                                   (ROPE ? WARPS * (sizeof(float4) + NQ * sizeof(float2)) * 64 : 0);
};

// The residual buffer's rows (full precision, at most 128) as one more part beside the cache's chunks.  A warp takes 32
// rows, 16 at a time in flight, four channels a lane, so every load is a row's contiguous 256 (or 512) bytes; the sixteen
// sums over the lanes are made together by halving exchanges (16 shuffles; one row at a time would take 80).
template <int NQ, bool ROPE, bool BF16>
__device__ __forceinline__ void residual_part(const AttnParams &p, float *sm, int h, int b, int hq0, int nq_here, int parts)
{
    using row_t = typename std::conditional<BF16, uint2, float4>::type;
    constexpr int ROWS = 16;
    float *w_sm = sm, *acc_sm = w_sm + NQ * D, *red = acc_sm + WARPS * NQ * D;                     // red: [2][WARPS][NQ]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long base = ((long long)b * p.H + h) * p.R * D;
    auto load_row = [&](const void *src, int r) {
        row_t v = {};
        if (r < p.R) v = __ldg(reinterpret_cast<const row_t *>(reinterpret_cast<const unsigned char *>(src) + (base + (long long)r * D) * (BF16 ? 2 : 4)) + lane);
        return v;
    };
    auto as_f4 = [](const row_t &r) {
        if constexpr (BF16) return make_float4(bf16lo_to_f32(r.x), bf16hi_to_f32(r.x), bf16lo_to_f32(r.y), bf16hi_to_f32(r.y));
        else return r;
    };
    float4 q[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        q[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (j < nq_here) {
            const long long at = ((long long)b * p.Hq + hq0 + j) * D + 4 * lane;
            q[j] = make_float4(p.scale * attn_load_elem(p.q, at, p.q_bf16), p.scale * attn_load_elem(p.q, at + 1, p.q_bf16),
                               p.scale * attn_load_elem(p.q, at + 2, p.q_bf16), p.scale * attn_load_elem(p.q, at + 3, p.q_bf16));
        }
    }
    // lane's own row: 16 (lane mod 2) + lane / 2 of the warp's 32
    const int my_row = 32 * warp + 16 * (lane & 1) + (lane >> 1);
    float s[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) s[j] = -INFINITY;
#pragma unroll 1
    for (int bt = 0; bt < 2; ++bt) {
        const int r0 = 32 * warp + ROWS * bt;
        if (r0 >= p.R) break;                                   // warp-uniform
        row_t k[ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) k[i] = load_row(p.k_res, r0 + i);
        float v[NQ][ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            float4 x = as_f4(k[i]);
            if (ROPE) {
                // row t turns at position first_pos + T + t; lane l < 16 holds channels 4 l .. 4 l + 3, lane l + 16 their partners
                const long long pos = p.first_pos + p.T + min(r0 + i, p.R - 1);
                const float sign = lane < 16 ? -1.0f : 1.0f;
                float *e = &x.x;
                const float4 o = make_float4(__shfl_xor_sync(0xffffffffu, x.x, 16), __shfl_xor_sync(0xffffffffu, x.y, 16),
                                             __shfl_xor_sync(0xffffffffu, x.z, 16), __shfl_xor_sync(0xffffffffu, x.w, 16));
                const float oth[4] = {o.x, o.y, o.z, o.w};
                const float4 *ta = reinterpret_cast<const float4 *>(p.rope_a + (pos >> 5) * 64 + 4 * (lane & 15));
                const float4 *tb = reinterpret_cast<const float4 *>(p.rope_b + (pos & 31) * 64 + 4 * (lane & 15));
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    const float4 ca = __ldg(ta + c / 2), cb = __ldg(tb + c / 2);
                    const float c0 = fmaf(ca.x, cb.x, -ca.y * cb.y), s0 = fmaf(ca.y, cb.x, ca.x * cb.y);
                    const float c1 = fmaf(ca.z, cb.z, -ca.w * cb.w), s1 = fmaf(ca.w, cb.z, ca.z * cb.w);
                    e[c] = fmaf(e[c], c0, sign * oth[c] * s0);
                    e[c + 1] = fmaf(e[c + 1], c1, sign * oth[c + 1] * s1);
                }
            }
#pragma unroll
            for (int j = 0; j < NQ; ++j) v[j][i] = fmaf(q[j].x, x.x, fmaf(q[j].y, x.y, fmaf(q[j].z, x.z, q[j].w * x.w)));
        }
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
#pragma unroll
            for (int o = 16; o >= 2; o >>= 1) {                 // lane bit o picks the half of the rows that the lane goes on with
                const int n = o / 2;
                const bool up = lane & o;
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    const float send = up ? v[j][i] : v[j][i + n], keep = up ? v[j][i + n] : v[j][i];
                    v[j][i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            v[j][0] += __shfl_xor_sync(0xffffffffu, v[j][0], 1);
            if ((lane & 1) == bt && my_row < p.R) s[j] = v[j][0];
        }
    }
    float mx[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        mx[j] = warp_max(s[j]);
        if (lane == 0) red[warp * NQ + j] = mx[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        mx[j] = max_nan(max_nan(red[j], red[NQ + j]), max_nan(red[2 * NQ + j], red[3 * NQ + j]));
        const float w = expf(s[j] - mx[j]);
        w_sm[j * D + my_row] = w;
        const float den = attn_warp_sum(w);
        if (lane == 0) red[(WARPS + warp) * NQ + j] = den;
    }
    __syncwarp();
    float4 acc[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) acc[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 1
    for (int bt = 0; bt < 2; ++bt) {
        const int r0 = 32 * warp + ROWS * bt;
        if (r0 >= p.R) break;
        row_t vr[ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) vr[i] = load_row(p.v_res, r0 + i);
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const float4 x = as_f4(vr[i]);
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                const float w = w_sm[j * D + r0 + i];           // 0 past the last row
                acc[j].x = fmaf(w, x.x, acc[j].x); acc[j].y = fmaf(w, x.y, acc[j].y);
                acc[j].z = fmaf(w, x.z, acc[j].z); acc[j].w = fmaf(w, x.w, acc[j].w);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < NQ; ++j) *reinterpret_cast<float4 *>(acc_sm + (warp * NQ + j) * D + 4 * lane) = acc[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        if (j >= nq_here) break;
        const long long row = ((long long)b * p.Hq + hq0 + j) * parts + p.nchunk;
        const float *a = acc_sm + j * D + tid;
        p.part[row * D + tid] = (a[0] + a[NQ * D]) + (a[2 * NQ * D] + a[3 * NQ * D]);
        if (tid == 0) {
            const float *dn = red + WARPS * NQ + j;
            *reinterpret_cast<float2 *>(p.ml + row * 2) = make_float2(mx[j], (dn[0] + dn[NQ]) + (dn[2 * NQ] + dn[3 * NQ]));
        }
    }
}

// (x & MASK) | c as one three-input logic instruction
template <uint32_t MASK>
__device__ __forceinline__ uint32_t and_or(uint32_t x, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(x), "n"(MASK), "r"(c));
    return d;
}
// A constant the compiler has to keep in a register: `(x & mask) | constant` is then ONE three-input logic instruction
// (mask as its immediate); with both as immediates it takes two.
__device__ __forceinline__ uint32_t in_register(uint32_t v)
{
    uint32_t r;
    asm volatile("mov.b32 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
// 1 + code / 2^BITS as a float, for the code at position i of a 32-bit word (low bits first).  one_bits: the bit pattern of 1.0f, held in a register (in_register)
template <int BITS>
__device__ __forceinline__ float code_as_float(uint32_t w, int i, uint32_t one_bits)
{
    constexpr int TOP = 23 - BITS;                              // the code's low bit lands here
    constexpr uint32_t MASK = ((1u << BITS) - 1u) << TOP;
    const int pos = BITS * i;
    uint32_t sh = pos <= TOP ? (w << (TOP - pos)) : (w >> (pos - TOP));
    asm("" : "+r"(sh));                                        // keep the shift where it is (not re-associated behind the mask)
    return __uint_as_float(and_or<MASK>(sh, one_bits));
}

template <int BITS, int NQ, int NG, bool M16, bool ROPE>
__global__ void __launch_bounds__(THREADS, ATTN_CTAS_PER_SM(NQ, ROPE)) attn_mma_kernel(AttnParams p)
{
    using S = Shape<BITS, NQ, NG, ROPE>;
    constexpr int G = D / NG, WPT = D * BITS / 32;              // tokens (or channels) per group; 32-bit words per token
    constexpr uint32_t MASK = BITS == 2 ? 0x03030303u : 0x0F0F0F0Fu;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *codes_sm = smem_raw + (1024 - (smem_u32(smem_raw) & 1023)) % 1024;      // [128 rows][128 bytes] of value codes, swizzled
    unsigned char *digits_sm = codes_sm + TILE * D;                                        // [2][N / 16][16][8][16 bytes]
    float *sc_sm = reinterpret_cast<float *>(digits_sm + 2 * S::DIG_BYTES) + threadIdx.x;  // [tiles][NQ][128]: this lane's scores
    __shared__ __align__(8) u64 mbar;
    __shared__ unsigned tmem_sm;
    __shared__ float2 qz_sm[MAX_TILES][NG][NQ];                 // inverse of the fixed point, sum of query x zero-point
    __shared__ float red_sm[WARPS][NG * NQ + NQ + 2], top_sm[WARPS][NG * NQ];
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);       // (uniform)
    const int parts = p.nchunk + (p.R > 0), chunk = blockIdx.x % parts, qpass = blockIdx.x / parts;
    const int h = blockIdx.y, b = blockIdx.z;
    const int qpk = p.Hq / p.H, hq0 = h * qpk + qpass * NQ, nq_here = min(NQ, qpk - qpass * NQ);
    grid_wait(p.q, p.kc, p.vc, p.ks, p.kz, p.vs, p.vz, p.k_res, p.v_res, p.rope_a, p.rope_b);
    if (chunk == p.nchunk) {
        if (p.res_bf16) residual_part<NQ, ROPE, true>(p, reinterpret_cast<float *>(smem_raw), h, b, hq0, nq_here, parts);
        else residual_part<NQ, ROPE, false>(p, reinterpret_cast<float *>(smem_raw), h, b, hq0, nq_here, parts);
        return;
    }
    const int t0 = chunk * p.chunk, n_tok = min(p.T - t0, p.chunk), tiles = (n_tok + TILE - 1) / TILE;
    const long long ctok0 = (long long)b * p.csb + (long long)h * p.csh + t0;               // first token of the chunk

    // Codes of a tile.  Keys: lane = token, its whole row.  Values: a warp's 32 rows as contiguous 512-byte pieces, LPT lanes a
    // row (half the cache lines of the other form per load).  Past the end of the chunk its last token stands in (its score
    // is -inf, its weight 0), so that no load hangs on a condition.
    constexpr int LPT = WPT / 4, TPL = 32 / LPT;
    const unsigned char *k_base = p.kc + ctok0 * (D * BITS / 8), *v_base = p.vc + ctok0 * (D * BITS / 8) + lane % LPT * 16;
    const int v_tok = 32 * warp + lane / LPT, last_tok = n_tok - 1;
    uint4 cw[LPT];
    auto load_keys = [&](int tile) {
        const uint4 *src = reinterpret_cast<const uint4 *>(k_base + min(tile * TILE + tid, last_tok) * (D * BITS / 8));
#pragma unroll
        for (int i = 0; i < LPT; ++i) cw[i] = __ldg(src + i);
    };
    auto load_values = [&](int tile) {
#pragma unroll
        for (int i = 0; i < LPT; ++i) cw[i] = ldg128(v_base + min(tile * TILE + v_tok + TPL * i, last_tok) * (D * BITS / 8));
    };
    load_keys(0);
    // Which (token group, head) digits a warp makes: 4 / NG warps share a group and deal its heads among them.  A lane makes
    // those of channels 4 lane .. 4 lane + 3.
    constexpr int WPG = WARPS / NG, HPW = (NQ + WPG - 1) / WPG;
    const int my_group = warp / WPG, my_head0 = warp % WPG * HPW;
    const bool makes = my_head0 < NQ;
    Meta<4, M16> ks_next, kz_next;                              // scales and zero-points of those channels in the warp's group
    auto load_kmeta = [&](int tile) {
        const long long at = (ctok0 + min(tile * TILE + my_group * G, n_tok - G)) / G * (D / 4) + lane;
        ks_next.load(p.ks, at);
        kz_next.load(p.kz, at);
    };
    Meta<NG, M16> vs_next, vz_next;                             // this lane's token's value scales and zero-points
    auto load_vs = [&](int tile) { vs_next.load(p.vs, ctok0 + min(tile * TILE + tid, last_tok)); };
    auto load_vz = [&](int tile) { vz_next.load(p.vz, ctok0 + min(tile * TILE + tid, last_tok)); };
    if (!ROPE) load_kmeta(0);
    load_vs(0);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sm)), "r"((unsigned)S::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    constexpr int QH = ROPE ? NQ : HPW;                         // heads whose queries this warp holds: channels 4 lane + i,
    float q[QH][4];                                             // or (ROPE) lane + 32 i
    int dig_at[4];                                              // where the lane's digits go
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < QH; ++j) {
            const int qi = ROPE ? j : my_head0 + j, ch = ROPE ? lane + 32 * i : 4 * lane + i;
            q[j][i] = qi < nq_here ? p.scale * attn_load_elem(p.q, ((long long)b * p.Hq + hq0 + qi) * D + ch, p.q_bf16) : 0.0f;
        }
        const int k = BITS == 2 ? 16 * (lane >> 2) + 4 * i + (lane & 3) : 8 * (lane >> 1) + 4 * (i & 1) + 2 * (lane & 1) + (i >> 1);
        const int n = (my_group * NQ + my_head0) * 4;
        dig_at[i] = n / 16 * DIG_CHUNK + k / 8 * DIG_PIECE + k % 8 * 16 + n % 16;
    }
    float2 *lane_turn = reinterpret_cast<float2 *>(codes_sm);   // ROPE: [64][32] cos/sin of (lane theta_i), until the values come
    if (ROPE)
        for (int i = tid; i < 64 * 32; i += THREADS) lane_turn[i] = __ldg(p.rope_b + (i & 31) * 64 + (i >> 5));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = __shfl_sync(0xffffffffu, tmem_sm, 0), t_lanes = tmem + ((unsigned)(warp * 32) << 16), t_mine = t_lanes + 32 + my_group * NQ * 4;
    bool ok = true;

    // a row of key codes as 128 bytes in tensor memory, this lane's
    auto unpack_keys = [&]() {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            uint32_t r[16];
#pragma unroll
            for (int w = 0; w < WPT / 2; ++w) {
                const uint4 &v = cw[(half * WPT / 2 + w) / 4];
                const uint32_t x = w % 4 == 0 ? v.x : w % 4 == 1 ? v.y : w % 4 == 2 ? v.z : v.w;
#pragma unroll
                for (int j = 0; j < 8 / BITS; ++j) r[w * (8 / BITS) + j] = x & (MASK << (BITS * j));
            }
            tmem_st16(t_lanes + 16 * half, r);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    };
    // rows of value codes as 128 bytes in shared memory: 16-byte piece c of row r sits at piece c ^ (r mod 8)
    auto unpack_values = [&]() {
#pragma unroll
        for (int i = 0; i < LPT; ++i) {
            const int r = v_tok + TPL * i, swz = r & 7, c0 = lane % LPT * (8 / LPT);
            unsigned char *row = codes_sm + r * D;
            const uint32_t x[4] = {cw[i].x, cw[i].y, cw[i].z, cw[i].w};
            if (BITS == 2) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    *reinterpret_cast<uint4 *>(row + (((c0 + e) ^ swz) << 4)) = make_uint4(x[e] & MASK, x[e] & (MASK << 2), x[e] & (MASK << 4), x[e] & (MASK << 6));
            } else {
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    *reinterpret_cast<uint4 *>(row + (((c0 + e) ^ swz) << 4)) =
                        make_uint4(x[2 * e] & MASK, x[2 * e] & (MASK << 4), x[2 * e + 1] & MASK, x[2 * e + 1] & (MASK << 4));
            }
        }
    };
    // The four 32-deep steps of a tile's product: the codes advance by 32 channels (keys) or 32 tokens (values), the digits by
    // 32 rows.  One product is in flight at a time; the digits of the next one are made meanwhile in the other buffer.
    unsigned issued = 0;
    auto issue = [&](int buf, bool values, bool accumulate) {
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            const u64 a = codes_desc(smem_u32(codes_sm)), dg = digits_desc(smem_u32(digits_sm + buf * S::DIG_BYTES));
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (values) mma_i8(tmem + 32, a + s * 32 * D / 16, dg + s * 4 * DIG_PIECE / 16, idesc_i8(S::N, true), s > 0 || accumulate);
                else mma_i8_ta(tmem + 32, tmem + 8 * s, dg + s * 4 * DIG_PIECE / 16, idesc_i8(S::N, false), s > 0);
            }
            tc_commit(smem_u32(&mbar));
        }
        ++issued;
    };
    auto wait_product = [&]() {
        ok = mbar_wait(smem_u32(&mbar), (issued - 1) & 1) && ok;
        tc_fence_after();
    };

    // ---------------------------------------------------------------- scores
    constexpr int P = NG * NQ;                                  // (channel group, head) pairs, g NQ + j
    float mx[NQ], vmax = 0.0f, vmin = INFINITY;                 // largest score of a head; largest and smallest |value scale|
#pragma unroll
    for (int j = 0; j < NQ; ++j) mx[j] = -INFINITY;
    auto widen = [&]() {                                        // by the token in vs_next
        float vs[NG];
        vs_next.get(vs);
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            vmax = max_nan(vmax, fabsf(vs[g]));
            vmin = fminf(vmin, fabsf(vs[g]));
        }
    };
    auto read_scores = [&](int tile) {
        wait_product();
        int d[NQ][4];
#pragma unroll
        for (int j = 0; j < NQ; ++j) tmem_ld4(t_mine + j * 4, d[j]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        const bool in = tile * TILE + tid < n_tok;
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const float2 iz = qz_sm[tile][my_group][j];
            const float s = in ? from_digits(d[j], iz.x) + iz.y : -INFINITY;
            sc_sm[(tile * NQ + j) * TILE] = s;
            mx[j] = max_nan(mx[j], s);
        }
    };
    if constexpr (ROPE) {
        // Keys stored before the rotary embedding: token first_pos + 32 a + l of a warp turns by a block turn (a: applied to
        // the query instead, with the opposite sign) and a lane turn.  Every pair of channels is dequantized (one
        // multiply-add per element), turned (4) and multiplied with the block-turned query of every head (2 per head).
        float4 *sz = reinterpret_cast<float4 *>(sc_sm - tid + MAX_TILES * TILE * NQ) + warp * 64;      // (S_i, Z_i, S_{i+64}, Z_{i+64})
        float2 *qb = reinterpret_cast<float2 *>(reinterpret_cast<float4 *>(sc_sm - tid + MAX_TILES * TILE * NQ) + WARPS * 64) + warp * 64 * NQ;
        const uint32_t one_bits = in_register(0x3F800000u);
        constexpr float LV = float(1 << BITS);
        // the next tile's block turn and key metadata, asked for a tile ahead like the codes
        float2 turn[2];
        Meta<1, M16> ms[4], mz[4];
        auto load_block = [&](int tile) {
            const int tok = min(tile * TILE + 32 * warp, n_tok - 32);
            const long long mrow = (ctok0 + tok) / G * D, a_blk = (p.first_pos + t0 + tok) >> 5;
#pragma unroll
            for (int i = 0; i < 2; ++i) turn[i] = __ldg(p.rope_a + a_blk * 64 + lane + 32 * i);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                ms[i].load(p.ks, mrow + lane + 32 * i);
                mz[i].load(p.kz, mrow + lane + 32 * i);
            }
        };
        load_block(0);
#pragma unroll 1
        for (int tile = 0; tile < tiles; ++tile) {
            const int tok = tile * TILE + 32 * warp;                   // the warp's first token; n_tok is a multiple of 32
            if (tok < n_tok) {
                __syncwarp();
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int i = lane + 32 * hh;
                    const float2 cs = turn[hh];
#pragma unroll
                    for (int j = 0; j < NQ; ++j)
                        qb[j * 64 + i] = make_float2(fmaf(q[j][hh], cs.x, q[j][hh + 2] * cs.y), fmaf(q[j][hh + 2], cs.x, -q[j][hh] * cs.y));
                    float s0[1], s1[1], z0[1], z1[1];
                    ms[hh].get(s0); ms[hh + 2].get(s1);
                    mz[hh].get(z0); mz[hh + 2].get(z1);
                    sz[i] = make_float4(s0[0] * LV, z0[0] - s0[0] * LV, s1[0] * LV, z1[0] - s1[0] * LV);
                }
                __syncwarp();
            }
            float acc[NQ][2];
#pragma unroll
            for (int j = 0; j < NQ; ++j) acc[j][0] = acc[j][1] = 0.0f;
            if (tok < n_tok) {
                uint32_t wd[WPT];
#pragma unroll
                for (int i = 0; i < LPT; ++i) { wd[4 * i] = cw[i].x; wd[4 * i + 1] = cw[i].y; wd[4 * i + 2] = cw[i].z; wd[4 * i + 3] = cw[i].w; }
                constexpr int CPW = 32 / BITS;
#pragma unroll
                for (int wi = 0; wi < WPT / 2; ++wi)
#pragma unroll
                    for (int pos = 0; pos < CPW; ++pos) {
                        const int i = wi * CPW + pos;                  // pair (i, i + 64): same code position, WPT / 2 words apart
                        const float4 m4 = sz[i];
                        const float k0 = fmaf(code_as_float<BITS>(wd[wi], pos, one_bits), m4.x, m4.y);
                        const float k1 = fmaf(code_as_float<BITS>(wd[wi + WPT / 2], pos, one_bits), m4.z, m4.w);
                        const float2 cs = lane_turn[i * 32 + lane];
                        const float r0 = fmaf(k0, cs.x, -k1 * cs.y), r1 = fmaf(k0, cs.y, k1 * cs.x);
#pragma unroll
                        for (int j = 0; j < NQ; ++j) {
                            const float2 qq = qb[j * 64 + i];
                            acc[j][pos & 1] = fmaf(r1, qq.y, fmaf(r0, qq.x, acc[j][pos & 1]));
                        }
                    }
            }
            if (tile + 1 < tiles) {
                load_keys(tile + 1);
                load_block(tile + 1);
            } else {
                load_values(0);
            }
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                const float s = tok < n_tok ? acc[j][0] + acc[j][1] : -INFINITY;
                sc_sm[(tile * NQ + j) * TILE] = s;
                mx[j] = max_nan(mx[j], s);
            }
            widen();
            load_vs(tile + 1 < tiles ? tile + 1 : 0);               // (0: for the weighted values)
        }
        load_vz(0);
    } else {
#pragma unroll 1
        for (int tile = 0; tile < tiles; ++tile) {
            const int buf = tile & 1;
            float ks[4], kz[4];
            ks_next.get(ks);
            kz_next.get(kz);
            uint32_t dig[4][HPW];
#pragma unroll
            for (int j = 0; j < HPW; ++j) {
                const float zs = attn_warp_sum(fmaf(q[j][0], kz[0], q[j][1] * kz[1]) + fmaf(q[j][2], kz[2], q[j][3] * kz[3]));
                constexpr float P1 = BITS == 2 ? 0.25f : 0.0625f, P2 = BITS == 2 ? 0.0625f : 1.0f, P3 = BITS == 2 ? 0.015625f : 0.0625f;
                const float f[4] = {q[j][0] * ks[0], q[j][1] * ks[1], q[j][2] * ks[2], q[j][3] * ks[3]};
                float inv;
                const float up = fixed_scale(warp_max(max_nan(max_nan(fabsf(f[0]), fabsf(f[1])), max_nan(fabsf(f[2]), fabsf(f[3])))), inv);
                if (lane == 0 && my_head0 + j < NQ) qz_sm[tile][my_group][my_head0 + j] = make_float2(inv, zs);
                dig[0][j] = digits_of(f[0] * up);
                dig[1][j] = digits_of(f[1] * (up * P1));
                dig[2][j] = digits_of(f[2] * (up * P2));
                dig[3][j] = digits_of(f[3] * (up * P3));
            }
            if (tile + 1 < tiles) load_kmeta(tile + 1);
            if (makes) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    unsigned char *dst = digits_sm + buf * S::DIG_BYTES + dig_at[i];
                    if constexpr (HPW == 4) *reinterpret_cast<uint4 *>(dst) = make_uint4(dig[i][0], dig[i][1], dig[i][2], dig[i][3]);
                    else if constexpr (HPW == 2) *reinterpret_cast<uint2 *>(dst) = make_uint2(dig[i][0], dig[i][1]);
                    else *reinterpret_cast<uint32_t *>(dst) = dig[i][0];
                }
            }
            widen();
            load_vs(tile + 1 < tiles ? tile + 1 : 0);               // (0: for the weighted values)
            if (tile > 0) read_scores(tile - 1);                    // also frees the keys' columns and the accumulator
            unpack_keys();
            if (tile + 1 < tiles) load_keys(tile + 1);
            else load_values(0);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            __syncthreads();
            issue(buf, false, false);
        }
        load_vz(0);
        read_scores(tiles - 1);
    }

    // ---------------------------------------------------------------- maxima over the chunk
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        mx[j] = warp_max(mx[j]);
        if (lane == 0) red_sm[warp][j] = mx[j];
    }
    vmax = warp_max(vmax);
    vmin = warp_max(-vmin);
    if (lane == 0) {
        red_sm[warp][NQ] = vmax;
        red_sm[warp][NQ + 1] = vmin;
    }
    tc_fence_before();                                          // the score columns have been read; the values' product reuses them
    __syncthreads();
    auto over_warps = [](const auto &part, int i) { return max_nan(max_nan(part[0][i], part[1][i]), max_nan(part[2][i], part[3][i])); };
#pragma unroll
    for (int j = 0; j < NQ; ++j) mx[j] = over_warps(red_sm, j);
    vmax = over_warps(red_sm, NQ);
    // The digits of weight x value scale are to hold about 31 bits of the largest product of each channel group and head.  Where
    // all scales of the chunk lie within a factor of 8 the largest stands for the products (the largest weight is 1, so 28 bits are
    // the least).  Otherwise the products are looked at: channel groups may lie far apart, and a token far above the others may
    // carry no weight.  That takes another pass over the scores and a barrier, with one token of 256 30 times the rest 271 -> 282 us
    // on 64 x 32 heads x 4096 and 69 -> 73 on 16 x 8 KV heads x 8160 (cold caches); for every chunk it cost 4 to 6 %, the same maxima
    // taken as logarithms beside the scores 1 to 5 %, this test 0 to 2 %.
    float inv_v[NQ], up_v[P];                                   // inv_v: of the channel group that the warp reads at the end
    if (__builtin_expect(vmax <= -8.0f * over_warps(red_sm, NQ + 1), 1)) {
        float inv;
        const float up = fixed_scale(vmax, inv);
#pragma unroll
        for (int i = 0; i < P; ++i) up_v[i] = up;
#pragma unroll
        for (int j = 0; j < NQ; ++j) inv_v[j] = inv;
    } else {
        float top[P];
#pragma unroll
        for (int i = 0; i < P; ++i) top[i] = 0.0f;
#pragma unroll 2
        for (int tile = 0; tile < tiles; ++tile) {
            Meta<NG, M16> m;
            m.load(p.vs, ctok0 + min(tile * TILE + tid, last_tok));
            float vs[NG];
            m.get(vs);
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                const float w = expf(sc_sm[(tile * NQ + j) * TILE] - mx[j]);
#pragma unroll
                for (int g = 0; g < NG; ++g) top[g * NQ + j] = max_nan(top[g * NQ + j], fabsf(w * vs[g]));
            }
        }
#pragma unroll
        for (int i = 0; i < P; ++i) {
            top[i] = warp_max(top[i]);
            if (lane == 0) top_sm[warp][i] = top[i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < P; ++i) {
            float inv;
            up_v[i] = fixed_scale(over_warps(top_sm, i), inv);
            if (i / NQ == my_group) inv_v[i % NQ] = inv;
        }
    }

    // ---------------------------------------------------------------- weights, weighted values
    float zacc[P], den[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) den[j] = 0.0f;
#pragma unroll
    for (int i = 0; i < P; ++i) zacc[i] = 0.0f;
    unsigned char *const my_dig = digits_sm + tid / 8 * DIG_PIECE + tid % 8 * 16;
#pragma unroll 1
    for (int tile = 0; tile < tiles; ++tile) {
        const int buf = tile & 1;
        float w[NQ];
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            w[j] = expf(sc_sm[(tile * NQ + j) * TILE] - mx[j]);
            den[j] += w[j];
        }
        float vs[NG], vz[NG];
        vs_next.get(vs);
        vz_next.get(vz);
        if (tile + 1 < tiles) {
            load_vs(tile + 1);
            load_vz(tile + 1);
        }
        uint32_t dig[S::N / 4];
        float ww[P], ss[P], zz[P], x[P];
#pragma unroll
        for (int i = 0; i < P; ++i) { ww[i] = w[i % NQ]; ss[i] = vs[i / NQ]; zz[i] = vz[i / NQ]; }
        fma_n(zacc, ww, zz, zacc);
        mul_n(x, ww, ss);
        mul_n(x, x, up_v);                                      // (exact: a power of two)
#pragma unroll
        for (int i = 0; i < P; ++i) dig[i] = digits_of(x[i]);
#pragma unroll
        for (int i = P; i < S::N / 4; ++i) dig[i] = 0;
#pragma unroll
        for (int c = 0; c < S::N / 16; ++c)
            *reinterpret_cast<uint4 *>(my_dig + buf * S::DIG_BYTES + c * DIG_CHUNK) = make_uint4(dig[4 * c], dig[4 * c + 1], dig[4 * c + 2], dig[4 * c + 3]);
        if (tile > 0) wait_product();
        unpack_values();
        if (tile + 1 < tiles) load_values(tile + 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        issue(buf, true, tile > 0);
    }
    // sums of the weights and of weight x zero-point over the chunk
    __syncthreads();                                            // the maxima in red_sm have been read
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        den[j] = attn_warp_sum(den[j]);
        if (lane == 0) red_sm[warp][P + j] = den[j];
    }
#pragma unroll
    for (int i = 0; i < P; ++i) {
        zacc[i] = attn_warp_sum(zacc[i]);
        if (lane == 0) red_sm[warp][i] = zacc[i];
    }
    wait_product();
    int d[NQ][4];
#pragma unroll
    for (int j = 0; j < NQ; ++j) tmem_ld4(t_mine + j * 4, d[j]);       // lane = channel: a warp's 32 channels share a group
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    if (!ok) atomicOr(p.status, SQUAT_FLAG_DEVICE_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((unsigned)S::TMEM_COLS) : "memory");
    const int c = channel_at<BITS>(tid);
    const float per_piece = 1.0f / (float)(1 << BITS * piece_at<BITS>(tid));
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        if (j >= nq_here) break;
        const int zi = my_group * NQ + j;
        const float z = (red_sm[0][zi] + red_sm[1][zi]) + (red_sm[2][zi] + red_sm[3][zi]);
        const long long row = ((long long)b * p.Hq + hq0 + j) * parts + chunk;
        p.part[row * D + c] = from_long_digits(d[j], inv_v[j] * per_piece) + z;
        if (tid == 0) {
            const int di = P + j;
            *reinterpret_cast<float2 *>(p.ml + row * 2) = make_float2(mx[j], (red_sm[0][di] + red_sm[1][di]) + (red_sm[2][di] + red_sm[3][di]));
        }
    }
}


// the grid: token chunks (and the residual buffer, if any) x query-head passes, KV heads, batch
template <bool ROPE, int BITS, int NQ, int NG, bool M16>
int launch(const AttnParams &p, int qpasses, cudaStream_t st)
{
    constexpr size_t smem = Shape<BITS, NQ, NG, ROPE>::SMEM;
    static std::atomic<unsigned long long> allowed{0};
    if (const int rc = squat_allow_smem(reinterpret_cast<const void *>(attn_mma_kernel<BITS, NQ, NG, M16, ROPE>), smem, allowed)) return rc;
    return squat_launch(attn_mma_kernel<BITS, NQ, NG, M16, ROPE>, dim3((p.nchunk + (p.R > 0)) * qpasses, p.H, p.B), THREADS, smem, st, p);
}
template <bool ROPE, int BITS, int NQ>
int launch_g(const AttnParams &p, int qpasses, cudaStream_t st)
{
    if (p.meta16)
        return p.G == 32 ? launch<ROPE, BITS, NQ, 4, true>(p, qpasses, st) : p.G == 64 ? launch<ROPE, BITS, NQ, 2, true>(p, qpasses, st)
                                                                                        : launch<ROPE, BITS, NQ, 1, true>(p, qpasses, st);
    return p.G == 32 ? launch<ROPE, BITS, NQ, 4, false>(p, qpasses, st) : p.G == 64 ? launch<ROPE, BITS, NQ, 2, false>(p, qpasses, st)
                                                                                     : launch<ROPE, BITS, NQ, 1, false>(p, qpasses, st);
}
template <bool ROPE, int BITS>
int launch_q(const AttnParams &p, cudaStream_t st)
{
    const int qpk = p.Hq / p.H;
    return qpk == 1 ? launch_g<ROPE, BITS, 1>(p, 1, st) : qpk == 2 ? launch_g<ROPE, BITS, 2>(p, 1, st) : launch_g<ROPE, BITS, 4>(p, (qpk + 3) / 4, st);
}

}  // namespace
