// Reader of the packed cache: one decode step of attention (Section 2, "(Masked) Attention mechanism";
// the score vector w^deq = <q, deq(k_i)> / sqrt(d) of the proof of Theorem 1; the most recent tokens come
// from the full-precision residual buffer of Algorithm 1).
//
//   out_hq = softmax_i( s <q_hq, k_i> ) . v_i ,   k_i, v_i = dequantized cache rows, then the residual rows
//
// The cache is never dequantized to memory.  attn_mma_kernel (attention_mma.cuh) writes (unnormalised sum, max, denominator)
// for every chunk of tokens and for the residual buffer; attn_combine_kernel merges them.  It is launched as a programmatic
// dependent: its blocks are in place when the last chunk ends, which takes the gap between the two launches out.
//
// Keys stored BEFORE the rotary position embedding (Section 4, the "pre" variant): the reader applies the
// embedding on the fly.  Token t of the cache sits at position P = first_pos + t; channel pair (i, i + 64) of its
// dequantized key turns by the angle P * base^(-2i/128).  With P = 32 a + l the turn is the product of a block
// turn (32 a theta_i: the same for the 32 tokens of a warp step, so it is applied to the query instead, with the
// opposite sign) and a lane turn (l theta_i: a table in shared memory, one entry per lane and pair).  Cosines and
// sines come from two tables the host fills in float64 (squat_rope_table_fill); the kernel only multiplies.
#include "attention.cuh"

namespace {

constexpr int D = SQUAT_D;

// One CTA per (batch, query head), thread = channel: parts rescaled to the common maximum and added.
__global__ void __launch_bounds__(D) attn_combine_kernel(AttnParams p)
{
    const int hq = blockIdx.x, b = blockIdx.y, c = threadIdx.x, parts = p.nchunk + (p.R > 0);
    grid_wait(p.part, p.ml);
    const long long row = ((long long)b * p.Hq + hq) * parts;
    const float2 *ml = reinterpret_cast<const float2 *>(p.ml) + row;
    const float *part = p.part + row * D + c;
    float m = -INFINITY, acc = 0.0f, den = 0.0f;
    constexpr int AT_ONCE = 8;                 // parts whose loads are in flight together
#pragma unroll 1
    for (int s0 = 0; s0 < parts; s0 += AT_ONCE) {
        float2 v[AT_ONCE];
        float x[AT_ONCE];
#pragma unroll
        for (int i = 0; i < AT_ONCE; ++i) {
            const bool in = s0 + i < parts;
            v[i] = in ? ml[s0 + i] : make_float2(-INFINITY, 0.0f);
            x[i] = in ? part[(long long)(s0 + i) * D] : 0.0f;
        }
        float mn = m;
#pragma unroll
        for (int i = 0; i < AT_ONCE; ++i) mn = fmaxf(mn, v[i].x);
        const float f0 = expf(m - mn);
        acc *= f0;
        den *= f0;
#pragma unroll
        for (int i = 0; i < AT_ONCE; ++i) {
            const float f = expf(v[i].x - mn);
            acc = fmaf(f, x[i], acc);
            den = fmaf(f, v[i].y, den);
        }
        m = mn;
    }
    p.out[((long long)b * p.Hq + hq) * D + c] = acc / den;
}

}  // namespace

size_t squat_attention_workspace_floats(int batch, int n_q_heads, int n_tokens)
{
    const long long nchunk = (n_tokens + 255) / 256 + 1;         // the smallest chunk the launcher may choose, and the residual buffer
    return (size_t)batch * n_q_heads * nchunk * (D + 2);
}

int squat_launch_decode_attention(const void *q, int q_dtype, int batch, int Hq, int H, int T,
                                  const unsigned char *kc, const void *ks, const void *kz,
                                  const unsigned char *vc, const void *vs, const void *vz,
                                  long long csb, long long csh, int bits, int G,
                                  const void *k_res, const void *v_res, int res_dtype, int R,
                                  float scale, float *out, float *workspace,
                                  const float *rope_table, int rope_blocks, long long first_pos, int meta16, cudaStream_t st)
{
    AttnParams p;
    p.meta16 = meta16;
    p.rope_a = reinterpret_cast<const float2 *>(rope_table);                     // NULL: keys were stored after the embedding
    p.rope_b = p.rope_a ? p.rope_a + (size_t)rope_blocks * 64 : nullptr;
    p.first_pos = first_pos;
    p.q = q; p.q_bf16 = q_dtype == SQUAT_BF16; p.B = batch; p.Hq = Hq; p.H = H; p.T = T;
    p.kc = kc; p.vc = vc; p.ks = ks; p.kz = kz; p.vs = vs; p.vz = vz; p.csb = csb; p.csh = csh; p.G = G;
    p.k_res = k_res; p.v_res = v_res; p.res_bf16 = res_dtype == SQUAT_BF16; p.R = R;
    p.scale = scale; p.out = out;
    p.status = squat_status_word();
    if (!p.status) return SQUAT_ERR_CUDA;
    // Tokens per CTA.  A CTA costs its tiles (2.2 times as much where the scores stay on the CUDA cores) and about 1.5 tiles (4,
    // with the rotary table) more to begin and end; once there are more CTAs than places, the last of them leave half a CTA's time idle.  Long chunks
    // win where there are many waves (64 x 32 heads x 4096 tokens: 1024 tokens 267 us, 512 288), short ones where there are
    // about two (5 x 32 x 3520, pre-rotary: 81, 74) or less than one.
    const int qpk = Hq / H, nq = qpk >= 3 ? 4 : qpk, passes = (qpk + nq - 1) / nq;
    const double slots = (double)squat_sm_count() * ATTN_CTAS_PER_SM(nq, p.rope_a != nullptr), units = (double)batch * H * passes, tile = p.rope_a ? 2.2 : 1.0, begin = p.rope_a ? 4.0 : 1.5;
    double best = 0.0;
    p.chunk = 256;
    for (int chunk = 256; chunk <= ATTN_MMA_TILE * ATTN_MMA_MAX_TILES; chunk *= 2) {
        const int n = (T + chunk - 1) / chunk;
        const double cta = (T < chunk ? T : chunk) / (double)ATTN_MMA_TILE * tile + begin;
        const double all = units * (T / (double)ATTN_MMA_TILE * tile + begin * n + (R > 0 ? 2.0 : 0.0)) / slots;
        const double cost = units * (n + (R > 0)) <= slots ? cta : all + 0.5 * cta;
        if (chunk == 256 || cost < best) { best = cost; p.chunk = chunk; }
    }
    p.nchunk = (T + p.chunk - 1) / p.chunk;
    p.part = workspace;
    p.ml = workspace + (size_t)batch * Hq * (p.nchunk + (R > 0)) * D;
    const int rc = p.rope_a ? squat_launch_attn_rope(p, bits, st) : squat_launch_attn_mma(p, bits, st);
    if (rc != SQUAT_OK) return rc;
    return squat_launch(attn_combine_kernel, dim3(Hq, batch), D, 0, st, p);
}
