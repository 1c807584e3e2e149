// Key quantization with error feedback (Algorithm 1, function Quant; any update matrix W): two or four tokens per lane, for groups of 64
// and 128 (keys_lane.cu: one token per lane; the rule is at the launcher below).
//
// A group is G consecutive tokens of one (batch, head); its channels must be visited in order, each channel's grid needs min /
// max over the group's tokens, and each token's rounding error is pushed through W onto its later channels:
//
//   m, M  = min / max                -> scale = (M-m)/L, zero = m
//   c     = rint((x_j - m)/scale),  e = c*scale - (x_j - m)       (= deq(qtz(x_j)) - x_j)
//   x_j' += e * W[j'][j]
//
// Within a block of 32 channels the pushes are CUDA-core work (packed fma.rn.f32x2), one after the other in the order of the channels that
// make them; onto the channels of later blocks they are a dense product on the tcgen05 tensor cores, tf32 operands split in two.  The
// order of the sums, the products' operands and the decisions are those of keys_lane.cu: both kernels give the same bytes.
//
// Who holds what.  A CTA is 4 sweeping warps on 2 tiles of 128 tokens, two CTAs per SM; for groups of 128 on 4 tiles, one CTA.  Row r of
// a tile = tensor-memory lane r; warp w, lane l holds row 32 w + l of every tile, as pairs of tokens, so a read of W and every packed
// instruction serve two tokens, and a warp's tokens are whole groups: they join their extremes in the lane before the
// warp-wide reduction and never meet another warp.  Tensor memory, per tile: the corrections D[128 x 96] of channels 32 .. 127, and 32 more
// columns for the errors of block 0.  The errors E_hi of block b > 0 take the columns whose corrections that block reads, half
// a block ahead.  E_lo goes to shared memory as a K-major operand.
//
// A block is swept in halves of 16 channels.  Between them the first half's errors, read back from tensor memory, are pushed onto the
// second half's values.  Straight code for 32 channels was slower by a third (50 KB and more for four tokens per lane).
//
// Hand-over from block b to b + 1 (a fifth warp issues the products: a sweeping one that did took 2 000 cycles a hand-over over it), onto
// slices of 32 channels so that all products into a column have the same shape and are ordered by that:
//       next slice     D += E_lo Whi + E_hi Wlo + E_hi Whi     (commit: the next sweep waits for this)
//       the others     D += E_lo Whi                           (commit: with one buffer of E_lo the next sweep waits for this too)
//                      D += E_hi Wlo + E_hi Whi                (done while the next sweep runs)
//
// Bound: latency.  A channel's chain (two reductions, reciprocal, rounding, push onto the next channel) is 71
// cycles; one or two warps per scheduler make 160 to 200 of it.  128 heads x 32768 tokens take, in cycles of a unit of 128 channels, 25 000 (four
// tokens per lane) in sweeps, 8 000 in pushes onto second halves, 6 000 in waits for products.  keys_lane.cu -> here: 128 heads x 32768, G = 128, 4
// bits 1719 -> 1277 us, G = 64 1583 -> 1198; 32 heads x 4096, G = 128 59.0 -> 46.4, G = 64 54.4 -> 44.7; 64 x 32 heads x 128, G = 128 116 -> 94.
// On the way: products of the first half's E_lo issued behind it slowed the pushes by as much as they took from the hand-over; the
// loads of a half's keys all at once hold up every read of W for 1 000 to 2 000 cycles a block.
//
// Rounding decision.  t = (x - m) / scale is formed with the hardware reciprocal, so c0 = rint(t) can be off by one when t is within
// ~1e-6 of a rounding midpoint.  Channels that earlier channels have corrected hold generic float32 values and such near-ties are as
// rare as that bound; but channels nothing has corrected yet (the first g channels, or all of them when W = 0) hold raw bf16 / f32
// inputs, where exact ties are structural (x exactly half way between min and max).  In every block of 32 channels that has such a channel,
// and so always in the first, the remainder e0 = c0*scale - (x - m), which is exact next to a midpoint, is compared with
// +-scale/2: that settles the rounding exactly as real arithmetic on the stored float32 scale would, ties going to the even code (the
// threshold of an odd c0 is one ulp lower, so "remainder == scale/2" moves it), and the stored scale is the correctly rounded quotient
// (bit-identical to plain round-to-nearest quantization); elsewhere it is the product with RN(1/L), within one ulp of it.
//
// M16: scale and zero-point are stored as binary16.  The float32 values are rounded once more, and the decision and the error fed
// back are taken against the rounded (stored) values: t = (x - z16) / s16, clamped to [0, L] because z16 can lie above the minimum.
#include "keys_common.cuh"

namespace {

constexpr int KEY_WARPS = 4, KEY_THREADS = 32 * (KEY_WARPS + 1);      // four sweeping warps, one that issues the products
constexpr int KEY_COLS = 128, KEY_E0_COL = 96;                           // per tile: [0, 96) corrections, [96, 128) E_hi of block 0
constexpr int KEY_E_FLOATS = 128 * KEY_BLK;                              // one tile's E_lo
constexpr unsigned KEY_A_LBO = 128 * 16, KEY_SBO = 128;
constexpr unsigned kMagicBits = 0x4B400000u;

struct KeyParams {
    const float *Wimg;        // [H, KEY_IMG_FLOATS] staged images of the update matrices
    const void *k;
    long long sb, sh, st;     // element strides of k
    unsigned char *codes;
    void *scales, *zeros;     // float32, or binary16 in the M16 instances
    long long osb, osh;       // output strides in tokens
    int groups_per_bh;        // T / G
    int groups_per_head;      // B * T / G
    int units_per_head;       // 256 tokens each (512 with two pairs per lane)
    int total_units;
    unsigned *status;
    const int *words;         // device words: leading channels that no earlier channel corrects, and the image's block size;
    int not_form;             // not 0: an image of that block size is not this kernel's (see quantize_keys_impl)
#ifdef SQUAT_CHECKED
    SqExtent x_k, x_codes, x_scales, x_zeros, x_img;      // what the caller's tensors and the handle's images span
#endif
};

// Pairs of tokens per lane, by group size.  One pair (G = 64): two CTAs of two tiles per SM.  Two pairs (G = 128): one CTA of four tiles, so
// that a group is one warp's and its extremes never leave it.
__host__ __device__ constexpr int key_np(int G) { return G == 128 ? 2 : 1; }

template <int NP>
struct alignas(128) KeyShared {
    float diag[KEY_DIAG_FLOATS];                     // the image: diagonal blocks of W^T,
    float panels[2 * KEY_PANEL_FLOATS];              // hi | lo panels
    float e_lo[NP][2 * NP][KEY_E_FLOATS];               // two pairs per lane: two buffers
    float grid[KEY_WARPS][2][KEY_BLK];               // scales | zero-points of a block's channels
    u64 mbar_e, mbar_d, mbar_r;                     // a block's errors are in place (4 warps); products: those for the next block are done, E_lo is free
    u64 mbar_diag, mbar_pan;                        // parts of the image staged
    unsigned tmem, timeout, exact_channels;
};
static_assert(sizeof(KeyShared<1>) <= 113 * 1024, "two CTAs per SM");
static_assert(sizeof(KeyShared<2>) > 114 * 1024, "one CTA per SM: it takes all of tensor memory");

__device__ __forceinline__ void key_tmem_st1(unsigned taddr, float v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(__float_as_uint(v)));
}
__device__ __forceinline__ void key_tmem_ld4(unsigned taddr, unsigned (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void key_tmem_ld16(unsigned taddr, unsigned (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}

// 16 channels of the lane's tokens as they are in memory
template <bool BF16, int NP>
struct PairRows {
    uint4 v[2 * NP][BF16 ? 2 : 4];
    __device__ __forceinline__ float get(int i, int c) const
    {
        if (BF16) {
            const uint4 &t = v[i][c >> 3];
            const unsigned w = (c & 7) < 2 ? t.x : (c & 7) < 4 ? t.y : (c & 7) < 6 ? t.z : t.w;
            return (c & 1) ? bf16hi_to_f32(w) : bf16lo_to_f32(w);
        }
        const uint4 &t = v[i][BF16 ? 0 : c >> 2];
        return __uint_as_float((c & 3) == 0 ? t.x : (c & 3) == 1 ? t.y : (c & 3) == 2 ? t.z : t.w);
    }
};

// Half a block, 16 channels, for the lane's 2 NP tokens (pair i of x[channel]: tokens 2 i and 2 i + 1) of the warp's group.
// x: the channels' values, and behind the sweep their errors.  diag: the half's own part of the image.
// Written in the order in which it should run: a channel's chain (reductions 24 cycles, reciprocal 24, six dependent
// operations of 4 to 6: 71 in all) goes on to the next channel's reductions before what does not hurry: the other pushes, the
// codes and the errors' stores fill the waits.  The next row of W is read before this channel's stores, which may be to the same
// memory for all the compiler knows.  The errors of the last block are stored like the others (a test per store would cut the
// code into pieces) and used by nobody.
// EXACT: decisions through the remainder.  The usual instance decides so in channel 0 alone (raw values; `head`).  In the other
// channels of block 0 (`first`) it stores the rounded quotient too and says in `open` whether a remainder reached half a step: one element in
// a million, and the block is swept again by the EXACT instance, which so does not run in every unit (128 heads x 32768, G = 128: 1355 -> 1269
// us).  Deciding again at once, behind a branch per channel, made the sweep 1.6 times as long, and settling every channel in one
// code the call 1.3 times.
// ahead(jj): what is to be asked for at channel jj.
template <int BITS, int NP, bool EXACT, bool M16, class Ahead>
__device__ __forceinline__ void sweep_half(const Ahead &ahead, bool head, bool first, bool &open, u64 (&x)[KEY_HALF][NP], const float *__restrict__ diag, unsigned e_hi, float *__restrict__ e_lo,
                                           int lane, float *__restrict__ gscale, float *__restrict__ gzero, unsigned (&cw)[2 * NP][BITS / 2])
{
    constexpr float L = float((1 << BITS) - 1);
    constexpr int PER_WORD = 32 / BITS, NT = 2 * NP;
    // what the constant upper bits of the rounded floats add up to in a packed word
    constexpr unsigned K = [] { unsigned k = 0; for (int i = 0; i < PER_WORD; ++i) k += kMagicBits << (BITS * i); return k; }();
    const u64 magic2 = pack2(kMagic, kMagic), negl2 = pack2(-L, -L);
    float el[NT][4];                                    // [token][channel % 4]
    float m, mx;
    auto extremes = [&](const u64 (&x)[NP]) {
        float v[NT];
#pragma unroll
        for (int i = 0; i < NP; ++i) unpack2(x[i], v[2 * i], v[2 * i + 1]);
        if (NT == 2) {
            m = warp_min(min_nan(v[0], v[1]));
            mx = warp_max(max_nan(v[0], v[1]));
        } else {
            m = warp_min(min_nan(min3_nan(v[0], v[1], v[NT - 2]), v[NT - 1]));
            mx = warp_max(max_nan(max3_nan(v[0], v[1], v[NT - 2]), v[NT - 1]));
        }
    };
    u64 w[KEY_HALF];                                     // row jj, channels jj + 1 .. 15
    auto read_row = [&](int jj) {
#pragma unroll
        for (int q = (jj + 1) / 2; q < KEY_HALF / 2; ++q) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(diag + 2 * KEY_HALF * jj + 4 * q);
            w[2 * q] = t.x;
            w[2 * q + 1] = t.y;
        }
    };
    read_row(0);
    extremes(x[0]);
#pragma unroll
    for (int jj = 0; jj < KEY_HALF; ++jj) {
        const float rng = __fsub_rn(mx, m);
        float z = m, scale = EXACT || first ? div_by_levels<BITS>(rng) : __fmul_rn(rng, 1.0f / L), inv;
        if (M16) {
            scale = __half2float(__float2half_rn(scale));
            z = __half2float(__float2half_rn(m));
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(scale));
            inv = scale > 0.0f ? -inv : 0.0f;                                                   // scale 0 (no range, or underflow): codes 0
        } else {
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(fmaxf(rng, 1e-30f)));            // constant group: x - m = 0 -> code 0
        }
        const u64 z2 = pack2(z, z), scale2 = pack2(scale, scale), inv2 = pack2(inv, inv);
        u64 e[NP];
        float y[NT];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const u64 n = fsub2(z2, x[jj][i]);                                              // -(x - m)
            u64 y2 = ffma2(M16 ? n : fmul2(n, negl2), inv2, magic2);
            float &y0 = y[2 * i], &y1 = y[2 * i + 1];
            unpack2(y2, y0, y1);
            if (M16 && !EXACT && jj > 0) {
                y0 = fminf(fmaxf(y0, kMagic), kMagic + L);
                y1 = fminf(fmaxf(y1, kMagic), kMagic + L);
                y2 = pack2(y0, y1);
            }
            e[i] = ffma2(fsub2(y2, magic2), scale2, n);
            if (EXACT || (jj == 0 && (head || M16))) {
                float e0, e1, n0, n1;
                unpack2(e[i], e0, e1);
                unpack2(n, n0, n1);
                auto decide = [&](float nd, float &yy, float &ee) {
                    if (EXACT || head) {
                        const float thr = __uint_as_float(__float_as_uint(0.5f * scale) - (__float_as_uint(yy) & 1u));
                        const float adj = ee > thr ? -1.0f : (ee < -thr ? 1.0f : 0.0f);
                        yy = __fadd_rn(yy, adj);
                        ee = __fmaf_rn(adj, scale, ee);
                    }
                    if (M16) {
                        const float cc = fminf(fmaxf(yy, kMagic), kMagic + L);
                        ee = cc == yy ? ee : __fmaf_rn(__fsub_rn(cc, kMagic), scale, nd);
                        yy = cc;
                    }
                };
                decide(n0, y0, e0);
                decide(n1, y1, e1);
                e[i] = pack2(e0, e1);
            }
        }
        // the largest remainder that is no open question
        const float most = first && !(jj == 0 && head) ? __uint_as_float(__float_as_uint(0.5f * scale) - 1u) : __int_as_float(0x7f800000);
        // the next channel's value and extremes first
        if (jj + 1 < KEY_HALF) {
#pragma unroll
            for (int i = 0; i < NP; ++i) x[jj + 1][i] = ffma2(e[i], w[jj + 1], x[jj + 1][i]);
            extremes(x[jj + 1]);
        }
        if (!EXACT)
#pragma unroll
            for (int t = 0; t < NT; ++t) open |= fabsf((t & 1) ? hi_of(e[t / 2]) : lo_of(e[t / 2])) > most;
#pragma unroll
        for (int c = jj + 2; c < KEY_HALF; ++c)
#pragma unroll
            for (int i = 0; i < NP; ++i) x[c][i] = ffma2(e[i], w[c], x[c][i]);
        ahead(jj);
        if (jj + 1 < KEY_HALF) read_row(jj + 1);
        if (lane == 0) {
            gscale[jj] = scale;
            gzero[jj] = z;
        }
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            // the low bits of a rounded float are its code
            unsigned &c = cw[t][jj / PER_WORD];
            if (jj % PER_WORD == 0) c = 0u - K;
            c += __float_as_uint(y[t]) << (BITS * (jj % PER_WORD));
            // tf32 split by truncation: the tensor core reads only the top 19 bits of each word, so e itself serves as E_hi =
            // trunc(e), and E_lo = e - trunc(e) is exact in fp32
            const float ev = (t & 1) ? hi_of(e[t / 2]) : lo_of(e[t / 2]);
            key_tmem_st1(e_hi + t * KEY_COLS + jj, ev);
            el[t][jj & 3] = __fsub_rn(ev, __uint_as_float(__float_as_uint(ev) & 0xffffe000u));
            if ((jj & 3) == 3)
                *reinterpret_cast<float4 *>(e_lo + t * KEY_E_FLOATS + (jj >> 2) * (KEY_A_LBO / 4)) = make_float4(el[t][0], el[t][1], el[t][2], el[t][3]);
        }
    }
}

// The errors of a block's first half, read back from tensor memory, pushed onto the second half's values one by one in the channels'
// order.  x: pairs of channels (2 q, 2 q + 1) of the lane's tokens, so that an entry of W is read once and not twice: a broadcast read is
// charged by its width, and reads of W are the most of what shared memory does.  A loop over quads of channels:
// against straight code for all 16 it is faster for groups of 128 (1376 -> 1269 us for 128 heads x 32768) and slower for 64 (1164 -> 1197).
template <int NT>
__device__ __forceinline__ void push_across(u64 (&x)[KEY_HALF / 2][NT], unsigned e_hi, const float *__restrict__ across)
{
    unsigned e[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t) key_tmem_ld4(e_hi + t * KEY_COLS, e[t]);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll 1
    for (int j = 0; j < KEY_HALF; j += 4) {
        unsigned next[NT][4];                            // (behind the last quad this one again)
#pragma unroll
        for (int t = 0; t < NT; ++t) key_tmem_ld4(e_hi + t * KEY_COLS + min(j + 4, KEY_HALF - 4), next[t]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            u64 w[KEY_HALF / 2];
#pragma unroll
            for (int q = 0; q < KEY_HALF / 4; ++q) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(across + (j + i) * KEY_HALF + 4 * q);
                w[2 * q] = t.x;
                w[2 * q + 1] = t.y;
            }
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const u64 ee = pack2(__uint_as_float(e[t][i]), __uint_as_float(e[t][i]));
#pragma unroll
                for (int q = 0; q < KEY_HALF / 2; ++q) x[q][t] = ffma2(ee, w[q], x[q][t]);
            }
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < 4; ++i) e[t][i] = next[t][i];
    }
}

template <int BITS, int G, bool BF16, bool M16>
__global__ void __launch_bounds__(KEY_THREADS, 2 / key_np(G)) quant_keys_kernel(const KeyParams p)
{
    constexpr int NP = key_np(G), NT = 2 * NP, ES = BF16 ? 2 : 4;
    static_assert(32 * NT == G, "a warp's tokens are one group");
    constexpr unsigned TMEM_COLS = NT * KEY_COLS;
    extern __shared__ __align__(128) unsigned char smem_bytes[];
    KeyShared<NP> &sm = *reinterpret_cast<KeyShared<NP> *>(smem_bytes);
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);      // (uniform: tensor-memory addresses go by it)

    const int u_lo = (int)((long long)p.total_units * blockIdx.x / gridDim.x);
    const int u_hi = (int)((long long)p.total_units * (blockIdx.x + 1) / gridDim.x);
    grid_wait();
    if (p.not_form && p.words[1] == p.not_form) return;
    volatile unsigned *timeout = &sm.timeout;
    const unsigned mbar_e = smem_u32(&sm.mbar_e), mbar_d = smem_u32(&sm.mbar_d), mbar_r = smem_u32(&sm.mbar_r), mbar_diag = smem_u32(&sm.mbar_diag), mbar_pan = smem_u32(&sm.mbar_pan);

    // where the lane's tokens (one in each tile) come from and go to
    struct Place {
        const char *row;          // the lane's first token
        unsigned char *codes;
        long long meta;
        bool active;              // the group exists (a head's last unit may be ragged: past its end the last group is redone and not stored)
    };
    const long long row_step = 32 * p.st * ES;           // to the lane's next token
    auto locate = [&](int unit, Place &t) {
        const int h = unit / p.units_per_head, g = (unit - h * p.units_per_head) * KEY_WARPS + warp;
        t.active = g < p.groups_per_head;
        const int in_head = t.active ? g : p.groups_per_head - 1;
        const int b = in_head / p.groups_per_bh, grp = in_head - b * p.groups_per_bh;
        const int tok = grp * G + lane;
        const long long out_tok0 = (long long)b * p.osb + (long long)h * p.osh;
        t.row = static_cast<const char *>(p.k) + ((long long)b * p.sb + (long long)h * p.sh + (long long)tok * p.st) * ES;
        t.codes = p.codes + (out_tok0 + tok) * (D * BITS / 8);
        t.meta = (out_tok0 / G + grp) * D + lane;
    };
    PairRows<BF16, NP> raw;                              // of the half to come
    constexpr int ROW_PIECES = BF16 ? 2 : 4, PIECES = NT * ROW_PIECES;       // 16 bytes each
    auto load_piece = [&](const char *row, int i) {
        const int t = i / ROW_PIECES, c = i % ROW_PIECES;
        const char *src = row + t * row_step + 16 * c;
        if (SQ_CHK_G(p.status, src, 16, p.x_k)) raw.v[t][c] = *reinterpret_cast<const uint4 *>(src);
    };
    Place cur;
    if (u_lo < u_hi && warp < KEY_WARPS) {               // the first rows are on their way while the CTA sets itself up
        locate(u_lo, cur);
#pragma unroll
        for (int i = 0; i < PIECES; ++i) load_piece(cur.row, i);
    }

    auto stage = [&](int h) {            // one head's image (one thread)
        const float *src = p.Wimg + (long long)h * KEY_IMG_FLOATS;
        if (!SQ_CHK_G(p.status, src, KEY_IMG_FLOATS * 4, p.x_img)) return;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        auto copy = [&](unsigned dst, const float *from, unsigned bytes, unsigned mbar) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(dst), "l"(from), "r"(bytes), "r"(mbar) : "memory");
        };
        copy(smem_u32(sm.diag), src + KEY_PLAIN_FLOATS + 2 * KEY_PANEL_FLOATS, KEY_DIAG_FLOATS * 4, mbar_diag);       // the sweeps need only these
        copy(smem_u32(sm.panels), src + KEY_PLAIN_FLOATS, 2 * KEY_PANEL_FLOATS * 4, mbar_pan);
    };
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_e), "r"(KEY_WARPS) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_d), "r"(1) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_r), "r"(1) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_diag), "r"(1) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_pan), "r"(1) : "memory");
        sm.timeout = 0;
        sm.exact_channels = (unsigned)p.words[0];
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (u_lo < u_hi) stage(u_lo / p.units_per_head);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = __shfl_sync(0xffffffffu, *const_cast<volatile unsigned *>(&sm.tmem), 0);
    const unsigned t_mine = tmem + ((unsigned)(warp * 32) << 16);
    const int exact_channels = (int)sm.exact_channels;
    unsigned phase = 0, img_phase = 0;

    auto bounded_wait = [&](unsigned mbar, unsigned parity) {
        if (!*timeout && !mbar_wait(mbar, parity)) {
            *timeout = 1;
            atomicOr(p.status, SQUAT_FLAG_DEVICE_TIMEOUT);
        }
    };
    if (warp == KEY_WARPS) {
        // The issuing warp: one lane of it, always the same, issues, so its commits cover all earlier products.
        const u64 a_lo0 = umma_desc(smem_u32(sm.e_lo[0][0]), KEY_A_LBO, KEY_SBO);
        const unsigned pan = smem_u32(sm.panels);
        int staged = -1;
#pragma unroll 1
        for (int unit = u_lo; unit < u_hi; ++unit) {
            const int h = unit / p.units_per_head;
            if (h != staged) {
                if (staged >= 0) __syncthreads();
                bounded_wait(mbar_pan, img_phase);
                img_phase ^= 1;
                staged = h;
            }
#pragma unroll 1
            for (int blk = 0; blk + 1 < KEY_NBLK; ++blk) {
                const int nb = D - (blk + 1) * KEY_BLK;             // channels still to come
                const unsigned b_lbo = 16u * nb, bhi = pan + 4 * key_panel_off(blk), idesc = tc_idesc(KEY_BLK);
                const u64 step = (2 * b_lbo) >> 4;                 // 8 source channels on
                if (!SQ_CHK_C(p.status, key_panel_off(blk) + nb * KEY_BLK <= KEY_PANEL_FLOATS)) continue;
                // E_lo (shared memory) x Whi onto the slice-th 32 channels behind the block
                auto low = [&](int slice, int i) {
                    const unsigned d = tmem + i * KEY_COLS + (blk + slice) * KEY_BLK;
                    const u64 a_lo = a_lo0 + ((NP == 2 ? (blk & 1) * NT : 0) + i) * (KEY_E_FLOATS * 4 / 16), hi = umma_desc(bhi + 16u * KEY_BLK * slice, b_lbo, KEY_SBO);
#pragma unroll
                    for (int ks = 0; ks < KEY_BLK / 8; ++ks) umma_tf32_ss(d, a_lo + ks * (2 * KEY_A_LBO / 16), hi + ks * step, idesc, (blk | ks) != 0);
                };
                // then E_hi (tensor memory) x Wlo and x Whi
                auto high = [&](int slice, int i) {
                    const unsigned d = tmem + i * KEY_COLS + (blk + slice) * KEY_BLK, a_hi = tmem + i * KEY_COLS + (blk == 0 ? KEY_E0_COL : (blk - 1) * KEY_BLK);
                    const u64 hi = umma_desc(bhi + 16u * KEY_BLK * slice, b_lbo, KEY_SBO), lo = hi + KEY_PANEL_FLOATS * 4 / 16;
#pragma unroll
                    for (int ks = 0; ks < KEY_BLK / 8; ++ks) umma_tf32_ts(d, a_hi + 8 * ks, lo + ks * step, idesc, 1u);
#pragma unroll
                    for (int ks = 0; ks < KEY_BLK / 8; ++ks) umma_tf32_ts(d, a_hi + 8 * ks, hi + ks * step, idesc, 1u);
                };
                bounded_wait(mbar_e, phase);
                phase ^= 1;
                tc_fence_after();
                if (elect_one()) {
                    const int slices = KEY_NBLK - 1 - blk;
#pragma unroll 1
                    for (int i = 0; i < NT; ++i) {
                        low(0, i);
                        high(0, i);
                    }
                    tc_commit(mbar_d);
#pragma unroll 1
                    for (int slice = 1; slice < slices; ++slice)
#pragma unroll 1
                        for (int i = 0; i < NT; ++i) low(slice, i);
                    if (NP == 1) tc_commit(mbar_r);
#pragma unroll 1
                    for (int slice = 1; slice < slices; ++slice)
#pragma unroll 1
                        for (int i = 0; i < NT; ++i) high(slice, i);
                }
                __syncwarp();
            }
        }
        // Every batch of products has been waited for by the sweeping warps unless a wait ran out; then commit once more and
        // give the tensor core a bounded time to drain before the columns are handed back.
        if (*timeout) {
            if (elect_one()) tc_commit(mbar_pan);
            mbar_wait(mbar_pan, img_phase);
        }
        tc_fence_before();
        __syncthreads();
        return;
    }

    int staged = -1;
#pragma unroll 1
    for (int unit = u_lo; unit < u_hi; ++unit) {
        const int h = unit / p.units_per_head;
        if (h != staged) {
            if (staged >= 0) {                           // (the first copy was started at kernel entry)
                // every read of the old image is over: by the lanes, and by the products, the last of which were waited for
                __syncthreads();
                if (threadIdx.x == 0) stage(h);
            }
            bounded_wait(mbar_diag, img_phase);
            img_phase ^= 1;
            staged = h;
        }
        Place nxt = cur;
        if (unit + 1 < u_hi) locate(unit + 1, nxt);
#pragma unroll 1
        for (int blk = 0; blk < KEY_NBLK; ++blk) {
            const bool more = blk + 1 < KEY_NBLK, first = blk == 0 && exact_channels > 0;
            bool exact = exact_channels > max(1, blk * KEY_BLK), open = false;
            const float *diag = sm.diag + blk * KEY_DIAG_BLK_FLOATS;
            const unsigned d_col = t_mine + (blk - 1) * KEY_BLK, e_hi = blk == 0 ? t_mine + KEY_E0_COL : d_col;
            float *e_lo = &sm.e_lo[NP == 2 ? blk & 1 : 0][0][(warp * 32 + lane) * 4];
            constexpr int E_HALF = KEY_HALF / 4 * (KEY_A_LBO / 4);
            // (recorded only: every address of a sweep is a constant away from these)
            (void)SQ_CHK_R(p.status, e_lo, (KEY_E_FLOATS * (NT - 1) + (KEY_BLK / 4 - 1) * KEY_A_LBO / 4 + 4) * 4, sm.e_lo[NP == 2 ? blk & 1 : 0], sizeof(sm.e_lo[0]));
            (void)SQ_CHK_R(p.status, diag, KEY_DIAG_BLK_FLOATS * 4, sm.diag, sizeof(sm.diag));
            (void)SQ_CHK_C(p.status, (e_hi & 0xffffu) >= (tmem & 0xffffu) && (e_hi & 0xffffu) + KEY_BLK <= (tmem & 0xffffu) + KEY_COLS);
            unsigned cw[NT][BITS / 2], cw_first[NT][BITS / 2];
            if (blk > 0) {
                bounded_wait(mbar_d, phase);             // the products that complete this block's corrections
                if (NP == 1) bounded_wait(mbar_r, phase);       // and have read E_lo, which is written next
                phase ^= 1;
                tc_fence_after();
            }
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                u64 x[KEY_HALF][NP];                     // the half's values
                {
                    u64 v[KEY_HALF / 2][NT];             // by pairs of channels
#pragma unroll
                    for (int q = 0; q < KEY_HALF / 2; ++q)
#pragma unroll
                        for (int t = 0; t < NT; ++t) v[q][t] = pack2(raw.get(t, 2 * q), raw.get(t, 2 * q + 1));
                    if (blk > 0) {
                        unsigned d[NT][16];
#pragma unroll
                        for (int t = 0; t < NT; ++t) key_tmem_ld16(d_col + t * KEY_COLS + half * KEY_HALF, d[t]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int q = 0; q < KEY_HALF / 2; ++q)
#pragma unroll
                            for (int t = 0; t < NT; ++t) v[q][t] = fadd2(v[q][t], pack2(__uint_as_float(d[t][2 * q]), __uint_as_float(d[t][2 * q + 1])));
                    }
                    if (half == 1) {
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                        push_across<NT>(v, e_hi, diag + KEY_OWN_FLOATS);
#pragma unroll
                        for (int i = 0; i < NT; ++i)
#pragma unroll
                            for (int w = 0; w < BITS / 2; ++w) cw_first[i][w] = cw[i][w];
                    }
#pragma unroll
                    for (int c = 0; c < KEY_HALF; ++c)
#pragma unroll
                        for (int i = 0; i < NP; ++i)
                            x[c][i] = (c & 1) ? pack2(hi_of(v[c / 2][2 * i]), hi_of(v[c / 2][2 * i + 1])) : pack2(lo_of(v[c / 2][2 * i]), lo_of(v[c / 2][2 * i + 1]));
                }
                const float *own = diag + half * (KEY_OWN_FLOATS + KEY_ACROSS_FLOATS);
                float *gscale = sm.grid[warp][0] + half * KEY_HALF, *gzero = sm.grid[warp][1] + half * KEY_HALF;
                // The keys of the next half, a few pieces at a channel: a lane's rows are 32 cache lines per load, so a half's loads at once
                // keep the load unit, and whoever reads W, waiting (1 000 to 2 000 cycles a block).  Behind a CTA's last half these again.
                const Place &place = half == 1 && !more ? nxt : cur;
                const int at = half == 0 ? blk * KEY_BLK + KEY_HALF : more ? (blk + 1) * KEY_BLK : 0;
                const char *row = place.row + at * ES;
                auto ahead = [&](int jj) {
                    constexpr int PER = PIECES > 8 ? PIECES / 8 : 1, STEP = PIECES < 8 ? 8 / PIECES : 1;
                    if (jj < 8 && jj % STEP == 0)
#pragma unroll
                        for (int i = 0; i < PER; ++i) load_piece(row, jj / STEP * PER + i);
                };
                if (exact) sweep_half<BITS, NP, true, M16>(ahead, false, false, open, x, own, e_hi + half * KEY_HALF, e_lo + half * E_HALF, lane, gscale, gzero, cw);
                else sweep_half<BITS, NP, false, M16>(ahead, first && half == 0, first, open, x, own, e_hi + half * KEY_HALF, e_lo + half * E_HALF, lane, gscale, gzero, cw);
                if (half == 1 && !exact && first && __any_sync(0xffffffffu, open)) {      // once more, from its keys
                    exact = true;
                    half = -1;
#pragma unroll
                    for (int i = 0; i < PIECES; ++i) load_piece(cur.row, i);
                }
            }

            // E_hi is in tensor memory; behind the last block too, whose columns the next unit's products, or another kernel, write next
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            if (more) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // E_lo rows, for the tensor core
                tc_fence_before();
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar_e) : "memory");
            }
            __syncwarp();                                // (the grids lane 0 wrote)
            const int at = blk * KEY_BLK;
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                unsigned char *cp = cur.codes + i * (32 * D * BITS / 8) + at * BITS / 8;
                if (cur.active && SQ_CHK_G(p.status, cp, 32 * BITS / 8, p.x_codes)) {
                    if (BITS == 2) *reinterpret_cast<uint2 *>(cp) = make_uint2(cw_first[i][0], cw[i][0]);
                    else *reinterpret_cast<uint4 *>(cp) = make_uint4(cw_first[i][0], cw_first[i][BITS / 2 - 1], cw[i][0], cw[i][BITS / 2 - 1]);
                }
            }
            {
                const float2 sz = make_float2(sm.grid[warp][0][lane], sm.grid[warp][1][lane]);
                const long long meta = cur.meta + at;
                if (cur.active && SQ_CHK_G(p.status, static_cast<char *>(p.scales) + meta * (M16 ? 2 : 4), M16 ? 2 : 4, p.x_scales) &&
                    SQ_CHK_G(p.status, static_cast<char *>(p.zeros) + meta * (M16 ? 2 : 4), M16 ? 2 : 4, p.x_zeros)) {
                    if (M16) {
                        static_cast<__half *>(p.scales)[meta] = __float2half_rn(sz.x);      // exact
                        static_cast<__half *>(p.zeros)[meta] = __float2half_rn(sz.y);
                    } else {
                        static_cast<float *>(p.scales)[meta] = sz.x;
                        static_cast<float *>(p.zeros)[meta] = sz.y;
                    }
                    if (!(sz.x > 0.0f && sz.x < __int_as_float(0x7f800000)))
                        atomicOr(p.status, sz.x == 0.0f ? SQUAT_FLAG_ZERO_RANGE : SQUAT_FLAG_NONFINITE);
                }
            }
            __syncwarp();                                // before the next sweep writes grids
        }
        cur = nxt;
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Writes, per head, the image from which the key kernels stage what they need:
//   diagonal          the four 32 x 32 blocks of W^T, row-major: block b, row jj, column c = W^T[32 b + jj][32 b + c]
//   hi panels         of source blocks b = 0, 1, 2: B_b(n, k) = W[32 (b + 1) + n][32 b + k] = W^T[32 b + k][32 (b + 1) + n],
//                     n < 96 - 32 b, k < 32, rounded to tf32, K-major in 8 x 16-byte core matrices:
//                     float index (k / 4) * 4 N + 4 n + k % 4 with N = 96 - 32 b
//   lo panels         tf32(W - hi), same layout
//   halves            of every diagonal block: its first half's rows and columns, row-major, every entry as a pair of equal floats;
//                     its first half's rows and second half's columns, row-major; its second half's rows and columns like the first's
// Grid (heads, slices): the kernel is a chain of two dependent global accesses, so more CTAs, not more work per thread, shorten
// it; each thread takes (panel, 4-k chunk, channel n): four coalesced row reads, one 16-byte store.
__global__ void __launch_bounds__(256) pack_w_kernel(const float *__restrict__ Wt, float *__restrict__ Wimg, int exact_channels,
                                                     int block_form, int *__restrict__ words_dev)
{
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {      // these travel with the matrices they describe
        words_dev[0] = exact_channels;
        words_dev[1] = block_form;
    }
    const float *src = Wt + (long long)blockIdx.x * D * D;
    float *img = Wimg + (long long)blockIdx.x * KEY_IMG_FLOATS;
    const int first = blockIdx.y * blockDim.x + threadIdx.x, stride = gridDim.y * blockDim.x;
    for (int i = first; i < KEY_PLAIN_FLOATS / 4; i += stride) {
        const int b = i / (KEY_BLK * KEY_BLK / 4), r = i % (KEY_BLK * KEY_BLK / 4), jj = r / (KEY_BLK / 4), c4 = r % (KEY_BLK / 4);
        reinterpret_cast<float4 *>(img)[i] = __ldg(reinterpret_cast<const float4 *>(src + (b * KEY_BLK + jj) * D + b * KEY_BLK + 4 * c4));
    }
    float *hi = img + KEY_PLAIN_FLOATS, *lo = hi + KEY_PANEL_FLOATS, *halves = lo + KEY_PANEL_FLOATS;
    for (int i = first; i < KEY_NBLK * KEY_DIAG_BLK_FLOATS / 4; i += stride) {
        const int b = i / (KEY_DIAG_BLK_FLOATS / 4), r = i % (KEY_DIAG_BLK_FLOATS / 4) * 4, part = (r >= KEY_OWN_FLOATS) + (r >= KEY_OWN_FLOATS + KEY_ACROSS_FLOATS);
        const float *from = src + (b * KEY_BLK + (part == 2 ? KEY_HALF : 0)) * D + b * KEY_BLK + (part > 0 ? KEY_HALF : 0);
        if (part == 1) {
            const int at = r - KEY_OWN_FLOATS;
            reinterpret_cast<float4 *>(halves)[i] = __ldg(reinterpret_cast<const float4 *>(from + at / KEY_HALF * D + at % KEY_HALF));
        } else {
            const int at = (r - (part == 2 ? KEY_OWN_FLOATS + KEY_ACROSS_FLOATS : 0)) / 2;
            const float2 v = __ldg(reinterpret_cast<const float2 *>(from + at / KEY_HALF * D + at % KEY_HALF));
            reinterpret_cast<float4 *>(halves)[i] = make_float4(v.x, v.x, v.y, v.y);
        }
    }
    for (int i = first; i < KEY_PANEL_FLOATS / 4; i += stride) {
        int b = 0;
#pragma unroll
        for (int t = 1; t < KEY_NBLK - 1; ++t) b += 4 * i >= key_panel_off(t);
        const int nb = D - (b + 1) * KEY_BLK, r = i - key_panel_off(b) / 4, kc = r / nb, n = r % nb;   // unit within the panel: kc * nb + n
        const float *g = src + (b * KEY_BLK + 4 * kc) * D + (b + 1) * KEY_BLK + n;
        const float w0 = __ldg(g), w1 = __ldg(g + D), w2 = __ldg(g + 2 * D), w3 = __ldg(g + 3 * D);
        const float4 whi = make_float4(__uint_as_float(tf32_of(w0)), __uint_as_float(tf32_of(w1)),
                                       __uint_as_float(tf32_of(w2)), __uint_as_float(tf32_of(w3)));
        reinterpret_cast<float4 *>(hi)[i] = whi;
        reinterpret_cast<float4 *>(lo)[i] =
            make_float4(__uint_as_float(tf32_of(__fsub_rn(w0, whi.x))), __uint_as_float(tf32_of(__fsub_rn(w1, whi.y))),
                        __uint_as_float(tf32_of(__fsub_rn(w2, whi.z))), __uint_as_float(tf32_of(__fsub_rn(w3, whi.w))));
    }
}

template <int BITS, int G, bool BF16, bool M16>
int launch_inst(const KeyParams &p, int grid, cudaStream_t st)
{
    static std::atomic<unsigned long long> allowed{0};
    if (const int rc = squat_allow_smem(reinterpret_cast<const void *>(quant_keys_kernel<BITS, G, BF16, M16>), sizeof(KeyShared<key_np(G)>), allowed)) return rc;
    return squat_launch(quant_keys_kernel<BITS, G, BF16, M16>, grid, KEY_THREADS, sizeof(KeyShared<key_np(G)>), st, p);
}
template <int BITS, int G>
int launch(const KeyParams &p, int grid, int dtype, int meta16, cudaStream_t st)
{
    if (dtype == SQUAT_BF16) return meta16 ? launch_inst<BITS, G, true, true>(p, grid, st) : launch_inst<BITS, G, true, false>(p, grid, st);
    return meta16 ? launch_inst<BITS, G, false, true>(p, grid, st) : launch_inst<BITS, G, false, false>(p, grid, st);
}

}  // namespace

int squat_launch_pack_update_matrices(const float *Wt, float *Wimg, int H, int exact_channels, int block_form, int *words_dev, cudaStream_t st)
{
    constexpr int PACK_SLICES = 8;
    pack_w_kernel<<<dim3(H, PACK_SLICES), 256, 0, st>>>(Wt, Wimg, exact_channels, block_form, words_dev);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    return SQUAT_OK;
}

int squat_launch_quant_keys(const float *Wimg, const void *k, int dtype, int batch, int H, int T,
                                 long long sb, long long sh, long long st_, int bits, int G,
                                 unsigned char *codes, void *scales, void *zeros,
                                 long long osb, long long osh, unsigned *status, const int *words, int not_form, int meta16, cudaStream_t st)
{
    // Which kernel: us of keys_lane.cu against this one, bf16 keys.  128 heads x 32768: G = 32 1298 / 1350, G = 64 1583 / 1198, G = 128 1719 / 1277.  32
    // heads x 4096: 45.0 / 49.8, 54.4 / 44.7, 59.0 / 46.4.  32 heads x 128 (one tile per CTA or less): 14.2 / 16.5, 18.2 / 16.0, 19.6 / 22.4.  So groups
    // of 32, which meet no other warp in either kernel, and those of 128 while there are no more tiles than SMs, where four tiles per CTA leave most of the
    // chip idle, have one token per lane.
    const long long tiles = H * (((long long)batch * (T / G) * G + 127) / 128);
    if (G == 32 || (G == 128 && tiles <= squat_sm_count()))
        return squat_launch_quant_keys_lane(Wimg, k, dtype, batch, H, T, sb, sh, st_, bits, G, codes, scales, zeros, osb, osh, status, words, not_form, meta16, st);
    KeyParams p;
    p.Wimg = Wimg; p.k = k; p.sb = sb; p.sh = sh; p.st = st_;
    p.codes = codes; p.scales = scales; p.zeros = zeros; p.osb = osb; p.osh = osh;
    p.groups_per_bh = T / G;
    p.status = status;
    p.words = words;
    p.not_form = not_form;
    const long long groups_per_head = (long long)batch * p.groups_per_bh;
    const int np = key_np(G), places = 2 / np * squat_sm_count();
    const long long unit = 256 * np / G;
    const long long units_per_head = (groups_per_head + unit - 1) / unit;
    if (groups_per_head > 0x3fffffffLL || units_per_head * H > 0x7fffffffLL) return SQUAT_ERR_UNSUPPORTED;      // counted in 32 bits
    if (units_per_head == 0) return SQUAT_OK;
    p.groups_per_head = (int)groups_per_head;
    p.units_per_head = (int)units_per_head;
    p.total_units = (int)(units_per_head * H);
#ifdef SQUAT_CHECKED
    {
        const unsigned long long es = dtype == SQUAT_BF16 ? 2 : 4, ms = meta16 ? 2 : 4;
        p.x_k = {k, (unsigned long long)((batch - 1) * sb + (H - 1) * sh + (long long)(T - 1) * st_ + D) * es};
        p.x_codes = {codes, (unsigned long long)((batch - 1) * osb + (H - 1) * osh + T) * (D * bits / 8)};
        const unsigned long long meta_elems = (unsigned long long)(((batch - 1) * osb + (H - 1) * osh) / G + T / G) * D;
        p.x_scales = {scales, meta_elems * ms};
        p.x_zeros = {zeros, meta_elems * ms};
        p.x_img = {Wimg, (unsigned long long)H * KEY_IMG_FLOATS * 4};
    }
#endif
    const int grid = p.total_units < places ? p.total_units : places;
    if (bits == 2) {
        if (G == 64) return launch<2, 64>(p, grid, dtype, meta16, st);
        if (G == 128) return launch<2, 128>(p, grid, dtype, meta16, st);
    } else if (bits == 4) {
        if (G == 64) return launch<4, 64>(p, grid, dtype, meta16, st);
        if (G == 128) return launch<4, 128>(p, grid, dtype, meta16, st);
    }
    return SQUAT_ERR_UNSUPPORTED;
}
