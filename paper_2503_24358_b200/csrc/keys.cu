// Key quantization with error feedback (Algorithm 1, function Quant; any update matrix W): two tokens per lane, blocks of 16
// channels.
//
// A group is G consecutive tokens of one (batch, head); its channels must be visited in order, each channel's grid needs min /
// max over the group's tokens, and each token's rounding error is pushed through W onto its later channels:
//
//   m, M  = min / max                -> scale = (M-m)/L, zero = m
//   c     = rint((x_j - m)/scale),  e = c*scale - (x_j - m)       (= deq(qtz(x_j)) - x_j)
//   x_j' += e * W[j'][j]
//
// Within a block of 16 channels the pushes are CUDA-core work (packed fma.rn.f32x2 on the lane's two tokens); onto the channels
// of later blocks they are a dense product on the tcgen05 tensor cores, tf32 operands split in two.
//
// Who holds what.  A CTA is 4 sweeping warps on 2 tiles of 128 tokens, two CTAs per SM; for groups of 128 on 4 tiles, one CTA.  Row r of
// a tile = tensor-memory lane r; warp w, lane l holds row 32 w + l of every tile, as pairs of tokens, so a read of W (stored
// twice) and every packed instruction serve two tokens, and a warp's tokens are whole groups: groups of 64 and 128 join their
// extremes in the lane before the warp-wide reduction and never meet another warp.  Tensor memory, per tile: the
// corrections D[128 x 112] of channels 16 .. 127, and 16 more columns for the errors of block 0.  The errors E_hi of block b > 0
// take the columns whose corrections that block has just read, so nothing waits for a free place.  E_lo goes to shared memory as
// a K-major operand, in two buffers.
//
// Hand-over from block b to b + 1 (a fifth warp issues the products: a sweeping one that did took 2 000 cycles a hand-over over it):
//       first   D[:, next 16]  += E_lo Whi + E_hi Wlo + E_hi Whi     (commit: the next sweep waits for this)
//       then    D[:, the rest] += the same                           (done while the next sweep runs)
// so a sweep waits for products of 16 columns, whatever is left of the row.
//
// Bound: latency.  A channel's chain (two reductions, reciprocal, rounding, push onto the next channel) is 71 cycles, a hand-over about
// 1 000, and tensor memory holds 512 tokens per SM, so two warps per scheduler have to cover each other's waits; issue slots are
// 30 % busy.  What this kernel replaced swept blocks of 32 channels with one token per lane (16 warps per SM): every warp made
// every channel's grid, read W for 32 tokens at a time and, for groups of 64 and 128, met the group's other warps for every
// channel.  128 heads x 32768 tokens, before -> now: G = 128, 4 bits 1715 -> 919 us; G = 64 1578 -> 1023; G = 32 1293 -> 1059; 32 heads
// x 4096, G = 32 47.2 -> 43.8; 64 x 32 heads x 128 89.6 -> 81.1; 32 heads x 128 15.0 -> 15.1.  On the way: four tokens per lane with
// blocks of 32 channels was slower (50 KB of straight code: instruction fetch); a sweeping warp that also issued the products lost
// 2 000 cycles a hand-over; converting the keys and asking for the next ones ahead of the wait instead of behind it was worth 6 to
// 10 %.
//
// Rounding decision.  t = (x - m) / scale is formed with the hardware reciprocal, so c0 = rint(t) can be off by one when t is within
// ~1e-6 of a rounding midpoint.  Channels that earlier channels have corrected hold generic float32 values and such near-ties are as
// rare as that bound; but channels nothing has corrected yet hold raw bf16 / f32 inputs, where exact ties are structural (x exactly
// half way between min and max).  These are channel 0; the channels that W leaves uncorrected (the first g, or all of them when W = 0);
// and those of a group in which no error has been made so far, as behind constant channels.  There the remainder
// e0 = c0*scale - (x - m), which is exact next to a midpoint, is compared with +-scale/2: that settles the rounding exactly as real
// arithmetic on the stored float32 scale would, ties going to the even code (the threshold of an odd c0 is one ulp lower, so
// "remainder == scale/2" moves it), and the stored scale is the correctly rounded quotient (bit-identical to plain round-to-nearest
// quantization); elsewhere it is the product with RN(1/L), within one ulp of it.  Channel 0 is settled in the usual code; for the
// others a block is swept by the EXACT instance: where W says so, or where the usual code, at the block's first channel, finds a group
// whose errors in channel 0 (block 0) or corrections (later blocks) are all 0.  That test is free behind the next channel's
// reductions; as a test of its own ahead of the block it cost 2 % at G = 32 (40.5 -> 41.3 us for 32 heads x 4096).  A block swept twice
// costs its time: keys that are all constant take 1.2 (G = 32) to 1.45 times (G = 128) as long as others.  Exact decisions in all of
// the first 32 channels, corrected or not, would cost 5 % (G = 32, 1062 -> 1115 us for 128 heads x 32768), 1 % (G = 64) and 12 % (G = 128).
//
// M16: scale and zero-point are stored as binary16.  The float32 values are rounded once more, and the decision and the error fed
// back are taken against the rounded (stored) values: t = (x - z16) / s16, clamped to [0, L] because z16 can lie above the minimum.
#include "keys_common.cuh"

namespace {

constexpr int KEY_WARPS = 4, KEY_THREADS = 32 * (KEY_WARPS + 1);      // four sweeping warps, one that issues the products
constexpr int KEY_COLS = 128, KEY_E0_COL = 112;                          // per tile: [0, 112) corrections, [112, 128) E_hi of block 0
// Accuracy (rms error of a group's minimum against 64 bits, as a part of its range; rank 32, 2 bits, G = 32).  Corrections are gathered
// apart from the keys and added once, when the channel's turn comes, so that a large key (an outlier channel) does not round every
// push.  The tensor core's accumulator truncates on every addition: without a remedy the error regressed on the sum that n = 1 .. 7
// source blocks have added to has slopes of -1.8, -4.5, -5.2, -8.3, -7.4, -11.5, -8.4 x 2^-24 (r = 64, 4 bits, G = 128: -1.3, -6.9, -4.6, -9.9,
// -7.4, -13.6, -7.3).  2, 4, 4, 6, 6, 6, 6 x 2^-24 of the sum are given back,
// fitted on the first setting alone: slopes of 1.3 at most there and 2.2 in the second (a standard error of about 1).  Rms 1.08e-7
// -> 0.70e-7, 0.56 -> 0.52, float32 keys with G = 64 1.04 -> 0.67, channels a factor of 1000 apart 4.4 -> 2.6.  The kernel of 32-channel
// blocks before this one: 0.93, 0.77, 0.90, 3.3e-7.  tests/test_gpu_keys_accuracy.py holds these.
__device__ __forceinline__ u64 key_untruncate(int n)
{
    const float f = 1.0f + (float)min((n + 2) / 2, 3) * 0x1p-23f;
    return pack2(f, f);
}
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
    int one_tile;             // G = 32, few tokens: a unit is one tile of 128 tokens (see the launcher)
    unsigned *status;
    const int *exact_channels;    // device word: leading channels that no earlier channel corrects
#ifdef SQUAT_CHECKED
    SqExtent x_k, x_codes, x_scales, x_zeros, x_img;      // what the caller's tensors and the handle's images span
#endif
};

// Pairs of tokens per lane, by group size.  One pair: two CTAs of two tiles per SM.  Two pairs: one CTA of four tiles, so that a group
// of 128 is one warp's and its extremes never leave it (128 heads x 32768 tokens, 4 bits: 1061 us when it was built; as two warps of one pair
// each that meet for every channel 1461).  Smaller groups lose with two pairs (G = 64: 1096 -> 1239, G = 32: 1210 -> 1633): nothing is left to
// run while one warp per scheduler waits.
__host__ __device__ constexpr int key_np(int G) { return G == 128 ? 2 : 1; }

template <int NP>
struct alignas(128) KeyShared {
    u64 diag[KEY_NBLK * KEY_BLK * KEY_BLK];            // the image: diagonal blocks of W^T, every entry twice,
    float panels[2 * KEY_PANEL_FLOATS];              // hi | lo panels
    float e_lo[2][2 * NP][KEY_E_FLOATS];
    float grid[KEY_WARPS][2][2 * KEY_BLK * 2 * NP];   // scales | zero-points of two blocks' channels, [channel][group of the warp]
    u64 mbar_e, mbar_d, mbar_diag, mbar_pan;        // errors of a block in place (4 warps), products done, parts of the image staged
    unsigned tmem, timeout, exact_channels;
};
static_assert(sizeof(KeyShared<1>) <= 113 * 1024, "two CTAs per SM");
static_assert(sizeof(KeyShared<2>) > 114 * 1024, "one CTA per SM: it takes all of tensor memory");

__device__ __forceinline__ void key_tmem_st1(unsigned taddr, float v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(__float_as_uint(v)));
}
// the values of N groups as one 8- or 16-byte store (N = 1: 4)
template <int N>
__device__ __forceinline__ void key_store_groups(float *dst, const float (&v)[N])
{
    if constexpr (N == 1) *dst = v[0];
    else if constexpr (N == 2) *reinterpret_cast<float2 *>(dst) = make_float2(v[0], v[1]);
    else *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void key_tmem_ld16(unsigned taddr, unsigned (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}

// which of the warp's groups have only zeros in v (warp-uniform)
template <int NP, int NGL>
__device__ __forceinline__ void key_raw_groups(const u64 (&v)[NP], bool (&raw)[NGL])
{
    constexpr int NT = 2 * NP, TPG = NT / NGL;
    bool nz[NGL] = {};
#pragma unroll
    for (int t = 0; t < NT; ++t) nz[t / TPG] |= !(((t & 1) ? hi_of(v[t / 2]) : lo_of(v[t / 2])) == 0.0f);
#pragma unroll
    for (int g = 0; g < NGL; ++g) raw[g] = !__any_sync(0xffffffffu, nz[g]);
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

// The 16 channels of one block for the lane's 2 NP tokens (pair i of x[channel]: tokens 2 i and 2 i + 1), which belong to NGL groups.
// EXACT: decisions are exact in the groups of raw[], and in channel 0 (the first of block 0: `first`).  The usual code decides channel 0 alone
// exactly; where it finds a group without errors or corrections so far it says so in raw[] and returns true, having changed nothing
// that the EXACT instance, which then sweeps the block from its start, does not write again.
// Written in the order in which it should run: a channel's chain (reductions 24 cycles, reciprocal 24, six dependent
// operations of 4 to 6: 71 in all) goes on to the next channel's reductions before what does not hurry: the other pushes, the
// codes and the errors' stores fill the waits.  The next row of W is read before this channel's stores, which may be to the same
// memory for all the compiler knows.  The errors of the last block are stored like the others (a test per store would cut the
// code into pieces) and used by nobody.
template <int BITS, int NP, int NGL, bool EXACT, bool M16>
__device__ __forceinline__ bool sweep_pairs(const u64 (&key)[KEY_BLK][NP], u64 (&cor)[KEY_BLK][NP], const u64 *__restrict__ diag, unsigned e_hi, float *__restrict__ e_lo,
                                            int lane, bool first, bool (&raw)[NGL], float *__restrict__ gscale, float *__restrict__ gzero, unsigned (&cw)[2 * NP][BITS / 2])
{
    constexpr float L = float((1 << BITS) - 1);
    constexpr int PER_WORD = 32 / BITS, NT = 2 * NP, TPG = NT / NGL;      // tokens of the lane per group
    // what the constant upper bits of the rounded floats add up to in a packed word
    constexpr unsigned K = [] { unsigned k = 0; for (int i = 0; i < PER_WORD; ++i) k += kMagicBits << (BITS * i); return k; }();
    const u64 magic2 = pack2(kMagic, kMagic), negl2 = pack2(-L, -L);
    float el[NT][4];                                    // [token][channel % 4]
    float m[NGL], mx[NGL];
    u64 x[NP];                                          // the channel's corrected values
    auto extremes = [&]() {
        float v[NT];
#pragma unroll
        for (int i = 0; i < NP; ++i) unpack2(x[i], v[2 * i], v[2 * i + 1]);
#pragma unroll
        for (int g = 0; g < NGL; ++g) {
            float lo = v[TPG * g], hi = lo;
            if (TPG == 2) { lo = min_nan(lo, v[TPG * g + 1]); hi = max_nan(hi, v[TPG * g + 1]); }
            if (TPG == 4) {
                lo = min_nan(min3_nan(v[0], v[1], v[NT > 2 ? 2 : 0]), v[NT > 2 ? 3 : 0]);
                hi = max_nan(max3_nan(v[0], v[1], v[NT > 2 ? 2 : 0]), v[NT > 2 ? 3 : 0]);
            }
            m[g] = warp_min(lo);
            mx[g] = warp_max(hi);
        }
    };
    u64 w[KEY_BLK];                                      // row jj of the diagonal block, channels jj + 1 .. 15
    auto read_row = [&](int jj) {
#pragma unroll
        for (int q = (jj + 1) / 2; q < KEY_BLK / 2; ++q) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(diag + jj * KEY_BLK + 2 * q);
            w[2 * q] = t.x;
            w[2 * q + 1] = t.y;
        }
    };
    read_row(0);
#pragma unroll
    for (int i = 0; i < NP; ++i) x[i] = fadd2(key[0][i], cor[0][i]);
    extremes();
#pragma unroll
    for (int jj = 0; jj < KEY_BLK; ++jj) {
        float scale[NGL], inv[NGL], z[NGL];
#pragma unroll
        for (int g = 0; g < NGL; ++g) {
            const float rng = __fsub_rn(mx[g], m[g]);
            z[g] = m[g];
            scale[g] = (EXACT && raw[g]) || (jj == 0 && first) ? div_by_levels<BITS>(rng) : __fmul_rn(rng, 1.0f / L);
            if (M16) {
                scale[g] = __half2float(__float2half_rn(scale[g]));
                z[g] = __half2float(__float2half_rn(m[g]));
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv[g]) : "f"(scale[g]));
                inv[g] = scale[g] > 0.0f ? -inv[g] : 0.0f;                                      // scale 0 (no range, or underflow): codes 0
            } else {
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv[g]) : "f"(fmaxf(rng, 1e-30f)));     // constant group: x - m = 0 -> code 0
            }
        }
        u64 pre[NP];                                    // the next channel, but for this channel's push
        if (jj + 1 < KEY_BLK) {
#pragma unroll
            for (int i = 0; i < NP; ++i) pre[i] = fadd2(key[jj + 1][i], cor[jj + 1][i]);
        }
        u64 e[NP];
        float y[NT];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int ga = 2 * i / TPG, gb = (2 * i + 1) / TPG;
            const u64 n = fsub2(pack2(z[ga], z[gb]), x[i]);                                 // -(x - m)
            u64 y2 = ffma2(M16 ? n : fmul2(n, negl2), pack2(inv[ga], inv[gb]), magic2);
            float &y0 = y[2 * i], &y1 = y[2 * i + 1];
            unpack2(y2, y0, y1);
            if (M16 && !EXACT && jj > 0) {
                y0 = fminf(fmaxf(y0, kMagic), kMagic + L);
                y1 = fminf(fmaxf(y1, kMagic), kMagic + L);
                y2 = pack2(y0, y1);
            }
            e[i] = ffma2(fsub2(y2, magic2), pack2(scale[ga], scale[gb]), n);
            if (EXACT || (jj == 0 && (first || M16))) {
                float e0, e1, n0, n1;
                unpack2(e[i], e0, e1);
                unpack2(n, n0, n1);
                auto decide = [&](float nd, int g, float &yy, float &ee) {
                    if (EXACT || first) {
                        const bool settle = !EXACT || raw[g] || (jj == 0 && first);      // (else nothing lies beyond, and 0 x 0 is added)
                        const float half = settle ? 0.5f * scale[g] : __int_as_float(0x7f800000), step = settle ? scale[g] : 0.0f;
                        const float thr = __uint_as_float(__float_as_uint(half) - (__float_as_uint(yy) & 1u));
                        const float adj = ee > thr ? -1.0f : (ee < -thr ? 1.0f : 0.0f);
                        yy = __fadd_rn(yy, adj);
                        ee = __fmaf_rn(adj, step, ee);
                    }
                    if (M16) {
                        const float cc = fminf(fmaxf(yy, kMagic), kMagic + L);
                        ee = cc == yy ? ee : __fmaf_rn(__fsub_rn(cc, kMagic), scale[g], nd);
                        yy = cc;
                    }
                };
                decide(n0, ga, y0, e0);
                decide(n1, gb, y1, e1);
                e[i] = pack2(e0, e1);
            }
        }
        // the next channel's value and extremes first
        if (jj + 1 < KEY_BLK) {
#pragma unroll
            for (int i = 0; i < NP; ++i) x[i] = ffma2(e[i], w[jj + 1], pre[i]);
            extremes();
        }
        if (!EXACT && jj == 0) {                        // (while those reductions run; no push has been made yet)
            bool any = false;
            u64 v[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) v[i] = first ? e[i] : cor[0][i];
            key_raw_groups<NP, NGL>(v, raw);
#pragma unroll
            for (int g = 0; g < NGL; ++g) any |= raw[g];
            if (any) return true;
        }
#pragma unroll
        for (int c = jj + 2; c < KEY_BLK; ++c)
#pragma unroll
            for (int i = 0; i < NP; ++i) cor[c][i] = ffma2(e[i], w[c], cor[c][i]);
        if (jj + 1 < KEY_BLK) read_row(jj + 1);
        if (lane == 0) {
            key_store_groups<NGL>(gscale + jj * NGL, scale);
            key_store_groups<NGL>(gzero + jj * NGL, z);
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
    return false;
}

template <int BITS, int G, bool BF16, bool M16>
__global__ void __launch_bounds__(KEY_THREADS, 2 / key_np(G)) quant_keys_kernel(const KeyParams p)
{
    constexpr int NP = key_np(G), NT = 2 * NP, NGL = 32 * NT / G, UNIT_GROUPS = KEY_WARPS * NGL, ES = BF16 ? 2 : 4;
    static_assert(NGL >= 1, "a group is one warp's");
    constexpr unsigned TMEM_COLS = NT * KEY_COLS;
    extern __shared__ __align__(128) unsigned char smem_bytes[];
    KeyShared<NP> &sm = *reinterpret_cast<KeyShared<NP> *>(smem_bytes);
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);      // (uniform: tensor-memory addresses go by it)

    const int u_lo = (int)((long long)p.total_units * blockIdx.x / gridDim.x);
    const int u_hi = (int)((long long)p.total_units * (blockIdx.x + 1) / gridDim.x);
    grid_wait();
    volatile unsigned *timeout = &sm.timeout;
    const unsigned mbar_e = smem_u32(&sm.mbar_e), mbar_d = smem_u32(&sm.mbar_d), mbar_diag = smem_u32(&sm.mbar_diag), mbar_pan = smem_u32(&sm.mbar_pan);

    // where the lane's tokens (one in each tile) and the warp's groups come from and go to
    struct Place {
        const char *row[NGL];     // the lane's first token of a group
        unsigned char *codes[NGL];
        long long meta[NGL];
        bool active[NGL];         // the group exists (a head's last unit may be ragged: past its end the last group is redone and not stored)
    };
    const long long row_step = 32 * p.st * ES;           // to the lane's next token of a group
    auto locate = [&](int unit, Place &t) {
        const int h = unit / p.units_per_head;
        const bool one = G == 32 && p.one_tile;
        const int g0 = one ? (unit - h * p.units_per_head) * KEY_WARPS + warp : (unit - h * p.units_per_head) * UNIT_GROUPS + NGL * warp;
#pragma unroll
        for (int g = 0; g < NGL; ++g) {
            t.active[g] = g0 + g < p.groups_per_head && (g == 0 || !one);
            const int in_head = t.active[g] ? g0 + g : p.groups_per_head - 1;
            const int b = in_head / p.groups_per_bh, grp = in_head - b * p.groups_per_bh;
            const int tok = grp * G + lane;
            const long long out_tok0 = (long long)b * p.osb + (long long)h * p.osh;
            t.row[g] = static_cast<const char *>(p.k) + ((long long)b * p.sb + (long long)h * p.sh + (long long)tok * p.st) * ES;
            t.codes[g] = p.codes + (out_tok0 + tok) * (D * BITS / 8);
            t.meta[g] = (out_tok0 / G + grp) * D + lane;
        }
    };
    PairRows<BF16, NP> raw;
    auto load_rows = [&](const Place &t, int blk) {
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            const char *src = t.row[i / (NT / NGL)] + i % (NT / NGL) * row_step + blk * (KEY_BLK * ES);
            if (SQ_CHK_G(p.status, src, KEY_BLK * ES, p.x_k)) {
#pragma unroll
                for (int c = 0; c < (BF16 ? 2 : 4); ++c) raw.v[i][c] = reinterpret_cast<const uint4 *>(src)[c];
            }
        }
    };
    Place cur;
    if (u_lo < u_hi && warp < KEY_WARPS) {               // the first rows are on their way while the CTA sets itself up
        locate(u_lo, cur);
        load_rows(cur, 0);
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
        copy(smem_u32(sm.diag), src, KEY_DIAG_FLOATS * 4, mbar_diag);                  // the sweeps need only these
        copy(smem_u32(sm.panels), src + KEY_DIAG_FLOATS, 2 * KEY_PANEL_FLOATS * 4, mbar_pan);
    };
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_e), "r"(KEY_WARPS) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_d), "r"(1) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_diag), "r"(1) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_pan), "r"(1) : "memory");
        sm.timeout = 0;
        sm.exact_channels = (unsigned)*p.exact_channels;
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
                bounded_wait(mbar_e, phase);
                phase ^= 1;
                tc_fence_after();
                const int nb = D - (blk + 1) * KEY_BLK;             // channels still to come
                const unsigned b_lbo = 16u * nb, bhi = pan + 4 * key_panel_off(blk);
                const u64 step = (2 * b_lbo) >> 4;                 // 8 channels on
                // onto n channels from the ch-th behind the block on, all tiles
                auto products = [&](int ch, int n) {
                    if (!SQ_CHK_C(p.status, key_panel_off(blk) + nb * KEY_BLK <= KEY_PANEL_FLOATS && ch + n <= nb)) return;
                    const unsigned idesc = tc_idesc(n);
                    const u64 hi = umma_desc(bhi + 16u * ch, b_lbo, KEY_SBO), lo = hi + KEY_PANEL_FLOATS * 4 / 16;
#pragma unroll
                    for (int i = 0; i < NT; ++i) {
                        if (G == 32 && i > 0 && p.one_tile) break;
                        const unsigned d = tmem + i * KEY_COLS + blk * KEY_BLK + ch, a_hi = tmem + i * KEY_COLS + (blk == 0 ? KEY_E0_COL : (blk - 1) * KEY_BLK);
                        const u64 a_lo = a_lo0 + ((blk & 1) * NT + i) * (KEY_E_FLOATS * 4 / 16);
                        umma_tf32_ss(d, a_lo, hi, idesc, blk != 0);                                            // E_lo (shared memory) x Whi
                        umma_tf32_ss(d, a_lo + 2 * KEY_A_LBO / 16, hi + step, idesc, 1u);
                        umma_tf32_ts(d, a_hi, lo, idesc, 1u);                                                   // E_hi (tensor memory) x Wlo
                        umma_tf32_ts(d, a_hi + 8, lo + step, idesc, 1u);
                        umma_tf32_ts(d, a_hi, hi, idesc, 1u);                                                   // E_hi x Whi
                        umma_tf32_ts(d, a_hi + 8, hi + step, idesc, 1u);
                    }
                };
                if (elect_one()) {
                    products(0, KEY_BLK);
                    tc_commit(mbar_d);
                    if (nb > KEY_BLK) products(KEY_BLK, nb - KEY_BLK);
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
        unsigned cw[NT][BITS / 2], cw_even[NT][BITS / 2];
#pragma unroll 1
        for (int blk = 0; blk < KEY_NBLK; ++blk) {
            const bool more = blk + 1 < KEY_NBLK;
            u64 key[KEY_BLK][NP], cor[KEY_BLK][NP];      // keys, and what earlier channels have pushed onto them
#pragma unroll
            for (int c = 0; c < KEY_BLK; ++c)
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    key[c][i] = pack2(raw.get(2 * i, c), raw.get(2 * i + 1, c));
                    cor[c][i] = 0;
                }
            if (more) load_rows(cur, blk + 1);           // (before the wait: what can be done ahead of it is)
            else if (unit + 1 < u_hi) load_rows(nxt, 0);
            if (blk > 0) {
                bounded_wait(mbar_d, phase);             // the products that complete this block's corrections
                phase ^= 1;
                tc_fence_after();
                unsigned d[NT][16];
                const u64 up = key_untruncate(blk);
#pragma unroll
                for (int t = 0; t < NT; ++t) key_tmem_ld16(t_mine + t * KEY_COLS + (blk - 1) * KEY_BLK, d[t]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int c = 0; c < KEY_BLK; ++c)
#pragma unroll
                    for (int i = 0; i < NP; ++i) cor[c][i] = fmul2(pack2(__uint_as_float(d[2 * i][c]), __uint_as_float(d[2 * i + 1][c])), up);
            }

            const u64 *diag = sm.diag + blk * KEY_BLK * KEY_BLK;
            const unsigned e_hi = t_mine + (blk == 0 ? KEY_E0_COL : (blk - 1) * KEY_BLK);
            float *e_lo = &sm.e_lo[blk & 1][0][(warp * 32 + lane) * 4];
            float *gscale = &sm.grid[warp][0][(blk & 1) * KEY_BLK * NGL], *gzero = &sm.grid[warp][1][(blk & 1) * KEY_BLK * NGL];
            // (recorded only: every address of a sweep is a constant away from these)
            (void)SQ_CHK_R(p.status, e_lo, (KEY_E_FLOATS * (NT - 1) + (KEY_BLK / 4 - 1) * KEY_A_LBO / 4 + 4) * 4, sm.e_lo[blk & 1], sizeof(sm.e_lo[0]));
            (void)SQ_CHK_R(p.status, diag, KEY_BLK * KEY_BLK * 8, sm.diag, sizeof(sm.diag));
            (void)SQ_CHK_C(p.status, (e_hi & 0xffffu) >= (tmem & 0xffffu) && (e_hi & 0xffffu) + KEY_BLK <= (tmem & 0xffffu) + KEY_COLS);
            // Where W leaves channels of the block uncorrected, every group is decided exactly; else the groups that the usual code finds raw.
            bool raw[NGL], exact = exact_channels > max(1, blk * KEY_BLK);
#pragma unroll
            for (int g = 0; g < NGL; ++g) raw[g] = true;
            if (!exact) exact = sweep_pairs<BITS, NP, NGL, false, M16>(key, cor, diag, e_hi, e_lo, lane, blk == 0, raw, gscale, gzero, cw);
            if (exact) sweep_pairs<BITS, NP, NGL, true, M16>(key, cor, diag, e_hi, e_lo, lane, blk == 0, raw, gscale, gzero, cw);

            if (more) {
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");   // E_hi is in tensor memory
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // E_lo rows, for the tensor core
                tc_fence_before();
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar_e) : "memory");
            }
            if (blk & 1) {                               // 32 channels are complete
                __syncwarp();                            // (the grids lane 0 wrote)
                const int at = (blk >> 1) * 32;
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    unsigned char *cp = cur.codes[i / (NT / NGL)] + i % (NT / NGL) * (32 * D * BITS / 8) + at * BITS / 8;
                    if (cur.active[i / (NT / NGL)] && SQ_CHK_G(p.status, cp, 32 * BITS / 8, p.x_codes)) {
                        if (BITS == 2) *reinterpret_cast<uint2 *>(cp) = make_uint2(cw_even[i][0], cw[i][0]);
                        else *reinterpret_cast<uint4 *>(cp) = make_uint4(cw_even[i][0], cw_even[i][BITS / 2 - 1], cw[i][0], cw[i][BITS / 2 - 1]);
                    }
                }
#pragma unroll
                for (int g = 0; g < NGL; ++g) {
                    const float2 sz = make_float2(sm.grid[warp][0][lane * NGL + g], sm.grid[warp][1][lane * NGL + g]);
                    const long long meta = cur.meta[g] + at;
                    if (cur.active[g] && SQ_CHK_G(p.status, static_cast<char *>(p.scales) + meta * (M16 ? 2 : 4), M16 ? 2 : 4, p.x_scales) &&
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
                __syncwarp();                            // before the next sweep writes grids
            } else {
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                    for (int w = 0; w < BITS / 2; ++w) cw_even[i][w] = cw[i][w];
            }
        }
        cur = nxt;
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Writes, per head, the image that quant_keys_kernel stages in shared memory:
//   u64 [8][16][16]   diagonal 16 x 16 blocks of W^T, row-major, every entry as a pair of equal floats
//   hi panels         of source blocks b = 0 .. 6: B_b(n, k) = W[16 (b + 1) + n][16 b + k] = W^T[16 b + k][16 (b + 1) + n],
//                     n < 112 - 16 b, k < 16, rounded to tf32, K-major in 8 x 16-byte core matrices:
//                     float index (k / 4) * 4 N + 4 n + k % 4 with N = 112 - 16 b
//   lo panels         tf32(W - hi), same layout
// Grid (heads, slices): the kernel is a chain of two dependent global accesses, so more CTAs, not more work per thread, shorten
// it; each thread takes (panel, 4-k chunk, channel n): four coalesced row reads, one 16-byte store.
__global__ void __launch_bounds__(256) pack_w_kernel(const float *__restrict__ Wt, float *__restrict__ Wimg, int exact_channels,
                                                        int *__restrict__ exact_channels_dev)
{
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *exact_channels_dev = exact_channels;    // travels with the matrices it describes
    const float *src = Wt + (long long)blockIdx.x * D * D;
    float *img = Wimg + (long long)blockIdx.x * KEY_IMG_FLOATS;
    const int first = blockIdx.y * blockDim.x + threadIdx.x, stride = gridDim.y * blockDim.x;
    for (int i = first; i < KEY_NBLK * KEY_BLK * KEY_BLK / 2; i += stride) {
        const int b = i / (KEY_BLK * KEY_BLK / 2), r = i % (KEY_BLK * KEY_BLK / 2), jj = r / (KEY_BLK / 2), c2 = r % (KEY_BLK / 2);
        const float2 v = __ldg(reinterpret_cast<const float2 *>(src + (b * KEY_BLK + jj) * D + b * KEY_BLK + 2 * c2));
        reinterpret_cast<float4 *>(img)[i] = make_float4(v.x, v.x, v.y, v.y);
    }
    float *hi = img + KEY_DIAG_FLOATS, *lo = hi + KEY_PANEL_FLOATS;
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

int squat_launch_pack_update_matrices(const float *Wt, float *Wimg, int H, int exact_channels, int *exact_channels_dev, cudaStream_t st)
{
    constexpr int PACK_SLICES = 8;
    pack_w_kernel<<<dim3(H, PACK_SLICES), 256, 0, st>>>(Wt, Wimg, exact_channels, exact_channels_dev);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    return SQUAT_OK;
}

int squat_launch_quant_keys(const float *Wimg, const void *k, int dtype, int batch, int H, int T,
                                 long long sb, long long sh, long long st_, int bits, int G,
                                 unsigned char *codes, void *scales, void *zeros,
                                 long long osb, long long osh, unsigned *status, const int *exact_channels, int meta16, cudaStream_t st)
{
    KeyParams p;
    p.Wimg = Wimg; p.k = k; p.sb = sb; p.sh = sh; p.st = st_;
    p.codes = codes; p.scales = scales; p.zeros = zeros; p.osb = osb; p.osh = osh;
    p.groups_per_bh = T / G;
    p.status = status;
    p.exact_channels = exact_channels;
    const long long groups_per_head = (long long)batch * p.groups_per_bh;
    const int np = key_np(G), places = 2 / np * squat_sm_count();
    // Where there is at most one tile of 128 tokens per SM (a window of a few sequences), a CTA takes one tile: a hand-over then
    // waits for half the products (4 x 32 heads x 128 tokens, G = 32: 16.3 -> 16.0 us; with 256 tiles two CTAs per SM of one tile
    // each take 22.4 us, one CTA of two 16.5).
    p.one_tile = G == 32 && H * ((groups_per_head + 3) / 4) <= squat_sm_count();
    const long long unit = p.one_tile ? 4 : 256 * np / G;
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
        if (G == 32) return launch<2, 32>(p, grid, dtype, meta16, st);
        if (G == 64) return launch<2, 64>(p, grid, dtype, meta16, st);
        if (G == 128) return launch<2, 128>(p, grid, dtype, meta16, st);
    } else if (bits == 4) {
        if (G == 32) return launch<4, 32>(p, grid, dtype, meta16, st);
        if (G == 64) return launch<4, 64>(p, grid, dtype, meta16, st);
        if (G == 128) return launch<4, 128>(p, grid, dtype, meta16, st);
    }
    return SQUAT_ERR_UNSUPPORTED;
}
