// Key quantization with block updates (Algorithm 1, function Quant, with g = 32 or 64 channels per iteration: Appendix A's
// block-wise quantization, the form of the paper's experiments; Eq. (update_block)).
//
// Within a block of g channels nothing depends on anything else: the diagonal blocks of W are zero, so the chain of 128
// dependent channels that the kernel of keys_lane.cu walks (lane = token, a warp-wide reduction and a push per channel) does not
// exist here.  What is left per block is one pass over memory and one dense product, and the mapping follows that:
//
//   a thread owns a quad of 4 channels x 8 tokens of a group; a warp 8 quads x 4 token phases = 32 channels x 32 tokens.
//   Minima and maxima are over the thread's own registers and two shuffle steps; the grid (scale, zero-point, reciprocal) is
//   formed once per channel and thread instead of once per element; arithmetic runs on packed pairs.  Groups of 64 and 128
//   tokens join 2 or 4 warps' extremes in shared memory once per block.
//
//   update of the later channels: D[128 tokens x later channels] += E [128 x g] * W panel on the tcgen05 tensor cores, tf32
//   operands split in two (E_lo Whi + E_hi Wlo + E_hi Whi, small terms first, as in keys.cu).  A thread's quad of errors is
//   exactly one 16-byte row of a K-major core matrix, so E goes to shared memory as it falls out of the quantizer.  D comes
//   back with lane = token; a warp reads precisely the 32 tokens x 32 channels it will quantize next, so the change to
//   quads is an exchange inside the warp, through its own (by then consumed) rows of the E_lo operand.
//
// g = 64: a tile of 128 tokens per CTA, 8 warps = 4 token quarters x 2 channel halves, two steps, one product of K = 64.
// g = 32: two tiles per CTA, 4 warps each, four steps and three products of K = 32.
// Two CTAs per SM, so one computes while the other's products run.  CTAs are persistent over a contiguous range of units
// (g = 64: a tile; g = 32: two tiles) in head-major order and stage a head's panels when the head changes.
//
// Bound: bytes first (304 per key vector with bf16 keys, 2 bits, G = 32, 16-bit scales), then the errors' trip through shared
// memory (8 B written, 12 B read by the tensor core per element).  Measured against the kernel of keys_lane.cu, which walks the chain
// of the element-wise form whatever g is: 16 x 8 heads x 8160 tokens, 2 bits, G = 32, 16-bit scales 365 -> 130 us at g = 64 and
// 357 -> 159 at g = 32; 4 bits, G = 128, g = 64 462 -> 142; 32 heads x 4096 48 -> 23; one window of 32 heads x 128 15.2 -> 6.6.
// What is left (ablations, g = 64): the wait for the products 27 us, the errors' stores 17, exact decisions 5; asking L2 for the
// next unit's keys ahead changed nothing, so it is the latency of a unit's steps at 16 warps per SM, not the loads.
// No size was found where the other kernel is faster, so every handle built with such a g comes here.
#include "keys_common.cuh"

namespace {

constexpr int BLK = 32;                               // channels per warp and step
constexpr int KB_THREADS = 256;
constexpr int KB_ROWS = 8;                            // tokens per thread and block
constexpr unsigned KB_LBO = 128 * 16 + 16, KB_SBO = 128;   // bytes between 4-channel chunks of an E operand (16 more than the 128
                                                      // rows take: a warp's 8 quads then fall on different banks), between 8 rows
constexpr int KB_CHUNK_FLOATS = KB_LBO / 4;

struct KeyBlockParams {
    const float *Wimg;        // [H, KEY_IMG_FLOATS] staged images of the update matrices (pack_w_kernel)
    const void *k;
    long long sb, sh, st;     // element strides of k
    unsigned char *codes;
    void *scales, *zeros;     // float32, or binary16 in the M16 instances
    long long osb, osh;       // output strides in tokens
    int groups_per_bh;        // T / G
    int groups_per_head;      // B * T / G
    int units_per_head;
    int total_units;
    unsigned *status;
    const int *form;          // not null: device word, the image's block size; one of another is not this kernel's (see quantize_keys_impl)
#ifdef SQUAT_CHECKED
    SqExtent x_k, x_codes, x_scales, x_zeros, x_img;      // what the caller's tensors and the handle's images span
#endif
};

// where the panel of step s starts (g = 32: 96, 64, 32 later channels)
__host__ __device__ constexpr int kb_panel_off(int s) { return s == 0 ? 0 : s == 1 ? 32 * 96 : 32 * (96 + 64); }

template <int GB>
struct KbLayout {
    static constexpr int SLOTS = 64 / GB;                         // tiles of 128 tokens per CTA
    static constexpr int STEPS = D / GB;
    static constexpr int CHUNKS = GB / 4;                         // 4-channel chunks of an operand
    static constexpr int E_FLOATS = CHUNKS * KB_CHUNK_FLOATS;     // one tile's E_hi (or E_lo)
    static constexpr int W_FLOATS = GB == 64 ? 64 * 64 : 32 * (96 + 64 + 32);    // hi (or lo) panels, K-major, GB source channels x the later ones
    static constexpr int SLOT_COLS = GB == 64 ? 64 : 128;
    static constexpr int TMEM_COLS = SLOTS * SLOT_COLS;
    static constexpr int WARPS_PER_TILE = 8 / SLOTS;
    static constexpr size_t SMEM = sizeof(float) * (2 * SLOTS * E_FLOATS + 2 * W_FLOATS) + sizeof(u64) * (SLOTS + 1) + 4 * (2 + SLOTS) + 8;
};

// 4 channels of the thread's 8 tokens as they are in memory
template <bool BF16>
struct QuadRows {
    uint4 v[BF16 ? KB_ROWS / 2 : KB_ROWS];      // bf16: two tokens per register quad
    __device__ __forceinline__ void load(int i, const void *p)
    {
        if (BF16) {
            const uint2 t = *reinterpret_cast<const uint2 *>(p);
            if (i & 1) { v[i >> 1].z = t.x; v[i >> 1].w = t.y; }
            else { v[i >> 1].x = t.x; v[i >> 1].y = t.y; }
        } else {
            v[BF16 ? 0 : i] = *reinterpret_cast<const uint4 *>(p);
        }
    }
    __device__ __forceinline__ uint2 words(int i) const      // bf16: channel pairs (0, 1) and (2, 3)
    {
        const uint4 &t = v[BF16 ? i >> 1 : 0];
        return (i & 1) ? make_uint2(t.z, t.w) : make_uint2(t.x, t.y);
    }
    __device__ __forceinline__ void get(int i, u64 &x01, u64 &x23) const
    {
        if (BF16) {
            const uint2 w = words(i);
            x01 = pack2(bf16lo_to_f32(w.x), bf16hi_to_f32(w.x));
            x23 = pack2(bf16lo_to_f32(w.y), bf16hi_to_f32(w.y));
        } else {
            const uint4 &t = v[BF16 ? 0 : i];
            x01 = pack2(__uint_as_float(t.x), __uint_as_float(t.y));
            x23 = pack2(__uint_as_float(t.z), __uint_as_float(t.w));
        }
    }
};

// Per-lane selectors of the transpositions below, fixed for the thread
struct CodeLanes {
    bool up4;                       // lane holds the upper four tokens after the first exchange
    unsigned keep2, send2, keep1, send1, out;
};
template <int BITS>
__device__ __forceinline__ CodeLanes code_lanes(int q)
{
    CodeLanes c;
    c.up4 = q & 4;
    c.keep2 = (q & 2) ? 0x7632u : 0x5410u;
    c.send2 = (q & 2) ? 0x5410u : 0x7632u;
    if (BITS == 2) {
        c.keep1 = (q & 1) ? 0x7531u : 0x6420u;
        c.send1 = (q & 1) ? 0x6420u : 0x7531u;
        c.out = 0;
#pragma unroll
        for (int l = 0; l < 4; ++l) {                  // where lane l's byte of the low word is (see below)
            const int x = (q & 3) ^ l;
            c.out |= (unsigned)(x == 0 ? 0 : x == 2 ? 2 : x == 1 ? 4 : 6) << (4 * l);
        }
    } else {
        c.keep1 = (q & 1) ? 0x7632u : 0x5410u;
        c.send1 = (q & 1) ? 0x5410u : 0x7632u;
        c.out = 0;
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const int x = (q & 3) ^ l;
            const unsigned half = x == 0 ? 0 : x == 2 ? 1 : x == 1 ? 2 : 3;
            c.out |= ((2 * half) | ((2 * half + 1) << 4)) << (8 * l);
        }
    }
    return c;
}

// The 8 lanes of a token phase hold, for 8 tokens i, the codes of 4 channels each (8 or 16 bits); returns the 32 channels'
// codes of token i = q to lane q: an 8 x 8 transposition in three exchanges.  `w` holds token i's codes at byte (2-bit) or
// half word (4-bit) i.
__device__ __forceinline__ uint2 transpose_codes2(const unsigned (&w)[2], const CodeLanes &c)
{
    const unsigned r4 = __shfl_xor_sync(0xffffffffu, c.up4 ? w[0] : w[1], 4), k4 = c.up4 ? w[1] : w[0];
    const unsigned lo = c.up4 ? r4 : k4, hi = c.up4 ? k4 : r4;               // from lanes q & 3 and (q & 3) + 4, four tokens each
    const unsigned r2 = __shfl_xor_sync(0xffffffffu, __byte_perm(lo, hi, c.send2), 2), k2 = __byte_perm(lo, hi, c.keep2);
    // k2: two tokens of (own lo, own hi), r2: of lane ^ 2
    const unsigned r1 = __shfl_xor_sync(0xffffffffu, __byte_perm(k2, r2, c.send1), 1), k1 = __byte_perm(k2, r2, c.keep1);
    // k1: token q of lanes (q, q + 4, q ^ 2, (q ^ 2) + 4) (mod the upper half), r1: the same of lane ^ 1
    return make_uint2(__byte_perm(k1, r1, c.out), __byte_perm(k1, r1, c.out + 0x1111u));
}
__device__ __forceinline__ uint4 transpose_codes4(const unsigned (&w)[4], const CodeLanes &c)
{
    const unsigned ra = __shfl_xor_sync(0xffffffffu, c.up4 ? w[0] : w[2], 4), rb = __shfl_xor_sync(0xffffffffu, c.up4 ? w[1] : w[3], 4);
    const unsigned ka = c.up4 ? w[2] : w[0], kb = c.up4 ? w[3] : w[1];
    const unsigned lo0 = c.up4 ? ra : ka, lo1 = c.up4 ? rb : kb, hi0 = c.up4 ? ka : ra, hi1 = c.up4 ? kb : rb;
    const bool up2 = c.keep2 == 0x7632u;
    const unsigned rl = __shfl_xor_sync(0xffffffffu, up2 ? lo0 : lo1, 2), rh = __shfl_xor_sync(0xffffffffu, up2 ? hi0 : hi1, 2);
    const unsigned kl = up2 ? lo1 : lo0, kh = up2 ? hi1 : hi0;
    const unsigned r0 = __shfl_xor_sync(0xffffffffu, __byte_perm(kl, rl, c.send1), 1), k0 = __byte_perm(kl, rl, c.keep1);
    const unsigned r1 = __shfl_xor_sync(0xffffffffu, __byte_perm(kh, rh, c.send1), 1), k1 = __byte_perm(kh, rh, c.keep1);
    return make_uint4(__byte_perm(k0, r0, c.out & 0xffffu), __byte_perm(k0, r0, c.out >> 16),
                      __byte_perm(k1, r1, c.out & 0xffffu), __byte_perm(k1, r1, c.out >> 16));
}

// The exact decision of one element of an uncorrected block whose remainder e is close to half a step (see the
// rounding decision in keys.cu): y, the rounded float, moves by one where the remainder says so, and the error with it.
template <int BITS, bool CLAMP>
__device__ __forceinline__ void decide_exactly(float nd, float scale, float neg_inv, float &y, float &e)
{
    constexpr float L = float((1 << BITS) - 1);
    if (CLAMP) {                                            // from the unclamped value
        y = __fmaf_rn(nd, neg_inv, kMagic);
        e = __fmaf_rn(__fsub_rn(y, kMagic), scale, nd);
    }
    const float thr = __uint_as_float(__float_as_uint(0.5f * scale) - (__float_as_uint(y) & 1u));
    const float adj = e > thr ? -1.0f : (e < -thr ? 1.0f : 0.0f);
    y = __fadd_rn(y, adj);
    e = __fmaf_rn(adj, scale, e);
    if (CLAMP) {
        const float c = fminf(fmaxf(y, kMagic), kMagic + L);
        e = c == y ? e : __fmaf_rn(__fsub_rn(c, kMagic), scale, nd);
        y = c;
    }
}

// Grids of a thread's 4 channels, as pairs
struct Grid4 {
    u64 m[2], scale[2], neg_inv[2];
};

// Codes of the thread's 4 channels x 8 tokens, and (STORE_E) the errors to the tile's E operands, a 16-byte row per token.
// EXACT: uncorrected inputs, where exact ties are structural: an element whose remainder is within 1e-4 of half a step is
// decided through that remainder as real arithmetic on the stored scale would; a row with such an element is looked at again.
// CLAMP: grids whose 16-bit zero-point or scale leaves an extreme half a step or more outside [0, L].
template <int BITS, bool CLAMP, bool EXACT, bool STORE_E>
__device__ __forceinline__ void quantize_quads(const u64 (&x)[KB_ROWS][2], const Grid4 &g, float *e_hi, float *e_lo, unsigned (&cw)[BITS])
{
    constexpr float L = float((1 << BITS) - 1);
    const u64 magic2 = pack2(kMagic, kMagic);
    float thr[4];
    if (EXACT) {
#pragma unroll
        for (int j = 0; j < 2; ++j) unpack2(fmul2(g.scale[j], pack2(0.4999f, 0.4999f)), thr[2 * j], thr[2 * j + 1]);
    }
#pragma unroll
    for (int i = 0; i < KB_ROWS; ++i) {
        u64 n[2], y[2], e[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            n[j] = fsub2(g.m[j], x[i][j]);                  // -(x - m)
            y[j] = ffma2(n[j], g.neg_inv[j], magic2);
            if (CLAMP) y[j] = pack2(fminf(fmaxf(lo_of(y[j]), kMagic), kMagic + L), fminf(fmaxf(hi_of(y[j]), kMagic), kMagic + L));
            if (EXACT || STORE_E) e[j] = ffma2(fsub2(y[j], magic2), g.scale[j], n[j]);
        }
        if (EXACT && ((fabsf(lo_of(e[0])) > thr[0]) | (fabsf(hi_of(e[0])) > thr[1]) | (fabsf(lo_of(e[1])) > thr[2]) | (fabsf(hi_of(e[1])) > thr[3]))) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float y0, y1, e0, e1;
                unpack2(y[j], y0, y1);
                unpack2(e[j], e0, e1);
                decide_exactly<BITS, CLAMP>(lo_of(n[j]), lo_of(g.scale[j]), lo_of(g.neg_inv[j]), y0, e0);
                decide_exactly<BITS, CLAMP>(hi_of(n[j]), hi_of(g.scale[j]), hi_of(g.neg_inv[j]), y1, e1);
                y[j] = pack2(y0, y1);
                e[j] = pack2(e0, e1);
            }
        }
        if (STORE_E) {
            // tf32 split by truncation: the tensor core reads the top 19 bits of a word, so e itself serves as E_hi
            ulonglong2 hi, lo;
            hi.x = e[0];
            hi.y = e[1];
            lo.x = fsub2(e[0], e[0] & 0xffffe000ffffe000ull);
            lo.y = fsub2(e[1], e[1] & 0xffffe000ffffe000ull);
            *reinterpret_cast<ulonglong2 *>(e_hi + i * 16) = hi;
            *reinterpret_cast<ulonglong2 *>(e_lo + i * 16) = lo;
        }
        // the low bits of a rounded float are its code; what is shifted in from above stays out of the 4 * BITS bits used
        const unsigned a = ((unsigned)(y[0] >> 32) << BITS) + (unsigned)y[0];
        const unsigned b = ((unsigned)(y[1] >> 32) << BITS) + (unsigned)y[1];
        const unsigned c4 = (b << (2 * BITS)) + a;
        if (BITS == 2) {                                    // byte i
            unsigned &d = cw[i >> 2];
            d = (i & 3) == 0 ? c4 : __byte_perm(d, c4, (i & 3) == 1 ? 0x3240u : (i & 3) == 2 ? 0x3410u : 0x4210u);
        } else {                                            // half word i
            unsigned &d = cw[i >> 1];
            d = (i & 1) == 0 ? c4 : __byte_perm(d, c4, 0x5410u);
        }
    }
}

// The grid of one channel: m becomes the stored zero-point; returns whether a code could leave [0, L].
template <int BITS, bool M16, bool EXACT>
__device__ __forceinline__ bool make_grid(float &m, float mx, float &scale, float &inv)
{
    constexpr float L = float((1 << BITS) - 1);
    const float rng = __fsub_rn(mx, m);
    scale = EXACT ? div_by_levels<BITS>(rng) : __fmul_rn(rng, 1.0f / L);                // as in keys.cu
    float rcp;
    if (!M16) {
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rcp) : "f"(fmaxf(rng, 1e-30f)));        // constant group: x - m = 0 -> code 0
        inv = __fmul_rn(rcp, L);
        return false;
    }
    const float lo = m;
    scale = __half2float(__float2half_rn(scale));
    m = __half2float(__float2half_rn(m));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rcp) : "f"(scale));
    inv = scale > 0.0f ? rcp : 0.0f;                                                    // scale 0 (no range, or underflow): codes 0
    return !(__fsub_rn(lo, m) >= -0.49f * scale && __fsub_rn(mx, m) <= (L + 0.49f) * scale);
}

template <int BITS, int NW, bool BF16, bool M16, int GB>
__global__ void __launch_bounds__(KB_THREADS, 2) quant_keys_block_kernel(const KeyBlockParams p)
{
    using Lay = KbLayout<GB>;
    constexpr int G = 32 * NW;
    constexpr int GPT = 4 / NW;                          // groups per tile
    constexpr int ES = BF16 ? 2 : 4;
    extern __shared__ __align__(128) float smem[];
    float *W_hi = smem, *W_lo = W_hi + Lay::W_FLOATS;    // the current head's panels
    float *E_all = W_lo + Lay::W_FLOATS;                 // per slot: E_hi, E_lo
    u64 *mbar = reinterpret_cast<u64 *>(E_all + 2 * Lay::SLOTS * Lay::E_FLOATS);       // [SLOTS] products done, [1] panels staged
    // [0] tensor-memory base, [1] a bounded wait ran out, [2 + slot] arrivals of the slot's warps
    volatile unsigned *shared_words = reinterpret_cast<volatile unsigned *>(mbar + Lay::SLOTS + 1);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wq = warp & 3;                             // quarter of the tile's tokens = of the tensor-memory lanes
    const int slot = GB == 64 ? 0 : warp >> 2;
    const int half = GB == 64 ? warp >> 2 : 0;           // which 32 channels of a block of 64
    const int q = lane & 7, s = lane >> 3;               // channel quad; token phase: tokens 4 i + s
    const int wteam = wq % NW;
    const int team_id = 1 + (warp >> 2) * GPT + wq / NW;

    const int u_lo = (int)((long long)p.total_units * blockIdx.x / gridDim.x);
    const int u_hi = (int)((long long)p.total_units * (blockIdx.x + 1) / gridDim.x);
    grid_wait();
    if (p.form && *p.form != GB) return;
    const unsigned img_mbar = smem_u32(mbar + Lay::SLOTS);

    // One head's panels into shared memory (one thread).  The image has them by 32 source channels with all later channels; of those
    // only the channels behind the block of g are taken, and the source blocks of a step put side by side along K.
    auto stage_panels = [&](int h) {
        const float *src = p.Wimg + (long long)h * KEY_IMG_FLOATS + KEY_PLAIN_FLOATS;
        if (!SQ_CHK_G(p.status, src, 2 * KEY_PANEL_FLOATS * 4, p.x_img)) return;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(img_mbar), "r"(2 * Lay::W_FLOATS * 4) : "memory");
        for (int part = 0; part < 2; ++part)
            for (int b = 0; b < (D - GB) / KEY_BLK; ++b) {                 // source blocks that lead anywhere
                const int step = b * KEY_BLK / GB, n = D - (step + 1) * GB, nb = D - (b + 1) * KEY_BLK;        // taken, present
                float *dst = (part ? W_lo : W_hi) + (GB == 64 ? 0 : kb_panel_off(step)) + (b * KEY_BLK - step * GB) * n;
                const float *from = src + part * KEY_PANEL_FLOATS + key_panel_off(b) + 4 * (nb - n);
                for (int kc = 0; kc < KEY_BLK / 4; ++kc)
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(smem_u32(dst + kc * 4 * n)), "l"(from + kc * 4 * nb), "r"(16u * n), "r"(img_mbar) : "memory");
            }
    };

    if (threadIdx.x == 0) {
#pragma unroll
        for (int t = 0; t < Lay::SLOTS; ++t) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar + t)), "r"(1) : "memory");
            shared_words[2 + t] = 0;
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(img_mbar), "r"(1) : "memory");
        shared_words[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (u_lo < u_hi) stage_panels(u_lo / p.units_per_head);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(const_cast<unsigned *>(shared_words))), "r"((unsigned)Lay::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = shared_words[0];
    const unsigned t_tile = tmem_base + slot * Lay::SLOT_COLS;
    const unsigned t_mine = t_tile + ((unsigned)(wq * 32) << 16);
    float *E_hi = E_all + slot * 2 * Lay::E_FLOATS, *E_lo = E_hi + Lay::E_FLOATS;
    // this warp's 8 chunks x 32 rows of an operand start here; the thread's first row of its quad
    const int e_warp = half * 8 * KB_CHUNK_FLOATS + wq * 32 * 4;
    const int e_mine = e_warp + q * KB_CHUNK_FLOATS + s * 4;
    const unsigned my_mbar = smem_u32(mbar + slot);
    unsigned phase = 0, img_phase = 0;
    const CodeLanes cl = code_lanes<BITS>(q);

    struct Place {
        bool active;              // the warp's group exists (a head's last unit may be ragged: its spare warps redo the last
                                  // group and store nothing)
        const char *row;          // the thread's first token at its quad of block 0
        unsigned char *codes;     // code row of the token the thread stores (4 q + s)
        long long meta;           // offset of the group's scales / zeros at the lane's own channel of block 0
    };
    auto locate = [&](int unit, Place &t) {
        const int h = unit / p.units_per_head;
        const int tile = (unit - h * p.units_per_head) * Lay::SLOTS + slot;
        const int g_raw = tile * GPT + wq / NW;
        t.active = g_raw < p.groups_per_head;
        const int in_head = t.active ? g_raw : p.groups_per_head - 1;
        const int b = in_head / p.groups_per_bh;
        const int grp = in_head - b * p.groups_per_bh;
        const int tok0 = grp * G + wteam * 32;
        const long long out_tok0 = (long long)b * p.osb + (long long)h * p.osh;
        t.codes = p.codes + (out_tok0 + tok0 + 4 * q + s) * (D * BITS / 8) + half * (BLK * BITS / 8);
        t.meta = (out_tok0 / G + grp) * D + half * BLK + 4 * q + s;
        const long long off = (long long)b * p.sb + (long long)h * p.sh + (long long)(tok0 + s) * p.st + half * BLK + 4 * q;
        t.row = static_cast<const char *>(p.k) + off * ES;
    };
    const long long row_step = 4 * p.st * ES;            // bytes between the thread's tokens

    QuadRows<BF16> raw;
    auto load_rows = [&](const char *row) {
#pragma unroll
        for (int i = 0; i < KB_ROWS; ++i) {
            const char *r = row + i * row_step;
            if (SQ_CHK_G(p.status, r, 4 * ES, p.x_k)) raw.load(i, r);
        }
    };

    Place cur;
    if (u_lo < u_hi) {
        locate(u_lo, cur);
        load_rows(cur.row);
    }
    int staged = -1;
    for (int unit = u_lo; unit < u_hi; ++unit) {
        const int h = unit / p.units_per_head;
        if (h != staged) {
            if (staged >= 0) {                           // (the first copy was started at kernel entry)
                __syncthreads();                         // every product that reads the old panels has been waited for
                if (threadIdx.x == 0) stage_panels(h);
            }
            if (!shared_words[1] && !mbar_wait(img_mbar, img_phase)) {
                shared_words[1] = 1;
                atomicOr(p.status, SQUAT_FLAG_DEVICE_TIMEOUT);
            }
            img_phase ^= 1;
            staged = h;
        }
        Place nxt = cur;
        if (unit + 1 < u_hi) locate(unit + 1, nxt);

#pragma unroll
        for (int step = 0; step < Lay::STEPS; ++step) {
            const bool last = step + 1 == Lay::STEPS;
            u64 x[KB_ROWS][2];
            float m, mx;                                 // extremes of the lane's own channel, 4 q + s: the quad's 4 lanes share out
                                                         // their channels in two halving exchanges
            if (step == 0) {
                if (BF16) {
                    unsigned a[2], b[2];
                    { const uint2 w = raw.words(0); a[0] = b[0] = w.x; a[1] = b[1] = w.y; }
#pragma unroll
                    for (int i = 1; i < KB_ROWS; ++i) {
                        const uint2 w = raw.words(i);
                        a[0] = hmin2_nan_bits(a[0], w.x); b[0] = hmax2_nan_bits(b[0], w.x);
                        a[1] = hmin2_nan_bits(a[1], w.y); b[1] = hmax2_nan_bits(b[1], w.y);
                    }
                    const bool u = s & 2;
                    unsigned ka = hmin2_nan_bits(u ? a[1] : a[0], __shfl_xor_sync(0xffffffffu, u ? a[0] : a[1], 16));
                    unsigned kb = hmax2_nan_bits(u ? b[1] : b[0], __shfl_xor_sync(0xffffffffu, u ? b[0] : b[1], 16));
                    ka = hmin2_nan_bits(ka, __shfl_xor_sync(0xffffffffu, ka, 8));
                    kb = hmax2_nan_bits(kb, __shfl_xor_sync(0xffffffffu, kb, 8));
                    m = (s & 1) ? bf16hi_to_f32(ka) : bf16lo_to_f32(ka);
                    mx = (s & 1) ? bf16hi_to_f32(kb) : bf16lo_to_f32(kb);
                }
#pragma unroll
                for (int i = 0; i < KB_ROWS; ++i) raw.get(i, x[i][0], x[i][1]);
            } else {
                // the products that complete this block's corrections were committed after the previous step
                if (!shared_words[1] && !mbar_wait(my_mbar, phase)) {
                    shared_words[1] = 1;
                    atomicOr(p.status, SQUAT_FLAG_DEVICE_TIMEOUT);
                }
                phase ^= 1;
                tc_fence_after();
                unsigned dv[32];
                const unsigned col = (step - 1) * GB + half * BLK;
                if (SQ_CHK_C(p.status, (int)col + 32 <= D - GB)) {
                    tmem_ld32(t_mine + col, dv);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) dv[i] = 0;
                }
                tc_fence_before();                       // the next product that writes these columns comes after this read
                __syncwarp();
                float *stage = E_lo + e_warp;            // lane = token writes its row, read back as quads: same 16-byte units
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    *reinterpret_cast<uint4 *>(stage + c * KB_CHUNK_FLOATS + lane * 4) = make_uint4(dv[4 * c], dv[4 * c + 1], dv[4 * c + 2], dv[4 * c + 3]);
                __syncwarp();
#pragma unroll
                for (int i = 0; i < KB_ROWS; ++i) {
                    const ulonglong2 dd = *reinterpret_cast<const ulonglong2 *>(E_lo + e_mine + i * 16);
                    u64 k01, k23;
                    raw.get(i, k01, k23);
                    // (the sum as it is, as in the other kernels, though the accumulator's truncation has made it smaller by 3 to 6 x 2^-24 on
                    // average.  Rms error of a group's minimum 0.20e-7 (g = 64) and 0.30 to 0.55e-7 (g = 32) of its range, no more than keys_lane.cu has)
                    x[i][0] = fadd2(k01, dd.x);
                    x[i][1] = fadd2(k23, dd.y);
                }
            }
            // the keys of the next block, or of the next unit's first, are on their way from here on
            auto load_next = [&] {
                if (!last) load_rows(cur.row + (step + 1) * (GB * ES));
                else if (unit + 1 < u_hi) load_rows(nxt.row);
            };
            if (BF16) load_next();                       // float32 rows take the registers that x still needs: later (32-channel
                                                         // blocks, 16-bit scales 111 -> 98 us for 8 x 8 heads x 8160)
            if (step != 0 || !BF16) {
                float a[4], b[4], v[4];
                unpack2(x[0][0], a[0], a[1]);
                unpack2(x[0][1], a[2], a[3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) b[j] = a[j];
#pragma unroll
                for (int i = 1; i + 1 < KB_ROWS; i += 2) {
                    float w[4];
                    unpack2(x[i][0], v[0], v[1]); unpack2(x[i][1], v[2], v[3]);
                    unpack2(x[i + 1][0], w[0], w[1]); unpack2(x[i + 1][1], w[2], w[3]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) { a[j] = min3_nan(a[j], v[j], w[j]); b[j] = max3_nan(b[j], v[j], w[j]); }
                }
                unpack2(x[KB_ROWS - 1][0], v[0], v[1]);
                unpack2(x[KB_ROWS - 1][1], v[2], v[3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) { a[j] = min_nan(a[j], v[j]); b[j] = max_nan(b[j], v[j]); }
                const bool u = s & 2, w = s & 1;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    a[j] = min_nan(u ? a[j + 2] : a[j], __shfl_xor_sync(0xffffffffu, u ? a[j] : a[j + 2], 16));
                    b[j] = max_nan(u ? b[j + 2] : b[j], __shfl_xor_sync(0xffffffffu, u ? b[j] : b[j + 2], 16));
                }
                m = min_nan(w ? a[1] : a[0], __shfl_xor_sync(0xffffffffu, w ? a[0] : a[1], 8));
                mx = max_nan(w ? b[1] : b[0], __shfl_xor_sync(0xffffffffu, w ? b[0] : b[1], 8));
            }
            // What the lanes and the team's warps tell each other goes through the first rows of each chunk of the warp's own
            // E_hi rows, which no product reads now: 0, 1, 2 zero-point, scale, reciprocal; 3, 4 extremes.
            float *own = E_hi + e_warp + q * KB_CHUNK_FLOATS + s;
            if (NW > 1) {
                own[12] = m;
                own[16] = mx;
                team_barrier(team_id, 32 * NW);
#pragma unroll
                for (int o = 1; o < NW; ++o) {
                    const float *peer = own + ((wteam ^ o) - wteam) * 128;
                    m = min_nan(m, peer[12]);
                    mx = max_nan(mx, peer[16]);
                }
            }
            float scale, inv;
            const bool outside = step == 0 ? make_grid<BITS, M16, true>(m, mx, scale, inv) : make_grid<BITS, M16, false>(m, mx, scale, inv);
            own[0] = m;
            own[4] = scale;
            own[8] = -inv;
            __syncwarp();
            Grid4 g;
            {
                const ulonglong2 *quad = reinterpret_cast<const ulonglong2 *>(E_hi + e_warp + q * KB_CHUNK_FLOATS);
                const ulonglong2 a = quad[0], b = quad[1], c = quad[2];
                g.m[0] = a.x; g.m[1] = a.y; g.scale[0] = b.x; g.scale[1] = b.y; g.neg_inv[0] = c.x; g.neg_inv[1] = c.y;
            }
            // all have read; the rows may be overwritten
            if (NW > 1) team_barrier(team_id, 32 * NW);
            else __syncwarp();
            const bool clamp = M16 && __any_sync(0xffffffffu, outside);

            unsigned cw[BITS];                           // 8 tokens x 4 channels x BITS bits
            float *eh = E_hi + e_mine, *el = E_lo + e_mine;
            if (!SQ_CHK_R(p.status, eh, (16 * (KB_ROWS - 1) + 4) * 4, E_hi, Lay::E_FLOATS * 4) ||
                !SQ_CHK_R(p.status, el, (16 * (KB_ROWS - 1) + 4) * 4, E_lo, Lay::E_FLOATS * 4)) {
                quantize_quads<BITS, false, true, false>(x, g, nullptr, nullptr, cw);
            } else if (step == 0) {
                if (clamp) quantize_quads<BITS, M16, true, true>(x, g, eh, el, cw);
                else quantize_quads<BITS, false, true, true>(x, g, eh, el, cw);
            } else if (!last) {
                if (clamp) quantize_quads<BITS, M16, false, true>(x, g, eh, el, cw);
                else quantize_quads<BITS, false, false, true>(x, g, eh, el, cw);
            } else {
                if (clamp) quantize_quads<BITS, M16, false, false>(x, g, nullptr, nullptr, cw);
                else quantize_quads<BITS, false, false, false>(x, g, nullptr, nullptr, cw);
            }

            if (!BF16) load_next();
            if (!last) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the E rows, for the tensor core
                tc_fence_before();
                __threadfence_block();
                __syncwarp();
                // the last of the tile's warps to get here issues the products; nobody waits at a barrier
                bool issue = false;
                if (lane == 0)
                    issue = (atomicAdd(const_cast<unsigned *>(shared_words) + 2 + slot, 1u) & (Lay::WARPS_PER_TILE - 1)) == Lay::WARPS_PER_TILE - 1;
                if (issue) {
                    __threadfence_block();
                    tc_fence_after();
                    const int nb = D - (step + 1) * GB;                 // channels still to come
                    const unsigned idesc = tc_idesc(nb), b_lbo = 16u * nb;
                    const unsigned a_hi = smem_u32(E_hi), a_lo = smem_u32(E_lo);
                    const int off = GB == 64 ? 0 : kb_panel_off(step);
                    const unsigned b_hi = smem_u32(W_hi + off), b_lo = smem_u32(W_lo + off);
                    const unsigned d = t_tile + step * GB;
                    if (SQ_CHK_C(p.status, off + nb * GB <= Lay::W_FLOATS && step * GB + nb <= Lay::SLOT_COLS)) {
#pragma unroll
                        for (int ks = 0; ks < GB / 8; ++ks)             // E_lo x Whi
                            umma_tf32_ss(d, umma_desc(a_lo + ks * 2 * KB_LBO, KB_LBO, KB_SBO), umma_desc(b_hi + ks * 2 * b_lbo, b_lbo, KB_SBO),
                                         idesc, (step | ks) != 0);
#pragma unroll
                        for (int ks = 0; ks < GB / 8; ++ks)             // E_hi x Wlo
                            umma_tf32_ss(d, umma_desc(a_hi + ks * 2 * KB_LBO, KB_LBO, KB_SBO), umma_desc(b_lo + ks * 2 * b_lbo, b_lbo, KB_SBO),
                                         idesc, 1u);
#pragma unroll
                        for (int ks = 0; ks < GB / 8; ++ks)             // E_hi x Whi
                            umma_tf32_ss(d, umma_desc(a_hi + ks * 2 * KB_LBO, KB_LBO, KB_SBO), umma_desc(b_hi + ks * 2 * b_lbo, b_lbo, KB_SBO),
                                         idesc, 1u);
                    }
                    tc_commit(my_mbar);
                }
                __syncwarp();
            }

            // codes and grids, while the products run
            unsigned char *cp = cur.codes + step * (GB * BITS / 8);
            const long long meta = cur.meta + step * GB;
            if (BITS == 2) {
                const uint2 c = transpose_codes2(reinterpret_cast<const unsigned(&)[2]>(cw), cl);
                if (cur.active && SQ_CHK_G(p.status, cp, 8, p.x_codes)) *reinterpret_cast<uint2 *>(cp) = c;
            } else {
                const uint4 c = transpose_codes4(reinterpret_cast<const unsigned(&)[4]>(cw), cl);
                if (cur.active && SQ_CHK_G(p.status, cp, 16, p.x_codes)) *reinterpret_cast<uint4 *>(cp) = c;
            }
            if (cur.active && wteam == 0 &&
                SQ_CHK_G(p.status, static_cast<char *>(p.scales) + meta * (M16 ? 2 : 4), M16 ? 2 : 4, p.x_scales) &&
                SQ_CHK_G(p.status, static_cast<char *>(p.zeros) + meta * (M16 ? 2 : 4), M16 ? 2 : 4, p.x_zeros)) {
                if (M16) {
                    static_cast<__half *>(p.scales)[meta] = __float2half_rn(scale);     // exact
                    static_cast<__half *>(p.zeros)[meta] = __float2half_rn(m);
                } else {
                    static_cast<float *>(p.scales)[meta] = scale;
                    static_cast<float *>(p.zeros)[meta] = m;
                }
                if (!(scale > 0.0f && scale < __int_as_float(0x7f800000)))
                    atomicOr(p.status, scale == 0.0f ? SQUAT_FLAG_ZERO_RANGE : SQUAT_FLAG_NONFINITE);
            }
        }
        cur = nxt;
    }

    // Every committed batch has been waited for unless a wait ran out; then commit once more per slot and give the
    // tensor core a bounded time to drain before the columns are handed back.
    if (shared_words[1] && wq == 0 && half == 0 && lane == 0) {
        tc_commit(my_mbar);
        mbar_wait(my_mbar, phase);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((unsigned)Lay::TMEM_COLS) : "memory");
}

template <int BITS, int NW, bool BF16, bool M16, int GB>
int launch_inst(const KeyBlockParams &p, int grid, cudaStream_t st)
{
    static std::atomic<unsigned long long> allowed{0};
    if (const int rc = squat_allow_smem(reinterpret_cast<const void *>(quant_keys_block_kernel<BITS, NW, BF16, M16, GB>), KbLayout<GB>::SMEM, allowed)) return rc;
    return squat_launch(quant_keys_block_kernel<BITS, NW, BF16, M16, GB>, grid, KB_THREADS, KbLayout<GB>::SMEM, st, p);
}

template <int GB, int BITS, int NW>
int launch(KeyBlockParams p, int H, int B, int dtype, int meta16, cudaStream_t st)
{
    constexpr int UNIT_GROUPS = KbLayout<GB>::SLOTS * (4 / NW);         // groups per unit
    const long long groups_per_head = (long long)B * p.groups_per_bh;
    const long long units_per_head = (groups_per_head + UNIT_GROUPS - 1) / UNIT_GROUPS;
    if (groups_per_head > 0x3fffffffLL || units_per_head * H > 0x7fffffffLL) return SQUAT_ERR_UNSUPPORTED;      // counted in 32 bits
    p.groups_per_head = (int)groups_per_head;
    p.units_per_head = (int)units_per_head;
    p.total_units = (int)(units_per_head * H);
    const int places = 2 * squat_sm_count();
    const int grid = p.total_units < places ? p.total_units : places;
    if (dtype == SQUAT_BF16) return meta16 ? launch_inst<BITS, NW, true, true, GB>(p, grid, st) : launch_inst<BITS, NW, true, false, GB>(p, grid, st);
    return meta16 ? launch_inst<BITS, NW, false, true, GB>(p, grid, st) : launch_inst<BITS, NW, false, false, GB>(p, grid, st);
}

}  // namespace

int squat_launch_quant_keys_block(int block_g, const float *Wimg, const void *k, int dtype, int batch, int H, int T,
                                  long long sb, long long sh, long long st_, int bits, int G,
                                  unsigned char *codes, void *scales, void *zeros,
                                  long long osb, long long osh, unsigned *status, const int *form, int meta16, cudaStream_t st)
{
    KeyBlockParams p;
    p.Wimg = Wimg; p.k = k; p.sb = sb; p.sh = sh; p.st = st_;
    p.codes = codes; p.scales = scales; p.zeros = zeros; p.osb = osb; p.osh = osh;
    p.groups_per_bh = T / G;
    p.status = status;
    p.form = form;
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
    if ((long long)H * batch * (T / G) == 0) return SQUAT_OK;
#define SQ_KB(GB, BITS)                                                          \
    switch (G) {                                                                 \
        case 32: return launch<GB, BITS, 1>(p, H, batch, dtype, meta16, st);     \
        case 64: return launch<GB, BITS, 2>(p, H, batch, dtype, meta16, st);     \
        case 128: return launch<GB, BITS, 4>(p, H, batch, dtype, meta16, st);    \
    }
    if (block_g == 32 && bits == 2) { SQ_KB(32, 2) }
    if (block_g == 32 && bits == 4) { SQ_KB(32, 4) }
    if (block_g == 64 && bits == 2) { SQ_KB(64, 2) }
    if (block_g == 64 && bits == 4) { SQ_KB(64, 4) }
#undef SQ_KB
    return SQUAT_ERR_UNSUPPORTED;
}
