// Gram matrices of bf16 queries on the integer tensor cores, exactly.
//
// M_h = sum over the stacked query rows of q q^T has to be known to fp64 accuracy (subspace.cu says why), and the fp64 pipe
// does 64 multiply-adds per clock and SM: 633 us for 32 heads of 32768 rows.  tcgen05.mma.kind::i8 does 8192.  A bf16 number
// has 8 significant bits, so with one power of two s_c per channel (from its largest element)
//     x s_c = h + 2^-15 l,   h = 256 d0 + d1,   l = 256 d2 + d3     (d1, d3 in [-128, 127], |d0|, |d2| <= 64)
// holds exactly for every element down to 2^-21 of the channel's largest, and M is a sum of ten integer products of digit
// planes, D_a^T D_b for a <= b (the ones with a > b are their transposes), accumulated in 32 bits in tensor memory without
// any rounding.  Elements below that (about one in a million of normally distributed ones) leave a remainder r; they are
// listed, and the reduction adds r x_i to row and column c in fp64.  A head whose list overflows (one token 40 times the rest is
// enough), or that holds a non-finite number, is left to the fp64 kernel of subspace.cu, which is launched in any case and
// returns at once for every other head.  A whole build of 8 heads x 32768 rows takes 318 us, with one token 1000 times the rest
// 495 us (378 in float32; with plain loops in the reduction instead of that kernel 7700).  The only roundings are those of the
// fp64 sums of the parts.
//
//   gram_max_kernel     largest |x| per channel and chunk of rows
//   gram_i8_kernel      one of three kinds of digit products (A = plane 0 with B = planes 0-3; 1 with 1-3; 2 with 2-3 and 3
//                       with 3: 4 + 3 + 3 products, all that the 512 tensor-memory columns hold at a time) on a chunk of
//                       rows.  Warps 0-15 turn rows into digit planes ([row][128 bytes], 128-byte swizzle, which the
//                       descriptors read as M-major A and N-major B), warp 16 issues the products; four stages of 64 rows.
//   (gram_kernel)       heads without the digits' help
//   gram_i8_reduce_kernel   M = sum of the parts S + S^T, remainders
//
// Bound: the instructions that make the digits (100 per eight elements and kind, 16 warps: 0.85 us for 64 rows; the products
// of a stage take 0.25).  32 heads x 32768 rows: 642 -> 367 us for the three kernels; 8 heads x 32640: 182 -> 121; 32 heads x
// 4096: 96 -> 81.
#include <type_traits>
#include "device_helpers.cuh"

namespace {

constexpr int D = SQUAT_D;
constexpr int MAX_ROWS_PER_PART = 1 << 16;     // products up to 2^14: the sum stays within 32 bits

struct GramArgs {
    const __nv_bfloat16 *q;
    int n_tokens, q_per_kv;
    long long stride_h, stride_t;
    int n_rows;                                // n_tokens * q_per_kv
    int parts[3], total_parts;                 // row chunks per kind of product
    int fp64_parts;                            // row chunks of the fp64 kernel, for the heads that it takes
    int max_chunks;                            // row chunks of the maximum kernel
    unsigned *maxima;                          // [H, max_chunks, D / 2] largest |x| bits, two channels a word
    int *rem_count;                            // [H] remainders listed (may exceed the capacity)
    SquatGramRem *rem;                         // [H, SQUAT_GRAM_REM_CAP]
    double *partial;                           // [total_parts, H, D, D]
    double *gram;
    unsigned *status;
};

// address of stacked row n of a KV head: token n mod n_tokens of its query head n / n_tokens
__device__ __forceinline__ const __nv_bfloat16 *row_ptr(const GramArgs &p, int h, int n)
{
    const int qh = n / p.n_tokens;
    return p.q + ((long long)h * p.q_per_kv + qh) * p.stride_h + (long long)(n - qh * p.n_tokens) * p.stride_t;
}

// ------------------------------------------------------------------------------------------------ maxima
constexpr int MAX_THREADS = 256;
__device__ __forceinline__ unsigned max2(unsigned a, unsigned b)
{
    unsigned r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__global__ void __launch_bounds__(MAX_THREADS) gram_max_kernel(const GramArgs p)
{
    __shared__ uint4 sm[MAX_THREADS];
    const int h = blockIdx.y, chunk = blockIdx.x, tid = threadIdx.x, c16 = tid & 15;
    const int per = (p.n_rows + p.max_chunks - 1) / p.max_chunks;
    const int lo = chunk * per, hi = min(p.n_rows, lo + per);
    uint4 m = make_uint4(0, 0, 0, 0);
    // Branch-free addresses (the wrap from one query head to the next is a select, rows past the end repeat the last one), so
    // that the eight loads of a step are in flight together.
    constexpr int STEP = MAX_THREADS / 16, AT_ONCE = 8;
    const long long step = STEP * p.stride_t, wrap = p.stride_h - p.n_tokens * p.stride_t;
    int n = lo + (tid >> 4), t = n % p.n_tokens;
    const __nv_bfloat16 *src = row_ptr(p, h, min(n, p.n_rows - 1)) + 8 * c16;
    for (; n < hi; ) {
        uint4 v[AT_ONCE];
#pragma unroll
        for (int i = 0; i < AT_ONCE; ++i) {
            v[i] = ldg128(src);
            n += STEP;
            t += STEP;
            const bool over = t >= p.n_tokens;
            const long long d = over ? step + wrap : step;
            t = over ? t - p.n_tokens : t;
            src = n < hi ? src + d : src;
        }
#pragma unroll
        for (int i = 0; i < AT_ONCE; ++i) {
            m.x = max2(m.x, v[i].x & 0x7fff7fffu);
            m.y = max2(m.y, v[i].y & 0x7fff7fffu);
            m.z = max2(m.z, v[i].z & 0x7fff7fffu);
            m.w = max2(m.w, v[i].w & 0x7fff7fffu);
        }
    }
    sm[tid] = m;
    __syncthreads();
    if (tid < 16) {
#pragma unroll
        for (int i = 1; i < MAX_THREADS / 16; ++i) {
            const uint4 v = sm[tid + 16 * i];
            m.x = max2(m.x, v.x);
            m.y = max2(m.y, v.y);
            m.z = max2(m.z, v.z);
            m.w = max2(m.w, v.w);
        }
        reinterpret_cast<uint4 *>(p.maxima + ((long long)h * p.max_chunks + chunk) * (D / 2))[tid] = m;
    }
    if (tid == 0 && chunk == 0) p.rem_count[h] = 0;
}

// biased exponent of channel c's largest element (1 for a channel of zeros or subnormals, 255: not finite), from the chunks' maxima
__device__ __forceinline__ int channel_exponent(const GramArgs &p, int h, int c)
{
    unsigned m = 0;
    const unsigned short *src = reinterpret_cast<const unsigned short *>(p.maxima + (long long)h * p.max_chunks * (D / 2)) + c;
#pragma unroll 8
    for (int i = 0; i < p.max_chunks; ++i) m = max(m, (unsigned)src[i * D]);
    return max((int)(m >> 7), 1);
}

// ------------------------------------------------------------------------------------------------ products
constexpr int ROWS = 64, STAGES = 4, CONV_WARPS = 16, CONV = 32 * CONV_WARPS, THREADS = CONV + 32;
constexpr int PLANE = ROWS * D, STAGE = 4 * PLANE;
constexpr size_t SMEM = 1024 + (size_t)STAGES * STAGE;

// planes: 128-byte rows (K), 128-byte swizzle, groups of 8 rows 1024 bytes apart; the next 128 columns of B are the next plane
__device__ __forceinline__ u64 plane_desc(unsigned addr)
{
    return (u64)((addr & 0x3FFFF) >> 4) | ((u64)(PLANE >> 4) << 16) | ((u64)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// int32 accumulator, signed bytes, A M-major, B N-major (one or two planes), M = 128
__host__ __device__ constexpr unsigned idesc(int n)
{
    return (2u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((unsigned)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void tmem_ld16(unsigned taddr, int (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}

// bytes 1 and 0 of eight words as 8 channels of two neighbouring planes (the first one left out if not WITH_HIGH)
template <bool WITH_HIGH>
__device__ __forceinline__ void store_planes(unsigned char *dst, const u64 (&b)[4])
{
    unsigned w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) w[e] = __byte_perm((unsigned)b[e], (unsigned)(b[e] >> 32), 0x5140);
    if (WITH_HIGH) *reinterpret_cast<uint2 *>(dst) = make_uint2(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632));
    *reinterpret_cast<uint2 *>(dst + PLANE) = make_uint2(__byte_perm(w[0], w[1], 0x5410) ^ 0x80808080u, __byte_perm(w[2], w[3], 0x5410) ^ 0x80808080u);
}

// what the digits of eight channels of a row leave over, for the reduction (rare; with a full list nothing more is listed)
__device__ __noinline__ void list_remainders(SquatGramRem *rem, int *rem_count, int row, int c16, uint4 raw, const double *unit, volatile unsigned *list_full)
{
    const unsigned w[4] = {raw.x, raw.y, raw.z, raw.w};
    for (int e = 0; e < 8; ++e) {
        const int c = 8 * c16 + e;
        const double u = unit[c], per_unit = __longlong_as_double((2046ll << 52) - __double_as_longlong(u));      // 1 / u: a power of two
        const double x = (double)((e & 1) ? bf16hi_to_f32(w[e >> 1]) : bf16lo_to_f32(w[e >> 1])) * per_unit;
        const double r = x * 32768.0 - rint(x * 32768.0);             // the digits hold the nearest multiple of 2^-15 units
        if (r == 0.0) continue;
        const int at = atomicAdd(rem_count, 1);
        if (at >= SQUAT_GRAM_REM_CAP) {
            *list_full = 1;
            return;
        }
        SquatGramRem &o = rem[at];
        o.row = row;
        o.channel = c;
        o.r = r * (1.0 / 32768.0) * u;
    }
}

__global__ void __launch_bounds__(THREADS, 1) gram_i8_kernel(const GramArgs p)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *planes = smem_raw + (1024 - (smem_u32(smem_raw) & 1023)) % 1024;       // [STAGES][4 planes][ROWS][128]
    __shared__ __align__(8) u64 full[STAGES], empty[STAGES];
    __shared__ double unit[D];                 // 2^(exponent) of a channel's digit unit
    __shared__ unsigned tmem_sm, timeout;
    __shared__ volatile unsigned list_full;    // the head's list has overflowed: its remainders need not be listed any more
    const int h = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int part = blockIdx.y, kind = part < p.parts[0] ? 0 : part < p.parts[0] + p.parts[1] ? 1 : 2;
    const int chunk = part - (kind > 0 ? p.parts[0] : 0) - (kind > 1 ? p.parts[1] : 0);
    const int lo = (int)((long long)p.n_rows * chunk / p.parts[kind]), hi = (int)((long long)p.n_rows * (chunk + 1) / p.parts[kind]);
    const int n_stages = (hi - lo + ROWS - 1) / ROWS;

    if (warp == CONV_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_sm)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        timeout = list_full = 0;
        for (int i = 0; i < STAGES; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[i])), "r"(CONV_WARPS) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[i])) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < D) {
        const int be = channel_exponent(p, h, tid);
        if (be == 255 && kind == 0 && chunk == 0) atomicAdd(&p.rem_count[h], SQUAT_GRAM_REM_CAP + 1);   // not finite
        unit[tid] = __longlong_as_double((long long)(max(min(be, 254), 13) - 140 + 1023) << 52);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = tmem_sm;

    if (warp < CONV_WARPS) {
        constexpr int STEP = CONV / 16, PER = ROWS / STEP;            // rows per pass of the converters, passes per stage
        const int c16 = tid & 15, r0 = tid >> 4;                      // channels 8 c16 .. 8 c16 + 7 of rows r0 + STEP i
        u64 s2[4];                                                    // 1 / unit, as the packed multiplicand of a channel pair
#pragma unroll
        for (int i = 0; i < 4; ++i) s2[i] = pack2((float)(1.0 / unit[8 * c16 + 2 * i]), (float)(1.0 / unit[8 * c16 + 2 * i + 1]));
        // 1.5 2^23: the integer in the low bits; + 128: the low digit's carry
        const u64 magic2 = pack2(12582912.0f + 128.0f, 12582912.0f + 128.0f), minus2 = pack2(-1.0f, -1.0f), frac2 = pack2(32768.0f, 32768.0f);
        // rows are addressed in 16-byte units from the head's first, with 32-bit steps; rows past the end are not loaded
        const uint4 *base = reinterpret_cast<const uint4 *>(p.q + (long long)h * p.q_per_kv * p.stride_h) + c16;
        int t = (lo + r0) % p.n_tokens, left = hi - lo - r0;
        int off = (int)(((lo + r0) / p.n_tokens * p.stride_h + t * p.stride_t) / 8);
        const int step = (int)(STEP * p.stride_t / 8), wrap = (int)((p.stride_h - p.n_tokens * p.stride_t) / 8);
        constexpr int AHEAD = 4;                                      // stages whose rows are on their way: 48 KB per SM
        uint4 raw[AHEAD][PER];
        auto fetch = [&](uint4 (&v)[PER]) {
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                if (left > 0) v[i] = __ldg(base + off);
                left -= STEP;
                t += STEP;
                off += step;
                if (t >= p.n_tokens) { t -= p.n_tokens; off += wrap; }
            }
        };
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) fetch(raw[u]);
        auto convert = [&](auto kind_constant) {
            constexpr int kind = decltype(kind_constant)::value;
            for (int s0 = 0; s0 < n_stages; s0 += AHEAD) {
#pragma unroll
                for (int u = 0; u < AHEAD; ++u) {
                    const int s = s0 + u;
                    if (s >= n_stages) break;
                    const int buf = s % STAGES;
                    if (s >= STAGES && !timeout && !mbar_wait(smem_u32(&empty[buf]), (s / STAGES - 1) & 1)) timeout = 1;
                    unsigned char *st = planes + buf * STAGE + (c16 & 1) * 8;
#pragma unroll
                    for (int i = 0; i < PER; ++i) {
                        const int r = r0 + STEP * i;
                        if (s == n_stages - 1 && lo + s * ROWS + r >= hi) raw[u][i] = make_uint4(0, 0, 0, 0);
                        const unsigned w[4] = {raw[u][i].x, raw[u][i].y, raw[u][i].z, raw[u][i].w};
                        u64 hb[4], lb[4];
                        unsigned any = 0;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const u64 x = pack2(bf16lo_to_f32(w[e]), bf16hi_to_f32(w[e]));
                            const u64 hm = ffma2(x, s2[e], magic2);
                            const u64 rr = ffma2(x, s2[e], ffma2(hm, minus2, magic2));
                            const u64 lm = ffma2(rr, frac2, magic2);
                            hb[e] = hm;
                            lb[e] = lm;
                            if (kind == 0) {
                                const u64 rem = ffma2(rr, frac2, ffma2(lm, minus2, magic2));
                                any |= (unsigned)rem | (unsigned)(rem >> 32);
                            }
                        }
                        unsigned char *dst = st + r * D + (((c16 >> 1) ^ (r & 7)) << 4);
                        if (kind < 2) store_planes<kind == 0>(dst, hb);
                        store_planes<true>(dst + 2 * PLANE, lb);
                        if (kind == 0 && (any & 0x7fffffffu) && !list_full)
                            list_remainders(p.rem + (long long)h * SQUAT_GRAM_REM_CAP, p.rem_count + h, lo + s * ROWS + r, c16, raw[u][i], unit, &list_full);
                    }
                    fetch(raw[u]);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();                      // one arrival a warp: they are handled one after another
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[buf])) : "memory");
                }
            }
        };
        if (kind == 0) convert(std::integral_constant<int, 0>{});
        else if (kind == 1) convert(std::integral_constant<int, 1>{});
        else convert(std::integral_constant<int, 2>{});
    } else if (lane == 0) {
        for (int s = 0; s < n_stages; ++s) {
            const int buf = s % STAGES;
            if (!timeout && !mbar_wait(smem_u32(&full[buf]), (s / STAGES) & 1)) timeout = 1;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned st = smem_u32(planes + buf * STAGE);
#pragma unroll
            for (int ks = 0; ks < ROWS / 32; ++ks) {
                const u64 p0 = plane_desc(st + ks * 32 * D), p1 = p0 + PLANE / 16, p2 = p0 + 2 * (PLANE / 16), p3 = p0 + 3 * (PLANE / 16);
                const bool acc = s > 0 || ks > 0;
                if (kind == 0) {
                    mma_i8(tmem, p0, p0, idesc(256), acc);
                    mma_i8(tmem + 256, p0, p2, idesc(256), acc);
                } else if (kind == 1) {
                    mma_i8(tmem, p1, p1, idesc(256), acc);
                    mma_i8(tmem + 256, p1, p3, idesc(128), acc);
                } else {
                    mma_i8(tmem, p2, p2, idesc(256), acc);
                    mma_i8(tmem + 256, p3, p3, idesc(128), acc);
                }
            }
            tc_commit(smem_u32(&empty[buf]));
        }
    }
    __syncwarp();
    if (n_stages > 0) {                        // the last stage's commit follows every product
        const int last = n_stages - 1;
        if (!timeout && !mbar_wait(smem_u32(&empty[last % STAGES]), (last / STAGES) & 1)) timeout = 1;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp < CONV_WARPS) {
        // S = 1/2 D_a^T D_a + sum over b > a of D_a^T D_b at the planes' weights 2^8, 1, 2^-7, 2^-15, in 64-bit integers
        const int i = 32 * (warp & 3) + lane, j0 = 128 / (CONV_WARPS / 4) * (warp >> 2);
        const unsigned at = tmem + ((unsigned)(32 * (warp & 3)) << 16);
        const int sh0 = kind == 0 ? 22 : kind == 1 ? 14 : 16, sh1 = kind == 0 ? 15 : kind == 1 ? 8 : 9, sh2 = kind == 0 ? 8 : 0;
        const double ui = unit[i] * (kind == 0 ? 1.0 / (1 << 7) : kind == 1 ? 1.0 / (1 << 15) : 1.0 / (1ull << 31));
        double *out = p.partial + ((long long)part * gridDim.x + h) * D * D + i * D;
#pragma unroll 1
        for (int j = j0; j < j0 + 128 / (CONV_WARPS / 4); j += 16) {
            int a0[16], a1[16], a2[16], a3[16];
            tmem_ld16(at + j, a0);
            tmem_ld16(at + 128 + j, a1);
            tmem_ld16(at + 256 + j, a2);
            if (kind == 0) tmem_ld16(at + 384 + j, a3);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                double v[2];
#pragma unroll
                for (int z = 0; z < 2; ++z) {
                    long long x = n_stages > 0 ? ((long long)a0[e + z] << sh0) + ((long long)a1[e + z] << sh1) + ((long long)a2[e + z] << sh2) : 0;
                    if (kind == 0 && n_stages > 0) x += a3[e + z];
                    v[z] = (double)x * ui * unit[j + e + z];
                }
                *reinterpret_cast<double2 *>(out + j + e) = make_double2(v[0], v[1]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == CONV_WARPS) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    if (tid == 0 && timeout) atomicOr(p.status, SQUAT_FLAG_DEVICE_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------ reduction
constexpr int RED_UNITS = 136 * 16, RED_THREADS = 128;    // tiles on or above the diagonal x 8 rows x halves of a row

__global__ void __launch_bounds__(RED_THREADS) gram_i8_reduce_kernel(const GramArgs p)
{
    __shared__ long long key_sm[SQUAT_GRAM_REM_CAP], sorted_sm[SQUAT_GRAM_REM_CAP];
    __shared__ double r_sm[SQUAT_GRAM_REM_CAP];
    const int h = blockIdx.y, H = gridDim.y, tid = threadIdx.x, unit_id = blockIdx.x * RED_THREADS + tid;
    grid_wait();
    int u = unit_id >> 4, ti = 0, len = 16;    // u-th tile of the upper triangle, row by row
    while (u >= len) { u -= len; --len; ++ti; }
    const int tj = ti + u, a = 8 * ti + ((unit_id >> 1) & 7), b = 8 * tj + 4 * (unit_id & 1);
    double m[4] = {0.0, 0.0, 0.0, 0.0};
    const bool digits = p.rem_count[h] <= SQUAT_GRAM_REM_CAP;             // or the fp64 kernel's parts, tiles of the upper triangle
    const int n_rem = digits ? p.rem_count[h] : 0, n_parts = digits ? p.total_parts : p.fp64_parts;
    const double *src = p.partial + (long long)h * D * D;
#pragma unroll 4
    for (int c = 0; c < n_parts; ++c, src += (long long)H * D * D) {
        const double2 x = *reinterpret_cast<const double2 *>(src + a * D + b), y = *reinterpret_cast<const double2 *>(src + a * D + b + 2);
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        if (digits) {
#pragma unroll
            for (int e = 0; e < 4; ++e) t[e] = src[(b + e) * D + a];
        }
        m[0] += x.x + t[0];
        m[1] += x.y + t[1];
        m[2] += y.x + t[2];
        m[3] += y.y + t[3];
    }
    // remainders, in the order of (row, channel) whatever order they were listed in
    const SquatGramRem *rem = p.rem + (long long)h * SQUAT_GRAM_REM_CAP;
    for (int k = tid; k < n_rem; k += RED_THREADS) key_sm[k] = (long long)rem[k].row * D + rem[k].channel;
    __syncthreads();
    for (int k = tid; k < n_rem; k += RED_THREADS) {
        const long long key = key_sm[k];
        int place = 0;
        for (int z = 0; z < n_rem; ++z) place += key_sm[z] < key;            // an element is listed once: all keys differ
        sorted_sm[place] = key;
        r_sm[place] = rem[k].r;
    }
    __syncthreads();
    for (int k = 0; k < n_rem; ++k) {
        const int c = (int)(sorted_sm[k] % D);
        if (c != a && (unsigned)(c - b) >= 4u) continue;
        const double r = r_sm[k];
        const __nv_bfloat16 *row = row_ptr(p, h, (int)(sorted_sm[k] / D));
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (c == a) m[e] = fma(r, (double)__bfloat162float(row[b + e]), m[e]);
            if (c == b + e) m[e] = fma(r, (double)__bfloat162float(row[a]), m[e]);
        }
    }
    double *g = p.gram + (long long)h * D * D;
    *reinterpret_cast<double2 *>(g + a * D + b) = make_double2(m[0], m[1]);
    *reinterpret_cast<double2 *>(g + a * D + b + 2) = make_double2(m[2], m[3]);
    if (ti != tj) {
#pragma unroll
        for (int e = 0; e < 4; ++e) g[(b + e) * D + a] = m[e];
    }
}

// Row chunks per kind of product: one wave of CTAs (one per SM) or two.  The kinds get equal shares (turning rows into digits
// takes them equally long, and longer than the products), so a wave lasts as long as the kind with the fewest CTAs per head needs
// for its share.  Two waves pay where one cannot be dealt out evenly -- four CTAs per head are 2 + 1 + 1 and last for all rows,
// nine in two waves for 2/3 of them -- and the rows saved are more than the 2048 that the second wave's beginnings, ends and parts
// cost.  Measured, one wave against two (whole power build): 32 heads x 4096 rows 163, 165 us; 5120 177, 177; 8192 218, 210; 32768
// 548, 450.  18 heads (4 + 2 + 2 or 6 + 5 + 5) x 16384 222, 226; 24576 280, 271.  24 heads (2 + 2 + 2 or 4 + 4 + 4) x 32768 364, 370.
bool plan(const squat_subspace *s, int n_rows, int (&parts)[3])
{
    long long best = -1;
    for (int waves = 1; waves <= 2; ++waves) {
        const int total = waves == 1 ? squat_sm_count() / s->n_kv_heads : s->gram_chunks_cap, fewest = total / 3;
        if (fewest < 1 || total > s->gram_chunks_cap || n_rows / fewest >= MAX_ROWS_PER_PART) continue;
        const long long cost = (long long)waves * (n_rows / fewest) + 2048 * (waves - 1);
        if (best >= 0 && cost >= best) continue;
        best = cost;
        parts[1] = parts[2] = fewest;
        parts[0] = total - 2 * fewest;
    }
    return best >= 0;
}

}  // namespace

// bf16 queries, and enough rows: the fp64 kernel's time grows with rows x heads, the integer kernels' beginnings, ends and parts
// cost about 25 us more than its own.  Both sides (whole power build, fp64 and integer): 8 heads x 4096 rows 124, 128 us; 6144 134,
// 132; 16 x 2560 124, 124; 4096 140, 130; 32 x 1536 126, 130; 2048 136, 135; 1 x 8192 136, 204; 1 x 65536 230, 230.  Above 49 heads there
// are two waves at any rate: 64 x 1280 146, 150; 1536 159, 155; 96 x 1024 153, 157.
// The loads step 32 tokens at a time and cross one query head at most.  Their offsets, in 16-byte units from a KV head's first row,
// are 32-bit and run on for up to 320 rows (that are not loaded) behind the last one, so views that spread a KV head over 32 GB
// go to the fp64 kernel.
bool squat_gram_i8_fits(const squat_subspace *s, int dtype, int n_q_heads, int n_tokens, long long stride_h, long long stride_t)
{
    int parts[3];
    const int q_per_kv = n_q_heads / s->n_kv_heads;
    const long long rows = (long long)n_tokens * q_per_kv;
    const double reach = ((double)(q_per_kv + 11) * stride_h + (double)(n_tokens + 320) * stride_t) / 8;
    const long long enough = squat_sm_count() / s->n_kv_heads >= 3 ? 3 << 14 : 3 << 15;
    return dtype == SQUAT_BF16 && n_tokens >= 32 && rows * s->n_kv_heads >= enough && rows < (1 << 30) && reach < 2147483648.0 && plan(s, (int)rows, parts);
}

int squat_launch_gram_i8(squat_subspace *s, const void *q, int n_q_heads, int n_tokens, long long stride_h, long long stride_t, cudaStream_t st)
{
    const int H = s->n_kv_heads;
    GramArgs p;
    p.q = static_cast<const __nv_bfloat16 *>(q);
    p.n_tokens = n_tokens;
    p.q_per_kv = n_q_heads / H;
    p.stride_h = stride_h;
    p.stride_t = stride_t;
    p.n_rows = n_tokens * p.q_per_kv;
    if (!plan(s, p.n_rows, p.parts)) return SQUAT_ERR_UNSUPPORTED;
    p.total_parts = p.parts[0] + p.parts[1] + p.parts[2];
    p.max_chunks = s->gram_chunks_cap < (p.n_rows + 255) / 256 ? s->gram_chunks_cap : (p.n_rows + 255) / 256;
    p.maxima = s->gram_max;
    p.rem_count = s->gram_rem_count;
    p.rem = s->gram_rem;
    p.partial = s->gram_partial;
    p.gram = s->gram;
    p.status = s->status;
    gram_max_kernel<<<dim3(p.max_chunks, H), MAX_THREADS, 0, st>>>(p);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    static std::atomic<unsigned long long> allowed{0};
    if (const int rc = squat_allow_smem(reinterpret_cast<const void *>(gram_i8_kernel), SMEM, allowed)) return rc;
    gram_i8_kernel<<<dim3(H, p.total_parts), THREADS, SMEM, st>>>(p);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    if (const int rc = squat_launch_gram_parts(q, SQUAT_BF16, H, p.n_tokens, p.q_per_kv, stride_h, stride_t, s->gram_chunks_cap, s->gram_rem_count, s->gram_partial, &p.fp64_parts, st)) return rc;
    return squat_launch(gram_i8_reduce_kernel, dim3(RED_UNITS / RED_THREADS, H), RED_THREADS, 0, st, p);
}
