// Step 1 of the write path: query subspace and update matrices, all in fp64.
//
//   gram_kernel      M_h = Qc^T Qc for the stacked prompt queries of KV head h (Section 3.2;
//                    Algorithm 1 line 5 needs only the right singular vectors and singular values
//                    of Qc, i.e. the eigen-pairs of M_h; GQA stacking rule of Appendix C).
//   (eig.cu)         eigen-decomposition of M_h: eigenvectors v_i and eigenvalues sigma_i^2.
//   assemble_kernel  P_inv = (I + lambda Qhat^T Qhat)^{-1} = I - sum_i s_i/(1+s_i) v_i v_i^T with
//                    s_i = lambda sigma_i^2 (Woodbury with orthonormal v_i; footnote of Prop. 4),
//                    then the update matrices B_t H_t of Lemma 3 read off the LDL^T factorisation
//                    P_inv = (I+W) D (I+W)^T: for g = 1, I+W is its unit lower factor (this equals
//                    the chain of Prop. 2 / Lemma 4 followed by B_t h_t, which the CPU oracle runs
//                    literally); for g > 1 each block column is multiplied by the inverse of its
//                    unit-lower diagonal block, which turns the scalar factor into the block one.
//
// The cut at rank r can fall between nearly equal eigenvalues whose directions still carry
// weight lambda sigma^2, so single precision anywhere in this step changes quantized codes
// downstream; products of bf16 inputs are exact in fp64 and everything stays fp64 until W is
// rounded to float32 at the very end.
#include <type_traits>
#include <utility>
#include "device_helpers.cuh"

namespace {

constexpr int D = SQUAT_D;

// ------------------------------------------------------------------------------------- Gram
// M = Qc^T Qc on the fp64 tensor-core path (mma.sync m8n8k4, fp64 operands and accumulators: products of bf16 or
// fp32 inputs are exact in fp64).  M is symmetric: of the 16 x 16 grid of 8 x 8 tiles only the 136 tiles on or above
// the diagonal are computed, 17 per warp, 8 warps per CTA.  The A fragment of tile row i (A[m][k] = Q[token k][8 i + m])
// and the B fragment of tile column i (B[k][n] = Q[token k][8 i + n]) are the same register, so a warp loads one
// fragment per 8-channel group and 4-token step and feeds it to every tile that touches the group.
constexpr int GRAM_THREADS = 256;
constexpr int GRAM_ROWS = 32;                  // token rows staged in shared memory per step
constexpr int GRAM_LDR = D + 4;                // row stride (doubles): 4 tokens x 8 channels of a fragment hit 32 distinct words
constexpr int GRAM_TILES_PER_WARP = 17;
constexpr int GRAM_CTAS_PER_SM = 2;

// u-th tile of the upper triangle, row by row: (ti, tj), ti <= tj
template <int U>
struct GramTile {
    static constexpr int row()
    {
        int u = U, ti = 0, len = 16;
        while (u >= len) { u -= len; --len; ++ti; }
        return ti;
    }
    static constexpr int ti = row();
    static constexpr int tj = ti + (U - (ti * 16 - ti * (ti - 1) / 2));
};


template <int W, int... N>
__device__ __forceinline__ void gram_warp_step(double (&acc)[GRAM_TILES_PER_WARP][2], const double (&F)[16],
                                               std::integer_sequence<int, N...>)
{
    (dmma(acc[N][0], acc[N][1], F[GramTile<GRAM_TILES_PER_WARP * W + N>::ti], F[GramTile<GRAM_TILES_PER_WARP * W + N>::tj]), ...);
}

template <int W, int... N>
__device__ __forceinline__ void gram_warp_store(const double (&acc)[GRAM_TILES_PER_WARP][2], double *out, int lane,
                                                std::integer_sequence<int, N...>)
{
    // C fragment: thread holds row lane / 4, columns 2 (lane % 4) and 2 (lane % 4) + 1 of the tile
    ((*reinterpret_cast<double2 *>(out + (GramTile<GRAM_TILES_PER_WARP * W + N>::ti * 8 + (lane >> 2)) * D +
                                   GramTile<GRAM_TILES_PER_WARP * W + N>::tj * 8 + 2 * (lane & 3)) = make_double2(acc[N][0], acc[N][1])), ...);
}

template <bool BF16, int W>
__device__ __forceinline__ void gram_warp_body(const double *rows, double (&acc)[GRAM_TILES_PER_WARP][2], int lane)
{
    const double *base = rows + (lane & 3) * GRAM_LDR + (lane >> 2);
#pragma unroll 2
    for (int k0 = 0; k0 < GRAM_ROWS; k0 += 4) {
        double F[16];
#pragma unroll
        for (int g = 0; g < 16; ++g) F[g] = base[k0 * GRAM_LDR + g * 8];
        gram_warp_step<W>(acc, F, std::make_integer_sequence<int, GRAM_TILES_PER_WARP>{});
    }
}

template <bool BF16>
__global__ void __launch_bounds__(GRAM_THREADS, GRAM_CTAS_PER_SM) gram_kernel(
    const void *q, int n_tokens, int q_per_kv, long long stride_h, long long stride_t,
    int rows_per_chunk, const int *list_counts, double *__restrict__ partial /* [chunks, H, D, D] */)
{
    __shared__ __align__(16) double rows[GRAM_ROWS * GRAM_LDR];
    const int h = blockIdx.y, chunk = blockIdx.x, H = gridDim.y;
    if (list_counts) {
        grid_wait(q);
        if (list_counts[h] <= SQUAT_GRAM_REM_CAP) return;                 // gram_i8.cu has this head's sums
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long N = (long long)n_tokens * q_per_kv;
    const long long row_lo = (long long)chunk * rows_per_chunk;
    long long row_hi = row_lo + rows_per_chunk;
    if (row_hi > N) row_hi = N;

    double acc[GRAM_TILES_PER_WARP][2];
#pragma unroll
    for (int n = 0; n < GRAM_TILES_PER_WARP; ++n) acc[n][0] = acc[n][1] = 0.0;

    // Staging: a thread moves pairs of neighbouring channels (4 bytes of bf16, 8 of fp32), so that a warp's
    // 16-byte stores of the converted pairs fall on consecutive words.  The global loads of step s + 1 are
    // issued before the arithmetic of step s, so their latency is hidden.
    constexpr int NPAIR = GRAM_ROWS * (D / 2) / GRAM_THREADS;          // 16
    using raw_t = typename std::conditional<BF16, uint32_t, uint2>::type;
    raw_t pre[NPAIR];
    // A thread's pairs of one step sit in rows r0 + rr0 + 4 it of the stack (rr0 = thread / 64) at a fixed channel pair.
    // Row n of the stack is token n mod n_tokens of query head n / n_tokens of the KV head: (head, token) of the
    // thread's first row are divided out once and then carried from row to row and from step to step (fetch is called
    // for consecutive steps), so the loop holds no division.
    static_assert(GRAM_THREADS / (D / 2) == 4 && NPAIR * 4 == GRAM_ROWS, "four rows per pass of the CTA over a step");
    const int c2 = threadIdx.x % (D / 2), rr0 = threadIdx.x / (D / 2);
    int q_next = 0, t_next = 0;                                     // query head and token of row (next r0) + rr0
    if (row_lo < row_hi) {
        const long long n0 = row_lo + rr0;
        q_next = (int)(n0 / n_tokens);
        t_next = (int)(n0 - (long long)q_next * n_tokens);
    }
    auto fetch = [&](long long r0) {
        int qh = q_next, t = t_next;
#pragma unroll
        for (int it = 0; it < NPAIR; ++it) {
            const long long n = r0 + rr0 + 4 * it;
            pre[it] = raw_t{};
            if (n < row_hi) {
                const long long off = ((long long)h * q_per_kv + qh) * stride_h + (long long)t * stride_t + c2 * 2;
                if constexpr (BF16) pre[it] = __ldg(reinterpret_cast<const uint32_t *>(reinterpret_cast<const __nv_bfloat16 *>(q) + off));
                else pre[it] = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const float *>(q) + off));
            }
            t += 4;
            while (t >= n_tokens) { t -= n_tokens; ++qh; }
        }
        q_next = qh;                                                // = (head, token) of row r0 + GRAM_ROWS + rr0
        t_next = t;
    };
    if (row_lo < row_hi) fetch(row_lo);
    for (long long r0 = row_lo; r0 < row_hi; r0 += GRAM_ROWS) {
        __syncthreads();
#pragma unroll
        for (int it = 0; it < NPAIR; ++it) {
            const int idx = threadIdx.x + it * GRAM_THREADS;
            const int rr = idx / (D / 2), c2 = idx % (D / 2);
            double2 v;
            if constexpr (BF16) { v.x = (double)bf16lo_to_f32(pre[it]); v.y = (double)bf16hi_to_f32(pre[it]); }
            else { v.x = (double)__uint_as_float(pre[it].x); v.y = (double)__uint_as_float(pre[it].y); }
            *reinterpret_cast<double2 *>(&rows[rr * GRAM_LDR + c2 * 2]) = v;
        }
        __syncthreads();
        if (r0 + GRAM_ROWS < row_hi) fetch(r0 + GRAM_ROWS);
        switch (warp) {
        case 0: gram_warp_body<BF16, 0>(rows, acc, lane); break;
        case 1: gram_warp_body<BF16, 1>(rows, acc, lane); break;
        case 2: gram_warp_body<BF16, 2>(rows, acc, lane); break;
        case 3: gram_warp_body<BF16, 3>(rows, acc, lane); break;
        case 4: gram_warp_body<BF16, 4>(rows, acc, lane); break;
        case 5: gram_warp_body<BF16, 5>(rows, acc, lane); break;
        case 6: gram_warp_body<BF16, 6>(rows, acc, lane); break;
        default: gram_warp_body<BF16, 7>(rows, acc, lane); break;
        }
    }
    double *out = partial + ((long long)chunk * H + h) * D * D;
    constexpr auto seq = std::make_integer_sequence<int, GRAM_TILES_PER_WARP>{};
    switch (warp) {
    case 0: gram_warp_store<0>(acc, out, lane, seq); break;
    case 1: gram_warp_store<1>(acc, out, lane, seq); break;
    case 2: gram_warp_store<2>(acc, out, lane, seq); break;
    case 3: gram_warp_store<3>(acc, out, lane, seq); break;
    case 4: gram_warp_store<4>(acc, out, lane, seq); break;
    case 5: gram_warp_store<5>(acc, out, lane, seq); break;
    case 6: gram_warp_store<6>(acc, out, lane, seq); break;
    default: gram_warp_store<7>(acc, out, lane, seq); break;
    }
}

// Sums the per-chunk partials in a fixed order and mirrors the upper tiles: gram[h] full symmetric.  One thread takes four
// neighbouring elements of a row of one of the 136 stored tiles (two 16-byte loads per chunk, all chunks' loads
// independent) and writes them and, for a tile above the diagonal, their mirror images.
constexpr int GRED_UNITS = 136 * 16;           // 136 tiles x 8 rows x 2 halves of a row
constexpr int GRED_THREADS = 128;
__global__ void __launch_bounds__(GRED_THREADS) gram_reduce_kernel(const double *__restrict__ partial, int chunks, int H, double *__restrict__ gram)
{
    const int h = blockIdx.y;
    const int unit = blockIdx.x * GRED_THREADS + threadIdx.x;
    if (unit >= GRED_UNITS) return;
    int u = unit >> 4, ti = 0, len = 16;       // u-th tile of the upper triangle, row by row
    while (u >= len) { u -= len; --len; ++ti; }
    const int tj = ti + u;
    const int a = 8 * ti + ((unit >> 1) & 7), b = 8 * tj + 4 * (unit & 1);
    const double *src = partial + (long long)h * D * D + a * D + b;
    double2 s0 = make_double2(0.0, 0.0), s1 = s0;
    for (int c = 0; c < chunks; ++c) {
        const double2 v0 = *reinterpret_cast<const double2 *>(src + (long long)c * H * D * D);
        const double2 v1 = *reinterpret_cast<const double2 *>(src + (long long)c * H * D * D + 2);
        s0.x += v0.x; s0.y += v0.y; s1.x += v1.x; s1.y += v1.y;
    }
    double *g = gram + (long long)h * D * D;
    *reinterpret_cast<double2 *>(g + a * D + b) = s0;
    *reinterpret_cast<double2 *>(g + a * D + b + 2) = s1;
    if (ti != tj) {
        g[(b + 0) * D + a] = s0.x;
        g[(b + 1) * D + a] = s0.y;
        g[(b + 2) * D + a] = s1.x;
        g[(b + 3) * D + a] = s1.y;
    }
}

static_assert(GRAM_TILES_PER_WARP * (GRAM_THREADS / 32) == 136, "the warps share the upper triangle evenly");


// ------------------------------------------------------------------------------------- assemble
// P_inv and its LDL^T factorisation, one CTA per head.  The 136 tiles of 8 x 8 on or below the diagonal live in registers
// as accumulators of the fp64 tensor path, dealt column by column to the 16 warps; the factorisation goes by panels of 8
// columns: the owners of a column of tiles publish it, four warps (a thread per row, the 8 x 8 diagonal block factored by
// each of them for itself, so that nothing is handed over in between) solve for the panel's rows, and every warp subtracts
// the panel's product from its later tiles.  Two barriers per panel, 32 in all; one column at a time took 128 steps of a
// barrier and a pass through shared memory each (36 us on 32 heads, of which the dependent divisions are 5).
constexpr int ASM_THREADS = 512, ASM_WARPS = 16;
constexpr int ASM_LD = D + 1;                  // row stride of L in shared memory (block updates)
constexpr int ASM_LDU = D + 4;                 // of the staged vectors: 4 mod 16, fragments without bank conflicts
constexpr int ASM_LDP = 12;                    // of a panel's rows: fragments without bank conflicts
constexpr int ASM_TILES = 9;                   // tiles per warp, at most
constexpr int ASM_STAGE = 32;                  // vectors staged at a time
constexpr size_t ASM_SMEM = sizeof(double) * (D * ASM_LD + 3 * D * ASM_LDP + D);
static_assert(2 * ASM_STAGE * ASM_LDU <= D * ASM_LD && ASM_SMEM <= 227 * 1024, "shared memory of assemble_kernel");

// row and column of the u-th tile of the lower triangle, column by column
__device__ __forceinline__ void asm_tile(int u, int &ti, int &tj)
{
    int c = 0, len = 16;
    while (u >= len) { u -= len; --len; ++c; }
    tj = c;
    ti = c + u;
}

// X <- X inverse(Lb) for the rows below a diagonal block Lb (unit lower, GB x GB, at A[c0][c0]): four lanes a row, columns
// dealt cyclically, from the last column down.
template <int GB>
__device__ __forceinline__ void block_solve(double *A, int tid)
{
    constexpr int PER = GB / 4, BLOCKS = D / GB - 1;
    const int sub = tid & 3;
    int item = tid >> 2;                       // (block, row below it)
    for (;; item += ASM_THREADS / 4) {
        int t = 0, row = item;
        while (t < BLOCKS && row >= D - (t + 1) * GB) { row -= D - (t + 1) * GB; ++t; }
        const bool live = t < BLOCKS;
        if (!__any_sync(0xffffffffu, live)) break;
        const int c0 = live ? t * GB : 0;
        double *x_sm = A + (live ? (t + 1) * GB + row : 0) * ASM_LD + c0;
        const double *lb = A + c0 * ASM_LD + c0;
        double x[PER];
#pragma unroll
        for (int m = 0; m < PER; ++m) x[m] = x_sm[4 * m + sub];
#pragma unroll
        for (int c = GB - 1; c >= 1; --c) {
            const double xc = __shfl_sync(0xffffffffu, x[c / 4], c % 4, 4);
#pragma unroll
            for (int m = 0; m <= (c - 1) / 4; ++m)
                if (4 * m + 3 < c || 4 * m + sub < c) x[m] = fma(-xc, lb[c * ASM_LD + 4 * m + sub], x[m]);
        }
        if (live) {
#pragma unroll
            for (int m = 0; m < PER; ++m) x_sm[4 * m + sub] = x[m];
        }
    }
}

__global__ void __launch_bounds__(ASM_THREADS, 1) assemble_kernel(
    const double *__restrict__ eigval, const double *__restrict__ eigvec, int rank_r, double lambda, int g,
    float *__restrict__ Wt, int left_rows)
{
    // left_rows = 0: P_inv = I - sum_i s_i/(1+s_i) v_i v_i^T from eigen-pairs (rows i of eigvec, eigval).
    // left_rows > 0: P_inv = I - sum_i z_i x_i^T with x_i = row i and z_i = row left_rows + i of eigvec (block power build).
    extern __shared__ __align__(16) double sm[];
    double *A = sm;                             // [D][ASM_LD] L, for block updates only
    double *U = A;                              // [ASM_STAGE][ASM_LDU] right vectors, before there is an L
    double *UL = U + ASM_STAGE * ASM_LDU;       // the same, left vectors times -coefficient
    double *P = A + D * ASM_LD;                 // [D][ASM_LDP] the panel's columns of the matrix
    double *Lp = P + D * ASM_LDP, *Vp = Lp + D * ASM_LDP;     // the panel's rows of L and of L D
    double *coef = Vp + D * ASM_LDP;            // -s_i / (1 + s_i)
    const int h = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int fr = lane >> 2, fk = lane & 3;
    const double *V = eigvec + (long long)h * D * D;
    float *out = Wt + (long long)h * D * D;

    if (tid < D) {
        double mu = eigval[(long long)h * D + tid];
        if (!(mu > 0.0)) mu = 0.0;
        const double s = lambda * mu;
        coef[tid] = (tid < rank_r) ? (left_rows > 0 ? -1.0 : -s / (1.0 + s)) : 0.0;
    }
    int ti[ASM_TILES], tj[ASM_TILES];
    double c[ASM_TILES][2];
#pragma unroll
    for (int n = 0; n < ASM_TILES; ++n) {
        const int u = warp + ASM_WARPS * n;
        ti[n] = tj[n] = 16;                     // no tile
        if (u < 136) asm_tile(u, ti[n], tj[n]);
        c[n][0] = ti[n] == tj[n] && fr == 2 * fk ? 1.0 : 0.0;
        c[n][1] = ti[n] == tj[n] && fr == 2 * fk + 1 ? 1.0 : 0.0;
    }
    for (int i0 = 0; i0 < rank_r; i0 += ASM_STAGE) {
        const int ni = rank_r - i0 < ASM_STAGE ? rank_r - i0 : ASM_STAGE, nk = (ni + 3) / 4 * 4;
        __syncthreads();
        for (int idx = tid; idx < nk * D; idx += ASM_THREADS) {
            const int e = idx / D, i = idx % D;
            U[e * ASM_LDU + i] = e < ni ? V[(long long)(i0 + e) * D + i] : 0.0;
            UL[e * ASM_LDU + i] = e < ni ? coef[i0 + e] * V[(long long)(left_rows + i0 + e) * D + i] : 0.0;
        }
        __syncthreads();
        for (int e = 0; e < nk; e += 4) {
#pragma unroll
            for (int n = 0; n < ASM_TILES; ++n) {
                if (ti[n] == 16) continue;      // warp-uniform
                dmma(c[n][0], c[n][1], UL[(e + fk) * ASM_LDU + 8 * ti[n] + fr], U[(e + fk) * ASM_LDU + 8 * tj[n] + fr]);
            }
        }
    }
    auto publish = [&](int p) {                 // the tiles of column p, as rows of 8
#pragma unroll
        for (int n = 0; n < ASM_TILES; ++n)
            if (tj[n] == p) *reinterpret_cast<double2 *>(&P[(8 * ti[n] + fr) * ASM_LDP + 2 * fk]) = make_double2(c[n][0], c[n][1]);
    };
    publish(0);
    __syncthreads();
#pragma unroll 1
    for (int p = 0; p < 16; ++p) {
        if (tid < D) {
            double d[8][8], v[8], l[8];         // the diagonal block (lower half) and this thread's row
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int k = 0; k <= i; ++k) d[i][k] = P[(8 * p + i) * ASM_LDP + k];
            const bool below = tid >= 8 * p;
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = below ? P[tid * ASM_LDP + k] : 0.0;
            // column k: v_k = L_rk d_k is final, l_k = v_k / d_k; later columns lose v_k times row element L_ck
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const double inv = rcp_nr(d[k][k]);
                l[k] = v[k] * inv;
#pragma unroll
                for (int i = k + 1; i < 8; ++i) {
                    const double li = d[i][k] * inv;                  // L_ik of the diagonal block
#pragma unroll
                    for (int z = i; z < 8; ++z) d[z][i] = fma(-li, d[z][k], d[z][i]);
                    v[i] = fma(-li, v[k], v[i]);
                }
            }
            if (below) {
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    *reinterpret_cast<double2 *>(&Lp[tid * ASM_LDP + k]) = make_double2(-l[k], -l[k + 1]);
                    *reinterpret_cast<double2 *>(&Vp[tid * ASM_LDP + k]) = make_double2(v[k], v[k + 1]);
                }
            }
            if (g == 1) {
                // Wt[j][j'] = W[j'][j] = L[j'][j] below the diagonal, zero on and above it
#pragma unroll
                for (int k = 0; k < 8; ++k) out[(8 * p + k) * D + tid] = tid > 8 * p + k ? (float)l[k] : 0.0f;
            } else if (below) {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (tid > 8 * p + k) A[tid * ASM_LD + 8 * p + k] = l[k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int n = 0; n < ASM_TILES; ++n) {
            if (tj[n] == 16 || tj[n] <= p) continue;
            const double *lp = Lp + (8 * ti[n] + fr) * ASM_LDP + fk, *vp = Vp + (8 * tj[n] + fr) * ASM_LDP + fk;
            dmma(c[n][0], c[n][1], lp[0], vp[0]);
            dmma(c[n][0], c[n][1], lp[4], vp[4]);
        }
        if (p < 15) publish(p + 1);
        __syncthreads();
    }
    if (g == 1) {
        asm volatile("griddepcontrol.wait;" ::: "memory");      // (see the launcher) what follows this kernel follows the tables' too
        return;
    }
    // g > 1: block column t becomes L[rest, blk] * inverse(unit-lower diagonal block)
    if (g == 64) block_solve<64>(A, tid);
    else if (g == 32) block_solve<32>(A, tid);
    else {
        const int T = D / g;
        for (int idx = tid; idx < D * (T - 1); idx += ASM_THREADS) {
            const int row = idx % D, t = idx / D;          // block t: columns [t*g, (t+1)*g)
            const int c0 = t * g;
            if (row < c0 + g) continue;
            double *x = A + row * ASM_LD + c0;
            for (int cc = g - 2; cc >= 0; --cc) {
                double s = x[cc];
                for (int cp = cc + 1; cp < g; ++cp) s = fma(-x[cp], A[(c0 + cp) * ASM_LD + c0 + cc], s);
                x[cc] = s;
            }
        }
    }
    __syncthreads();
    // Wt[j][j'] = W[j'][j]: zero on and above the block diagonal
    for (int idx = tid; idx < D * D; idx += ASM_THREADS) {
        const int j = idx / D, jp = idx % D;
        const int blk_end = (j / g + 1) * g;
        out[idx] = (jp >= blk_end) ? (float)A[jp * ASM_LD + j] : 0.0f;
    }
}

}  // namespace

int squat_launch_gram_parts(const void *q, int dtype, int H, int n_tokens, int q_per_kv, long long stride_h, long long stride_t,
                            int chunks_cap, const int *list_counts, double *partial, int *chunks, cudaStream_t st)
{
    const long long N = (long long)n_tokens * q_per_kv;
    long long rows_per_chunk = (N + chunks_cap - 1) / chunks_cap;
    rows_per_chunk = (rows_per_chunk + GRAM_ROWS - 1) / GRAM_ROWS * GRAM_ROWS;
    if (rows_per_chunk < 2 * GRAM_ROWS) rows_per_chunk = 2 * GRAM_ROWS;
    *chunks = (int)((N + rows_per_chunk - 1) / rows_per_chunk);
    if (*chunks < 1) *chunks = 1;
    const dim3 grid(*chunks, H);
    if (list_counts) return squat_launch(gram_kernel<true>, grid, GRAM_THREADS, 0, st, q, n_tokens, q_per_kv, stride_h, stride_t, (int)rows_per_chunk, list_counts, partial);
    if (dtype == SQUAT_BF16)
        gram_kernel<true><<<grid, GRAM_THREADS, 0, st>>>(q, n_tokens, q_per_kv, stride_h, stride_t, (int)rows_per_chunk, list_counts, partial);
    else
        gram_kernel<false><<<grid, GRAM_THREADS, 0, st>>>(q, n_tokens, q_per_kv, stride_h, stride_t, (int)rows_per_chunk, list_counts, partial);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    return SQUAT_OK;
}

int squat_launch_gram(squat_subspace *s, const void *q, int dtype, int n_q_heads, int n_tokens,
                      long long stride_h, long long stride_t, cudaStream_t st)
{
    if (squat_gram_i8_fits(s, dtype, n_q_heads, n_tokens, stride_h, stride_t)) return squat_launch_gram_i8(s, q, n_q_heads, n_tokens, stride_h, stride_t, st);
    const int H = s->n_kv_heads;
    int chunks = 0;
    if (const int rc = squat_launch_gram_parts(q, dtype, H, n_tokens, n_q_heads / H, stride_h, stride_t, s->gram_chunks_cap, nullptr, s->gram_partial, &chunks, st)) return rc;
    gram_reduce_kernel<<<dim3(GRED_UNITS / GRED_THREADS, H), GRED_THREADS, 0, st>>>(s->gram_partial, chunks, H, s->gram);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    return SQUAT_OK;
}

int squat_launch_assemble(squat_subspace *s, int rank_r, double lambda, int block_g, int left_rows, int exact_channels, int block_form, cudaStream_t st)
{
    constexpr size_t smem = ASM_SMEM;
    static std::atomic<unsigned long long> allowed{0};
    if (const int rc = squat_allow_smem(reinterpret_cast<const void *>(assemble_kernel), smem, allowed)) return rc;
    // Behind the tables of the rank-r form the assembly is a programmatic dependent that waits only at its end: the tables' kernel
    // lets its dependents start at once, both read the eigen-pairs, which were complete before that kernel began, and neither
    // reads what the other writes.  Two short kernels of few CTAs side by side: 8 heads x 256 tokens, r = 8,
    // whole prompt pass 239.7 -> 229.0 us.
    if (s->lowrank_r > 0) {
        const double *vals = s->eigval, *vecs = s->eigvec;
        const int rc = squat_launch(assemble_kernel, s->n_kv_heads, ASM_THREADS, smem, st, vals, vecs, rank_r, lambda, block_g, s->Wt, left_rows);
        if (rc != SQUAT_OK) return rc;
    } else {
        assemble_kernel<<<s->n_kv_heads, ASM_THREADS, smem, st>>>(s->eigval, s->eigvec, rank_r, lambda, block_g, s->Wt, left_rows);
        squat_count_launch();
        SQUAT_LAUNCH_CHECK();
    }
    return squat_launch_pack_update_matrices(s->Wt, s->Wimg, s->n_kv_heads, exact_channels, block_form, s->words, st);
}

// ------------------------------------------------------------------------- allocation-free Gram entry
// Scratch for squat_gram_static: the per-chunk partial Gram matrices live in this fixed array instead of
// memory obtained from cudaMalloc.  64 units of one d x d fp64 matrix = 8 MiB, held by every GPU that loads
// the library until the process exits.
namespace {
constexpr int GRAM_STATIC_MAX_UNITS = 64;            // n_kv_heads x row chunks
static __device__ __align__(256) double g_gram_static_scratch[(size_t)GRAM_STATIC_MAX_UNITS * D * D];
double *g_gram_static_ptr[64] = {nullptr};           // device address of the array, per device ordinal
}  // namespace

extern "C" int squat_gram_static(const void *q, int dtype, int n_q_heads, int n_kv_heads, int n_tokens,
                                 int head_dim, long long stride_h, long long stride_t, double *gram_out,
                                 void *stream)
{
    if (!q || !gram_out || (dtype != SQUAT_F32 && dtype != SQUAT_BF16)) return SQUAT_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(q) & 15u) || (reinterpret_cast<uintptr_t>(gram_out) & 15u)) return SQUAT_ERR_INVALID_ARG;
    if (n_q_heads <= 0 || n_kv_heads <= 0 || n_tokens <= 0) return SQUAT_ERR_INVALID_ARG;
    if (head_dim != D) return SQUAT_ERR_UNSUPPORTED;
    if (n_kv_heads > GRAM_STATIC_MAX_UNITS) return SQUAT_ERR_UNSUPPORTED;      // beyond the fixed scratch
    if (n_q_heads % n_kv_heads != 0) return SQUAT_ERR_SHAPE;
    const long long vec = dtype == SQUAT_BF16 ? 8 : 4;
    if (stride_t < D || stride_h < 0 || stride_t % vec || stride_h % vec) return SQUAT_ERR_INVALID_ARG;

    // set-up, once per device, with that device current: the array's name is only a host-side handle here;
    // kernels must be given the device address that cudaGetSymbolAddress reports
    int dev = 0;
    SQUAT_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return SQUAT_ERR_UNSUPPORTED;
    if (!g_gram_static_ptr[dev]) {
        double *ptr = nullptr;
        SQUAT_CUDA(cudaGetSymbolAddress((void **)&ptr, g_gram_static_scratch));
        g_gram_static_ptr[dev] = ptr;
    }
    double *partial = g_gram_static_ptr[dev];

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int H = n_kv_heads;
    // every element the reduction reads is written by this call's first kernel, so nothing left in the
    // array by an earlier call is ever seen and nothing needs clearing
    int chunks = 0;
    if (const int rc = squat_launch_gram_parts(q, dtype, H, n_tokens, n_q_heads / H, stride_h, stride_t, GRAM_STATIC_MAX_UNITS / H, nullptr, partial, &chunks, st)) return rc;
    gram_reduce_kernel<<<dim3(GRED_UNITS / GRED_THREADS, H), GRED_THREADS, 0, st>>>(partial, chunks, H, gram_out);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    return SQUAT_OK;
}

