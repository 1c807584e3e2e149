// Eigen-decomposition of the Gram matrices of step 1 (sigma_i^2 and v_i of the SVD of Algorithm 1 line 5), fp64.
//
//   tridiag_kernel   Householder reduction M = H T H^T, one CTA per head, the matrix in registers.
//   dc_kernel        divide and conquer on T (Cuppen's rank-one tearing, Gu and Eisenstat's recomputed weights), one
//                    cluster of 4 CTAs per head, then the reflectors applied to the eigenvectors of T.
//
// Both are bound by latency: the first by 126 dependent steps (a column norm, a matrix-vector product and two barriers
// each), the second by six dependent merges (a few secular-equation iterations each).  The flops of neither would fill a
// tenth of the time.  Measured on the 32 heads of a 4096-token prompt: 97 + 72 us.  What was here before, one-sided Jacobi
// on a Cholesky factor, needed 10 sweeps of 127 dependent rounds: 677 us.
#include <cooperative_groups.h>
#include <type_traits>
#include "device_helpers.cuh"

namespace {

namespace cg = cooperative_groups;
constexpr int D = SQUAT_D;



__device__ __forceinline__ double sqrt_nr(double x) { return x > 1e-290 ? x * rsqrt_nr(x) : 0.0; }

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    return v;
}


// ------------------------------------------------------------------------------------------------ tridiagonalisation
// Step k zeroes column k below the subdiagonal with the reflector I - u u^T / h (u_i = 0 for i <= k):
//     y = A u,  w = y / h - K u  with  K = u.y / (2 h^2),  A <- A - u w^T - w u^T.
// Warps 0-7 hold A, 4 rows x 16 columns a thread: rows 32 i + 4 warp + lane / 8, columns 16 m + 2 (lane % 8) + {0, 1}.
// Eight lanes share a row, so y needs three shuffle steps, and finished rows and columns drop out of the unrolled loops
// every 32 and 16 steps.  Warp 8 holds the vectors (index lane + 32 m) and runs the scalar chain: it forms row k of the
// current A itself from the row as it was before the last update, so the column norm and the new u are made while the
// other warps apply that update (rank two, twice the product's work).  Two barriers a step:
//     A  warp 8: w, row k, norm, new u   | others: w, rank-two update with the previous u, publish row k + 1
//     B  warp 8: 1 / h                   | others: y = A u and u.y
// Sums over a warp go through two fp64 tensor-core products with ones (77 cycles against 178 for five shuffle steps).
// Eight warps of 64 elements instead of sixteen of 32: what a step costs per warp (K, w, barriers) is most of the time.
constexpr int TRI_WARPS = 8;
constexpr int TRI_THREADS = 32 * (TRI_WARPS + 1);

__device__ __forceinline__ double warp_sum_mma(double v)
{
    double c0 = 0.0, c1 = 0.0;
    dmma(c0, c1, 1.0, v);                      // column sums of v seen as 4 x 8: lane (r, q) gets columns 2 q and 2 q + 1
    double t0 = 0.0, t1 = 0.0;
    dmma(t0, t1, c0 + c1, 1.0);                // the four q of every row added up
    return t0;
}

struct TriShared {
    double us[2][D], ys[D], rows[2][D], dots[TRI_WARPS], hinvs[2], mhs[2], red[TRI_WARPS];    // mhs: -1 / (2 h^2)
};

// registers of the chain warp: u (index lane + 32 m) and row k of the matrix before the last update, their elements k + 1,
// 1 / h, c1 = u_k / h, c3 = u_k / h^2
struct TriChain {
    double u[4], row[4], u1, row1, hinv, c1, c3, h, un1;
};

template <int KB>
__device__ __forceinline__ void tridiag_chain(TriShared &sm, TriChain &ch, double *dout, double *eout, double *hout, double *uout, int lane)
{
    constexpr int I0 = KB / 2;                 // first 32-row block that is not finished
#pragma unroll 1
    for (int k = 16 * KB; k < 16 * KB + 16; ++k) {
        double *un = sm.us[k & 1];
        const double2 p0 = *reinterpret_cast<const double2 *>(&sm.dots[0]), p1 = *reinterpret_cast<const double2 *>(&sm.dots[2]);
        const double2 p2 = *reinterpret_cast<const double2 *>(&sm.dots[4]), p3 = *reinterpret_cast<const double2 *>(&sm.dots[6]);
        // with w = y / h - K u:  x_i = row_i - u_i w_k - w_i u_k = (row_i - y_i u_k / h) - u_i (y_k / h - 2 K u_k)
        const double yk = sm.ys[k], y1 = sm.ys[(k + 1) & (D - 1)];
        double x[4], yi[4];
#pragma unroll
        for (int m = I0; m < 4; ++m) yi[m] = sm.ys[lane + 32 * m];
        const double sum = ((p0.x + p0.y) + (p1.x + p1.y)) + ((p2.x + p2.y) + (p3.x + p3.y));
        const double c2 = fma(ch.hinv, yk, -ch.c3 * sum);
        const double al = fma(-ch.u1, c2, fma(-y1, ch.c1, ch.row1));
        double s2[2] = {0.0, 0.0};
#pragma unroll
        for (int m = I0; m < 4; ++m) {
            const int i = lane + 32 * m;
            x[m] = fma(-ch.u[m], c2, fma(-yi[m], ch.c1, ch.row[m]));
            const double xm = i > k + 1 ? x[m] : 0.0;
            s2[m & 1] = fma(xm, xm, s2[m & 1]);
            if (i != k + 1) un[i] = xm;
            ch.u[m] = xm;
        }
        const double ss = warp_sum_mma(s2[0] + s2[1]);
        // a column that is tridiagonal already (or smaller than 1e-140) keeps h = infinity: its u has no effect
        const double n2 = fma(al, al, 1e-290) + ss;
        const double nrm = n2 * rsqrt_nr(n2);
        const double un1 = al + copysign(nrm, al);
        if (lane == ((k + 1) & 31)) un[(k + 1) & (D - 1)] = un1;
        const bool live = ss > 1e-280;
        ch.un1 = un1;
        ch.h = live ? nrm * (nrm + fabs(al)) : 0.0;
#pragma unroll
        for (int m = I0; m < 4; ++m) {
            const int i = lane + 32 * m;
            if (i == k) dout[k] = x[m];
            if (i == k + 1) ch.u[m] = un1;
        }
        if (lane == 0 && k < D - 1) eout[k] = live ? -copysign(nrm, al) : al;
        __syncthreads();
        ch.hinv = ch.h > 0.0 ? rcp_nr(ch.h) : 0.0;
        if (lane == 0) {
            sm.hinvs[k & 1] = ch.hinv;
            sm.mhs[k & 1] = -0.5 * ch.hinv * ch.hinv;
            hout[k] = ch.hinv;
        }
        // what the next step needs of this u and of the row the other warps have published
        const double *row = sm.rows[(k + 1) & 1];
        ch.c1 = ch.hinv * ch.un1;
        ch.c3 = ch.hinv * ch.c1;
        ch.u1 = un[(k + 2) & (D - 1)];
        ch.row1 = row[(k + 2) & (D - 1)];
#pragma unroll
        for (int m = I0; m < 4; ++m) {
            ch.row[m] = row[lane + 32 * m];
            uout[k * D + lane + 32 * m] = ch.u[m];
        }
        __syncthreads();
    }
}

template <int KB>
__device__ __forceinline__ void tridiag_work(TriShared &sm, double (&a)[4][16], int warp, int lane)
{
    const int rg = lane >> 3, r0 = 4 * warp + rg, cg2 = 2 * (lane & 7);
    constexpr int I0 = KB / 2;
#pragma unroll 1
    for (int k = 16 * KB; k < 16 * KB + 16; ++k) {
        const double *uo = sm.us[(k + 1) & 1], *un = sm.us[k & 1];
        const double2 p0 = *reinterpret_cast<const double2 *>(&sm.dots[0]), p1 = *reinterpret_cast<const double2 *>(&sm.dots[2]);
        const double2 p2 = *reinterpret_cast<const double2 *>(&sm.dots[4]), p3 = *reinterpret_cast<const double2 *>(&sm.dots[6]);
        const double hinv = sm.hinvs[(k + 1) & 1];
        const double sum = ((p0.x + p0.y) + (p1.x + p1.y)) + ((p2.x + p2.y) + (p3.x + p3.y));
        const double mk = sum * sm.mhs[(k + 1) & 1];              // -K of the previous step
        double wr[4], ur[4];
#pragma unroll
        for (int i = I0; i < 4; ++i) {
            ur[i] = uo[r0 + 32 * i];
            wr[i] = fma(hinv, sm.ys[r0 + 32 * i], mk * ur[i]);
        }
#pragma unroll
        for (int m = KB; m < 8; ++m) {
            const double2 u2 = *reinterpret_cast<const double2 *>(&uo[16 * m + cg2]);
            const double2 y2 = *reinterpret_cast<const double2 *>(&sm.ys[16 * m + cg2]);
            const double w0 = fma(hinv, y2.x, mk * u2.x), w1 = fma(hinv, y2.y, mk * u2.y);
#pragma unroll
            for (int i = I0; i < 4; ++i) {
                a[i][2 * m] = fma(-ur[i], w0, fma(-wr[i], u2.x, a[i][2 * m]));
                a[i][2 * m + 1] = fma(-ur[i], w1, fma(-wr[i], u2.y, a[i][2 * m + 1]));
            }
        }
        if (r0 == ((k + 1) & 31)) {                               // row k + 1 belongs to this thread's 32-row block (k + 1) / 32
            double *row = sm.rows[(k + 1) & 1];
            constexpr int I1 = (KB + 1) / 2 < 4 ? (KB + 1) / 2 : 3;
            const bool nextb = I1 != I0 && ((k + 1) & 15) == 0;
#pragma unroll
            for (int m = KB; m < 8; ++m)
                *reinterpret_cast<double2 *>(&row[16 * m + cg2]) =
                    nextb ? make_double2(a[I1][2 * m], a[I1][2 * m + 1]) : make_double2(a[I0][2 * m], a[I0][2 * m + 1]);
        }
        __syncthreads();
        double y[4], y1[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = y1[i] = 0.0;
#pragma unroll
        for (int m = KB; m < 8; ++m) {
            const double2 u2 = *reinterpret_cast<const double2 *>(&un[16 * m + cg2]);
#pragma unroll
            for (int i = I0; i < 4; ++i) {
                y[i] = fma(a[i][2 * m], u2.x, y[i]);
                y1[i] = fma(a[i][2 * m + 1], u2.y, y1[i]);
            }
        }
        double dt = 0.0;
#pragma unroll
        for (int i = I0; i < 4; ++i) {
            y[i] += y1[i];
            dt = fma(y[i], un[r0 + 32 * i], dt);
        }
        // four rows over eight lanes: lane bits 2 and 1 pick the row a lane finishes
        const bool b2 = lane & 4, b1 = lane & 2;
        double s0 = b2 ? y[0] : y[2], s1 = b2 ? y[1] : y[3];
        s0 = (b2 ? y[2] : y[0]) + __shfl_xor_sync(0xffffffffu, s0, 4);
        s1 = (b2 ? y[3] : y[1]) + __shfl_xor_sync(0xffffffffu, s1, 4);
        double t = b1 ? s0 : s1;
        t = (b1 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, t, 2);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        dt = warp_sum_mma(dt);
        const int r = r0 + 32 * ((lane >> 1) & 3 ? ((lane & 4) >> 1) + ((lane & 2) >> 1) : 0);
        if ((lane & 1) == 0) sm.ys[r] = r > k ? t : 0.0;          // finished rows are left alone
        if (lane == 0) sm.dots[warp] = dt;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(TRI_THREADS, 1) tridiag_kernel(
    const double *__restrict__ gram, double *__restrict__ tri /* [H, 3, D]: diagonal, subdiagonal, 1 / h */,
    double *__restrict__ refl /* [H, D, D]: row k = u of step k */, double *__restrict__ scale_out /* [H] */)
{
    __shared__ __align__(16) TriShared sm;
    const int h = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const double *M = gram + (long long)h * D * D;
    double *dout = tri + (long long)h * 3 * D, *eout = dout + D, *hout = dout + 2 * D;
    double *uout = refl + (long long)h * D * D;
    const int r0 = 4 * warp + (lane >> 3), cg2 = 2 * (lane & 7);

    double a[4][16];
    if (warp < TRI_WARPS) {
        double tr = 0.0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const double2 v = *reinterpret_cast<const double2 *>(M + (r0 + 32 * i) * D + 16 * m + cg2);
                a[i][2 * m] = v.x;
                a[i][2 * m + 1] = v.y;
                if (r0 + 32 * i == 16 * m + cg2) tr += v.x;
                if (r0 + 32 * i == 16 * m + cg2 + 1) tr += v.y;
            }
        tr = warp_sum(tr);
        if (lane == 0) { sm.red[warp] = tr; sm.dots[warp] = 0.0; }
    }
    if (tid < D) { sm.us[0][tid] = sm.us[1][tid] = 0.0; sm.ys[tid] = 0.0; }
    for (int i = tid; i < D * D; i += TRI_THREADS)                    // what the steps below leave out of the reflectors' rows
        if (i % D < i / D / 32 * 32) uout[i] = 0.0;
    if (tid == 0) sm.hinvs[1] = sm.mhs[1] = 0.0;
    __syncthreads();
    double trace = 0.0;
#pragma unroll
    for (int w = 0; w < TRI_WARPS; ++w) trace += sm.red[w];
    // a power of two near 1 / trace keeps every square and product below in range, whatever the queries' scale
    const int ebits = (int)((__double_as_longlong(trace) >> 52) & 0x7ff);
    const bool plain = !(trace > 0.0) || ebits == 0x7ff;              // zero or non-finite: nothing to scale
    const double scale = plain ? 1.0 : __longlong_as_double((long long)(2046 - (ebits < 1 ? 1 : ebits)) << 52);
    if (tid == 0) scale_out[h] = plain ? 1.0 : __longlong_as_double((long long)(ebits < 1 ? 1 : ebits) << 52);   // 1 / scale
    if (warp < TRI_WARPS) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 16; ++j) a[i][j] *= scale;
        if (r0 == 0) {
#pragma unroll
            for (int m = 0; m < 8; ++m) *reinterpret_cast<double2 *>(&sm.rows[0][16 * m + cg2]) = make_double2(a[0][2 * m], a[0][2 * m + 1]);
        }
    }
    __syncthreads();
    // the two roles meet at the same number of barriers
    if (warp == TRI_WARPS) {
        TriChain ch = {};
#pragma unroll
        for (int m = 0; m < 4; ++m) ch.row[m] = sm.rows[0][lane + 32 * m];
        ch.row1 = sm.rows[0][1];
        tridiag_chain<0>(sm, ch, dout, eout, hout, uout, lane);
        tridiag_chain<1>(sm, ch, dout, eout, hout, uout, lane);
        tridiag_chain<2>(sm, ch, dout, eout, hout, uout, lane);
        tridiag_chain<3>(sm, ch, dout, eout, hout, uout, lane);
        tridiag_chain<4>(sm, ch, dout, eout, hout, uout, lane);
        tridiag_chain<5>(sm, ch, dout, eout, hout, uout, lane);
        tridiag_chain<6>(sm, ch, dout, eout, hout, uout, lane);
        tridiag_chain<7>(sm, ch, dout, eout, hout, uout, lane);
    } else {
        tridiag_work<0>(sm, a, warp, lane);
        tridiag_work<1>(sm, a, warp, lane);
        tridiag_work<2>(sm, a, warp, lane);
        tridiag_work<3>(sm, a, warp, lane);
        tridiag_work<4>(sm, a, warp, lane);
        tridiag_work<5>(sm, a, warp, lane);
        tridiag_work<6>(sm, a, warp, lane);
        tridiag_work<7>(sm, a, warp, lane);
    }
}

// ------------------------------------------------------------------------------------------------ divide and conquer
// T is torn at every second off-diagonal element e: with rho = |e| the two halves lose rho at their touching corners and
// T = diag(T1, T2) + rho v v^T, so with the halves' eigen-pairs (d, Q) a merge is the eigenproblem of D + rho z z^T, z =
// Q^T v (last row of Q1, first row of Q2).  Its eigenvalues are the roots of 1/rho + sum z_j^2 / (d_j - lambda), one
// between any two neighbouring d.  A root is kept as (nearest pole K, offset mu), so that d_j - lambda_i = (d_j - d_K) -
// mu_i keeps its relative accuracy; the weights z are then recomputed from the roots (Gu and Eisenstat), for which the
// computed roots are exact, and the vectors z_j / (d_j - lambda_i) come out orthogonal to working precision.
// Nothing is deflated: neighbouring d are pushed at least DC_SEP apart (a few units in the last place of ||T||) and |z| is
// kept above DC_ZMIN instead, so the work does not depend on the data.  The pushes are backward errors; they add up over the
// copies of a multiple eigenvalue and over the merges, to at most (1 + 3 + 7 + .. + 127) DC_SEP = 2.2e-13 of ||T|| (measured on
// a multiple of the identity: 1.5e-13; on simple spectra eigenvalues and residuals are within 2.4e-15).
//
// Four CTAs work on a head.  Each solves a 32 x 32 diagonal block alone (rotations to 2, merges to 4, 8, .. 32), two share a merge to 64
// and four the one to 128; a CTA always owns 32 roots, eight lanes each, and the 32 eigenvectors that belong to them.
// What the next merge needs (eigenvalues, eigenvectors, roots) is written straight into the peers' shared memory.
// Warps 8-15 meanwhile make the triangular factors of the blocked reflectors and then help to apply them.
constexpr int DC_CTAS = 4;
constexpr int DC_THREADS = 512;
constexpr int DC_WORK = 256;                   // threads of the merges
constexpr int DC_LD = 36;                      // row stride of 32-column matrices: 4 mod 16, DMMA fragments without conflicts
constexpr int DC_LDQ = 68;                     // row stride of 64-column matrices, likewise
constexpr int DC_LDU = 132;                    // row stride of staged reflectors, likewise
constexpr double DC_SEP = 8.8817841970012523e-16;     // 2^-50
constexpr double DC_ZMIN = 5.5511151231257827e-17;    // 2^-54
constexpr double DC_RHOMIN = 2.2204460492503131e-16;  // 2^-52
constexpr double DC_EPS = 1.1102230246251565e-16;     // 2^-53
constexpr int DC_MAX_ITER = 60;

struct DcShared {
    double q32[2][32 * DC_LD];                 // this CTA's block, old and new
    double qa[2 * 32 * DC_LD];                 // the two children of the merge to 64
    union {
        double qb[2 * 64 * DC_LDQ];            // the two children of the merge to 128
        double u[2][16 * DC_LDU];              // afterwards: reflectors of one block, double-buffered
    };
    double s[D * DC_LD];                       // vectors of D + rho z z^T, rows in the children's column order
    double x[D * DC_LD];                       // eigenvectors: of T, then of M
    double t[8][16 * 17];                      // triangular factors of the eight blocks
    double y[2][16 * DC_LD], z[16 * DC_LD];
    double d32[2][32], da[64], db[D];          // children's eigenvalues per merge size
    double mu32[32], mua[64], mub[D];          // roots
    double dsort[D], ds[D], zs[D], zh[D], norm[32];
    double e[D], hinv[D];
    int k32[32], ka[64], kb[D];
    int perm[D];
    double wmax[16];
    int iters[8];
};

static_assert(sizeof(DcShared) <= 227 * 1024, "one CTA's shared memory");

__device__ __forceinline__ void work_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// One root of 1/rho + sum_j z_j^2 / (d_j - lambda) in (d_i, d_{i+1}) (beyond d_{n-1}: up to rho |z|^2), by eight lanes.
// Start: the two nearest poles kept exactly, the rest frozen at the middle of the interval.  Then the "middle way" of
// R.-C. Li ("Solving secular equations stably and efficiently", 1993), from which this start is taken too: both
// sums replaced by one pole each that matches value and slope, whose root is a quadratic's; a step that leaves the bracket
// or (every fifth) one that has not paid is replaced by a bisection, geometric where the bracket spans orders of magnitude.
template <int N>
__device__ __forceinline__ void secular_root(const double *ds, const double *zs, double rho, int i, int sub, double &mu_out, int &k_out, int &iters)
{
    constexpr int TERMS = (N + 7) / 8;
    double dl[TERMS], z[TERMS];
    const double rinv = 1.0 / rho;
    const bool last = i == N - 1;
    double z2 = 0.0;
#pragma unroll
    for (int t = 0; t < TERMS; ++t) {
        const int j = sub + 8 * t;
        const bool in = N >= 8 || j < N;
        dl[t] = in ? ds[j] - ds[i] : 1.0;
        z[t] = in ? zs[j] : 0.0;
        z2 = fma(z[t], z[t], z2);
    }
#pragma unroll
    for (int m = 4; m >= 1; m >>= 1) z2 += __shfl_xor_sync(0xffffffffu, z2, m);
    const double gap = last ? rho * z2 : ds[last ? i : i + 1] - ds[i];
    const double zi2 = zs[i] * zs[i], zr = last ? 0.0 : zs[last ? i : i + 1] * zs[last ? i : i + 1];
    double psi, phi, dpsi, dphi;
    auto eval = [&](double mu) {
        psi = phi = dpsi = dphi = 0.0;
#pragma unroll
        for (int t = 0; t < TERMS; ++t) {
            const double q = z[t] * rcp_nr(dl[t] - mu);
            if (sub + 8 * t <= i) { psi = fma(z[t], q, psi); dpsi = fma(q, q, dpsi); }
            else { phi = fma(z[t], q, phi); dphi = fma(q, q, dphi); }
        }
#pragma unroll
        for (int m = 4; m >= 1; m >>= 1) {
            psi += __shfl_xor_sync(0xffffffffu, psi, m);
            phi += __shfl_xor_sync(0xffffffffu, phi, m);
            dpsi += __shfl_xor_sync(0xffffffffu, dpsi, m);
            dphi += __shfl_xor_sync(0xffffffffu, dphi, m);
        }
    };
    const double mid = 0.5 * gap;
    eval(mid);
    const double f = rinv + psi + phi;
    const bool right = !last && f < 0.0;
    const int k = right ? i + 1 : i;
    double lo = right ? -mid : (last && f < 0.0 ? mid : 0.0), hi = right ? 0.0 : (last && f < 0.0 ? gap : mid);
    double mu;
    {
        const double rmid = rcp_nr(mid);
        const double c = f + zi2 * rmid - zr * rmid;                  // the poles' terms at the middle taken out
        if (last) mu = zi2 * rcp_nr(c);
        else {
            const double sg = right ? -1.0 : 1.0;
            const double a = fma(c, gap, sg * (zi2 + zr)), b = (right ? zr : zi2) * gap;
            const double r = sqrt_nr(fabs(fma(a, a, -sg * 4.0 * b * c)));
            // left: a > 0 ? 2b / (a + r) : (a - r) / 2c;   right: a < 0 ? 2b / (a - r) : -(a + r) / 2c
            const bool first = right ? a < 0.0 : a > 0.0;
            const double num = first ? 2.0 * b : sg * (a - sg * r), den = first ? a + sg * r : 2.0 * c;
            mu = num * rcp_nr(den);
        }
        if (!(mu > lo && mu < hi)) mu = 0.5 * (lo + hi);
    }
    const double dli = right ? ds[i] - ds[i + 1] : 0.0, dlr = right ? 0.0 : gap;
    if (right) {
#pragma unroll
        for (int t = 0; t < TERMS; ++t) {
            const int j = sub + 8 * t;
            if (N >= 8 || j < N) dl[t] = ds[j] - ds[i + 1];
        }
    }
    bool done = false;
    double pw = 1e300;
    int it = 0;
    for (; it < DC_MAX_ITER; ++it) {
        eval(mu);
        const double w = rinv + psi + phi;
        if (!done) {
            if (w < 0.0) lo = mu;
            else hi = mu;
        }
        const double alo = fmin(fabs(lo), fabs(hi)), ahi = fmax(fabs(lo), fabs(hi));
        done = done || fabs(w) <= 8.0 * DC_EPS * (rinv + phi - psi) || hi - lo <= 4.0 * DC_EPS * alo || !(w == w);
        if (__all_sync(0xffffffffu, done)) break;
        if (!done) {
            const double di = dli - mu, dr = dlr - mu;
            double num, den;
            if (last) {
                num = dpsi * di * di;
                den = fma(-dpsi, di, rinv + psi);
            } else {
                const double c = fma(-dr, dphi, fma(-di, dpsi, w));
                const double a = fma(di + dr, w, -di * dr * (dpsi + dphi)), b = di * dr * w;
                const double disc = sqrt_nr(fma(a, a, -4.0 * b * c));
                num = a <= 0.0 ? a - disc : 2.0 * b;
                den = a <= 0.0 ? 2.0 * c : a + disc;
            }
            double nw = mu + (last ? di : 0.0) + num * rcp_nr(den);     // a zero den: not a number, bisected
            if (!(nw > lo && nw < hi) || (it % 5 == 4 && fabs(w) > 0.1 * pw)) {
                const double g = sqrt_nr(fmax(alo, 1e-34 * ahi) * ahi);
                nw = ahi > 8.0 * alo ? (right ? -g : g) : 0.5 * (lo + hi);
            }
            pw = fabs(w);
            mu = nw;
        }
    }
    mu_out = mu;
    k_out = k;
    iters = it;
}

// The steps of a merge to N that are the same in every form.  din: the children's eigenvalues (problem by problem, N
// entries each), TOTAL = max(32, N) of them in this CTA.  last_row / first_row(col): the z vector's source.
template <int N>
__device__ __forceinline__ void dc_sort(DcShared &sm, const double *din, const double *q, int ldq, int child_rows, int tid, int e0)
{
    constexpr int TOTAL = N > 32 ? N : 32, M = N / 2;
    if (tid < TOTAL) {
        const int p = tid / N, l = tid % N, second = l >= M;
        const double dv = din[tid];
        const double *sib = din + p * N + (second ? 0 : M);
        int lo = 0, cnt = M;                   // how many of the sibling's (ascending) values come before this one
        while (cnt > 0) {
            const int half = cnt >> 1;
            const bool before = second ? sib[lo + half] <= dv : sib[lo + half] < dv;
            if (before) { lo += half + 1; cnt -= half + 1; }
            else cnt = half;
        }
        const int pos = p * N + (second ? l - M : l) + lo;
        // z: the last row of the first child's vectors, the first row of the second child's (times the sign of e)
        double z;
        if (N <= 32) z = q[(p * N + (second ? M : M - 1)) * ldq + tid];
        else z = second ? q[child_rows * ldq + (l - M)] : q[(M - 1) * ldq + l];
        if (second && sm.e[e0 + p * N + M - 1] < 0.0) z = -z;
        if (!(fabs(z) >= DC_ZMIN)) z = z < 0.0 ? -DC_ZMIN : DC_ZMIN;
        sm.dsort[pos] = dv;
        sm.zs[pos] = z;
        sm.perm[pos] = tid;
    }
    work_sync();
    if (tid < 32) {                            // separation: running maximum of d_l - l DC_SEP within each problem
        constexpr int EPL = TOTAL / 32;
        double v[EPL];
        double run = -1e300;
#pragma unroll
        for (int c = 0; c < EPL; ++c) {
            const int id = tid * EPL + c;
            v[c] = fmax(run, fma(-(double)(id % N), DC_SEP, sm.dsort[id]));
            run = v[c];
        }
        constexpr int W = N > 32 ? 32 : N;     // lanes per problem
#pragma unroll
        for (int o = 1; o < W; o <<= 1) {
            const double up = __shfl_up_sync(0xffffffffu, run, o, W);
            if ((tid & (W - 1)) >= o) run = fmax(run, up);
        }
        double before = __shfl_up_sync(0xffffffffu, run, 1, W);
        if ((tid & (W - 1)) == 0) before = -1e300;
#pragma unroll
        for (int c = 0; c < EPL; ++c) {
            const int id = tid * EPL + c;
            sm.ds[id] = fma((double)(id % N), DC_SEP, fmax(v[c], before));
        }
    }
    work_sync();
}

// weights recomputed from the roots: z_j^2 = (lambda_{n-1} - d_j) prod_{i<j} (lambda_i - d_j) / (d_i - d_j)
// prod_{j<=i<n-1} (lambda_i - d_j) / (d_{i+1} - d_j), up to a common factor
template <int N>
__device__ __forceinline__ void dc_weights(DcShared &sm, const double *mu, const int *kk, int tid)
{
    constexpr int TOTAL = N > 32 ? N : 32, TPJ = DC_WORK / TOTAL;
    const int g = tid / TPJ, sub = tid % TPJ, base = g / N * N, j = g % N;
    const double dj = sm.ds[g];
    double prod = 1.0;
    constexpr int CNT = (N + TPJ - 1) / TPJ;
    constexpr int STEP = CNT < 4 ? CNT : 4;
#pragma unroll 1
    for (int c0 = 0; c0 < CNT; c0 += STEP) {
        double num = 1.0, den = 1.0;
#pragma unroll
        for (int c = 0; c < STEP; ++c) {
            const int i = sub + TPJ * (c0 + c);
            if (i < N) {
                num *= (sm.ds[base + kk[base + i]] - dj) + mu[base + i];
                if (i < N - 1) den *= sm.ds[base + (i < j ? i : i + 1)] - dj;
            }
        }
        prod *= num * rcp_nr(den);
    }
#pragma unroll
    for (int m = TPJ / 2; m >= 1; m >>= 1) prod *= __shfl_xor_sync(0xffffffffu, prod, m);
    if (sub == 0) sm.zh[g] = copysign(sqrt_nr(fabs(prod)), sm.zs[g]);
}

// unnormalised vectors of this CTA's 32 roots into s (rows in the children's column order) and the norms' reciprocals
template <int N>
__device__ __forceinline__ void dc_vectors(DcShared &sm, const double *mu, const int *kk, int i0, int tid)
{
    const int slot = tid >> 3, sub = tid & 7;
    const int base = N > 32 ? 0 : slot / N * N, i = N > 32 ? i0 + slot : slot;
    const double dk = sm.ds[base + kk[i]], m = mu[i];
    double ss = 0.0;
#pragma unroll
    for (int t = 0; t < (N + 7) / 8; ++t) {
        const int j = sub + 8 * t;
        if (N >= 8 || j < N) {
            const double v = sm.zh[base + j] * rcp_nr((sm.ds[base + j] - dk) - m);
            ss = fma(v, v, ss);
            sm.s[sm.perm[base + j] * DC_LD + slot] = v;
        }
    }
#pragma unroll
    for (int o = 4; o >= 1; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (sub == 0) sm.norm[slot] = rsqrt_nr(ss);
}

// a merge inside the CTA's 32 x 32 block (32 / N problems)
template <int N>
__device__ __forceinline__ void dc_merge_local(DcShared &sm, int &buf, int blk, int tid, int &most)
{
    constexpr int M = N / 2;
    const double *q = sm.q32[buf];
    double *qn = sm.q32[buf ^ 1];
    dc_sort<N>(sm, sm.d32[buf], q, DC_LD, 0, tid, 32 * blk);
    {
        const int slot = tid >> 3, base = slot / N * N;
        double mu;
        int k, it;
        const double rho = fmax(fabs(sm.e[32 * blk + base + M - 1]), DC_RHOMIN);
        secular_root<N>(sm.ds + base, sm.zs + base, rho, slot - base, tid & 7, mu, k, it);
        most = max(most, it);
        if ((tid & 7) == 0) {
            sm.mu32[slot] = mu;
            sm.k32[slot] = k;
            sm.d32[buf ^ 1][slot] = sm.ds[base + k] + mu;
        }
    }
    work_sync();
    dc_weights<N>(sm, sm.mu32, sm.k32, tid);
    work_sync();
    dc_vectors<N>(sm, sm.mu32, sm.k32, 0, tid);
    work_sync();
    if constexpr (N >= 16) {                   // 8 x 8 tiles on the problems' diagonal blocks, two a warp at most
        const int warp = tid >> 5, lane = tid & 31;
        constexpr int PER_ROW = N / 8, TILES = 4 * PER_ROW;
#pragma unroll
        for (int u = warp; u < TILES; u += DC_WORK / 32) {
            const int ti = u / PER_ROW, tj = ti / PER_ROW * PER_ROW + u % PER_ROW;       // tile row and column in the 32 x 32 block
            const int k0 = 8 * ti / M * M;     // the columns of the child that the row belongs to
            double acc[2] = {0.0, 0.0};
#pragma unroll
            for (int kx = 0; kx < M; kx += 4)
                dmma(acc[0], acc[1], q[(8 * ti + (lane >> 2)) * DC_LD + k0 + kx + (lane & 3)], sm.s[(k0 + kx + (lane & 3)) * DC_LD + 8 * tj + (lane >> 2)]);
            const int r = 8 * ti + (lane >> 2), c = 8 * tj + 2 * (lane & 3);
            *reinterpret_cast<double2 *>(&qn[r * DC_LD + c]) = make_double2(acc[0] * sm.norm[c], acc[1] * sm.norm[c + 1]);
        }
    } else {
        const int c = tid & 31, p = c / N * N;
        const double nv = sm.norm[c];
#pragma unroll
        for (int rr = tid >> 5; rr < N; rr += DC_WORK / 32) {
            const int k0 = p + (rr >= M ? M : 0);
            double acc = 0.0;
#pragma unroll
            for (int kx = 0; kx < M; ++kx) acc = fma(q[(p + rr) * DC_LD + k0 + kx], sm.s[(k0 + kx) * DC_LD + c], acc);
            qn[(p + rr) * DC_LD + c] = acc * nv;
        }
    }
    work_sync();
    buf ^= 1;
}

// rows x 32 product: out[r][c] = norm[c] sum_k q[r][k] s[k0(r) + k][c]; rows of the first child take s rows 0 .. M-1, of
// the second M .. 2M-1.  One warp: 16 rows (N = 128) or 8 rows (N = 64).
template <int N, class Store>
__device__ __forceinline__ void dc_product(DcShared &sm, const double *q, int ldq, int warp, int lane, Store store)
{
    constexpr int M = N / 2, RT = N / 64;      // 8-row tiles per warp
    double acc[RT][4][2];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[i][n][0] = acc[i][n][1] = 0.0;
    const int r0 = warp * 8 * RT, k0 = r0 >= M ? M : 0;
    const double *qa = q + (r0 + (lane >> 2)) * ldq + (lane & 3);
    const double *sb = sm.s + (k0 + (lane & 3)) * DC_LD + (lane >> 2);
#pragma unroll 4
    for (int kx = 0; kx < M; kx += 4) {
        double a[RT], b[4];
#pragma unroll
        for (int i = 0; i < RT; ++i) a[i] = qa[i * 8 * ldq + kx];
#pragma unroll
        for (int n = 0; n < 4; ++n) b[n] = sb[kx * DC_LD + 8 * n];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int n = 0; n < 4; ++n) dmma(acc[i][n][0], acc[i][n][1], a[i], b[n]);
    }
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int r = r0 + 8 * i + (lane >> 2), c = 8 * n + 2 * (lane & 3);
            store(r, c, acc[i][n][0] * sm.norm[c], acc[i][n][1] * sm.norm[c + 1]);
        }
}

// Triangular factor of reflector block b (16 reflectors, H_{k0} .. H_{k0+15} = I - U^T T U with the rows of U the
// reflectors): T_ii = 1/h_i, T[a][i] = -T_ii sum_{a <= c < i} T[a][c] (u_c . u_i).  One warp per block.
__device__ __forceinline__ void wy_factor(DcShared &sm, const double *refl, int b, int lane)
{
    double acc[3][2] = {};                     // tiles (0,0), (0,1), (1,1) of the 16 x 16 Gram matrix
    const double *u0 = refl + (16 * b + (lane >> 2)) * D + (lane & 3), *u1 = u0 + 8 * D;
#pragma unroll 8
    for (int i = 16 * b; i < D; i += 4) {      // u_k is zero up to index k
        const double x = u0[i], y = u1[i];
        dmma(acc[0][0], acc[0][1], x, x);
        dmma(acc[1][0], acc[1][1], x, y);
        dmma(acc[2][0], acc[2][1], y, y);
    }
    double *t = sm.t[b];
    const int r = lane >> 2, c = 2 * (lane & 3);
#pragma unroll
    for (int e = 0; e < 2; ++e) {              // the Gram matrix, transposed into the lower triangle: t[i][c] = u_c . u_i
        t[(c + e) * 17 + r] = acc[0][e];
        t[(8 + c + e) * 17 + r] = acc[1][e];
        t[(8 + c + e) * 17 + 8 + r] = acc[2][e];
    }
    __syncwarp();
    double row[16];                            // lane a < 16 makes row a of T
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const double hi = sm.hinv[16 * b + i];
        double s = 0.0;
#pragma unroll
        for (int cc = 0; cc < i; ++cc) s = fma(row[cc], t[i * 17 + cc], s);
        row[i] = lane == i ? hi : (lane < i ? -hi * s : 0.0);
    }
    __syncwarp();
    if (lane < 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) t[lane * 17 + i] = row[i];
    }
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

__global__ void __cluster_dims__(DC_CTAS, 1, 1) __launch_bounds__(DC_THREADS, 1) dc_kernel(
    const double *__restrict__ tri, const double *__restrict__ refl_all, const double *__restrict__ scale_in,
    double *__restrict__ eigval, double *__restrict__ eigvec, int *__restrict__ iters_out, unsigned *__restrict__ status)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DcShared &sm = *reinterpret_cast<DcShared *>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int h = blockIdx.x / DC_CTAS, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const double *refl = refl_all + (long long)h * D * D;
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");     // waited for before the first store to a peer

    // T scaled by a power of two to a largest element in [1/2, 1): the separations above are relative to it
    double dv = 0.0;
    if (tid < D) {
        const double *t = tri + (long long)h * 3 * D;
        dv = t[tid];
        const double ev = tid < D - 1 ? t[D + tid] : 0.0;
        sm.e[tid] = ev;
        sm.hinv[tid] = t[2 * D + tid];
        sm.perm[tid] = tid & 31;
        double m = fmax(fabs(dv), fabs(ev));
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) sm.wmax[warp] = m;
    }
    __syncthreads();
    const double tmax = fmax(fmax(sm.wmax[0], sm.wmax[1]), fmax(sm.wmax[2], sm.wmax[3]));
    const int ebits = (int)((__double_as_longlong(tmax) >> 52) & 0x7ff);
    const bool zero = !(tmax > 1e-290);
    const double sc = zero ? 0.0 : __longlong_as_double((long long)(2045 - ebits) << 52);
    const double back = zero ? 0.0 : scale_in[h] * __longlong_as_double((long long)(ebits + 1) << 52);
    __syncthreads();
    if (tid < D) sm.e[tid] *= sc;
    __syncthreads();
    if (tid >= 32 * rank && tid < 32 * rank + 32) {
        double v = dv * sc;
        if (tid > 0) v -= fmax(fabs(sm.e[tid - 1]), DC_RHOMIN);
        if (tid < D - 1) v -= fmax(fabs(sm.e[tid]), DC_RHOMIN);
        sm.d32[0][tid & 31] = v;
    }
    for (int i = tid; i < 32 * DC_LD; i += DC_THREADS) sm.q32[0][i] = 0.0;
    __syncthreads();
    if (tid < 16) {                            // the 2 x 2 diagonal blocks by one rotation each
        const int i = 2 * tid;
        const double a = sm.d32[0][i], c = sm.d32[0][i + 1], e = sm.e[32 * rank + i];
        // the corners between the two were not torn: a and c have lost |e| in vain
        const double add = fmax(fabs(e), DC_RHOMIN), a1 = a + add, c1 = c + add;
        const double half = 0.5 * (c1 - a1), r = sqrt_nr(fma(half, half, e * e));
        const double den = fabs(half) + r, tn = den > 1e-290 ? (half >= 0.0 ? e : -e) * rcp_nr(den) : 0.0;   // tan of the angle, at most 1
        const double cs = rsqrt_nr(fma(tn, tn, 1.0)), sn = tn * cs;
        const double lo = fma(-tn, e, a1), hi = fma(tn, e, c1);       // of (cs, -sn) and (sn, cs)
        const bool swap = lo > hi;
        sm.d32[0][i] = swap ? hi : lo;
        sm.d32[0][i + 1] = swap ? lo : hi;
        const double v0[2] = {cs, sn}, v1[2] = {-sn, cs};             // rows of the matrix whose columns are the vectors
        sm.q32[0][i * DC_LD + i] = v0[swap];
        sm.q32[0][i * DC_LD + i + 1] = v0[!swap];
        sm.q32[0][(i + 1) * DC_LD + i] = v1[swap];
        sm.q32[0][(i + 1) * DC_LD + i + 1] = v1[!swap];
    }
    __syncthreads();

    int most = 0;
    if (warp < DC_WORK / 32) {
        int buf = 0;
        dc_merge_local<4>(sm, buf, rank, tid, most);
        dc_merge_local<8>(sm, buf, rank, tid, most);
        dc_merge_local<16>(sm, buf, rank, tid, most);
        dc_merge_local<32>(sm, buf, rank, tid, most);
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        // the block's eigen-pairs to this CTA and its partner: child rank & 1 of the merge to 64
#pragma unroll
        for (int to = 0; to < 2; ++to) {
            double *qd = cluster.map_shared_rank(sm.qa, (rank & 2) + to) + (rank & 1) * 32 * DC_LD;
            double *dd = cluster.map_shared_rank(sm.da, (rank & 2) + to) + (rank & 1) * 32;
            for (int i = tid; i < 32 * 32; i += DC_WORK) qd[i / 32 * DC_LD + i % 32] = sm.q32[buf][i / 32 * DC_LD + i % 32];
            if (tid < 32) dd[tid] = sm.d32[buf][tid];
        }
        cluster.sync();

        const int slot = tid >> 3, sub = tid & 7, half = rank & 1, pair = rank >> 1;
        {
            dc_sort<64>(sm, sm.da, sm.qa, DC_LD, 32, tid, 64 * pair);
            double mu;
            int k, it;
            const double rho = fmax(fabs(sm.e[64 * pair + 31]), DC_RHOMIN);
            secular_root<64>(sm.ds, sm.zs, rho, 32 * half + slot, sub, mu, k, it);
            most = max(most, it);
            if (sub < 2) {
                cluster.map_shared_rank(sm.mua, (rank & 2) + sub)[32 * half + slot] = mu;
                cluster.map_shared_rank(sm.ka, (rank & 2) + sub)[32 * half + slot] = k;
            }
        }
        cluster.sync();
        dc_weights<64>(sm, sm.mua, sm.ka, tid);
        work_sync();
        dc_vectors<64>(sm, sm.mua, sm.ka, 32 * half, tid);
        work_sync();
        {
            double *qd[DC_CTAS];
#pragma unroll
            for (int to = 0; to < DC_CTAS; ++to) qd[to] = cluster.map_shared_rank(sm.qb, to) + pair * 64 * DC_LDQ + 32 * half;
            dc_product<64>(sm, sm.qa, DC_LD, warp, lane, [&](int r, int c, double v0, double v1) {
#pragma unroll
                for (int to = 0; to < DC_CTAS; ++to) *reinterpret_cast<double2 *>(&qd[to][r * DC_LDQ + c]) = make_double2(v0, v1);
            });
            if (sub < DC_CTAS)
                cluster.map_shared_rank(sm.db, sub)[64 * pair + 32 * half + slot] = sm.ds[sm.ka[32 * half + slot]] + sm.mua[32 * half + slot];
        }
        cluster.sync();
        {
            dc_sort<128>(sm, sm.db, sm.qb, DC_LDQ, 64, tid, 0);
            double mu;
            int k, it;
            const double rho = fmax(fabs(sm.e[63]), DC_RHOMIN);
            secular_root<128>(sm.ds, sm.zs, rho, 32 * rank + slot, sub, mu, k, it);
            most = max(most, it);
            if (sub < DC_CTAS) {
                cluster.map_shared_rank(sm.mub, sub)[32 * rank + slot] = mu;
                cluster.map_shared_rank(sm.kb, sub)[32 * rank + slot] = k;
            }
        }
        cluster.sync();
        dc_weights<128>(sm, sm.mub, sm.kb, tid);
        work_sync();
        dc_vectors<128>(sm, sm.mub, sm.kb, 32 * rank, tid);
        work_sync();
        dc_product<128>(sm, sm.qb, DC_LDQ, warp, lane, [&](int r, int c, double v0, double v1) {
            *reinterpret_cast<double2 *>(&sm.x[r * DC_LD + c]) = make_double2(v0, v1);
        });
        if (lane == 0) sm.iters[warp] = most;
    } else {
        wy_factor(sm, refl, warp - DC_WORK / 32, lane);
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
#pragma unroll 1
        for (int i = 0; i < 4; ++i) cluster.sync();
    }

    // eigenvectors of M: the reflectors' blocks, last first, X <- X - U^T (T (U X))
    auto stage = [&](int b) {
        for (int i = tid; i < 16 * (D / 2); i += DC_THREADS)
            cp_async16(&sm.u[b & 1][i / (D / 2) * DC_LDU + i % (D / 2) * 2], refl + (16 * b + i / (D / 2)) * D + i % (D / 2) * 2);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    __syncthreads();                           // the merges are done with qb, which the reflectors now share
    stage(7);
#pragma unroll 1
    for (int b = 7; b >= 0; --b) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                       // block b is staged; X is up to date; the other buffer is free
        if (b > 0) stage(b - 1);
        const double *u = sm.u[b & 1];
        {   // Y = U X: 2 x 4 tiles, the rows 16 b .. 127 that U touches in two interleaved halves
            const int tile = warp & 7, half = warp >> 3, ti = tile >> 2, tj = tile & 3;
            double acc[4][2] = {};
            const double *ua = u + (8 * ti + (lane >> 2)) * DC_LDU + (lane & 3);
            const double *xb = sm.x + (lane & 3) * DC_LD + 8 * tj + (lane >> 2);
            for (int i = 16 * b + 8 * half; i < D; i += 32) {          // four products in flight
                const bool two = i + 16 < D;
                const double a0 = ua[i], b0 = xb[i * DC_LD], a1 = ua[i + 4], b1 = xb[(i + 4) * DC_LD];
                const double a2 = two ? ua[i + 16] : 0.0, b2 = two ? xb[(i + 16) * DC_LD] : 0.0;
                const double a3 = two ? ua[i + 20] : 0.0, b3 = two ? xb[(i + 20) * DC_LD] : 0.0;
                dmma(acc[0][0], acc[0][1], a0, b0);
                dmma(acc[1][0], acc[1][1], a1, b1);
                dmma(acc[2][0], acc[2][1], a2, b2);
                dmma(acc[3][0], acc[3][1], a3, b3);
            }
            const int r = 8 * ti + (lane >> 2), c = 8 * tj + 2 * (lane & 3);
            *reinterpret_cast<double2 *>(&sm.y[half][r * DC_LD + c]) = make_double2((acc[0][0] + acc[1][0]) + (acc[2][0] + acc[3][0]), (acc[0][1] + acc[1][1]) + (acc[2][1] + acc[3][1]));
        }
        __syncthreads();
        if (warp < 8) {                        // Z = T Y
            const int ti = warp >> 2, tj = warp & 3;
            double acc[2][2] = {};
            const double *ta = sm.t[b] + (8 * ti + (lane >> 2)) * 17 + (lane & 3);
            const double *y0 = sm.y[0] + (lane & 3) * DC_LD + 8 * tj + (lane >> 2), *y1 = y0 + 16 * DC_LD;
#pragma unroll
            for (int kx = 0; kx < 16; kx += 4) dmma(acc[kx / 4 & 1][0], acc[kx / 4 & 1][1], ta[kx], y0[kx * DC_LD] + y1[kx * DC_LD]);
            const int r = 8 * ti + (lane >> 2), c = 8 * tj + 2 * (lane & 3);
            *reinterpret_cast<double2 *>(&sm.z[r * DC_LD + c]) = make_double2(-(acc[0][0] + acc[1][0]), -(acc[0][1] + acc[1][1]));
        }
        __syncthreads();
        {   // X += U^T (-Z): tile column warp % 4, tile rows 2 b + warp / 4, + 4, .. (four at most, in flight together)
            const int tj = warp & 3, c = 8 * tj + 2 * (lane & 3), rt0 = 2 * b + (warp >> 2);
            const double *zb = sm.z + (lane & 3) * DC_LD + 8 * tj + (lane >> 2);
            double z[4];
#pragma unroll
            for (int kx = 0; kx < 4; ++kx) z[kx] = zb[4 * kx * DC_LD];
            auto update = [&](auto count) {
                constexpr int NT = decltype(count)::value;
                double2 acc[NT];
#pragma unroll
                for (int n = 0; n < NT; ++n) acc[n] = *reinterpret_cast<const double2 *>(&sm.x[(8 * (rt0 + 4 * n) + (lane >> 2)) * DC_LD + c]);
#pragma unroll
                for (int kx = 0; kx < 4; ++kx)
#pragma unroll
                    for (int n = 0; n < NT; ++n) dmma(acc[n].x, acc[n].y, u[(4 * kx + (lane & 3)) * DC_LDU + 8 * (rt0 + 4 * n) + (lane >> 2)], z[kx]);
#pragma unroll
                for (int n = 0; n < NT; ++n) *reinterpret_cast<double2 *>(&sm.x[(8 * (rt0 + 4 * n) + (lane >> 2)) * DC_LD + c]) = acc[n];
            };
            switch ((19 - rt0) / 4) {          // warp-uniform
            case 4: update(std::integral_constant<int, 4>{}); break;
            case 3: update(std::integral_constant<int, 3>{}); break;
            case 2: update(std::integral_constant<int, 2>{}); break;
            case 1: update(std::integral_constant<int, 1>{}); break;
            default: break;
            }
        }
    }
    __syncthreads();
    // descending order: root 32 rank + c of the ascending list is eigen-pair 127 - that
    for (int i = tid; i < 32 * D; i += DC_THREADS) {
        const int c = i / D, r = i % D;
        eigvec[((long long)h * D + (D - 1 - 32 * rank - c)) * D + r] = sm.x[r * DC_LD + c];
    }
    if (tid < 32) {
        const double lam = (sm.ds[sm.kb[32 * rank + tid]] + sm.mub[32 * rank + tid]) * back;
        eigval[(long long)h * D + (D - 1 - 32 * rank - tid)] = lam > 0.0 ? lam : 0.0;
    }
    if (tid == 0 && rank == 0) {
        int m = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) m = max(m, sm.iters[w]);
        iters_out[h] = m;
        if (m >= DC_MAX_ITER) atomicOr(status, SQUAT_FLAG_NO_CONVERGE);
    }
}

}  // namespace

int squat_launch_eig(squat_subspace *s, cudaStream_t st)
{
    const int H = s->n_kv_heads;
    tridiag_kernel<<<H, TRI_THREADS, 0, st>>>(s->gram, s->tri, s->gram_partial, s->eig_scale);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    static std::atomic<unsigned long long> allowed{0};
    if (const int rc = squat_allow_smem(reinterpret_cast<const void *>(dc_kernel), sizeof(DcShared), allowed)) return rc;
    dc_kernel<<<H * DC_CTAS, DC_THREADS, sizeof(DcShared), st>>>(s->tri, s->gram_partial, s->eig_scale, s->eigval, s->eigvec,
                                                                 s->eig_sweeps, s->status);
    squat_count_launch();
    SQUAT_LAUNCH_CHECK();
    return SQUAT_OK;
}
