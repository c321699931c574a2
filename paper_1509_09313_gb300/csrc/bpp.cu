// Batched NLS by block principal pivoting (Eq. 3, Eq. 4, Sec. 4.2).
//
// Every right-hand side j solves  min_{x >= 0} 0.5 x^T G x - g_j^T x  with one
// shared k x k Gram G. BPP partitions the indices into a passive set F (free)
// and an active set (x_i = 0); for a partition the candidate is
//   x_F = G_FF^{-1} g_F, x_A = 0, y = G x - g (y_F = 0),
// and the exchange rules of the cited method (full exchange while the number
// of infeasible indices drops, three more full exchanges otherwise, then the
// backup single exchange of the largest infeasible index) move infeasible
// indices (x_i < 0 on F, y_i < 0 off F) across until Eq. 4 holds.
//
// GPU design (differs from the paper's column grouping; same result):
//  * bpp_prep_kernel (one CTA, or a cluster of eight where k is large and
//    nothing runs beside it; FP64) turns the usable part of G into M = G^{-1}
//    once per half-step by symmetric Gauss-Jordan sweeps in registers (indices
//    with G_ii <= 0 are never passive), and forms the condition number cond_1(S G S) = ||S G S||_1
//    ||S^-1 M S^-1||_1 of G with its diagonal scaled to one (S = diag(G)^-1/2),
//    and picks the arithmetic of the solves: FP32 when it is <= 1e4 (mode 0),
//    FP64 otherwise (mode 1), FP64 without M when G is numerically singular
//    (mode 2). The scaled number is the one that bounds the FP32 error: every
//    FP32 step here (rounding G and M, Cholesky, the matrix-vector products)
//    perturbs entry (i, j) relative to sqrt(G_ii G_jj), so a factor that is
//    merely badly scaled (one row of H much smaller than the rest, common in
//    early iterations) costs nothing.
//  * solve kernels: persistent, one warp per right-hand side, G and M in
//    shared memory. Lane l holds indices l, l+32, ... of g, x, y and of the
//    unconstrained solution u = M g. Each exchange round solves the smaller of
//    two equivalent systems:
//      direct      G_FF x_F = g_F                          (|F| x |F|)
//      complement  M_AA y_A = -u_A,  x_F = u_F + M_FA y_A  (|A| x |A|)
//    (the second follows from G x = g + y with y supported on A and x_A = 0),
//    by a warp-cooperative factorisation with shuffle-broadcast
//    substitutions. Cost per round O(min(|F|,|A|)^3 + k |F|) instead of
//    O(|F|^3). bpp_solve32_kernel (bpp32.cu) runs mode 0: it refines once
//    (residual g_F - G_FF x_F solved through the same factor: the explicit
//    inverse alone is not backward stable), recomputes y from G, and counts a
//    sign test as violated only beyond 2^-20 of the problem's scale in the
//    diagonally scaled variables (x_i sqrt(G_ii) against max over F of
//    |x_j| sqrt(G_jj); y_i / sqrt(G_ii) against max of |g_j| / sqrt(G_jj)):
//    values within FP32 noise of zero are degenerate ties that would
//    otherwise make the exchange rules cycle. The final x is clamped at 0
//    there. A system whose FP32 pivot falls below 1e-4 of its diagonal
//    defers its right-hand side to a second pass of bpp_solve_kernel in FP64.
//    bpp_solve_kernel (here) runs modes 1 and 2 in FP64 with the strict sign
//    test and no refinement.
//  * Every loop is bounded: a solve stops at max_rounds with status
//    NOT_CONVERGED; there are no spin-waits.
//
// Roofline: FP32 ALU for the pivoting; HBM traffic is nrhs * k * 8 bytes
// (right-hand sides in, solutions out) plus bitmasks.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <iterator>
#include <mutex>

#include "bpp_internal.cuh"

namespace nmf {
namespace {

using namespace bpp;

constexpr int BPP_WARPS = 8;               // most warps per CTA (launch bound)
constexpr int BPP_THREADS = BPP_WARPS * 32;

// Workspace layout (bytes, 256-aligned pieces).
struct WorkLayout {
    size_t g32, m32, m64, usable, flags, counters, defer, total;
};

WorkLayout layout(int k)
{
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    WorkLayout w;
    size_t off = 0;
    w.g32 = off; off += al(sizeof(float) * k * k);
    w.m32 = off; off += al(sizeof(float) * k * k);
    w.m64 = off; off += al(sizeof(double) * k * k);
    w.usable = off; off += al(sizeof(uint32_t) * 4);
    w.flags = off; off += al(sizeof(int) * 4);
    w.counters = off; off += al(sizeof(unsigned long long) * CNT_WORDS);
    w.defer = off; off += al(sizeof(int64_t) * DEFER_CAP);
    w.total = off;
    return w;
}

// Row of entry e of a lower triangle stored row by row (e = a (a + 1) / 2 + b,
// b <= a): the FP32 estimate of the root of a (a + 1) / 2 = e, corrected.
__device__ __forceinline__ int tri_row(int e)
{
    int a = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    while (a * (a + 1) / 2 > e)
        --a;
    while ((a + 1) * (a + 2) / 2 <= e)
        ++a;
    return a;
}

// ---------------------------------------------------------------------------
// Prep: M = G_UU^{-1} in FP64, the scaled cond_1, FP32 copies of G and M.
// flags[0] = mode (0 FP32, 1 FP64 with M, 2 FP64 without M), flags[1] = |U|.
//
// G_UU is inverted in place by Gauss-Jordan sweeps over its lower triangle:
// sweep p takes the Schur complement's pivot d = A_pp (the square of the
// Cholesky pivot, tested against the same floor), and sets A_ij -= A_ip A_pj /
// d, A_ip /= d, A_pp = -1 / d; after the last one A = -M. On positive definite
// matrices that is as accurate as the inverse through the factor (condition
// 30 to 4e10, k = 20 to 100, against extended precision: 1.6 to 4 times less
// error than M = L^{-T} L^{-1}), has the same k^3 / 2 multiply-adds, and one
// barrier per pivot: the threads keep the triangle in registers, four
// consecutive entries of a row each, and a pivot's column goes through shared
// memory (two buffers).
//
// Bound by FP64: a quarter of an SM takes one warp instruction in 63-76 cycles,
// one after the other, whatever its active lanes, and a division in 340. Warp 0
// therefore keeps the diagonal (lane l: entries l, l + 32, ...) and has the
// next pivot's reciprocal ready at the barrier, while the others update the
// triangle. Above k = PREP_ONE_K a cluster of C = 8 CTAs shares the triangle
// out and writes each pivot's column into every CTA's buffer, unless a product
// runs beside it, which fills the SMs a cluster would have to wait for (C = 1).
// Measured, k = 10, 20, 33, 50, 100: 11, 19, 28, 55 and (C = 8) 110 us, where an
// FP64 Cholesky with three more kernels for the inverse (k >= 48) took 19, 40,
// 75, 96 and 257.
// Pairs of floats in place of FP64 were as fast (36 us at k = 50, 131 at 100),
// but leave M's FP32 rounding to chance in one entry of 1e4 (condition 150).
// ---------------------------------------------------------------------------
constexpr int PREP_THREADS = 1024;
constexpr int PREP_ONE_K = 52;

// Segment s of the lower triangle (rows in order, row i in i / 4 + 1 segments
// of four columns): row i, first column j0.
__device__ __forceinline__ void prep_segment(int s, int &i, int &j0)
{
    int a = (int)((sqrtf(2.0f * (float)s + 1.0f) - 1.0f) * 0.5f);
    while (2 * a * (a + 1) > s)
        --a;
    while (2 * (a + 1) * (a + 2) <= s)
        ++a;
    const int rem = s - 2 * a * (a + 1);   // rows 4 a .. 4 a + 3 have a + 1 each
    i = 4 * a + rem / (a + 1);
    j0 = 4 * (rem % (a + 1));
}
__host__ __device__ inline int prep_segments(int u)
{
    const int a = u >> 2;
    return 2 * a * (a + 1) + (u & 3) * (a + 1);
}

// Thread t's part of sum_a |Ms_ac| w_a: column c = t mod 128, every (threads /
// 128)-th row.
__device__ __forceinline__ float prep_colsum(const float *__restrict__ Ms, int u,
                                             const float *__restrict__ w)
{
    const int c = threadIdx.x & 127, part = threadIdx.x >> 7, parts = blockDim.x >> 7;
    float s = 0.0f;
    if (c < u && part < parts)
        for (int a = part; a < u; a += parts)
            s = fmaf(fabsf(Ms[a * u + c]), w[a], s);
    return s;
}

template <int C, int NSEG>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(C == 1 ? PREP_THREADS : PREP_THREADS / 2)
    bpp_prep_kernel(const double *__restrict__ G, int k, float *__restrict__ G32,
                    float *__restrict__ M32, double *__restrict__ M64,
                    uint32_t *__restrict__ usable_words, int *__restrict__ flags,
                    unsigned long long *__restrict__ counters, BppStats *__restrict__ stats)
{
    constexpr int DS = NMF_MAX_K / 32;
    extern __shared__ float Ms[];                           // u x u, CTA 0: G, then M, in FP32
    __shared__ __align__(16) double col[2][NMF_MAX_K + 4];  // the pivot's column
    __shared__ double rpiv[2];                              // 1 / pivot; 0: below the floor
    __shared__ double floor_[NMF_MAX_K];                    // the pivots' floors
    __shared__ float dsq[NMF_MAX_K], rdsq[NMF_MAX_K];       // sqrt(G_aa) and its reciprocal
    __shared__ int uidx[NMF_MAX_K];
    __shared__ uint32_t words[4];
    __shared__ float red[2][PREP_THREADS];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int rank = C == 1 ? 0 : (int)blockIdx.x;
    namespace cg = cooperative_groups;
    auto sync = [&]() {
        if constexpr (C == 1)
            __syncthreads();
        else
            cg::this_cluster().sync();
    };
    auto at = [&](auto *ptr, int r) {
        if constexpr (C == 1)
            return ptr;
        else
            return cg::this_cluster().map_shared_rank(ptr, r);
    };

    // Usable indices (G_ii > 0), in order.
    double gii = 0.0;
    if (tid < NMF_MAX_K) {   // (at least 128 threads)
        gii = tid < k ? G[tid * (k + 1)] : 0.0;
        const uint32_t b = __ballot_sync(FULL, gii > 0.0);
        if (lane == 0)
            words[tid >> 5] = b;
    }
    for (int e = tid; e < 2 * (NMF_MAX_K + 4); e += nt)
        (&col[0][0])[e] = 0.0;
#pragma unroll 4
    for (int e = rank * nt + tid; e < k * k; e += C * nt)
        G32[e] = (float)G[e];
    __syncthreads();
    int u = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w)
        u += __popc(words[w]);
    if (gii > 0.0) {
        int a = __popc(words[tid >> 5] & lanemask_lt(lane));
        for (int w = 0; w < (tid >> 5); ++w)
            a += __popc(words[w]);
        uidx[a] = tid;
        floor_[a] = PIVOT_TOL64 * gii;
        const float d = sqrtf((float)gii);
        dsq[a] = d;
        rdsq[a] = 1.0f / d;
    }
    if (rank == 0) {
        if (tid < 4)
            usable_words[tid] = words[tid];
        if (tid < CNT_WORDS)
            counters[tid] = 0ull;
    }
    if (u < k)
        for (int e = rank * nt + tid; e < k * k; e += C * nt) {
            const int a = e / k, b = e - a * k;
            if (!((words[a >> 5] >> (a & 31)) & (words[b >> 5] >> (b & 31)) & 1u)) {
                M32[e] = 0.0f;
                M64[e] = 0.0;
            }
        }
    __syncthreads();

    int row[NSEG], j0[NSEG];
    double A[NSEG][4];
    const int nseg = prep_segments(u);
#pragma unroll
    for (int q = 0; q < NSEG; ++q) {
        const int sg = (q * (nt - 32) + tid - 32) * C + rank;
        row[q] = -1;
        j0[q] = 0;
        if (tid >= 32 && sg < nseg)
            prep_segment(sg, row[q], j0[q]);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            A[q][e] = j0[q] + e <= row[q] ? G[uidx[row[q]] * k + uidx[j0[q] + e]] : 0.0;
    }
    double diag[DS];
#pragma unroll
    for (int t = 0; t < DS; ++t) {
        const int i = lane + 32 * t;
        diag[t] = tid < 32 && i < u ? G[uidx[i] * (k + 1)] : 1.0;
    }
    if (C > 1)
        sync();   // every CTA's buffers are cleared
    // sign times the entries to both triangles of CTA 0's Ms.
    auto to_shared = [&](float sign) {
        float *dst = at(Ms, 0);
#pragma unroll
        for (int q = 0; q < NSEG; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = row[q], j = j0[q] + e;
                if (j <= i) {
                    const float v = sign * (float)A[q][e];
                    dst[i * u + j] = v;
                    dst[j * u + i] = v;
                }
            }
    };
    auto put = [&](double v, int i, int p) {   // entry i of pivot p's column
        for (int t = 0; t < C; ++t)
            *at(&col[p & 1][i], t) = v;
    };
    // A segment's entries of pivot p's column: row p itself, or column p.
    auto put_segment = [&](double a0, double a1, double a2, double a3, int i, int j, int p) {
        if (i == p) {
            put(a0, j, p);
            if (j + 1 <= p)
                put(a1, j + 1, p);
            if (j + 2 <= p)
                put(a2, j + 2, p);
            if (j + 3 <= p)
                put(a3, j + 3, p);
        } else if (i > p && j == (p & ~3)) {
            const int e = p & 3;
            put(e == 0 ? a0 : e == 1 ? a1 : e == 2 ? a2 : a3, i, p);
        }
    };
    to_shared(1.0f);
#pragma unroll
    for (int q = 0; q < NSEG; ++q)
        put_segment(A[q][0], A[q][1], A[q][2], A[q][3], row[q], j0[q], 0);
    if (tid == 0)
        rpiv[0] = diag[0] > floor_[0] ? 1.0 / diag[0] : 0.0;
    sync();
    const float sg = rank == 0 ? prep_colsum(Ms, u, rdsq) : 0.0f;
    bool ok = u > 0;
    for (int p = 0; p < u; ++p) {
        const double *c = col[p & 1];
        const double r = rpiv[p & 1];
        if (!(r > 0.0)) {
            ok = false;   // (the same in every thread)
            break;
        }
        const int np = p + 1;
        if (tid < 32) {
            // The diagonal, the next pivot's part first (entries already swept
            // carry values of no use).
            const int tn = np >> 5;
            double d = diag[0];
#pragma unroll
            for (int t = 1; t < DS; ++t)
                if (t == tn)
                    d = diag[t];
            const double cn = c[(lane + 32 * tn) & (NMF_MAX_K - 1)];
            d = fma(-(cn * r), cn, d);
            if (lane == (np & 31) && np < u) {
                const double rn = 1.0 / d;
                rpiv[np & 1] = d > floor_[np] ? rn : 0.0;
            }
#pragma unroll
            for (int t = 0; t < DS; ++t) {
                if (t == tn) {
                    diag[t] = d;
                } else if (t > tn && 32 * t < u) {
                    const double ct = c[lane + 32 * t];
                    diag[t] = fma(-(ct * r), ct, diag[t]);
                }
            }
        } else {
#pragma unroll
            for (int q = 0; q < NSEG; ++q) {
                if (row[q] < 0)
                    continue;
                // Row p itself becomes c r: the same products with -r for c_i r
                // and zero for A.
                const bool prow = row[q] == p;
                const double s = (prow ? -1.0 : c[row[q]]) * r;
                const double2 c01 = *reinterpret_cast<const double2 *>(c + j0[q]);
                const double2 c23 = *reinterpret_cast<const double2 *>(c + j0[q] + 2);
                const double cj[4] = {c01.x, c01.y, c23.x, c23.y};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const double v = fma(-s, cj[e], prow ? 0.0 : A[q][e]);
                    A[q][e] = j0[q] + e == p ? s : v;
                }
                put_segment(A[q][0], A[q][1], A[q][2], A[q][3], row[q], j0[q], np);
            }
        }
        sync();
    }
    if (!ok) {
        if (rank == 0 && tid == 0) {
            flags[0] = 2;
            flags[1] = u;
            atomicAdd(&stats->fp64_halfsteps, 1ull);
        }
        return;   // (the loop ended at a barrier all CTAs passed)
    }
    // M = -A to both triangles.
#pragma unroll
    for (int q = 0; q < NSEG; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i = row[q], j = j0[q] + e;
            if (j <= i) {
                const double m = -A[q][e];
                const int gi = uidx[i], gj = uidx[j];
                M64[gi * k + gj] = m;
                M64[gj * k + gi] = m;
                M32[gi * k + gj] = (float)m;
                M32[gj * k + gi] = (float)m;
            }
        }
    to_shared(-1.0f);
    sync();
    if (rank != 0)
        return;
    // cond_1 of the scaled matrix, max column sum of |G_ac| / (d_a d_c) times
    // max column sum of |M_ac| d_a d_c with d_a = sqrt(G_aa). In FP32 first: with
    // the diagonal far from the ends of the range that estimate is within 150 x
    // 2^-24 per factor of the FP64 number (one rounding of G or M, two of each
    // scale, at most 128 additions), so that 2^-13 away from the line it decides
    // alike. Nearer, or with such a diagonal, the FP64 number does. Where FP32
    // cannot hold G or M, FP64 solves.
    red[0][tid] = sg;
    red[1][tid] = prep_colsum(Ms, u, dsq);
    __syncthreads();
    if (tid >= 32)
        return;
    const int parts = nt >> 7;
    float mg = 0.0f, mm = 0.0f;
    bool fine = true, in_range = true;
    for (int c = lane; c < u; c += 32) {
        float tg = 0.0f, tm = 0.0f;
        for (int q = 0; q < parts; ++q) {
            tg += red[0][c + 128 * q];
            tm += red[1][c + 128 * q];
        }
        tg *= rdsq[c];
        tm *= dsq[c];
        fine &= isfinite(tg) && isfinite(tm);
        in_range &= dsq[c] >= 0x1p-50f && dsq[c] <= 0x1p50f;
        mg = fmaxf(mg, tg);
        mm = fmaxf(mm, tm);
    }
    fine = __all_sync(FULL, fine);
    in_range = __all_sync(FULL, in_range);
    double cond = (double)warp_max(mg) * (double)warp_max(mm);
    if (fine && (!in_range || fabs(cond - COND_FP32) <= 0x1p-13 * COND_FP32)) {
        double *d = floor_;   // (the floors are done with)
        for (int a = lane; a < u; a += 32)
            d[a] = sqrt(G[uidx[a] * (k + 1)]);
        __syncwarp();
        double dg = 0.0, dm = 0.0;
        for (int c = lane; c < u; c += 32) {
            double tg = 0.0, tm = 0.0;
            for (int a = 0; a < u; ++a) {
                const int e = uidx[a] * k + uidx[c];
                tg += fabs(G[e]) / d[a];
                tm += fabs(M64[e]) * d[a];
            }
            dg = fmax(dg, tg / d[c]);
            dm = fmax(dm, tm * d[c]);
        }
        cond = warp_max(dg) * warp_max(dm);
    }
    if (lane == 0) {
        const int mode = fine && cond <= COND_FP32 ? 0 : 1;
        flags[0] = mode;
        flags[1] = u;
        if (mode)
            atomicAdd(&stats->fp64_halfsteps, 1ull);
    }
}

// FP64 Cholesky of S_ab = Src[idx[a] * ld + idx[b]], right-looking: after
// each pivot the trailing lower triangle is updated with its (a, b) entries
// spread over the 32 lanes. Output: L in the lower triangle of Lw (row stride
// LS), invd = 1 / L_jj; false, uniformly across the warp, on a pivot
// <= tol * S_jj. The FP64 solves are bound by GB300's narrow FP64 pipe (two
// lanes per clock per SM). The lane-per-row form gave step j to rows a >= j,
// j FMAs each: p^2 / 2 warp FMA instructions with most lanes idle. The
// trailing update takes about p^3 / 192 + p.
__device__ bool warp_chol_factor_rl(const double *__restrict__ Src, int ld,
                                    const int *__restrict__ idx, int p, double *__restrict__ Lw,
                                    int LS, double *__restrict__ invd, double tol, int lane)
{
    for (int e = lane; e < p * (p + 1) / 2; e += 32) {
        const int a = tri_row(e), b = e - a * (a + 1) / 2;
        Lw[a * LS + b] = Src[idx[a] * ld + idx[b]];
    }
    __syncwarp();
    for (int j = 0; j < p; ++j) {
        const double d = Lw[j * LS + j];
        const double dorig = Src[idx[j] * ld + idx[j]];
        if (!(d > tol * dorig))
            return false;
        const double l = sqrt(d);
        const double inv = 1.0 / l;
        for (int a = j + 1 + lane; a < p; a += 32)
            Lw[a * LS + j] *= inv;
        __syncwarp();
        if (lane == 0) {
            Lw[j * LS + j] = l;
            invd[j] = inv;
        }
        const int t = p - j - 1;
        for (int e = lane; e < t * (t + 1) / 2; e += 32) {
            const int a = tri_row(e), b = e - a * (a + 1) / 2;
            const int ra = j + 1 + a, rb = j + 1 + b;
            Lw[ra * LS + rb] -= Lw[ra * LS + j] * Lw[rb * LS + j];
        }
        __syncwarp();
    }
    return true;
}

// Solve L L^T z = r with the factor from warp_chol_factor_rl; row a of r / z in
// lane a % 32, slot a / 32 (shuffle-broadcast substitutions).
template <typename T, int PT>
__device__ void warp_chol_subst(int p, const T *__restrict__ Lw, int LS,
                                const T *__restrict__ invd, T (&r)[PT], int lane)
{
    for (int j = 0; j < p; ++j) {
        const int tj = j >> 5, owner = j & 31;
        T rj = r[0];
#pragma unroll
        for (int t = 1; t < PT; ++t)
            if (tj == t)
                rj = r[t];
        const T zj = __shfl_sync(FULL, rj, owner) * invd[j];
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            const int i = lane + 32 * t;
            if (i > j && i < p)
                r[t] -= Lw[i * LS + j] * zj;
            if (t == tj && lane == owner)
                r[t] = zj;
        }
    }
    for (int j = p - 1; j >= 0; --j) {
        const int tj = j >> 5, owner = j & 31;
        T rj = r[0];
#pragma unroll
        for (int t = 1; t < PT; ++t)
            if (tj == t)
                rj = r[t];
        const T xj = __shfl_sync(FULL, rj, owner) * invd[j];
        const T *lj = Lw + j * LS;
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            const int i = lane + 32 * t;
            if (i < j)
                r[t] -= lj[i] * xj;
            if (t == tj && lane == owner)
                r[t] = xj;
        }
    }
    __syncwarp();
}

template <typename T, int KW>
__device__ __forceinline__ void warp_matvec(const T *__restrict__ Mat, int k, const T (&v)[KW],
                                            T (&out)[KW], T *__restrict__ stage, int lane)
{
#pragma unroll
    for (int s = 0; s < KW; ++s)
        stage[32 * s + lane] = v[s];
    __syncwarp();
    int j = 0;
    for (; j + 4 <= k; j += 4) {
        T vj[4];
        if constexpr (sizeof(T) == 4) {
            const float4 q = *reinterpret_cast<const float4 *>(stage + j);
            vj[0] = q.x;
            vj[1] = q.y;
            vj[2] = q.z;
            vj[3] = q.w;
        } else {
            const double2 q0 = *reinterpret_cast<const double2 *>(stage + j);
            const double2 q1 = *reinterpret_cast<const double2 *>(stage + j + 2);
            vj[0] = q0.x;
            vj[1] = q0.y;
            vj[2] = q1.x;
            vj[3] = q1.y;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const T *row = Mat + (j + t) * k;
#pragma unroll
            for (int s = 0; s < KW; ++s) {
                const int i = lane + 32 * s;
                if (i < k)
                    out[s] = fma(row[i], vj[t], out[s]);
            }
        }
    }
    for (; j < k; ++j) {
        const T vj = stage[j];
        const T *row = Mat + j * k;
#pragma unroll
        for (int s = 0; s < KW; ++s) {
            const int i = lane + 32 * s;
            if (i < k)
                out[s] = fma(row[i], vj, out[s]);
        }
    }
    __syncwarp();
}

// Per warp: index list (128 ints), right-hand side and reciprocal pivots of
// the compact system (128 doubles each), the matrix-vector staging vector
// (128 doubles), the p x LS factor; rounded to 16 bytes.
__host__ __device__ inline size_t per_warp_bytes(int pmax, int LS)
{
    const size_t b = 128 * sizeof(int) + 384 * sizeof(double) + sizeof(double) * (size_t)pmax * LS;
    return (b + 15) & ~size_t(15);
}

// Shared-memory matrices of a mode: mode 1 G64 and M64, mode 2 none (no M;
// G64 read through L1/L2).
__host__ __device__ inline size_t mats_bytes(int k, int mode)
{
    const size_t b = mode == 1 ? 2 * sizeof(double) * (size_t)k * k : 0;
    return (b + 15) & ~size_t(15);
}

// How a mode's FP64 solves use the CTA: systems of up to pmax rows (row stride
// LS), warps that solve (the others of the CTA return), G and M staged in
// shared memory or not.
struct Solve64Shape {
    int pmax, LS, warps, staged;
};

// FP64 solves of one mode. KW = index slots per lane (k <= 32 KW); PT =
// compact-system rows per lane (pmax <= 32 PT). The right-hand sides are pin's
// batch, or, with use_list, those the FP32 kernel deferred.
template <int KW, int PT, int MODE>
__device__ __forceinline__ void solve64(const SolveParams &P, const Solve64Shape &sh,
                                        const uint64_t *__restrict__ pin, int64_t nwork,
                                        bool use_list, unsigned long long *counter)
{
    using T = double;
    constexpr bool HAVE_M = MODE != 2;
    const int pmax = sh.pmax, LS = sh.LS, staged = sh.staged;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int k = P.k;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const T *Gs;
    const T *Ms = nullptr;
    if (!staged) {
        // Matrices too large for shared memory next to the per-warp space:
        // read them through L1/L2 (mode 1 at k > ~100, mode 2 always).
        Gs = P.G64;
        if (HAVE_M)
            Ms = P.M64;
    } else {
        T *gsh = reinterpret_cast<T *>(smem_raw);
        T *msh = gsh + k * k;
        for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
            gsh[e] = P.G64[e];
            msh[e] = P.M64[e];
        }
        Gs = gsh;
        Ms = msh;
    }
    unsigned char *wp =
        smem_raw + (staged ? mats_bytes(k, MODE) : 0) + warp * per_warp_bytes(pmax, LS);
    int *widx = reinterpret_cast<int *>(wp);
    T *zbuf = reinterpret_cast<T *>(wp + 128 * sizeof(int));
    T *invd = zbuf + 128;
    T *stage = invd + 128;
    T *Lw = stage + 128;
    __syncthreads();
    if (warp >= sh.warps)
        return;

    bool usable[KW];
    int nU = 0;
#pragma unroll
    for (int s = 0; s < KW; ++s) {
        const uint32_t w = P.usable_words[s];
        usable[s] = (w >> lane) & 1u;
        nU += __popc(w);
    }

    unsigned long long st_rounds = 0, st_max = 0, st_nc = 0, st_sing = 0, st_nf = 0, st_rhs = 0;

    for (;;) {
        unsigned long long j0 = 0;
        if (lane == 0)
            j0 = atomicAdd(counter, (unsigned long long)P.chunk);
        j0 = __shfl_sync(FULL, j0, 0);
        if (j0 >= (unsigned long long)nwork)
            break;
        const int64_t jend = min((int64_t)j0 + P.chunk, nwork);
        for (int64_t jj = (int64_t)j0; jj < jend; ++jj) {
            const int64_t j = use_list ? P.defer[jj] : jj;
            T g[KW], u[KW], x[KW], y[KW];
            bool inF[KW];
            bool bad = false;
#pragma unroll
            for (int s = 0; s < KW; ++s) {
                const int i = lane + 32 * s;
                g[s] = i < k ? (T)P.B[j * k + i] : (T)0;
                bad |= !isfinite(g[s]);
                u[s] = 0;
                x[s] = 0;
                y[s] = -g[s];
                inF[s] = false;
            }
            bad = __any_sync(FULL, bad);
            int status = NMF_OK;
            int rounds = 0;
            if (bad) {
                status = NMF_ERR_NONFINITE;
#pragma unroll
                for (int s = 0; s < KW; ++s)
                    x[s] = 0;
            } else {
                // Starting partition: empty (cold) or the given bitmask (warm).
                if (pin) {
#pragma unroll
                    for (int s = 0; s < KW; ++s) {
                        const int i = lane + 32 * s;
                        bool f = false;
                        if (i < k) {
                            const uint64_t wv = pin[j * P.nwords + (i >> 6)];
                            f = (wv >> (i & 63)) & 1ull;
                        }
                        inF[s] = f && usable[s];
                    }
                }
                bool have_u = false;   // u = M g, formed when a complement solve first needs it

                // Candidate point of the current partition: fills x and y.
                auto solve = [&]() -> int {
                    int nF = 0;
#pragma unroll
                    for (int s = 0; s < KW; ++s)
                        nF += __popc(__ballot_sync(FULL, inF[s]));
                    const int nA = nU - nF;
                    const bool comp = HAVE_M && nA < nF;
                    if (comp && !have_u) {
                        warp_matvec<T, KW>(Ms, k, g, u, stage, lane);
                        have_u = true;
                    }
                    bool inS[KW];
                    int rank[KW];
                    int pos = 0;
#pragma unroll
                    for (int s = 0; s < KW; ++s) {
                        inS[s] = comp ? (usable[s] && !inF[s]) : inF[s];
                        const unsigned mk = __ballot_sync(FULL, inS[s]);
                        rank[s] = pos + __popc(mk & lanemask_lt(lane));
                        if (inS[s]) {
                            widx[rank[s]] = lane + 32 * s;
                            zbuf[rank[s]] = comp ? -u[s] : g[s];
                        }
                        pos += __popc(mk);
                    }
                    const int p = pos;
                    __syncwarp();
                    if (p > 0) {
                        if (!warp_chol_factor_rl(comp ? Ms : Gs, k, widx, p, Lw, LS, invd,
                                                 PIVOT_TOL64, lane))
                            return NMF_ERR_SINGULAR_GRAM;
                        T r[PT];
#pragma unroll
                        for (int t = 0; t < PT; ++t) {
                            const int a = lane + 32 * t;
                            r[t] = a < p ? zbuf[a] : (T)0;
                        }
                        warp_chol_subst<T, PT>(p, Lw, LS, invd, r, lane);
#pragma unroll
                        for (int t = 0; t < PT; ++t) {
                            const int a = lane + 32 * t;
                            if (a < p)
                                zbuf[a] = r[t];
                        }
                        __syncwarp();
                    }
                    // The compact solution z (zbuf, p entries) against the
                    // rows it touches: x_F = u_F + M_FA z in the complement
                    // form; y = G_{:,F} x_F - g in the direct form. Both loop
                    // over the p-entry list, not over all k rows.
                    const T *Lst = comp ? Ms : Gs;
                    T acc[KW];
#pragma unroll
                    for (int s = 0; s < KW; ++s)
                        acc[s] = comp ? u[s] : -g[s];
                    for (int a = 0; a < p; ++a) {
                        const T za = zbuf[a];
                        const T *row = Lst + widx[a] * k;
#pragma unroll
                        for (int s = 0; s < KW; ++s) {
                            const int i = lane + 32 * s;
                            if (i < k)
                                acc[s] = fma(row[i], za, acc[s]);
                        }
                    }
#pragma unroll
                    for (int s = 0; s < KW; ++s) {
                        if (comp) {
                            // y_A is the complement solution itself (accurate in FP64).
                            x[s] = inF[s] ? acc[s] : (T)0;
                            y[s] = inS[s] ? zbuf[rank[s]] : (inF[s] ? (T)0 : -g[s]);
                        } else {
                            x[s] = inF[s] ? zbuf[rank[s]] : (T)0;
                            y[s] = inF[s] ? (T)0 : acc[s];
                        }
                    }
                    __syncwarp();
                    return NMF_OK;
                };

                // One solve per exchange round, from a single call site.
                bool anyF = false;
#pragma unroll
                for (int s = 0; s < KW; ++s)
                    anyF |= inF[s];
                bool need = __any_sync(FULL, anyF);   // else x = 0, y = -g already
                int alpha = 3, beta = k + 1;
                for (;;) {
                    if (need) {
                        status = solve();
                        if (status != NMF_OK)
                            break;
                    }
                    need = true;
                    bool inf[KW];
                    unsigned vm[KW];
                    int nV = 0;
#pragma unroll
                    for (int s = 0; s < KW; ++s) {
                        inf[s] = usable[s] && (inF[s] ? (x[s] < (T)0) : (y[s] < (T)0));
                        vm[s] = __ballot_sync(FULL, inf[s]);
                        nV += __popc(vm[s]);
                    }
                    if (nV == 0)
                        break;
                    if (rounds >= P.max_rounds) {
                        status = NMF_ERR_NOT_CONVERGED;
                        break;
                    }
                    if (nV < beta || alpha >= 1) {   // full exchange
                        if (nV < beta) {
                            beta = nV;
                            alpha = 3;
                        } else {
                            alpha -= 1;
                        }
#pragma unroll
                        for (int s = 0; s < KW; ++s)
                            inF[s] = inF[s] != inf[s];
                    } else {   // backup rule: the largest infeasible index alone
                        int top = -1;
#pragma unroll
                        for (int s = KW - 1; s >= 0; --s)
                            if (top < 0 && vm[s])
                                top = 32 * s + 31 - __clz(vm[s]);
#pragma unroll
                        for (int s = 0; s < KW; ++s)
                            if (lane + 32 * s == top)
                                inF[s] = !inF[s];
                    }
                    rounds += 1;
                }
                bool nf = false;
#pragma unroll
                for (int s = 0; s < KW; ++s) {
                    x[s] = x[s] > (T)0 ? x[s] : (T)0;
                    nf |= !isfinite(x[s]);
                }
                if (__any_sync(FULL, nf) && status == NMF_OK)
                    status = NMF_ERR_NONFINITE;
            }
#pragma unroll
            for (int s = 0; s < KW; ++s) {
                const int i = lane + 32 * s;
                if (i < k)
                    P.X[j * k + i] = (float)x[s];
            }
            if (P.pout) {
                unsigned bm[KW];
#pragma unroll
                for (int s = 0; s < KW; ++s)
                    bm[s] = __ballot_sync(FULL, inF[s]);
                if (lane == 0) {
#pragma unroll
                    for (int w = 0; w < (KW + 1) / 2; ++w) {
                        const uint64_t lo = bm[2 * w];
                        const uint64_t hi = (2 * w + 1 < KW) ? bm[2 * w + 1] : 0u;
                        P.pout[j * P.nwords + w] = lo | (hi << 32);
                    }
                }
            }
            if (lane == 0) {
                if (P.rounds_out)
                    P.rounds_out[j] = rounds;
                if (P.status_out)
                    P.status_out[j] = (int8_t)status;
                st_rhs += 1;
                st_rounds += rounds;
                st_max = st_max > (unsigned long long)rounds ? st_max : (unsigned long long)rounds;
                st_nc += status == NMF_ERR_NOT_CONVERGED;
                st_sing += status == NMF_ERR_SINGULAR_GRAM;
                st_nf += status == NMF_ERR_NONFINITE;
            }
        }
    }
    // (After an overflow of the deferral list the second pass re-solves the
    // whole batch, and the right-hand-side and round counts include both
    // passes.)
    if (lane == 0 && st_rhs) {
        atomicAdd(&P.stats->rhs, st_rhs);
        atomicAdd(&P.stats->rounds, st_rounds);
        atomicMax(&P.stats->max_rounds, st_max);
        if (st_nc) atomicAdd(&P.stats->not_converged, st_nc);
        if (st_sing) atomicAdd(&P.stats->singular, st_sing);
        if (st_nf) atomicAdd(&P.stats->nonfinite, st_nf);
    }
}

// One launch for every FP64 case, so that the host never waits for the mode the
// preparation chose and an FP32 half-step pays for one kernel that returns at
// once instead of three (2.4 us each): mode 1 (from the predicted partitions
// where the FP32 kernel made them), mode 2, and, in mode 0, the second pass
// that re-solves, from their starting partitions, the right-hand sides the FP32
// kernel deferred (all of them if more than DEFER_CAP were). For large k mode
// 2 has a launch of its own; `modes` has a bit for each mode a launch serves.
template <int KW>
__global__ void __launch_bounds__(BPP_THREADS, 2)
    bpp_solve_kernel(const SolveParams P, const Solve64Shape sh1, const Solve64Shape sh2,
                     int modes)
{
    const int mode = P.flags[0];
    if (!((modes >> mode) & 1))
        return;
    if (mode == 2) {
        solve64<KW, KW, 2>(P, sh2, P.pin, P.nrhs, false, &P.counters[CNT_WORK]);
        return;
    }
    int64_t nwork = P.nrhs;
    bool use_list = false;
    const uint64_t *pin = P.pin;
    unsigned long long *counter = &P.counters[CNT_WORK];
    if (mode == 0) {
        // Written by the FP32 kernel earlier in the same stream.
        const unsigned long long nd = P.counters[CNT_DEFERRED];
        if (nd == 0)
            return;
        use_list = nd <= (unsigned long long)DEFER_CAP;
        nwork = use_list ? (int64_t)nd : P.nrhs;
        counter = &P.counters[CNT_DEFER_WORK];
    } else if (P.predict) {
        pin = P.predict;
    }
    solve64<KW, (KW + 1) / 2, 1>(P, sh1, pin, nwork, use_list, counter);
}

constexpr size_t SMEM_LIMIT = 227 * 1024;
constexpr size_t SMEM_HALF = 112 * 1024;   // two CTAs per SM

template <int KW>
nmf_status launch_solve64(const SolveParams &P, cudaStream_t s)
{
    const int k = P.k;
    const int warps = P.warps < BPP_WARPS ? P.warps : BPP_WARPS;
    Solve64Shape sh1, sh2;
    sh1.pmax = k / 2 < 1 ? 1 : k / 2;
    sh2.pmax = k;
    sh1.LS = sh1.pmax | 1;   // odd row stride: conflict-free lane-per-row reads
    sh2.LS = sh2.pmax | 1;
    // Mode 1 stages G and M in shared memory when they leave room for >= 2
    // warps.
    const size_t pw1 = per_warp_bytes(sh1.pmax, sh1.LS), pw2 = per_warp_bytes(sh2.pmax, sh2.LS);
    sh1.staged = mats_bytes(k, 1) + 2 * pw1 <= SMEM_LIMIT;
    sh2.staged = 0;
    const size_t mats = sh1.staged ? mats_bytes(k, 1) : 0;
    auto fit = [&](size_t base, size_t pw, size_t limit) {   // warps of pw bytes beside base
        return (int)std::min<size_t>(warps, limit > base ? (limit - base) / pw : 0);
    };
    sh1.warps = fit(mats, pw1, SMEM_LIMIT);
    sh2.warps = fit(0, pw2, SMEM_LIMIT);
    if (sh1.warps < 1 || sh2.warps < 1)
        return NMF_ERR_INVALID_ARG;
    const size_t smem1 = mats + sh1.warps * pw1, smem2 = sh2.warps * pw2;
    auto launch = [&](int modes, int nwarps, int least, size_t smem) -> nmf_status {
        static SmemOptIn opt_in;
        NMF_TRY(ensure_smem(bpp_solve_kernel<KW>, opt_in, smem));
        int per_sm = 0;
        NMF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bpp_solve_kernel<KW>,
                                                               nwarps * 32, smem));
        if (per_sm < 1)
            return NMF_ERR_INVALID_ARG;
        int64_t blocks = (int64_t)per_sm * sm_count();
        SolveParams Q = P;
        Q.chunk = grab_size(P, blocks * nwarps);
        // As many CTAs as the batch has grabs for (the second pass's size is
        // known only on the device).
        const int64_t need = cdiv(cdiv(P.nrhs, (int64_t)Q.chunk), least);
        if (need < blocks)
            blocks = need < 1 ? 1 : need;
        bpp_solve_kernel<KW><<<(unsigned)blocks, nwarps * 32, smem, s>>>(Q, sh1, sh2, modes);
        NMF_LAUNCHED("bpp_solve_kernel");
        return NMF_OK;
    };
    // Mode 2 reads G through the L1 cache, which has what the CTA's shared memory
    // leaves: where its own shape takes less than mode 1's (k >= 83: three warps
    // and fewer), it has a launch of its own (30000 right-hand sides, k = 88, 100,
    // 128: 4.2, 7.5, 22.9 ms in a common launch, 3.3, 6.1, 16.5 so).
    if (smem1 > smem2 && smem1 > SMEM_HALF) {
        NMF_TRY(launch(1 << 2, sh2.warps, sh2.warps, smem2));
        return launch(1 << 0 | 1 << 1, sh1.warps, sh1.warps, smem1);
    }
    // A common launch: where mode 1 leaves room for two CTAs per SM, mode 2
    // takes what half an SM holds, else all it can use.
    const size_t most = smem1 <= SMEM_HALF ? SMEM_HALF : SMEM_LIMIT;
    sh2.warps = std::max(1, fit(0, pw2, std::max(most, smem1)));
    const size_t smem = std::max(smem1, sh2.warps * pw2);
    return launch(7, std::max(sh1.warps, sh2.warps), std::min(sh1.warps, sh2.warps), smem);
}

template <int KW>
nmf_status launch_modes(SolveParams P, cudaStream_t s)
{
    // Mode 0 (FP32): the group-tile pass for the all-passive group first,
    // then the per-warp solves of what it left.
    if (P.group && !P.fused) {
        if (P.group == 2)
            NMF_TRY(launch_group_tc(P, s));
        else
            NMF_TRY(launch_group32(P, s));
    }
    if (P.fused) {
        // FP64 half-step: the right-hand sides are formed here instead of
        // inside the FP32 solves.
        NMF_TRY(launch_spmm_unless_fp32(P.gat.rowptr, P.gat.colidx, P.gat.vals, P.nrhs,
                                        P.gat.cols, P.gat.F, P.k, const_cast<float *>(P.B),
                                        P.flags, s));
    }
    // Mode 1 (FP64): the FP32 kernel first predicts each right-hand side's
    // partition, and the FP64 solves start from it: they need fewer rounds (16000
    // right-hand sides, k = 50, from the signs of the unconstrained solution: 0.32
    // ms, 1.25 from that start itself). Each NLS has one minimiser, but a
    // degenerate index (x_i = y_i = 0) may come out at rounding noise or at zero,
    // passive or not, by the start, and a batch that the cap on rounds stopped
    // short of an answer may now reach it. Not under a tight cap, which keeps its
    // meaning.
    if (P.max_rounds < 2 * PREDICT_ROUNDS)
        P.predict = nullptr;
    NMF_TRY(launch_solve32(P, s));
    return launch_solve64<KW>(P, s);
}

}  // namespace

size_t bpp_work_bytes(int k) { return layout(k).total; }

namespace {

// Launch shape of the solve kernels per k (warps per CTA, right-hand sides per
// grab of the work counter, whether the group-tile pass runs first):
// {8, 8, group pass on} until bpp_tune has measured the batch or the caller
// set one; the group pass runs on the tensor cores (2) for 65 <= k <= 112,
// else on the SIMT pipes (1). Shapes with group 0 or 1 compute the same results
// (a right-hand side's arithmetic does not depend on where it runs); group 2
// solves the all-passive group with tensor-core products, to FP32 accuracy
// but not the same bits.
struct BppShape {
    int warps = BPP_WARPS, chunk = 8, group = -1;   // -1: the default for k
};
std::mutex g_shape_mu;
BppShape g_shape[NMF_MAX_K + 1];

BppShape shape_for(int k)
{
    std::lock_guard<std::mutex> lock(g_shape_mu);
    BppShape sh = g_shape[k];
    if (sh.group < 0)   // measured: the tensor-core pass wins from k = 65 (k = 100: 2.5x), the
                        // SIMT pass at k = 50 (dense ANLS, 127.1 against 126.4 iter/s)
        sh.group = k >= 65 && group_tc_supported(k) ? 2 : 1;
    return sh;
}

SolveParams solve_params(int k, int64_t nrhs, const double *G, const float *B, float *X,
                         const uint64_t *passive_in, uint64_t *passive_out, int32_t *rounds_out,
                         int8_t *status_out, int max_rounds, void *work, BppStats *stats_dev)
{
    const WorkLayout L = layout(k);
    unsigned char *w = static_cast<unsigned char *>(work);
    SolveParams P;
    P.k = k;
    P.nwords = (k + 63) / 64;
    P.max_rounds = max_rounds;
    P.nrhs = nrhs;
    P.G32 = reinterpret_cast<float *>(w + L.g32);
    P.M32 = reinterpret_cast<float *>(w + L.m32);
    P.G64 = G;
    P.M64 = reinterpret_cast<double *>(w + L.m64);
    P.usable_words = reinterpret_cast<uint32_t *>(w + L.usable);
    P.flags = reinterpret_cast<int *>(w + L.flags);
    P.B = B;
    P.X = X;
    P.pin = passive_in;
    P.pout = passive_out;
    P.rounds_out = rounds_out;
    P.status_out = status_out;
    P.counters = reinterpret_cast<unsigned long long *>(w + L.counters);
    P.predict = passive_out;
    P.fused = 0;
    P.gat = CsrGather{nullptr, nullptr, nullptr, nullptr, 0};
    P.defer = reinterpret_cast<int64_t *>(w + L.defer);
    P.stats = stats_dev;
    const BppShape sh = shape_for(k);
    P.warps = sh.warps;
    P.chunk = sh.chunk;
    P.group = sh.group;
    return P;
}

nmf_status launch_solves(const SolveParams &P, cudaStream_t s)
{
    if (P.k <= 32)
        return launch_modes<1>(P, s);
    if (P.k <= 64)
        return launch_modes<2>(P, s);
    if (P.k <= 96)
        return launch_modes<3>(P, s);
    return launch_modes<4>(P, s);
}

}  // namespace

namespace {

constexpr size_t PREP_STATIC = 16 * 1024;   // at least the kernel's static shared memory

template <int C, int NSEG>
nmf_status launch_prep(const SolveParams &P, BppStats *stats_dev, cudaStream_t s)
{
    const int k = P.k;
    const size_t smem = sizeof(float) * (size_t)k * k;
    static SmemOptIn opt_in;
    NMF_TRY(ensure_smem(bpp_prep_kernel<C, NSEG>, opt_in, smem + PREP_STATIC));
    // A thread per segment of the triangle beside warp 0, 128 at a time.
    const int64_t want = cdiv(cdiv(prep_segments(k), C) + 32, 128) * 128;
    const int threads = (int)std::min<int64_t>(want, C == 1 ? PREP_THREADS : PREP_THREADS / 2);
    bpp_prep_kernel<C, NSEG><<<C, threads, smem, s>>>(
        P.G64, k, const_cast<float *>(P.G32), const_cast<float *>(P.M32),
        const_cast<double *>(P.M64), const_cast<uint32_t *>(P.usable_words),
        const_cast<int *>(P.flags), P.counters, stats_dev);
    NMF_LAUNCHED("bpp_prep_kernel");
    return NMF_OK;
}

}  // namespace

nmf_status launch_bpp_prep(int k, const double *G, void *work, BppStats *stats_dev, cudaStream_t s,
                           bool alone)
{
    const SolveParams P = solve_params(k, 0, G, nullptr, nullptr, nullptr, nullptr, nullptr,
                                       nullptr, 0, work, stats_dev);
    if (k > PREP_ONE_K && alone)
        return launch_prep<8, 1>(P, stats_dev, s);
    // Segments per thread (k = 128: 2112).
    const int nseg = prep_segments(k), nt = PREP_THREADS - 32;
    return nseg <= nt       ? launch_prep<1, 1>(P, stats_dev, s)
           : nseg <= 2 * nt ? launch_prep<1, 2>(P, stats_dev, s)
                            : launch_prep<1, 3>(P, stats_dev, s);
}

nmf_status launch_bpp_solve(int k, int64_t nrhs, const double *G, const float *B, float *X,
                            const uint64_t *passive_in, uint64_t *passive_out, int32_t *rounds_out,
                            int8_t *status_out, int max_rounds, void *work, BppStats *stats_dev,
                            cudaStream_t s, const CsrGather *gather, uint64_t *predict)
{
    if (nrhs == 0)
        return NMF_OK;
    SolveParams P = solve_params(k, nrhs, G, B, X, passive_in, passive_out, rounds_out,
                                 status_out, max_rounds, work, stats_dev);
    if (gather) {
        P.fused = 1;
        P.gat = *gather;
    }
    if (!P.predict)
        P.predict = predict;
    return launch_solves(P, s);
}

// Times every candidate launch shape on this batch (after one warm-up each;
// the passive-set, round and status outputs are left out so every candidate
// starts from the same partitions) and keeps the fastest for k. X receives
// the solution.
nmf_status bpp_tune(int k, int64_t nrhs, const double *G, const float *B, float *X,
                    const uint64_t *passive_in, int max_rounds, void *work, BppStats *stats_dev,
                    cudaStream_t s, int *warps_out, int *chunk_out, int *group_out)
{
    // The candidates keep the group mode of the current shape (and try the
    // pass off only beside the SIMT pass, whose results it shares), so every
    // candidate gives the same bits.
    const int gm = shape_for(k).group;
    const BppShape cand[] = {{16, 4, gm}, {16, 8, gm}, {8, 1, gm},  {8, 4, gm},
                             {8, 8, gm},  {8, 32, gm}, {4, 16, gm}, {8, 8, gm == 1 ? 0 : gm}};
    NMF_TRY(launch_bpp_prep(k, G, work, stats_dev, s));
    SolveParams P = solve_params(k, nrhs, G, B, X, passive_in, nullptr, nullptr, nullptr,
                                 max_rounds, work, stats_dev);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    NMF_CUDA(cudaEventCreate(&e0));
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return NMF_ERR_CUDA;
    }
    BppShape best;
    float best_ms = -1.0f;
    nmf_status st = NMF_OK;
    for (const BppShape &c : cand) {
        // The same launch as another candidate: above k = 64 the FP32 solves
        // take twice the shape's warps, at most 16, and the FP64 ones at most 8;
        // the last one differs only in its group pass.
        if ((c.warps == 16 && k > 64) || (&c == std::end(cand) - 1 && c.group == gm))
            continue;
        P.warps = c.warps;
        P.chunk = c.chunk;
        P.group = c.group;
        float ms = 0.0f;
        for (int rep = 0; rep < 2 && st == NMF_OK; ++rep) {
            // The prep kernel resets the work counter; re-run it per solve.
            st = launch_bpp_prep(k, G, work, stats_dev, s);
            if (st == NMF_OK && cudaEventRecord(e0, s) != cudaSuccess)
                st = NMF_ERR_CUDA;
            if (st == NMF_OK)
                st = launch_solves(P, s);
            if (st == NMF_OK && (cudaEventRecord(e1, s) != cudaSuccess ||
                                 cudaEventSynchronize(e1) != cudaSuccess ||
                                 cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess))
                st = NMF_ERR_CUDA;
        }
        if (st != NMF_OK)
            break;
        if (best_ms < 0.0f || ms < best_ms) {
            best_ms = ms;
            best = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    NMF_TRY(st);
    {
        std::lock_guard<std::mutex> lock(g_shape_mu);
        g_shape[k] = best;
    }
    if (warps_out)
        *warps_out = best.warps;
    if (chunk_out)
        *chunk_out = best.chunk;
    if (group_out)
        *group_out = best.group;
    return NMF_OK;
}

nmf_status bpp_set_shape(int k, int warps, int chunk, int group)
{
    if (k < 1 || k > NMF_MAX_K || warps < 1 || warps > 16 || chunk < 1 || chunk > 1024 ||
        group < 0 || group > 2 || (group == 2 && !group_tc_supported(k)))
        return NMF_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_shape_mu);
    g_shape[k].warps = warps;
    g_shape[k].chunk = chunk;
    g_shape[k].group = group;
    return NMF_OK;
}

nmf_status bpp_get_shape(int k, int *warps, int *chunk, int *group)
{
    if (k < 1 || k > NMF_MAX_K)
        return NMF_ERR_INVALID_ARG;
    const BppShape sh = shape_for(k);
    if (warps)
        *warps = sh.warps;
    if (chunk)
        *chunk = sh.chunk;
    if (group)
        *group = sh.group;
    return NMF_OK;
}

nmf_status launch_bpp(int k, int64_t nrhs, const double *G, const float *B, float *X,
                      const uint64_t *passive_in, uint64_t *passive_out, int32_t *rounds_out,
                      int8_t *status_out, int max_rounds, void *work, BppStats *stats_dev,
                      cudaStream_t s, uint64_t *predict)
{
    NMF_TRY(launch_bpp_prep(k, G, work, stats_dev, s));
    return launch_bpp_solve(k, nrhs, G, B, X, passive_in, passive_out, rounds_out, status_out,
                            max_rounds, work, stats_dev, s, nullptr, predict);
}

}  // namespace nmf
