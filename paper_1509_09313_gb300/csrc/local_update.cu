// The paper's alternative local updates for the two steps of Alg. 1: MU
// (Eq. 5) and HALS (Eq. 6). Both take the same inputs as the BPP solves, the
// k x k Gram G of the fixed factor and the right-hand sides R (A H^T for W,
// (W^T A)^T for H^T), and update the rows of the other factor X in place.
//
//   MU    x_ij <- x_ij R_ij / (X G)_ij, all from the X before the step; where
//         (X G)_ij is not positive x_ij is left as it is (0 is a fixed point).
//   HALS  for i = 0..k-1 in order: x_i <- [R_i - sum_{l != i} G_li x_l]_+ / G_ii,
//         with the newest values of the other entries; a column with
//         G_ii <= 0 is set to 0.
//
// Rows are independent. row_update_kernel gives a warp a tile of 64 rows, held
// transposed in shared memory (entry l of every row side by side), lane l
// owning rows 2 l and 2 l + 1; the coordinates are taken in blocks of 8. For
// a block, the sums over the entries outside it, sum_l G_li x_l, are a small
// matrix product (the lane's two rows are the halves of packed FP32x2 FMAs, G
// is staged with every value twice as their other operand); HALS then takes the
// block's coordinates in turn, adding each new value to the sums still open. Every sum consists of
// the terms of its own definition: keeping x G and adding d times row i of G
// after each change would save the products but loses digits. HALS often
// drives whole columns to zero, and the large steps d = -x_i leave the updated
// sums as the rounding residue of a cancellation (measured on the sparse 20000
// x 10000 test: 1e-3 relative factor error after five iterations, against 1e-7
// for the direct form). Eight terms at a time are summed apart and then added
// to the total.
//
// local_update_kernel (one warp per row) serves batches too small for tiles, and
// MU where the last wave of tiles would be too empty: lane l holds entries l, l +
// 32, ... (KW slots), G in FP32 in shared memory lane-interleaved (entry (r, c) at
// r * 32 KW + (c % 32) * KW + c / 32) so that a lane reads its KW entries of a row
// as one vector; MU forms X G with one product, HALS each coordinate's sum with a
// butterfly. It also forms the projected-gradient norm of the stopping rule (Lin
// 2007): grad = X G - R, an entry counting where x_ij > 0 and, where x_ij = 0, only
// if negative; squares summed in FP32 per row, FP64 across rows, per-CTA partials
// added in a fixed order. The two kernels' sums round differently: a row's last
// bits depend on how many rows the call has.
//
// Roofline: HBM (12 k bytes per row: R and X in, X out); 2 k^2 FLOPs per row.
// The tile kernel is bound by the latency of its instruction stream (some ten
// warps per SM, one instruction in four cycles each). Measured, 96000 x 50:
// HALS 45 us, MU 37 us (one warp per row: 272 and 51 us; HBM alone 8.5 us);
// 1000000 x 50: HALS 411 us (2785), MU 356 us (478). 128-row tiles, four rows
// per lane, were slower at 96000 rows (50 and 46 us) and 1000000 (457, 421).
#include <algorithm>

#include "common.cuh"

namespace nmf {
namespace {

constexpr int LU_WARPS = 8;
enum LuOp { LU_MU = 0, LU_HALS = 1, LU_PGRAD = 2 };
constexpr int RU_WARPS = 12;     // warps per CTA of row_update_kernel
constexpr int RU_ROWS = 64;      // rows per warp tile, two per lane
constexpr int RU_BLOCK = 8;      // coordinates per block, terms per partial sum
constexpr int RU_DUP_K = 64;     // G staged with every value twice up to this k
constexpr size_t LU_SMEM = 227 * 1024;

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool live)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(live ? 4 : 0)
                 : "memory");
}

// a / g rounded to nearest for a >= 0 (or infinite), g > 0 and rg = 1 / g rounded:
// the quotient corrected by its exact remainder (Markstein 1990), with the plain
// division where one of the three is so large or small that a step could
// overflow or lose bits (1 / g is infinite up to g = 2^-128, and 0 times that a
// NaN; the remainder of a < 1e-31 is not exact). Zero, the common numerator, is
// its own quotient.
__device__ __forceinline__ float quotient(float a, float g, float rg)
{
    constexpr float LO = 1e-30f, HI = 1e30f;
    const float q = a * rg;
    if (!(a > 0.0f))
        return 0.0f;
    if (!(a > LO && a < HI && g > LO && g < HI && q > LO && q < HI))
        return a / g;
    return fmaf(fmaf(-q, g, a), rg, q);
}

// Shared memory: G (k rows of k rounded up to 8; every value twice when DUP, as
// the operand pair of a packed FMA), then per warp the tile of X (k x RS) and
// the block's panel of R, later of its new values (8 x RS); RS = 66.
__host__ __device__ inline size_t ru_g_floats(int k, bool dup)
{
    return (size_t)k * ((k + 7) & ~7) * (dup ? 2 : 1);
}
__host__ __device__ inline size_t ru_warp_floats(int k)
{
    return (size_t)(k + RU_BLOCK) * (RU_ROWS + 2);
}

template <bool HALS, bool DUP>
__global__ void __launch_bounds__(RU_WARPS * 32, 1)
    row_update_kernel(const double *__restrict__ G, int k, const float *__restrict__ R,
                      float *__restrict__ X, int64_t rows, int nw)
{
    constexpr int TR = RU_ROWS, RS = RU_ROWS + 2, D = DUP ? 2 : 1;
    extern __shared__ __align__(16) float lu_smem[];
    const int KP = (k + 7) & ~7;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *Gs = lu_smem;
    float *Xs = Gs + ru_g_floats(k, DUP) + warp * ru_warp_floats(k);
    float *Ps = Xs + k * RS;
    const uint32_t magic = 0xffffffffu / (uint32_t)k + 1u;   // e / k for e < 2^16
    const int64_t ntiles = cdiv(rows, TR);
    int64_t tile = warp < nw ? (int64_t)blockIdx.x * nw + warp : ntiles;
    // A tile of X (its rows are one stretch), transposed on the way; all of it
    // in flight at once.
    auto load_tile = [&]() {
        const float *src = X + tile * TR * k;
        const int ne = (int)min((int64_t)TR, rows - tile * TR) * k;
#pragma unroll 4
        for (int e = lane; e < ne; e += 32) {
            const int r = k == 1 ? e : (int)__umulhi((uint32_t)e, magic);
            cp_async4(Xs + (e - r * k) * RS + r, src + e, true);
        }
    };
    if (tile < ntiles)
        load_tile();
    // All the CTA's warps stage G; those without a tile of their own then leave.
#pragma unroll 4
    for (int e = threadIdx.x; e < k * KP; e += RU_WARPS * 32) {
        const int r = e / KP, c = e - r * KP;
        const float g = c < k ? (float)G[r * k + c] : 0.0f;
        if (DUP)
            reinterpret_cast<float2 *>(Gs)[e] = make_float2(g, g);
        else
            Gs[e] = g;
    }
    __syncthreads();
    const float2 zero2 = make_float2(0.0f, 0.0f), neg1 = make_float2(-1.0f, -1.0f);
    const int pr = lane >> 3, pc = lane & 7;   // panel copies: row pr + 4 t, column pc
    while (tile < ntiles) {
        const int64_t row0 = tile * TR;
        const int nr = (int)min((int64_t)TR, rows - row0);
        asm volatile("cp.async.wait_all;" ::: "memory");
        for (int i0 = 0; i0 < k; i0 += RU_BLOCK) {
            const int nb = min(RU_BLOCK, k - i0);
            __syncwarp();   // X staged; the last panel is read
            // The block's panel of R, in flight while the sums are formed.
            {
                const float *src = R + (row0 + pr) * k + i0 + pc;
                float *dst = Ps + pc * RS + pr;
#pragma unroll 4
                for (int t = 0; t < TR / 4; ++t) {
                    const bool live = pr + 4 * t < nr && pc < nb;
                    cp_async4(dst + 4 * t, live ? src : R, live);
                    src += 4 * k;
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            // Lane l: rows 2 l and 2 l + 1, as the pairs of packed FMAs.
            // HALS keeps the total's rounding errors beside it (Dekker's
            // two-sum: exact while the total is the larger), since the
            // coordinate is a small difference of two large sums: plain adds
            // lost 1.3 times what the warp's butterfly sum loses, this loses
            // half as much (2 us of 43).
            float2 tot[RU_BLOCK], err[RU_BLOCK], part[RU_BLOCK];
#pragma unroll
            for (int b = 0; b < RU_BLOCK; ++b)
                tot[b] = err[b] = zero2;
            auto add = [&](int b) {   // tot + err += part
                const float2 s = __fadd2_rn(tot[b], part[b]);
                if (HALS) {
                    const float2 d = __ffma2_rn(tot[b], neg1, s);
                    err[b] = __fadd2_rn(err[b], __ffma2_rn(d, neg1, part[b]));
                }
                tot[b] = s;
            };
            auto pair_of_x = [&](int l) {
                return *reinterpret_cast<const float2 *>(Xs + l * RS + 2 * lane);
            };
            // v += G[l][i0 + lo .. hi) x_l.
            auto term = [&](int l, float2 (&v)[RU_BLOCK], int lo, int hi) {
                const float4 *gr = reinterpret_cast<const float4 *>(Gs + (l * KP + i0) * D);
                const float2 x = pair_of_x(l);
#pragma unroll
                for (int h = 0; h < 2 * D; ++h) {
                    const float4 g = gr[h];
                    constexpr int W = 4 / D;   // coordinates per 16 bytes
#pragma unroll
                    for (int b = 0; b < W; ++b) {
                        const int i = W * h + b;
                        const float2 gg = DUP ? (b ? make_float2(g.z, g.w) : make_float2(g.x, g.y))
                                          : b == 0 ? make_float2(g.x, g.x)
                                          : b == 1 ? make_float2(g.y, g.y)
                                          : b == 2 ? make_float2(g.z, g.z)
                                                   : make_float2(g.w, g.w);
                        if (i >= lo && i < hi)
                            v[i] = __ffma2_rn(gg, x, v[i]);
                    }
                }
            };
            for (int l0 = 0; l0 < k; l0 += RU_BLOCK) {
                if (HALS && l0 == i0)
                    continue;
#pragma unroll
                for (int b = 0; b < RU_BLOCK; ++b)
                    part[b] = zero2;
                if (l0 + RU_BLOCK <= k) {
#pragma unroll
                    for (int j = 0; j < RU_BLOCK; ++j)
                        term(l0 + j, part, 0, RU_BLOCK);
                } else {
                    for (int l = l0; l < k; ++l)
                        term(l, part, 0, RU_BLOCK);
                }
#pragma unroll
                for (int b = 0; b < RU_BLOCK; ++b)
                    add(b);
            }
            // HALS: the terms of the block's own entries, summed apart: first
            // those still to come (coordinates below j), before they change.
#pragma unroll
            for (int b = 0; b < RU_BLOCK; ++b)
                part[b] = zero2;
            if (HALS) {
#pragma unroll
                for (int j = 1; j < RU_BLOCK; ++j)
                    if (j < nb)
                        term(i0 + j, part, 0, j);
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
#pragma unroll
            for (int i = 0; i < RU_BLOCK; ++i) {
                if (i >= nb)
                    break;
                const float gii = Gs[((i0 + i) * KP + i0 + i) * D];
                const float rg = 1.0f / gii;
                float *pp = Ps + i * RS + 2 * lane;
                const float2 r = *reinterpret_cast<const float2 *>(pp);
                float2 x;
                if (HALS) {
                    add(i);
                    // max(n, 0), where the error of a sum that overflowed, a NaN,
                    // does not take an infinite n for zero.
                    const float d0 = r.x - tot[i].x, d1 = r.y - tot[i].y;
                    const float n0 = fmaxf(d0 - err[i].x, d0 == INFINITY ? d0 : 0.0f);
                    const float n1 = fmaxf(d1 - err[i].y, d1 == INFINITY ? d1 : 0.0f);
                    x.x = gii > 0.0f ? quotient(n0, gii, rg) : 0.0f;
                    x.y = gii > 0.0f ? quotient(n1, gii, rg) : 0.0f;
                    *reinterpret_cast<float2 *>(Xs + (i0 + i) * RS + 2 * lane) = x;
                } else {
                    const float2 t = tot[i];
                    x = pair_of_x(i0 + i);   // (stays for the blocks to come)
                    if (t.x > 0.0f)
                        x.x = x.x * r.x / t.x;
                    if (t.y > 0.0f)
                        x.y = x.y * r.y / t.y;
                }
                *reinterpret_cast<float2 *>(pp) = x;
                // ... then the new values, as they come.
                if (HALS)
                    term(i0 + i, part, i + 1, RU_BLOCK);
            }
            __syncwarp();
            {
                float *dst = X + (row0 + pr) * k + i0 + pc;
                const float *src = Ps + pc * RS + pr;
#pragma unroll 4
                for (int t = 0; t < TR / 4; ++t) {
                    if (pr + 4 * t < nr && pc < nb)
                        *dst = src[4 * t];
                    dst += 4 * k;
                }
            }
        }
        __syncwarp();   // the next tile overwrites Xs
        tile += (int64_t)gridDim.x * nw;
        if (tile < ntiles)
            load_tile();
    }
}

template <int KW>
__device__ __forceinline__ void lu_row_fma(const float *__restrict__ p, float a, float (&acc)[KW])
{
    if constexpr (KW == 1) {
        acc[0] = fmaf(p[0], a, acc[0]);
    } else if constexpr (KW == 2) {
        const float2 q = *reinterpret_cast<const float2 *>(p);
        acc[0] = fmaf(q.x, a, acc[0]);
        acc[1] = fmaf(q.y, a, acc[1]);
    } else {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        acc[0] = fmaf(q.x, a, acc[0]);
        acc[1] = fmaf(q.y, a, acc[1]);
        acc[2] = fmaf(q.z, a, acc[2]);
        acc[3] = fmaf(q.w, a, acc[3]);
    }
}

template <int KW, int OP>
__global__ void __launch_bounds__(LU_WARPS * 32)
    local_update_kernel(const double *__restrict__ G, int k, const float *__restrict__ R,
                        float *__restrict__ X, int64_t rows, double *__restrict__ partials)
{
    constexpr bool HALS = OP == LU_HALS;
    constexpr int RS = 32 * KW;
    extern __shared__ __align__(16) float lu_smem[];
    const int k4 = (k + 3) & ~3;
    float *Gs = lu_smem;                                    // k4 x RS
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *stage = Gs + k4 * RS + warp * RS;                // per-warp vector
    for (int e = threadIdx.x; e < k4 * RS; e += blockDim.x) {
        const int r = e / RS, q = e - r * RS;
        const int c = q / KW + 32 * (q % KW);
        Gs[e] = (r < k && c < k && !(HALS && r == c)) ? (float)G[r * k + c] : 0.0f;
    }
    __syncthreads();
    float gdiag[KW];   // G_ii of the lane's entries
#pragma unroll
    for (int s = 0; s < KW; ++s) {
        const int i = lane + 32 * s;
        gdiag[s] = i < k ? (float)G[i * k + i] : 0.0f;
    }
    const int64_t nwarps = (int64_t)gridDim.x * LU_WARPS;
    double pg = 0.0;   // LU_PGRAD: this lane's sum of squares
    for (int64_t row = (int64_t)blockIdx.x * LU_WARPS + warp; row < rows; row += nwarps) {
        float x[KW], r[KW], t[KW];
#pragma unroll
        for (int s = 0; s < KW; ++s) {
            const int i = lane + 32 * s;
            x[s] = i < k ? X[row * k + i] : 0.0f;
            r[s] = i < k ? R[row * k + i] : 0.0f;
            t[s] = 0.0f;
            if (!HALS)
                stage[32 * s + lane] = x[s];
        }
        __syncwarp();
        const float *base = Gs + lane * KW;
        if (!HALS) {
            // t = x G (G symmetric: t_i = sum_l x_l G_li, row l of G times x_l).
            for (int l = 0; l < k4; l += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(stage + l);
                lu_row_fma<KW>(base + (l + 0) * RS, v.x, t);
                lu_row_fma<KW>(base + (l + 1) * RS, v.y, t);
                lu_row_fma<KW>(base + (l + 2) * RS, v.z, t);
                lu_row_fma<KW>(base + (l + 3) * RS, v.w, t);
            }
            __syncwarp();   // stage is rewritten for the next row
            if constexpr (OP == LU_PGRAD) {
                float sq = 0.0f;
#pragma unroll
                for (int s = 0; s < KW; ++s) {
                    const float gr = t[s] - r[s];
                    const float pj = x[s] > 0.0f ? gr : fminf(gr, 0.0f);
                    sq = fmaf(pj, pj, sq);
                }
                pg += (double)sq;
            } else {
#pragma unroll
                for (int s = 0; s < KW; ++s)
                    if (t[s] > 0.0f)
                        x[s] = x[s] * r[s] / t[s];
            }
        } else {
            for (int i = 0; i < k; ++i) {
                // sum_{l != i} G_il x_l: this lane's entries of row i (the
                // staged diagonal is zero), then a butterfly sum (fixed order).
                float part[KW];
#pragma unroll
                for (int s = 0; s < KW; ++s)
                    part[s] = 0.0f;
                lu_row_fma<KW>(base + i * RS, 1.0f, part);
                float sum = 0.0f;
#pragma unroll
                for (int s = 0; s < KW; ++s)
                    sum = fmaf(part[s], x[s], sum);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    sum += __shfl_xor_sync(FULL, sum, o);
                const int si = i >> 5, owner = i & 31;
#pragma unroll
                for (int s = 0; s < KW; ++s)
                    if (s == si && lane == owner) {
                        const float gii = gdiag[s];
                        const float num = r[s] - sum;
                        x[s] = gii > 0.0f ? (num > 0.0f ? num : 0.0f) / gii : 0.0f;
                    }
            }
        }
        if (OP != LU_PGRAD) {
#pragma unroll
            for (int s = 0; s < KW; ++s) {
                const int i = lane + 32 * s;
                if (i < k)
                    X[row * k + i] = x[s];
            }
        }
    }
    if (OP == LU_PGRAD) {
        __shared__ double red[LU_WARPS];
        for (int o = 16; o > 0; o >>= 1)
            pg += __shfl_xor_sync(FULL, pg, o);
        if (lane == 0)
            red[warp] = pg;
        __syncthreads();
        if (threadIdx.x == 0) {
            double b = 0.0;
            for (int w = 0; w < LU_WARPS; ++w)
                b += red[w];
            partials[blockIdx.x] = b;
        }
    }
}

// out = sum of partials[0..n) in index order.
__global__ void lu_sum_kernel(const double *__restrict__ partials, int n, double *__restrict__ out)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < n; ++i)
            s += partials[i];
        *out = s;
    }
}

// Warps per CTA (one CTA per SM) of the tile kernel that the shared memory holds.
int ru_warps(int k, bool dup)
{
    const size_t g = sizeof(float) * ru_g_floats(k, dup), w = sizeof(float) * ru_warp_floats(k);
    return (int)std::min<size_t>(RU_WARPS, (LU_SMEM - g) / w);
}

template <bool HALS, bool DUP>
nmf_status launch_rows(const double *G, int k, const float *R, float *X, int64_t rows,
                       cudaStream_t s)
{
    const int64_t tiles = cdiv(rows, RU_ROWS);
    // As many warps as share the tiles out evenly, so that G is staged once per
    // SM.
    const int64_t nw = std::min<int64_t>(cdiv(tiles, sm_count()), ru_warps(k, DUP));
    const size_t smem = sizeof(float) * (ru_g_floats(k, DUP) + nw * ru_warp_floats(k));
    static SmemOptIn opt_in;
    NMF_TRY(ensure_smem(row_update_kernel<HALS, DUP>, opt_in, smem));
    int64_t blocks = cdiv(tiles, nw);
    if (blocks > sm_count())
        blocks = sm_count();
    row_update_kernel<HALS, DUP><<<(unsigned)blocks, 32 * RU_WARPS, smem, s>>>(G, k, R, X, rows,
                                                                                  (int)nw);
    NMF_LAUNCHED(HALS ? "row_update_kernel<hals>" : "row_update_kernel<mu>");
    return NMF_OK;
}

// LU_PGRAD writes one partial per CTA (at most max_parts); *nparts gets the
// count.
template <int KW, int OP>
nmf_status launch_lu(const double *G, int k, const float *R, float *X, int64_t rows,
                     double *partials, int max_parts, int *nparts, cudaStream_t s)
{
    const size_t smem = sizeof(float) * (size_t)(((k + 3) & ~3) + LU_WARPS) * 32 * KW;
    static SmemOptIn opt_in;
    NMF_TRY(ensure_smem(local_update_kernel<KW, OP>, opt_in, smem));
    int per_sm = 0;
    NMF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, local_update_kernel<KW, OP>, LU_WARPS * 32, smem));
    int64_t blocks = (int64_t)(per_sm > 0 ? per_sm : 1) * sm_count();
    const int64_t need = cdiv(rows, LU_WARPS);
    if (need < blocks)
        blocks = need;
    if (OP == LU_PGRAD && blocks > max_parts)
        blocks = max_parts;
    if (blocks < 1)
        blocks = 1;
    local_update_kernel<KW, OP><<<(unsigned)blocks, LU_WARPS * 32, smem, s>>>(G, k, R, X, rows,
                                                                            partials);
    NMF_LAUNCHED(OP == LU_HALS ? "local_update_kernel<hals>"
                 : OP == LU_MU ? "local_update_kernel<mu>"
                               : "local_update_kernel<pgrad>");
    *nparts = (int)blocks;
    return NMF_OK;
}

template <int OP>
nmf_status launch_lu_k(const double *G, int k, const float *R, float *X, int64_t rows,
                       double *partials, int max_parts, int *nparts, cudaStream_t s)
{
    if (k <= 32)
        return launch_lu<1, OP>(G, k, R, X, rows, partials, max_parts, nparts, s);
    if (k <= 64)
        return launch_lu<2, OP>(G, k, R, X, rows, partials, max_parts, nparts, s);
    return launch_lu<4, OP>(G, k, R, X, rows, partials, max_parts, nparts, s);
}

// Whether the tile kernel is the faster one. HALS: from the row count on where a
// wave of tiles (20-25 us at k = 50, whatever the batch) passes that of single
// rows (17); no k up to 128 and no partial wave after it is slower (k = 128, 7297
// rows 94 / 115 us, 38913 rows, one tile past a wave, 178 / 405; k = 50, 96000
// rows 45 / 264).
// MU: single rows cost little more than the tiles' terms, so the last wave of
// tiles has to be full enough: the time of full waves stands against that of
// their rows, done singly, like 1 to 1.4 for 25 to 32 coordinates (one slot per
// lane there), 1.6-1.8 up to 48, 1.5 up to 56 and 1.2-1.4 up to 64 (two slots, 12
// and 10 warps of tiles), 1.65 and more with at least 7 warps (four slots), 1.65
// (to k = 104) and 1.5 with 6, 1.25 with 5 and 1.05 with 4. Measured, tiles / single rows: k = 32,
// 175200 rows 40.9 / 40.9 us, 117000 rows (half of the second wave) 40.9 / 30.5; k
// = 64, 90000 rows 51 / 59, 97300 rows 86 / 63; k = 100, 80000 rows 121 / 141,
// 58369 rows 125 / 108; k = 128, 77900 rows 213 / 168.
bool rows_in_tiles(bool hals, int k, int64_t rows)
{
    if (rows < (hals ? 48 : 384) * (int64_t)sm_count())
        return false;
    if (hals || k <= 24)
        return true;
    const int nw = ru_warps(k, k <= RU_DUP_K);
    const int64_t tiles = cdiv(rows, RU_ROWS), slots = (int64_t)nw * sm_count();
    const double fill = (double)tiles / (double)(cdiv(tiles, slots) * slots);
    return fill >= (k <= 32   ? 0.75
                    : k <= 48 ? 0.6
                    : k <= 64 ? (nw == RU_WARPS ? 0.67 : 0.82)
                    : nw >= 7 ? 0.0
                    : nw == 6 ? (k <= 104 ? 0.66 : 0.75)
                    : nw == 5 ? 0.83
                              : 0.95);
}

}  // namespace

nmf_status launch_local_update(int solver, const double *G, int k, const float *R, float *X,
                               int64_t rows, cudaStream_t s)
{
    if (rows == 0)
        return NMF_OK;
    if (solver != NMF_SOLVER_MU && solver != NMF_SOLVER_HALS)
        return NMF_ERR_INVALID_ARG;
    const bool hals = solver == NMF_SOLVER_HALS;
    if (!rows_in_tiles(hals, k, rows)) {
        int np = 0;
        if (hals)
            return launch_lu_k<LU_HALS>(G, k, R, X, rows, nullptr, 0, &np, s);
        return launch_lu_k<LU_MU>(G, k, R, X, rows, nullptr, 0, &np, s);
    }
    if (hals)
        return k <= RU_DUP_K ? launch_rows<true, true>(G, k, R, X, rows, s)
                             : launch_rows<true, false>(G, k, R, X, rows, s);
    return k <= RU_DUP_K ? launch_rows<false, true>(G, k, R, X, rows, s)
                         : launch_rows<false, false>(G, k, R, X, rows, s);
}

int pgrad_partials_len() { return 2 * sm_count(); }

nmf_status launch_pgrad_sq(const double *G, int k, const float *R, const float *X, int64_t rows,
                           double *partials, double *out, cudaStream_t s)
{
    int np = 0;
    if (rows > 0)
        NMF_TRY(launch_lu_k<LU_PGRAD>(G, k, R, const_cast<float *>(X), rows, partials,
                                      pgrad_partials_len(), &np, s));
    lu_sum_kernel<<<1, 32, 0, s>>>(partials, np, out);
    NMF_LAUNCHED("lu_sum_kernel");
    return NMF_OK;
}

}  // namespace nmf

extern "C" nmf_status nmf_update_mu(int32_t k, int64_t rows, const double *G, const float *R,
                                    float *X, void *stream)
{
    if (k < 1 || k > NMF_MAX_K || rows < 0 || !G || (rows > 0 && (!R || !X)))
        return NMF_ERR_INVALID_ARG;
    return nmf::launch_local_update(NMF_SOLVER_MU, G, k, R, X, rows,
                                    static_cast<cudaStream_t>(stream));
}

extern "C" nmf_status nmf_update_hals(int32_t k, int64_t rows, const double *G, const float *R,
                                      float *X, void *stream)
{
    if (k < 1 || k > NMF_MAX_K || rows < 0 || !G || (rows > 0 && (!R || !X)))
        return NMF_ERR_INVALID_ARG;
    return nmf::launch_local_update(NMF_SOLVER_HALS, G, k, R, X, rows,
                                    static_cast<cudaStream_t>(stream));
}
