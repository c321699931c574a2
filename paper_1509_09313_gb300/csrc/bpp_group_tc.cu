// Group-tile pass of the FP32 batched BPP (Sec. 4.2) for the all-passive
// group, on the 5th-generation tensor cores (launch shape group = 2; the
// SIMT pass of bpp_group.cu is group = 1).
//
// Membership, outputs and the hand-over to the per-warp kernel are those of
// the SIMT pass: a right-hand side joins the group when its first candidate
// partition is U, all usable indices (a warm start covering U, or from the
// empty start every usable y_i = -g_i infeasible); for the group F = U and the
// factor is the inverse M = G_UU^{-1} the preparation holds, so
//     x0 = M g,   r = g - G x0 (on U),   x1 = x0 + M r,
// and x1 is kept where it passes the sign test. A member whose solution is not
// kept (or not formed, when a wait timed out) is marked GROUP_PENDING and goes
// to the per-warp kernel.
//
// The three products run as tcgen05 MMAs (M = 128 right-hand sides, N = k
// padded to 16, K = 16) on BF16 splits, accumulated in FP32 in TMEM:
//   x0 = g M:   g = g_hi + g_lo, M = M_hi + M_lo   (3 MMAs per step)
//   G x0':      x0' = hi + lo of x0 (exact: the vector whose residual is
//               taken, and the one x1 is built on), G = G_hi + G_mid + G_lo
//               (5 MMAs per step; G is represented to 2^-24)
//   M r:        r = r_hi + r_lo, M 2-way (3 MMAs per step).
// M's 16-bit representation only slows the refinement's contraction (x1 -
// x* = (I - M'G)(x0' - x*) + O(FP32 rounding of r)), so x1 is within the FP32
// solve's cond(G) 6e-8 bound; the results are not bitwise those of the SIMT
// pass or of the per-warp kernel.
//
// Kernel: one persistent CTA per SM walking 128-right-hand-side tiles, 16
// warps. Warp 0 allocates TMEM (three accumulators of N columns); thread 0
// also issues each product's MMAs once all threads have written its A
// operand (mbarrier bar_a), and commits them to bar_d.
//   all warps  four threads per right-hand side (its TMEM lane), each with
//              a quarter of the 16-column chunks: membership, the A operands
//              (split in registers, stored in the canonical K-major
//              128-byte-swizzled layout), the masks, the sign test and the
//              outputs; per-row decisions combine the four threads' partial
//              results through shared memory (a named barrier of the four
//              warps that share 32 rows).
// M and G (split) stay in shared memory for the whole kernel: with the A tiles
// they fill it, so one tile is in flight per SM and its chain of phases bounds
// the kernel. What shortens the chain: the next tile's right-hand sides are
// loaded into registers while the last product runs (four lanes to a row: 64
// us less than a row to a lane); results leave through
// the A tiles in bulk copies (rows of k floats: a warp's own stores touch 32
// lines each); membership divides only where products cannot decide it; one
// exchange per decision. 1e6 right-hand sides, k = 100: 33000 cycles per tile
// without these (888 us for the kernel), 20000 with them (570 us); by memory traffic
// it would be 120 us.
// Every mbarrier wait is bounded (~2 s).
#include <math.h>

#include "bpp_internal.cuh"
#include "tc_ptx.cuh"

namespace nmf {
namespace bpp {
namespace {

using namespace tc;

constexpr int GC_BM = 128;         // right-hand sides per tile (MMA M)
constexpr int GC_PARTS = 4;        // threads per right-hand side
constexpr int GC_THREADS = GC_PARTS * GC_BM;   // 16 warps; thread 0 also issues the MMAs
constexpr int GC_MAX_K = 112;

template <int NP>   // k padded to 16: the MMA N and the columns of each accumulator
struct GcLayout {
    static constexpr int NKB = (NP + 63) / 64;       // K-blocks of 64 (K padded to 64 NKB)
    static constexpr int A_TILE = GC_BM * 128;       // 16 KB: 128 rows x 64 BF16
    static constexpr int B_TILE = NP * 128;          // NP rows x 64 BF16
    static constexpr int OFF_AHI = 0;
    static constexpr int OFF_ALO = NKB * A_TILE;
    static constexpr int OFF_B = 2 * NKB * A_TILE;   // M_hi, M_lo, G_hi, G_mid, G_lo
    static constexpr int PART = NKB * B_TILE;
    static constexpr int OFF_BAR = OFF_B + 5 * PART;
    static constexpr int OFF_TMEM = OFF_BAR + 16;
    static constexpr int OFF_ABORT = OFF_TMEM + 4;
    static constexpr int OFF_DSQ = OFF_BAR + 32;     // GC_MAX_K floats
    static constexpr int OFF_RD = OFF_DSQ + 4 * GC_MAX_K;        // GC_MAX_K float2
    static constexpr int OFF_XCH = OFF_RD + 8 * GC_MAX_K;        // twice [part][row] float2
    static constexpr int BYTES = OFF_XCH + 2 * 8 * GC_PARTS * GC_BM;
    static_assert(OFF_RD % 16 == 0 && OFF_XCH % 16 == 0, "alignment");
    static constexpr int TMEM_COLS = 3 * NP <= 64 ? 64 : 3 * NP <= 128 ? 128
                                   : 3 * NP <= 256 ? 256 : 512;
    static_assert(NP % 16 == 0 && NP <= GC_MAX_K, "MMA N");
    static_assert(B_TILE % 1024 == 0 && OFF_B % 1024 == 0, "128-byte-swizzled tiles");
    static_assert(BYTES + 1024 <= 227 * 1024, "shared memory budget");
};

// 16 consecutive FP32 columns of this warp's 32 TMEM lanes (no wait).
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// v = hi + mid + lo to 2^-24 |v| (each step's remainder is exact in FP32).
__device__ __forceinline__ void split8_3(const float (&v)[8], uint4 &hi, uint4 &mid, uint4 &lo)
{
    uint32_t hw[4], mw[4], lw[4];
    const float2 neg1 = make_float2(-1.0f, -1.0f);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 v2 = make_float2(v[2 * i], v[2 * i + 1]);
        const __nv_bfloat162 hb = __floats2bfloat162_rn(v2.x, v2.y);
        const float2 r1 = __ffma2_rn(__bfloat1622float2(hb), neg1, v2);   // exact
        const __nv_bfloat162 mb = __floats2bfloat162_rn(r1.x, r1.y);
        const float2 r2 = __ffma2_rn(__bfloat1622float2(mb), neg1, r1);   // exact
        const __nv_bfloat162 lb = __floats2bfloat162_rn(r2.x, r2.y);
        hw[i] = *reinterpret_cast<const uint32_t *>(&hb);
        mw[i] = *reinterpret_cast<const uint32_t *>(&mb);
        lw[i] = *reinterpret_cast<const uint32_t *>(&lb);
    }
    hi = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    mid = make_uint4(mw[0], mw[1], mw[2], mw[3]);
    lo = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}

// v = hi + lo within 2^-17 |v|; s = hi + lo (exact in FP32).
__device__ __forceinline__ void split8_sum(const float (&v)[8], uint4 &hi, uint4 &lo,
                                           float (&s)[8])
{
    uint32_t hw[4], lw[4];
    const float2 neg1 = make_float2(-1.0f, -1.0f);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 v2 = make_float2(v[2 * i], v[2 * i + 1]);
        const __nv_bfloat162 hb = __floats2bfloat162_rn(v2.x, v2.y);
        const float2 hf = __bfloat1622float2(hb);
        const float2 d = __ffma2_rn(hf, neg1, v2);   // v - hi, exact
        const __nv_bfloat162 lb = __floats2bfloat162_rn(d.x, d.y);
        const float2 lf = __bfloat1622float2(lb);
        const float2 sm = __fadd2_rn(hf, lf);
        s[2 * i] = sm.x;
        s[2 * i + 1] = sm.y;
        hw[i] = *reinterpret_cast<const uint32_t *>(&hb);
        lw[i] = *reinterpret_cast<const uint32_t *>(&lb);
    }
    hi = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    lo = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}

template <int NP>
__global__ void __launch_bounds__(GC_THREADS, 1) bpp_group_tc_kernel(const SolveParams P)
{
    if (P.flags[0] != 0)
        return;   // not an FP32 half-step
    using L = GcLayout<NP>;
    constexpr int NKB = L::NKB;
    extern __shared__ unsigned char gc_smem_dyn[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(gc_smem_dyn) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int k = P.k;
    const uint32_t bar_a = sbase + L::OFF_BAR, bar_d = bar_a + 8;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + L::OFF_TMEM);
    volatile int *abort = reinterpret_cast<volatile int *>(smem + L::OFF_ABORT);
    float *dsq = reinterpret_cast<float *>(smem + L::OFF_DSQ);
    float2 *rd = reinterpret_cast<float2 *>(smem + L::OFF_RD);

    int nU = 0;
    uint64_t umask[2] = {0ull, 0ull};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        nU += __popc(P.usable_words[q]);
        umask[q >> 1] |= (uint64_t)P.usable_words[q] << (32 * (q & 1));
    }
    if (tid == 0) {
        mbar_init(bar_a, GC_PARTS * GC_BM);   // the row threads
        mbar_init(bar_d, 1);     // the MMA commits
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // sqrt(G_ii); its reciprocal with, where the column is not usable, the
    // infinity that takes the column out of a minimum. In range: the
    // reciprocals' products decide the membership (below).
    bool dr = true;
    for (int i = tid; i < NP; i += GC_THREADS) {
        const bool u = i < k && ((P.usable_words[i >> 5] >> (i & 31)) & 1u);
        const float d = u ? sqrtf(P.G32[i * k + i]) : 1.0f;
        dr = dr && d >= 0x1p-40f && d <= 0x1p40f;
        dsq[i] = d;
        rd[i] = make_float2(1.0f / d, u ? 0.0f : INFINITY);
    }
    const bool scales_ok = __syncthreads_and(dr);
    // B operands: row n (the output index i), 16-byte chunk c along K (the
    // contraction index j): M[n][j] 2-way, G[n][j] 3-way, zero past k.
    for (int e = tid; e < NP * NKB * 8; e += GC_THREADS) {
        const int n = e / (NKB * 8), c = e - n * (NKB * 8);
        float mv[8], gv[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int j = 8 * c + t;
            const bool in = n < k && j < k;
            mv[t] = in ? P.M32[n * k + j] : 0.0f;
            gv[t] = in ? P.G32[n * k + j] : 0.0f;
        }
        uint4 mh, ml, gh, gm, gl;
        split8(mv, mh, ml);
        split8_3(gv, gh, gm, gl);
        const uint32_t off = (uint32_t)((c >> 3) * L::B_TILE) + sw128_off(n, c & 7);
        unsigned char *b = smem + L::OFF_B + off;
        *reinterpret_cast<uint4 *>(b) = mh;
        *reinterpret_cast<uint4 *>(b + L::PART) = ml;
        *reinterpret_cast<uint4 *>(b + 2 * L::PART) = gh;
        *reinterpret_cast<uint4 *>(b + 3 * L::PART) = gm;
        *reinterpret_cast<uint4 *>(b + 4 * L::PART) = gl;
    }
    fence_proxy_async();   // these writes are read by the tensor cores
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"((uint32_t)L::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int64_t ntiles = cdiv(P.nrhs, (int64_t)GC_BM);

    // The MMAs of one product (thread 0, after the row threads' arrivals on
    // bar_a): x0 = g M (step 0), G x0' (1), M r (2), committed to bar_d.
    // kind::f16, BF16 A and B (both K-major), FP32 D, M = 128, N = NP.
    uint32_t ph_a = 0;
    auto issue = [&](int step) -> bool {
        if (!mbar_wait_fast(bar_a, ph_a & 1u, abort))
            return false;
        ++ph_a;
        tc_fence_after();
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                               ((uint32_t)(NP >> 3) << 17) | ((uint32_t)(GC_BM >> 4) << 24);
        const uint64_t ahi = sw128_desc(sbase + L::OFF_AHI), alo = sw128_desc(sbase + L::OFF_ALO);
        const uint64_t b0 = sw128_desc(sbase + L::OFF_B);
        constexpr uint64_t A16 = (uint64_t)(L::A_TILE >> 4), B16 = (uint64_t)(L::B_TILE >> 4);
        constexpr uint64_t P16 = (uint64_t)(L::PART >> 4);
        const uint64_t mhi = b0, mlo = b0 + P16, ghi = b0 + 2 * P16, gmid = b0 + 3 * P16,
                       glo = b0 + 4 * P16;
        const uint32_t d = tmem + (uint32_t)(step * NP);
#pragma unroll
        for (int kb = 0; kb < NKB; ++kb)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                if (4 * kb + kk >= NP / 16)   // (columns past NP are zero)
                    continue;
                const uint64_t oa = kb * A16 + (uint64_t)(kk * 2);
                const uint64_t ob = kb * B16 + (uint64_t)(kk * 2);
                const uint32_t acc = (kb | kk) ? 1u : 0u;
                if (step != 1) {   // x0 = g M, then M r
                    mma_bf16(d, ahi + oa, mhi + ob, idesc, acc);
                    mma_bf16(d, ahi + oa, mlo + ob, idesc, 1u);
                    mma_bf16(d, alo + oa, mhi + ob, idesc, 1u);
                } else {           // G x0'
                    mma_bf16(d, ahi + oa, ghi + ob, idesc, acc);
                    mma_bf16(d, ahi + oa, gmid + ob, idesc, 1u);
                    mma_bf16(d, alo + oa, ghi + ob, idesc, 1u);
                    mma_bf16(d, ahi + oa, glo + ob, idesc, 1u);
                    mma_bf16(d, alo + oa, gmid + ob, idesc, 1u);
                }
            }
        mma_commit(bar_d);
        return true;
    };

    {
        // ------------------------------------------------ right-hand sides
        // Four threads per right-hand side (warps w and w + 4, w + 8, w + 12
        // share a TMEM lane quarter): part p takes the 16-column chunks p,
        // p + 4, ... of the row; per-row decisions combine the parts' partial
        // results through shared memory.
        const int quarter = warp & 3;            // TMEM lane quarter of this warp
        const int part = warp >> 2;              // 0..3
        const int rl = quarter * 32 + lane;      // row of the tile = TMEM lane
        const uint32_t tq = tmem + ((uint32_t)(quarter * 32) << 16);
        constexpr int NCH = NP / 16;                       // 16-column chunks
        constexpr int MYCH = (NCH + GC_PARTS - 1) / GC_PARTS;   // chunks per part (at most)
        float2 *xch = reinterpret_cast<float2 *>(smem + L::OFF_XCH);
        uint32_t xph = 0;
        auto quarter_sync = [&] {
            asm volatile("bar.sync %0, %1;" ::"r"(1 + quarter), "n"(GC_PARTS * 32) : "memory");
        };
        unsigned char *arow_hi = smem + L::OFF_AHI, *arow_lo = smem + L::OFF_ALO;
        auto put_a = [&](int c8, const uint4 &h, const uint4 &l) {
            const uint32_t off = (uint32_t)((c8 >> 3) * L::A_TILE) + sw128_off(rl, c8 & 7);
            *reinterpret_cast<uint4 *>(arow_hi + off) = h;
            *reinterpret_cast<uint4 *>(arow_lo + off) = l;
        };
        // This thread's usable columns, bit 16 m + i for column 16 (part + 4 m)
        // + i (formed once: the per-column tests below are one bit test).
        uint32_t mymask = 0;
#pragma unroll
        for (int m = 0; m < MYCH; ++m)
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int c = 16 * (part + GC_PARTS * m) + i;
                if (c < k && (((c < 64 ? umask[0] : umask[1]) >> (c & 63)) & 1ull))
                    mymask |= 1u << (16 * m + i);
            }
        mymask = __reduce_or_sync(FULL, mymask);   // (the same in the whole warp)
        auto use_mi = [&](int m, int i) { return (mymask >> (16 * m + i)) & 1u; };
        // The parts' partial results of one decision: max and min over the
        // row, ok where no part gave the max a sign (every part gets the same
        // result). A barrier of the four warps that share the rows; two sets
        // of slots in turn, so that one barrier orders the reads and the
        // writes after the next.
        auto combine = [&](float mxp, float mnp, float &mx, float &mn) -> bool {
            float2 *x = xch + (xph & 1u) * (GC_PARTS * GC_BM);
            ++xph;
            x[part * GC_BM + rl] = make_float2(mxp, mnp);
            quarter_sync();
            uint32_t sgn = 0;
            mx = 0.0f;
            mn = INFINITY;
#pragma unroll
            for (int q = 0; q < GC_PARTS; ++q) {
                const float2 v = x[q * GC_BM + rl];
                sgn |= __float_as_uint(v.x);
                mx = fmaxf(mx, fabsf(v.x));
                mn = fminf(mn, v.y);
            }
            return !(sgn >> 31);
        };
        uint32_t st_rhs = 0, st_nf = 0, pending = 0;   // (at most one a tile and thread)
        const int rounds = P.pin ? 0 : 1;
        uint32_t ph = 0;
        bool dead = false;   // a wait of this warp timed out: only mark from now on
        // Rows of B and X start on 16 bytes when k is a multiple of 4 (the
        // bases come from the allocator, 256-byte aligned, checked here).
        const bool vec4 = (k & 3) == 0 &&
                          ((reinterpret_cast<uintptr_t>(P.B) | reinterpret_cast<uintptr_t>(P.X)) & 15) == 0;
        // This part's columns of a tile's right-hand sides, in registers.
        // Where rows are 16-byte aligned, four lanes read 64 contiguous bytes
        // of each of their four rows in turn (8 rows per load instead of 32:
        // the cost is in the lines an instruction touches), and own_rows
        // exchanges them before use.
        float g[MYCH][16];
        auto relu = [](float x) { return x > 0.0f ? x : 0.0f; };   // (a NaN gives 0)
        auto load_g = [&](int64_t t) {
            if (vec4) {
                const int64_t j4 = t * GC_BM + (rl & ~3);
                const float *rows = P.B + (j4 < P.nrhs ? j4 : 0) * k;
#pragma unroll
                for (int m = 0; m < MYCH; ++m) {
                    const int c = 16 * (part + GC_PARTS * m) + 4 * (lane & 3);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 v = j4 + q < P.nrhs && c < k
                                             ? *reinterpret_cast<const float4 *>(rows + q * k + c)
                                             : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        g[m][4 * q] = v.x;
                        g[m][4 * q + 1] = v.y;
                        g[m][4 * q + 2] = v.z;
                        g[m][4 * q + 3] = v.w;
                    }
                }
            } else {
                const int64_t j = t * GC_BM + rl;
                const bool live = j < P.nrhs;
                const float *row = P.B + (live ? j : 0) * k;
#pragma unroll
                for (int m = 0; m < MYCH; ++m)
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int c = 16 * (part + GC_PARTS * m) + i;
                        g[m][i] = live && c < k ? row[c] : 0.0f;
                    }
            }
        };
        // Quads q of lane b of four <- quad b of lane q: a 4 x 4 transpose in
        // two exchanges.
        auto own_rows = [&] {
            if (!vec4)
                return;
#pragma unroll
            for (int m = 0; m < MYCH; ++m)
#pragma unroll
                for (int s = 1; s <= 2; s *= 2) {
                    const bool up = lane & s;
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if ((e >> 2) & s)
                            continue;
                        float &a = g[m][e], &b = g[m][e + 4 * s];
                        const float o = __shfl_xor_sync(FULL, up ? a : b, s);
                        a = up ? o : a;
                        b = up ? b : o;
                    }
                }
        };
        load_g(blockIdx.x);
        for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
            const int64_t j = t * GC_BM + rl;
            const bool live = j < P.nrhs;
            own_rows();
            // Membership: the first candidate partition is U (the test of the
            // SIMT pass and of the per-warp kernel: every usable g_i above
            // FEAS_TOL32 max_c |g_c| / d_c times d_i). The products g_i (1 /
            // d_i) stand within 2^-22 of the quotients, and the test's own
            // roundings within as much of its exact value, so where the
            // least product is further than 2^-19 from the bound they decide
            // alike; elsewhere, and where scales near the ends of the range
            // could round further, the quotients decide. (28 divisions per
            // thread and tile otherwise: a third of the instructions.)
            int member;
            {
                float fsum = 0.0f, mxp = 0.0f, mnp = INFINITY;
#pragma unroll
                for (int m = 0; m < MYCH; ++m) {
                    const int c16 = part + GC_PARTS * m;
                    if (c16 >= NCH)
                        continue;   // warp-uniform
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float4 r = *reinterpret_cast<const float4 *>(rd + 16 * c16 + i);
                        fsum = __fmaf_rn(g[m][i], 0.0f, fsum);   // NaN from any Inf or NaN
                        fsum = __fmaf_rn(g[m][i + 1], 0.0f, fsum);
                        mxp = fmaxf(mxp, fmaxf(fabsf(g[m][i] * r.x), fabsf(g[m][i + 1] * r.z)));
                        mnp = fminf(mnp, fminf(__fmaf_rn(g[m][i], r.x, r.y),
                                               __fmaf_rn(g[m][i + 1], r.z, r.w)));
                    }
                }
                const bool okp = fsum == 0.0f;
                // The last tile's results are out of the A tiles before the
                // exchange lets this one's right-hand sides into them.
                if (part == 0 && lane == 0)
                    bulk_wait_read();
                float mx, mn;
                const bool ok = combine(okp ? mxp : -1.0f, mnp, mx, mn) && live && nU > 0;
                if (P.pin) {
                    bool inp = ok;
                    if (ok)
                        for (int w = 0; w < P.nwords; ++w)
                            if ((P.pin[j * P.nwords + w] & umask[w]) != umask[w])
                                inp = false;
                    member = inp;
                } else if (P.max_rounds < 1) {
                    member = 0;
                } else {
                    const float bound = FEAS_TOL32 * mx;
                    const bool far = scales_ok && mx >= 0x1p-60f && mx <= 0x1p60f &&
                                     fabsf(mn - bound) > 0x1p-19f * bound;
                    member = ok && mn > bound;
                    if (__any_sync(FULL, ok && !far)) {   // (the same in the four warps)
                        float gmp = 0.0f;
#pragma unroll
                        for (int m = 0; m < MYCH; ++m)
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const int c = 16 * (part + GC_PARTS * m) + i;
                                if (c < k)
                                    gmp = fmaxf(gmp, fabsf(g[m][i]) / dsq[c]);
                            }
                        float gmax, unused;
                        combine(gmp, 0.0f, gmax, unused);
                        const float ytol = FEAS_TOL32 * gmax;
                        bool inp = true;
#pragma unroll
                        for (int m = 0; m < MYCH; ++m)
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const int c = 16 * (part + GC_PARTS * m) + i;
                                if (use_mi(m, i) && !(-g[m][i] < -ytol * dsq[c]))
                                    inp = false;
                            }
                        const bool all_in = combine(inp ? 0.0f : -1.0f, 0.0f, gmax, unused);
                        member = ok && all_in;
                    }
                }
            }
            if (!dead) {
                // Step 1: A = g.
#pragma unroll
                for (int m = 0; m < MYCH; ++m) {
                    const int c16 = part + GC_PARTS * m;
                    if (c16 < NCH)
#pragma unroll
                        for (int h8 = 0; h8 < 2; ++h8) {
                            float v[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                v[i] = member ? g[m][8 * h8 + i] : 0.0f;
                            uint4 h, l;
                            split8(v, h, l);
                            put_a(2 * c16 + h8, h, l);
                        }
                }
                fence_proxy_async();
                tc_fence_before();
                mbar_arrive(bar_a);
                if (tid == 0)
                    issue(0);
                // Step 2: x0 (masked to U) -> x0' = hi + lo, back into its
                // accumulator columns and into A.
                dead = !__all_sync(FULL, mbar_wait(bar_d, ph & 1u, abort));
                ++ph;
            }
            if (!dead) {
                tc_fence_after();
#pragma unroll
                for (int m = 0; m < MYCH; ++m) {
                    const int c16 = part + GC_PARTS * m;
                    if (c16 >= NCH)
                        continue;   // warp-uniform
                    uint32_t raw[16];
                    tmem_ld16_nowait(tq + (uint32_t)(16 * c16), raw);
                    tmem_wait_ld();
#pragma unroll
                    for (int h8 = 0; h8 < 2; ++h8) {
                        float v[8], sm[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            v[i] = use_mi(m, 8 * h8 + i) ? __uint_as_float(raw[8 * h8 + i]) + 0.0f
                                                         : 0.0f;
                        }
                        uint4 h, l;
                        split8_sum(v, h, l, sm);
                        put_a(2 * c16 + h8, h, l);
                        tmem_st8(tq + (uint32_t)(16 * c16 + 8 * h8), sm);
                    }
                }
                tmem_wait_st();
                fence_proxy_async();
                tc_fence_before();
                mbar_arrive(bar_a);
                if (tid == 0)
                    issue(1);
                // Step 3: r = g - G x0' on U.
                dead = !__all_sync(FULL, mbar_wait(bar_d, ph & 1u, abort));
                ++ph;
            }
            if (!dead) {
                tc_fence_after();
#pragma unroll
                for (int m = 0; m < MYCH; ++m) {
                    const int c16 = part + GC_PARTS * m;
                    if (c16 >= NCH)
                        continue;
                    uint32_t raw[16];
                    tmem_ld16_nowait(tq + (uint32_t)(NP + 16 * c16), raw);
                    tmem_wait_ld();
#pragma unroll
                    for (int h8 = 0; h8 < 2; ++h8) {
                        float v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            v[i] = member && use_mi(m, 8 * h8 + i)
                                       ? g[m][8 * h8 + i] - __uint_as_float(raw[8 * h8 + i])
                                       : 0.0f;
                        }
                        uint4 h, l;
                        split8(v, h, l);
                        put_a(2 * c16 + h8, h, l);
                    }
                }
                fence_proxy_async();
                tc_fence_before();
                mbar_arrive(bar_a);
                if (tid == 0)
                    issue(2);
            }
            // The next tile's right-hand sides, while the last product runs and
            // this tile's results go out (g is not read again in this tile).
            load_g(t + gridDim.x);
            if (!dead) {
                // Step 4: x1 = x0' + M r, the sign test, the outputs.
                dead = !__all_sync(FULL, mbar_wait(bar_d, ph & 1u, abort));
                ++ph;
            }
            // The exchanges below take every warp, dead or not.
            float x1[MYCH][16];
            float xmp = 0.0f, xnp = 0.0f;
            if (!dead) {
                tc_fence_after();
#pragma unroll
                for (int m = 0; m < MYCH; ++m) {
                    const int c16 = part + GC_PARTS * m;
                    if (c16 >= NCH) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            x1[m][i] = 0.0f;
                        continue;
                    }
#pragma unroll
                    for (int h8 = 0; h8 < 2; ++h8) {   // (16 columns at once spill)
                        uint32_t a0[8], a2[8];
                        tmem_ld8_nowait(tq + (uint32_t)(16 * c16 + 8 * h8), a0);
                        tmem_ld8_nowait(tq + (uint32_t)(2 * NP + 16 * c16 + 8 * h8), a2);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int ci = 8 * h8 + i;
                            const float x = use_mi(m, ci) ? __uint_as_float(a0[i]) +
                                                                (__uint_as_float(a2[i]) + 0.0f)
                                                          : 0.0f;
                            x1[m][ci] = x;
                            const float xd = x * dsq[16 * c16 + ci];   // (not usable: 0)
                            xmp = fmaxf(xmp, fabsf(xd));
                            xnp = fminf(xnp, xd);
                        }
                    }
                }
                tc_fence_before();   // the accumulators are read before the next tile's MMAs
            } else {
#pragma unroll
                for (int m = 0; m < MYCH; ++m)
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        x1[m][i] = 0.0f;
            }
            float xm, xn;
            const bool okall = combine(dead ? -1.0f : xmp, xnp, xm, xn);
            const bool feasible = !(xn < -(FEAS_TOL32 * xm));
            bool fin = true;
            if (__any_sync(FULL, isinf(xm))) {   // (no x is infinite otherwise; the same in the four warps)
                float big = 0.0f, unused;
#pragma unroll
                for (int m = 0; m < MYCH; ++m)
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        big = fmaxf(big, x1[m][i]);
                combine(big, 0.0f, big, unused);
                fin = !isinf(big);
            }
            const bool keep = okall && member && feasible;
            if (vec4 && __all_sync(FULL, keep)) {   // (the same in the four warps)
                // The quarter's 32 rows are one piece of X: through the rows'
                // part of the A tiles (every product of this tile has read
                // them), 4 KB of each in turn, and out in bulk copies.
#pragma unroll
                for (int m = 0; m < MYCH; ++m)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int c = 16 * (part + GC_PARTS * m) + 4 * q;
                        const uint32_t o = (uint32_t)(lane * k + c) * 4u;
                        if (c < k)
                            *reinterpret_cast<float4 *>(arow_hi + (o >> 12) * L::A_TILE +
                                                        quarter * 4096 + (o & 4095u)) =
                                make_float4(relu(x1[m][4 * q]), relu(x1[m][4 * q + 1]),
                                            relu(x1[m][4 * q + 2]), relu(x1[m][4 * q + 3]));
                    }
                fence_proxy_async();
                quarter_sync();
                if (part == 0 && lane == 0) {
                    float *x = P.X + (t * GC_BM + quarter * 32) * k;
                    for (uint32_t o = 0; o < 128u * (uint32_t)k; o += 4096u)
                        bulk_store(x + o / 4, sbase + L::OFF_AHI + (o >> 12) * L::A_TILE + quarter * 4096,
                                   min(128u * (uint32_t)k - o, 4096u));
                    bulk_commit();
                }
            } else if (keep) {
                float *xr = P.X + j * k;
#pragma unroll
                for (int m = 0; m < MYCH; ++m)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int c = 16 * (part + GC_PARTS * m) + 4 * q;
                        if (vec4) {
                            if (c < k)
                                *reinterpret_cast<float4 *>(xr + c) =
                                    make_float4(relu(x1[m][4 * q]), relu(x1[m][4 * q + 1]),
                                                relu(x1[m][4 * q + 2]), relu(x1[m][4 * q + 3]));
                        } else {
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (c + i < k)
                                    xr[c + i] = relu(x1[m][4 * q + i]);
                        }
                    }
            }
            if (keep) {
                if (part == 0) {
                    if (P.pout)
                        for (int w = 0; w < P.nwords; ++w)
                            P.pout[j * P.nwords + w] = umask[w];
                    if (P.rounds_out)
                        P.rounds_out[j] = rounds;
                    if (P.status_out)
                        P.status_out[j] = (int8_t)(fin ? NMF_OK : NMF_ERR_NONFINITE);
                    st_rhs += 1;
                    st_nf += fin ? 0 : 1;
                }
            }
            // The others go to the per-warp kernel, members with their mark.
            if (part == 0 && live && !keep) {
                if (member)
                    reinterpret_cast<uint32_t *>(P.X)[j * k] = GROUP_PENDING;
                pending += 1;
            }
        }
        if (part == 0 && lane == 0)
            bulk_wait_all();
        for (int o = 16; o > 0; o >>= 1) {
            pending += __shfl_xor_sync(FULL, pending, o);
            st_rhs += __shfl_xor_sync(FULL, st_rhs, o);
            st_nf += __shfl_xor_sync(FULL, st_nf, o);
        }
        if (lane == 0) {
            if (pending)
                atomicAdd(&P.counters[CNT_PENDING], pending);
            if (st_rhs) {
                atomicAdd(&P.stats->rhs, st_rhs);
                atomicAdd(&P.stats->rounds, (unsigned long long)(rounds * st_rhs));
                atomicMax(&P.stats->max_rounds, (unsigned long long)rounds);
                if (st_nf)
                    atomicAdd(&P.stats->nonfinite, st_nf);
            }
        }
    }


    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"((uint32_t)L::TMEM_COLS)
                     : "memory");
    }
}

template <int NP>
nmf_status launch_np(const SolveParams &P, cudaStream_t s)
{
    using L = GcLayout<NP>;
    const size_t smem = (size_t)L::BYTES + 1024;
    static SmemOptIn opt_in;
    NMF_TRY(ensure_smem(bpp_group_tc_kernel<NP>, opt_in, smem));
    const int64_t ntiles = cdiv(P.nrhs, (int64_t)GC_BM);
    const unsigned grid = (unsigned)std::min<int64_t>(ntiles < 1 ? 1 : ntiles, sm_count());
    bpp_group_tc_kernel<NP><<<grid, GC_THREADS, smem, s>>>(P);
    NMF_LAUNCHED("bpp_group_tc_kernel");
    return NMF_OK;
}

}  // namespace

bool group_tc_supported(int k) { return k >= 1 && k <= GC_MAX_K; }

nmf_status launch_group_tc(const SolveParams &P, cudaStream_t s)
{
    switch ((P.k + 15) / 16) {
    case 1: return launch_np<16>(P, s);
    case 2: return launch_np<32>(P, s);
    case 3: return launch_np<48>(P, s);
    case 4: return launch_np<64>(P, s);
    case 5: return launch_np<80>(P, s);
    case 6: return launch_np<96>(P, s);
    case 7: return launch_np<112>(P, s);
    default: return NMF_ERR_INVALID_ARG;
    }
}

}  // namespace bpp
}  // namespace nmf
