// Sparse products of Alg. 1 with CSR A (the sparse "MM" task of Sec. 4.3):
// out (rows x k) = S F, one warp per CSR row. The warp reads its row's
// (column, value) pairs 32 at a time with one coalesced load each, then
// broadcasts them by shuffle; lane l accumulates columns l, l+32, ... of the
// output, gathering the matching rows of F (k contiguous floats each). Sums
// run in the row's stored order, so results are deterministic.
//
// W^T A needs the CSR of A^T: csr_transpose builds it on the device (count
// per column, prefix sum, scatter, then each output row sorted by index so
// the layout does not depend on scheduling).
//
// Roofline: HBM. Compulsory bytes per product: rowptr + colidx + vals +
// F + out; the gathers of F rows add up to nnz * k * 4 bytes when F is not
// L2-resident. While it is, 64 warps per SM with one or two rows in flight
// each are best (200000 x 10^6, 10^7 entries, k = 20: 237 us against 360 with
// spmm_stream_kernel; 100000 x 50000, 10^6 entries, k = 50: 40 against 52);
// beyond, fewer warps with eight in flight (10^6 x 10^6, 10^7 entries: k = 50
// 609 us against 480, k = 33, 132 MB, 532 against 449).
#include "common.cuh"

namespace nmf {
namespace {

constexpr int SPMM_THREADS = 256;

template <int KW>
__global__ void __launch_bounds__(SPMM_THREADS)
    spmm_kernel(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                const float *__restrict__ vals, int64_t rows, const float *__restrict__ F, int k,
                float *__restrict__ out, const int *__restrict__ mode_flag)
{
    if (mode_flag && *mode_flag == 0)
        return;   // FP32 half-step: its solves form the product rows themselves
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * SPMM_THREADS + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * SPMM_THREADS) >> 5;
    for (int64_t i = warp0; i < rows; i += nw) {
        float acc[KW];
#pragma unroll
        for (int s = 0; s < KW; ++s)
            acc[s] = 0.0f;
        const int64_t beg = rowptr[i], end = rowptr[i + 1];
        for (int64_t p0 = beg; p0 < end; p0 += 32) {
            const int64_t p = p0 + lane;
            const int c = p < end ? colidx[p] : 0;
            const float v = p < end ? vals[p] : 0.0f;
            const int cnt = (int)min((int64_t)32, end - p0);
            for (int l = 0; l < cnt; ++l) {
                const int64_t cl = __shfl_sync(FULL, c, l);
                const float vl = __shfl_sync(FULL, v, l);
                const float *frow = F + cl * k;
#pragma unroll
                for (int s = 0; s < KW; ++s) {
                    const int r = lane + 32 * s;
                    if (r < k)
                        acc[s] = fmaf(vl, frow[r], acc[s]);
                }
            }
        }
#pragma unroll
        for (int s = 0; s < KW; ++s) {
            const int r = lane + 32 * s;
            if (r < k)
                out[i * k + r] = acc[s];
        }
    }
}

// Rows of F gathered from beyond the L2 cache: a warp takes up to STREAM_ROWS
// consecutive rows, whose stored entries are one stretch, reads the entries 32
// at a time, the next 32 while these are used, and keeps STREAM_BATCH gathered
// rows in flight, in 24 to 32 warps per SM. The same sums in the same order as
// spmm_kernel. VEC = 2: k even and F, out 8-byte aligned; lane l owns columns
// 2 l + 64 s and the next (KW slots). VEC = 1: columns l + 32 s.
//
// Stretches of more than STREAM_HEAVY entries a row are left for the end and
// dealt out row by row, neighbouring ones to different warps: the long rows of a
// matrix often lie together (sorted by degree), and a warp with 16 of them kept
// the whole GPU waiting (1000 rows of 9000 entries side by side among 10^6 rows of
// one, k = 50: 18.4 ms, 1.3 so, 3.9 with spmm_kernel; without such rows the search
// for them costs 2 us of 480). As a function of its own, a heavy row takes no
// registers from the stretches (inlined: 483 to 950 us at k = 50 to 100).
constexpr int STREAM_ROWS = 16, STREAM_BATCH = 8, STREAM_HEAVY = 128;

// One row of the product, a warp to it.
template <int KW, int VEC>
__device__ __noinline__ void stream_row(const int64_t *__restrict__ rowptr,
                                        const int32_t *__restrict__ colidx,
                                        const float *__restrict__ vals, int64_t row,
                                        const float *__restrict__ F, int k, float *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    float acc[KW][VEC];
#pragma unroll
    for (int s = 0; s < KW; ++s)
#pragma unroll
        for (int e = 0; e < VEC; ++e)
            acc[s][e] = 0.0f;
    int64_t p = rowptr[row];
    const int64_t end = rowptr[row + 1];
    int cn = p + lane < end ? colidx[p + lane] : 0;
    float vn = p + lane < end ? vals[p + lane] : 0.0f;
    for (; p < end; p += 32) {
        const int c = cn;
        const float v = vn;
        const int64_t pn = p + 32 + lane;
        cn = pn < end ? colidx[pn] : 0;
        vn = pn < end ? vals[pn] : 0.0f;
        const int cnt = (int)min((int64_t)32, end - p);
        for (int l = 0; l < cnt;) {
            const int n = min(cnt - l, STREAM_BATCH);
            float f[STREAM_BATCH][KW][VEC], w[STREAM_BATCH];
#pragma unroll
            for (int q = 0; q < STREAM_BATCH; ++q)
                if (q < n) {
                    const int64_t cl = __shfl_sync(FULL, c, l + q);
                    w[q] = __shfl_sync(FULL, v, l + q);
                    const float *frow = F + cl * k;
#pragma unroll
                    for (int s = 0; s < KW; ++s) {
                        const int cc = VEC * (lane + 32 * s);
                        if constexpr (VEC == 2) {
                            const float2 t =
                                cc < k ? *reinterpret_cast<const float2 *>(frow + cc)
                                       : make_float2(0.0f, 0.0f);
                            f[q][s][0] = t.x;
                            f[q][s][1] = t.y;
                        } else {
                            f[q][s][0] = cc < k ? frow[cc] : 0.0f;
                        }
                    }
                }
#pragma unroll
            for (int q = 0; q < STREAM_BATCH; ++q)
                if (q < n)
#pragma unroll
                    for (int s = 0; s < KW; ++s)
#pragma unroll
                        for (int e = 0; e < VEC; ++e)
                            acc[s][e] = fmaf(w[q], f[q][s][e], acc[s][e]);
            l += n;
        }
    }
#pragma unroll
    for (int s = 0; s < KW; ++s) {
        const int c = VEC * (lane + 32 * s);
        if (c < k) {
            float *o = out + row * k + c;
            if constexpr (VEC == 2)
                *reinterpret_cast<float2 *>(o) = make_float2(acc[s][0], acc[s][1]);
            else
                *o = acc[s][0];
        }
    }
}

template <int KW, int VEC>
__global__ void __launch_bounds__(SPMM_THREADS)
    spmm_stream_kernel(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                       const float *__restrict__ vals, int64_t rows, const float *__restrict__ F,
                       int k, float *__restrict__ out, const int *__restrict__ mode_flag,
                       int chunk)
{
    if (mode_flag && *mode_flag == 0)
        return;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * SPMM_THREADS + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * SPMM_THREADS) >> 5;
    for (int64_t r0 = warp0 * chunk; r0 < rows; r0 += nw * chunk) {
        const int nr = (int)min((int64_t)chunk, rows - r0);
        const int64_t rp = rowptr[r0 + min(lane, nr)];   // lane l: the start of row r0 + l
        const int64_t end = __shfl_sync(FULL, rp, nr);
        if (chunk > 1 && end - __shfl_sync(FULL, rp, 0) > STREAM_HEAVY * chunk)
            continue;   // (dealt out below)
        float acc[KW][VEC];
#pragma unroll
        for (int s = 0; s < KW; ++s)
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                acc[s][e] = 0.0f;
        int r = 0;
        int64_t p = __shfl_sync(FULL, rp, 0), rend = __shfl_sync(FULL, rp, 1);
        auto put_row = [&]() {   // row r is complete
#pragma unroll
            for (int s = 0; s < KW; ++s) {
                const int c = VEC * (lane + 32 * s);
                if (c < k) {
                    float *o = out + (r0 + r) * k + c;
                    if constexpr (VEC == 2)
                        *reinterpret_cast<float2 *>(o) = make_float2(acc[s][0], acc[s][1]);
                    else
                        *o = acc[s][0];
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e)
                    acc[s][e] = 0.0f;
            }
            ++r;
            rend = __shfl_sync(FULL, rp, min(r + 1, nr));
        };
        int c = 0, cn = 0;
        float v = 0.0f, vn = 0.0f;
        if (p + lane < end) {
            cn = colidx[p + lane];
            vn = vals[p + lane];
        }
        while (p < end) {
            c = cn;
            v = vn;
            const int64_t pn = p + 32 + lane;
            cn = pn < end ? colidx[pn] : 0;
            vn = pn < end ? vals[pn] : 0.0f;
            const int cnt = (int)min((int64_t)32, end - p);
            for (int l = 0; l < cnt;) {
                while (r < nr && rend <= p + l)
                    put_row();
                if (r == nr)
                    break;
                const int n = (int)min((int64_t)min(cnt - l, STREAM_BATCH), rend - (p + l));
                float f[STREAM_BATCH][KW][VEC], w[STREAM_BATCH];
#pragma unroll
                for (int q = 0; q < STREAM_BATCH; ++q)
                    if (q < n) {
                        const int64_t cl = __shfl_sync(FULL, c, l + q);
                        w[q] = __shfl_sync(FULL, v, l + q);
                        const float *frow = F + cl * k;
#pragma unroll
                        for (int s = 0; s < KW; ++s) {
                            const int cc = VEC * (lane + 32 * s);
                            if constexpr (VEC == 2) {
                                const float2 t = cc < k
                                                     ? *reinterpret_cast<const float2 *>(frow + cc)
                                                     : make_float2(0.0f, 0.0f);
                                f[q][s][0] = t.x;
                                f[q][s][1] = t.y;
                            } else {
                                f[q][s][0] = cc < k ? frow[cc] : 0.0f;
                            }
                        }
                    }
#pragma unroll
                for (int q = 0; q < STREAM_BATCH; ++q)
                    if (q < n)
#pragma unroll
                        for (int s = 0; s < KW; ++s)
#pragma unroll
                            for (int e = 0; e < VEC; ++e)
                                acc[s][e] = fmaf(w[q], f[q][s][e], acc[s][e]);
                l += n;
            }
            p += 32;
        }
        while (r < nr)
            put_row();
    }
    if (chunk == 1)
        return;
    // The heavy stretches: warp j of a group of `chunk` warps takes row j of each
    // of them among the group's (every groups-th).
    const int64_t group = warp0 / chunk, groups = nw / chunk;
    const int j = (int)(warp0 - group * chunk);
    if (group >= groups)
        return;
    for (int64_t c0 = group; c0 * chunk < rows; c0 += 32 * groups) {
        const int64_t a = min((c0 + lane * groups) * chunk, rows);
        unsigned todo = __ballot_sync(
            FULL, rowptr[min(a + chunk, rows)] - rowptr[a] > STREAM_HEAVY * chunk);
        for (; todo; todo &= todo - 1) {
            const int64_t row = (c0 + (__ffs(todo) - 1) * groups) * chunk + j;
            if (row >= rows)
                continue;
            stream_row<KW, VEC>(rowptr, colidx, vals, row, F, k, out);
        }
    }
}

__global__ void count_cols_kernel(const int32_t *__restrict__ colidx, int64_t nnz,
                                  unsigned long long *__restrict__ counts)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz;
         p += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&counts[colidx[p] + 1], 1ull);
}

// In-place inclusive scan of counts[0..len) by one CTA of 1024 threads,
// walking 1024-element chunks with a running carry (init-time only).
__global__ void __launch_bounds__(1024) scan_kernel(unsigned long long *__restrict__ a, int64_t len)
{
    __shared__ unsigned long long buf[1024];
    __shared__ unsigned long long carry;
    if (threadIdx.x == 0)
        carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < len; base += 1024) {
        const int64_t i = base + threadIdx.x;
        buf[threadIdx.x] = i < len ? a[i] : 0ull;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {
            const unsigned long long v = threadIdx.x >= o ? buf[threadIdx.x - o] : 0ull;
            __syncthreads();
            buf[threadIdx.x] += v;
            __syncthreads();
        }
        if (i < len)
            a[i] = buf[threadIdx.x] + carry;
        __syncthreads();
        if (threadIdx.x == 1023)
            carry += buf[1023];
        __syncthreads();
    }
}

__global__ void scatter_kernel(const int64_t *__restrict__ rowptr,
                               const int32_t *__restrict__ colidx, const float *__restrict__ vals,
                               int64_t m, unsigned long long *__restrict__ cursor,
                               int32_t *__restrict__ t_colidx, float *__restrict__ t_vals)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x)
        for (int64_t p = rowptr[i]; p < rowptr[i + 1]; ++p) {
            const unsigned long long pos = atomicAdd(&cursor[colidx[p]], 1ull);
            t_colidx[pos] = (int32_t)i;
            t_vals[pos] = vals[p];
        }
}

__global__ void sort_rows_kernel(const int64_t *__restrict__ t_rowptr, int64_t n,
                                 int32_t *__restrict__ t_colidx, float *__restrict__ t_vals)
{
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = t_rowptr[j], e = t_rowptr[j + 1];
        for (int64_t p = b + 1; p < e; ++p) {
            const int32_t c = t_colidx[p];
            const float v = t_vals[p];
            int64_t q = p - 1;
            while (q >= b && t_colidx[q] > c) {
                t_colidx[q + 1] = t_colidx[q];
                t_vals[q + 1] = t_vals[q];
                --q;
            }
            t_colidx[q + 1] = c;
            t_vals[q + 1] = v;
        }
    }
}

}  // namespace

namespace {

double l2_bytes()
{
    static const double bytes = [] {   // (initialised once, whatever the threads)
        int dev = 0, b = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&b, cudaDevAttrL2CacheSize, dev);
        return b > 0 ? (double)b : 1.0;
    }();
    return bytes;
}

// cols: the rows of F.
nmf_status spmm_launch(const int64_t *rowptr, const int32_t *colidx, const float *vals,
                       int64_t rows, int64_t cols, const float *F, int k, float *out,
                       const int *mode_flag, cudaStream_t s)
{
    if (rows == 0)
        return NMF_OK;
    const int64_t frows = cols < 0 ? 0 : cols;
    if ((double)frows * k * sizeof(float) > 0.9 * l2_bytes()) {
        const bool pairs = k % 2 == 0 && ((reinterpret_cast<uintptr_t>(F) |
                                           reinterpret_cast<uintptr_t>(out)) & 7) == 0;
        const int kw = (int)cdiv(k, pairs ? 64 : 32);
        auto kernel = pairs ? (kw == 1 ? spmm_stream_kernel<1, 2> : spmm_stream_kernel<2, 2>)
                      : kw == 1 ? spmm_stream_kernel<1, 1>
                      : kw == 2 ? spmm_stream_kernel<2, 1>
                      : kw == 3 ? spmm_stream_kernel<3, 1>
                                : spmm_stream_kernel<4, 1>;
        int per_sm = 0;
        NMF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, SPMM_THREADS, 0));
        const int64_t most = (int64_t)(per_sm > 0 ? per_sm : 1) * sm_count();
        // Chunks of STREAM_ROWS rows, shorter where that leaves warps without
        // one.
        const int64_t warps = most * (SPMM_THREADS / 32), share = rows / (2 * warps);
        const int chunk = (int)(share < 1 ? 1 : share < STREAM_ROWS ? share : STREAM_ROWS);
        const int64_t want = cdiv(cdiv(rows, chunk) * 32, SPMM_THREADS);
        kernel<<<(unsigned)(want < most ? want : most), SPMM_THREADS, 0, s>>>(
            rowptr, colidx, vals, rows, F, k, out, mode_flag, chunk);
        NMF_LAUNCHED("spmm_stream_kernel");
        return NMF_OK;
    }
    int64_t blocks = cdiv(rows * 32, SPMM_THREADS);
    const int64_t cap = 16LL * sm_count();
    if (blocks > cap)
        blocks = cap;
    const unsigned g = (unsigned)blocks;
    if (k <= 32)
        spmm_kernel<1><<<g, SPMM_THREADS, 0, s>>>(rowptr, colidx, vals, rows, F, k, out, mode_flag);
    else if (k <= 64)
        spmm_kernel<2><<<g, SPMM_THREADS, 0, s>>>(rowptr, colidx, vals, rows, F, k, out, mode_flag);
    else if (k <= 96)
        spmm_kernel<3><<<g, SPMM_THREADS, 0, s>>>(rowptr, colidx, vals, rows, F, k, out, mode_flag);
    else
        spmm_kernel<4><<<g, SPMM_THREADS, 0, s>>>(rowptr, colidx, vals, rows, F, k, out, mode_flag);
    NMF_LAUNCHED("spmm_kernel");
    return NMF_OK;
}
}  // namespace

nmf_status launch_spmm(const int64_t *rowptr, const int32_t *colidx, const float *vals,
                       int64_t rows, int64_t cols, const float *F, int k, float *out,
                       cudaStream_t s)
{
    return spmm_launch(rowptr, colidx, vals, rows, cols, F, k, out, nullptr, s);
}

nmf_status launch_spmm_unless_fp32(const int64_t *rowptr, const int32_t *colidx,
                                   const float *vals, int64_t rows, int64_t cols,
                                   const float *F, int k, float *out, const int *mode_flag,
                                   cudaStream_t s)
{
    return spmm_launch(rowptr, colidx, vals, rows, cols, F, k, out, mode_flag, s);
}

nmf_status launch_csr_transpose(const int64_t *rowptr, const int32_t *colidx, const float *vals,
                                int64_t m, int64_t n, int64_t nnz, int64_t *t_rowptr,
                                int32_t *t_colidx, float *t_vals,
                                unsigned long long *cursor, cudaStream_t s)
{
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(t_rowptr);
    NMF_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int64_t) * (size_t)(n + 1), s));
    const unsigned g = (unsigned)(4 * sm_count());
    if (nnz > 0) {
        count_cols_kernel<<<g, 256, 0, s>>>(colidx, nnz, cnt);
        NMF_LAUNCHED("count_cols_kernel");
    }
    scan_kernel<<<1, 1024, 0, s>>>(cnt, n + 1);
    NMF_LAUNCHED("scan_kernel");
    if (n > 0)
        NMF_CUDA(cudaMemcpyAsync(cursor, cnt, sizeof(int64_t) * (size_t)n,
                                 cudaMemcpyDeviceToDevice, s));
    if (m > 0 && nnz > 0) {
        scatter_kernel<<<g, 256, 0, s>>>(rowptr, colidx, vals, m, cursor, t_colidx, t_vals);
        NMF_LAUNCHED("scatter_kernel");
        sort_rows_kernel<<<g, 256, 0, s>>>(t_rowptr, n, t_colidx, t_vals);
        NMF_LAUNCHED("sort_rows_kernel");
    }
    return NMF_OK;
}

}  // namespace nmf
