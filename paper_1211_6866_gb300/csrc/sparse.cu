// sparse.cu -- device-wide scan, CSC validation, CSC->CSR transpose and the
// multi-right-hand-side CSR SpMM used by every Krylov iteration.
#include <stdio.h>

#include "internal.h"

// ------------------------------------------------------------------ buffers
sai_status Buf::alloc(size_t nbytes, cudaStream_t s, bool use_async)
{
    release();
    st = s;
    async = use_async;
    bytes = nbytes;
    dev = -1;
    if (nbytes == 0) return SAI_OK;
    const cudaMemPool_t pool = !use_async && nbytes <= HANDLE_POOL_MAX ? sai_handle_pool() : nullptr;
    int d = -1;
    if (pool && cudaGetDevice(&d) != cudaSuccess) return SAI_CUDA_ERROR;
    cudaError_t e = use_async ? cudaMallocAsync(&p, nbytes, s)
                    : pool    ? cudaMallocFromPoolAsync(&p, nbytes, pool, s)
                              : cudaMalloc(&p, nbytes);
    if (e == cudaSuccess) dev = d;
    if (e != cudaSuccess) {
        p = nullptr;
        (void)cudaGetLastError();  // the status carries it: a caller may go on without the buffer
        sai_internal_note_cuda_error(e, "device allocation", __FILE__, __LINE__);
        return e == cudaErrorMemoryAllocation ? SAI_OOM : SAI_CUDA_ERROR;
    }
    return SAI_OK;
}

void Buf::release()
{
    if (p && async) {
        cudaFreeAsync(p, st);
    } else if (p && dev >= 0) {
        int cur = -1;
        const bool other = cudaGetDevice(&cur) == cudaSuccess && cur != dev && cudaSetDevice(dev) == cudaSuccess;
        cudaFreeAsync(p, st);  // chosen by free_on
        if (other) cudaSetDevice(cur);
    } else if (p) {
        cudaFree(p);
    }
    p = nullptr;
    bytes = 0;
    dev = -1;
}

cudaStream_t sai_free_stream()
{
    static std::mutex mu;
    static cudaStream_t streams[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    if (!streams[dev] && cudaStreamCreateWithFlags(&streams[dev], cudaStreamNonBlocking) != cudaSuccess) {
        (void)cudaGetLastError();
        streams[dev] = nullptr;
    }
    return streams[dev];
}

cudaMemPool_t sai_handle_pool()
{
    static std::mutex mu;
    static cudaMemPool_t pools[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || !sai_free_stream()) return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    if (!pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        uint64_t keep = HANDLE_POOL_KEEP;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) == cudaSuccess &&
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess)
            pools[dev] = pool;
        else if (pool)
            cudaMemPoolDestroy(pool);
        (void)cudaGetLastError();
    }
    return pools[dev];
}

void HandleUses::record(cudaStream_t s)
{
    cudaStreamCaptureStatus cs;
    if (cudaStreamIsCapturing(s, &cs) != cudaSuccess) {
        (void)cudaGetLastError();
        return;
    }
    if (cs != cudaStreamCaptureStatusNone) return;
    std::lock_guard<std::mutex> lk(mu);
    int q = 0;
    while (q < cnt && st[q] != s) ++q;
    bool ok = true;
    if (q == cnt && cnt < MAX) {
        ok = (dev >= 0 || cudaGetDevice(&dev) == cudaSuccess) &&
             cudaEventCreateWithFlags(&ev[q], cudaEventDisableTiming) == cudaSuccess;
        if (ok) ++cnt;
    } else {
        // the event moves on to this use and stays behind its earlier ones: of
        // another stream (the table is full, or a new stream has an old one's
        // handle) or of this one, for which the wait is nothing
        if (q == cnt) q = MAX - 1;
        ok = cudaStreamWaitEvent(s, ev[q], 0) == cudaSuccess;
    }
    if (ok) {
        st[q] = s;
        ok = cudaEventRecord(ev[q], s) == cudaSuccess;
    }
    if (!ok) {
        (void)cudaGetLastError();
        cudaStreamSynchronize(s);
    }
}

cudaStream_t HandleUses::before_free(const Buf& b)
{
    if (b.async) return nullptr;  // no handle: a call's own buffers
    const int d = b.dev >= 0 ? b.dev : dev;
    int cur = -1;
    const bool other = d >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != d && cudaSetDevice(d) == cudaSuccess;
    cudaStream_t f = nullptr;
    // not the legacy stream while one that it would wait for captures
    cudaStreamCaptureStatus cs;
    if ((b.st != nullptr && b.st != cudaStreamLegacy) || cudaStreamIsCapturing(nullptr, &cs) != cudaSuccess ||
        cs != cudaStreamCaptureStatusNone)
        f = sai_free_stream();
    for (int q = 0; q < cnt; ++q) {
        if (cudaStreamWaitEvent(f, ev[q], 0) != cudaSuccess) cudaEventSynchronize(ev[q]);
        cudaEventDestroy(ev[q]);
    }
    (void)cudaGetLastError();
    cnt = 0;
    if (other) cudaSetDevice(cur);
    return f;
}

// ------------------------------------------------------------------ scan
// Three passes: per-tile sums, one-block scan of the tile sums, per-tile scan.
#define SCAN_THREADS 512
#define SCAN_ITEMS 8
#define SCAN_TILE (SCAN_THREADS * SCAN_ITEMS)

__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* sh, int64_t* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(SAI_FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < nw ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(SAI_FULL, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) sh[lane] = w;
    }
    __syncthreads();
    int64_t off = warp > 0 ? sh[warp - 1] : 0;
    *total = sh[nw - 1];
    __syncthreads();
    return off + x - v;
}

template <class T>
__global__ void k_scan_tilesum(const T* in, int64_t n, int64_t* tsum)
{
    __shared__ int64_t sh[32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int64_t s = 0;
#pragma unroll
    for (int q = 0; q < SCAN_ITEMS; ++q)
        if (base + q < n) s += (int64_t)in[base + q];
    int64_t tot;
    block_exclusive_scan(s, sh, &tot);
    if (threadIdx.x == 0) tsum[blockIdx.x] = tot;
}

__global__ void k_scan_tiles(int64_t* tsum, int64_t ntiles)
{
    __shared__ int64_t sh[32];
    int64_t carry = 0;
    for (int64_t base = 0; base < ntiles; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        int64_t v = i < ntiles ? tsum[i] : 0;
        int64_t tot;
        int64_t ex = block_exclusive_scan(v, sh, &tot);
        if (i < ntiles) tsum[i] = carry + ex;
        carry += tot;
    }
}

template <class T>
__global__ void k_scan_apply(const T* in, int64_t n, const int64_t* toff, int64_t* out)
{
    __shared__ int64_t sh[32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int64_t vals[SCAN_ITEMS];
    int64_t s = 0;
#pragma unroll
    for (int q = 0; q < SCAN_ITEMS; ++q) {
        vals[q] = (base + q < n) ? (int64_t)in[base + q] : 0;
        s += vals[q];
    }
    int64_t tot;
    int64_t ex = block_exclusive_scan(s, sh, &tot) + toff[blockIdx.x];
#pragma unroll
    for (int q = 0; q < SCAN_ITEMS; ++q) {
        if (base + q < n) out[base + q] = ex;
        ex += vals[q];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) out[n] = toff[blockIdx.x] + tot;
}

template <class T>
static sai_status scan_counts(const T* in, int64_t* out, int64_t n, cudaStream_t st)
{
    int64_t ntiles = n > 0 ? (n + SCAN_TILE - 1) / SCAN_TILE : 1;
    Buf tsum;
    SAI_TRY(tsum.alloc(sizeof(int64_t) * ntiles, st, true));
    k_scan_tilesum<T><<<SAI_GRID((unsigned)ntiles), SCAN_THREADS, 0, st>>>(in, n, tsum.as<int64_t>());
    k_scan_tiles<<<SAI_GRID(1), 1024, 0, st>>>(tsum.as<int64_t>(), ntiles);
    k_scan_apply<T><<<SAI_GRID((unsigned)ntiles), SCAN_THREADS, 0, st>>>(in, n, tsum.as<int64_t>(), out);
    SAI_CUDA(cudaGetLastError());
    return SAI_OK;
}

sai_status sai_scan_counts_i32(const int32_t* in, int64_t* out, int64_t n, cudaStream_t st)
{
    return scan_counts<int32_t>(in, out, n, st);
}
sai_status sai_scan_counts_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t st)
{
    return scan_counts<int64_t>(in, out, n, st);
}

// ------------------------------------------------------------------ validate
// one warp per column: the column's bounds, every row index in range and
// each one above its predecessor
__global__ void k_validate_csc(int32_t nrows, int32_t ncols, int64_t nnz, const int64_t* cp, const int32_t* ri,
                               int* bad)
{
    const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= ncols) return;
    const int64_t b = cp[j], e = cp[j + 1];
    if (lane == 0) {
        if (j == 0 && b != 0) atomicOr(bad, 1);
        if (j == ncols - 1 && e != nnz) atomicOr(bad, 2);
    }
    if (e < b || b < 0 || e > nnz) {
        if (lane == 0) atomicOr(bad, 4);
        return;
    }
    bool ok = true;
    for (int64_t t0 = b + lane; t0 < e; t0 += 32 * 4) {
        int32_t i[4], nx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t t = t0 + 32 * u;
            i[u] = t < e ? ri[t] : 0;
            nx[u] = t + 1 < e ? ri[t + 1] : INT32_MAX;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t t = t0 + 32 * u;
            if (t < e && (i[u] < 0 || i[u] >= nrows || nx[u] <= i[u])) ok = false;
        }
    }
    if (!__all_sync(SAI_FULL, ok) && lane == 0) atomicOr(bad, 8);
}

sai_status sai_validate_csc(int32_t nrows, int32_t ncols, int64_t nnz, const int64_t* cp, const int32_t* ri,
                            cudaStream_t st)
{
    if (ncols == 0) return SAI_OK;
    Buf bad;
    SAI_TRY(bad.alloc(sizeof(int), st, true));
    SAI_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
    k_validate_csc<<<SAI_GRID(sai_div_up((int64_t)ncols * 32, 256)), 256, 0, st>>>(nrows, ncols, nnz, cp, ri,
                                                                                  bad.as<int>());
    SAI_CUDA(cudaGetLastError());
    int h = 0;
    SAI_CUDA(cudaMemcpyAsync(&h, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    SAI_CUDA(cudaStreamSynchronize(st));
    return h ? SAI_INVALID_ARG : SAI_OK;
}

// ------------------------------------------------------------------ transpose
__global__ void k_row_hist(int64_t nnz, const int32_t* ri, int32_t* cnt)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nnz; t += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[ri[t]], 1);
}

// One warp per column: scatter the column's entries into their rows' segments.
__global__ void k_scatter_rows(int32_t ncols, const int64_t* cp, const int32_t* ri, const double* cv,
                               int64_t* fill, int32_t* tci, double* tv)
{
    int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (w >= ncols) return;
    for (int64_t t = cp[w] + lane; t < cp[w + 1]; t += 32) {
        unsigned long long q = atomicAdd((unsigned long long*)&fill[ri[t]], 1ull);
        tci[q] = (int32_t)w;
        tv[q] = cv[t];
    }
}

// One warp per row: rank sort of the (unique) column indices of the row.
__global__ void k_sort_rows(int32_t nrows, const int64_t* rp, const int32_t* tci, const double* tv, int32_t* ci,
                            double* v)
{
    int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (w >= nrows) return;
    int64_t b = rp[w], e = rp[w + 1];
    for (int64_t t = b + lane; t < e; t += 32) {
        int32_t c = tci[t];
        int64_t rank = 0;
        for (int64_t u = b; u < e; ++u) rank += (tci[u] < c);
        ci[b + rank] = c;
        v[b + rank] = tv[t];
    }
}

sai_status sai_csc_to_csr(int32_t nrows, int32_t ncols, int64_t nnz, const int64_t* cp, const int32_t* ri,
                          const double* cv, Buf& rp, Buf& ci, Buf& rv, cudaStream_t st, bool mode_async)
{
    SAI_TRY(rp.alloc(sizeof(int64_t) * ((size_t)nrows + 1), st, mode_async));
    SAI_TRY(ci.alloc(sizeof(int32_t) * (size_t)nnz, st, mode_async));
    SAI_TRY(rv.alloc(sizeof(double) * (size_t)nnz, st, mode_async));
    Buf cnt, fill, tci, tv;
    SAI_TRY(cnt.alloc(sizeof(int32_t) * ((size_t)nrows + 1), st, true));
    SAI_TRY(fill.alloc(sizeof(int64_t) * ((size_t)nrows + 1), st, true));
    SAI_TRY(tci.alloc(sizeof(int32_t) * (size_t)nnz, st, true));
    SAI_TRY(tv.alloc(sizeof(double) * (size_t)nnz, st, true));
    SAI_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int32_t) * ((size_t)nrows + 1), st));
    if (nnz > 0) {
        unsigned g = sai_div_up(nnz, 256);
        if (g > 152 * 64) g = 152 * 64;
        k_row_hist<<<SAI_GRID(g), 256, 0, st>>>(nnz, ri, cnt.as<int32_t>());
    }
    SAI_TRY(sai_scan_counts_i32(cnt.as<int32_t>(), rp.as<int64_t>(), nrows, st));
    SAI_CUDA(cudaMemcpyAsync(fill.p, rp.p, sizeof(int64_t) * ((size_t)nrows + 1), cudaMemcpyDeviceToDevice, st));
    if (ncols > 0)
        k_scatter_rows<<<SAI_GRID(sai_div_up((int64_t)ncols * 32, 256)), 256, 0, st>>>(ncols, cp, ri, cv, fill.as<int64_t>(),
                                                                         tci.as<int32_t>(), tv.as<double>());
    if (nrows > 0)
        k_sort_rows<<<SAI_GRID(sai_div_up((int64_t)nrows * 32, 256)), 256, 0, st>>>(nrows, rp.as<int64_t>(), tci.as<int32_t>(),
                                                                         tv.as<double>(), ci.as<int32_t>(),
                                                                         rv.as<double>());
    SAI_CUDA(cudaGetLastError());
    return SAI_OK;
}

// ------------------------------------------------------------------ SpMM
// Lane groups of G = next power of two >= k (capped at 32) own one row each;
// lane c of a group accumulates column c (and c+32, ... when k > 32). The
// k values of a row of X are contiguous, so each gathered row is one
// coalesced segment.
template <int G, int MODE>
__global__ void __launch_bounds__(256) k_spmm(int32_t n, const int64_t* __restrict__ rp,
                                              const int32_t* __restrict__ ci, const double* __restrict__ v,
                                              int32_t k, const double* __restrict__ X, double* __restrict__ Y,
                                              const double* __restrict__ B)
{
    constexpr int RPW = 32 / G;  // rows per warp
    const int lane = threadIdx.x & 31;
    const int sub = lane / G, c0 = lane % G;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t row0 = warp * RPW; row0 < n; row0 += nwarps * RPW) {
        int64_t row = row0 + sub;
        if (row >= n) continue;
        int64_t b = rp[row], e = rp[row + 1];
        for (int c = c0; c < k; c += G) {
            double acc = 0.0;
            for (int64_t t = b; t < e; ++t) acc = fma(v[t], X[(int64_t)ci[t] * k + c], acc);
            if (MODE == 0) Y[row * k + c] = acc;
            else Y[row * k + c] = B[row * k + c] - acc;
        }
    }
}

template <int MODE>
static void launch_spmm(int32_t n, const int64_t* rp, const int32_t* ci, const double* v, int32_t k,
                        const double* X, double* Y, const double* B, cudaStream_t st)
{
    int G = 1;
    while (G < k && G < 32) G <<= 1;
    int rpw = 32 / G;
    int64_t warps = (n + rpw - 1) / rpw;
    int64_t blocks = (warps * 32 + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    if (blocks < 1) blocks = 1;
    switch (G) {
    case 1: k_spmm<1, MODE><<<SAI_GRID((unsigned)blocks), 256, 0, st>>>(n, rp, ci, v, k, X, Y, B); break;
    case 2: k_spmm<2, MODE><<<SAI_GRID((unsigned)blocks), 256, 0, st>>>(n, rp, ci, v, k, X, Y, B); break;
    case 4: k_spmm<4, MODE><<<SAI_GRID((unsigned)blocks), 256, 0, st>>>(n, rp, ci, v, k, X, Y, B); break;
    case 8: k_spmm<8, MODE><<<SAI_GRID((unsigned)blocks), 256, 0, st>>>(n, rp, ci, v, k, X, Y, B); break;
    case 16: k_spmm<16, MODE><<<SAI_GRID((unsigned)blocks), 256, 0, st>>>(n, rp, ci, v, k, X, Y, B); break;
    default: k_spmm<32, MODE><<<SAI_GRID((unsigned)blocks), 256, 0, st>>>(n, rp, ci, v, k, X, Y, B); break;
    }
}

sai_status sai_spmm(int32_t n, const int64_t* rp, const int32_t* ci, const double* v, int32_t k, const double* X,
                    double* Y, const double* B, int mode, cudaStream_t st)
{
    if (n == 0 || k == 0) return SAI_OK;
    if (mode == 0) launch_spmm<0>(n, rp, ci, v, k, X, Y, B, st);
    else launch_spmm<1>(n, rp, ci, v, k, X, Y, B, st);
    SAI_CUDA(cudaGetLastError());
    return SAI_OK;
}

// ------------------------------------------------------------------ residual norms with A in CSC
// Pass 1 scatters A x into y with a warp per column (atomic adds, fixed grid);
// to stay deterministic the product is instead formed by a CSR copy in the
// callers that need bit-stable results. This helper is only used for the
// final rr check, where a last-bit variation is irrelevant.
__global__ void k_csc_axpy(int32_t n, const int64_t* cp, const int32_t* ri, const double* cv, const double* x,
                           double* y)
{
    int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (w >= n) return;
    const double xj = x[w];
    const int64_t e = cp[w + 1];
    for (int64_t t0 = cp[w] + lane; t0 < e; t0 += 32 * 8) {  // eight entries in flight per lane
        int32_t r[8];
        double a[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t t = t0 + 32 * u;
            r[u] = t < e ? ri[t] : 0;
            a[u] = t < e ? cv[t] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (t0 + 32 * u < e) atomicAdd(&y[r[u]], a[u] * xj);
    }
}

__global__ void k_resid_norms(int32_t n, const double* b, const double* ax, double* out)
{
    __shared__ double sh[2][32];
    double s0 = 0.0, s1 = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double d = b[i] - ax[i];
        s0 += d * d;
        s1 += b[i] * b[i];
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sh[0][wid] = s0;
        sh[1][wid] = s1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, c = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
            a += sh[0][q];
            c += sh[1][q];
        }
        out[2 * blockIdx.x] = a;
        out[2 * blockIdx.x + 1] = c;
    }
}

// Fixed-order sum of the per-block partial pairs (one warp).
__global__ void k_sum_pairs(const double* part, int nb, double* out)
{
    double a = 0.0, c = 0.0;
    for (int q = threadIdx.x; q < nb; q += 32) {
        a += part[2 * q];
        c += part[2 * q + 1];
    }
    a = warp_sum(a);
    c = warp_sum(c);
    if (threadIdx.x == 0) {
        out[0] = a;
        out[1] = c;
    }
}

sai_status sai_csc_residual_norms(int32_t n, const int64_t* cp, const int32_t* ri, const double* cv,
                                  const double* b, const double* x, double* out2_host, cudaStream_t st)
{
    Buf ax, part;
    const int nb = 152 * 4;
    SAI_TRY(ax.alloc(sizeof(double) * (size_t)(n > 0 ? n : 1), st, true));
    SAI_TRY(part.alloc(sizeof(double) * (2 * nb + 2), st, true));
    SAI_CUDA(cudaMemsetAsync(ax.p, 0, sizeof(double) * (size_t)n, st));
    if (n > 0) k_csc_axpy<<<SAI_GRID(sai_div_up((int64_t)n * 32, 256)), 256, 0, st>>>(n, cp, ri, cv, x, ax.as<double>());
    k_resid_norms<<<SAI_GRID(nb), 256, 0, st>>>(n, b, ax.as<double>(), part.as<double>());
    k_sum_pairs<<<SAI_GRID(1), 32, 0, st>>>(part.as<double>(), nb, part.as<double>() + 2 * nb);
    SAI_CUDA(cudaGetLastError());
    SAI_CUDA(cudaMemcpyAsync(out2_host, part.as<double>() + 2 * nb, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    SAI_CUDA(cudaStreamSynchronize(st));
    return SAI_OK;
}
