// sorted_rows.cuh -- a CSR matrix as slices of 32 rows of nearly equal length.
//
// A lane per CSR row takes a memory transaction per lane and entry, and the
// lanes of a warp wait (and, on the FP64 pipe, pay) for its longest row. Here
// the rows of each block are sorted by length, the longest first, and stored
// column-major in slices of 32; position i of a block holds its row ord[i]
// (-1: none). A row's entries keep their order, so its sum does too. Included
// inside the anonymous namespace of the file that uses it.

// Blocks of R rows (a multiple of 32): consecutive rows of an order-n matrix,
// or (first row, rows, column subtracted from the indices, 0) per block.
struct RowBlocks {
    int n, R;
    const int4* tab;
    __device__ int4 operator()(int b) const
    {
        return tab ? tab[b] : make_int4(b * R, max(0, min(R, n - b * R)), 0, 0);
    }
};

__global__ void __launch_bounds__(512) k_sorted_order(RowBlocks Q, const int64_t* __restrict__ rp, int32_t* ord,
                                                      int64_t* __restrict__ cnt)
{
    constexpr int NB = 1024;  // bins by length, the longest first
    __shared__ int off[NB];
    __shared__ int ws[16];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int4 bl = Q((int)blockIdx.x);
    const int base = bl.x, nrow = bl.y;
    const int64_t at = (int64_t)blockIdx.x * Q.R;
    auto bin = [&](int r) {  // steps of 96 from 512 entries on
        const int len = (int)(rp[base + r + 1] - rp[base + r]);
        return NB - 1 - min(NB - 1, len < 512 ? len : 512 + (len - 512) / 96);
    };
    for (int i = tid; i < NB; i += 512) off[i] = 0;
    for (int i = tid; i < Q.R; i += 512) ord[at + i] = -1;
    __syncthreads();
    for (int r = tid; r < nrow; r += 512) atomicAdd(&off[bin(r)], 1);
    __syncthreads();
    // exclusive prefix over the bins, two per thread
    const int c0 = off[2 * tid], c1 = off[2 * tid + 1];
    int incl = c0 + c1;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(SAI_FULL, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) ws[wid] = incl;
    __syncthreads();
    int before = incl - c0 - c1;
    for (int w = 0; w < wid; ++w) before += ws[w];
    off[2 * tid] = before;
    off[2 * tid + 1] = before + c0;
    __syncthreads();
    // rows of equal length land in any order: a row's product does not depend on its place
    for (int r = tid; r < nrow; r += 512) ord[at + atomicAdd(&off[bin(r)], 1)] = r;
    __syncthreads();
    for (int s = wid; s < Q.R / 32; s += 16) {
        const int r = ord[at + 32 * s + lane];
        const unsigned len = r >= 0 ? (unsigned)(rp[base + r + 1] - rp[base + r]) : 0u;
        const unsigned w = __reduce_max_sync(SAI_FULL, len);
        if (lane == 0) cnt[at / 32 + s] = (int64_t)w * 32;
    }
}

template <class T>
__global__ void k_sorted_fill(int nsl, RowBlocks Q, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                              const T* __restrict__ v, const int32_t* __restrict__ ord, const int64_t* __restrict__ sp,
                              int32_t* __restrict__ sci, T* __restrict__ sv)
{
    const int sl = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (sl >= nsl) return;
    const int4 bl = Q(sl / (Q.R / 32));
    const int r = ord[(int64_t)sl * 32 + lane];
    const int64_t b = sp[sl], w = (sp[sl + 1] - b) / 32;
    const int64_t r0 = r >= 0 ? rp[bl.x + r] : 0, len = r >= 0 ? rp[bl.x + r + 1] - r0 : 0;
#pragma unroll 4
    for (int64_t k = 0; k < w; ++k) {
        const int64_t q = b + k * 32 + lane;
        sci[q] = k < len ? ci[r0 + k] - bl.z : -1;  // not multiplied: its factor may be infinite
        sv[q] = k < len ? v[r0 + k] : T(0);
    }
}

// buf: ord (R per block), slice offsets (int64), columns, values. Waits once for the size.
template <class T>
sai_status sorted_rows(const RowBlocks& Q, int nblk, const int64_t* rp, const int32_t* ci, const T* v, Buf (&buf)[4],
                       cudaStream_t st)
{
    const int64_t nsl = (int64_t)nblk * (Q.R / 32);
    Buf cnt;
    SAI_TRY(cnt.alloc(sizeof(int64_t) * (size_t)nsl, st, true));
    SAI_TRY(buf[0].alloc(sizeof(int32_t) * (size_t)nsl * 32, st, true));
    SAI_TRY(buf[1].alloc(sizeof(int64_t) * ((size_t)nsl + 1), st, true));
    k_sorted_order<<<SAI_GRID(nblk), 512, 0, st>>>(Q, rp, buf[0].as<int32_t>(), cnt.as<int64_t>());
    SAI_TRY(sai_scan_counts_i64(cnt.as<int64_t>(), buf[1].as<int64_t>(), nsl, st));
    int64_t total = 0;
    SAI_CUDA(cudaMemcpyAsync(&total, buf[1].as<int64_t>() + nsl, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    SAI_CUDA(cudaStreamSynchronize(st));
    SAI_TRY(buf[2].alloc(sizeof(int32_t) * (size_t)(total > 0 ? total : 1), st, true));
    SAI_TRY(buf[3].alloc(sizeof(T) * (size_t)(total > 0 ? total : 1), st, true));
    k_sorted_fill<T><<<SAI_GRID(sai_div_up(nsl * 32, 256)), 256, 0, st>>>(
        (int)nsl, Q, rp, ci, v, buf[0].as<int32_t>(), buf[1].as<int64_t>(), buf[2].as<int32_t>(), buf[3].as<T>());
    SAI_CUDA(cudaGetLastError());
    return SAI_OK;
}
