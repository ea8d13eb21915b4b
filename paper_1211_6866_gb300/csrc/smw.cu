// smw.cu -- Sherman-Morrison-Woodbury recovery of x (Theorem 1; eq.
// (composi)): xhat = yhat - What (I + V^T What)^{-1} (V^T yhat), with
// V = [e_J0 .. e_J(s-1)], so V^T What is What(J,:) and V^T yhat is yhat(J).
//   k_smw_gather   C = I + What(J,:) (column-major s x s), g = yhat(J)
//   k_lu_solve     Gaussian elimination with partial pivoting (first largest
//                  |pivot| wins), one block; z = C^{-1} g, c = ||z|| (a blocked
//                  LU above LU_SMEM)
//   k_smw_update   xhat(i) = yhat(i) - sum_t What(i,t) z_t, one thread per row
// and its adjoint for A^T = A~^T + V U^T (the backward pass), where the small
// system is C = I + U^T What, g = U^T yhat (k_smw_gather_adj).
#include <math.h>

#include "internal.h"

namespace {

// |v| as an integer that orders like it (NaN below everything): pivot
// searches compare on the integer units, not on the FP64 pipe
__device__ __forceinline__ long long mag_bits(double v)
{
    const long long b = __double_as_longlong(v) & 0x7fffffffffffffffll;
    return b > 0x7ff0000000000000ll ? -1 : b;
}

// the largest key of the warp and its smallest row
__device__ __forceinline__ void warp_best(long long& key, int& row)
{
    for (int o = 16; o > 0; o >>= 1) {
        const long long ok = __shfl_xor_sync(SAI_FULL, key, o);
        const int orow = __shfl_xor_sync(SAI_FULL, row, o);
        if (ok > key || (ok == key && orow < row)) {
            key = ok;
            row = orow;
        }
    }
}

int g_smw_sms = 0;
int g_num_sms_smw()
{
    if (g_smw_sms == 0) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            g_smw_sms = v;
        else
            return 1;
    }
    return g_smw_sms;
}

__global__ void k_smw_gather(int32_t n, int32_t s, const int32_t* J, const double* Y, double* C, double* g)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)s * s) return;
    const int col = (int)(t / s), row = (int)(t - (int64_t)col * s);  // C(row, col)
    const int64_t ld = (int64_t)s + 1;
    C[(int64_t)col * s + row] = (row == col ? 1.0 : 0.0) + Y[(int64_t)J[row] * ld + 1 + col];
    if (col == 0) g[row] = Y[(int64_t)J[row] * ld];
}

// Adjoint form (A^T = A~^T + V U^T): C = I + U^T What (column-major s x s),
// g = U^T yhat. One warp per (row a of U^T, column b of Y), b = 0 is yhat.
__global__ void k_smw_gather_adj(int32_t s, const int64_t* Ucp, const int32_t* Uri, const double* Uv,
                                 const double* Y, double* C, double* g)
{
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= (int64_t)s * (s + 1)) return;
    const int a = (int)(w % s), b = (int)(w / s);
    const int64_t ld = (int64_t)s + 1;
    double acc = 0.0;
    for (int64_t q = Ucp[a] + lane; q < Ucp[a + 1]; q += 32) acc = fma(Uv[q], Y[(int64_t)Uri[q] * ld + b], acc);
    acc = warp_sum(acc);
    if (lane == 0) {
        if (b == 0) g[a] = acc;
        else C[(int64_t)(b - 1) * s + a] = (a == b - 1 ? 1.0 : 0.0) + acc;
    }
}

// Gaussian elimination with partial pivoting (the largest |pivot|, the first
// row on ties) and back substitution for s <= 1024 / 4 in one block. The
// matrix is worked on in shared memory when SMEM (ld = s | 1, s <= LU_SMEM),
// in place otherwise. A column costs two barriers: the multipliers, then one
// pass in which a warp per trailing column (g among them) swaps the pivot row
// in and updates it; the warp of the next column searches its pivot in the
// values it has just written. One warp does the back substitution with its
// rows in registers. (With a tree search, a swap and a thread per row, each
// behind barriers, s = 123 took 1.44 ms and s = 3 51 us; this form 0.57 ms and
// 9 us.)
constexpr int LU_T = 1024;
constexpr int LU_SMALL = 256;  // largest s of this kernel
constexpr int LU_SMEM = 160;   // largest s in shared memory (206 KB)
inline size_t lu_smem(int s) { return s <= LU_SMEM ? sizeof(double) * (size_t)s * (s | 1) : 0; }

template <bool SMEM>
__global__ void __launch_bounds__(LU_T) k_lu_solve(int32_t s, double* C, double* g, double* z, double* c_out, int* err)
{
    extern __shared__ double csm[];
    __shared__ double l[LU_SMALL], gs[LU_SMALL];
    __shared__ int piv_s;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int NW = LU_T / 32;
    const int ld = SMEM ? (s | 1) : s;
    double* A = SMEM ? csm : C;  // column j at A + j ld
    if (SMEM)
        for (int e = tid; e < s * s; e += LU_T) csm[(e / s) * ld + e % s] = C[e];
    for (int i = tid; i < s; i += LU_T) gs[i] = g[i];
    __syncthreads();
    if (wid == 0) {
        long long best = -1;
        int row = s;
        for (int i = lane; i < s; i += 32)
            if (mag_bits(A[i]) > best) {
                best = mag_bits(A[i]);
                row = i;
            }
        warp_best(best, row);
        if (lane == 0) piv_s = best > 0 ? row : -1;
    }
    __syncthreads();
    for (int k = 0; k < s; ++k) {
        const int p = piv_s;
        if (p < 0) {
            if (tid == 0) *err = 1;
            return;
        }
        double* ck = A + (size_t)k * ld;
        for (int i = k + 1 + tid; i < s; i += LU_T) l[i] = ck[i == p ? k : i] / ck[p];
        __syncthreads();
        if (tid == 0) ck[k] = ck[p];  // read as U(k, k) by the back substitution only
        for (int j = k + 1 + wid; j <= s; j += NW) {
            double* c = j < s ? A + (size_t)j * ld : gs;
            const double old = c[k], u = c[p];
            __syncwarp();
            long long best = -1;
            int row = s;
            for (int i = k + 1 + lane; i < s; i += 32) {
                const double v = fma(-l[i], u, i == p ? old : c[i]);
                c[i] = v;
                if (mag_bits(v) > best) {
                    best = mag_bits(v);
                    row = i;
                }
            }
            if (lane == 0) c[k] = u;
            if (j == k + 1 && j < s) {
                warp_best(best, row);
                if (lane == 0) piv_s = best > 0 ? row : -1;
            }
        }
        __syncthreads();
    }
    if (wid == 0) {
        // U z = g: lane keeps rows lane + 32 q; the pivots' reciprocals side by side
        constexpr int RPL = LU_SMALL / 32;
        double t[RPL], rd[RPL];
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q;
            t[q] = i < s ? gs[i] : 0.0;
            rd[q] = i < s ? 1.0 / A[(size_t)i * ld + i] : 0.0;
        }
        for (int j = s - 1; j >= 0; --j) {
            double zj = 0.0;
#pragma unroll
            for (int q = 0; q < RPL; ++q)
                if (j / 32 == q) {
                    if (lane == j % 32) t[q] = div_by(t[q], A[(size_t)j * ld + j], rd[q]);
                    zj = __shfl_sync(SAI_FULL, t[q], j % 32);
                }
#pragma unroll
            for (int q = 0; q < RPL; ++q) {
                const int i = lane + 32 * q;
                if (32 * q < j && i < j) t[q] = fma(-A[(size_t)j * ld + i], zj, t[q]);
            }
        }
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q;
            if (i < s) z[i] = t[q];
            acc = fma(t[q], t[q], acc);
        }
        acc = warp_sum(acc);
        if (lane == 0) *c_out = sqrt(acc);
    }
}

sai_status lu_small(int32_t s, double* C, double* g, double* z, double* c_out, int* err, cudaStream_t st)
{
    if (s <= LU_SMEM) {
        SAI_CUDA(sai_smem_limit(k_lu_solve<true>, lu_smem(LU_SMEM)));
        k_lu_solve<true><<<SAI_GRID(1), LU_T, lu_smem(s), st>>>(s, C, g, z, c_out, err);
    } else {
        k_lu_solve<false><<<SAI_GRID(1), LU_T, 0, st>>>(s, C, g, z, c_out, err);
    }
    return SAI_OK;
}

__global__ void k_smw_update(int32_t n, int32_t s, const double* Y, const double* z, double* x)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t ld = (int64_t)s + 1;
    const double* row = Y + i * ld;
    double v = row[0];
    for (int t = 0; t < s; ++t) v = fma(-row[1 + t], z[t], v);
    x[i] = v;
}


// ---------------------------------------------------------------- large s
// For s > LU_SMEM the s x s system is solved by a blocked right-looking LU
// with the same partial pivoting (largest |pivot|, the first row on ties),
// panels of LU_NB columns:
//   k_lu_panel   one block factors columns [k0, k0 + kb) over rows [k0, s)
//                (k_lu_panel_cluster, up to LU_CL LU_PROWS rows: one cluster)
//   k_lu_swap    applies the panel's interchanges to the other columns and g
//   k_lu_trsm    U12 = L11^{-1} A12, one thread per trailing column
//   k_lu_gemm    A22 -= L21 U12 on 64 x 64 tiles in FP64
//   k_lu_trsv    L y = Pg, U z = y in blocks of 32 rows, one cluster; c = ||z||
// After a zero pivot the panel sets *err and every later kernel returns
// without touching C, so no unwritten pivot index is ever read.
constexpr int LU_NB = 16;

// The panel over a cluster of blocks: each keeps PROWS of its rows in shared
// memory, row by row (17 values apart, the lanes of a warp in different
// banks), a thread per row. Per column every block sends its largest
// candidate row, and the owner of row j that row, to all blocks; after one
// cluster barrier each knows the pivot row, takes its part of the swap and
// updates its rows with the pivot's reciprocal, tracking the next column's
// largest value. One SM's FP64 pipe bounds a panel of many rows (s = 1051:
// 119 us in one block with the panel in global memory, 56 us over the cluster).
constexpr int LU_PLD = LU_NB + 1;
constexpr int LU_CL = 8;        // blocks per cluster
constexpr int LU_CT = 256;      // threads per block
constexpr int LU_PROWS = 1600;  // rows per block (218 KB)
constexpr size_t LU_PANEL_SMEM = sizeof(double) * LU_PROWS * LU_PLD;
// of the triangular solves, a value per row of a block: s up to 8 * 24576, whose matrix would take 309 GB
constexpr size_t LU_TRSV_SMEM = sizeof(double) * 24576;

__device__ __forceinline__ uint32_t smw_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t smw_map(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void smw_st(uint32_t a, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void smw_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __launch_bounds__(LU_CT) k_lu_panel_cluster(int32_t s, int32_t k0, int32_t kb, int rows, double* C,
                                                            int32_t* piv, int* err)
{
    extern __shared__ double P[];  // rows x LU_PLD
    // by column parity: every block's candidate (its 16 values, the key, the
    // row) and row j of the panel
    __shared__ double cand[2][LU_CL][LU_NB + 2], rowj[2][LU_NB];
    __shared__ long long wk[LU_CT / 32];
    __shared__ int wr[LU_CT / 32];
    __shared__ int best_s;
    if (*err) return;  // set by an earlier launch only: the same in every block
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int m = s - k0;
    const int b0 = (int)rank * rows, nr = max(0, min(rows, m - b0));  // this block's rows of the panel
    for (int c = 0; c < kb; ++c)
        for (int r = tid; r < nr; r += LU_CT) P[r * LU_PLD + c] = C[(int64_t)(k0 + c) * s + k0 + b0 + r];
    long long key = -1;
    int row = m;
    for (int r = tid; r < nr; r += LU_CT) {  // the rows this thread has written
        const long long a = mag_bits(P[r * LU_PLD]);
        if (a > key) {
            key = a;
            row = b0 + r;
        }
    }
    smw_cluster_sync();  // every block runs before its memory is written
    for (int j = 0; j < kb; ++j) {
        const int pb = j & 1;
        warp_best(key, row);
        if (lane == 0) {
            wk[wid] = key;
            wr[wid] = row;
        }
        __syncthreads();
        if (wid == 0) {
            key = lane < LU_CT / 32 ? wk[lane] : -1;
            row = lane < LU_CT / 32 ? wr[lane] : m;
            warp_best(key, row);
            if (lane == 0) {
                wk[0] = key;
                wr[0] = row;
            }
        }
        __syncthreads();
        key = wk[0];
        row = wr[0];
        {  // thread (block, value) sends one value of the candidate and of row j
            const int to = tid >> 5;
            if (lane < LU_NB + 2) {
                double v = 0.0;
                if (lane < LU_NB) v = key > 0 ? P[(row - b0) * LU_PLD + lane] : 0.0;
                else v = __longlong_as_double(lane == LU_NB ? key : (long long)row);
                smw_st(smw_map(smw_smem(&cand[pb][rank][lane]), (uint32_t)to), v);
            }
            if (j >= b0 && j < b0 + nr && lane < LU_NB)
                smw_st(smw_map(smw_smem(&rowj[pb][lane]), (uint32_t)to), P[(j - b0) * LU_PLD + lane]);
        }
        smw_cluster_sync();
        if (wid == 0) {
            long long bk = lane < LU_CL ? __double_as_longlong(cand[pb][lane][LU_NB]) : -1;
            int br = lane < LU_CL ? (int)__double_as_longlong(cand[pb][lane][LU_NB + 1]) : m;
            warp_best(bk, br);
            if (lane == 0) best_s = bk > 0 ? br : -1;
        }
        __syncthreads();
        const int p = best_s;
        if (p < 0) {  // the same in every block, none of which writes to another after this
            if (rank == 0 && tid == 0) *err = 1;
            break;
        }
        const int own = p / rows;  // the block of row p
        if (rank == 0 && tid == 0) piv[k0 + j] = k0 + p;
        const double* uj = cand[pb][own];
        // the swap: row p takes row j's values, row j the pivot row
        if (p != j && (int)rank == own && tid < kb) P[(p - b0) * LU_PLD + tid] = rowj[pb][tid];
        if (j >= b0 && j < b0 + nr && tid < kb) P[(j - b0) * LU_PLD + tid] = uj[tid];
        __syncthreads();
        double u[LU_NB];
#pragma unroll
        for (int c = 0; c < LU_NB; ++c) u[c] = uj[c];
        const double inv = 1.0 / uj[j];
        key = -1;
        row = m;
        for (int r = tid; r < nr; r += LU_CT) {
            if (b0 + r <= j) continue;
            double* x = P + r * LU_PLD;
            const double l = div_by(x[j], uj[j], inv);
            x[j] = l;
#pragma unroll
            for (int c = 1; c < LU_NB; ++c)
                if (c > j && c < kb) x[c] = fma(-l, u[c], x[c]);
            if (j + 1 < kb) {
                const long long a = mag_bits(x[j + 1]);
                if (a > key) {
                    key = a;
                    row = b0 + r;
                }
            }
        }
    }
    __syncthreads();
    for (int c = 0; c < kb; ++c)
        for (int r = tid; r < nr; r += LU_CT) C[(int64_t)(k0 + c) * s + k0 + b0 + r] = P[r * LU_PLD + c];
    smw_cluster_sync();  // no block leaves while another may write to it
}

__global__ void __launch_bounds__(1024) k_lu_panel(int32_t s, int32_t k0, int32_t kb, double* C, int32_t* piv,
                                                   int* err)
{
    __shared__ double wv[32];
    __shared__ int wi[32];
    __shared__ int pv_s;
    if (*err) return;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nwarps = nt >> 5;
    for (int j = k0; j < k0 + kb; ++j) {
        double* cj = C + (int64_t)j * s;
        double best = -1.0;
        int bidx = s;
        for (int i = j + tid; i < s; i += nt) {
            const double a = fabs(cj[i]);
            if (a > best) {
                best = a;
                bidx = i;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(SAI_FULL, best, o);
            const int oi = __shfl_xor_sync(SAI_FULL, bidx, o);
            if (ov > best || (ov == best && oi < bidx)) {
                best = ov;
                bidx = oi;
            }
        }
        if (lane == 0) {
            wv[wid] = best;
            wi[wid] = bidx;
        }
        __syncthreads();
        if (wid == 0) {
            best = lane < nwarps ? wv[lane] : -1.0;
            bidx = lane < nwarps ? wi[lane] : s;
            for (int o = 16; o > 0; o >>= 1) {
                const double ov = __shfl_xor_sync(SAI_FULL, best, o);
                const int oi = __shfl_xor_sync(SAI_FULL, bidx, o);
                if (ov > best || (ov == best && oi < bidx)) {
                    best = ov;
                    bidx = oi;
                }
            }
            if (lane == 0) pv_s = (best > 0.0 && bidx < s) ? bidx : -1;
        }
        __syncthreads();
        const int p = pv_s;
        if (p < 0) {
            if (tid == 0) *err = 1;
            return;
        }
        if (tid == 0) piv[j] = p;
        if (p != j)
            for (int c = k0 + tid; c < k0 + kb; c += nt) {
                const double t = C[(int64_t)c * s + j];
                C[(int64_t)c * s + j] = C[(int64_t)c * s + p];
                C[(int64_t)c * s + p] = t;
            }
        __syncthreads();
        const double ajj = cj[j];
        for (int i = j + 1 + tid; i < s; i += nt) {
            const double l = cj[i] / ajj;
            cj[i] = l;
            for (int c = j + 1; c < k0 + kb; ++c) C[(int64_t)c * s + i] -= l * C[(int64_t)c * s + j];
        }
        __syncthreads();
    }
}

// thread t < s: column t (outside the panel); thread s: g
__global__ void k_lu_swap(int32_t s, int32_t k0, int32_t kb, double* C, double* g, const int32_t* piv,
                          const int* err)
{
    if (*err) return;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t > s || (t >= k0 && t < k0 + kb)) return;
    double* v = t < s ? C + t * s : g;
    for (int j = k0; j < k0 + kb; ++j) {
        const int p = piv[j];
        if (p <= j || p >= s) continue;
        const double a = v[j];
        v[j] = v[p];
        v[p] = a;
    }
}

__global__ void k_lu_trsm(int32_t s, int32_t k0, int32_t kb, double* C, const int* err)
{
    if (*err) return;
    const int64_t c = (int64_t)k0 + kb + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s) return;
    double x[LU_NB];
    double* col = C + c * s + k0;
#pragma unroll
    for (int r = 0; r < LU_NB; ++r) {
        if (r < kb) {
            double v = col[r];
            for (int q = 0; q < r; ++q) v -= C[(int64_t)(k0 + q) * s + k0 + r] * x[q];
            x[r] = v;
            col[r] = v;
        }
    }
}

__global__ void __launch_bounds__(256) k_lu_gemm(int32_t s, int32_t k0, int32_t kb, double* C, const int* err)
{
    __shared__ double Ls[LU_NB][64];
    __shared__ double Us[LU_NB][65];
    if (*err) return;
    const int k1 = k0 + kb;
    const int m = s - k1;
    const int nt = (m + 63) / 64;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int64_t blk = blockIdx.x; blk < (int64_t)nt * nt; blk += gridDim.x) {
        const int i0 = k1 + (int)(blk % nt) * 64, c0 = k1 + (int)(blk / nt) * 64;
        for (int e = tid; e < kb * 64; e += 256) {
            const int q = e / 64, ii = e % 64;
            Ls[q][ii] = i0 + ii < s ? C[(int64_t)(k0 + q) * s + i0 + ii] : 0.0;
        }
        for (int e = tid; e < kb * 64; e += 256) {
            const int q = e % kb, cc = e / kb;
            Us[q][cc] = c0 + cc < s ? C[(int64_t)(c0 + cc) * s + k0 + q] : 0.0;
        }
        __syncthreads();
        double acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
        for (int q = 0; q < kb; ++q) {
            double l[4], u[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) l[a] = Ls[q][tx + 16 * a];
#pragma unroll
            for (int b = 0; b < 4; ++b) u[b] = Us[q][ty + 16 * b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fma(l[a], u[b], acc[a][b]);
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int c = c0 + ty + 16 * b;
            if (c >= s) continue;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int i = i0 + tx + 16 * a;
                if (i < s) C[(int64_t)c * s + i] -= acc[a][b];
            }
        }
        __syncthreads();
    }
}

// L y = Pg (unit diagonal), U z = y in blocks of 32 rows over one cluster:
// block r of the cluster keeps rows [r R, (r + 1) R) of the vector in shared
// memory, warp 0 of the diagonal block's owner solves it (from a staged copy,
// with the pivots' reciprocals) and sends the 32 values to all, and after one
// cluster barrier every block takes them out of its own rows. (One block, its
// FP64 pipe the bound, took 1.58 ms at s = 1051, the cluster 0.67 ms.)
__global__ void __launch_bounds__(LU_CT) k_lu_trsv(int32_t s, int R, const double* C, const double* g, double* z,
                                                   double* c_out, const int* err)
{
    extern __shared__ double zs[];  // R
    __shared__ double yb[2][32], D[32][33], red[LU_CT / 32], part[LU_CL];
    if (*err) return;
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int b0 = (int)rank * R, nr = max(0, min(R, s - b0));  // R is a multiple of 32
    for (int i = tid; i < nr; i += LU_CT) zs[i] = g[b0 + i];
    const int nb = (s + 31) / 32;
    __syncthreads();
    smw_cluster_sync();
    for (int pass = 0; pass < 2; ++pass)
        for (int q = 0; q < nb; ++q) {
            const int t = pass == 0 ? q : nb - 1 - q;  // diagonal block
            const int j0 = 32 * t, jb = min(32, s - j0);
            double* y = yb[(pass * nb + q) & 1];
            if (j0 / R == (int)rank) {
                for (int e = tid; e < 32 * 32; e += LU_CT) {
                    const int c = e >> 5, r = e & 31;
                    D[c][r] = c < jb && r < jb ? C[(int64_t)(j0 + c) * s + j0 + r] : 0.0;
                }
                __syncthreads();
                if (wid == 0) {
                    double v = lane < jb ? zs[j0 - b0 + lane] : 0.0;
                    if (pass == 0) {
                        for (int jj = 0; jj < jb; ++jj) {
                            const double yj = __shfl_sync(SAI_FULL, v, jj);
                            if (lane > jj) v = fma(-D[jj][lane], yj, v);
                        }
                    } else {
                        const double rd = lane < jb ? 1.0 / D[lane][lane] : 0.0;
                        for (int jj = jb - 1; jj >= 0; --jj) {
                            if (lane == jj) v = div_by(v, D[jj][jj], rd);
                            const double zj = __shfl_sync(SAI_FULL, v, jj);
                            if (lane < jj) v = fma(-D[jj][lane], zj, v);
                        }
                    }
                    if (lane < jb) zs[j0 - b0 + lane] = v;
                    for (int to = 0; to < LU_CL; ++to) smw_st(smw_map(smw_smem(y + lane), (uint32_t)to), lane < jb ? v : 0.0);
                }
            }
            smw_cluster_sync();
            const int a = pass == 0 ? max(0, j0 + jb - b0) : 0, b = pass == 0 ? nr : min(nr, j0 - b0);
            for (int i = a + tid; i < b; i += LU_CT) {
                double v = zs[i];
                for (int q0 = 0; q0 < jb; q0 += 8) {
                    double c[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) c[u] = q0 + u < jb ? C[(int64_t)(j0 + q0 + u) * s + b0 + i] : 0.0;
#pragma unroll
                    for (int u = 0; u < 8; ++u) v = fma(-c[u], y[q0 + u], v);
                }
                zs[i] = v;
            }
            __syncthreads();
        }
    double acc = 0.0;
    for (int i = tid; i < nr; i += LU_CT) {
        z[b0 + i] = zs[i];
        acc = fma(zs[i], zs[i], acc);
    }
    acc = warp_sum(acc);
    if (lane == 0) red[wid] = acc;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < LU_CT / 32; ++w) t += red[w];
        smw_st(smw_map(smw_smem(&part[rank]), 0), t);
    }
    smw_cluster_sync();
    if (rank == 0 && tid == 0) {
        double t = 0.0;
        for (int w = 0; w < LU_CL; ++w) t += part[w];
        *c_out = sqrt(t);
    }
}

// a launch of one cluster of LU_CL blocks; limit: the most dynamic shared memory of kern's launches
template <class... Args>
sai_status lu_cluster(void (*kern)(Args...), size_t limit, size_t smem, cudaStream_t st, Args... args)
{
    SAI_CUDA(sai_smem_limit(kern, limit));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SAI_GRID(LU_CL));
    cfg.blockDim = dim3(LU_CT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = LU_CL;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    SAI_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
    return SAI_OK;
}

// C = I + U^T What, g = U^T yhat for large s: a warp forms 64 consecutive
// columns b of Y = [yhat, What] for one column a of U, summing over U's
// entries in stored order. Items are column-chunk-major, so the warps
// running together read the same 64 columns of Y (n x 64 values, in L2).
__global__ void k_smw_gather_adj_big(int32_t s, const int64_t* Ucp, const int32_t* Uri, const double* Uv,
                                     const double* Y, double* C, double* g)
{
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t ld = (int64_t)s + 1;
    const int64_t nbc = (ld + 63) / 64;
    for (int64_t it = w0; it < (int64_t)s * nbc; it += nw) {
        const int a = (int)(it % s);
        const int64_t b0 = (it / s) * 64;
        const int64_t ba = b0 + lane, bb = b0 + 32 + lane;
        double acc0 = 0.0, acc1 = 0.0;
        const int64_t q0 = Ucp[a], q1 = Ucp[a + 1];
        for (int64_t qb = q0; qb < q1; qb += 32) {
            const int64_t q = qb + lane;
            const int32_t ri = q < q1 ? Uri[q] : 0;
            const double uv = q < q1 ? Uv[q] : 0.0;
            const int m = q1 - qb < 32 ? (int)(q1 - qb) : 32;
            for (int e = 0; e < m; ++e) {
                const int64_t i = __shfl_sync(SAI_FULL, ri, e);
                const double u = __shfl_sync(SAI_FULL, uv, e);
                const double* row = Y + i * ld;
                if (ba < ld) acc0 = fma(u, row[ba], acc0);
                if (bb < ld) acc1 = fma(u, row[bb], acc1);
            }
        }
        if (ba < ld) {
            if (ba == 0) g[a] = acc0;
            else C[(ba - 1) * s + a] = (a == ba - 1 ? 1.0 : 0.0) + acc0;
        }
        if (bb < ld) C[(bb - 1) * s + a] = (a == bb - 1 ? 1.0 : 0.0) + acc1;
    }
}

// xhat(i) = yhat(i) - sum_t What(i,t) z_t for large s, one warp per row
__global__ void k_smw_update_big(int32_t n, int32_t s, const double* Y, const double* z, double* x)
{
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    const int64_t ld = (int64_t)s + 1;
    const double* row = Y + i * ld;
    double v = 0.0;
    for (int t = lane; t < s; t += 32) v = fma(row[1 + t], z[t], v);
    v = warp_sum(v);
    if (lane == 0) x[i] = row[0] - v;
}

// LU solve of the s x s system C z = g (C, g overwritten) for large s.
sai_status lu_big(int32_t s, double* C, double* g, double* z, double* c_out, int* err, cudaStream_t st)
{
    Buf pivb;
    SAI_TRY(pivb.alloc(sizeof(int32_t) * (size_t)s, st, true));
    int32_t* piv = pivb.as<int32_t>();
    for (int k0 = 0; k0 < s; k0 += LU_NB) {
        const int kb = s - k0 < LU_NB ? s - k0 : LU_NB;
        const int rows = (s - k0 + LU_CL - 1) / LU_CL;
        if (rows <= LU_PROWS)
            SAI_TRY(lu_cluster(k_lu_panel_cluster, LU_PANEL_SMEM, sizeof(double) * rows * LU_PLD, st, s, k0, kb, rows, C,
                               piv, err));
        else
            k_lu_panel<<<SAI_GRID(1), 1024, 0, st>>>(s, k0, kb, C, piv, err);
        k_lu_swap<<<SAI_GRID(sai_div_up((int64_t)s + 1, 256)), 256, 0, st>>>(s, k0, kb, C, g, piv, err);
        const int m = s - k0 - kb;
        if (m > 0) {
            k_lu_trsm<<<SAI_GRID(sai_div_up(m, 128)), 128, 0, st>>>(s, k0, kb, C, err);
            const int64_t nt = (m + 63) / 64;
            const int64_t gb = nt * nt < (int64_t)g_num_sms_smw() * 8 ? nt * nt : (int64_t)g_num_sms_smw() * 8;
            k_lu_gemm<<<SAI_GRID(gb), 256, 0, st>>>(s, k0, kb, C, err);
        }
    }
    const int R = (((int)s + LU_CL - 1) / LU_CL + 31) / 32 * 32;
    SAI_TRY(lu_cluster(k_lu_trsv, LU_TRSV_SMEM, sizeof(double) * R, st, s, R, (const double*)C, (const double*)g, z,
                       c_out, (const int*)err));
    SAI_CUDA(cudaGetLastError());
    return SAI_OK;
}

}  // namespace

namespace {

sai_status smw_common(const sai_split_s* h, const double* Y, double* x, double* c_out, bool adjoint, cudaStream_t st)
{
    if (!h || (h->n > 0 && (!Y || !x))) return SAI_INVALID_ARG;
    const int32_t n = h->n, s = h->s;
    const size_t ss = (size_t)(s > 0 ? s : 1);
    Buf C, g, z, cbuf, err;
    SAI_TRY(C.alloc(sizeof(double) * ss * ss, st, true));
    SAI_TRY(g.alloc(sizeof(double) * ss, st, true));
    SAI_TRY(z.alloc(sizeof(double) * ss, st, true));
    SAI_TRY(cbuf.alloc(sizeof(double), st, true));
    SAI_TRY(err.alloc(sizeof(int), st, true));
    SAI_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
    SAI_CUDA(cudaMemsetAsync(cbuf.p, 0, sizeof(double), st));
    if (s > 0) {
        if (!adjoint)
            k_smw_gather<<<SAI_GRID(sai_div_up((int64_t)s * s, 256)), 256, 0, st>>>(n, s, h->J.as<int32_t>(), Y,
                                                                                   C.as<double>(), g.as<double>());
        else if (s <= LU_SMALL)
            k_smw_gather_adj<<<SAI_GRID(sai_div_up((int64_t)s * (s + 1) * 32, 256)), 256, 0, st>>>(
                s, h->U_cp.as<int64_t>(), h->U_ri.as<int32_t>(), h->U_v.as<double>(), Y, C.as<double>(),
                g.as<double>());
        else {
            const int64_t items = (int64_t)s * (((int64_t)s + 1 + 63) / 64);
            const int64_t gb = sai_div_up(items, 8) < (int64_t)g_num_sms_smw() * 16 ? sai_div_up(items, 8)
                                                                                   : (int64_t)g_num_sms_smw() * 16;
            k_smw_gather_adj_big<<<SAI_GRID(gb), 256, 0, st>>>(s, h->U_cp.as<int64_t>(), h->U_ri.as<int32_t>(),
                                                               h->U_v.as<double>(), Y, C.as<double>(),
                                                               g.as<double>());
        }
        if (s <= LU_SMEM)
            SAI_TRY(lu_small(s, C.as<double>(), g.as<double>(), z.as<double>(), cbuf.as<double>(), err.as<int>(), st));
        else
            SAI_TRY(lu_big(s, C.as<double>(), g.as<double>(), z.as<double>(), cbuf.as<double>(), err.as<int>(), st));
    }
    if (n > 0 && s <= LU_SMALL) k_smw_update<<<SAI_GRID(sai_div_up(n, 256)), 256, 0, st>>>(n, s, Y, z.as<double>(), x);
    else if (n > 0)
        k_smw_update_big<<<SAI_GRID(sai_div_up((int64_t)n * 32, 256)), 256, 0, st>>>(n, s, Y, z.as<double>(), x);
    SAI_CUDA(cudaGetLastError());
    int herr = 0;
    double hc = 0.0;
    SAI_CUDA(cudaMemcpyAsync(&herr, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    SAI_CUDA(cudaMemcpyAsync(&hc, cbuf.p, sizeof(double), cudaMemcpyDeviceToHost, st));
    SAI_CUDA(cudaStreamSynchronize(st));
    if (herr) return SAI_SINGULAR;
    if (c_out) *c_out = hc;
    return SAI_OK;
}

}  // namespace

sai_status sai_smw_run(const sai_split_s* h, const double* Y, double* x, double* c_out, cudaStream_t st)
{
    return smw_common(h, Y, x, c_out, false, st);
}

sai_status sai_smw_adj_run(const sai_split_s* h, const double* Y, double* x, double* c_out, cudaStream_t st)
{
    return smw_common(h, Y, x, c_out, true, st);
}

// ---------------------------------------------------------------- allocation-free variant
// sai_smw_recover_noalloc: the same SMW recovery for callers that cannot
// allocate device memory -- code that runs where every device byte is owned
// by a host framework's own pool or a fixed budget, or where an allocation
// would synchronise or is not permitted. Its scratch (the s x s matrix, two
// s-vectors, c and an error flag) is this file-scope array, reserved once on
// every device that loads the library and held until the process exits.
namespace {

constexpr int NOALLOC_MAX_S = 256;
constexpr size_t NOALLOC_C_OFF = 0;
constexpr size_t NOALLOC_G_OFF = NOALLOC_C_OFF + sizeof(double) * NOALLOC_MAX_S * NOALLOC_MAX_S;
constexpr size_t NOALLOC_Z_OFF = NOALLOC_G_OFF + sizeof(double) * NOALLOC_MAX_S;
constexpr size_t NOALLOC_CV_OFF = NOALLOC_Z_OFF + sizeof(double) * NOALLOC_MAX_S;
constexpr size_t NOALLOC_ERR_OFF = NOALLOC_CV_OFF + 256;
constexpr size_t NOALLOC_BYTES = NOALLOC_ERR_OFF + 256;

static __device__ __align__(256) unsigned char g_smw_noalloc_scratch[NOALLOC_BYTES];

// Device address of the scratch array in the current device's context (the
// host-side symbol is only a stand-in, not a device address). Looked up on
// every call: the lookup allocates nothing, and an address kept from an
// earlier context (before a cudaDeviceReset, say) would no longer be valid.
sai_status noalloc_scratch(unsigned char** out)
{
    void* p = nullptr;
    SAI_CUDA(cudaGetSymbolAddress(&p, g_smw_noalloc_scratch));
    *out = (unsigned char*)p;
    return SAI_OK;
}

}  // namespace

extern "C" sai_status sai_smw_recover_noalloc(int32_t n, int32_t s, const int32_t* J, const double* Y, double* x,
                                              double* c_out, sai_stream_t stream)
{
    if (n < 0 || s < 0 || s > n || (n > 0 && (!Y || !x)) || (s > 0 && !J)) return SAI_INVALID_ARG;
    if (s > NOALLOC_MAX_S) return SAI_INVALID_ARG;  // beyond the static scratch
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char* base = nullptr;
    SAI_TRY(noalloc_scratch(&base));
    double* C = (double*)(base + NOALLOC_C_OFF);
    double* g = (double*)(base + NOALLOC_G_OFF);
    double* z = (double*)(base + NOALLOC_Z_OFF);
    double* cval = (double*)(base + NOALLOC_CV_OFF);
    int* err = (int*)(base + NOALLOC_ERR_OFF);
    // the array keeps the previous call's contents: clear what must start at
    // zero; z too, so that a zero pivot (z left unwritten) gives x = yhat
    SAI_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
    SAI_CUDA(cudaMemsetAsync(cval, 0, sizeof(double), st));
    if (s > 0) SAI_CUDA(cudaMemsetAsync(z, 0, sizeof(double) * (size_t)s, st));
    if (s > 0) {
        k_smw_gather<<<SAI_GRID(sai_div_up((int64_t)s * s, 256)), 256, 0, st>>>(n, s, J, Y, C, g);
        SAI_TRY(lu_small(s, C, g, z, cval, err, st));
    }
    if (n > 0) k_smw_update<<<SAI_GRID(sai_div_up(n, 256)), 256, 0, st>>>(n, s, Y, z, x);
    SAI_CUDA(cudaGetLastError());
    int herr = 0;
    double hc = 0.0;
    SAI_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    SAI_CUDA(cudaMemcpyAsync(&hc, cval, sizeof(double), cudaMemcpyDeviceToHost, st));
    SAI_CUDA(cudaStreamSynchronize(st));
    if (herr) return SAI_SINGULAR;
    if (c_out) *c_out = hc;
    return SAI_OK;
}
