// bicg_cluster.cuh -- the whole BiCGStab of one system in one thread-block
// cluster, for orders up to CL_MAXN (included by krylov.cu inside its
// namespace).
//
// At these orders an iteration of the multi-kernel form is nine launches of a
// few microseconds each, whatever the work. Here a cluster of 1, 2, 4 or 8
// blocks keeps all nine vectors of its system in shared memory (block b the
// rows [b R, (b + 1) R)), reads the matrices through L1, gathers x across the
// cluster by distributed-shared-memory loads and runs every iteration without
// leaving the kernel; a phase costs a cluster barrier.
//
// A system's bits do not depend on the cluster size or on the other systems:
// row sums run over the row's entries in order, and an inner product is a
// fixed tree per unit of 64 rows (two rows per lane, five shuffle levels)
// followed by the units' sums in a fixed order (lane l takes units l, l + 32,
// .., then five shuffle levels), those of rhat^T v and rhat^T r in twice the
// working precision as in the multi-kernel form.

constexpr int CL_T = 512;        // threads per block
constexpr int CL_MAXR = 2560;    // rows per block: nine vectors of 20 KB
constexpr int CL_MAXC = 8;       // blocks per cluster (the portable limit; 16 where all systems run at once)
constexpr int CL_MAXN = CL_MAXR * CL_MAXC;
constexpr int CL_UNIT = 64;      // rows per reduction unit
constexpr int CL_VECS = 9;
constexpr int CL_SLOTS = 6;      // partial sums: rhat^T v; ||s||; t^T s, t^T t; ||r||, rhat^T r

// CSR, or its sliced-ELL copy when sp is given (row0 = 0 then)
template <class T>
struct ClMat {
    const int64_t* rp;
    const int32_t* ci;
    const T* v;
    const int64_t* sp;
    const int32_t* sci;
    const T* sv;
};

template <bool MULTI>
__device__ __forceinline__ void cl_barrier()
{
    if (MULTI) {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else {
        __syncthreads();
    }
}

__device__ __forceinline__ uint32_t cl_map(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

template <class T>
__device__ __forceinline__ T cl_ld(uint32_t addr);
template <>
__device__ __forceinline__ double cl_ld<double>(uint32_t addr)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
template <>
__device__ __forceinline__ float cl_ld<float>(uint32_t addr)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ void cl_st(uint32_t addr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// The block's part of the system.
struct ClRows {
    int n, R, base, nrow;  // order, rows per block, first row, rows of this block
    int row0;              // the system's first row in the matrices
    uint32_t inv;          // ceil(2^32 / R): row / R = umulhi(row, inv) for rows below 2^32 / R
    int units;             // units of this block
    int unit0;             // index of its first unit in the system
    int nunits;            // units of the system
};

// y (two rows per lane of the unit at local row lr0) = the rows of A times
// the vector at shared offset `x` (bytes) of every block of the cluster
template <class T, bool MULTI>
__device__ __forceinline__ void cl_spmv(const ClMat<T>& A, const ClRows& W, const T* xs, uint32_t x, int lr0, T (&y)[2])
{
    const int lane = threadIdx.x & 31;
    const int32_t* ci[2];
    const T* va[2];
    int len[2], stride;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int lr = lr0 + 32 * h + lane;  // local row
        if (A.sp) {
            const int sl = (W.base + lr0) / 32 + h;
            const bool in = lr0 + 32 * h < W.nrow;
            const int64_t b = in ? A.sp[sl] : 0, e = in ? A.sp[sl + 1] : 0;
            ci[h] = A.sci + b + lane;
            va[h] = A.sv + b + lane;
            len[h] = (int)(e - b) / 32;
            stride = 32;
        } else {
            const bool in = lr < W.nrow;
            const int64_t g = (int64_t)W.row0 + W.base + lr;
            const int64_t b = in ? A.rp[g] : 0, e = in ? A.rp[g + 1] : 0;
            ci[h] = A.ci + b;
            va[h] = A.v + b;
            len[h] = (int)(e - b);
            stride = 1;
        }
        y[h] = 0;
    }
    // BT entries of both rows at a time: their indices and values, then their
    // gathers (from this block's shared memory when all of the warp's columns
    // are its own, as most are on a grid: 30 cycles against 250 across the
    // cluster), then their products in order
    constexpr int BT = sizeof(T) == 4 ? 8 : 4;
    // the warp's longest row: its votes below need every lane in every round
    const int most = __reduce_max_sync(SAI_FULL, max(len[0], len[1]));
    for (int k0 = 0; k0 < most; k0 += BT) {
        int col[2][BT];
        T a[2][BT], xv[2][BT];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int u = 0; u < BT; ++u) {
                const bool in = k0 + u < len[h];
                col[h][u] = in ? __ldg(ci[h] + (int64_t)(k0 + u) * stride) - W.row0 : W.base;
                a[h][u] = in ? __ldg(va[h] + (int64_t)(k0 + u) * stride) : T(0);
            }
        bool own = true;
        if (MULTI) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int u = 0; u < BT; ++u) own &= (unsigned)(col[h][u] - W.base) < (unsigned)W.R;
            own = __all_sync(SAI_FULL, own);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int u = 0; u < BT; ++u) {
                if (!MULTI || own) {
                    xv[h][u] = xs[col[h][u] - W.base];
                } else {
                    const uint32_t rk = __umulhi((uint32_t)col[h][u], W.inv);
                    xv[h][u] = cl_ld<T>(cl_map(x + (uint32_t)sizeof(T) * ((uint32_t)col[h][u] - rk * (uint32_t)W.R), rk));
                }
            }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int u = 0; u < BT; ++u)
                if (k0 + u < len[h]) y[h] = fma(a[h][u], xv[h][u], y[h]);
    }
}

// Stores a unit's partial sum in slot `slot` of every block of the cluster.
template <bool MULTI>
__device__ __forceinline__ void cl_put(double v, int slot, int unit, double* parts, int pstride, int nranks)
{
    v = warp_sum(v);
    const int lane = threadIdx.x & 31;
    double* p = parts + slot * pstride + unit;
    if (MULTI) {
        if (lane < nranks) cl_st(cl_map(smem_u32(p), (uint32_t)lane), v);
    } else if (lane == 0) {
        *p = v;
    }
}

// The sum of a slot's units (one warp; the same bits in every block).
__device__ __forceinline__ double cl_total(const double* parts, int slot, int pstride, int nunits, bool comp)
{
    const int lane = threadIdx.x & 31;
    const double* p = parts + slot * pstride;
    double h = 0.0, l = 0.0;
    if (!comp) {
        for (int u = lane; u < nunits; u += 32) h += p[u];
        return warp_sum(h);
    }
    for (int u = lane; u < nunits; u += 32) two_add(h, l, p[u]);
    // up the tree the sums alone wait for one another; a node's rounding error
    // is known to all 2^(level + 1) lanes below it and enters with that weight,
    // so that the lanes' errors add up to the tree's (exact scalings)
    double w = 0.5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1, w *= 0.5) {
        const double h2 = __shfl_xor_sync(SAI_FULL, h, o);
        const bool lo = (lane & o) == 0;
        double a = lo ? h : h2, e = 0.0;  // the same operands in the same order in both lanes
        two_add(a, e, lo ? h2 : h);
        h = a;
        l = fma(w, e, l);
    }
    return h + warp_sum(l);
}

// sqrt(x) < t, with the root taken only where the squares are too close to tell
__device__ __forceinline__ bool cl_below(double x, double t)
{
    const double t2 = t * t;
    if (x > t2 * (1.0 + 1e-14)) return false;
    if (x < t2 * (1.0 - 1e-14)) return true;
    return sqrt(x) < t;
}

// One cluster per system (blockIdx.x / cluster size = index in `pick`, or the
// system itself). B, X: the system's vectors at off[c] (c * ld without off).
template <bool MULTI>
__global__ void __launch_bounds__(CL_T, 1)
k_bicg_cluster(ClMat<double> A, ClMat<double> M, int n1, int64_t ld, const int64_t* __restrict__ off, const int32_t* __restrict__ lens,
               const int32_t* __restrict__ row0s, const int32_t* __restrict__ pick, int rmax, int umax,
               const double* __restrict__ B, double* __restrict__ X, const double* __restrict__ thr, int maxit,
               int* __restrict__ iters, int* __restrict__ status)
{
    extern __shared__ __align__(16) double sm[];
    __shared__ double sc[5];  // alpha, omega, beta, alpha / (omega rho), rho of the running iteration
    __shared__ int flag;      // 0 go on (first iteration), 1 half step, then stop, 2 stop, 3 go on
    uint32_t rank = 0, nranks = 1;
    if (MULTI) {
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nranks));
    }
    const int q = blockIdx.x / nranks;
    const int c = pick ? pick[q] : q;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int NW = CL_T / 32;
    ClRows W;
    W.n = lens ? lens[c] : n1;
    W.row0 = row0s ? row0s[c] : 0;
    W.R = ((W.n + (int)nranks - 1) / (int)nranks + CL_UNIT - 1) / CL_UNIT * CL_UNIT;
    W.base = (int)rank * W.R;
    W.nrow = max(0, min(W.R, W.n - W.base));
    W.inv = (uint32_t)((0x100000000ull + (unsigned)W.R - 1) / (unsigned)W.R);
    W.units = (W.nrow + CL_UNIT - 1) / CL_UNIT;
    W.unit0 = W.base / CL_UNIT;
    W.nunits = (W.n + CL_UNIT - 1) / CL_UNIT;
    const int64_t o = (off ? off[c] : (int64_t)c * ld) + W.base;
    double *p = sm, *ph = p + rmax, *s = ph + rmax, *sh = s + rmax;  // gathered by the cluster
    double *r = sh + rmax, *rh = r + rmax, *v = rh + rmax, *t = v + rmax, *x = t + rmax;
    double* parts = x + rmax;  // [slot][unit]
    const uint32_t pa = smem_u32(p), pha = smem_u32(ph), sa = smem_u32(s), sha = smem_u32(sh);
    const double th = thr[c];
    // r = rhat = p = b (the rows past the end are zero and stay so), x = 0
    for (int i = threadIdx.x; i < rmax; i += CL_T) {
        const double b = i < W.nrow ? B[o + i] : 0.0;
        r[i] = rh[i] = p[i] = b;
        x[i] = v[i] = t[i] = s[i] = ph[i] = sh[i] = 0.0;
    }
    __syncthreads();
    cl_barrier<MULTI>();  // every block of the cluster runs before its memory is written
    for (int u = wid; u < W.units; u += NW) {
        const double a = r[u * CL_UNIT + lane], b = r[u * CL_UNIT + 32 + lane];
        cl_put<MULTI>(fma(b, b, a * a), 1, W.unit0 + u, parts, umax, (int)nranks);
    }
    cl_barrier<MULTI>();
    // control values live in warp 0, lane by lane the same
    double rho = 0.0, omega = 1.0;
    int it = 0, stat = ST_OK;
    // the next iteration's start: count it, test rho, form beta
    auto next = [&]() {
        if (it >= maxit) {
            stat = ST_MAXITER;
            return 2;
        }
        ++it;
        if (rho == 0.0) {
            stat = ST_BREAKDOWN;
            return 2;
        }
        // beta = (rho / rho_old) (alpha / omega), the quotient without rho formed earlier
        if (lane == 0) sc[2] = it == 1 ? 0.0 : rho * sc[3];
        return 0;
    };
    if (wid == 0) {
        rho = cl_total(parts, 1, umax, W.nunits, false);
        int f = 2;
        if (!(sqrt(rho) < th)) f = next();
        if (lane == 0) flag = f;
    }
    __syncthreads();
    while (flag != 2) {
        if (flag == 3) {  // p = r + beta (p - omega v); the first iteration's p = r is in place
            const double be = sc[2], om = sc[1];
            for (int u = wid; u < W.units; u += NW)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = u * CL_UNIT + 32 * h + lane;
                    p[i] = fma(be, fma(-om, v[i], p[i]), r[i]);
                }
        }
        cl_barrier<MULTI>();
        for (int u = wid; u < W.units; u += NW) {
            double y[2];
            cl_spmv<double, MULTI>(M, W, p, pa, u * CL_UNIT, y);
            ph[u * CL_UNIT + lane] = y[0];
            ph[u * CL_UNIT + 32 + lane] = y[1];
        }
        cl_barrier<MULTI>();
        for (int u = wid; u < W.units; u += NW) {
            double y[2];
            cl_spmv<double, MULTI>(A, W, ph, pha, u * CL_UNIT, y);
            const int i = u * CL_UNIT + lane;
            v[i] = y[0];
            v[i + 32] = y[1];
            cl_put<MULTI>(fma(rh[i + 32], y[1], rh[i] * y[0]), 0, W.unit0 + u, parts, umax, (int)nranks);
        }
        cl_barrier<MULTI>();
        if (wid == 0) {
            const double rv = cl_total(parts, 0, umax, W.nunits, true);
            int f = 0;
            if (rv == 0.0) {
                stat = ST_BREAKDOWN;
                f = 2;
            } else {
                const double alpha = rho / rv;
                if (lane == 0) {
                    sc[0] = alpha;
                    sc[4] = rho;
                }
            }
            if (lane == 0) flag = f;
        }
        __syncthreads();
        if (flag == 2) break;
        {
            const double al = sc[0];
            for (int u = wid; u < W.units; u += NW) {
                const int i = u * CL_UNIT + lane;
                const double s0 = fma(-al, v[i], r[i]), s1 = fma(-al, v[i + 32], r[i + 32]);
                s[i] = s0;
                s[i + 32] = s1;
                cl_put<MULTI>(fma(s1, s1, s0 * s0), 1, W.unit0 + u, parts, umax, (int)nranks);
            }
        }
        cl_barrier<MULTI>();
        if (wid == 0) {
            const double ss = cl_total(parts, 1, umax, W.nunits, false);
            if (lane == 0) flag = cl_below(ss, th) ? 1 : 0;
        }
        __syncthreads();
        if (flag == 1) {  // the half step
            const double al = sc[0];
            for (int u = wid; u < W.units; u += NW) {
                const int i = u * CL_UNIT + lane;
                x[i] = fma(al, ph[i], x[i]);
                x[i + 32] = fma(al, ph[i + 32], x[i + 32]);
            }
            stat = ST_OK;
            break;
        }
        for (int u = wid; u < W.units; u += NW) {
            double y[2];
            cl_spmv<double, MULTI>(M, W, s, sa, u * CL_UNIT, y);
            sh[u * CL_UNIT + lane] = y[0];
            sh[u * CL_UNIT + 32 + lane] = y[1];
        }
        cl_barrier<MULTI>();
        for (int u = wid; u < W.units; u += NW) {
            double y[2];
            cl_spmv<double, MULTI>(A, W, sh, sha, u * CL_UNIT, y);
            const int i = u * CL_UNIT + lane;
            t[i] = y[0];
            t[i + 32] = y[1];
            cl_put<MULTI>(fma(y[1], s[i + 32], y[0] * s[i]), 2, W.unit0 + u, parts, umax, (int)nranks);
            cl_put<MULTI>(fma(y[1], y[1], y[0] * y[0]), 3, W.unit0 + u, parts, umax, (int)nranks);
        }
        cl_barrier<MULTI>();
        if (wid == 0) {
            const double ts = cl_total(parts, 2, umax, W.nunits, false);
            const double tt = cl_total(parts, 3, umax, W.nunits, false);
            int f = 0;
            if (tt == 0.0) {
                stat = ST_BREAKDOWN;
                f = 2;
            } else {
                omega = ts / tt;
                if (lane == 0) sc[1] = omega;
            }
            if (lane == 0) flag = f;
        }
        __syncthreads();
        if (flag == 2) break;
        {
            const double al = sc[0], om = sc[1];
            // beside the update, in the warp that has the fewest units
            if (wid == NW - 1 && lane == 0) sc[3] = al / (om * sc[4]);
            for (int u = wid; u < W.units; u += NW) {
                const int i = u * CL_UNIT + lane;
                double rv[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int e = i + 32 * h;
                    x[e] = fma(om, sh[e], fma(al, ph[e], x[e]));
                    rv[h] = fma(-om, t[e], s[e]);
                    r[e] = rv[h];
                }
                cl_put<MULTI>(fma(rv[1], rv[1], rv[0] * rv[0]), 4, W.unit0 + u, parts, umax, (int)nranks);
                cl_put<MULTI>(fma(rh[i + 32], rv[1], rh[i] * rv[0]), 5, W.unit0 + u, parts, umax, (int)nranks);
            }
        }
        cl_barrier<MULTI>();
        if (wid == 0) {
            const double rr = cl_total(parts, 4, umax, W.nunits, false);
            const double rhr = cl_total(parts, 5, umax, W.nunits, true);
            int f = 2;
            if (cl_below(rr, th)) {
                stat = ST_OK;
            } else if (omega == 0.0) {
                stat = ST_BREAKDOWN;
            } else {
                rho = rhr;
                f = next();
                if (f == 0) f = 3;  // p is formed with beta from here on
            }
            if (lane == 0) flag = f;
        }
        __syncthreads();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < W.nrow; i += CL_T) X[o + i] = x[i];
    if (rank == 0 && threadIdx.x == 0) {
        iters[c] = it;
        status[c] = stat;
    }
    cl_barrier<MULTI>();  // no block leaves while another may read its memory
}

// algorithmic work of a finished launch (only while a profile is open): the
// matrices once per iteration of the longest system, each system's vectors
__global__ void k_cl_work(int k, const int* iters, Dims D)
{
    double sum = 0.0, most = 0.0;
    for (int c = 0; c < k; ++c) {
        sum += iters[c];
        most = fmax(most, (double)iters[c]);
    }
    const double nz = D.nnzA + D.nnzM;
    kwork_add(PROF_SPMM, 2.0 * most * (12.0 * nz + 16.0 * (D.n + 1)) + 64.0 * D.n * sum, 4.0 * nz * sum);
    kwork_add(PROF_BICG_VEC, 8.0 * D.n * 19 * sum, D.n * 23.0 * sum);
}

// blocks per cluster for k systems of order at most n: enough for the rows,
// then as many as leave every system on the GPU at once with two units of
// rows per block (the reductions' cost does not shrink with more)
inline int cl_blocks(int k, int n)
{
    int C = 1;
    while (C < CL_MAXC && (int64_t)C * CL_MAXR < n) C *= 2;
    while (C < CL_MAXC && (int64_t)2 * C * k <= (int64_t)g_sms * 7 / 8 && n / (2 * C) >= 2 * CL_UNIT) C *= 2;
    return C;
}

// true when the GPU holds k clusters of 16 blocks of kern at once
template <class... Params>
bool cl_fits16(void (*kern)(Params...), int k, int threads, size_t smem)
{
    if (16 * (int64_t)k > g_sms) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16u * (unsigned)k);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 16;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int most = 0;
    const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&most, kern, &cfg) == cudaSuccess;
    if (!ok) (void)cudaGetLastError();
    return ok && most >= k;
}

// Launches kern with k clusters of C blocks; false when the device refuses the shape.
template <class... Params, class... Args>
bool cl_run(void (*kern)(Params...), int k, int C, int threads, size_t smem, cudaStream_t st, Args... args)
{
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SAI_GRID(k * C));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...) != cudaSuccess) {
        (void)cudaGetLastError();
        sai_count_grid_add(-1);
        return false;
    }
    return true;
}

inline bool cl_launch(const ClMat<double>& A, const ClMat<double>& M, int k, int n, int64_t ld, const int64_t* off,
                      const int32_t* lens, const int32_t* row0s, const int32_t* pick, const double* B, double* X,
                      const double* thr, int maxit, int* iters, int* status, cudaStream_t st)
{
    int C = cl_blocks(k, n);
    const int umax = (n + CL_UNIT - 1) / CL_UNIT;
    int rmax = 0;
    size_t smem = 0;
    auto shape = [&](int blocks) {
        C = blocks;
        rmax = ((n + C - 1) / C + CL_UNIT - 1) / CL_UNIT * CL_UNIT;
        smem = sizeof(double) * ((size_t)CL_VECS * rmax + (size_t)CL_SLOTS * umax);
    };
    shape(C);
    // from 512 rows per block on the FP64 pipe outweighs the barriers
    if (C == CL_MAXC && rmax >= 512) {
        shape(16);
        if (!cl_fits16(k_bicg_cluster<true>, k, CL_T, smem)) shape(CL_MAXC);
    }
    return cl_run(C > 1 ? k_bicg_cluster<true> : k_bicg_cluster<false>, k, C, CL_T, smem, st, A, M, n, ld, off, lens,
                  row0s, pick, rmax, umax, B, X, thr, maxit, iters, status);
}
