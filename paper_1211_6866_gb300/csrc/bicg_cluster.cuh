// bicg_cluster.cuh -- the whole BiCGStab of one system in one thread-block
// cluster, for orders up to CL_MAXN (included by krylov.cu inside its
// namespace).
//
// At these orders an iteration of the multi-kernel form is nine launches of a
// few microseconds each, whatever the work. Here a cluster of 1, 2, 4, 8 or 16
// blocks keeps all nine vectors of its system in shared memory (block b the
// rows [b R, (b + 1) R)), reads the matrices through L1, gathers x across the
// cluster by distributed-shared-memory loads and runs every iteration without
// leaving the kernel; a phase costs a cluster barrier. A 45 x 45 grid with four
// systems, 80 iterations: 11.5 ms per call at first, 2.5 ms here, 22 us per
// iteration (seven barriers, four products, three scalar chains).
//
// A system's bits do not depend on the cluster size, nor on the systems that
// run with it as long as their number leaves the form in use (the limits below;
// the multi-kernel form adds in another order):
// row sums run over the row's entries in order, and an inner product is a
// fixed tree per unit of 64 rows (two rows per lane, five shuffle levels)
// followed by the units' sums in a fixed order (lane l takes units l, l + 32,
// .., then five shuffle levels), those of rhat^T v and rhat^T r in twice the
// working precision as in the multi-kernel form.

constexpr int CL_T = 512;        // threads per block
constexpr int CL_MAXR = 2560;    // rows per block: nine vectors of 20 KB
constexpr int CL_MAXC = 8;       // blocks per cluster (the portable limit; 16 where all systems run at once)
constexpr int CL_MAXN = CL_MAXR * CL_MAXC;
// Limits of the form, against the multi-kernel form (40 iterations unless
// stated, in ms):
// - systems: at 10000 rows of a power-law matrix 52 against 56 with 511, 101
//   against 33 with 1020, for which the other form goes over to panels of
//   systems;
constexpr int CL_MAXK = 256;
// - a scattered matrix, most of whose gathers cross the cluster, up to this
//   order only (in GMRES too): with 8, 32 and 128 systems 4.9, 7.0 and 27
//   against 5.0, 9.3 and 28 at 10000 rows, 6.6, 20 and 29 (of half the
//   iterations) against 5.4, 11 and 17 at 14500;
constexpr int CL_FAR_N = 10240;
// - above this order only so many systems (60 iterations on a grid): 8, 64 and
//   256 systems 3.0, 14.0 and 49.7 against 5.8, 15.0 and 50.2 at 12167 rows, 3.6,
//   17.0 and 60.6 against 5.7, 15.4 and 53.3 at 15625, 4.1, 19.8 and 70.5 against
//   6.4, 16.1 and 53.5 at 19683. (From 17 on, which take two rounds, the other
//   form is up to a fifth faster; the line lies higher so that a system keeps its
//   bits among a few dozen others.)
constexpr int CL_MANY_N = 14336, CL_MANY_K = 64;
constexpr int CL_UNIT = 64;      // rows per reduction unit
constexpr int CL_VECS = 9;
constexpr int CL_SLOTS = 6;      // partial sums: rhat^T v; ||s||; t^T s, t^T t; ||r||, rhat^T r
constexpr size_t CL_SMEM = sizeof(double) * ((size_t)CL_VECS * CL_MAXR + (size_t)CL_SLOTS * (CL_MAXN / CL_UNIT));  // at most

// A matrix in slices of 32 rows, entries column-major within a slice (slice q
// at sp[q] .. sp[q + 1]). With ord, the rows of each block are sorted by
// length and position i holds row ord[i] of its block (-1: none): slices of
// unsorted rows of unequal length would be mostly padding, and a CSR row per
// lane takes a memory transaction per lane and entry (a 2000-row power-law
// system forward and backward, build included: 15.6 ms with CSR rows, 12.1 ms sorted).
template <class T>
struct ClMat {
    const int64_t* sp;
    const int32_t* sci;
    const T* sv;
    const int32_t* ord;
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
    uint32_t inv;          // ceil(2^32 / R): row / R = umulhi(row, inv) for rows below 2^32 / R
    int units;             // units of this block
    int unit0;             // index of its first unit in the system
    int nunits;            // units of the system
};

__device__ __forceinline__ ClRows cl_rows(int n, int R, int rank)
{
    ClRows W;
    W.n = n;
    W.R = R;
    W.base = rank * R;
    W.nrow = max(0, min(R, n - W.base));
    W.inv = (uint32_t)((0x100000000ull + (unsigned)R - 1) / (unsigned)R);
    W.units = (W.nrow + CL_UNIT - 1) / CL_UNIT;
    W.unit0 = W.base / CL_UNIT;
    W.nunits = (n + CL_UNIT - 1) / CL_UNIT;
    return W;
}

// dst = A src (MODE 0), dst += A src (1) or dst = b - A src (2) on the block's
// rows, src spread over the cluster. A warp takes 64 positions, two per lane.
// Not inlined: the kernels are one long pass per iteration, and its copies
// would push that pass out of the instruction cache. Ends without a barrier.
template <class T, bool MULTI, int MODE>
__device__ __noinline__ void cl_apply(const ClMat<T>* Am, const ClRows* Wp, const T* src, T* dst, const T* b)
{
    const ClMat<T> A = *Am;
    const ClRows W = *Wp;
    const int lane = threadIdx.x & 31;
    const uint32_t sa = smem_u32(src);
    __builtin_assume(__isShared(src));
    __builtin_assume(__isShared(dst));
    // BT entries of both rows at a time: their indices and values, then their
    // gathers (from this block's shared memory when all of the warp's columns
    // are its own, as most are on a grid: 30 cycles against 250 across the
    // cluster), then their products in order
    constexpr int BT = sizeof(T) == 4 ? 8 : 4;
#pragma unroll 1
    for (int q = threadIdx.x >> 5; q < W.units; q += blockDim.x >> 5) {
        const int32_t* ci[2];
        const T* va[2];
        int len[2], row[2];
        T y[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int at = q * CL_UNIT + 32 * h;
            const bool in = at < W.nrow;
            const int64_t sl = (W.base + at) / 32;
            const int64_t e0 = in ? A.sp[sl] : 0, e1 = in ? A.sp[sl + 1] : 0;
            row[h] = !in ? -1 : A.ord ? A.ord[W.base + at + lane] : (at + lane < W.nrow ? at + lane : -1);
            ci[h] = A.sci + e0 + lane;
            va[h] = A.sv + e0 + lane;
            len[h] = (int)(e1 - e0) / 32;
            y[h] = 0;
        }
        const int most = max(len[0], len[1]);  // the same in every lane: the votes below need all of them
#pragma unroll 1
        for (int k0 = 0; k0 < most; k0 += BT) {
            int col[2][BT];
            T a[2][BT], xv[2][BT];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int u = 0; u < BT; ++u) {
                    const bool in = k0 + u < len[h];
                    col[h][u] = in ? __ldg(ci[h] + (k0 + u) * 32) : -1;
                    a[h][u] = in ? __ldg(va[h] + (k0 + u) * 32) : T(0);
                }
            bool own = true;
            if (MULTI) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int u = 0; u < BT; ++u) own &= col[h][u] < 0 || (unsigned)(col[h][u] - W.base) < (unsigned)W.R;
                own = __all_sync(SAI_FULL, own);
            }
            if (!MULTI || own) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int u = 0; u < BT; ++u) xv[h][u] = src[max(col[h][u], W.base) - W.base];
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int u = 0; u < BT; ++u) {
                        const uint32_t j = (uint32_t)max(col[h][u], 0), rk = __umulhi(j, W.inv);
                        xv[h][u] = cl_ld<T>(cl_map(sa + (uint32_t)sizeof(T) * (j - rk * (uint32_t)W.R), rk));
                    }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int u = 0; u < BT; ++u)
                    if (col[h][u] >= 0) y[h] = fma(a[h][u], xv[h][u], y[h]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (row[h] >= 0) {
                if (MODE == 0) dst[row[h]] = y[h];
                else if (MODE == 1) dst[row[h]] += y[h];
                else dst[row[h]] = b[row[h]] - y[h];
            }
    }
}

// The matrix of a cluster kernel: its sliced-ELL copy, or the sorted form of
// its CSR arrays for C blocks of R rows in buf (live until the kernel has run).
template <class T>
sai_status cl_matrix(const Mat<T>& X, int n, int R, int C, Buf (&buf)[4], ClMat<T>& out, cudaStream_t st)
{
    if (X.sp) {
        out = {X.sp, X.sci, X.sv, nullptr};
        return SAI_OK;
    }
    SAI_TRY(sorted_rows<T>(RowBlocks{n, R, nullptr}, C, X.rp, X.ci, X.v, buf, st));
    out = {buf[1].as<int64_t>(), buf[2].as<int32_t>(), buf[3].as<T>(), buf[0].as<int32_t>()};
    return SAI_OK;
}

// The two matrices of a cluster kernel, formed once per call of the solver (a
// refined solve runs GMRES once per outer step; the blocks stay the same).
template <class T>
struct ClPair {
    ClMat<T> A, M;
    Buf ab[4], mb[4];
    bool ready = false;
    // SAI_OOM: no memory for the sorted forms, of which the multi-kernel form needs none
    sai_status form(const Mat<T>& a, const Mat<T>& m, int n, int R, int C, cudaStream_t st)
    {
        if (ready) return SAI_OK;
        SAI_TRY(cl_matrix(a, n, R, C, ab, A, st));
        SAI_TRY(cl_matrix(m, n, R, C, mb, M, st));
        ready = true;
        return SAI_OK;
    }
};

// Stores a unit's partial sum in slot `slot` of every block of the cluster.
template <bool MULTI>
__device__ __noinline__ void cl_put(double v, int slot, int unit, double* parts, int pstride, int nranks)
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
__device__ __noinline__ double cl_total(const double* parts, int slot, int pstride, int nunits, bool comp)
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

// One cluster per system (blockIdx.x / cluster size). B, X: the system's vectors at c * ld.
template <bool MULTI>
__global__ void __launch_bounds__(CL_T, 1)
k_bicg_cluster(ClMat<double> A, ClMat<double> M, int n, int64_t ld, int rmax, int umax,
               const double* __restrict__ B, double* __restrict__ X, const double* __restrict__ thr, int maxit,
               int* __restrict__ iters, int* __restrict__ status)
{
    extern __shared__ __align__(16) double sm[];
    // alpha, omega, beta, alpha / (omega rho f), rho of the running iteration, f = the power of two that
    // takes rho near 1 (the quotient must not overflow where rho is small, as it is when b is)
    __shared__ double sc[6];
    __shared__ int flag;      // 0 go on (first iteration), 1 half step, then stop, 2 stop, 3 go on
    uint32_t rank = 0, nranks = 1;
    if (MULTI) {
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nranks));
    }
    const int c = blockIdx.x / nranks;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int NW = CL_T / 32;
    __shared__ ClRows W;
    __shared__ ClMat<double> As, Ms;
    if (threadIdx.x == 0) {
        W = cl_rows(n, rmax, (int)rank);
        As = A;
        Ms = M;
    }
    __syncthreads();
    const int64_t o = (int64_t)c * ld + W.base;
    double *p = sm, *ph = p + rmax, *s = ph + rmax, *sh = s + rmax;  // gathered by the cluster
    double *r = sh + rmax, *rh = r + rmax, *v = rh + rmax, *t = v + rmax, *x = t + rmax;
    double* parts = x + rmax;  // [slot][unit]
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
        if (lane == 0) sc[2] = it == 1 ? 0.0 : rho * sc[5] * sc[3];
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
        cl_apply<double, MULTI, 0>(&Ms, &W, p, ph, nullptr);
        cl_barrier<MULTI>();
        cl_apply<double, MULTI, 0>(&As, &W, ph, v, nullptr);
        __syncthreads();
        for (int u = wid; u < W.units; u += NW) {
            const int i = u * CL_UNIT + lane;
            cl_put<MULTI>(fma(rh[i + 32], v[i + 32], rh[i] * v[i]), 0, W.unit0 + u, parts, umax, (int)nranks);
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
        cl_apply<double, MULTI, 0>(&Ms, &W, s, sh, nullptr);
        cl_barrier<MULTI>();
        cl_apply<double, MULTI, 0>(&As, &W, sh, t, nullptr);
        __syncthreads();
        for (int u = wid; u < W.units; u += NW) {
            const int i = u * CL_UNIT + lane;
            cl_put<MULTI>(fma(t[i + 32], s[i + 32], t[i] * s[i]), 2, W.unit0 + u, parts, umax, (int)nranks);
            cl_put<MULTI>(fma(t[i + 32], t[i + 32], t[i] * t[i]), 3, W.unit0 + u, parts, umax, (int)nranks);
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
            if (wid == NW - 1 && lane == 0) {
                const int e = ((__double2hiint(sc[4]) >> 20) & 0x7ff) - 1023;
                const double f = __hiloint2double((1023 - min(max(e, -1022), 1022)) << 20, 0);
                sc[5] = f;
                sc[3] = al / (om * (sc[4] * f));
            }
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

// Clusters of C blocks of kern that the GPU holds at once, by log2 C (0: not
// asked yet). A block's registers leave room for no second one on its SM
// whatever its shared memory, so the answer depends on the GPU and C alone and is
// kept: asking takes 20 to 30 us, 2% of a small solve.
using ClHeld = std::atomic<int>[5];

// true when the GPU holds k clusters of C blocks of kern at once (fewer than its
// SMs suggest: a cluster stays within one group of them, and sixteen clusters of
// eight blocks take two rounds on 152 SMs); limit: the most dynamic shared memory
// of kern's launches
template <class... Params>
bool cl_fits(void (*kern)(Params...), int k, int C, int threads, size_t limit, ClHeld& held)
{
    if ((int64_t)C * k > g_sms) return false;
    if (C <= CL_MAXC && (int64_t)2 * C * k <= g_sms) return true;
    int lg = 0;
    while ((1 << lg) < C) ++lg;
    if (held[lg].load(std::memory_order_relaxed) > 0) return held[lg].load(std::memory_order_relaxed) >= k;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C * (unsigned)k);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = limit;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int most = 0;
    const bool ok = (C <= CL_MAXC ||
                     cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
                    sai_smem_limit(kern, limit) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&most, kern, &cfg) == cudaSuccess;
    if (!ok) (void)cudaGetLastError();
    if (ok && most > 0) held[lg].store(most, std::memory_order_relaxed);
    return ok && most >= k;
}

// Launches kern with k clusters of C blocks; false when the device refuses the shape.
template <class... Params, class... Args>
bool cl_run(void (*kern)(Params...), int k, int C, int threads, size_t limit, size_t smem, cudaStream_t st, Args... args)
{
    if (sai_smem_limit(kern, limit) != cudaSuccess ||
        (C > CL_MAXC && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
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

// BiCGStab of k systems in clusters; *ran is false when the form does not take
// them or the device refuses the shape.
inline sai_status cl_bicgstab(const Ops<double>& A, int k, int n, int64_t ld, const double* B, double* X,
                              const double* thr, int maxit, int* iters, int* status, cudaStream_t st, bool* ran)
{
    *ran = false;
    if (n > CL_MAXN || k > (n > CL_MANY_N ? CL_MANY_K : CL_MAXK) || (n > CL_FAR_N && A.scattered)) return SAI_OK;
    const int umax = (n + CL_UNIT - 1) / CL_UNIT;
    auto rows = [&](int blocks) { return ((n + blocks - 1) / blocks + CL_UNIT - 1) / CL_UNIT * CL_UNIT; };
    auto bytes = [&](int blocks) {
        return sizeof(double) * ((size_t)CL_VECS * rows(blocks) + (size_t)CL_SLOTS * umax);
    };
    static ClHeld held;
    auto fits = [&](int blocks) { return cl_fits(k_bicg_cluster<true>, k, blocks, CL_T, CL_SMEM, held); };
    // enough blocks for the rows, then as many as leave every system on the GPU
    // at once with two units of rows per block (the reductions' cost does not
    // shrink with more); sixteen where the FP64 pipe outweighs the barriers, from
    // 512 rows per block on
    int C = 1;
    while (C < CL_MAXC && (int64_t)C * CL_MAXR < n) C *= 2;
    while (C < CL_MAXC && n / (2 * C) >= 2 * CL_UNIT && fits(2 * C)) C *= 2;
    if (C == CL_MAXC && rows(C) >= 512 && fits(16)) C = 16;
    const int rmax = rows(C);
    const size_t smem = bytes(C);
    ClPair<double> F;
    const sai_status fs = F.form(A.A, A.M, n, rmax, C, st);
    if (fs == SAI_OOM) return SAI_OK;
    SAI_TRY(fs);
    *ran = cl_run(C > 1 ? k_bicg_cluster<true> : k_bicg_cluster<false>, k, C, CL_T, CL_SMEM, smem, st, F.A, F.M, n, ld, rmax,
                  umax, B, X, thr, maxit, iters, status);
    return SAI_OK;
}
