// gmres_cluster.cuh -- restarted GMRES of one system in one thread-block
// cluster (included by krylov.cu inside its namespace).
//
// The Arnoldi process with delayed re-orthogonalisation of k_dc_dots /
// k_dc_step / k_dc_update, restarts included, without leaving the kernel: at
// small orders a step of the multi-kernel form is five launches that wait for
// one another (45 us at 35937 rows and 6 systems, most of it latency; the
// whole call 10.4 ms, 6.9 ms here). Block
// b of the cluster owns rows [b R, (b + 1) R): the candidate u, t = M u, z =
// A~ t and x live in its shared memory, its rows of the basis in global
// memory (read by this block only, so from L1 while they fit). Products
// gather u, t and x across the cluster; a step has three cluster barriers.
// Every block keeps the small Hessenberg problem itself and runs the same
// control arithmetic on the same sums, so no value has to be sent back.
//
// A system's bits depend on n, m, T and the matrices, not on the systems that
// run with it: the number of blocks follows k, but a sum is a tree per unit of
// rows (GcUnits, gc_dots) and the units' sums added pairwise in FP64, each block
// holding whole units. With sums per block instead, this form took 2.94, 4.02
// and 11.7 ms where it takes 2.90, 4.2 and 12.2 (35937 rows in FP32, 6, 11 and 40
// systems, 101 steps), and 6.3 where it takes 6.8 (1728 rows in FP64, 256
// systems, 60 steps). The Hessenberg columns are kept in T, the type k_dc_step
// uses them in (its rotated columns are T values stored as FP64).

constexpr int GC_T = 512;      // threads per block
constexpr int GC_UT = GC_T - 32;  // of them in the update; the last warp runs the Givens rotations meanwhile
constexpr int GC_MAXU = 16;    // units of a system
constexpr int GC_MAXR = 6144;  // rows per block
// orders up to which the form is used, by n alone. FP32: at 46656 rows a few
// systems take 3.08, 3.10 and 4.93 ms (2, 6 and 11) against 4.37, 5.05 and 6.11 in
// the multi-kernel form, which is the faster one there from 16 systems on (9.7 and
// 7.6 ms, 15.2 and 14.6 with 40, 29.8 and 25.7 with 77); at 35937 rows the two
// meet at 153 systems (43.4 and 42.7; 12.2 and 13.1 with 40). A split's systems are
// its dense columns and one, so the few decide. FP64: above, the
// FP64 pipes of eight SMs are slower than those of all.
constexpr size_t GC_SMEM = 220 * 1024;  // shared memory of a block, at most
constexpr int GC_MAXN32 = 49152, GC_MAXN64 = 10240;
// of a scattered matrix in FP32 (8, 16, 19 and 76 systems of 12000 rows: 2.88,
// 3.9, 4.0 and 4.9 ms against 3.1, 4.0, 4.4 and 12.0; 4, 16 and 76 systems of 20000
// rows 3.0, 7.6 and 16 against 2.7, 4.4 and 13.8)
constexpr int GC_FAR_N32 = 12288;

// Shared-memory layout of one block (bytes from the start).
template <class T>
struct GcLayout {
    size_t u, t, z, x, hb, r, cs, sn, rc, s, c, parts, red, hp, g, y, bytes;
    int ns;  // slots of a unit's partial sums
    GcLayout(int R, int m, int units)
    {
        ns = 2 * m + 4;
        size_t o = 0;
        auto take = [&](size_t b) {
            const size_t at = o;
            o += (b + 15) / 16 * 16;
            return at;
        };
        u = take(sizeof(T) * R);
        t = take(sizeof(T) * R);
        z = take(sizeof(T) * R);
        x = take(sizeof(T) * R);
        hb = take(sizeof(T) * ((size_t)m * (m + 3) / 2));  // Hbar, column q: q + 2 entries from q (q + 3) / 2
        r = take(sizeof(T) * ((size_t)m * (m + 1) / 2));   // R, column q: q + 1 entries from q (q + 1) / 2
        cs = take(sizeof(T) * m);
        sn = take(sizeof(T) * m);
        rc = take(sizeof(T) * (m + 2));
        s = take(sizeof(T) * (m + 1));
        c = take(sizeof(T) * (m + 1));
        parts = take(sizeof(double) * (size_t)units * ns);
        red = take(sizeof(double) * ns);
        hp = take(sizeof(double) * (m + 2));
        g = take(sizeof(double) * (m + 2));
        y = take(sizeof(T) * (m + 1));
        bytes = o;
    }
};

struct GcArgs {
    int n, m, R, k;
    int64_t ld, vs;
    double tiny;
    int units, U, ns;  // GcUnits; ns as in GcLayout
    uint32_t u, t, z, x, hb, r, cs, sn, rc, s, c, parts, red, hp, g, y;  // offsets of GcLayout
};

// two sums over the warp at once: lane 0 gets a's, lane 16 b's
template <class T>
__device__ __forceinline__ T gc_sum2(T a, T b)
{
    const bool up = (threadIdx.x & 16) != 0;
    T w = (up ? b : a) + __shfl_xor_sync(SAI_FULL, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) w += __shfl_xor_sync(SAI_FULL, w, o);
    return w;
}

// The units of a system: a power of two of them, of U rows (the last ones
// fewer, or none). A block of the cluster holds units / C of them, so the order
// of every sum depends on n alone: a tree per unit (gc_dots), and the units'
// sums added pairwise.
struct GcUnits {
    int units, U;
    explicit GcUnits(int n)
    {
        // at least 128 rows per unit; sixteen from 512 rows per eighth on, where the work outweighs the barriers
        units = 1;
        while (units < 8 && n / (2 * units) >= 2 * CL_UNIT) units *= 2;
        if (units == 8 && n > 8 * (512 - CL_UNIT)) units = GC_MAXU;
        U = ((n + units - 1) / units + 31) / 32 * 32;
    }
};

template <class T>
struct Comp;  // the components of a Vec<T>
template <>
struct Comp<float> {
    __device__ static void fma4(const float4& a, const float4& b, float4& c)
    {
        c.x = fmaf(a.x, b.x, c.x);
        c.y = fmaf(a.y, b.y, c.y);
        c.z = fmaf(a.z, b.z, c.z);
        c.w = fmaf(a.w, b.w, c.w);
    }
    __device__ static float sum(const float4& a) { return (a.x + a.y) + (a.z + a.w); }
};
template <>
struct Comp<double> {
    __device__ static void fma4(const double2& a, const double2& b, double2& c)
    {
        c.x = fma(a.x, b.x, c.x);
        c.y = fma(a.y, b.y, c.y);
    }
    __device__ static double sum(const double2& a) { return a.x + a.y; }
};

// v^T u and v^T z over rows [at, at + U) below nrow by one warp, in FP32: plain
// sums over at most eight row pieces per lane and component and, for more than
// 512 rows, those and the tree over the lanes with their rounding errors carried
// along. (A plain tree over 2048 rows has twice the error of the multi-kernel
// form's four over 512 rows each, added in FP64.) Lane 0 returns v^T u, lane 16
// v^T z. Two basis vectors at a time, sharing the loads of u and z, were no
// faster; as a call it is slower (13.8 against 13.1 us a step at 2500 rows, 23.7
// against 22.6 at 27000) by the registers saved around it.
__device__ __forceinline__ double gc_dots(const float* v, const float* u, const float* z, int at, int U, int nrow, int)
{
    __builtin_assume(__isShared(u));
    __builtin_assume(__isShared(z));
    const int lane = threadIdx.x & 31, r1 = min(nrow, at + U);
    auto add = [](float& h, float& l, float x) {  // (h, l) += x (Knuth's two-sum)
        const float s = h + x, t = s - h;
        l += (h - (s - t)) + (x - t);
        h = s;
    };
    float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
#pragma unroll 1
    for (int r0 = at + 4 * lane; r0 - 4 * lane < r1;) {
        float4 as = {}, ac = {};
#pragma unroll 1
        for (int half = 0; half < 2; ++half, r0 += 512) {
            float4 x[4];
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (r0 + 128 * s < r1) x[s] = *reinterpret_cast<const float4*>(v + r0 + 128 * s);
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (r0 + 128 * s < r1) {
                    Comp<float>::fma4(x[s], *reinterpret_cast<const float4*>(u + r0 + 128 * s), as);
                    Comp<float>::fma4(x[s], *reinterpret_cast<const float4*>(z + r0 + 128 * s), ac);
                }
        }
        const float a = Comp<float>::sum(as), c = Comp<float>::sum(ac);
        if (U <= 512) return (double)gc_sum2(a, c);
        add(h0, l0, a);
        add(h1, l1, c);
    }
    const bool up = (lane & 16) != 0;
    float h = up ? h1 : h0, l = up ? l1 : l0;
    const float hx = __shfl_xor_sync(SAI_FULL, up ? h0 : h1, 16), lx = __shfl_xor_sync(SAI_FULL, up ? l0 : l1, 16);
    add(h, l, hx);
    l += lx;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        const float hy = __shfl_xor_sync(SAI_FULL, h, o), ly = __shfl_xor_sync(SAI_FULL, l, o);
        add(h, l, hy);
        l += ly;
    }
    return (double)h + (double)l;
}

// Sums a[0..7] over the warp, each with the additions of gc_sum2's tree: lanes
// 4 i to 4 i + 3 get the sum of a[i].
__device__ __forceinline__ double gc_sum8(double (&a)[8])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 2; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o / 4; ++i) {
            const double keep = up ? a[i + o / 4] : a[i], send = up ? a[i] : a[i + o / 4];
            a[i] = keep + __shfl_xor_sync(SAI_FULL, send, o);
        }
    }
    double w = a[0];
    w += __shfl_xor_sync(SAI_FULL, w, 2);
    return w + __shfl_xor_sync(SAI_FULL, w, 1);
}

// The same in FP64 for 2 or 4 units of U rows at a time, whose trees share their
// additions (9 for four units, 5 for one). Unit e's sums: lanes 8 e and 8 e + 4.
__device__ __noinline__ double gc_dots_units(const double* v, const double* u, const double* z, int at, int U, int nrow, int uw)
{
    __builtin_assume(__isShared(u));
    __builtin_assume(__isShared(z));
    const int lane = threadIdx.x & 31;
    double sums[8];
#pragma unroll
    for (int e = 0; e < 4; ++e, at += U) {
        const int r1 = e < uw ? min(nrow, at + U) : 0;
        double a = 0.0, b = 0.0;
#pragma unroll 1
        for (int r0 = at + 2 * lane; r0 - 2 * lane < r1; r0 += 256) {
            double2 x[4];
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (r0 + 64 * s < r1) x[s] = *reinterpret_cast<const double2*>(v + r0 + 64 * s);
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (r0 + 64 * s < r1) {
                    a = Vec<double>::dot(x[s], *reinterpret_cast<const double2*>(u + r0 + 64 * s), a);
                    b = Vec<double>::dot(x[s], *reinterpret_cast<const double2*>(z + r0 + 64 * s), b);
                }
        }
        sums[2 * e] = a;
        sums[2 * e + 1] = b;
    }
    return gc_sum8(sums);
}

// uw units in FP64; one alone in line (2401 rows: a step 26.9 -> 24.1 us)
__device__ __forceinline__ double gc_dots(const double* v, const double* u, const double* z, int at, int U, int nrow, int uw)
{
    if (uw > 1) return gc_dots_units(v, u, z, at, U, nrow, uw);
    const int r1 = min(nrow, at + U);
    double a = 0.0, b = 0.0;
#pragma unroll 4
    for (int r = at + 2 * (threadIdx.x & 31); r < r1; r += 64) {
        const double2 x = *reinterpret_cast<const double2*>(v + r);
        a = Vec<double>::dot(x, *reinterpret_cast<const double2*>(u + r), a);
        b = Vec<double>::dot(x, *reinterpret_cast<const double2*>(z + r), b);
    }
    return gc_sum2(a, b);
}

// v_j = ia (u - V s), u <- ia (z - V c - dd v_j) on the block's rows: a thread
// per row (W = 1) or per 16-byte piece
template <class T, int W>
__device__ __forceinline__ void gc_update(int j, int nrow, const T* V, int64_t vs, T* Vj, T* u, const T* z, const T* sT,
                                          const T* cT, T ia, T dd)
{
    for (int r = (int)threadIdx.x * W; r < nrow; r += GC_UT * W) {
        T a_s[W], a_c[W];
#pragma unroll
        for (int e = 0; e < W; ++e) a_s[e] = a_c[e] = 0;
        for (int i0 = 0; i0 < j; i0 += 8) {
            T v[8][W];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const bool in = i0 + q < j;
                const T* p = V + (int64_t)(in ? i0 + q : i0) * vs + r;
                if (W == 1) {
                    v[q][0] = in ? *p : T(0);
                } else {
                    const typename Vec<T>::type x = *reinterpret_cast<const typename Vec<T>::type*>(p);
                    const T* xe = reinterpret_cast<const T*>(&x);
#pragma unroll
                    for (int e = 0; e < W; ++e) v[q][e] = in ? xe[e] : T(0);
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (i0 + q < j) {
                    const T s = sT[i0 + q], c = cT[i0 + q];
#pragma unroll
                    for (int e = 0; e < W; ++e) {
                        a_s[e] = fma(s, v[q][e], a_s[e]);
                        a_c[e] = fma(c, v[q][e], a_c[e]);
                    }
                }
        }
#pragma unroll
        for (int e = 0; e < W; ++e)
            if (r + e < nrow) {
                const T v = ia * (u[r + e] - a_s[e]);
                Vj[r + e] = v;
                u[r + e] = ia * fma(-dd, v, z[r + e] - a_c[e]);
            }
    }
}

template <class T, bool MULTI>
__global__ void __launch_bounds__(GC_T, 1)
k_gmres_cluster(ClMat<T> A, ClMat<T> M, GcArgs P, Basis<T> Bv, const T* __restrict__ B, T* __restrict__ X,
                const double* __restrict__ thr, const int* __restrict__ cap, int* __restrict__ iters,
                int* __restrict__ status, Dims D)
{
    using VT = typename Vec<T>::type;
    constexpr int VW = Vec<T>::W;
    constexpr int NW = GC_T / 32;
    extern __shared__ __align__(16) unsigned char gsm[];
    __shared__ double sh[3];  // alpha, d, 1 / alpha
    __shared__ int flag;      // of the last control step: 0 go on, 1 the cycle ends
    __shared__ int done;      // of the cycle's end: 0 another cycle, 1 stop
    uint32_t rank = 0, nranks = 1;
    if (MULTI) {
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nranks));
    }
    const int c = blockIdx.x / nranks;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int m = P.m;
    __shared__ ClRows W;
    __shared__ ClMat<T> As, Ms;
    if (tid == 0) {
        W = cl_rows(P.n, P.R, (int)rank);
        As = A;
        Ms = M;
    }
    __syncthreads();
    const int64_t o = (int64_t)c * P.ld + W.base;
    T* V = Bv.V + o;  // the block's rows of v_0; v_i at V + i vs
    T *u = (T*)(gsm + P.u), *t = (T*)(gsm + P.t), *z = (T*)(gsm + P.z), *x = (T*)(gsm + P.x);
    T *hb = (T*)(gsm + P.hb), *Rm = (T*)(gsm + P.r), *cs = (T*)(gsm + P.cs), *sn = (T*)(gsm + P.sn), *rc = (T*)(gsm + P.rc);
    T *sT = (T*)(gsm + P.s), *cT = (T*)(gsm + P.c), *yT = (T*)(gsm + P.y);
    double *parts = (double*)(gsm + P.parts), *red = (double*)(gsm + P.red), *hp = (double*)(gsm + P.hp), *g = (double*)(gsm + P.g);
    const double th = thr[c];
    const int most = cap[c];
    int it = 0, stat = ST_OK;         // the same in every thread of the cluster
    double wsteps = 0.0, wj = 0.0;    // work: steps, and basis vectors over the steps
    const int lr = 31 - __clz((int)nranks), ub = P.units >> lr;  // ub: units of this block
    // v^T u and v^T zz on units g w to g w + w - 1 of the block, stored in slots sl, sl + 1 of every block (one warp; the
    // sums do not depend on w)
    auto dots = [&](const T* v, const T* zz, int g, int w, int sl) {
        const double d = gc_dots(v, u, zz, g * w * P.U, P.U, W.nrow, w);
        // a store per lane: (unit, part, block)
        const int vi = lane >> lr, to = lane & ((int)nranks - 1);
        const int e = vi >> 1, b = vi & 1;
        const double val = __shfl_sync(SAI_FULL, d, (w > 1 ? 8 * e + 4 * b : 16 * b) & 31);
        if (vi < 2 * w) {
            double* p = parts + (size_t)((int)rank * ub + g * w + e) * P.ns + sl + b;
            if (MULTI) cl_st(cl_map(smem_u32(p), (uint32_t)to), val);
            else *p = val;
        }
    };
    // red[t] = the sum of slot t over the units, t < cnt
    auto total = [&](int cnt) {
        for (int q = tid; q < cnt; q += GC_T) {
            auto eight = [&](int e0) {  // of units e0 to e0 + 7
                double a[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) a[e] = e0 + e < P.units ? parts[(size_t)(e0 + e) * P.ns + q] : 0.0;
#pragma unroll
                for (int w = 1; w < 8; w *= 2)
                    if (w < P.units)
#pragma unroll
                        for (int e = 0; e < 8; e += 2 * w) a[e] += a[e + w];
                return a[0];
            };
            double a = eight(0);
            if (P.units > 8) a += eight(8);
            red[q] = a;
        }
        __syncthreads();
    };
    // the block's rows of u = r: ||r||^2 into slot 0 (and 1)
    auto norm = [&]() {
        for (int g = wid; g < ub; g += NW) dots(u, u, g, 1, 0);
    };
    for (int i = tid; i < P.R; i += GC_T) {
        u[i] = i < W.nrow ? B[o + i] : T(0);
        t[i] = z[i] = x[i] = 0;
    }
    __syncthreads();
    cl_barrier<MULTI>();  // every block of the cluster runs before its memory is written
    norm();
    cl_barrier<MULTI>();
    for (;;) {
        // cycle start: true residual norm, stop tests
        total(1);
        const double beta = sqrt(red[0]);
        if (beta < th) {
            stat = ST_OK;
            break;
        }
        if (it >= most) {
            stat = ST_MAXITER;
            break;
        }
        int jd = 0;
        bool conv = false;
        for (int j = 0; j <= m; ++j) {
            if (j < m) {  // the last step of a cycle needs no operator application
                cl_apply<T, MULTI, 0>(&Ms, &W, u, t, nullptr);
                cl_barrier<MULTI>();
                cl_apply<T, MULTI, 0>(&As, &W, t, z, nullptr);
                __syncthreads();
            }
            // s = V^T u, c = V^T z (slots 2 i, 2 i + 1), u^T u, u^T z (2 j, 2 j + 1)
            int w = sizeof(T) == 4 ? 1 : min(4, ub);  // units a warp takes at a time: fewer while warps would idle
            while (w > 1 && (j + 1) * (ub / w) < NW) w >>= 1;
            const int lu = 31 - __clz(ub / w);
            for (int q = wid; q < (j + 1) << lu; q += NW) {
                const int i = q >> lu;
                dots(i < j ? V + (int64_t)i * P.vs : u, z, q - (i << lu), w, 2 * i);
            }
            cl_barrier<MULTI>();
            total(2 * j + 2);
            wsteps += 1.0;
            wj += j;
            // alpha, d = v_j^T z
            if (wid == 0) {
                double ss = 0.0, sc = 0.0;
                for (int i = lane; i < j; i += 32) {
                    ss = fma(red[2 * i], red[2 * i], ss);
                    sc = fma(red[2 * i], red[2 * i + 1], sc);
                }
                const double w = gc_sum2(ss, sc);
                ss = __shfl_sync(SAI_FULL, w, 0);
                sc = __shfl_sync(SAI_FULL, w, 16);
                const double uu = red[2 * j], a2 = uu - ss;
                const bool ok = a2 > P.tiny * uu;
                const double ial = ok ? rsqrt(a2) : 0.0;
                if (lane == 0) {
                    sh[0] = ok ? a2 * ial : 0.0;
                    sh[1] = (red[2 * j + 1] - sc) * ial;
                    sh[2] = ial;
                }
            }
            for (int i = tid; i < j; i += GC_T) {
                sT[i] = (T)red[2 * i];
                cT[i] = (T)red[2 * i + 1];
            }
            __syncthreads();
            const double al = sh[0], d = sh[1], ial = sh[2];
            if (j >= 1) {
                // column j - 1: first-pass coefficients + s, subdiagonal alpha
                T* hc = hb + (size_t)(j - 1) * (j + 2) / 2;
                for (int i = tid; i <= j; i += GC_T) hc[i] = rc[i] = (T)(i < j ? hp[i] + red[2 * i] : al);
                ++it;
                jd = j;
            }
            __syncthreads();
            // column j - 1 rotated, the residual estimate and the stop tests by
            // the last warp, whose result the others need only after the update
            // (a stopping step's update is not used)
            if (tid == GC_UT) {
                if (j >= 1) {
                    T* rr = Rm + (size_t)(j - 1) * j / 2;
                    T ri = rc[0];
                    for (int i = 0; i < j - 1; ++i) {
                        const T b = rc[i + 1], ci = cs[i], si = sn[i];
                        rr[i] = ci * ri + si * b;
                        ri = -si * ri + ci * b;
                    }
                    const T a = ri, b = rc[j];
                    const T den = sqrt(a * a + b * b);
                    const T cn = den == (T)0 ? (T)1 : a / den, s_ = den == (T)0 ? (T)0 : b / den;
                    cs[j - 1] = cn;
                    sn[j - 1] = s_;
                    rr[j - 1] = cn * a + s_ * b;
                    const T gj1 = (T)g[j - 1];
                    const double gj = (double)(-s_ * gj1);
                    g[j] = gj;
                    g[j - 1] = (double)(cn * gj1);
                    // bit 0: the cycle ends; bit 1: converged
                    flag = fabs(gj) < th ? 3 : (al == 0.0 || it >= most || j >= m ? 1 : 0);
                } else {
                    g[0] = al;  // v_0 = r0 / alpha
                    flag = al == 0.0 ? 3 : 0;
                }
            }
            // first-pass coefficients of column j: ([c; d] - Hbar s) / alpha
            for (int i = tid; i <= j && tid < GC_UT; i += GC_UT) {
                T hs = 0;
                for (int q = i > 0 ? i - 1 : 0; q < j; ++q) hs = fma(hb[(size_t)q * (q + 3) / 2 + i], sT[q], hs);
                const double cz = i < j ? red[2 * i + 1] : d;
                hp[i] = (cz - (double)hs) * ial;
            }
            if (tid < GC_UT) {
                if (W.nrow >= GC_T * 2)
                    gc_update<T, VW>(j, W.nrow, V, P.vs, V + (int64_t)j * P.vs, u, z, sT, cT, (T)ial, (T)d);
                else
                    gc_update<T, 1>(j, W.nrow, V, P.vs, V + (int64_t)j * P.vs, u, z, sT, cT, (T)ial, (T)d);
            }
            cl_barrier<MULTI>();  // u is gathered next; red, hp, flag are rewritten after it
            const int f = flag;
            if (f) {
                conv = (f & 2) != 0;
                break;
            }
        }
        __syncthreads();
        // y = R^{-1} g by one warp, column by column, with the pivots' reciprocals
        if (wid == 0) {
            constexpr int RPL = GM_MAXM / 32;
            double w[RPL], rd[RPL];
            bool bad = false;
#pragma unroll
            for (int q = 0; q < RPL; ++q) {
                const int i = lane + 32 * q;
                w[q] = i < jd ? g[i] : 0.0;
                const double dg = i < jd ? (double)Rm[(size_t)i * (i + 1) / 2 + i] : 1.0;
                bad |= dg == 0.0;
                rd[q] = 1.0 / dg;
            }
            bad = __any_sync(SAI_FULL, bad);
            for (int q = jd - 1; q >= 0; --q) {
                double yq = 0.0;
#pragma unroll
                for (int e = 0; e < RPL; ++e)
                    if (q / 32 == e) {
                        if (lane == q % 32) w[e] = div_by(w[e], (double)Rm[(size_t)q * (q + 1) / 2 + q], rd[e]);
                        yq = __shfl_sync(SAI_FULL, w[e], q % 32);
                    }
#pragma unroll
                for (int e = 0; e < RPL; ++e) {
                    const int i = lane + 32 * e;
                    if (32 * e < q && i < q) w[e] = fma(-(double)Rm[(size_t)q * (q + 1) / 2 + i], yq, w[e]);
                }
            }
#pragma unroll
            for (int q = 0; q < RPL; ++q)
                if (lane + 32 * q < jd) yT[lane + 32 * q] = (T)w[q];
            if (lane == 0) done = bad;
        }
        __syncthreads();
        if (done) {
            stat = ST_BREAKDOWN;
            break;
        }
        // u = V y, x += M u
        for (int r = tid; r < W.nrow; r += GC_T) {
            T a = 0;
#pragma unroll 8
            for (int i = 0; i < jd; ++i) a = fma(yT[i], V[(int64_t)i * P.vs + r], a);
            u[r] = a;
        }
        cl_barrier<MULTI>();
        cl_apply<T, MULTI, 1>(&Ms, &W, u, x, nullptr);
        if (conv) {
            stat = ST_OK;
            break;
        }
        if (it >= most) {
            stat = ST_MAXITER;
            break;
        }
        cl_barrier<MULTI>();
        cl_apply<T, MULTI, 2>(&As, &W, x, u, B + o);  // r = b - A~ x
        __syncthreads();
        norm();
        cl_barrier<MULTI>();
    }
    __syncthreads();
    for (int i = tid; i < W.nrow; i += GC_T) X[o + i] = x[i];
    if (rank == 0 && tid == 0) {
        iters[c] = it;
        status[c] = stat;
        const double nz = D.nnzA + D.nnzM;
        kwork_add(D.site_spmm, wsteps * (((4.0 + D.esz) * nz + 16.0 * (D.n + 1)) / P.k + 4.0 * D.esz * D.n),
                  wsteps * 2.0 * nz);
        kwork_add(D.site_dots, D.esz * D.n * (wj + 2.0 * wsteps), D.n * 4.0 * (wj + wsteps));
        kwork_add(D.site_upd, D.esz * D.n * (wj + 4.0 * wsteps), D.n * (4.0 * wj + 6.0 * wsteps));
    }
    cl_barrier<MULTI>();  // no block leaves while another may read its memory
}

// Runs the k systems in clusters when they fit (*ran).
template <class T>
sai_status gc_launch(int n, int64_t ld, int k, int m, const Ops<T>& A, ClPair<T>& F, const T* Bs, T* Xs,
                     const GmWork<T>& Wk, Sys& S, const int* cap, const Dims& D, double tiny, cudaStream_t st, bool* ran)
{
    *ran = false;
    if (n < 1 || n > (sizeof(T) == 4 ? GC_MAXN32 : GC_MAXN64) || (n > (sizeof(T) == 4 ? GC_FAR_N32 : CL_FAR_N) && A.scattered))
        return SAI_OK;
    // whether the form is used depends on n and m alone, as the sums do: a
    // system's bits do not depend on the systems that run with it
    const GcUnits N(n);
    auto rows = [&](int blocks) { return N.U * (N.units / blocks); };
    const int most = N.units < CL_MAXC ? N.units : CL_MAXC;
    int C = 1;
    while (C < most && (rows(C) > GC_MAXR || GcLayout<T>(rows(C), m, N.units).bytes > GC_SMEM)) C *= 2;
    if (rows(C) > GC_MAXR || GcLayout<T>(rows(C), m, N.units).bytes > GC_SMEM) return SAI_OK;
    // then as many blocks as leave every system on the GPU at once
    static ClHeld held;
    auto fits = [&](int blocks) { return cl_fits(k_gmres_cluster<T, true>, k, blocks, GC_T, GC_SMEM, held); };
    while (C < most && fits(2 * C)) C *= 2;
    if (C == CL_MAXC && N.units == GC_MAXU && fits(16)) C = 16;
    const int R = rows(C);
    const GcLayout<T> L(R, m, N.units);
    GcArgs P;
    P.n = n;
    P.m = m;
    P.R = R;
    P.k = k;
    P.ld = ld;
    P.vs = Wk.B.vs;
    P.tiny = tiny;
    P.units = N.units;
    P.U = N.U;
    P.ns = L.ns;
    P.u = (uint32_t)L.u;
    P.t = (uint32_t)L.t;
    P.z = (uint32_t)L.z;
    P.x = (uint32_t)L.x;
    P.hb = (uint32_t)L.hb;
    P.r = (uint32_t)L.r;
    P.cs = (uint32_t)L.cs;
    P.sn = (uint32_t)L.sn;
    P.rc = (uint32_t)L.rc;
    P.s = (uint32_t)L.s;
    P.c = (uint32_t)L.c;
    P.parts = (uint32_t)L.parts;
    P.red = (uint32_t)L.red;
    P.hp = (uint32_t)L.hp;
    P.g = (uint32_t)L.g;
    P.y = (uint32_t)L.y;
    const sai_status fs = F.form(A.A, A.M, n, R, C, st);
    if (fs == SAI_OOM) return SAI_OK;
    SAI_TRY(fs);
    *ran = cl_run(C > 1 ? k_gmres_cluster<T, true> : k_gmres_cluster<T, false>, k, C, GC_T, GC_SMEM, L.bytes, st, F.A, F.M, P,
                  Wk.B, Bs, Xs, (const double*)S.thr, cap, S.iters, S.status, D);
    return SAI_OK;
}
