// internal.h -- host-side declarations shared by the saismw CUDA sources.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "common.cuh"
#include "saismw.h"

// Ownership mode of a device buffer. CALL: lives inside one call, from the
// stream-ordered pool, freed on the call's stream. HANDLE: part of a handle
// returned to the user; up to HANDLE_POOL_MAX bytes from a pool of the
// handles' own (a handle has ten to twelve buffers, and cudaMalloc / cudaFree
// of them took a third of a small split or build), larger ones from
// cudaMalloc. What is free in that pool above HANDLE_POOL_KEEP bytes goes back
// to the driver at the next synchronisation, as destroyed handles' memory
// should; the call pool keeps all of its scratch. A
// handle's creation synchronises its stream before it returns; its pooled
// buffers are freed after the work of every stream that has used the handle
// (HandleUses), on the legacy stream if they come from there, else on a stream
// of their own (the creating one may be gone), from which the next handle's
// creation takes them a little later: 4096 rows split in 0.24 and 0.27 ms.
constexpr size_t HANDLE_POOL_MAX = size_t(32) << 20;
constexpr size_t HANDLE_POOL_KEEP = size_t(256) << 20;  // two handles of 262144 rows
struct Buf {
    void* p = nullptr;
    size_t bytes = 0;
    cudaStream_t st = nullptr;
    int dev = -1;  // device of a HANDLE buffer from the pool (-1: another kind)
    bool async = false;
    Buf() = default;
    Buf(const Buf&) = delete;
    Buf& operator=(const Buf&) = delete;
    ~Buf() { release(); }
    sai_status alloc(size_t nbytes, cudaStream_t s, bool use_async);
    void release();
    // the stream that a pooled HANDLE buffer will be freed on
    void free_on(cudaStream_t s)
    {
        if (dev >= 0) st = s;
    }
    template <class T> T* as() const { return static_cast<T*>(p); }
};

// Exclusive scan of n counts into out[0..n] (out[n] = total), int64 output.
sai_status sai_scan_counts_i32(const int32_t* in, int64_t* out, int64_t n, cudaStream_t st);
sai_status sai_scan_counts_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t st);

// CSC (ncols columns, rows < nrows) -> CSR with ascending column indices.
// Output buffers are allocated in `mode_async` mode on st.
sai_status sai_csc_to_csr(int32_t nrows, int32_t ncols, int64_t nnz, const int64_t* cp, const int32_t* ri,
                          const double* cv, Buf& rp, Buf& ci, Buf& rv, cudaStream_t st, bool mode_async);

// Checks CSC structure on the device: col_ptr[0]=0, nondecreasing, last = nnz,
// rows in [0,nrows) strictly ascending per column.
sai_status sai_validate_csc(int32_t nrows, int32_t ncols, int64_t nnz, const int64_t* cp, const int32_t* ri,
                            cudaStream_t st);

// Y = A X (mode 0) or Y = B - A X (mode 1), A in CSR (n rows), X/Y/B n x k row-major.
sai_status sai_spmm(int32_t n, const int64_t* rp, const int32_t* ci, const double* v, int32_t k, const double* X,
                    double* Y, const double* B, int mode, cudaStream_t st);

// y = A x for a CSC matrix via gather over a CSR copy is done by callers; this
// helper computes ||b - A x||^2 and ||b||^2 with A in CSC (one pass, atomics-free).
sai_status sai_csc_residual_norms(int32_t n, const int64_t* cp, const int32_t* ri, const double* cv,
                                  const double* b, const double* x, double* out2_host, cudaStream_t st);

// Handle internals --------------------------------------------------------
// Library-owned non-blocking stream of the current device on which handles'
// pooled buffers are freed (nothing else runs on it, and it is never captured),
// or nullptr; and the pool they come from, nullptr without either.
cudaStream_t sai_free_stream();
cudaMemPool_t sai_handle_pool();

// The streams that have used a handle, each with an event behind its last use.
// A handle's destruction makes the freeing stream wait for these events. It does
// not synchronise the device: that is not permitted while another thread
// captures a stream (every GMRES call of a large order does) and would break
// that capture.
class HandleUses {
  public:
    // The work enqueued on st so far may use the handle. A stream in capture
    // runs nothing: whoever replays its graph keeps the handle alive.
    void record(cudaStream_t st);
    // The stream to free the handle's buffers on (b: one of them), ordered after every recorded use.
    cudaStream_t before_free(const Buf& b);

  private:
    static constexpr int MAX = 16;  // further streams share the last event
    std::mutex mu;
    int cnt = 0, dev = -1;
    cudaStream_t st[MAX];
    cudaEvent_t ev[MAX];
};

struct sai_split_s {
    sai_split_s() = default;
    ~sai_split_s()
    {
        const cudaStream_t f = uses.before_free(J);
        for (Buf* b : {&At_cp, &At_ri, &At_v, &Atr_rp, &Atr_ci, &Atr_v, &U_cp, &U_ri, &U_v, &J, &colnorm2}) b->free_on(f);
    }
    mutable HandleUses uses;
    int32_t n = 0, s = 0, p = 0, p_keep = 0;
    double tau = 0.0, norm1 = 0.0;
    int64_t nnz_At = 0, nnz_U = 0;
    Buf At_cp, At_ri, At_v;      // CSC of A~
    Buf Atr_rp, Atr_ci, Atr_v;   // CSR of A~
    Buf U_cp, U_ri, U_v;         // CSC of U (n x s)
    Buf J;                       // int32[s]
    Buf colnorm2;                // ||A~ e_j||^2
    float ms = 0.f;
};

struct sai_precond_s {
    sai_precond_s() = default;
    ~sai_precond_s()
    {
        const cudaStream_t f = uses.before_free(loops);
        for (Buf* b : {&M_cp, &M_ri, &M_v, &Mr_rp, &Mr_ci, &Mr_v, &loops, &res, &res_post}) b->free_on(f);
    }
    mutable HandleUses uses;
    int32_t n = 0;
    int64_t nnz = 0;
    int32_t n_c = 0, l_m = 0;
    int32_t n_tier[6] = {0, 0, 0, 0, 0, 0};
    float ms = 0.f;
    Buf M_cp, M_ri, M_v;     // CSC
    Buf Mr_rp, Mr_ci, Mr_v;  // CSR
    Buf loops, res, res_post;
};

// Records the use of handles (nullptr: none) by a call on st when it ends, unless
// it ended synchronised: an error may leave work in flight.
struct HandleUse {
    const sai_split_s* h;
    const sai_precond_s* P;
    cudaStream_t st;
    bool idle = false;
    // passes on the status of a call that synchronises st before it returns without an error
    sai_status synced(sai_status r)
    {
        idle = r == SAI_OK || r == SAI_MAXITER || r == SAI_BREAKDOWN;
        return r;
    }
    ~HandleUse()
    {
        if (h && !idle) h->uses.record(st);
        if (P && !idle) P->uses.record(st);
    }
};

sai_status sai_split_build(const sai_csc_view* A, const sai_split_params* prm, cudaStream_t st, bool async,
                           sai_split_s* h);
sai_status sai_spai_build(const sai_split_s* h, const sai_spai_params* prm, cudaStream_t st, bool async,
                          sai_precond_s* P);
sai_status sai_psai_build(const sai_split_s* h, const sai_psai_params* prm, cudaStream_t st, bool async,
                          sai_precond_s* P);
sai_status sai_krylov_run(const sai_split_s* h, const sai_precond_s* P, int32_t k, const double* B,
                          const double* thr, const sai_krylov_params* prm, double* X, int32_t* iters,
                          int32_t* status, cudaStream_t st);
sai_status sai_smw_run(const sai_split_s* h, const double* Y, double* x, double* c_out, cudaStream_t st);
sai_status sai_build_autotune_run(const sai_split_s* h, int32_t sai, const sai_spai_params* sp,
                                  const sai_psai_params* pp, cudaStream_t st, sai_build_tuning* out);
sai_status sai_build_set_config_run(const sai_build_config* cfg);
// Theorem 1 for A^T = A~^T + V U^T: x = yhat - What (I + U^T What)^{-1} (U^T yhat)
sai_status sai_smw_adj_run(const sai_split_s* h, const double* Y, double* x, double* c_out, cudaStream_t st);

// Zero-diagonal repair (section 5): maximum transversal p (p[j] = row of
// column j, -1 if unmatched), B = A(p,:), and y = x(p).
sai_status sai_dmperm_run(const sai_csc_view* A, int32_t* p, int32_t* rank_out, int32_t* moved_out, cudaStream_t st);
sai_status sai_permute_rows_run(const sai_csc_view* A, const int32_t* p, int64_t* Bcp, int32_t* Bri, double* Bv,
                                cudaStream_t st);
sai_status sai_gather_vec(int32_t n, const int32_t* p, const double* x, double* y, cudaStream_t st);

void sai_pool_init_once();
// A library-owned non-blocking stream of the current device for graph capture
// and replay, held by one call at a time (of two calls that capture on one
// stream the second would join, or end, the first one's capture) and given back
// at the end of the scope. s is nullptr when no stream can be had.
struct AuxStream {
    cudaStream_t s = nullptr;
    int dev = -1;
    void lease();
    AuxStream() = default;
    AuxStream(const AuxStream&) = delete;
    AuxStream& operator=(const AuxStream&) = delete;
    ~AuxStream();
};

// Device-side algorithmic work per profiled site ([site][0] bytes, [1] flops),
// one accumulator per translation unit.
sai_status sai_krylov_work_reset();
sai_status sai_krylov_work_read(double* out /* PROF_NSITES x 2 */);
sai_status sai_build_work_reset();
sai_status sai_build_work_read(double* out /* PROF_NSITES x 2 */, double* flops32 /* FP32 flops of the build */);
sai_status sai_batch_work_reset();
sai_status sai_batch_work_read(double* out /* PROF_NSITES x 2 */);
