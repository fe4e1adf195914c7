// Internal declarations shared by the translation units of librpa.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "rpa.h"

namespace rpa {

constexpr int kRadius = 6;              // 12th-order centred differences
constexpr int kMaxOmega = 64;
constexpr int kMaxSqOrder = 32;     // largest Gauss spectral quadrature order
constexpr int kMaxBlock = 16;       // largest block of block COCG

// ------------------------------------------------------------------------------------------
// Errors: every internal failure throws rpa::Error; the C entry points catch it and turn it
// into a status code plus a thread-local message.
// ------------------------------------------------------------------------------------------
struct Error {
    rpa_status status;
    std::string msg;
};

[[noreturn]] void fail(rpa_status st, const char *fmt, ...);

// Raise a kernel's dynamic shared-memory limit to the device maximum (once; the value never
// depends on the call, so contexts on different threads cannot lower each other's limit between
// setting it and launching) and fail with RPA_ERR_INVALID if `need` bytes exceed that maximum.
void allow_dynamic_smem(const void *kernel, size_t need);

// Kernel launches issued by the library on this thread (reported in rpa_stats.launches).
extern thread_local long long g_launches;
inline void count_launches(long long n) { g_launches += n; }
void check_cuda(cudaError_t e, const char *what, const char *file, int line);
#define RPA_CUDA(call) ::rpa::check_cuda((call), #call, __FILE__, __LINE__)
#define RPA_LAUNCH(what) ::rpa::check_cuda(cudaGetLastError(), what, __FILE__, __LINE__)

// cudaMalloc, again after the Lanczos workspaces that no running queue uses are given back (all contexts').
cudaError_t device_malloc(void **p, size_t bytes);
template <typename T> cudaError_t device_malloc(T **p, size_t bytes) { return device_malloc((void **)p, bytes); }

// ------------------------------------------------------------------------------------------
// Device buffer that only grows.
// ------------------------------------------------------------------------------------------
struct DevBuf {
    void *ptr = nullptr;
    size_t bytes = 0;
    void *ensure(size_t need);
    bool room(size_t need);       // the same, for a buffer that one can do without: false where memory is short
    void release();
    template <typename T> T *as() const { return static_cast<T *>(ptr); }
};

// Shifted Hamiltonian stencil: (H + sigma) v = (diag + V + sigma) v + sum_k a_k (six neighbours
// at distance k), with a_k = -w_k / (2 h^2) and diag = 3 a_0.
struct StencilCoef {
    double a[kRadius + 1];
};

// Per-system COCG scalars (one slot of a batch).
struct SysState {
    double rho_re, rho_im;        // r^T r (unconjugated)
    double alpha_re, alpha_im;
    double beta_re, beta_im;
    double ref_norm;              // ||b|| (outer) for the FP64 form; ||r64|| for a mixed inner solve
    double bnorm;                 // ||b||
    double rnorm;                 // latest ||r||
    double shift_re, shift_im;    // sigma = -eps_n + i omega
    int n, j;                     // orbital, column
    int active;                   // inner COCG running
    int outer_active;             // mixed: refinement running
    int iters;                    // inner iterations in the current solve
    int total_iters;              // all inner iterations
    int refines;                  // FP64 residual evaluations
    int status;
};

// Summary of the Sternheimer queues run since the last read-back, accumulated on the device (so
// that a queue needs no host synchronisation) and added to rpa_stats at the next one.
struct QueueStats {
    long long solves, iters, refines, nearb, launches;
    int worst;          // largest per-system status
    int unfinished;     // a queue stopped at its epoch bound with systems left
};

// How a queue's systems are spread over the SMs by the Lanczos kernel (lanczos.cu): a cluster of
// ncl blocks per system, `clusters` of them resident, each thread with W x 2 x zc points (W = 16 bytes).
struct LanczosPlan {
    int variant, mixed, zc, ncl, clusters, threads;
    int hw, hh, nch;               // units per row, row pairs, z chunks of a block
    int pitch, plane, lead;        // elements of a slab row and plane, and before the first plane
    int reach, hist;
    int stream, bh, depth, unit_rows;   // the streaming kernel: rows of a band, planes in flight, rows a thread
    size_t smem, ws_stride, ws_bytes;
    void *ws;                      // ws_bytes of workspace, set by the caller
};

struct BatchCoord;   // rendezvous of rpa_ec_batch's threads (api.cu)

// ------------------------------------------------------------------------------------------
// Context
// ------------------------------------------------------------------------------------------
struct Ctx {
    int nx = 0, ny = 0, nz = 0, ns = 0;
    long long nd = 0;
    double h = 0;
    rpa_options opt{};
    StencilCoef coef{};
    int device = 0;

    // inputs (device copies)
    double *vloc64 = nullptr;
    float *vloc32 = nullptr;
    float *vloc_lo = nullptr;     // V_loc - vloc32 in FP32: V_loc as an FP32 pair
    double *psi64 = nullptr;      // ns x nd (row s = orbital s)
    float *psi32 = nullptr;       // FP32 copy (projection of the mixed form's FP32 residuals)
    std::vector<double> eps;
    double *eps_dev = nullptr;

    // Kronecker Coulomb operator: 1D eigenvectors Q_a (n_a x n_a, row-major Q[i*n+a]) and the
    // summed eigenvalue grid lam = mu_x + mu_y + mu_z (nd).
    double *Q[3] = {nullptr, nullptr, nullptr};
    double *lam = nullptr;
    // The same eigenvectors by parity, in the same allocation (null: not every one has a parity), h = ceil(n_a / 2): h x h components
    // i < h of the symmetric ones and of the antisymmetric ones, then their indices a (two lists of h ints).
    double *Qpar[3] = {nullptr, nullptr, nullptr};
    // Laplacian preconditioner of COCG: the 1D eigenvalues mu_a (FP64), FP32 copies of Q_a and mu_a,
    // and the mean of V_loc
    double *mu[3] = {nullptr, nullptr, nullptr};
    float *Qf[3] = {nullptr, nullptr, nullptr};
    float *muf[3] = {nullptr, nullptr, nullptr};
    double vbar = 0.0;

    // workspaces
    DevBuf cocg_state;            // complex vectors of the systems in flight
    DevBuf cocg_partials;
    DevBuf sys_state;             // SysState[slots]
    DevBuf rhs;                   // real right-hand sides of the systems in flight
    DevBuf pc_coef;               // P_c coefficients
    DevBuf coul_tmp;              // Kronecker scratch
    DevBuf blockA, blockB, blockC, blockD;   // N_d x N_r blocks for rpa_ec / apply
    DevBuf small;                 // N_r x N_r matrices and scalars
    DevBuf slot_idx;              // (n, j) of the slots
    DevBuf proj_buf;              // occupied-space projection of finished solutions
    DevBuf coef_buf;              // per-column coefficients of the gradient pass
    DevBuf blockE;                // subspace of the previous iteration (gradient)
    DevBuf dense_scratch;         // split-K partial sums
    // Lanczos vectors of the systems in flight.  One can do without them (the COCG kernels run): any
    // allocation of the library that fails takes them back from the contexts whose queue does not hold them
    // (lz_held; lz_done: the last that did has run on the device), see LanczosHold.
    DevBuf lanczos_ws;
    bool lz_held = false;
    cudaEvent_t lz_done = nullptr;
    LanczosPlan lz_plan{};        // the last queue's plan, for lz_key = {slots, form, batch_load}
    int lz_key[3] = {-1, -1, -1};
    bool lz_ok = false;
    // Set while rpa_ec_gradient iterates its subspace: the COCG kernels.  A subspace is R L^-T with the conditioning of R,
    // and after the exact integer pieces of the tensor-core contractions (whose last digits turn on
    // 1e-12 of their operands) the Lanczos kernel's rounding moves it by 2e-9 relative, more than a change
    // of kernels may; the energies and the gradient move by 1e-10.  It is one rule for every call, so that
    // they do not depend on whether the subspace is an output.
    bool keep_cocg = false;
    SysState *h_state = nullptr;  // pinned host mirror of the slot states
    size_t h_state_cap = 0;
    int *h_count = nullptr;       // pinned host counter
    int *d_tc_err = nullptr;      // set by a kernel that gave up waiting: 1 a tensor-core contraction, 2 Lanczos
    QueueStats *d_qstats = nullptr;   // device accumulator of queue statistics
    int *d_loop = nullptr;            // epoch counter of a device-driven queue
    char *h_rb = nullptr;             // pinned read-back block (Ritz values, scalars, statistics)
    long long host_syncs = 0;         // host synchronisations of the current call
    // events of the last chi0 application (Coulomb / COCG phase times, read at the next sync)
    cudaEvent_t ev_apply[4] = {nullptr, nullptr, nullptr, nullptr};
    bool apply_timed = false;

    // per-call statistics
    rpa_stats stats{};
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    // profiling (rpa_options.profile): event pool and per-kernel point counters on the device
    std::vector<cudaEvent_t> ev_pool;
    unsigned long long *d_prof_points = nullptr;   // RPA_PROF_SLOTS counters
    // rpa_ec_batch: the rendezvous this context's chi0 applications go to (nullptr otherwise)
    BatchCoord *coord = nullptr;
    // a batch without block COCG: this context's stream, and the systems of the whole batch
    cudaStream_t batch_stream = nullptr;
    int batch_load = 0;
    // CUDA graphs: epochs of COCG iterations are captured on a private stream and replayed
    bool use_graphs = true;
    cudaStream_t cap_stream = nullptr;

    ~Ctx();
};

// ------------------------------------------------------------------------------------------
// Operations (each enqueues work on `stream`)
// ------------------------------------------------------------------------------------------
// Kronecker Coulomb operator nu^power on ncols columns.
void coulomb_apply(Ctx &c, double power, const double *in, double *out, int ncols, cudaStream_t s,
                   bool tensor = false);
// Whether the dense contractions of this context run on the tensor cores (rpa_options.contractions):
// the P_c coefficients and C = V^T R, and the Kronecker transforms of nu^1/2.
inline bool use_tensor_cores(const Ctx &c) {
    return c.opt.contractions >= 2 || (c.opt.contractions == 0 && c.opt.prec == RPA_MIXED);
}
// A queue's hold on its context's Lanczos workspace, from its request (after every other buffer that the queue
// needs) to the end of the work that the queue has put on its stream.
struct LanczosHold {
    Ctx &c;
    cudaStream_t s;
    bool held = false;
    LanczosHold(Ctx &ctx, cudaStream_t st) : c(ctx), s(st) {}
    LanczosHold(const LanczosHold &) = delete;
    bool take(size_t bytes);      // false where memory is short
    ~LanczosHold();
};

inline bool use_tensor_cores_kronecker(const Ctx &c) {
    return c.opt.contractions == 2 || (c.opt.contractions == 0 && c.opt.prec == RPA_MIXED);
}
// Fails with RPA_ERR_CUDA if a kernel reported a timed-out wait (synchronises s).
void check_tensor_core_status(Ctx &c, cudaStream_t s);
void coulomb_setup(Ctx &c);
// Same operator with its scratch in the library's fixed device array (no allocation).
void coulomb_apply_noalloc(Ctx &c, double power, const double *in, double *out, int ncols, cudaStream_t s);

// Synchronise s and count it in the call's statistics.
void sync_stream(Ctx &c, cudaStream_t s);
// After a synchronisation: add the device queue statistics read back into h (pinned) to the
// call's statistics and return the worst per-system status seen.
int add_queue_stats(Ctx &c, const QueueStats &h);

// Sternheimer solves for the systems given by (n, j) pairs with real right-hand sides b
// (nsys x nd, row per system) -> complex solutions x (nsys x nd interleaved, FP64).
// Returns the worst per-system status; fills per-system iterations/status (host vectors).
int sternheimer_batch(Ctx &c, double omega, const int *orb, int nsys, const double *b, double *x,
                      std::vector<int> *iters, std::vector<int> *status, cudaStream_t s);

// chi0 on ncols real columns: drho = (4/h^3) Re sum_n u_n x_n with the projected right-hand
// sides -P_c(u_n dV_j).  Returns the worst status.
int chi0_apply(Ctx &c, double omega, const double *dv, double *drho, int ncols, cudaStream_t s);

// grad += sum_j coef[j] (4/h^3) Re sum_n (P_c x_{n,j})^2 for the projected Sternheimer solutions of
// dV_j (ncols rows of dv); coef: ncols doubles on the device.  Returns the worst status known on
// the host (a device-driven queue reports through the device statistics).
int response_square(Ctx &c, double omega, const double *dv, const double *coef, double *grad, int ncols,
                    cudaStream_t s);

// Host symmetric eigendecomposition (cyclic Jacobi): A = Q diag(w) Q^T, Q[i*n+a] = component i of
// eigenvector a; w ascending is not guaranteed.  (The 1D matrices of the Coulomb operator.)
void jacobi_eigh(std::vector<double> A, int n, std::vector<double> &w, std::vector<double> &Q);
// The same on the device (parallel cyclic Jacobi, one block; A destroyed); work: 3 (n + 1) doubles.
void jacobi_eigh_device(double *A, int n, double *Q, double *w, double *work, cudaStream_t s);
// S = Q^T and coef[i] = weight * g'(w_i), g'(x) = -x / (1 - x) (the adjoint's Ritz rotation, device).
void ritz_rotation(const double *Q, const double *w, int n, double weight, double *S, double *coef, cudaStream_t s);

// Whether the fused single-pass COCG kernel applies to this context's grid (a whole xy plane fits
// its shared-memory ring); the mixed form then uses it by default.
bool fused_kernel_applies(const Ctx &c, bool warp_specialised = false, bool cluster = false);

// Block COCG (block_cocg.cu) for systems grouped by orbital: chi0 on ncols columns (as chi0_apply)
// and the Sternheimer solves of rpa_sternheimer_solve (as sternheimer_batch; Tc: P_c coefficients
// of the rows of b, or nullptr).
int chi0_apply_block(Ctx &c, double omega, const double *dv, double *drho, int ncols, cudaStream_t s);
int sternheimer_block(Ctx &c, double omega, const int *orb, int nsys, const double *b, const double *Tc,
                      double *x, std::vector<int> *iters, std::vector<int> *status, cudaStream_t s);
// One context's chi0 application within a batch.
struct Chi0Request {
    Ctx *c;
    double omega;
    const double *dv;
    double *drho;
    int ncols;
};
// chi0 for several contexts (distinct, on one device, with equal precision and COCG settings) in
// one set of launches: the block COCG kernels over all their groups at once, with block size
// max(1, block_cocg) and the iteration settings and workspaces of the first context.  The
// statistics of each context get its own systems.
int chi0_apply_batch(const std::vector<Chi0Request> &reqs, cudaStream_t s, std::vector<int> *status = nullptr);
// While a context with block_cocg > 0 is attached to a BatchCoord, its chi0 applications are posted there
// and run together with the other contexts' (batch_chi0).
int batch_chi0(Ctx &c, double omega, const double *dv, double *drho, int ncols, cudaStream_t s);

// Same as sternheimer_batch, with b replaced by P_c b first.
int sternheimer_batch_projected(Ctx &c, double omega, const int *orb, int nsys, const double *b, double *x,
                                std::vector<int> *iters, std::vector<int> *status, cudaStream_t s);

// Dense FP64 helpers (dense.cu)
// G (na x nb, row-major) = A B^T with A: na rows of length len, B: nb rows of length len.
void gram(const double *A, int na, const double *B, int nb, long long len, double *G, cudaStream_t s,
          DevBuf &scratch);
// T[(n, j)][k] = sum_r u_k[r] u_n[r] dv_j[r], row n ncols + j of ns values.
void gram_pairs(const double *psi, int ns, const double *dv, int ncols, long long len, double *T, cudaStream_t s,
                DevBuf &scratch);
// Y (nc rows) = S X, S: nc x nk row-major (device), X: nk rows of length len.
void combine_rows(const double *S, int nc, int nk, const double *X, long long len, double *Y,
                  cudaStream_t s);
// Cholesky of the n x n SPD matrix M (row-major, device) in place -> lower L; returns via
// *dev_info (0 ok, k+1 = failed pivot k).
void cholesky(double *M, int n, int *dev_info, cudaStream_t s);
// Linv = L^{-1} (lower), n x n row-major.
void tri_inverse(const double *L, int n, double *Linv, cudaStream_t s);
// Ascending eigenvalues of the symmetric n x n matrix C (row-major, destroyed), then
// e_out = weight * sum_i [log1p(-lam_i) + lam_i].
// e_out = weight * Tr g(C) by Gauss spectral quadrature of order n_o (part: n doubles of scratch)
void sq_trace(const double *C, int n, int n_o, double *part, double weight, double *e_out, cudaStream_t s);
void sym_eigvals(double *C, int n, double *lam, double *work, double weight, double *e_out,
                 cudaStream_t s);
void symmetrize(double *C, int n, cudaStream_t s);

// Contractions on the tensor cores (tcgen05, exact integer pieces; tc_gemm.cu).  *err_dev is set to 1 if
// the kernel gave up waiting on its MMAs.
// D (M x N, row-major) = sum_k A[m a_m + k] B[n b_n + k].
void tc_gemm(const double *A, long long a_m, const double *B, long long b_n, int M, int N, long long K, double *D,
             cudaStream_t s, DevBuf &scratch, int *err_dev);
// The same for the products of rows: D[(i nv + j) N + n] = sum_k U[i K + k] V[j K + k] B[n K + k], i < nu, j < nv.
void tc_gemm_pairs(const double *U, int nu, const double *V, int nv, const double *B, int N, long long K, double *D,
                   cudaStream_t s, DevBuf &scratch, int *err_dev);
// Transform of lines of n values: line r starts at in + (r / mi) mo + (r % mi) ms, its values ks apart;
// out (same places) = sum_k Q(a, k) in(k), Q(a, k) = Q[a q_n + k q_k]; optionally times scale[(r % mi) ms + a ks].
void tc_lines(const double *in, double *out, long long rows, int mi, long long mo, long long ms, long long ks, int n,
              const double *Q, long long q_n, long long q_k, const double *scale, cudaStream_t s, int *err_dev);

// Profiling helpers: register a kernel name in the stats table (returns its slot) and add
// launches/time/points/bytes to it.
int prof_slot(Ctx &c, const char *name);

}  // namespace rpa

struct rpa_ctx {
    rpa::Ctx impl;
};
