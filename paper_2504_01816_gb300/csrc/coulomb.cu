// Coulomb operator nu^p = (4 pi)^p (-L_h)^{-p} by the Kronecker-product formalism
// (arXiv 2504.01816, Section "Implementation"; Poisson equation, Eq. 5).
//
// With zero values outside the box, -L_h = K_x (+) K_y (+) K_z (Kronecker sum) where K_a is
// the n_a x n_a matrix of the 1D centred second difference (symmetric Toeplitz, SPD).  With
// K_a = Q_a diag(mu_a) Q_a^T:
//     nu^p f = (Q_z x Q_y x Q_x) diag((4 pi)^p (mu_x + mu_y + mu_z)^{-p}) (Q_z x Q_y x Q_x)^T f
// i.e. three per-axis transforms with Q^T, a pointwise scale, three transforms with Q.
// The 1D eigendecompositions are computed once per context on the host (cyclic Jacobi in
// FP64; n_a is at most a few hundred).
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "internal.cuh"

namespace rpa {

// Symmetric eigendecomposition A = Q diag(w) Q^T (row-major n x n, Q[i*n+a] = component i of
// eigenvector a) by cyclic Jacobi rotations.
void jacobi_eigh(std::vector<double> A, int n, std::vector<double> &w, std::vector<double> &Q) {
    Q.assign((size_t)n * n, 0.0);
    for (int i = 0; i < n; ++i) Q[(size_t)i * n + i] = 1.0;
    for (int sweep = 0; sweep < 100; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) {
                const double a = A[(size_t)i * n + j];
                tot += a * a;
                if (i != j) off += a * a;
            }
        if (off <= 1e-30 * tot) break;
        for (int p = 0; p < n - 1; ++p)
            for (int q = p + 1; q < n; ++q) {
                const double apq = A[(size_t)p * n + q];
                if (apq == 0.0) continue;
                const double app = A[(size_t)p * n + p], aqq = A[(size_t)q * n + q];
                const double theta = (aqq - app) / (2.0 * apq);
                const double t = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
                const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
                for (int k = 0; k < n; ++k) {   // columns p, q
                    const double akp = A[(size_t)k * n + p], akq = A[(size_t)k * n + q];
                    A[(size_t)k * n + p] = c * akp - s * akq;
                    A[(size_t)k * n + q] = s * akp + c * akq;
                }
                for (int k = 0; k < n; ++k) {   // rows p, q
                    const double apk = A[(size_t)p * n + k], aqk = A[(size_t)q * n + k];
                    A[(size_t)p * n + k] = c * apk - s * aqk;
                    A[(size_t)q * n + k] = s * apk + c * aqk;
                }
                for (int k = 0; k < n; ++k) {
                    const double qkp = Q[(size_t)k * n + p], qkq = Q[(size_t)k * n + q];
                    Q[(size_t)k * n + p] = c * qkp - s * qkq;
                    Q[(size_t)k * n + q] = s * qkp + c * qkq;
                }
            }
    }
    w.resize(n);
    for (int i = 0; i < n; ++i) w[i] = A[(size_t)i * n + i];
}

namespace {

// out[o][a][i] = sum_b M[a][b] in[o][b][i]; M = Q^T (forward) or Q (back).  The data are viewed
// as [outer][n][inner].  Each block takes one outer index and 32 consecutive inner indices
// (inner > 1), or 32 consecutive outer indices (inner == 1); lines are staged in shared memory.
__global__ void __launch_bounds__(256) k_axis(const double *__restrict__ in, double *__restrict__ out,
                                              const double *__restrict__ Q, int n, long long inner,
                                              long long outer, int forward, const double *__restrict__ scale,
                                              long long nd) {
    extern __shared__ double sh[];
    double *Ms = sh;                 // n x n, Ms[a*n+b] = M[a][b]
    double *X = sh + (size_t)n * n;  // n x 32, X[b*33 + w]
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int a = e / n, b = e % n;
        Ms[e] = forward ? Q[(size_t)b * n + a] : Q[(size_t)a * n + b];
    }
    long long o0, i0;
    int wcount;
    if (inner > 1) {
        const long long tiles = (inner + 31) / 32;
        o0 = blockIdx.x / tiles;
        i0 = (blockIdx.x % tiles) * 32;
        wcount = (int)min(32LL, inner - i0);
    } else {
        o0 = (long long)blockIdx.x * 32;
        i0 = 0;
        wcount = (int)min(32LL, outer - o0);
    }
    // load
    for (int e = threadIdx.x; e < n * 32; e += blockDim.x) {
        int b, w;
        if (inner > 1) { b = e / 32; w = e % 32; }
        else { w = e / n; b = e % n; }
        double v = 0.0;
        if (w < wcount) {
            const long long addr = inner > 1 ? (o0 * n + b) * inner + i0 + w : (o0 + w) * n + b;
            v = in[addr];
        }
        X[b * 33 + w] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n * 32; e += blockDim.x) {
        int a, w;
        if (inner > 1) { a = e / 32; w = e % 32; }
        else { w = e / n; a = e % n; }
        if (w >= wcount) continue;
        double acc = 0.0;
        for (int b = 0; b < n; ++b) acc += Ms[a * n + b] * X[b * 33 + w];
        const long long addr = inner > 1 ? (o0 * n + a) * inner + i0 + w : (o0 + w) * n + a;
        if (scale) acc *= scale[addr % nd];
        out[addr] = acc;
    }
}

// The same transform for eigenvectors that are symmetric or antisymmetric about the middle of the line, as
// those of a symmetric Toeplitz matrix are: with s_i = x_i + x_{n-1-i} and d_i = x_i - x_{n-1-i} (i < h)
// a symmetric component takes only the s_i and an antisymmetric one only the d_i, and back: half the
// multiply-adds of the n x n product.  The FP64 pipe bounds it (two multiply-adds a clock and SM).  One
// thread takes one symmetric and one antisymmetric sum of a line (two chains), a warp 32 lines, so that
// the matrix is read by broadcast.  40^3, 64 columns, a pass: 341 -> 200 us, the pipe 89% busy.
__global__ void __launch_bounds__(256) k_axis_par(const double *__restrict__ in, double *__restrict__ out,
                                                  const double *__restrict__ Qp, int n, long long inner,
                                                  long long outer, int forward, const double *__restrict__ scale,
                                                  long long nd) {
    extern __shared__ double sh[];
    const int h = (n + 1) / 2;
    double *Ms = sh;                 // h x h, Ms[r * h + c]: result r from term c, symmetric; then antisymmetric
    double *X = Ms + 2 * h * h;      // h x 33 of s (or symmetric components), then of d
    double *Y = X + 2 * h * 33;      // inner == 1: results, n x 33
    int *idx = reinterpret_cast<int *>(Y + (inner == 1 ? n * 33 : 0));   // eigenvectors: symmetric, antisymmetric
    for (int e = threadIdx.x; e < 2 * h * h; e += blockDim.x) {
        const int p = e / (h * h), r = (e - p * h * h) / h, c = e - p * h * h - r * h;
        Ms[e] = Qp[(size_t)p * h * h + (forward ? r * h + c : c * h + r)];
    }
    for (int e = threadIdx.x; e < 2 * h; e += blockDim.x) idx[e] = reinterpret_cast<const int *>(Qp + 2 * h * h)[e];
    long long o0, i0;
    int wcount;
    if (inner > 1) {
        const long long tiles = (inner + 31) / 32;
        o0 = blockIdx.x / tiles;
        i0 = (blockIdx.x % tiles) * 32;
        wcount = (int)min(32LL, inner - i0);
    } else {
        o0 = (long long)blockIdx.x * 32;
        i0 = 0;
        wcount = (int)min(32LL, outer - o0);
    }
    // element b of line w
    auto addr = [&](int b, int w) { return inner > 1 ? (o0 * n + b) * inner + i0 + w : (o0 + w) * n + b; };
    __syncthreads();                 // idx
    for (int e = threadIdx.x; e < h * 32; e += blockDim.x) {
        int i, w;
        if (inner > 1) { i = e / 32; w = e % 32; }
        else { w = e / h; i = e % h; }
        double s = 0.0, d = 0.0;
        if (w < wcount) {
            const int b0 = forward ? i : idx[i], b1 = forward ? n - 1 - i : idx[h + i];   // -1: no such component
            const double v0 = in[addr(b0, w)], v1 = b1 >= 0 ? in[addr(b1, w)] : 0.0;
            s = !forward || b0 == b1 ? v0 : v0 + v1;
            d = !forward ? v1 : b0 == b1 ? 0.0 : v0 - v1;
        }
        X[i * 33 + w] = s;
        X[(h + i) * 33 + w] = d;
    }
    __syncthreads();
    const int w = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < h; r += (int)blockDim.x >> 5) {
        const double *ms = Ms + r * h, *ma = ms + h * h, *xs = X + w, *xd = xs + h * 33;
        double s = 0.0, d = 0.0;
        for (int c = 0; c < h; ++c) {
            s += ms[c] * xs[c * 33];
            d += ma[c] * xd[c * 33];
        }
        if (w >= wcount) continue;
        const int b0 = forward ? idx[r] : r, b1 = forward ? idx[h + r] : n - 1 - r;
        const double v0 = forward ? s : s + d, v1 = forward ? d : s - d;
        if (inner == 1) {
            Y[b0 * 33 + w] = v0;
            if (b1 >= 0 && b1 != b0) Y[b1 * 33 + w] = v1;
            continue;
        }
        const long long a0 = addr(b0, w);
        out[a0] = scale ? v0 * scale[a0 % nd] : v0;
        if (b1 >= 0 && b1 != b0) {
            const long long a1 = addr(b1, w);
            out[a1] = scale ? v1 * scale[a1 % nd] : v1;
        }
    }
    if (inner > 1) return;
    __syncthreads();
    for (int e = threadIdx.x; e < n * wcount; e += blockDim.x) {
        const int l = e / n, b = e - l * n;
        const long long a = addr(b, l);
        out[a] = scale ? Y[b * 33 + l] * scale[a % nd] : Y[b * 33 + l];
    }
}

// The eigenvectors by parity for k_axis_par (empty: one has no parity, as within the degenerate pairs of a
// periodic axis).  The part of the other parity that is dropped is the eigensolver's error: rounding over the gap to
// the next eigenvalue, 1e-13 at n = 40 and 6e-12 at n = 150.  It mixes neighbours, on which nu^p differs by as little as
// their gap, so the operator is not the worse for it (against a long double eigensolver, p = 1/2: 3.46e-14
// with all of Q, 3.42e-14 by parity at n = 40; 7.0e-13 and 5.6e-13 at n = 150), and the vectors stay orthonormal
// (5e-14).
std::vector<double> by_parity(const std::vector<double> &Q, int n) {
    const int h = (n + 1) / 2;
    std::vector<double> F((size_t)2 * h * h + h, 0.0);
    std::vector<int> idx(2 * (size_t)h, -1);
    int cnt[2] = {0, 0};
    for (int a = 0; a < n; ++a) {
        double even = 0.0, odd = 0.0;
        for (int i = 0; i < n; ++i) {
            const double u = Q[(size_t)i * n + a], v = Q[(size_t)(n - 1 - i) * n + a];
            even += 0.25 * (u + v) * (u + v);
            odd += 0.25 * (u - v) * (u - v);
        }
        const int p = even < odd;
        if (std::min(even, odd) > 1e-22 || cnt[p] >= (p ? n - h : h)) return {};
        const int j = cnt[p]++;
        idx[(size_t)p * h + j] = a;
        for (int i = 0; i < h; ++i) {
            const double u = Q[(size_t)i * n + a], v = Q[(size_t)(n - 1 - i) * n + a];
            F[((size_t)p * h + j) * h + i] = 0.5 * (p ? u - v : u + v);
        }
    }
    std::memcpy(F.data() + (size_t)2 * h * h, idx.data(), sizeof(int) * idx.size());
    return F;
}

// Pointwise factor (4 pi / lam)^power of nu^power in the eigenbasis; lam = 0 only for the G = 0
// mode of a periodic grid, which nu^power maps to zero.
__global__ void k_scale_grid(const double *__restrict__ lam, double *__restrict__ sc, long long nd, double power) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nd) sc[i] = lam[i] > 0.0 ? pow(4.0 * 3.14159265358979323846, power) * pow(lam[i], -power) : 0.0;
}

}  // namespace

void coulomb_setup(Ctx &c) {
    const int dims[3] = {c.nx, c.ny, c.nz};
    std::vector<double> mu[3];
    for (int a = 0; a < 3; ++a) {
        const int n = dims[a];
        std::vector<double> K((size_t)n * n, 0.0), Q;
        // K = -D, D the 1D second difference with weights w_k / h^2;  c.coef.a = -w/(2h^2).
        // Dirichlet: taps past the ends are dropped (Toeplitz); periodic: taps wrap, and taps
        // that land on the same point add up (circulant).
        for (int i = 0; i < n; ++i)
            for (int d = -kRadius; d <= kRadius; ++d) {
                int j = i + d;
                if (c.opt.periodic) j = ((j % n) + n) % n;
                else if (j < 0 || j >= n) continue;
                K[(size_t)i * n + j] += 2.0 * c.coef.a[std::abs(d)];
            }
        jacobi_eigh(K, n, mu[a], Q);
        if (c.opt.periodic) {
            // one zero eigenvalue (the constant mode), returned to rounding: made exactly zero so
            // that the G = 0 mode of the 3D operator is the one point where lam = 0
            double top = 0.0;
            for (double m : mu[a]) top = std::max(top, std::fabs(m));
            int zi = 0;
            for (int i = 1; i < n; ++i)
                if (std::fabs(mu[a][i]) < std::fabs(mu[a][zi])) zi = i;
            if (!(std::fabs(mu[a][zi]) <= 1e-10 * top)) fail(RPA_ERR_INVALID, "periodic 1D Laplacian: no zero mode (n=%d)", n);
            mu[a][zi] = 0.0;
            for (int i = 0; i < n; ++i)
                if (i != zi && !(mu[a][i] > 0.0)) fail(RPA_ERR_INVALID, "periodic 1D Laplacian not semidefinite (n=%d)", n);
        } else {
            for (double m : mu[a])
                if (!(m > 0.0)) fail(RPA_ERR_INVALID, "1D Laplacian not positive definite (n=%d)", n);
        }
        const std::vector<double> qp = by_parity(Q, n);
        std::vector<double> both(Q);                     // one allocation and copy
        both.insert(both.end(), qp.begin(), qp.end());
        RPA_CUDA(device_malloc(&c.Q[a], sizeof(double) * both.size()));
        RPA_CUDA(cudaMemcpy(c.Q[a], both.data(), sizeof(double) * both.size(), cudaMemcpyHostToDevice));
        if (!qp.empty()) c.Qpar[a] = c.Q[a] + (size_t)n * n;
        // the same factors for the Laplacian preconditioner of COCG, in FP64 and FP32
        std::vector<float> qf(Q.begin(), Q.end()), mf(mu[a].begin(), mu[a].end());
        RPA_CUDA(device_malloc(&c.mu[a], sizeof(double) * n));
        RPA_CUDA(cudaMemcpy(c.mu[a], mu[a].data(), sizeof(double) * n, cudaMemcpyHostToDevice));
        RPA_CUDA(device_malloc(&c.Qf[a], sizeof(float) * n * n));
        RPA_CUDA(cudaMemcpy(c.Qf[a], qf.data(), sizeof(float) * n * n, cudaMemcpyHostToDevice));
        RPA_CUDA(device_malloc(&c.muf[a], sizeof(float) * n));
        RPA_CUDA(cudaMemcpy(c.muf[a], mf.data(), sizeof(float) * n, cudaMemcpyHostToDevice));
    }
    std::vector<double> lam((size_t)c.nd);
    for (int k = 0; k < c.nz; ++k)
        for (int j = 0; j < c.ny; ++j)
            for (int i = 0; i < c.nx; ++i)
                lam[(size_t)i + (size_t)c.nx * (j + (size_t)c.ny * k)] = mu[0][i] + mu[1][j] + mu[2][k];
    RPA_CUDA(device_malloc(&c.lam, sizeof(double) * c.nd));
    RPA_CUDA(cudaMemcpy(c.lam, lam.data(), sizeof(double) * c.nd, cudaMemcpyHostToDevice));
}

static void axis_pass(Ctx &c, int axis, const double *in, double *out, int ncols, int forward, const double *scale,
                      cudaStream_t s) {
    const int n = axis == 0 ? c.nx : axis == 1 ? c.ny : c.nz;
    const long long inner = axis == 0 ? 1 : axis == 1 ? c.nx : (long long)c.nx * c.ny;
    const long long outer = (long long)ncols * c.nd / ((long long)n * inner);
    const size_t sh = sizeof(double) * ((size_t)n * n + (size_t)n * 33);
    allow_dynamic_smem((const void *)k_axis, sh);   // rejects grid dimensions above ~150
    const long long blocks = inner > 1 ? outer * ((inner + 31) / 32) : (outer + 31) / 32;
    if (c.Qpar[axis]) {
        const int h = (n + 1) / 2;
        const size_t shp = sizeof(double) * ((size_t)2 * h * h + (size_t)2 * h * 33 + (inner == 1 ? (size_t)n * 33 : 0) + h);
        allow_dynamic_smem((const void *)k_axis_par, shp);
        k_axis_par<<<(unsigned)blocks, 256, shp, s>>>(in, out, c.Qpar[axis], n, inner, outer, forward, scale, c.nd);
        RPA_LAUNCH("coulomb axis transform by parity");
        return;
    }
    k_axis<<<(unsigned)blocks, 256, sh, s>>>(in, out, c.Q[axis], n, inner, outer, forward, scale, c.nd);
    RPA_LAUNCH("coulomb axis transform");
}

// Fixed scratch for rpa_coulomb_apply_noalloc.  Every device that loads the library holds
// RPA_STATIC_SCRATCH_BYTES of it until the process exits.  In host code the symbol is only a
// stand-in: the device address is looked up once per device with cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_scratch[RPA_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void *g_scratch_addr[kMaxDevices] = {};

// Device address of g_static_scratch on the current device (looked up on first use).
void *static_scratch(int dev) {
    if (dev < 0 || dev >= kMaxDevices) fail(RPA_ERR_INVALID, "device ordinal %d not supported", dev);
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_addr[dev]) {
        void *ptr = nullptr;
        RPA_CUDA(cudaGetSymbolAddress(&ptr, g_static_scratch));
        g_scratch_addr[dev] = ptr;
    }
    return g_scratch_addr[dev];
}
}  // namespace

// The same per-axis transform on the tensor cores: the grid's lines along the axis are the rows of one
// contraction with M = Q^T (forward) or Q (back), Q[i*n+a] row-major, so its 128-row tiles are full
// whatever the axis.
static void axis_pass_tc(Ctx &c, int axis, const double *in, double *out, int ncols, int forward,
                         const double *scale, cudaStream_t s) {
    const int n = axis == 0 ? c.nx : axis == 1 ? c.ny : c.nz;
    const double *Q = c.Q[axis];
    // M(a, b) = Q[b][a] (forward) or Q[a][b] (back): element strides of (a, b)
    const long long ma = forward ? 1 : n, mb = forward ? n : 1;
    const long long lines = (long long)ncols * c.nd / n, plane = (long long)c.nx * c.ny;
    if (plane > (long long)INT32_MAX) fail(RPA_ERR_INVALID, "plane too large for the tensor-core transform");
    // x: the line of row o starts at o n_x (taken n_y n_z lines, a column, at a time); y: line (slab, i) at
    // slab n_x n_y + i; z: line (column, i) at column N_d + i
    if (axis == 0) tc_lines(in, out, lines, c.ny * c.nz, c.nd, n, 1, n, Q, ma, mb, scale, s, c.d_tc_err);
    else if (axis == 1) tc_lines(in, out, lines, c.nx, plane, 1, c.nx, n, Q, ma, mb, scale, s, c.d_tc_err);
    else tc_lines(in, out, lines, (int)plane, c.nd, 1, plane, n, Q, ma, mb, scale, s, c.d_tc_err);
}

static void coulomb_passes_tc(Ctx &c, double power, const double *in, double *out, int ncols, double *t1, double *t2,
                              double *sc, cudaStream_t s) {
    k_scale_grid<<<(unsigned)((c.nd + 255) / 256), 256, 0, s>>>(c.lam, sc, c.nd, power);
    RPA_LAUNCH("coulomb scale");
    count_launches(1);
    axis_pass_tc(c, 0, in, t1, ncols, 1, nullptr, s);
    axis_pass_tc(c, 1, t1, t2, ncols, 1, nullptr, s);
    axis_pass_tc(c, 2, t2, t1, ncols, 1, sc, s);
    axis_pass_tc(c, 2, t1, t2, ncols, 0, nullptr, s);
    axis_pass_tc(c, 1, t2, t1, ncols, 0, nullptr, s);
    axis_pass_tc(c, 0, t1, out, ncols, 0, nullptr, s);
}

static void coulomb_passes(Ctx &c, double power, const double *in, double *out, int ncols, double *t1, double *t2,
                           double *sc, cudaStream_t s) {
    k_scale_grid<<<(unsigned)((c.nd + 255) / 256), 256, 0, s>>>(c.lam, sc, c.nd, power);
    RPA_LAUNCH("coulomb scale");
    count_launches(7);   // scale + six axis passes
    axis_pass(c, 0, in, t1, ncols, 1, nullptr, s);
    axis_pass(c, 1, t1, t2, ncols, 1, nullptr, s);
    axis_pass(c, 2, t2, t1, ncols, 1, sc, s);
    axis_pass(c, 2, t1, t2, ncols, 0, nullptr, s);
    axis_pass(c, 1, t2, t1, ncols, 0, nullptr, s);
    axis_pass(c, 0, t1, out, ncols, 0, nullptr, s);
}

void coulomb_apply_noalloc(Ctx &c, double power, const double *in, double *out, int ncols, cudaStream_t s) {
    if (ncols <= 0) return;
    const size_t blk = (sizeof(double) * (size_t)ncols * c.nd + 255) / 256 * 256;
    const size_t need = 2 * blk + sizeof(double) * (size_t)c.nd;
    if (need > (size_t)RPA_STATIC_SCRATCH_BYTES)
        fail(RPA_ERR_INVALID, "rpa_coulomb_apply_noalloc: %d columns of %lld points need %zu bytes of scratch, "
                              "more than the fixed %zu", ncols, c.nd, need, (size_t)RPA_STATIC_SCRATCH_BYTES);
    int dev = 0;
    RPA_CUDA(cudaGetDevice(&dev));
    if (dev != c.device) fail(RPA_ERR_INVALID, "the current device is not the context's device");
    char *base = (char *)static_scratch(dev);
    double *t1 = (double *)base, *t2 = (double *)(base + blk), *sc = (double *)(base + 2 * blk);
    // every scratch word is written before it is read: nothing needs clearing
    coulomb_passes(c, power, in, out, ncols, t1, t2, sc, s);
}

void coulomb_apply(Ctx &c, double power, const double *in, double *out, int ncols, cudaStream_t s, bool tensor) {
    if (ncols <= 0) return;
    const size_t blk = sizeof(double) * (size_t)ncols * c.nd;
    char *base = (char *)c.coul_tmp.ensure(2 * blk + sizeof(double) * c.nd);
    double *t1 = (double *)base, *t2 = (double *)(base + blk), *sc = (double *)(base + 2 * blk);
    if (tensor)
        coulomb_passes_tc(c, power, in, out, ncols, t1, t2, sc, s);
    else
        coulomb_passes(c, power, in, out, ncols, t1, t2, sc, s);
}

}  // namespace rpa
