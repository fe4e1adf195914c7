// Sternheimer inner solves by real Lanczos recurrences, a whole system on chip (arXiv 2504.01816:
// Sternheimer equation, Eq. 9; COCG, Section "Implementation").
//
// COCG for (B + i w) x = b with B = H - eps_n real symmetric and a real b builds its iterates in the
// real Krylov space of B and b: its residuals are complex multiples of the real Lanczos vectors v_k
// of B.  This kernel runs the Lanczos recurrence itself,
//     u = B v_k - c_k v_{k-1},  a_k = u.v_k / v_k.v_k,  v_{k+1} = (u - a_k v_k) / g_{k+1},  c_k = g_k,
// and takes the COCG iterate from the LU factors of the tridiagonal T + i w (d_k = a_k + i w -
// g_k c_k / d_{k-1}, z_k = -g_k z_{k-1} / d_{k-1}, ||r_k|| = g_{k+1} |z_k / d_k|): the same iterates as
// COCG for half the stencil arithmetic and half the state.  |d_k| >= |w|, so for w != 0 the factors
// cannot break down.  A complex right-hand side r (the residual of a refinement) is turned to
// e^{-i phi} r = r_a + i r_b with r_a.r_b = 0 and ||r_a|| largest, and its two real parts are solved one
// after the other; after a first inner solve r_b is the rounding noise of that solve (1e-3..1e-2 of
// r_a) and takes a third of r_a's steps.
//
// A thread-block cluster of C blocks owns one system at a time.  Block c keeps the planes
// [c nz / C, (c + 1) nz / C) of v_k with six halo planes on either side in shared memory; v_{k-1}, u and
// v_{k+1} share one register array (each thread owns W x 2 x ZC points: W = 16 bytes of x, two rows, ZC
// planes), so an iteration reads nothing from memory but V_loc (from L2) and writes only v_k, by a bulk
// copy from shared memory, kept for the solution x = sum_k y_k v_k.  That sum is formed by two extra warps
// while the others are at the next solve, from a history of two buffers; warps that come to the end of that
// solve before take part in what is left of it (or, when the history is full, all form it at once, with
// the COCG direction p handed over).  Between blocks an iteration has two dependences and no cluster
// barrier: the halo planes arrive by bulk copies through distributed shared memory that count on the
// receiver's mbarrier, and overlap the x and y neighbours' part of the stencil; the three dot products are
// sent to every block with st.async, which also tells a block that its neighbours' halos may be
// overwritten.  Every block of a cluster computes the same scalars from the same sums in the same order,
// so all take the same decisions.  The factors, the stopping test and the slot's state belong to an extra
// warp that works while the others compute the next stencil; a solve therefore ends one stencil late.
// In the mixed form the dot products, a_k, g_k and the right-hand side's norms are FP32 throughout (the COCG
// kernels add the threads' sums in FP64): what that costs in a solve its FP64 refinement makes good.  The
// factors are FP64.
//
// What bounds it: shared-memory loads.  A unit of W x 2 points and ZC planes takes 2 (ZC + 12) 16-byte
// loads for the z neighbours of all its planes (held against the ZC accumulators in turn), and per
// plane 12 for the y and 2 XL for the x neighbours: 58 bytes a point for ZC = 5 in FP32 against 240 for
// a plane-by-plane march on complex values; the FP64 form is bound by the FP64 pipe (46 operations a
// point).  Measured (GB300, tol 1e-11, whole chi0 application, against the fused and split COCG kernels):
// 40^3, 1024 systems 212 -> 98 ms; 24^3, 4 systems 9.9 -> 1.9 ms; 37 x 43 x 29, 77 systems 25 -> 6.8 ms;
// FP64 15^3, 32 systems 15.9 -> 2.6 ms, 32^3, 128 systems 197 -> 78 ms.  At 40^3 (four blocks a system) an
// iteration takes 20 thousand cycles: x and y neighbours 9.4 (5.7 of shared-memory loads and 2.5 of
// copies), z neighbours 2.8, sums 2.3, update 2.2, halo 0.3, and per iteration of a solve 1.4 of waiting for
// the solution before it and 2.0 for the start.  With the solution formed at the end of each solve, by all
// warps: 22.4 thousand, 3.8 of them for it (and 9.6 of 26 where a system lies on two blocks).  One form with
// 64-bit index arithmetic per halo store took 230 ms, one with cluster barriers 138 ms, one with the
// solution's code inlined (spills) 158 ms, one that stored the history from registers 102 ms against 98.
#include <algorithm>
#include <cmath>

#include "lanczos.cuh"

namespace rpa {

namespace {

constexpr int kHistMax = 128;            // Lanczos vectors kept between two updates of x

// FP64 form: where g^2 = u.u - (u.v)^2 / v.v comes out below this share of u.u (half its digits are gone: v is
// nearly in an invariant subspace, as a right-hand side next to an eigenvector is), g is taken from the
// sums of u - a' v itself.  Without it g is rounding noise and, where that is negative, the solve ends
// with a residual of 1e-9 that it takes for 0.  The mixed form need not: its refinement forms the residual.
constexpr double kNearSpace = 0x1p-26;

constexpr int kFlushThreads = 64;        // two warps that form the solutions
constexpr int kExtra = 32 + kFlushThreads;   // threads without points: the scalar warp, the flush warps

// W values of one row: 16 bytes.
template <typename T> struct Pk;
template <> struct Pk<float> {
    static constexpr int W = 4;
    float2 p[2];
    __device__ __forceinline__ float get(int i) const { return i & 1 ? p[i >> 1].y : p[i >> 1].x; }
    __device__ __forceinline__ void set(int i, float v) { (i & 1 ? p[i >> 1].y : p[i >> 1].x) = v; }
    __device__ __forceinline__ void fma(float c, const Pk &v) {
        const float2 cc = make_float2(c, c);
        p[0] = __ffma2_rn(cc, v.p[0], p[0]);
        p[1] = __ffma2_rn(cc, v.p[1], p[1]);
    }
    __device__ __forceinline__ void fma(const Pk &c, const Pk &v) {
        p[0] = __ffma2_rn(c.p[0], v.p[0], p[0]);
        p[1] = __ffma2_rn(c.p[1], v.p[1], p[1]);
    }
    __device__ __forceinline__ void mul(float c) {
        const float2 cc = make_float2(c, c);
        p[0] = __fmul2_rn(cc, p[0]);
        p[1] = __fmul2_rn(cc, p[1]);
    }
    __device__ __forceinline__ void mul(const Pk &c) {
        p[0] = __fmul2_rn(c.p[0], p[0]);
        p[1] = __fmul2_rn(c.p[1], p[1]);
    }
    __device__ __forceinline__ float sum() const { return (p[0].x + p[0].y) + (p[1].x + p[1].y); }
    __device__ __forceinline__ void zero() { p[0] = p[1] = make_float2(0.f, 0.f); }
};
template <> struct Pk<double> {
    static constexpr int W = 2;
    double2 p;
    __device__ __forceinline__ double get(int i) const { return i ? p.y : p.x; }
    __device__ __forceinline__ void set(int i, double v) { (i ? p.y : p.x) = v; }
    __device__ __forceinline__ void fma(double c, const Pk &v) {
        p.x = ::fma(c, v.p.x, p.x);
        p.y = ::fma(c, v.p.y, p.y);
    }
    __device__ __forceinline__ void fma(const Pk &c, const Pk &v) {
        p.x = ::fma(c.p.x, v.p.x, p.x);
        p.y = ::fma(c.p.y, v.p.y, p.y);
    }
    __device__ __forceinline__ void mul(double c) {
        p.x *= c;
        p.y *= c;
    }
    __device__ __forceinline__ void mul(const Pk &c) {
        p.x *= c.p.x;
        p.y *= c.p.y;
    }
    __device__ __forceinline__ double sum() const { return p.x + p.y; }
    __device__ __forceinline__ void zero() { p = make_double2(0.0, 0.0); }
};
__device__ __forceinline__ Pk<float> pk_load(const float *a) {
    const float4 t = *reinterpret_cast<const float4 *>(a);
    Pk<float> r;
    r.p[0] = make_float2(t.x, t.y);
    r.p[1] = make_float2(t.z, t.w);
    return r;
}
__device__ __forceinline__ Pk<double> pk_load(const double *a) {
    Pk<double> r;
    r.p = *reinterpret_cast<const double2 *>(a);
    return r;
}
// The same from a byte offset in the block's shared memory (a thread's offset plus ones that are the same for
// all threads, which stay in the uniform registers of the load's address).
template <typename T> __device__ __forceinline__ Pk<T> lds(int off);
// The same from the history, past L1: the bulk stores that write it do not update L1's lines.
__device__ __forceinline__ Pk<float> pk_load_l2(const float *a) {
    const float4 t = __ldcg(reinterpret_cast<const float4 *>(a));
    Pk<float> r;
    r.p[0] = make_float2(t.x, t.y);
    r.p[1] = make_float2(t.z, t.w);
    return r;
}
__device__ __forceinline__ Pk<double> pk_load_l2(const double *a) {
    Pk<double> r;
    r.p = __ldcg(reinterpret_cast<const double2 *>(a));
    return r;
}
__device__ __forceinline__ void pk_store(float *a, const Pk<float> &v) {
    *reinterpret_cast<float4 *>(a) = make_float4(v.p[0].x, v.p[0].y, v.p[1].x, v.p[1].y);
}
__device__ __forceinline__ void pk_store(double *a, const Pk<double> &v) { *reinterpret_cast<double2 *>(a) = v.p; }
__device__ __forceinline__ unsigned map_rank(unsigned addr, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();                        // the aligned forms need the warp together
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_init(unsigned long long *b) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(b)) : "memory");
}
// Wait for a phase of an mbarrier; false after `limit` cycles (~1 s; the flush warps' wait for a whole solve longer).
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, long long limit = 2000000000LL) {
    const long long t0 = clock64();
    for (;;) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > limit) return false;
    }
}

// acc += sum_d cf[d] (x - d and x + d neighbours) for W values; X holds the row from x - PAD on.
__device__ __forceinline__ void x_part(Pk<float> &acc, const Pk<float> (&X)[5], const Coef<float> &cf) {
    auto at = [&](int o) -> float { return X[(8 + o) >> 2].get((8 + o) & 3); };
    auto pr = [&](int o) -> float2 { return X[(8 + o) >> 2].p[((8 + o) & 3) >> 1]; };   // o even
#pragma unroll
    for (int d = 1; d <= kRadius; ++d) {
        if (d & 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i) acc.set(i, fmaf(cf.a[d], at(i - d) + at(i + d), acc.get(i)));
        } else {
            const float2 c = make_float2(cf.a[d], cf.a[d]);
#pragma unroll
            for (int i = 0; i < 2; ++i) acc.p[i] = __ffma2_rn(c, __fadd2_rn(pr(2 * i - d), pr(2 * i + d)), acc.p[i]);
        }
    }
}
__device__ __forceinline__ void x_part(Pk<double> &acc, const Pk<double> (&X)[7], const Coef<double> &cf) {
    auto at = [&](int o) -> double { return X[(6 + o) >> 1].get((6 + o) & 1); };
#pragma unroll
    for (int d = 1; d <= kRadius; ++d)
#pragma unroll
        for (int i = 0; i < 2; ++i) acc.set(i, ::fma(cf.a[d], at(i - d) + at(i + d), acc.get(i)));
}

// Three sums into a block of the cluster, counted on its barrier.
__device__ __forceinline__ void send_sums(unsigned to, unsigned bar, float a, float b, float c) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(to),
                 "f"(a), "f"(b), "f"(c), "f"(0.f), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send_sums(unsigned to, unsigned bar, double a, double b, double c) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(to), "d"(a),
                 "d"(b), "r"(bar)
                 : "memory");
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(to + 16),
                 "d"(c), "d"(0.0), "r"(bar)
                 : "memory");
}

template <typename T> struct Vec4;
template <> struct Vec4<float> { using t = float4; };
template <> struct Vec4<double> { using t = double4_16a; };

// The scalar lane's state of a solve (in shared memory: the other threads' registers hold points).
struct ScalarState {
    double dr, di;                       // 1 / d_{k-1}
    double zr, zi;                       // z_{k-1}
    double gam;                          // g_k
    double ak, ck, ig;                   // the step whose factors are pending: a_k, c_k, 1 / g_{k+1}
    double thr, d0, w, rn2;              // threshold, diagonal of B but V_loc, omega, sum of ||r||^2
    int sweeps, fail;                    // fail: 1 limit, 2 breakdown, 3 non-finite
};

// A solution to form, for the flush warps: slot s (-1: no more), n vectors of history buffer buf, the part's phase.
struct Job {
    int s, n, buf, have_p;
    double er, ei;
};

// Shared memory of a block, before its slab of planes.
template <typename T> struct Shared {
    using V4 = typename Vec4<T>::t;
    V4 coef[kHistMax];                   // y_j (re, im), direction coefficient (re, im)
    V4 prev;                             // the same for the direction handed over
    T part[2][16][4];                    // the blocks' sums of a reduction (alternating)
    T red[3][32];
    T vec[4];                            // a', 1/g, g (FP64)
    double dr[2][kHistMax], di[2][kHistMax], zr[2][kHistMax], zi[2][kHistMax], g[2][kHistMax];   // factors by history place
    double start[4];                     // cos phi, sin phi, ||r_a||, ||r_b||
    ScalarState F;
    unsigned long long bar, pbar[2];     // arrival of the halo, of the sums
    union {
        struct {
            unsigned long long ibar[2];              // arrival of the next system
            unsigned long long job_full, job_done;   // a job for the flush warps, and its end
        };
        unsigned long long full[4];      // streaming kernel: arrival of a stage's planes
    };
    Job job;
    int next;                            // its first place that no warp has taken
    unsigned opened;                     // jobs whose coefficients are there
    int item[2], flag;
    unsigned gone;                       // a wait ran out (wait_lost; 0: none did)
    int tell;                            // the blocks told of it (0: this one)
    int taken;                           // on chip: the system taken last (first block)
    int nto, to[4 * 12];                 // the copies that fill the neighbours' halos
    unsigned expect;                     // bytes that arrive in this block's halo
    LanczosArgs<T> A;                    // for the functions off the hot path
};
template <typename T> constexpr int shared_bytes() { return (int)((sizeof(Shared<T>) + 127) / 128 * 128); }

extern __shared__ __align__(128) unsigned char lz_smem[];
template <typename T> __device__ __forceinline__ Pk<T> lds(int off) {
    return pk_load(reinterpret_cast<const T *>(lz_smem + off));
}
template <typename T> __device__ __forceinline__ Shared<T> &sh() { return *reinterpret_cast<Shared<T> *>(lz_smem); }

// A thread's points: W values of x from gx, rows gy and gy + 1, local planes lz0 .. lz0 + ZC - 1.
template <typename T, int ZC> struct Geo {
    static constexpr int W = Pk<T>::W, PAD = W == 4 ? 8 : 6;   // PAD: elements before a row, at least the radius
    int rank, z0, nzl;                   // the block's planes
    bool unit, row1;                     // has points; row gy + 1 lies inside the box
    int gx, gy, lz0, nvx, nvz;           // nvx, nvz: points of a row, planes inside the box
    int c0, c1;                          // its rows' first points in the slab (plane lz0)
    int nthr;                            // threads that may hold points
    __device__ __forceinline__ Geo(const LanczosArgs<T> &A) {
        const int tid = threadIdx.x, per_chunk = A.hw * A.hh;
        rank = (int)(blockIdx.x % (unsigned)A.ncl);
        z0 = rank * A.nz / A.ncl;
        nzl = (rank + 1) * A.nz / A.ncl - z0;
        unit = tid < per_chunk * A.nch;
        const int ch = unit ? tid / per_chunk : 0;
        const int by = unit ? (tid - ch * per_chunk) / A.hw : 0;
        gx = unit ? W * (tid - ch * per_chunk - by * A.hw) : 0;
        gy = 2 * by;
        lz0 = ch * ZC;
        nvx = min(W, A.nx - gx);
        row1 = gy + 1 < A.ny;
        nvz = unit ? max(0, min(ZC, nzl - lz0)) : 0;
        c0 = (lz0 + kRadius) * A.plane + gy * A.pitch + PAD + gx;
        c1 = row1 ? c0 + A.pitch : c0;
        nthr = (int)blockDim.x - kExtra;
    }
    // private 16-byte place of (z, r) in a vector of the workspace, in elements
    __device__ __forceinline__ size_t priv(int z, int r) const { return ((size_t)(2 * z + r) * nthr + threadIdx.x) * W; }
    // index of the row's first point on the grid
    __device__ __forceinline__ long long grid(const LanczosArgs<T> &A, int z, int r) const {
        return ((long long)(z0 + lz0 + z) * A.ny + gy + r) * A.nx + gx;
    }
};
// The block's arrays in the workspace: V_loc by threads; the direction (re, im) and the history, laid out as in
// the slab.
template <typename T, int ZC> struct Work {
    T *V, *Pd, *H;                       // H: two buffers, buf elements apart
    size_t vec, hvec, buf;
    __device__ __forceinline__ Work(const LanczosArgs<T> &A) {
        vec = (size_t)2 * ZC * (blockDim.x - kExtra) * Pk<T>::W;
        hvec = (size_t)A.nch * ZC * A.plane;
        V = A.ws + (size_t)blockIdx.x * A.ws_stride;
        Pd = V + vec;
        H = Pd + 2 * hvec;
        buf = (size_t)A.hist * hvec;
    }
};
template <typename T> __device__ __forceinline__ T *slab_of(const LanczosArgs<T> &A) {
    return reinterpret_cast<T *>(lz_smem + shared_bytes<T>()) + A.lead;   // after the zero word or the first rows of zeros
}

// W values of a row into the slab (periodic: and the images past the row's ends).
template <typename T, int MODE>
__device__ __forceinline__ void put(T *own, int gx, int nvx, int nx, const Pk<T> &v) {
    constexpr int W = Pk<T>::W, PAD = W == 4 ? 8 : 6;
    if (nvx == W) {
        pk_store(own, v);
    } else {
        for (int i = 0; i < nvx; ++i) own[i] = v.get(i);
    }
    if (MODE == 1) {
        if (nx % W == 0) {
            if (gx < PAD) pk_store(own + nx, v);
            if (gx >= nx - PAD) pk_store(own - nx, v);
        } else {
            for (int i = 0; i < nvx; ++i) {
                const int x = gx + i;
                if (x < kRadius) own[i + nx] = v.get(i);
                if (x >= nx - kRadius) own[i - nx] = v.get(i);
            }
        }
    }
}

// A wait ran out.  The threads of a block (on chip) or of a cluster (streaming: its blocks meet at cluster barriers) have
// to go on alike: they end the solve when they next decide on it, behind a barrier (`left`), start no other
// (start_part), and leave the launch before the next system.  The mark is the number of reductions (ng)
// behind that barrier: a decision counts the marks up to its own number only, so that one made meanwhile by a
// thread that is ahead does not divide those that still have to decide.
template <typename T> __device__ __noinline__ void wait_lost(unsigned mark) {
    Shared<T> &S = sh<T>();
    const int ncl = S.tell;
    atomicExch(S.A.err, 2);
    if (ncl == 0) atomicCAS(&S.gone, 0u, mark);          // this block; the first mark stands
    for (int t = 0; t < ncl; ++t) {
        unsigned old;
        asm volatile("atom.relaxed.cluster.shared::cluster.cas.b32 %0, [%1], 0, %2;"
                     : "=r"(old)
                     : "r"(map_rank((unsigned)__cvta_generic_to_shared(&S.gone), t)), "r"(mark)
                     : "memory");
    }
}
template <typename T> __device__ __forceinline__ bool left(unsigned ng) {
    const unsigned d = *(volatile unsigned *)&sh<T>().gone;
    return d != 0 && d <= ng;
}

// Barrier of the threads that iterate (the flush warps run beside them).
__device__ __forceinline__ void main_sync(int nmain) { asm volatile("bar.sync 1, %0;" ::"r"(nmain) : "memory"); }
// The same, and whether any of them says so.
__device__ __forceinline__ bool main_any(int nmain, bool say) {
    int r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.s32 p, %2, 0;\n bar.red.or.pred q, 1, %1, p;\n selp.s32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(nmain), "r"((int)say)
        : "memory");
    return r != 0;
}
// The block's own planes are stored: before the bulk copies read them.
__device__ __forceinline__ void planes_stored(int nmain) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    main_sync(nmain);
}
// The planes to the halos of the blocks that need them (one bulk copy a block and side), by the scalar
// lane once they are stored and no block reads its last halo any more; the phase of sh().bar is complete
// when this block's own halo has arrived.
template <typename T> __device__ __forceinline__ void send_halos(T *slab) {
    Shared<T> &S = sh<T>();
    const unsigned bar = (unsigned)__cvta_generic_to_shared(&S.bar), base = (unsigned)__cvta_generic_to_shared(slab);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(S.expect) : "memory");
    for (int e = 0; e < S.nto; ++e) {
        const int t = S.to[4 * e];
        asm volatile(
            "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                map_rank(base, t) + (unsigned)S.to[4 * e + 1]),
            "r"(base + (unsigned)S.to[4 * e + 2]), "r"(S.to[4 * e + 3]), "r"(map_rank(bar, t))
            : "memory");
    }
}
// The block's planes to place h of the history, by the scalar lane once they are stored; they may change
// again after keep_wait.
template <typename T> __device__ __forceinline__ void keep(const T *slab, T *H, size_t hvec, int h, int nzl, int plane) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                     __cvta_generic_to_global(H + (size_t)h * hvec)),
                 "r"((unsigned)__cvta_generic_to_shared(slab + kRadius * plane)), "r"(nzl * plane * (int)sizeof(T))
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void keep_wait() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// Block sums of three values per thread, all-gathered over the cluster into part[ng & 1]: every block
// sends its sums to all (st.async, which counts on the receiver's barrier) and waits for all.  A block
// sends only after all its threads are done with the stencil, so the wait also says that no block reads
// its halo any more.  The sums alternate between two buffers and barriers: a block may be one
// reduction ahead of another, never two.
template <typename T>
__device__ __forceinline__ void gather3(T a, T b, T c, unsigned &ng, int ncl, int rank, int nmain) {
    Shared<T> &S = sh<T>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = nmain >> 5;
    T v[3] = {a, b, c};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 3; ++q) S.red[q][warp] = v[q];
    main_sync(nmain);
    const unsigned pb = (unsigned)__cvta_generic_to_shared(&S.pbar[ng & 1]);
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q] = lane < nwarp ? S.red[q][lane] : (T)0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < 3; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(pb),
                         "r"((unsigned)(ncl * 4 * (int)sizeof(T)))
                         : "memory");
        if (lane < ncl)
            send_sums(map_rank((unsigned)__cvta_generic_to_shared(&S.part[ng & 1][rank][0]), lane), map_rank(pb, lane),
                      v[0], v[1], v[2]);
        __syncwarp();
    }
    if (!mbar_wait(pb, (ng >> 1) & 1)) wait_lost<T>(ng + 1);
    ++ng;
}
template <typename T> __device__ __forceinline__ void sum_parts(unsigned ng, int ncl, T &a, T &b, T &c) {   // after gather3
    const T(&pp)[16][4] = sh<T>().part[(ng & 1) ^ 1];
    a = b = c = (T)0;
    for (int t = 0; t < ncl; ++t) {
        a += pp[t][0];
        b += pp[t][1];
        c += pp[t][2];
    }
}

// The pending step's factors, by the scalar lane while the others compute the next stencil: d_k and z_k of
// the LU of T + i w, the residual and the stopping test (flag: 0 go on, 1 converged, 2 limit, 3 breakdown,
// 4 non-finite); j its place in the history, steps the steps so far.
template <typename T> __device__ __forceinline__ void factor(int buf, int j, int steps, int maxit) {
    Shared<T> &S = sh<T>();
    ScalarState &F = S.F;
    const double ig = F.ig, g1 = ig > 0.0 ? 1.0 / ig : 0.0;
    const double lr = F.gam * F.dr, li = F.gam * F.di;               // l_k = g_k / d_{k-1}
    const double er = F.ak - lr * F.ck, ei = F.w - li * F.ck;
    const double q = er * er + ei * ei, iq = 1.0 / q;
    const double zr = steps > 1 ? -(lr * F.zr - li * F.zi) : F.zr;
    const double zi = steps > 1 ? -(lr * F.zi + li * F.zr) : 0.0;
    const double dr = er * iq, di = -ei * iq;
    const double yr = zr * dr - zi * di, yi = zr * di + zi * dr;
    const double rn = g1 * sqrt(yr * yr + yi * yi);
    S.dr[buf][j] = F.dr = dr;
    S.di[buf][j] = F.di = di;
    S.zr[buf][j] = F.zr = zr;
    S.zi[buf][j] = F.zi = zi;
    S.g[buf][j] = F.gam;
    F.gam = g1;
    F.sweeps += 1;
    int flag = 0;
    if (!isfinite(rn) || !(ig == ig)) flag = 4;
    else if (!(q > 0.0)) flag = 3;
    else if (rn <= F.thr) flag = 1;
    else if (steps >= maxit) flag = 2;
    if (flag) F.rn2 += flag < 3 ? rn * rn : (double)INFINITY;
    if (flag > 1) F.fail = max(F.fail, flag - 1);
    S.flag = flag;
}

// Off the hot path, in functions of their own so that the iteration keeps its registers.

// The scalar lane, from the right-hand side's sums (Re^2, Im^2, Re Im): its phase phi = arg(r^T r) / 2 and the
// norms of its two parts, r_a^2 = sum + |r^T r| / 2, r_b^2 = sum - |r^T r| / 2.
template <typename T> __device__ __noinline__ void start_state(T a, T b, T c, double d0, double w) {
    Shared<T> &S = sh<T>();
    const double sum = 0.5 * ((double)a + (double)b), D = 0.5 * ((double)a - (double)b), O = (double)c;
    const double m = sqrt(D * D + O * O);
    double cs = 1.0, sn = 0.0;
    if (m > 0.0 && (double)b > 0.0) {
        cs = sqrt(fmax(0.0, 0.5 * (1.0 + D / m)));
        sn = copysign(sqrt(fmax(0.0, 0.5 * (1.0 - D / m))), O);
    }
    S.start[0] = cs;
    S.start[1] = sn;
    S.start[2] = sqrt(sum + m);
    S.start[3] = (double)b > 0.0 ? sqrt(fmax(0.0, sum - m)) : 0.0;
    S.F.sweeps = S.F.fail = 0;
    S.F.rn2 = 0.0;
    S.F.d0 = d0;                                         // 3 a_0 and the shift of H: -eps_n
    S.F.w = w;
}

// Start of part pt of slot s's solve (every thread): false if there is nothing to solve for (uniform over
// the cluster), else v_0 = f_re Re(r) + f_im Im(r).
template <typename T> __device__ __noinline__ bool start_part(const LanczosArgs<T> &A, int s, int pt, bool scalar, unsigned ng, T &f_re,
                                                                T &f_im) {
    Shared<T> &S = sh<T>();
    if (left<T>(ng)) {                                   // no solve, and the system has failed
        if (scalar) S.F.fail = 3;
        return false;
    }
    const Slot &sl = A.slots[s];
    const double thr_all = A.mixed ? fmax(A.inner_tol * sl.ref_norm, 0.3 * A.tol * sl.bnorm * sl.scale)
                                   : A.tol * sl.bnorm;
    const double na = S.start[2], nb = S.start[3], beta = pt ? nb : na;
    // The parts' residuals add as orthogonal vectors nearly do.  A small r_b (rounding noise of the last inner
    // solve) gets a small share of the threshold, comparable parts equal shares.
    const double thr = thr_all * (nb == 0.0 ? 1.0 : nb > 0.1 * na ? 0.7 : pt ? 0.3 : 0.95);
    if (!(beta > thr)) {
        if (scalar) {
            S.F.rn2 += beta * beta;
            if (!(beta <= thr)) S.F.fail = 3;            // not a number
        }
        return false;
    }
    if (scalar) {
        S.F.dr = S.F.di = S.F.zi = S.F.gam = 0.0;
        S.F.zr = beta;
        S.F.thr = thr;
        S.flag = 0;
    }
    const double ib = 1.0 / beta;
    f_re = (T)((pt ? -S.start[1] : S.start[0]) * ib);
    f_im = (T)((pt ? S.start[0] : S.start[1]) * ib);
    return true;
}

// The slot's state after its solve (the scalar lane of the cluster's first block).
template <typename T> __device__ __noinline__ void end_state(const LanczosArgs<T> &A, int s) {
    Slot &sl = A.slots[s];
    const ScalarState &F = sh<T>().F;
    sl.iters = F.sweeps;
    sl.total_iters += F.sweeps;
    sl.rnorm = sqrt(F.rn2);
    if (A.mixed) {
        if (F.fail == 3) sl.discard = 1;
        if (F.fail >= 2) sl.status = RPA_ERR_BREAKDOWN;
        sl.phase = kInnerDone;
    } else {
        sl.status = F.fail == 0 ? RPA_OK : F.fail == 1 ? RPA_ERR_NOT_CONVERGED : RPA_ERR_BREAKDOWN;
        sl.phase = kFinished;
    }
}

// A wait ran out, in this launch or before it: the call fails (err is set) and its systems end unsolved, so that the
// queue does.  A slot that no cluster goes on with, and every system that none has taken yet.
template <typename T> __device__ __noinline__ void fail_slot(const LanczosArgs<T> &A, int s) {
    A.slots[s].status = RPA_ERR_CUDA;
    A.slots[s].phase = kFinished;
}
template <typename T> __device__ __noinline__ void fail_rest(const LanczosArgs<T> &A, int n_items) {
    for (int it; (it = atomicAdd(A.grab, 1)) < n_items;) fail_slot(A, A.list[n_items - 1 - it]);
}

// The thread's sums of Re(r)^2, Im(r)^2 and Re(r) Im(r) over its points of slot s.
template <typename T, int ZC> __device__ __noinline__ void start_sums(int s, T &rr, T &ii, T &ri) {
    using C = typename Cx<T>::t;
    const LanczosArgs<T> &A = sh<T>().A;
    const Geo<T, ZC> G(A);
    const C *const rg = A.r + (long long)s * A.nd;
    T a = 0, b = 0, c = 0;
#pragma unroll
    for (int r = 0; r < 2; ++r)
        if (r == 0 || G.row1) {
            C v[ZC][G.W];
#pragma unroll
            for (int z = 0; z < ZC; ++z) {
                const C *src = rg + G.grid(A, z, r);
#pragma unroll
                for (int i = 0; i < G.W; ++i) v[z][i] = z < G.nvz && i < G.nvx ? src[i] : C{0, 0};
            }
#pragma unroll
            for (int z = 0; z < ZC; ++z)
#pragma unroll
                for (int i = 0; i < G.W; ++i) {
                    a += v[z][i].x * v[z][i].x;
                    b += v[z][i].y * v[z][i].y;
                    c += v[z][i].x * v[z][i].y;
                }
        }
    rr = a;
    ii = b;
    ri = c;
}

// v_0 = f_re Re(r) + f_im Im(r) of slot s into the slab.
template <typename T, int ZC, int MODE> __device__ __noinline__ void start_vector(int s, T f_re, T f_im) {
    using C = typename Cx<T>::t;
    const LanczosArgs<T> &A = sh<T>().A;
    const Geo<T, ZC> G(A);
    const C *const rg = A.r + (long long)s * A.nd;
    T *const slab = slab_of(A);
#pragma unroll
    for (int r = 0; r < 2; ++r)
        if (r == 0 || G.row1) {
            C v[ZC][G.W];
#pragma unroll
            for (int z = 0; z < ZC; ++z) {
                const C *src = rg + G.grid(A, z, r);
#pragma unroll
                for (int i = 0; i < G.W; ++i) v[z][i] = z < G.nvz && i < G.nvx ? src[i] : C{0, 0};
            }
#pragma unroll
            for (int z = 0; z < ZC; ++z)
                if (z < G.nvz) {
                    Pk<T> w;
#pragma unroll
                    for (int i = 0; i < G.W; ++i) w.set(i, f_re * v[z][i].x + f_im * v[z][i].y);
                    put<T, MODE>(slab + (r ? G.c1 : G.c0) + z * A.plane, G.gx, G.nvx, A.nx, w);
                }
        }
}

// The solution's coefficients, by one thread: x += sum_j y_j v_j over the n vectors of history buffer buf, y from
// U y = z backwards (times the part's phase er + i ei), prev: of the direction handed over by the last time; the
// COCG direction of the last vector, p = sum_j q_j v_j + q_prev p_prev, likewise.
template <typename T> __device__ __noinline__ void coefficients(int buf, int n, double er, double ei) {
    using V4 = typename Vec4<T>::t;
    Shared<T> &S = sh<T>();
    double yr = 0, yi = 0, qr = 0, qi = 0;
    for (int j = n - 1; j >= 0; --j) {
        const double cn = j + 1 < n ? (double)(T)S.g[buf][j + 1] : 0.0, dr = S.dr[buf][j], di = S.di[buf][j];
        const double tr = S.zr[buf][j] - cn * yr, ti = S.zi[buf][j] - cn * yi;
        yr = tr * dr - ti * di;
        yi = tr * di + ti * dr;
        const double ur = j == n - 1 ? 1.0 : -cn * qr, ui = j == n - 1 ? 0.0 : -cn * qi;
        qr = ur * dr - ui * di;
        qi = ur * di + ui * dr;
        V4 c;
        c.x = (T)(er * yr - ei * yi);
        c.y = (T)(er * yi + ei * yr);
        c.z = (T)qr;
        c.w = (T)qi;
        S.coef[j] = c;
    }
    const double c0 = (double)(T)S.g[buf][0];
    V4 c;
    c.x = (T)(-c0 * (er * yr - ei * yi));
    c.y = (T)(-c0 * (er * yi + ei * yr));
    c.z = (T)(-c0 * qr);
    c.w = (T)(-c0 * qi);
    S.prev = c;
}

// x of slot s += the history's sum at the 16-byte places e, e + nt .. of the block's planes (GO: and the
// direction handed over formed anew), NP places a thread.  Two warps have to keep up with the others' iterations, and one warp
// issues an instruction every four to five cycles: four 16-byte places at a time, so that a coefficient is
// read once for four loads, whose addresses advance by additions (a first form with two places and products
// in the addresses took 29 to 42 thousand cycles a vector of 16000 points, 9 with all 13 warps).
template <typename T, int ZC, bool GO, int NP> __device__ __forceinline__ void add_history(const Job &J, int e, int nt) {
    using P = Pk<T>;
    using C = typename Cx<T>::t;
    using V4 = typename Vec4<T>::t;
    constexpr int W = P::W, PAD = Geo<T, ZC>::PAD;
    Shared<T> &S = sh<T>();
    const LanczosArgs<T> &A = S.A;
    const Work<T, ZC> K(A);
    const int rank = (int)(blockIdx.x % (unsigned)A.ncl), z0 = rank * A.nz / A.ncl, nzl = (rank + 1) * A.nz / A.ncl - z0;
    const int rows = nzl * A.ny, total = rows * A.hw, n = J.n;
    const T *const H = K.H + J.buf * K.buf;
    const size_t step = K.hvec;
    const T *q[NP];
    int o[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        const int m = min(e + h * nt, total - 1);    // past the end: the last place again, not stored
        const int row = m / A.hw, z = row / A.ny;
        o[h] = z * A.plane + (row - z * A.ny) * A.pitch + PAD + W * (m - row * A.hw);
        q[h] = H + o[h];
    }
    P xr[NP], xi[NP], pr[NP], pi[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        xr[h].zero();
        xi[h].zero();
        pr[h].zero();
        pi[h].zero();
    }
    auto add = [&](int j, const P (&v)[NP]) {
        const V4 c = S.coef[j];
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            xr[h].fma(c.x, v[h]);
            xi[h].fma(c.y, v[h]);
            if (GO) {
                pr[h].fma(c.z, v[h]);
                pi[h].fma(c.w, v[h]);
            }
        }
    };
    auto load = [&](P (&v)[NP]) {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            v[h] = pk_load_l2(q[h]);
            q[h] += step;
        }
    };
    int j = 0;
    for (; j + 4 <= n; j += 4) {
        P v0[NP], v1[NP], v2[NP], v3[NP];
        load(v0);
        load(v1);
        load(v2);
        load(v3);
        add(j, v0);
        add(j + 1, v1);
        add(j + 2, v2);
        add(j + 3, v3);
    }
    for (; j < n; ++j) {
        P v0[NP];
        load(v0);
        add(j, v0);
    }
    const V4 pv = S.prev;
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        if (e + h * nt >= total) continue;
        if (J.have_p) {
            const P qr = pk_load_l2(K.Pd + o[h]), qi = pk_load_l2(K.Pd + K.hvec + o[h]);
            xr[h].fma(pv.x, qr);
            xr[h].fma(-pv.y, qi);
            xi[h].fma(pv.x, qi);
            xi[h].fma(pv.y, qr);
            if (GO) {
                pr[h].fma(pv.z, qr);
                pr[h].fma(-pv.w, qi);
                pi[h].fma(pv.z, qi);
                pi[h].fma(pv.w, qr);
            }
        }
        if (GO) {
            pk_store(K.Pd + o[h], pr[h]);
            pk_store(K.Pd + K.hvec + o[h], pi[h]);
        }
        const int m = e + h * nt, row = m / A.hw, gx = W * (m - row * A.hw), nvx = min(W, A.nx - gx);
        C *dst = A.x + (long long)J.s * A.nd + ((long long)z0 * A.ny + row) * A.nx + gx;
        C c[W];
#pragma unroll
        for (int i = 0; i < W; ++i) c[i] = i < nvx ? __ldcg(dst + i) : C{0, 0};
#pragma unroll
        for (int i = 0; i < W; ++i)
            if (i < nvx) {
                c[i].x += xr[h].get(i);
                c[i].y += xi[h].get(i);
                dst[i] = c[i];
            }
    }
}

// The places of the job in hand that no warp has taken, NP rows of 32 at a time: by the flush warps, and by
// the others once they are at the end of the next part (a place's sum is the same whoever forms it).
template <typename T, int ZC, int NP> __device__ __noinline__ void take_places() {
    Shared<T> &S = sh<T>();
    const int rank = (int)(blockIdx.x % (unsigned)S.A.ncl), lane = (int)threadIdx.x & 31;
    const int total = ((rank + 1) * S.A.nz / S.A.ncl - rank * S.A.nz / S.A.ncl) * S.A.ny * S.A.hw;
    for (;;) {
        int e = 0;
        if (lane == 0) e = atomicAdd(&S.next, 32 * NP);
        e = __shfl_sync(0xffffffffu, e, 0);
        if (e >= total) break;
        __threadfence_block();
        add_history<T, ZC, false, NP>(S.job, e + lane, 32);
    }
    __threadfence();
}

// The flush warps: forms the solution of every finished part while the other warps go on with the next.
template <typename T, int ZC> __device__ __noinline__ void flush_warps() {
    Shared<T> &S = sh<T>();
    const int t = (int)threadIdx.x - ((int)blockDim.x - kFlushThreads);
    const unsigned full = (unsigned)__cvta_generic_to_shared(&S.job_full), done = (unsigned)__cvta_generic_to_shared(&S.job_done);
    for (unsigned job = 1;; ++job) {
        if (!mbar_wait(full, (job - 1) & 1, 200000000000LL)) {
            atomicExch(S.A.err, 2);
            return;
        }
        const Job J = S.job;
        if (J.s < 0) return;
        if (t == 0) {
            coefficients<T>(J.buf, J.n, J.er, J.ei);
            __threadfence_block();
            atomicExch(&S.next, 0);
            *(volatile unsigned *)&S.opened = job;
        }
        asm volatile("bar.sync 2, %0;" ::"r"(kFlushThreads) : "memory");
        take_places<T, ZC, 4>();
        asm volatile("bar.sync 2, %0;" ::"r"(kFlushThreads) : "memory");
        if (t == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(done) : "memory");
    }
}

// The threads that iterate, before the history's next use: the last job is done.
template <typename T, int ZC> __device__ __forceinline__ void finish_job(int nmain) {
    take_places<T, ZC, 2>();
    main_sync(nmain);
}
// The scalar lane then: the flush warps are done with it too (njobs posted so far).  False where the wait ran out.
template <typename T> __device__ __forceinline__ bool jobs_done(unsigned njobs, unsigned ng) {
    const bool ok = njobs == 0 || mbar_wait((unsigned)__cvta_generic_to_shared(&sh<T>().job_done), (njobs - 1) & 1);
    if (!ok) wait_lost<T>(ng + 1);
    return ok;
}
// ... and the next (not posted where the wait ran out: the flush warps still read the last).
template <typename T> __device__ __forceinline__ void post_job(const Job &J, unsigned &njobs, unsigned ng) {
    Shared<T> &S = sh<T>();
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");    // the history is written
    if (!jobs_done<T>(njobs, ng)) return;
    S.job = J;
    ++njobs;
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"((unsigned)__cvta_generic_to_shared(&S.job_full)) : "memory");
}

// The history is full: its sum into x, the direction handed over, by the threads that iterate.
template <typename T, int ZC> __device__ __noinline__ void flush_full(const Job &J, unsigned njobs, unsigned ng, int nmain) {
    finish_job<T, ZC>(nmain);
    if ((int)threadIdx.x == nmain - 32) {
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        if (jobs_done<T>(njobs, ng)) coefficients<T>(J.buf, J.n, J.er, J.ei);
    }
    main_sync(nmain);
    const int rank = (int)(blockIdx.x % (unsigned)sh<T>().A.ncl), nz = sh<T>().A.nz, ncl = sh<T>().A.ncl;
    const int total = ((rank + 1) * nz / ncl - rank * nz / ncl) * sh<T>().A.ny * sh<T>().A.hw;
    for (int e = threadIdx.x; e < total; e += 2 * nmain) add_history<T, ZC, true, 2>(J, e, nmain);
    __threadfence();
    main_sync(nmain);
}

// The end of a block that leaves after a wait has run out, by the scalar lane: the system taken last is given up,
// the block's own copies are waited for, the flush warps sent home (they end by themselves where even their
// last job's end does not come), and what is on its way to this block, sent before another one left, is given
// half a millisecond to arrive.  The other blocks of the cluster leave likewise: they wait for this one's
// sums, each wait for a second at most.
template <typename T> __device__ __noinline__ void leave(int rank, int n_items, unsigned njobs, unsigned ng) {
    Shared<T> &S = sh<T>();
    const LanczosArgs<T> &A = S.A;
    if (rank == 0) {
        if (S.taken < n_items) fail_slot(A, A.list[n_items - 1 - S.taken]);
        fail_rest(A, n_items);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    post_job<T>(Job{-1, 0, 0, 0, 0.0, 0.0}, njobs, ng);
    const long long t0 = clock64();
    while (clock64() - t0 < 1000000LL) {}
}

// Once a block: its slab cleared, barriers, the halo copies, V_loc by threads.
template <typename T, int ZC> __device__ __noinline__ void block_setup(const LanczosArgs<T> *args, bool per) {
    Shared<T> &S = sh<T>();
    const LanczosArgs<T> &A = *args;
    const Geo<T, ZC> G(A);
    const Work<T, ZC> K(A);
    for (int e = threadIdx.x; e < A.smem_words; e += blockDim.x)
        reinterpret_cast<int4 *>(lz_smem + shared_bytes<T>())[e] = make_int4(0, 0, 0, 0);
    if ((int)threadIdx.x < G.nthr)
        for (int z = 0; z < ZC; ++z)
            for (int r = 0; r < 2; ++r) {
                Pk<T> v;
#pragma unroll
                for (int i = 0; i < G.W; ++i)
                    v.set(i, z < G.nvz && (r == 0 || G.row1) && i < G.nvx ? A.vloc[G.grid(A, z, r) + i] : (T)0);
                pk_store(K.V + G.priv(z, r), v);
            }
    if ((int)threadIdx.x == G.nthr) {
        mbar_init(&S.bar);
        for (int q = 0; q < 2; ++q) mbar_init(&S.pbar[q]);
        for (int q = 0; q < 2; ++q) mbar_init(&S.ibar[q]);
        mbar_init(&S.job_full);
        mbar_init(&S.job_done);
        S.next = 1 << 30;                                // no job
        S.gone = 0;
        S.tell = 0;
        S.taken = 1 << 30;
        S.opened = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // the copies: this block's planes [g0, g1) that lie in the halo of rank t (periodic: of its image)
        const int ncl = A.ncl, nz = A.nz, z0 = G.z0, z1 = G.z0 + G.nzl, pb = A.plane * (int)sizeof(T);
        int n = 0, bytes = 0;
        for (int dt = -A.reach; dt <= A.reach; ++dt) {
            int t = G.rank + dt, base = 0;
            if (dt == 0) continue;
            if (t < 0 || t >= ncl) {
                if (!per) continue;
                const int w = t < 0 ? -((ncl - 1 - t) / ncl) : t / ncl;
                t -= w * ncl;
                base = w * nz;
            }
            const int t0 = base + t * nz / ncl, t1 = base + (t + 1) * nz / ncl;   // rank t's planes
            const int g0 = max(z0, t0 - kRadius), g1 = min(z1, t1 + kRadius);
            if (g0 < g1) {
                S.to[4 * n] = t;
                S.to[4 * n + 1] = (g0 - t0 + kRadius) * pb;
                S.to[4 * n + 2] = (g0 - z0 + kRadius) * pb;
                S.to[4 * n + 3] = (g1 - g0) * pb;
                ++n;
            }
            // and rank t's planes in this block's halo
            bytes += max(0, min(t1, z1 + kRadius) - max(t0, z0 - kRadius)) * pb;
        }
        S.nto = n;
        S.expect = (unsigned)bytes;
    }
}

// MODE: 0 zero values outside the box, kept as rows of zeros between the planes; 1 periodic; 2 zero
// values outside the box, read from a zero word (less shared memory, a select per row)
template <typename T, int ZC, int MAXT, int MODE>
__global__ void __launch_bounds__(MAXT, 1) k_lanczos(const __grid_constant__ LanczosArgs<T> A, const __grid_constant__ Coef<T> cf) {
    using P = Pk<T>;
    constexpr bool PER = MODE == 1;
    constexpr int W = P::W;
    constexpr int PAD = Geo<T, ZC>::PAD;
    constexpr int XL = (2 * PAD + W) / W;               // 16-byte loads of a row's x neighbours
    Shared<T> &S = sh<T>();
    const int tid = threadIdx.x, ncl = A.ncl;
    if (tid == 0) S.A = A;
    __syncthreads();
    block_setup<T, ZC>(&S.A, PER);
    const Geo<T, ZC> G(A);
    const int nmain = G.nthr + 32;                      // threads that iterate: points and the scalar warp
    const bool scalar = tid == G.nthr;
    T *const slab = slab_of(A);
    const int slab_off = shared_bytes<T>() + A.lead * (int)sizeof(T);
    const int pb = A.plane * (int)sizeof(T), rb = A.pitch * (int)sizeof(T);   // bytes of a plane, a row
    constexpr int QB = 16;                              // bytes of W values
    const int n_items = *A.cnt;
    unsigned phase = 0, ng = 0, ns = 0, njobs = 0;      // halo phase; reductions, systems, jobs so far
    int buf = 0;                                        // history buffer
    // the next system, by the scalar lane of the first block, from the end of the list (the highest orbitals,
    // the longest solves, first); every block receives its number in item[m & 1]
    auto fetch = [&](unsigned m) {
        if (G.rank == 0) {
            const int err = *(volatile int *)A.err;
            int it = atomicAdd(A.grab, 1);
            if (err) {                                   // no more
                if (it < n_items) fail_slot(A, A.list[n_items - 1 - it]);
                fail_rest(A, n_items);
                it = 1 << 30;
            }
            S.taken = it;
            for (int t = 0; t < ncl; ++t)
                asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                                 map_rank((unsigned)__cvta_generic_to_shared(&S.item[m & 1]), t)),
                             "r"(it), "r"(map_rank((unsigned)__cvta_generic_to_shared(&S.ibar[m & 1]), t))
                             : "memory");
        }
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], 4;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(&S.ibar[m & 1]))
                     : "memory");
    };
    cluster_barrier();                                  // every block runs, has cleared its slab and set its barriers
    if (tid >= nmain) {
        flush_warps<T, ZC>();
        cluster_barrier();
        return;
    }
    if (scalar) fetch(0);
    for (;; ++ns) {
        const bool here = mbar_wait((unsigned)__cvta_generic_to_shared(&S.ibar[ns & 1]), (ns >> 1) & 1);
        if (!here) wait_lost<T>(ng + 1);
        if (main_any(nmain, !here || left<T>(ng))) {    // the item is not to be read, or a solve has ended so
            if (scalar) leave<T>(G.rank, n_items, njobs, ng);
            cluster_barrier();
            return;
        }
        const int it = S.item[ns & 1];
        if (it >= n_items) break;
        const int s = A.list[n_items - 1 - it];
        // the right-hand side's phase and the norms of its two parts
        {
            T rr, ii, ri;
            start_sums<T, ZC>(s, rr, ii, ri);
            gather3(rr, ii, ri, ng, ncl, G.rank, nmain);
            if (scalar && !left<T>(ng)) {
                fetch(ns + 1);                           // every block has read the number before this one
                T a, b, c;
                sum_parts(ng, ncl, a, b, c);
                start_state<T>(a, b, c, A.d0 + A.slots[s].shift_re, A.slots[s].shift_im);
            }
            main_sync(nmain);
        }
        for (int pt = 0; pt < 2; ++pt) {
            T f_re, f_im;
            if (!start_part<T>(A, s, pt, scalar, ng, f_re, f_im)) continue;
            start_vector<T, ZC, MODE>(s, f_re, f_im);
            planes_stored(nmain);
            if (scalar) {
                const Work<T, ZC> K(A);
                send_halos(slab);
                keep(slab, K.H + buf * K.buf, K.hvec, 0, G.nzl, A.plane);
            }
            P acc[ZC][2];
#pragma unroll
            for (int z = 0; z < ZC; ++z) {
                acc[z][0].zero();
                acc[z][1].zero();
            }
            T dg = (T)S.F.d0, cc = 0;                    // diagonal used (shifted by the last a_k), c_k
            int k = 0, kb = 0, n = 0;                    // step, first vector of the history, vectors to flush
            bool have_p = false;
            for (;;) {
                // byte offsets of the unit's rows: made opaque so that the hundreds of addresses formed from
                // them are not kept (and spilled) across iterations
                int o0 = slab_off + G.c0 * (int)sizeof(T), o1 = slab_off + G.c1 * (int)sizeof(T);
                asm volatile("" : "+r"(o0), "+r"(o1));
                if (scalar) {
                    if (k > kb) factor<T>(buf, k - 1 - kb, k, A.maxit);
                    if (left<T>(ng)) {
                        S.F.fail = 3;
                        S.flag = 4;
                    }
                    keep_wait();
                }
                // ---- u = B v_k - c_k v_{k-1} (shifted), sums v.v, u.v, u.u.  The x and y neighbours and the
                // diagonal lie in the block's own planes: first, while the halo is on its way.
                T svv = 0, suv = 0, suu = 0;
                P mask;                                  // 1 for points inside the box
#pragma unroll
                for (int i = 0; i < W; ++i) mask.set(i, i < G.nvx ? (T)1 : (T)0);
                if (G.unit) {
                    // the row r rows from the unit's first, at offset o
                    auto yrow = [&](int o, int r) -> P {
                        if (MODE == 0) return lds<T>(o + r * rb);
                        int y = G.gy + r;
                        if (MODE == 2) return lds<T>(y >= 0 && y < A.ny ? o + r * rb : shared_bytes<T>());
                        y = y < 0 ? y + A.ny : y >= A.ny ? y - A.ny : y;
                        return lds<T>(o + (y - G.gy) * rb);
                    };
                    const T *const wv = A.ws + (size_t)blockIdx.x * A.ws_stride + (size_t)tid * W;
                    const int vs = G.nthr * W;
                    P vn[2];
                    vn[0] = pk_load(wv);
                    vn[1] = pk_load(wv + vs);
#pragma unroll
                    for (int z = 0; z < ZC; ++z) {
                        P &a0 = acc[z][0], &a1 = acc[z][1];
                        a0.mul(-cc);
                        a1.mul(-cc);
                        if (z < G.nvz) {
                            const int q0 = o0 + z * pb, q1 = o1 + z * pb;
                            const P pv0 = vn[0], pv1 = vn[1];
                            if (z + 1 < ZC) {
                                vn[0] = pk_load(wv + (2 * z + 2) * vs);
                                vn[1] = pk_load(wv + (2 * z + 3) * vs);
                            }
                            P ctr0, ctr1, nb1;
                            {
                                P X[XL];
#pragma unroll
                                for (int m = 0; m < XL; ++m) X[m] = lds<T>(q0 + (m - PAD / W) * QB);
                                ctr0 = X[PAD / W];
                                x_part(a0, X, cf);
                            }
                            {
                                P X[XL];
#pragma unroll
                                for (int m = 0; m < XL; ++m) X[m] = lds<T>(q1 + (m - PAD / W) * QB);
                                ctr1 = X[PAD / W];
                                x_part(a1, X, cf);
                            }
                            nb1 = G.row1 ? ctr1 : yrow(q0, 1);
                            a0.fma(cf.a[1], nb1);
                            a1.fma(cf.a[1], ctr0);
#pragma unroll
                            for (int d = 1; d <= kRadius; ++d) {
                                const P lo = yrow(q0, -d), hi = yrow(q0, 1 + d);
                                a0.fma(cf.a[d], lo);
                                a1.fma(cf.a[d], hi);
                                if (d < kRadius) {
                                    a1.fma(cf.a[d + 1], lo);
                                    a0.fma(cf.a[d + 1], hi);
                                }
                            }
                            a0.fma(dg, ctr0);
                            a1.fma(dg, ctr1);
                            a0.fma(pv0, ctr0);
                            a1.fma(pv1, ctr1);
                            if (PER) {                   // a periodic row's images are no points
                                ctr0.mul(mask);
                                ctr1.mul(mask);
                            }
                            P t;
                            t.zero();
                            t.fma(ctr0, ctr0);
                            if (G.row1) t.fma(ctr1, ctr1);
                            svv += t.sum();
                        }
                    }
                }
                const bool halo = mbar_wait((unsigned)__cvta_generic_to_shared(&S.bar), phase);
                if (!halo) wait_lost<T>(ng + 1);
                phase ^= 1u;
                if (G.unit) {
#pragma unroll
                    for (int p = 0; p < ZC + 2 * kRadius; ++p) {
                        const P v0 = lds<T>(o0 + (p - kRadius) * pb), v1 = lds<T>(o1 + (p - kRadius) * pb);
#pragma unroll
                        for (int z = 0; z < ZC; ++z) {
                            const int d = p - z - kRadius < 0 ? z + kRadius - p : p - z - kRadius;
                            if (d >= 1 && d <= kRadius) {
                                acc[z][0].fma(cf.a[d], v0);
                                acc[z][1].fma(cf.a[d], v1);
                            }
                        }
                    }
                    P t1, t2;
                    t1.zero();
                    t2.zero();
#pragma unroll
                    for (int z = 0; z < ZC; ++z)
                        if (z < G.nvz) {
                            P &a0 = acc[z][0], &a1 = acc[z][1];
                            a0.mul(mask);                // u = 0 outside the box
                            a1.mul(mask);
                            const P v0 = lds<T>(o0 + z * pb), v1 = lds<T>(o1 + z * pb);
                            t1.fma(a0, v0);
                            t2.fma(a0, a0);
                            if (G.row1) {
                                t1.fma(a1, v1);
                                t2.fma(a1, a1);
                            }
                        }
                    suv = t1.sum();
                    suu = t2.sum();
                }
                gather3(svv, suv, suu, ng, ncl, G.rank, nmain);
                if (S.flag) {                            // the last step ended the solve (k = kb: a lost wait)
                    n = k - kb;
                    break;
                }
                // ---- a' = u.v / v.v, 1/g with g = ||u - a' v||
                T ap = 0, ig = 0;
                if (sizeof(T) == 4 || scalar) {
                    T a, b, c;
                    sum_parts(ng, ncl, a, b, c);
                    ap = b / a;
                    const T b2 = c - ap * b;
                    ig = b2 > (T)0 ? (T)1 / sqrt(b2) : (T)0;
                    if (!isfinite(a) || !isfinite(c)) ig = (T)nan("");
                    if (sizeof(T) == 8) {
                        S.vec[0] = ap;
                        S.vec[1] = ig;
                        S.vec[2] = ig > (T)0 ? (T)1 / ig : (T)0;
                        S.vec[3] = b2 < (T)kNearSpace * c ? a : (T)0;
                    }
                }
                if (sizeof(T) == 8) {
                    main_sync(nmain);
                    const T vv = S.vec[3];
                    ap = S.vec[0];
                    if (vv > (T)0) {                     // g by the sums of w = u - a' v itself, a' with w's rest along v
                        P t1, t2;
                        t1.zero();
                        t2.zero();
                        if (G.unit) {
#pragma unroll
                            for (int z = 0; z < ZC; ++z)
                                if (z < G.nvz) {
#pragma unroll
                                    for (int r = 0; r < 2; ++r)
                                        if (r == 0 || G.row1) {
                                            const P v = lds<T>((r ? o1 : o0) + z * pb);
                                            P w = acc[z][r];
                                            w.fma(-ap, v);
                                            w.mul(mask);
                                            t1.fma(w, v);
                                            t2.fma(w, w);
                                        }
                                }
                        }
                        gather3((T)0, t1.sum(), t2.sum(), ng, ncl, G.rank, nmain);
                        if (scalar) {
                            T a, b, c;
                            sum_parts(ng, ncl, a, b, c);
                            const T da = b / vv, b2 = c - da * b;
                            ig = b2 > (T)0 ? (T)1 / sqrt(b2) : (T)0;
                            if (!isfinite(c)) ig = (T)nan("");
                            S.vec[0] = ap + da;
                            S.vec[1] = ig;
                            S.vec[2] = ig > (T)0 ? (T)1 / ig : (T)0;
                        }
                        main_sync(nmain);
                        ap = S.vec[0];
                    }
                    ig = S.vec[1];
                }
                if (scalar) {
                    S.F.ak = S.F.d0 - (double)dg + (double)ap;   // a_k of B
                    S.F.ck = (double)cc;
                    S.F.ig = (double)ig;
                    if (A.prof && G.rank == 0) atomicAdd(A.prof + 1, (unsigned long long)A.nd);
                }
                // ---- v_{k+1} into the slab; the registers keep v_k
                const T m_ag = -ap * ig;
#pragma unroll
                for (int z = 0; z < ZC; ++z)
                    if (z < G.nvz) {
#pragma unroll
                        for (int r = 0; r < 2; ++r)
                            if (r == 0 || G.row1) {
                                T *const own = reinterpret_cast<T *>(lz_smem + (r ? o1 : o0) + z * pb);
                                const P v = pk_load(own);
                                P w = acc[z][r];
                                w.mul(ig);
                                w.fma(m_ag, v);
                                put<T, MODE>(own, G.gx, G.nvx, A.nx, w);
                                acc[z][r] = v;
                            }
                    }
                // the next stencil: its diagonal shifted by a_k (u.v stays small against u.u)
                cc = sizeof(T) == 8 ? S.vec[2] : ig > (T)0 ? (T)1 / ig : (T)0;
                dg -= ap;
                planes_stored(nmain);
                ++k;
                if (k - kb == A.hist) {                  // the history is full: into x and p
                    if (scalar) factor<T>(buf, k - 1 - kb, k, A.maxit);
                    main_sync(nmain);
                    n = k - kb;
                    if (S.flag) break;
                    flush_full<T, ZC>(Job{s, n, buf, have_p, pt ? -S.start[1] : S.start[0], pt ? S.start[0] : S.start[1]},
                                      njobs, ng, nmain);
                    have_p = true;
                    kb = k;
                    const Work<T, ZC> K(A);
                    const T *const hl = K.H + buf * K.buf + (size_t)(A.hist - 1) * K.hvec - kRadius * A.plane;   // v_{k-1} again
#pragma unroll
                    for (int z = 0; z < ZC; ++z) {
                        acc[z][0] = pk_load_l2(hl + G.c0 + z * A.plane);
                        acc[z][1] = pk_load_l2(hl + G.c1 + z * A.plane);
                    }
                }
                if (scalar && halo) {                    // (a lost halo's barrier is not armed again)
                    const Work<T, ZC> K(A);
                    send_halos(slab);
                    keep(slab, K.H + buf * K.buf, K.hvec, k - kb, G.nzl, A.plane);
                }
            }
            finish_job<T, ZC>(nmain);
            if (S.flag < 4) {                            // nothing is kept of a solve that went non-finite
                if (scalar)
                    post_job<T>(Job{s, n, buf, have_p, pt ? -S.start[1] : S.start[0], pt ? S.start[0] : S.start[1]}, njobs, ng);
                buf ^= 1;                                // free again: its last job ended before this one was posted
            } else if (scalar) {
                asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // its places are written anew
            }
            main_sync(nmain);                            // no thread still reads the flag
        }
        if (scalar && G.rank == 0) end_state(A, s);
    }
    // nothing is left to go on with: the last job by all warps, once its coefficients are there
    if (scalar)
        for (int i = 0; i < 1 << 20 && *(volatile unsigned *)&S.opened != njobs; ++i) {}
    main_sync(nmain);
    finish_job<T, ZC>(nmain);
    if (scalar) post_job<T>(Job{-1, 0, 0, 0, 0.0, 0.0}, njobs, ng);
    cluster_barrier();                                  // no block leaves while another may write its memory
}

// ---------------------------------------------------------------------------------------------
// The same solve for grids that do not fit on chip (mixed form): u and the
// vectors stay in memory and a cluster of C blocks marches along z, block c over a band of rows.  One
// sweep is one Lanczos step: at step f a thread (4 x 1 or 4 x 2 points) forms v_k = (u - a' v_{k-1}) / g of plane f
// from the last sweep's u and v_{k-1}, stores it in a plane in shared memory and as vector k of the history,
// and after one barrier applies the x and y neighbours and the diagonal of the stencil.  Along z its values go
// into sums for the planes f-6 .. f+6, which it holds in registers and shifts as it adds (a multiply-add
// writes where the last one read), and plane f-6 of u = B v_k - c v_{k-1} is complete.  u.v is summed with
// the sums that plane f has received so far, twice (B is symmetric).  The six halo rows on either side of
// a band are formed by every block that reads them, so that bands exchange nothing within a sweep.  u and v_{k-1}
// of the planes ahead, and V_loc, arrive by bulk copies, A.depth planes in flight.  v_{k-1} is vector
// k - 1 of the history, so the history costs no traffic of its own: a point takes 16 bytes an iteration (u
// and v_{k-1} in, u and v_k out) and 4 at the end, when the history comes back through the same stages,
// against 64 of the fused COCG kernel on complex vectors.
//
// What bounds it: the latency of a plane's step (loads from a stage, one barrier, 16 to 20 loads of neighbours, a
// hundred dependent multiply-adds) with the 7 to 14 warps that the sums' registers allow, and memory
// bandwidth above 64^3.  A form that kept 14 planes in a shared-memory ring for the z neighbours took 46
// shared-memory loads for 8 points against 20, and twice the bands.  Measured, whole chi0 application: 56^3,
// 256 systems 239 ms with the COCG kernels, 111 with the ring, 83 in this form; 72^3, 256 systems 691, 352, 213.
// ---------------------------------------------------------------------------------------------
constexpr int kStages = 4;               // planes in flight, at most

struct StreamArgs {
    LanczosArgs<float> L;                // slots, queue, tolerances, workspace; pitch, plane: in shared memory
    const float *v;                      // V_loc, rows padded to px
    int bh;                              // rows of a band (even)
    int px;                              // padded row length in memory (a multiple of 4)
    int depth;                           // planes in flight
    size_t nv;                           // elements of a vector in memory: nz ny px
};

// rows of nx values -> rows padded to px
__global__ void k_pad_rows(const float *__restrict__ in, float *__restrict__ out, int nx, int px, long long rows) {
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < rows * px; e += (long long)gridDim.x * blockDim.x) {
        const long long r = e / px;
        const int i = (int)(e - r * px);
        out[e] = i < nx ? in[r * nx + i] : 0.f;
    }
}

// A thread's points of a plane: 4 values of x from gx, R rows from gy.
template <int R> struct StreamGeo {
    int rank, y0, rows, gx, gy, nvx;     // the band's first row and rows inside the box; the unit's first point
    bool own, row1;                      // has points; of R = 2 row gy + 1, too, lies inside the box
    int mem;                             // the first point in a plane in memory
    __device__ __forceinline__ StreamGeo(const StreamArgs &A) {
        const int t = threadIdx.x, hw = A.L.hw, pair = t / hw;
        rank = (int)(blockIdx.x % (unsigned)A.L.ncl);
        y0 = rank * A.bh;
        rows = min(A.bh, A.L.ny - y0);
        gx = 4 * (t - pair * hw);
        gy = y0 + R * pair;
        own = R * pair < rows;
        row1 = R == 2 && own && R * pair + 1 < rows;
        nvx = min(4, A.L.nx - gx);
        mem = own ? gy * A.px + gx : 0;
    }
};
__device__ __forceinline__ void bulk_load(unsigned to, const float *from, int bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(to),
                 "l"(__cvta_generic_to_global(from)), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void expect_bytes(unsigned bar, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Values written by the threads, before bulk copies (after a barrier) read them from memory.
__device__ __forceinline__ void before_bulk() { asm volatile("fence.proxy.async;" ::: "memory"); }

// The stages: planes in flight, each with its barrier; every thread counts along.
struct Stages {
    int st;                              // next stage
    unsigned ph;                         // bit s: parity of stage s's next arrival
    bool ok;
    __device__ __forceinline__ unsigned bar(int s) const {
        return (unsigned)__cvta_generic_to_shared(&sh<float>().full[0]) + 8u * (unsigned)s;
    }
    __device__ __forceinline__ void wait(int *err) {   // !ok: no more copies; the scalar lane tells the cluster
        if (ok && !mbar_wait(bar(st), (ph >> st) & 1)) {
            ok = false;
            atomicExch(err, 2);
        }
    }
    __device__ __forceinline__ void next(int depth) {
        ph ^= 1u << st;
        st = st + 1 == depth ? 0 : st + 1;
    }
};

// x += sum_j y_j v_j over the n vectors of the history (go_on: by plain loads, and the COCG direction; else
// three planes of the band of one vector a stage).
template <int R>
__device__ __noinline__ Stages stream_flush(const StreamArgs *args, int s, int n, bool go_on, bool have_p, double er,
                                            double ei, Stages G4) {
    using P = Pk<float>;
    constexpr int NP = 3;                // planes of the band that a stage holds
    Shared<float> &S = sh<float>();
    const StreamArgs &A = *args;
    const StreamGeo<R> G(A);
    const int ncl = A.L.ncl;
    const bool scalar = (int)threadIdx.x == (int)blockDim.x - 32;
    float *const U = A.L.ws + (size_t)(blockIdx.x / (unsigned)ncl) * A.L.ws_stride;
    float *const Pd = U + 2 * A.nv, *const H = Pd + 2 * A.nv;
    float2 *const xg = A.L.x + (long long)s * A.L.nd;
    if (scalar) coefficients<float>(0, n, er, ei);
    __syncthreads();
    auto add_x = [&](int z, int r, P xr, P xi, P pr, P pi) {
        const size_t o = ((size_t)z * A.L.ny + r) * A.px + G.mem;
        if (have_p) {
            const float4 c = S.prev;
            const P qr = pk_load(Pd + o), qi = pk_load(Pd + A.nv + o);
            xr.fma(c.x, qr);
            xr.fma(-c.y, qi);
            xi.fma(c.x, qi);
            xi.fma(c.y, qr);
            pr.fma(c.z, qr);
            pr.fma(-c.w, qi);
            pi.fma(c.z, qi);
            pi.fma(c.w, qr);
        }
        if (go_on) {
            pk_store(Pd + o, pr);
            pk_store(Pd + A.nv + o, pi);
        }
        float2 *dst = xg + ((long long)z * A.L.ny + G.gy + r) * A.L.nx + G.gx;
        float2 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = i < G.nvx ? dst[i] : make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < G.nvx) dst[i] = make_float2(q[i].x + xr.get(i), q[i].y + xi.get(i));
    };
    if (go_on) {
        if (G.own)
            for (int z = 0; z < A.L.nz; ++z)
                for (int r = 0; r < (G.row1 ? 2 : 1); ++r) {
                    const float *h = H + ((size_t)z * A.L.ny + r) * A.px + G.mem;
                    P xr, xi, pr, pi;
                    xr.zero();
                    xi.zero();
                    pr.zero();
                    pi.zero();
#pragma unroll 8
                    for (int j = 0; j < n; ++j) {
                        const float4 c = S.coef[j];
                        const P v = pk_load(h + (size_t)j * A.nv);
                        xr.fma(c.x, v);
                        xi.fma(c.y, v);
                        pr.fma(c.z, v);
                        pi.fma(c.w, v);
                    }
                    add_x(z, r, xr, xi, pr, pi);
                }
        __syncthreads();
        return G4;
    }
    const size_t pl = (size_t)A.L.ny * A.px;
    const int band = G.rows * A.px, su = (A.bh + 2 * kRadius) * A.px, stb = (2 * su + A.bh * A.px) * 4;
    const int s0 = shared_bytes<float>() + (2 * A.L.plane + 16) * 4;
    const int own_at = s0 + (G.own ? ((G.gy - G.y0) * A.px + G.gx) * 4 : 0), second = G.row1 ? A.px * 4 : 0;
    const int npair = (A.L.nz + NP - 1) / NP, total = npair * n;
    // planes NP zi .. of vector j into stage q
    auto issue = [&](int zi, int j, int q) {
        const int np = min(NP, A.L.nz - NP * zi);
        expect_bytes(G4.bar(q), np * band * 4);
        for (int m = 0; m < np; ++m)
            bulk_load((unsigned)__cvta_generic_to_shared(lz_smem) + (unsigned)(s0 + q * stb + m * band * 4),
                      H + (size_t)j * A.nv + (size_t)(NP * zi + m) * pl + (size_t)G.y0 * A.px, band * 4, G4.bar(q));
    };
    int iz = 0, ij = 0, iq = G4.st;      // the next to issue (the scalar lane's)
    auto issue_next = [&]() {
        if (iz >= npair || !G4.ok) return;
        issue(iz, ij, iq);
        if (++ij == n) {
            ij = 0;
            ++iz;
        }
        iq = iq + 1 == A.depth ? 0 : iq + 1;
    };
    if (scalar) {
        before_bulk();
        for (int i = 0; i < min(total, A.depth); ++i) issue_next();
    }
    for (int zi = 0; zi < npair; ++zi) {
        P xr[NP][R], xi[NP][R];
#pragma unroll
        for (int m = 0; m < NP; ++m)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                xr[m][r].zero();
                xi[m][r].zero();
            }
        for (int j = 0; j < n; ++j) {
            G4.wait(A.L.err);
            const int b = G4.st * stb;
            P v[NP][R];
#pragma unroll
            for (int m = 0; m < NP; ++m)
#pragma unroll
                for (int r = 0; r < R; ++r) v[m][r] = lds<float>(own_at + b + m * band * 4 + r * second);
            const float4 c = S.coef[j];
#pragma unroll
            for (int m = 0; m < NP; ++m)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    xr[m][r].fma(c.x, v[m][r]);
                    xi[m][r].fma(c.y, v[m][r]);
                }
            G4.next(A.depth);
            __syncthreads();             // the stage is read
            if (scalar) issue_next();
        }
        if (G.own)
#pragma unroll
            for (int m = 0; m < NP; ++m)
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (NP * zi + m < A.L.nz && (r == 0 || G.row1)) add_x(NP * zi + m, r, xr[m][r], xi[m][r], xr[m][r], xi[m][r]);
    }
    __syncthreads();
    return G4;
}

// Sums of the right-hand side (f_re = f_im = 0: into sums) or u = f_re Re(r) + f_im Im(r).
template <int R>
__device__ __noinline__ void stream_start(const StreamArgs *args, int s, float f_re, float f_im, bool store, float &rr,
                                          float &ii, float &ri) {
    const StreamArgs &A = *args;
    const StreamGeo<R> G(A);
    float *const U = A.L.ws + (size_t)(blockIdx.x / (unsigned)A.L.ncl) * A.L.ws_stride;
    const float2 *const rg = A.L.r + (long long)s * A.L.nd;
    float a = 0.f, b = 0.f, c = 0.f;
    if (G.own)
#pragma unroll 4
        for (int z = 0; z < A.L.nz; ++z)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (r == 0 || G.row1) {
                    const float2 *src = rg + ((long long)z * A.L.ny + G.gy + r) * A.L.nx + G.gx;
                    Pk<float> w;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 v = i < G.nvx ? src[i] : make_float2(0.f, 0.f);
                        a += v.x * v.x;
                        b += v.y * v.y;
                        c += v.x * v.y;
                        w.set(i, f_re * v.x + f_im * v.y);
                    }
                    if (store) pk_store(U + (size_t)z * A.L.ny * A.px + G.mem + r * A.px, w);
                }
    rr = a;
    ii = b;
    ri = c;
}

// PER: periodic boundaries (R = 1): rows past the box are staged and formed at their images, a row's images beside
// it in its padding, and the planes nz-6 .. nz-1 before and 0 .. 5 after the sweep, for their part along z alone
// (the COCG kernels before: chi0 at 48^3, 128 systems 127 ms, now 55).
template <int R, int MAXT, bool PER>
__global__ void __launch_bounds__(MAXT, 1)
    k_lanczos_stream(const __grid_constant__ StreamArgs A, const __grid_constant__ Coef<float> cf) {
    using P = Pk<float>;
    Shared<float> &S = sh<float>();
    const int tid = threadIdx.x, ncl = A.L.ncl, nz = A.L.nz, depth = A.depth;
    const StreamGeo<R> G(A);
    const bool scalar = tid == (int)blockDim.x - 32;
    // byte offsets in shared memory: the unit's rows in plane 0; bytes of a plane, of a row; the stages (u with
    // its halo rows, v_{k-1} likewise, V_loc)
    const int pb = A.L.plane * 4, rb = A.L.pitch * 4, mb = A.px * 4;
    const int o0 = shared_bytes<float>() + ((G.gy - G.y0 + kRadius) * A.L.pitch + 8 + G.gx) * 4;
    const int s0 = shared_bytes<float>() + 2 * pb + 64, su = (A.bh + 2 * kRadius) * mb, stb = 2 * su + A.bh * mb;
    // rows staged; planes before the first
    const int r0 = PER ? G.y0 - kRadius : max(0, G.y0 - kRadius), nrow = PER ? G.rows + 2 * kRadius : min(A.L.ny, G.y0 + A.bh + kRadius) - r0;
    constexpr int GH = PER ? kRadius : 0;
    // the unit's second row, if it lies outside the box: the first again, with factors 0
    const int uo = G.own ? (G.gy - r0) * mb + G.gx * 4 : 0, vo = 2 * su + (G.own ? (G.gy - G.y0) * mb + G.gx * 4 : 0);
    const int mb1 = G.row1 ? mb : 0;
    const float in1 = G.row1 ? 1.f : 0.f;
    // halo rows: units of one row by all threads that have points
    const int nhalo = PER || ncl > 1 ? 2 * kRadius * A.L.hw : 0, nthr = A.bh / R * A.L.hw;
    // unit e: its place in a stage (-1: outside the box) and in plane 0
    auto halo = [&](int e, int &from, int &to) {
        const int hr = e / A.L.hw, lr = hr < kRadius ? hr - kRadius : G.rows + hr - kRadius, y = G.y0 + lr;
        const int x = 4 * (e - hr * A.L.hw);
        from = e < nhalo && (PER || (y >= 0 && y < A.L.ny)) ? (y - r0) * mb + 4 * x : -1;
        to = shared_bytes<float>() + ((lr + kRadius) * A.L.pitch + 8 + x) * 4;
    };
    int h_from = -1, h_to = 0;                           // the thread's first
    if (tid < nthr) halo(tid, h_from, h_to);
    for (int e = tid; e < A.L.smem_words; e += blockDim.x)
        reinterpret_cast<int4 *>(lz_smem + shared_bytes<float>())[e] = make_int4(0, 0, 0, 0);
    if (scalar) {
        for (int q = 0; q < 2; ++q) mbar_init(&S.pbar[q]);
        for (int q = 0; q < kStages; ++q) mbar_init(&S.full[q]);
        S.gone = 0;
        S.tell = ncl;
        S.A.err = A.L.err;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    before_bulk();                                       // the zeros, before bulk copies into the same memory
    float *const U = A.L.ws + (size_t)(blockIdx.x / (unsigned)ncl) * A.L.ws_stride;
    float *const H = U + 4 * A.nv;                       // after u (two buffers) and the direction (re, im)
    const size_t pl = (size_t)A.L.ny * A.px;             // a plane in memory
    const int n_items = *A.L.cnt;
    unsigned ng = 0;
    Stages G4{0, 0u, true};
    P mask;                                              // 1 for points inside the box
#pragma unroll
    for (int i = 0; i < 4; ++i) mask.set(i, i < G.nvx ? 1.f : 0.f);
    cluster_barrier();
    for (;;) {
        if (G.rank == 0 && tid < ncl) {
            int it = 0;
            if (tid == 0) {
                if (*(volatile int *)A.L.err) fail_rest(A.L, n_items);   // no more
                it = atomicAdd(A.L.grab, 1);
            }
            it = __shfl_sync((1u << ncl) - 1u, it, 0);
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(
                             map_rank((unsigned)__cvta_generic_to_shared(&S.item[0]), tid)),
                         "r"(it)
                         : "memory");
        }
        cluster_barrier();
        if (S.item[0] >= n_items) break;
        const int s = A.L.list[n_items - 1 - S.item[0]];
        {
            float rr, ii, ri;
            stream_start<R>(&A, s, 0.f, 0.f, false, rr, ii, ri);
            gather3(rr, ii, ri, ng, ncl, G.rank, (int)blockDim.x);
            if (scalar) {
                float a, b, c;
                sum_parts(ng, ncl, a, b, c);
                start_state(a, b, c, A.L.d0 + A.L.slots[s].shift_re, A.L.slots[s].shift_im);
            }
            cluster_barrier();                           // and every block knows of a lost wait (start_part)
        }
        for (int pt = 0; pt < 2; ++pt) {
            float f_re, f_im;
            if (!start_part<float>(A.L, s, pt, scalar, ng, f_re, f_im)) continue;
            {
                float d0, d1, d2;
                stream_start<R>(&A, s, f_re, f_im, true, d0, d1, d2);
            }
            before_bulk();
            cluster_barrier();                           // u is stored in every band
            float ap = 0.f, ig = 1.f, cc = 0.f, dg = (float)S.F.d0;   // the first sweep: v_0 = u
            int k = 0, kb = 0, n = 0;
            bool have_p = false;
            for (;;) {
                // u alternates between two buffers: a band may be planes ahead of one that reads its rows
                const float *const ui = U + (size_t)(k & 1) * A.nv;
                float *const uout = U + (size_t)((k & 1) ^ 1) * A.nv + G.mem;
                const float *const vp = k == 0 ? U : H + (size_t)(k == kb ? A.L.hist - 1 : k - 1 - kb) * A.nv;
                float *const vk = H + (size_t)(k - kb) * A.nv + G.mem;
                auto issue = [&](int f, int q) {
                    const unsigned to = (unsigned)__cvta_generic_to_shared(lz_smem) + (unsigned)(s0 + q * stb);
                    if (PER) f = f < 0 ? f + nz : f >= nz ? f - nz : f;
                    expect_bytes(G4.bar(q), 2 * nrow * mb + G.rows * mb);
                    for (int i = 0; i < nrow;) {         // once, but for a periodic band at the box's edge
                        int y = r0 + i;
                        if (PER) y = y < 0 ? y + A.L.ny : y % A.L.ny;
                        const int m = PER ? min(nrow - i, A.L.ny - y) : nrow;
                        const size_t o = f * pl + (size_t)y * A.px;
                        bulk_load(to + i * mb, ui + o, m * mb, G4.bar(q));
                        bulk_load(to + su + i * mb, vp + o, m * mb, G4.bar(q));
                        i += m;
                    }
                    bulk_load(to + 2 * su, A.v + f * pl + (size_t)G.y0 * A.px, G.rows * mb, G4.bar(q));
                };
                if (scalar && G4.ok) {
                    before_bulk();
                    for (int i = 0, q = G4.st; i < min(depth, nz + 2 * GH); ++i, q = q + 1 == depth ? 0 : q + 1) issue(i - GH, q);
                }
                const float m_ag = -ap * ig, ig1 = ig * in1, m_ag1 = m_ag * in1;
                float *pu = uout, *pv = vk;              // planes f - 6 of u, f of v_k
                float2 svv = make_float2(0.f, 0.f), suv = svv, suu = svv;
                P acc[12][R];                            // sums of planes f-6 .. f+5
#pragma unroll
                for (int j = 0; j < 12; ++j)
#pragma unroll
                    for (int r = 0; r < R; ++r) acc[j][r].zero();
                // the next plane of u
                auto put_u = [&](const P (&u)[R]) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        P t = u[r];
                        t.mul(mask);
                        if (r) t.mul(in1);
                        if (r == 0 || G.row1) pk_store(pu + r * A.px, t);
#pragma unroll
                        for (int i = 0; i < 2; ++i) suu = __ffma2_rn(t.p[i], t.p[i], suu);
                    }
                    pu += pl;
                };
                for (int f = -GH; f < nz + GH; ++f) {
                    const bool real = !PER || (f >= 0 && f < nz);
                    const int sb = s0 + G4.st * stb, po = (f & 1) * pb;
                    int q0 = o0 + po;
                    asm volatile("" : "+r"(q0));
                    G4.wait(A.L.err);
                    P w[R], a[R];
                    if (G.own) {
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            a[r] = lds<float>(sb + su + uo + r * mb1);
                            w[r] = lds<float>(sb + uo + r * mb1);
                            w[r].mul(r ? ig1 : ig);
                            w[r].fma(r ? m_ag1 : m_ag, a[r]);
                            if (PER) {
                                if (!real) continue;
                                put<float, 1>(reinterpret_cast<float *>(lz_smem + q0), G.gx, G.nvx, A.L.nx, w[r]);
                            } else {
                                pk_store(reinterpret_cast<float *>(lz_smem + q0 + r * rb), w[r]);
                            }
                            if (r == 0 || G.row1) pk_store(pv + r * A.px, w[r]);
                            a[r].mul(-cc);
                            a[r].fma(lds<float>(sb + vo + r * mb1), w[r]);
                            a[r].fma(dg, w[r]);
                        }
                        if (real) pv += pl;
                    }
                    auto form_halo = [&](int from, int to) {
                        if (from < 0) return;
                        P h = lds<float>(sb + from);
                        h.mul(ig);
                        h.fma(m_ag, lds<float>(sb + su + from));
                        float *const at = reinterpret_cast<float *>(lz_smem + po + to);
                        const int x = from % mb / 4;
                        if (PER) put<float, 1>(at, x, min(4, A.L.nx - x), A.L.nx, h);
                        else pk_store(at, h);
                    };
                    if (real) form_halo(h_from, h_to);
                    if (tid < nthr && real)
                        for (int e = tid + nthr; e < nhalo; e += nthr) {   // bands of fewer than 24 rows
                            int from, to;
                            halo(e, from, to);
                            form_halo(from, to);
                        }
                    const int freed = G4.st;
                    G4.next(depth);
                    __syncthreads();                     // the plane is there, the stage is read
                    if (scalar && G4.ok && f + depth < nz + GH) issue(f + depth, freed);
                    if (!G.own) continue;
                    if (!real) {                         // its part along z alone
                        P u = acc[0][0];
                        u.fma(cf.a[6], w[0]);
#pragma unroll
                        for (int j = 1; j < 12; ++j) {
                            acc[j - 1][0] = acc[j][0];
                            if (j != 6) acc[j - 1][0].fma(cf.a[j < 6 ? 6 - j : j - 6], w[0]);
                        }
                        acc[11][0] = w[0];
                        acc[11][0].mul(cf.a[6]);
                        if (f >= nz) {
                            P t[R];
                            t[0] = u;
                            put_u(t);
                        }
                        continue;
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        P X[5];
#pragma unroll
                        for (int m = 0; m < 5; ++m) X[m] = m == 2 && !PER ? w[r] : lds<float>(q0 + r * rb + (m - 2) * 16);
                        x_part(a[r], X, cf);
                    }
                    if (R == 2) {
                        a[0].fma(cf.a[1], w[R - 1]);
                        a[R - 1].fma(cf.a[1], w[0]);
                    }
#pragma unroll
                    for (int d = 1; d <= kRadius; ++d) {
                        const P lo = lds<float>(q0 - d * rb), hi = lds<float>(q0 + (R - 1 + d) * rb);
                        a[0].fma(cf.a[d], lo);
                        a[R - 1].fma(cf.a[d], hi);
                        if (R == 2 && d < kRadius) {
                            a[R - 1].fma(cf.a[d + 1], lo);
                            a[0].fma(cf.a[d + 1], hi);
                        }
                    }
                    P u[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        // acc[6]: plane f's neighbours below; the ones above give w.(B w) the same again
                        P t = a[r];
                        t.fma(2.f, acc[6][r]);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            svv = __ffma2_rn(w[r].p[i], w[r].p[i], svv);
                            suv = __ffma2_rn(t.p[i], w[r].p[i], suv);
                        }
                        u[r] = acc[0][r];
                        u[r].fma(cf.a[6], w[r]);
#pragma unroll
                        for (int j = 1; j < 12; ++j) {
                            acc[j - 1][r] = acc[j][r];
                            if (j == 6) acc[j - 1][r].fma(1.f, a[r]);   // plane f
                            else acc[j - 1][r].fma(cf.a[j < 6 ? 6 - j : j - 6], w[r]);
                        }
                        acc[11][r] = w[r];
                        acc[11][r].mul(cf.a[6]);
                    }
                    if (f >= kRadius) put_u(u);
                }
                if (G.own && !PER)
#pragma unroll
                    for (int j = 0; j < kRadius; ++j) put_u(acc[j]);
                before_bulk();                           // u and v_k, for the next sweep's copies
                gather3(svv.x + svv.y, suv.x + suv.y, suu.x + suu.y, ng, ncl, G.rank, (int)blockDim.x);
                {
                    float a, b, c;
                    sum_parts(ng, ncl, a, b, c);
                    ap = b / a;
                    const float b2 = c - ap * b;
                    ig = b2 > 0.f ? 1.f / sqrtf(b2) : 0.f;
                    if (!isfinite(a) || !isfinite(c)) ig = nanf("");
                }
                ++k;
                if (scalar) {
                    S.F.ak = S.F.d0 - (double)dg + (double)ap;
                    S.F.ck = (double)cc;
                    S.F.ig = (double)ig;
                    factor<float>(0, k - 1 - kb, k, A.L.maxit);
                    if (!G4.ok) wait_lost<float>(ng);
                    if (A.L.prof && G.rank == 0) atomicAdd(A.L.prof + 1, (unsigned long long)A.L.nd);
                }
                cc = ig > 0.f ? 1.f / ig : 0.f;
                dg -= ap;
                cluster_barrier();                       // u and v_k of every band are written; the decision is taken
                n = k - kb;
                // (a vote: as a plain condition it costs the plane loop 8 registers and 2.5% of the call, and wait_lost with
                // the cluster's size as an argument 2% at 51 x 44 x 51)
                if (S.flag || __any_sync(0xffffffffu, left<float>(ng))) break;
                if (n == A.L.hist) {                     // the history is full: into x and p
                    G4 = stream_flush<R>(&A, s, n, true, have_p, pt ? -S.start[1] : S.start[0], pt ? S.start[0] : S.start[1], G4);
                    have_p = true;
                    kb = k;
                }
            }
            if (S.flag < 4)
                G4 = stream_flush<R>(&A, s, n, false, have_p, pt ? -S.start[1] : S.start[0], pt ? S.start[0] : S.start[1], G4);
            cluster_barrier();                           // no thread still reads the flag or this part's vectors
        }
        if (scalar && G.rank == 0) end_state(A.L, s);
    }
    if (!G4.ok) {                                        // planes that were asked for may still arrive: a second more
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000000LL) {}
    }
    cluster_barrier();
}

struct Variant {
    int zc, max_threads;
};
constexpr Variant kVar32[3] = {{3, 640}, {4, 640}, {5, 512}};
constexpr Variant kVar64[3] = {{2, 640}, {4, 640}, {8, 384}};

using Fn32 = void (*)(LanczosArgs<float>, Coef<float>);
using Fn64 = void (*)(LanczosArgs<double>, Coef<double>);
// by variant and MODE (FP64 has no rows of zeros: its arithmetic, not its loads, is the limit)
const Fn32 kFn32[3][2] = {{k_lanczos<float, 3, 640, 0>, k_lanczos<float, 3, 640, 1>},
                          {k_lanczos<float, 4, 640, 0>, k_lanczos<float, 4, 640, 1>},
                          {k_lanczos<float, 5, 512, 0>, k_lanczos<float, 5, 512, 1>}};
const Fn64 kFn64[3][2] = {{k_lanczos<double, 2, 640, 2>, k_lanczos<double, 2, 640, 1>},
                          {k_lanczos<double, 4, 640, 2>, k_lanczos<double, 4, 640, 1>},
                          {k_lanczos<double, 8, 384, 2>, k_lanczos<double, 8, 384, 1>}};

const void *stream_kernel(int rows, int threads, bool per) {
    return per ? (const void *)k_lanczos_stream<1, 512, true>
               : rows == 1 ? (const void *)k_lanczos_stream<1, 512, false>
                           : threads <= 256 ? (const void *)k_lanczos_stream<2, 256, false>
                                            : (const void *)k_lanczos_stream<2, 384, false>;
}

const void *kernel_of(bool mixed, int v, bool per) {
    return mixed ? (const void *)kFn32[v][per] : (const void *)kFn64[v][per];
}

void cluster_config(cudaLaunchConfig_t &lc, cudaLaunchAttribute &at, int ncl, int blocks, int threads, size_t smem,
                    cudaStream_t s) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)ncl;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    lc.gridDim = dim3((unsigned)blocks, 1, 1);
    lc.blockDim = dim3((unsigned)threads, 1, 1);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    lc.attrs = &at;
    lc.numAttrs = 1;
}

}  // namespace

// Bytes of a history buffer: `most` for a context by itself, the share (by systems) of four times that for a batch's
// (of twice that, a history of 113 vectors instead of 128 cost a batch of 29 x 34 x 26 .. 33 x 25 x 34, 177 solves, 1%).
static size_t history_budget(const Ctx &c, int nsys, size_t most) {
    if (c.batch_load <= nsys) return most;
    return std::min(most, (size_t)(4.0 * (double)most * nsys / c.batch_load));
}

// Plan of the streaming kernel: threads of one or two rows and 1 to 8 bands, of which a block's threads take every
// point and whose planes fit, two in flight at least.  A plane of a band of bh rows takes time as bh + 10 (its
// halo rows are only formed), three quarters of that for each of the blocks that share an SM (one waits
// where another computes), and never less than one step's latency, which is longer for two rows a thread.
// Measured, whole chi0 application in ms, with (rows, bands): 56^3, 256 systems (1, 2) 88, (1, 3) 108,
// (1, 4) 82.5, (1, 5) 93, (1, 6) 118, (2, 2) 83, (2, 3) 123, (2, 4) 134; 72^3, 256 systems (1, 3) 246, (1, 4) 264,
// (1, 6) 238, (2, 2) 213, (2, 3) 232, (2, 4) 289, (2, 6) 357.
static bool stream_plan(const Ctx &c, int nsys, int sms, int optin, LanczosPlan &p, double &cycles) {
    if (c.opt.prec != RPA_MIXED) return false;
    const bool per = c.opt.periodic != 0;
    const int hw = (c.nx + 3) / 4, px = 4 * hw;
    double best = 1e300;
    for (int q = 0; q < (per ? 8 : 16); ++q) {
        const int rows = 1 + q / 8, ncl = 1 + q % 8;
        const int bh = ((c.ny + ncl - 1) / ncl + 1) / 2 * 2;
        if (bh < 2 || (long long)bh * (ncl - 1) >= c.ny) continue;
        const long long units = (long long)hw * (bh / rows);
        const int threads = (int)std::min<long long>((units + 31) / 32 * 32 + 32, 1 << 20);
        if (threads > (rows == 1 ? 512 : 384)) continue;
        int p16 = per ? (16 + c.nx + 3) / 4 : 2 + hw;   // 16-byte words of a row: a unit's rows span hw of them modulo 8
        while ((rows * p16 - (hw + (rows == 2 ? hw % 2 : 0))) % 8 != 0) ++p16;
        const int pitch = 4 * p16, plane = pitch * (bh + 2 * kRadius);
        const size_t stage = sizeof(float) * (size_t)px * (3 * bh + 4 * kRadius);
        const size_t fixed = shared_bytes<float>() + sizeof(float) * (2 * (size_t)plane + 16);
        if (fixed + 2 * stage > (size_t)optin) continue;
        const int depth = (int)std::min<size_t>(kStages, ((size_t)optin - fixed) / stage);
        const size_t smem = fixed + depth * stage;
        const void *fn = stream_kernel(rows, threads, per);
        RPA_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        allow_dynamic_smem(fn, smem);
        cudaLaunchConfig_t lc{};
        cudaLaunchAttribute at{};
        cluster_config(lc, at, ncl, ncl * sms, threads, smem, nullptr);
        int ncs = 0;
        if (cudaOccupancyMaxActiveClusters(&ncs, fn, &lc) != cudaSuccess || ncs < 1) {
            (void)cudaGetLastError();
            continue;
        }
        const int all = std::max(nsys, c.batch_load);
        const double share = (double)std::min(ncs, all) * ncl / sms, load = (rows == 1 ? 1.0 : 0.92) * hw * (bh + 10);
        // cycles of a sweep (and what it costs at its end), times the rounds the systems take
        const double cost = (all <= ncs ? 1.0 : (double)all / ncs + 0.3) *
                            (20e3 + 5.4 * (c.nz + (per ? 8 : 0)) * std::max(rows == 1 ? 250.0 : 500.0, load * std::max(1.0, 0.75 * share)));
        if (cost >= best) continue;
        best = cost;
        p = LanczosPlan{};
        p.stream = 1;
        p.mixed = 1;
        p.ncl = ncl;
        p.clusters = std::min(ncs, nsys);
        p.threads = threads;
        p.smem = smem;
        p.hw = hw;
        p.pitch = pitch;
        p.plane = plane;
        p.bh = bh;
        p.depth = depth;
        p.unit_rows = rows;
    }
    if (best == 1e300) return false;
    cycles = best;
    const size_t nv = (size_t)c.nz * c.ny * px;
    // history: as many vectors as 8 GB hold, 16 .. kHistMax (a batch: its share of 32 GB, by systems)
    const size_t most = history_budget(c, nsys, (size_t)8 << 30);
    p.hist = (int)std::max<size_t>(16, std::min<size_t>(kHistMax, most / (nv * 4 * p.clusters)));
    p.ws_stride = nv * (4 + p.hist);
    p.ws_bytes = sizeof(float) * (p.ws_stride * p.clusters + nv);         // and V_loc
    return true;
}

bool lanczos_plan(const Ctx &c, int nsys, LanczosPlan &best) {
    if (c.opt.precondition || c.nz < kRadius + 2 || c.ny < kRadius || c.nx < kRadius) return false;
    const bool mixed = c.opt.prec == RPA_MIXED;
    int sms = 0, optin = 0;
    RPA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c.device));
    RPA_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c.device));
    const int W = mixed ? 4 : 2, pad = mixed ? 8 : 6;
    const size_t tsz = mixed ? 4 : 8;
    const int hw = (c.nx + W - 1) / W, hh = (c.ny + 1) / 2;
    // row pitch in 16-byte words: the row and its padding (periodic: images on both sides), and two rows
    // spanning hw words modulo 8 (odd hw: one more), so that 8 consecutive units hit different banks
    int p16 = c.opt.periodic ? (2 * pad + c.nx + W - 1) / W : (pad + hw * W) / W;
    if (mixed)
        while ((2 * p16 - (hw + hw % 2)) % 8 != 0) ++p16;
    // FP32, zero values outside the box: planes follow each other with kRadius rows of zeros in between
    const int zrows = c.opt.periodic || !mixed ? 0 : kRadius;
    const int pitch = p16 * W, plane = pitch * (c.ny + zrows), lead = std::max(W, pitch * zrows);
    const int nvar = 3;
    double best_cost = 1e300;
    bool found = false;
    for (int v = 0; v < nvar; ++v) {
        const Variant var = mixed ? kVar32[v] : kVar64[v];
        const void *fn = kernel_of(mixed, v, c.opt.periodic != 0);
        cudaFuncAttributes fa{};
        RPA_CUDA(cudaFuncGetAttributes(&fa, fn));
        for (int ncl = 1; ncl <= 16; ncl *= 2) {
            if (ncl > c.nz) break;
            const int nzl = (c.nz + ncl - 1) / ncl, nch = (nzl + var.zc - 1) / var.zc;
            const long long units = (long long)hw * hh * nch;
            const int threads = (int)std::min<long long>((units + 31) / 32 * 32 + kExtra, 1 << 20);
            if (threads > var.max_threads) continue;
            const size_t elems = (size_t)lead + (size_t)plane * (nch * var.zc + 2 * kRadius) + 2 * pad;
            const size_t smem = (elems * tsz + 15) / 16 * 16 + (mixed ? shared_bytes<float>() : shared_bytes<double>());
            if (smem + fa.sharedSizeBytes > (size_t)optin) continue;
            RPA_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            allow_dynamic_smem(fn, smem);
            cudaLaunchConfig_t lc{};
            cudaLaunchAttribute at{};
            cluster_config(lc, at, ncl, ncl * sms, threads, smem, nullptr);
            int ncs = 0;
            if (cudaOccupancyMaxActiveClusters(&ncs, fn, &lc) != cudaSuccess || ncs < 1) {
                (void)cudaGetLastError();
                continue;
            }
            // cycles per iteration of the blocks sharing an SM, and the rounds the systems take
            const double pts = (double)(threads - kExtra) * 2 * W * var.zc;
            // (a batch's other contexts run beside this one)
            const int used = std::min(ncs, nsys), all = std::max(nsys, c.batch_load), busy = std::min(ncs, all);
            const double share = std::max(1.0, (double)busy * ncl / sms);
            const double sync = 3500.0 + 300.0 * std::log2((double)ncl);
            const double cyc = std::max(share * pts * (mixed ? 0.6 : 24.0), pts * (mixed ? 0.6 : 24.0) + sync);
            const double rounds = all <= ncs ? 1.0 : (double)all / ncs + 0.3;
            const double cost = rounds * cyc;
            if (cost < best_cost) {
                best_cost = cost;
                found = true;
                best.variant = v;
                best.mixed = mixed;
                best.ncl = ncl;
                best.clusters = used;
                best.threads = threads;
                best.smem = smem;
                best.hw = hw;
                best.hh = hh;
                best.nch = nch;
                best.pitch = pitch;
                best.plane = plane;
                best.lead = lead;
                best.reach = (kRadius + c.nz / ncl - 1) / (c.nz / ncl);
                best.zc = var.zc;
            }
        }
    }
    // Clusters of 8 or 16 blocks leave SMs idle (15 and 7 are resident, of 19 and 9.5): with many systems the
    // streaming kernel is faster then.  An iteration on chip takes 1.5 times the cycles above.  Measured, chi0 in
    // ms, on chip and streaming: 44^3 32 systems 7.7, 15.4, 128 systems 23.7, 28.1, 256 systems 45.0, 40.7; 48^3
    // 11.0, 19.0; 38.1, 30.4; 73.3, 46.4; with four blocks, 40^3, 4096 systems 357, 429; with two, 32^3 175, 212.
    // Periodic (one row a thread, 16 blocks on chip): 44^3 16.4, 23.9; 59.3, 51.8; 114.9, 86.5; 48^3 16.1, 31.8; 57.9,
    // 58.2; 112.7, 96.8: the rule takes the dearer at 44^3 with 128 and at 48^3 with 256 systems (14 and 16%).
    LanczosPlan sp;
    double sc = 0.0;
    if (stream_plan(c, nsys, sms, optin, sp, sc) && (!found || sc < 0.93 * 1.5 * best_cost)) {
        best = sp;
        return true;
    }
    if (!found) return false;
    best.stream = 0;
    const size_t vec = (size_t)2 * best.zc * (best.threads - kExtra) * W, hvec = (size_t)best.nch * best.zc * best.plane;
    // history: as many vectors as 2 GB hold in each of its two buffers, 16 .. kHistMax (a batch: its share of 8 GB)
    const size_t per_vec = hvec * tsz * best.clusters * best.ncl;
    best.hist = (int)std::max<size_t>(16, std::min<size_t>(kHistMax, history_budget(c, nsys, (size_t)2 << 30) / per_vec));
    best.ws_stride = vec + 2 * hvec + 2 * hvec * best.hist;
    best.ws_bytes = best.ws_stride * tsz * best.clusters * best.ncl;
    return true;
}

template <typename T> static void fill_args(const Ctx &c, const LanczosPlan &p, LanczosArgs<T> &a) {
    a.ws = (T *)p.ws;
    a.ws_stride = p.ws_stride;
    a.nd = c.nd;
    a.nx = c.nx;
    a.ny = c.ny;
    a.nz = c.nz;
    a.tol = c.opt.tol;
    a.inner_tol = c.opt.inner_tol;
    a.maxit = c.opt.maxit;
    a.mixed = p.mixed;
    a.ncl = p.ncl;
    a.hw = p.hw;
    a.hh = p.hh;
    a.nch = p.nch;
    a.pitch = p.pitch;
    a.plane = p.plane;
    a.lead = p.lead;
    a.err = c.d_tc_err;
    a.reach = p.reach;
    a.hist = p.hist;
    a.smem_words = (int)((p.smem - shared_bytes<T>()) / 16);
    a.d0 = 3.0 * c.coef.a[0];
}

template <typename T> static void launch(const Ctx &c, const LanczosPlan &p, LanczosArgs<T> a, cudaStream_t s) {
    fill_args(c, p, a);
    const Coef<T> cf = cast_coef<T>(c.coef);
    const void *fn = kernel_of(p.mixed, p.variant, c.opt.periodic != 0);
    allow_dynamic_smem(fn, p.smem);
    RPA_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t lc{};
    cudaLaunchAttribute at{};
    cluster_config(lc, at, p.ncl, p.ncl * p.clusters, p.threads, p.smem, s);
    void *args[2] = {(void *)&a, (void *)&cf};
    RPA_CUDA(cudaLaunchKernelExC(&lc, fn, args));
}

void lanczos_prepare(const Ctx &c, const LanczosPlan &p, cudaStream_t s) {
    if (!p.stream) return;
    const size_t nv = (size_t)c.nz * c.ny * 4 * p.hw;
    k_pad_rows<<<(unsigned)std::min<size_t>((nv + 255) / 256, 2048), 256, 0, s>>>(
        c.vloc32, (float *)p.ws + p.ws_stride * p.clusters, c.nx, 4 * p.hw, (long long)c.nz * c.ny);
    RPA_LAUNCH("V_loc rows");
    count_launches(1);
}

void lanczos_launch(const Ctx &c, const LanczosPlan &p, const LanczosArgs<float> &args, cudaStream_t s) {
    if (!p.stream) {
        launch(c, p, args, s);
        return;
    }
    StreamArgs a{};
    a.L = args;
    fill_args(c, p, a.L);
    a.px = 4 * p.hw;
    a.nv = (size_t)c.nz * c.ny * a.px;
    a.v = (const float *)p.ws + p.ws_stride * p.clusters;
    a.bh = p.bh;
    a.depth = p.depth;
    const Coef<float> cf = cast_coef<float>(c.coef);
    const void *fn = stream_kernel(p.unit_rows, p.threads, c.opt.periodic != 0);
    allow_dynamic_smem(fn, p.smem);
    cudaLaunchConfig_t lc{};
    cudaLaunchAttribute at{};
    cluster_config(lc, at, p.ncl, p.ncl * p.clusters, p.threads, p.smem, s);
    void *kargs[2] = {(void *)&a, (void *)&cf};
    RPA_CUDA(cudaLaunchKernelExC(&lc, fn, kargs));
}
void lanczos_launch(const Ctx &c, const LanczosPlan &p, const LanczosArgs<double> &a, cudaStream_t s) { launch(c, p, a, s); }

}  // namespace rpa
