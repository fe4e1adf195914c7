// Dense contractions of the subspace step on the 5th-generation tensor cores (tcgen05, sm_103a):
//
//     D[m][n] = sum_k A(m, k) B(n, k),   A(m, k) = A[m * a_m + k * a_k],  B(n, k) = B[n * b_n + k * b_k]
//
// for FP64 operands, as BF16 tensor-core products that are exact.  The scheme is the error-free
// splitting of Ozaki, Ogita and Oishi (error-free transformation of matrix products into sums of
// products of low-precision pieces) with per-chunk power-of-two scaling:
//
//   * k is walked in chunks of kTcK = 64.  Within a chunk every row m of A gets the power of two
//     s_m = 2^(e_m + 1) above its largest |A(m, k)| (e_m its binary exponent), every row n of B
//     likewise s_n, so that |A(m, k) / s_m| < 1.
//   * |x| = |A(m, k)| / s_m * 2^7 <= 128 is rounded to 2^-24 and cut into four balanced integer
//     digits, read off the bits of the FP64 significand with integer instructions:
//       |x| = a1 + 2^-8 a2 + 2^-16 a3 + 2^-24 a4 + r,  0 <= a1 <= 128, |a2..a4| <= 128, |r| <= 2^-25,
//     each times the sign of A(m, k) and exactly representable in BF16 (8 significant bits).
//   * Products a_i b_j are integers of magnitude at most 2^14, so over one chunk (64 values of k)
//     every partial sum the tensor core forms -- inside one MMA of 16 k values, or accumulated over
//     the chunk's four MMAs -- is an integer below 2^24 (the largest tile, L3, sums at most 256
//     products: below 2^22) and therefore exact in its FP32 accumulator, whatever the rounding of
//     the hardware's additions.  The ten products of weight 2^0 .. 2^-24 go to four tensor-memory tiles by weight:
//     L0 = a1.b1; L1 = a1.b2 + a2.b1; L2 = a1.b3 + a3.b1 + a2.b2; L3 = a1.b4 + a4.b1 + a2.b3 + a3.b2.
//   * After each chunk the tiles are read back (tcgen05.ld), combined exactly in 64-bit integers
//     as 2^24 L0 + 2^16 L1 + 2^8 L2 + L3, and the chunk's contribution s_m s_n 2^-38 times that
//     integer is added in FP64 (one conversion and one multiply-add per output and chunk).
// The only errors are the truncated remainders and the neglected products (weights 2^-31 and
// below, relative to s_m s_n) and the FP64 additions: about 1e-9 of the chunk-row maxima.
//
// Used for the projection C = V^T R of the Rayleigh-Ritz step (Algorithm 1), the P_c coefficients
// T_{k,(n,j)} = u_k . (u_n (.) nu^1/2 v_j) of the Sternheimer right-hand sides (Eqs. 7-9), and the
// per-axis transforms of the Kronecker-product Coulomb operator (Eq. 5), in the mixed-precision form.
//
// Blocking.  A block computes one 128 x kTcN tile of D over one range of k (split-K, blockIdx.z).  Per
// chunk a warp takes 8 rows of an operand at a time: lane l holds 16 values of row l % 8 (two groups
// of 8 consecutive k), the row's exponent is a maximum over four lanes (two shuffles), and the pieces
// go to shared memory as 16-byte stores, 8 lanes to the 8 rows of a core matrix, in the canonical K-major
// layout without swizzle (8-row x 16-byte core matrices, 128 bytes each): every value is loaded once and
// nothing is exchanged between warps before the tiles are complete.  One thread issues 4 (k slices of
// 16) x 10 (products) MMAs and commits them to an mbarrier, which every thread waits on before the
// tiles are read back and the shared tiles rewritten.  The FP64 tile goes to the output or to a
// split-K partial; a second kernel adds the partials in a fixed order (deterministic).  An operand row
// may be the product of two arrays' rows (the pairs u_n (.) dv_j), formed as it is loaded.
//
// What bounds it: the instructions that cut the pieces and the FP64 pipe that combines them (two
// conversions and a multiply-add per output and chunk); rows and columns past the operands cost
// nothing.  Measured at 40^3, 64 columns: a per-axis transform 200 -> 85 us (loading every value
// twice, shared-memory atomics for the exponents, 2-byte stores), the P_c coefficients of 16 x 64
// pairs 4.5 -> 0.72 ms (one contraction per orbital, 64 of 128 rows used).
//
// Bounded waits: every wait on the mbarrier gives up after ~1 s of clock cycles, sets the error
// flag, waits (again bounded) for the block's MMAs, frees the tensor memory and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "internal.cuh"

namespace rpa {

namespace {

constexpr int kTcM = 128;                // tile rows (MMA M)
constexpr int kTcN = 64;                 // tile columns (MMA N)
constexpr int kTcK = 64;                 // k chunk staged per round
constexpr int kTcThreads = 256;
constexpr int kTcPieces = 4;             // integer pieces per operand value
constexpr int kTcLevels = 4;             // product weights 2^0, 2^-8, 2^-16, 2^-24
constexpr uint32_t kTcCoreBytes = 128;   // one 8 x 16-byte core matrix
constexpr uint32_t kTcSbo = (kTcK / 8) * kTcCoreBytes;            // next 8-row group
constexpr uint32_t kTcLbo = kTcCoreBytes;                         // next 8 k values
constexpr uint32_t kTcTileA = kTcM * kTcK * 2;                    // bytes of one BF16 A tile
constexpr uint32_t kTcTileB = kTcN * kTcK * 2;
constexpr uint32_t kTcSmem = kTcPieces * (kTcTileA + kTcTileB) + 64;
constexpr long long kTcWaitCycles = 2000000000LL;                 // ~1 s at 2 GHz

// Operand rows: X(r, k) = p[(r / mi) mo + (r % mi) ms + k ks], times q[(r / mi) qmo + (r % mi) qms + k ks] if q is set.
struct TcRows {
    const double *p, *q;
    long long mo, ms, qmo, qms, ks;
    int mi;
};
struct TcArgs {
    TcRows A, B;
    int M, N;                            // output size
    long long K;
    long long kchunk;                    // k range per split (multiple of kTcK)
    double *D;                           // split-K: partials [splits][M][N]; else the output
    int lines;                           // != 0: no split; D[(m / di) do_ + (m % di) dm + n dn]
    long long do_, dm, dn;
    int di;
    const double *scale;                 // lines only: times scale[(m % di) dm + n dn] (nullptr = none)
    int *err;                            // set on a timed-out wait
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor: K-major canonical layout without swizzle.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((kTcLbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((kTcSbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;              // descriptor version of the 5th-generation tensor cores
    return d;                            // base offset 0, swizzle mode 0 (none)
}

// Instruction descriptor of kind::f16: D in FP32, A and B in BF16, both K-major, M x N.
constexpr uint32_t tc_idesc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Biased binary exponent field of |x| (0 for zero).
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// The four BF16 pieces of x for the row exponent field e (see above), from the significand bits:
// I = round(|x| / 2^(e - 1022) * 2^31) = round(significand / 2^(22 + e - e_x)), then balanced base-256
// digits I = a1 2^24 + a2 2^16 + a3 2^8 + a4 with a2..a4 in [-128, 127] and 0 <= a1 <= 128 (balanced
// digits keep the neglected products unbiased).  An integer of magnitude <= 256 converts to FP32
// exactly with no bits below the top 8 of its significand, so the upper half of its FP32 pattern
// is the same value in BF16.
__device__ __forceinline__ void cut4(double x, int e, __nv_bfloat16 (&p)[4]) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7FF);
    const int sh = 22 + e - ex;
    long long I = 0;
    if (ex > 0 && sh < 64)
        I = (long long)((((bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) + (1ull << (sh - 1))) >> sh);
    int dg[4];
#pragma unroll
    for (int i = 3; i >= 1; --i) {
        dg[i] = (int)(((I + 128) & 255) - 128);
        I = (I - dg[i]) >> 8;
    }
    dg[0] = (int)I;
    const unsigned short sx = (unsigned short)((bits >> 48) & 0x8000u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const unsigned int v = (unsigned int)abs(dg[i]);
        const unsigned short h = (unsigned short)(__float_as_uint(__uint2float_rn(v)) >> 16);
        const unsigned short sg = dg[i] < 0 ? (unsigned short)(sx ^ 0x8000u) : sx;
        p[i] = __ushort_as_bfloat16(v ? (unsigned short)(h | sg) : (unsigned short)0);
    }
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > kTcWaitCycles) return false;
    }
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

// Rows 8 g .. 8 g + 7 of an operand's tile, by one warp: row exponents and integer pieces of the 64 values from
// k = kb on (zeros from k1 on and for rows past the operand).
__device__ __forceinline__ void tc_stage(const TcRows &X, int r0, int rows, int g, long long kb, long long k1,
                                         unsigned char *tile, uint32_t tile_bytes, int *ex) {
    const int lane = threadIdx.x & 31, lr = 8 * g + (lane & 7), kg = lane >> 3, r = r0 + lr;
    double x[2][8];
    int e = 0;
    const bool in = r < rows;
    const int hi = in ? r / X.mi : 0, lo = in ? r - hi * X.mi : 0;
    const double *p = X.p + hi * X.mo + lo * X.ms, *q = X.q ? X.q + hi * X.qmo + lo * X.qms : nullptr;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const long long k = kb + 8 * (kg + 4 * h) + i;
            x[h][i] = in && k < k1 ? p[k * X.ks] : 0.0;
        }
    if (q) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const long long k = kb + 8 * (kg + 4 * h) + i;
                if (in && k < k1) x[h][i] *= q[k * X.ks];
            }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 8; ++i) e = max(e, exp_field(x[h][i]));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 8));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
    if (lane < 8) ex[lr] = e;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t w[kTcPieces][4];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            __nv_bfloat16 a[4], b[4];
            cut4(x[h][i], e, a);
            cut4(x[h][i + 1], e, b);
#pragma unroll
            for (int c = 0; c < kTcPieces; ++c)
                w[c][i >> 1] = (uint32_t)__bfloat16_as_ushort(a[c]) | ((uint32_t)__bfloat16_as_ushort(b[c]) << 16);
        }
        const uint32_t o = (uint32_t)g * kTcSbo + (uint32_t)(kg + 4 * h) * kTcCoreBytes + (uint32_t)(lane & 7) * 16u;
#pragma unroll
        for (int c = 0; c < kTcPieces; ++c)
            *reinterpret_cast<uint4 *>(tile + c * tile_bytes + o) = make_uint4(w[c][0], w[c][1], w[c][2], w[c][3]);
    }
}

__global__ void __launch_bounds__(kTcThreads, 2) k_tc_gemm(const __grid_constant__ TcArgs a) {
    extern __shared__ __align__(1024) unsigned char tsm[];
    unsigned char *tA = tsm;                                       // [4][kTcTileA]
    unsigned char *tB = tsm + kTcPieces * kTcTileA;                // [4][kTcTileB]
    uint64_t *bar = reinterpret_cast<uint64_t *>(tsm + kTcPieces * (kTcTileA + kTcTileB));
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + 1);
    __shared__ int abort_flag;
    __shared__ int expA[kTcM], expB[kTcN];                         // row exponents of the chunk
    const int tid = threadIdx.x, warp = tid >> 5;
    const int m0 = blockIdx.x * kTcM, n0 = blockIdx.y * kTcN;
    const long long k0 = (long long)blockIdx.z * a.kchunk;
    const long long k1 = min(a.K, k0 + a.kchunk);
    const uint32_t bar_addr = smem_u32(bar);
    constexpr uint32_t kCols = kTcLevels * kTcN;                  // one accumulator tile per weight
    // groups of 8 rows with values; the tiles' other rows stay zero
    const int ga = (min(kTcM, a.M - m0) + 7) / 8, gb = (min(kTcN, a.N - n0) + 7) / 8;
    for (uint32_t e = tid; e < kTcPieces * (kTcTileA + kTcTileB) / 16; e += kTcThreads)
        reinterpret_cast<uint4 *>(tsm)[e] = make_uint4(0, 0, 0, 0);
    for (int e = tid; e < kTcM; e += kTcThreads) expA[e] = 0;
    for (int e = tid; e < kTcN; e += kTcThreads) expB[e] = 0;

    if (tid == 0) {
        abort_flag = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_addr) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    // epilogue mapping: warp w reads tile rows 32 (w % 4) .. +31 (its tensor-memory lanes) and
    // columns 32 (w / 4) .. +31
    const int lane_base = 32 * (warp & 3), col0 = 32 * (warp >> 2);
    const int my_row = lane_base + (tid & 31);
    const uint32_t t_base = tmem + ((uint32_t)lane_base << 16) + (uint32_t)col0;
    // a warp whose rows or columns all lie past the output reads nothing back
    const int my_cols = m0 + lane_base < a.M ? max(0, min(32, a.N - n0 - col0)) : 0;
    double acc[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) acc[c] = 0.0;

    uint32_t phase = 0;
    bool ok = true, pending = false;
    for (long long kb = k0; kb < k1; kb += kTcK) {
        // 1. row exponents and integer pieces into the K-major core-matrix tiles
        for (int g = warp; g < ga + gb; g += kTcThreads / 32) {
            if (g < ga) tc_stage(a.A, m0, a.M, g, kb, k1, tA, kTcTileA, expA);
            else tc_stage(a.B, n0, a.N, g - ga, kb, k1, tB, kTcTileB, expB);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> tensor core
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr uint32_t idesc = tc_idesc(kTcM, kTcN);
            // (A piece, B piece, weight level) of the ten products a_i b_j with i + j <= 5
            constexpr int np = 10;
            const int pa[np] = {0, 0, 1, 0, 2, 1, 0, 3, 1, 2};
            const int pb[np] = {0, 1, 0, 2, 0, 1, 3, 0, 2, 1};
            const int lv[np] = {0, 1, 1, 2, 2, 2, 3, 3, 3, 3};
#pragma unroll
            for (int t = 0; t < kTcK / 16; ++t)
#pragma unroll
                for (int pr = 0; pr < np; ++pr) {
                    const uint64_t da = tc_desc(smem_u32(tA + pa[pr] * kTcTileA) + t * 2 * kTcCoreBytes);
                    const uint64_t db = tc_desc(smem_u32(tB + pb[pr] * kTcTileB) + t * 2 * kTcCoreBytes);
                    const uint32_t d = tmem + (uint32_t)(lv[pr] * kTcN);
                    // each chunk starts every level's tile afresh with its first product
                    const bool first = t == 0 && (pr == 0 || pr == 1 || pr == 3 || pr == 6);
                    const uint32_t accum = first ? 0u : 1u;
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                        "l"(da), "l"(db), "r"(idesc), "r"(accum)
                        : "memory");
                }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_addr)
                         : "memory");
        }
        pending = true;
        if (!mbar_wait(bar_addr, phase)) {
            ok = false;
            atomicExch(&abort_flag, 1);
        }
        phase ^= 1u;
        __syncthreads();
        if (abort_flag) break;
        pending = false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // 2. read the four weight tiles back (8 columns at a time) and add the chunk in FP64
        const int ea = expA[my_row];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (8 * h >= my_cols) break;                           // uniform per warp
            uint32_t l0[8], l1[8], l2[8], l3[8];
            tmem_ld8(t_base + 8 * h, l0);
            tmem_ld8(t_base + kTcN + 8 * h, l1);
            tmem_ld8(t_base + 2 * kTcN + 8 * h, l2);
            tmem_ld8(t_base + 3 * kTcN + 8 * h, l3);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int eb = expB[col0 + 8 * h + c];
                // the tiles hold integers below 2^24: exact in int64 as 2^24 L0 + 2^16 L1 + 2^8 L2 + L3
                const long long v = ((long long)__float2int_rn(__uint_as_float(l0[c])) << 24) +
                                    ((long long)__float2int_rn(__uint_as_float(l1[c])) << 16) +
                                    ((long long)__float2int_rn(__uint_as_float(l2[c])) << 8) +
                                    (long long)__float2int_rn(__uint_as_float(l3[c]));
                // s_m s_n 2^-38 = 2^(ea - 1022 + eb - 1022 - 38); zero rows have exponent field 0
                // (a scale below the normal range -- rows of magnitude ~1e-150 -- counts as zero)
                const double sc = (ea == 0 || eb == 0 || ea + eb < 1060) ? 0.0
                                                                          : __hiloint2double((ea + eb - 1059) << 20, 0);
                acc[8 * h + c] = fma(sc, (double)v, acc[8 * h + c]);
            }
        }
        // the next chunk's MMAs rewrite tensor memory and its loads the shared tiles and exponents
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    if (ok && !abort_flag) {
        const int m = m0 + my_row;
        if (m < a.M) {
            if (a.lines) {
                const int hi = m / a.di;
                const long long in = (m - hi * a.di) * a.dm, off = hi * a.do_ + in;
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const int n = n0 + col0 + c;
                    if (n < a.N) a.D[off + n * a.dn] = a.scale ? acc[c] * a.scale[in + n * a.dn] : acc[c];
                }
            } else {
                double *out = a.D + ((long long)blockIdx.z * a.M + m) * a.N;
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const int n = n0 + col0 + c;
                    if (n < a.N) out[n] = acc[c];
                }
            }
        }
    } else if (tid == 0) {
        atomicExch(a.err, 1);
        if (pending) (void)mbar_wait(bar_addr, phase ^ 1u);          // let the block's MMAs finish
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

__global__ void k_tc_sum_splits(const double *__restrict__ part, int splits, long long n, double *__restrict__ D) {
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        double s = 0.0;
        int z = 0;
        for (; z + 16 <= splits; z += 16) {              // 16 loads in flight, added in order
            double v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = part[(long long)(z + i) * n + e];
#pragma unroll
            for (int i = 0; i < 16; ++i) s += v[i];
        }
        for (; z < splits; ++z) s += part[(long long)z * n + e];
        D[e] = s;
    }
}

inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

}  // namespace

// D (M x N, row-major) over split ranges of k, as if the rows came ref_rows at a time (which sets the ranges).
static void tc_split(TcArgs a, int ref_rows, double *D, cudaStream_t s, DevBuf &scratch) {
    const int tm = (int)cdiv(a.M, kTcM), tn = (int)cdiv(a.N, kTcN), rm = (int)cdiv(ref_rows, kTcM);
    int dev = 0, sms = 0;
    RPA_CUDA(cudaGetDevice(&dev));
    RPA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // split K so that the grid covers the SMs about three times, with at least two chunks per split
    long long splits = std::max(1LL, std::min<long long>(a.K / (2 * kTcK), (3LL * sms + rm * tn - 1) / (rm * tn)));
    a.kchunk = ((a.K + splits - 1) / splits + kTcK - 1) / kTcK * kTcK;
    splits = std::max(1LL, (a.K + a.kchunk - 1) / a.kchunk);
    a.D = (double *)scratch.ensure(sizeof(double) * (size_t)splits * a.M * a.N);
    allow_dynamic_smem((const void *)k_tc_gemm, kTcSmem);
    k_tc_gemm<<<dim3(tm, tn, (unsigned)splits), kTcThreads, kTcSmem, s>>>(a);
    const long long n = (long long)a.M * a.N;
    k_tc_sum_splits<<<std::min<unsigned>(cdiv(n, 64), 4096u), 64, 0, s>>>(a.D, (int)splits, n, D);
    RPA_LAUNCH("tensor-core contraction");
    count_launches(2);
}

void tc_gemm(const double *A, long long a_m, const double *B, long long b_n, int M, int N, long long K, double *D,
             cudaStream_t s, DevBuf &scratch, int *err_dev) {
    if (M <= 0 || N <= 0) return;
    TcArgs a{};
    a.A = TcRows{A, nullptr, 0, a_m, 0, 0, 1, M};
    a.B = TcRows{B, nullptr, 0, b_n, 0, 0, 1, N};
    a.M = M;
    a.N = N;
    a.K = K;
    a.err = err_dev;
    tc_split(a, M, D, s, scratch);
}

void tc_gemm_pairs(const double *U, int nu, const double *V, int nv, const double *B, int N, long long K, double *D,
                   cudaStream_t s, DevBuf &scratch, int *err_dev) {
    if (nu <= 0 || nv <= 0 || N <= 0) return;
    const size_t limit = (size_t)256 << 20;              // bytes of partials: orbitals are taken in groups
    const size_t per = sizeof(double) * (size_t)nv * N * 512;
    const int step = (int)std::max<size_t>(1, std::min<size_t>(nu, limit / per));
    for (int n = 0; n < nu; n += step) {
        const int m = std::min(step, nu - n);
        TcArgs a{};
        a.A = TcRows{U + (size_t)n * K, V, K, 0, 0, K, 1, nv};
        a.B = TcRows{B, nullptr, 0, K, 0, 0, 1, N};
        a.M = m * nv;
        a.N = N;
        a.K = K;
        a.err = err_dev;
        tc_split(a, nv, D + (size_t)n * nv * N, s, scratch);
    }
}

void tc_lines(const double *in, double *out, long long rows, int mi, long long mo, long long ms, long long ks, int n,
              const double *Q, long long q_n, long long q_k, const double *scale, cudaStream_t s, int *err_dev) {
    // whole groups of mi lines per launch, the line index in 32 bits
    const long long per = std::max<long long>(1, (1LL << 30) / mi) * mi;
    for (long long r = 0; r < rows; r += per) {
        TcArgs a{};
        const double *x = in + r / mi * mo;
        a.A = TcRows{x, nullptr, mo, ms, 0, 0, ks, mi};
        a.B = TcRows{Q, nullptr, 0, q_n, 0, 0, q_k, n};
        a.M = (int)std::min(per, rows - r);
        a.N = n;
        a.K = n;
        a.kchunk = n;
        a.D = out + r / mi * mo;
        a.lines = 1;
        a.di = mi;
        a.do_ = mo;
        a.dm = ms;
        a.dn = ks;
        a.scale = scale;
        a.err = err_dev;
        allow_dynamic_smem((const void *)k_tc_gemm, kTcSmem);
        k_tc_gemm<<<dim3(cdiv(a.M, kTcM), cdiv(n, kTcN), 1), kTcThreads, kTcSmem, s>>>(a);
        RPA_LAUNCH("tensor-core transform");
        count_launches(1);
    }
}

}  // namespace rpa
