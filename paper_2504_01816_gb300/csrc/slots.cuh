// Slots of the Sternheimer queue and the stencil coefficients, shared by the COCG kernels (cocg.cu)
// and the Lanczos kernel (lanczos.cu).
#pragma once

#include "internal.cuh"

namespace rpa {

enum Phase : int { kEmpty = 0, kInner = 1, kInnerDone = 2, kFinished = 3, kLoading = 4 };

struct Slot {
    double rho_re[2], rho_im[2];    // r^T r of the last two iterations (by parity of the iteration)
    double alpha_re, alpha_im, beta_re, beta_im;
    double shift_re, shift_im;
    double bnorm, ref_norm, rnorm;  // ||b||; inner solve: norms of the scaled FP32 residual
    double scale;                   // mixed: the FP32 inner solve works on scale * (b - A x64)
    int phase, sys, n, j;
    int iters, total_iters, refines, status;
    int discard;                    // mixed: the inner solve went non-finite; its correction is dropped
    int nearbreak;                  // mixed: inner solves ended at a near-breakdown
};

template <typename T> struct Cx;
template <> struct Cx<float> { using t = float2; };
template <> struct Cx<double> { using t = double2; };

template <typename T> struct Coef {
    T a[kRadius + 1];
};

template <typename T> Coef<T> cast_coef(const StencilCoef &c) {
    Coef<T> r;
    for (int k = 0; k <= kRadius; ++k) r.a[k] = (T)c.a[k];
    return r;
}

}  // namespace rpa
