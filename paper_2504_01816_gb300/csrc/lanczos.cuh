// The Lanczos kernel of the Sternheimer inner solves (lanczos.cu): its plan and launch.
#pragma once

#include "slots.cuh"

namespace rpa {

template <typename T> struct LanczosArgs {
    Slot *slots;
    const int *list, *cnt;         // slots whose inner solve runs, and their number
    int *grab;                     // systems taken so far (zero at the launch)
    const typename Cx<T>::t *r;    // right-hand sides of the inner solves [S][nd]
    typename Cx<T>::t *x;          // solutions, added to [S][nd]
    const T *vloc;
    unsigned long long *prof;      // [1] grid points processed (nullptr = off)
    // filled in by lanczos_launch
    T *ws;
    size_t ws_stride;
    long long nd;
    int nx, ny, nz;
    double tol, inner_tol;
    int maxit, mixed;
    int ncl, hw, hh, nch, pitch, plane, lead, reach, hist, smem_words;
    int *err;                      // set on a timed-out wait
    double d0;                     // 3 a_0
};

// Plan for nsys systems of this context; false where the grid neither fits on chip nor streams (fewer than 6 points
// along x or y or 8 along z, planes too wide for the streaming kernel, or FP64) and the COCG kernels run instead.
bool lanczos_plan(const Ctx &c, int nsys, LanczosPlan &p);
// Once a queue, before its launches (p.ws set).
void lanczos_prepare(const Ctx &c, const LanczosPlan &p, cudaStream_t s);
void lanczos_launch(const Ctx &c, const LanczosPlan &p, const LanczosArgs<float> &a, cudaStream_t s);
void lanczos_launch(const Ctx &c, const LanczosPlan &p, const LanczosArgs<double> &a, cudaStream_t s);

}  // namespace rpa
