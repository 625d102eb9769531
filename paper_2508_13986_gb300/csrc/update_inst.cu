// Instantiations of the flux-update kernels and of the step-loop kernels for one
// precision and dimension (the drift model is a run-time parameter: velocities
// are evaluated once per cell). The build compiles this file once per
// (GBEES_PREC, GBEES_DIM) pair so that the instantiations compile in parallel:
//   GBEES_PREC   64 (FP64) or 32 (FP32 storage and fluxes)
//   GBEES_DIM    1..6
#include "gbees_persistent.cuh"

#ifndef GBEES_PREC
#error "GBEES_PREC must be 32 or 64"
#endif
#ifndef GBEES_DIM
#error "GBEES_DIM must be 1..6"
#endif

namespace gbees {

#if GBEES_PREC == 64
using Real = double;
#else
using Real = float;
#endif

#define GBEES_JOIN2(a, b) a##b
#define GBEES_JOIN(a, b) GBEES_JOIN2(a, b)
#define GBEES_ENTRY GBEES_JOIN(GBEES_JOIN(update_kernels_p, GBEES_PREC), GBEES_JOIN(_n, GBEES_DIM))

// pre: the kernels before the link phase (grow, halo); post: after it (all
// take (Model, Bufs)).
void GBEES_ENTRY(Kernels* k) {
    constexpr int N = GBEES_DIM;
    k->persist = (void*)k_persistent<N, Real>;
    k->batch = (void*)k_batch<N, Real>;
    k->pre[0] = (void*)k_grow_mark<Real>;
    k->pre[1] = (void*)k_grow_list<N, Real>;
    k->pre[2] = (void*)k_halo<N, Real, 1>;
    k->npre = 3;
    k->post[0] = (void*)k_waves<N, Real>;
#if GBEES_PREC == 64
    k->post[1] = (void*)k_faces<N, Real>;
    k->post[2] = (void*)k_apply<N, Real>;
    k->npost = 3;
#else
    k->post[1] = (void*)k_update<N, Real>;
    k->npost = 2;
#endif
}

}  // namespace gbees
