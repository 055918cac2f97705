// Sums that the next kernel takes over (small lattices).
//
// There every launch lasts a few microseconds, and a reduction that ends in
// its own kernel costs as much again: partial, fence, ticket, and the last
// block's loads one after the other (at 8^4 the M Dslash took 8.5 us with the
// ticket and takes 4.6 without).  The M Dslash leaves its block partials of
// <p, Ap> instead, and each block of the next kernel sums them for itself, in
// the same order, so all blocks get the same alpha.
#pragma once
#include "cg_state.cuh"
#include "reduce.cuh"

namespace stag {

// the M Dslash's partials of <p, Ap>; n = 0: alpha is in the scalars already
struct PapPartials {
    const double *v = nullptr;
    int n = 0;
};

// sum of n partials, valid in every thread
template <int BLOCK> STAG_D double sum_partials(const double *__restrict__ v, int n, double *smem) {
    __shared__ double all;
    const double t = block_sum<BLOCK>(partials_share<BLOCK>(v, n), smem);
    if (threadIdx.x == 0)
        all = t;
    __syncthreads();
    return all;
}

// alpha = rr / <p, Ap> of this iteration and the solve's status with the
// breakdown test on <p, Ap> applied, in every thread; block 0 also stores pAp
// and alpha, which no block of the kernel may read from the scalars then (nor
// write rr or status before every block has called this).  Without partials
// (SMALL false: the kernels of larger lattices, which the sum's registers
// would cost occupancy) both are the scalars' own.
template <bool SMALL, int BLOCK>
STAG_D int iteration_alpha(const PapPartials &pap, CgScalars *sc, double *smem, dpair &alpha) {
    const int status = sc->status;
    if (!SMALL || status != CG_RUNNING) {
        alpha = sc->alpha;
        return status;
    }
    __shared__ dpair salpha;
    __shared__ int sstatus;
    const double total = sum_partials<BLOCK>(pap.v, pap.n, smem);
    if (threadIdx.x == 0) {
        sstatus = total > 0.0 && total < INFINITY ? CG_RUNNING : CG_BREAKDOWN;
        salpha = make_dpair(sstatus == CG_RUNNING ? sc->rr / total : 0.0);
        if (blockIdx.x == 0) {
            sc->pAp = total;
            sc->alpha = salpha;
        }
    }
    __syncthreads();
    alpha = salpha;
    return sstatus;
}

}  // namespace stag
