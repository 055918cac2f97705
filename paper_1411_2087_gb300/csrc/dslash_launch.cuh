// Launcher template of the Dslash kernels; each precision is instantiated in
// its own translation unit (dslash_<prec>.cu) so that they compile in parallel.
#pragma once
#include "dslash_split.cuh"
#include "kernels.h"

namespace stag {

// Which kernels run under the register cap by default (before tuning):
// FP32 and 16-bit (the figures are at kCapThreads).  The FP64 kernel is
// bound by the FP64 pipe and keeps the compiler's choice.
template <int P>
constexpr bool kCapped = P == P_F16 || P == P_F32;

template <int P, int EPI, int BLOCK, int CM>
static void launch_capped(int grid, const DslashArgs &a, cudaStream_t s) {
    constexpr int least = cap_blocks_least<P, CM>(BLOCK);
    const int blocks = cap_blocks<P, CM>(BLOCK, grid, a.keep);
    if constexpr (P == P_F32 && least < 1024 / BLOCK)
        if (blocks > least) {
            dslash_kernel_capped<P, EPI, BLOCK, CM, 1024 / BLOCK><<<grid, BLOCK, 0, s>>>(a);
            return;
        }
    dslash_kernel_capped<P, EPI, BLOCK, CM, least><<<grid, BLOCK, 0, s>>>(a);
}

// The plain stencil and the M stencil with <p, Mp> partials (the solvers'
// two kernels per iteration) are instantiated in both register variants, so
// that the autotuner can time them; the other epilogues use the default.
template <int P, int EPI, int BLOCK, int CM>
static void launch_one(int grid, const DslashArgs &a, cudaStream_t s) {
    constexpr bool tunable = EPI == EPI_NONE || EPI == EPI_M_PART;
    const bool capped = tunable && a.regs != REGS_DEFAULT && a.regs != REGS_PAIR ? a.regs == REGS_CAPPED
                                                                                 : kCapped<P>;
    if constexpr (tunable) {
        if (capped)
            launch_capped<P, EPI, BLOCK, CM>(grid, a, s);
        else
            dslash_kernel<P, EPI, BLOCK, CM><<<grid, BLOCK, 0, s>>>(a);
    } else if constexpr (kCapped<P>) {
        launch_capped<P, EPI, BLOCK, CM>(grid, a, s);
    } else {
        dslash_kernel<P, EPI, BLOCK, CM><<<grid, BLOCK, 0, s>>>(a);
    }
}

// the split form with NG warps per block
template <int P, int NG, int CM>
static cudaError_t launch_split_g(int epi, const DslashArgs &a, cudaStream_t s) {
    const dim3 grid(dslash_blocks(P, epi, a, 0), a.nbatch > 1 ? a.nbatch : 1);
    const int block = 32 * NG;
    if (grid.x == 0)
        return cudaSuccess;
    if (grid.y > 1 && epi != EPI_NONE && epi != EPI_M)
        return cudaErrorInvalidValue;
    switch (epi) {
    case EPI_NONE: dslash_split_kernel<P, EPI_NONE, NG, CM><<<grid, block, 0, s>>>(a); break;
    case EPI_M: dslash_split_kernel<P, EPI_M, NG, CM><<<grid, block, 0, s>>>(a); break;
    case EPI_M_PAP: dslash_split_kernel<P, EPI_M_PAP, NG, CM><<<grid, block, 0, s>>>(a); break;
    case EPI_RESID: dslash_split_kernel<P, EPI_RESID, NG, CM><<<grid, block, 0, s>>>(a); break;
    case EPI_RESID_STORE: dslash_split_kernel<P, EPI_RESID_STORE, NG, CM><<<grid, block, 0, s>>>(a); break;
    case EPI_M_PART: dslash_split_kernel<P, EPI_M_PART, NG, CM><<<grid, block, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int P, int CM>
static cudaError_t launch_split(int epi, const DslashArgs &a, cudaStream_t s) {
    switch (split_warps(P, a)) {
    case 4: return launch_split_g<P, 4, CM>(epi, a, s);
    case 8: return launch_split_g<P, 8, CM>(epi, a, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int P, int BLOCK, int CM>
static cudaError_t launch_p_b_c(int epi, const DslashArgs &a, cudaStream_t s) {
    if constexpr (P == P_F16 && pair16_ring<BLOCK, CM>() > 0) {
        if (pair16_used(P, epi, a, BLOCK)) {
            const int grid = dslash_pair16_grid(a.g, BLOCK);
            if (epi == EPI_NONE)
                dslash_pair16_kernel<EPI_NONE, BLOCK, CM><<<grid, BLOCK, 0, s>>>(a);
            else
                dslash_pair16_kernel<EPI_M_PART, BLOCK, CM><<<grid, BLOCK, 0, s>>>(a);
            return cudaGetLastError();
        }
    }
    const int grid = dslash_blocks(P, epi, a, BLOCK);
    if (grid == 0)
        return cudaSuccess;
    if (a.nbatch > 1)  // the split form only
        return cudaErrorInvalidValue;
    switch (epi) {
    case EPI_NONE: launch_one<P, EPI_NONE, BLOCK, CM>(grid, a, s); break;
    case EPI_M: launch_one<P, EPI_M, BLOCK, CM>(grid, a, s); break;
    case EPI_M_PAP: launch_one<P, EPI_M_PAP, BLOCK, CM>(grid, a, s); break;
    case EPI_RESID: launch_one<P, EPI_RESID, BLOCK, CM>(grid, a, s); break;
    case EPI_RESID_STORE: launch_one<P, EPI_RESID_STORE, BLOCK, CM>(grid, a, s); break;
    case EPI_M_PART: launch_one<P, EPI_M_PART, BLOCK, CM>(grid, a, s); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// the 12-real layout exists for FP32 and 16-bit links only: every link
// 12-real (mask 3), or the three-link ones only (mask 2)
template <int P, int BLOCK>
static cudaError_t launch_p_b(int epi, const DslashArgs &a, cudaStream_t s) {
    if constexpr (P == P_F32 || P == P_F16) {
        switch (a.compressed) {
        case 0: return launch_p_b_c<P, BLOCK, 0>(epi, a, s);
        case 2: return launch_p_b_c<P, BLOCK, 2>(epi, a, s);
        case 3: return launch_p_b_c<P, BLOCK, 3>(epi, a, s);
        default: return cudaErrorInvalidValue;
        }
    } else {
        if (a.compressed)
            return cudaErrorInvalidValue;
        return launch_p_b_c<P, BLOCK, 0>(epi, a, s);
    }
}

template <int P> cudaError_t launch_dslash_p(int epi, const DslashArgs &a, int block, cudaStream_t s) {
    if constexpr (P != P_F16) {
        if (split_warps(P, a) > 0) {
            if constexpr (P == P_F32) {
                if (a.compressed == 2)
                    return launch_split<P, 2>(epi, a, s);
                if (a.compressed == 3)
                    return launch_split<P, 3>(epi, a, s);
            }
            return a.compressed ? cudaErrorInvalidValue : launch_split<P, 0>(epi, a, s);
        }
    }
    switch (block) {
    case 64: return launch_p_b<P, 64>(epi, a, s);
    case 128: return launch_p_b<P, 128>(epi, a, s);
    case 256: return launch_p_b<P, 256>(epi, a, s);
    case 512: return launch_p_b<P, 512>(epi, a, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace stag
