// CG vector kernels and field import/export.
#include "dslash.cuh"
#include "kernels.h"
#include "small_sums.cuh"

#include <cfloat>

namespace stag {

// --------------------------------------------------------------------------
// CG vector kernels.  Each reads the device scalars written by the previous
// kernel; the last block of a reducing kernel updates them and, inside the
// solve graph, sets the loop condition.
// --------------------------------------------------------------------------

STAG_D void set_loop_condition(CgScalars *sc) {
    if (sc->has_cond)
        cudaGraphSetConditional(sc->cond, sc->status == CG_RUNNING ? 1u : 0u);
}

// x = 0, r = b, p = b, |b|^2
template <int P, int BLOCK>
__global__ void __launch_bounds__(BLOCK)
cg_init_kernel(Geom g, typename Fmt<P>::Elem *x, typename Fmt<P>::Elem *r,
               typename Fmt<P>::Elem *p, const typename Fmt<P>::Elem *b, double *partial,
               CgScalars *sc) {
    using F = Fmt<P>;
    using R = typename F::R;
    __shared__ double smem[32];
    const int c = blockIdx.x * BLOCK + threadIdx.x;
    red_t<R> dot = red_zero<red_t<R>>();
    if (c < g.Vh) {
        cplx<R> bv[3], z[3];
        load_vec<P>(b, g.stride, c, bv);
#pragma unroll
        for (int k = 0; k < 3; k++)
            z[k] = czero<R>();
        store_vec<P>(x, g.stride, c, z);
        store_vec<P>(r, g.stride, c, bv);
        store_vec<P>(p, g.stride, c, bv);
        dot = re_dot3<R>(bv, bv);
    }
    double total;
    if (grid_sum<BLOCK>(dot, partial, &sc->ticket, smem, total) && threadIdx.x == 0) {
        sc->bb = total;
        sc->rr = total;
        sc->rr_stop = sc->tol2 * total;
        sc->iter = 0;
        sc->alpha = make_dpair(0.0);
        sc->beta = make_dpair(0.0);
        if (!(total < INFINITY))
            sc->status = CG_BREAKDOWN;
        else if (total <= sc->rr_stop)
            sc->status = CG_CONVERGED;
        else if (sc->max_iter <= 0)
            sc->status = CG_MAXITER;
        else
            sc->status = CG_RUNNING;
        set_loop_condition(sc);
    }
}

// x += alpha p, r -= alpha Ap, |r|^2 -> beta, convergence
template <int P, int BLOCK>
__global__ void __launch_bounds__(BLOCK)
cg_update_kernel(Geom g, typename Fmt<P>::Elem *x, typename Fmt<P>::Elem *r,
                 const typename Fmt<P>::Elem *p, const typename Fmt<P>::Elem *Ap,
                 double *partial, CgScalars *sc) {
    using F = Fmt<P>;
    using R = typename F::R;
    __shared__ double smem[32];
    const bool run = sc->status == CG_RUNNING;
    const R alpha = scalar_as<R>(sc->alpha);
    const R malpha = -alpha;
    red_t<R> dot = red_zero<red_t<R>>();
    if (run)
        for (int c = blockIdx.x * BLOCK + threadIdx.x; c < g.Vh; c += gridDim.x * BLOCK) {
            cplx<R> xv[3], rv[3], pv[3], av[3];
            load_vec<P>(x, g.stride, c, xv);
            load_vec<P>(r, g.stride, c, rv);
            load_vec<P>(p, g.stride, c, pv);
            load_vec<P>(Ap, g.stride, c, av);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                mac(xv[k].re, alpha, pv[k].re);
                mac(xv[k].im, alpha, pv[k].im);
                mac(rv[k].re, malpha, av[k].re);
                mac(rv[k].im, malpha, av[k].im);
                xv[k].re = rnorm<R>(xv[k].re);
                xv[k].im = rnorm<R>(xv[k].im);
                rv[k].re = rnorm<R>(rv[k].re);
                rv[k].im = rnorm<R>(rv[k].im);
            }
            store_vec<P>(x, g.stride, c, xv);
            store_vec<P>(r, g.stride, c, rv);
            dot = red_add(dot, re_dot3<R>(rv, rv));
        }
    double total;
    if (grid_sum<BLOCK>(dot, partial, &sc->ticket, smem, total) && threadIdx.x == 0) {
        if (sc->status == CG_RUNNING) {
            const double beta = total / sc->rr;
            sc->beta = make_dpair(beta);
            sc->rr = total;
            sc->iter += 1;
            if (!(total < INFINITY))
                sc->status = CG_BREAKDOWN;
            else if (total <= sc->rr_stop)
                sc->status = CG_CONVERGED;
            else if (sc->iter >= sc->max_iter)
                sc->status = CG_MAXITER;
        } else {
            sc->beta = make_dpair(0.0);
        }
        set_loop_condition(sc);
    }
}

// p = r + beta p
template <int P, int BLOCK>
__global__ void __launch_bounds__(BLOCK)
cg_p_kernel(Geom g, const typename Fmt<P>::Elem *r, typename Fmt<P>::Elem *p, const CgScalars *sc) {
    using F = Fmt<P>;
    using R = typename F::R;
    const int c = blockIdx.x * BLOCK + threadIdx.x;
    // after convergence or breakdown p is no longer used
    if (c >= g.Vh || sc->status != CG_RUNNING)
        return;
    const R beta = scalar_as<R>(sc->beta);
    cplx<R> rv[3], pv[3];
    load_vec<P>(r, g.stride, c, rv);
    load_vec<P>(p, g.stride, c, pv);
#pragma unroll
    for (int k = 0; k < 3; k++) {
        mac(rv[k].re, beta, pv[k].re);
        mac(rv[k].im, beta, pv[k].im);
        rv[k].re = rnorm<R>(rv[k].re);
        rv[k].im = rnorm<R>(rv[k].im);
    }
    store_vec<P>(p, g.stride, c, rv);
}

// one block: sum of the block partials of an EPI_M_PART Dslash, then alpha
constexpr int FINISH_BLOCK = 1024;

__global__ void __launch_bounds__(FINISH_BLOCK)
pap_finish_kernel(const double *__restrict__ partial, int n, CgScalars *sc, int skip_if_done, const int *gate) {
    __shared__ double smem[32];
    // the scalars are read together with the partials, not before them
    const double rr = sc->rr;
    const int status = sc->status;
    const int open = gate ? *gate : 1;
    const double share = partials_share<FINISH_BLOCK>(partial, n);
    if ((skip_if_done && status != CG_RUNNING) || open == 0)
        return;
    const double total = block_sum<FINISH_BLOCK>(share, smem);
    if (threadIdx.x == 0) {
        sc->pAp = total;
        const bool ok = total > 0.0 && total < INFINITY;
        if (status == CG_RUNNING && !ok)
            sc->status = CG_BREAKDOWN;
        sc->alpha = make_dpair(status == CG_RUNNING && ok ? rr / total : 0.0);
    }
}

cudaError_t launch_pap_finish(const double *partial, int n, CgScalars *sc, bool skip_if_done, cudaStream_t s,
                              const int *gate) {
    pap_finish_kernel<<<1, FINISH_BLOCK, 0, s>>>(partial, n, sc, skip_if_done ? 1 : 0, gate);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// The vector kernels of plain CG on small lattices: <p, Ap> and |r|^2 are
// both summed by the kernel after the one that leaves their partials
// (small_sums.cuh; the update at 8^4 took 6.9 us with a ticket, now 4.4).  No
// kernel reads a scalar that it writes: the update kernel reads rr, iter,
// status and writes alpha, pAp, up_*; the direction kernel reads up_* and
// writes the others.
// --------------------------------------------------------------------------
// x += alpha p, r -= alpha Ap with alpha = rr / <p, Ap> from the M Dslash's
// npap partials; one partial of |r|^2 per block
template <int P, int BLOCK>
__global__ void __launch_bounds__(BLOCK)
cg_small_update_kernel(Geom g, typename Fmt<P>::Elem *x, typename Fmt<P>::Elem *r, const typename Fmt<P>::Elem *p,
                       const typename Fmt<P>::Elem *Ap, PapPartials pap, double *rr_part, CgScalars *sc) {
    using R = typename Fmt<P>::R;
    __shared__ double smem[32];
    dpair alpha_k;
    const int c = blockIdx.x * BLOCK + threadIdx.x;
    cplx<R> xv[3], rv[3], pv[3], av[3];
    if (c < g.Vh) {  // in flight while the partials are summed
        load_vec<P>(x, g.stride, c, xv);
        load_vec<P>(r, g.stride, c, rv);
        load_vec<P>(p, g.stride, c, pv);
        load_vec<P>(Ap, g.stride, c, av);
    }
    const int status = iteration_alpha<true, BLOCK>(pap, sc, smem, alpha_k);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->up_rr = sc->rr;
        sc->up_iter = sc->iter;
        sc->up_status = status;
    }
    if (status != CG_RUNNING)
        return;
    red_t<R> dot = red_zero<red_t<R>>();
    if (c < g.Vh) {
        const R alpha = scalar_as<R>(alpha_k);
        const R malpha = -alpha;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            mac(xv[k].re, alpha, pv[k].re);
            mac(xv[k].im, alpha, pv[k].im);
            mac(rv[k].re, malpha, av[k].re);
            mac(rv[k].im, malpha, av[k].im);
            xv[k].re = rnorm<R>(xv[k].re);
            xv[k].im = rnorm<R>(xv[k].im);
            rv[k].re = rnorm<R>(rv[k].re);
            rv[k].im = rnorm<R>(rv[k].im);
        }
        store_vec<P>(x, g.stride, c, xv);
        store_vec<P>(r, g.stride, c, rv);
        dot = re_dot3<R>(rv, rv);
    }
    const double s = block_sum<BLOCK>(dot, smem);
    if (threadIdx.x == 0)
        rr_part[blockIdx.x] = s;
}

// |r|^2 from the update's nrr partials, beta, the stopping test, p = r + beta p
template <int P, int BLOCK>
__global__ void __launch_bounds__(BLOCK)
cg_small_p_kernel(Geom g, const typename Fmt<P>::Elem *r, typename Fmt<P>::Elem *p, const double *rr_part, int nrr,
                  CgScalars *sc) {
    using R = typename Fmt<P>::R;
    __shared__ double smem[32];
    __shared__ dpair sbeta;
    __shared__ int sstatus;
    const int c = blockIdx.x * BLOCK + threadIdx.x;
    cplx<R> rv[3], pv[3];
    if (c < g.Vh) {
        load_vec<P>(r, g.stride, c, rv);
        load_vec<P>(p, g.stride, c, pv);
    }
    int status = sc->up_status;
    if (status == CG_RUNNING) {
        const double total = sum_partials<BLOCK>(rr_part, nrr, smem);
        if (threadIdx.x == 0) {
            const double beta = total / sc->up_rr;
            const int iter = sc->up_iter + 1;
            sbeta = make_dpair(beta);
            sstatus = !(total < INFINITY)      ? CG_BREAKDOWN
                      : total <= sc->rr_stop   ? CG_CONVERGED
                      : iter >= sc->max_iter   ? CG_MAXITER
                                               : CG_RUNNING;
            if (blockIdx.x == 0) {
                sc->beta = sbeta;
                sc->rr = total;
                sc->iter = iter;
            }
        }
        __syncthreads();
        status = sstatus;
    } else if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->beta = make_dpair(0.0);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->status = status;
        set_loop_condition(sc);
    }
    // after convergence or breakdown p is no longer used
    if (c >= g.Vh || status != CG_RUNNING)
        return;
    const R beta = scalar_as<R>(sbeta);
#pragma unroll
    for (int k = 0; k < 3; k++) {
        mac(rv[k].re, beta, pv[k].re);
        mac(rv[k].im, beta, pv[k].im);
        rv[k].re = rnorm<R>(rv[k].re);
        rv[k].im = rnorm<R>(rv[k].im);
    }
    store_vec<P>(p, g.stride, c, rv);
}

static int cg_grid(const Geom &g) { return (g.Vh + CG_BLOCK - 1) / CG_BLOCK; }

#define STAG_PREC_SWITCH(prec, ...)                                   \
    switch (prec) {                                                   \
    case P_F64: { constexpr int P = P_F64; __VA_ARGS__; } break;      \
    case P_DF64: { constexpr int P = P_DF64; __VA_ARGS__; } break;    \
    case P_F32: { constexpr int P = P_F32; __VA_ARGS__; } break;      \
    case P_F16: { constexpr int P = P_F16; __VA_ARGS__; } break;      \
    default: return cudaErrorInvalidValue;                            \
    }

cudaError_t launch_cg_init(int prec, const Geom &g, void *x, void *r, void *p, const void *b,
                           double *partial, CgScalars *sc, cudaStream_t s) {
    STAG_PREC_SWITCH(prec, {
        using E = typename Fmt<P>::Elem;
        cg_init_kernel<P, CG_BLOCK><<<cg_grid(g), CG_BLOCK, 0, s>>>(g, (E *)x, (E *)r, (E *)p,
                                                                    (const E *)b, partial, sc);
    });
    return cudaGetLastError();
}

cudaError_t launch_cg_update(int prec, const Geom &g, void *x, void *r, const void *p,
                             const void *Ap, double *partial, CgScalars *sc, cudaStream_t s) {
    STAG_PREC_SWITCH(prec, {
        using E = typename Fmt<P>::Elem;
        cg_update_kernel<P, CG_BLOCK><<<sum_grid(g.Vh, CG_BLOCK), CG_BLOCK, 0, s>>>(
            g, (E *)x, (E *)r, (const E *)p, (const E *)Ap, partial, sc);
    });
    return cudaGetLastError();
}

cudaError_t launch_cg_p_update(int prec, const Geom &g, const void *r, void *p,
                               const CgScalars *sc, cudaStream_t s) {
    STAG_PREC_SWITCH(prec, {
        using E = typename Fmt<P>::Elem;
        cg_p_kernel<P, CG_BLOCK><<<cg_grid(g), CG_BLOCK, 0, s>>>(g, (const E *)r, (E *)p, sc);
    });
    return cudaGetLastError();
}

constexpr int SMALL_BLOCK = 256;
static int small_grid(const Geom &g) { return (g.Vh + SMALL_BLOCK - 1) / SMALL_BLOCK; }

cudaError_t launch_cg_small_vectors(int prec, const Geom &g, void *x, void *r, void *p, const void *Ap,
                                    const PapPartials &pap, double *rr_part, CgScalars *sc, cudaStream_t s) {
    const int grid = small_grid(g);
    STAG_PREC_SWITCH(prec, {
        using E = typename Fmt<P>::Elem;
        cg_small_update_kernel<P, SMALL_BLOCK><<<grid, SMALL_BLOCK, 0, s>>>(g, (E *)x, (E *)r, (const E *)p,
                                                                           (const E *)Ap, pap, rr_part, sc);
        cg_small_p_kernel<P, SMALL_BLOCK><<<grid, SMALL_BLOCK, 0, s>>>(g, (const E *)r, (E *)p, rr_part, grid, sc);
    });
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// import / export between canonical complex128 [Vh][3] and the SoA layout
// --------------------------------------------------------------------------
template <int P>
__global__ void import_kernel(Geom g, const double *__restrict__ canon, typename Fmt<P>::Elem *f) {
    using R = typename Fmt<P>::R;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.Vh)
        return;
    cplx<R> w[3];
#pragma unroll
    for (int a = 0; a < 3; a++)
        w[a] = Fmt<P>::make(canon[(3 * (size_t)c + a) * 2], canon[(3 * (size_t)c + a) * 2 + 1]);
    store_vec<P>(f, g.stride, c, w);
}

template <int P>
__global__ void export_kernel(Geom g, const typename Fmt<P>::Elem *f, double *__restrict__ canon) {
    using R = typename Fmt<P>::R;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.Vh)
        return;
    cplx<R> w[3];
    load_vec<P>(f, g.stride, c, w);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        canon[(3 * (size_t)c + a) * 2] = to_double<R>(w[a].re);
        canon[(3 * (size_t)c + a) * 2 + 1] = to_double<R>(w[a].im);
    }
}

cudaError_t launch_import(int prec, const Geom &g, const double *canon, void *field, cudaStream_t s) {
    const int grid = (g.Vh + 255) / 256;
    STAG_PREC_SWITCH(prec, {
        import_kernel<P><<<grid, 256, 0, s>>>(g, canon, (typename Fmt<P>::Elem *)field);
    });
    return cudaGetLastError();
}

cudaError_t launch_export(int prec, const Geom &g, const void *field, double *canon, cudaStream_t s) {
    const int grid = (g.Vh + 255) / 256;
    STAG_PREC_SWITCH(prec, {
        export_kernel<P><<<grid, 256, 0, s>>>(g, (const typename Fmt<P>::Elem *)field, canon);
    });
    return cudaGetLastError();
}

// *flag = 1 if a finite entry lies beyond the FP32 range (NaN and infinity
// pass: the solvers report them as breakdowns)
__global__ void finite_overflow_kernel(const double *__restrict__ a, long long n, unsigned *flag) {
    int bad = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double v = fabs(a[i]);
        bad |= v > (double)FLT_MAX && v < INFINITY;
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0)
        atomicOr(flag, 1u);
}

cudaError_t launch_finite_overflow(const double *a, long long n, unsigned *flag, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(unsigned), s);
    if (e != cudaSuccess)
        return e;
    finite_overflow_kernel<<<1024, 256, 0, s>>>(a, n, flag);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// exact power-of-two rescaling of a colour field (the solvers' source
// normalisation): the largest |component| (double-float: of the hi parts)
// as float bits, and v *= 2^e
// --------------------------------------------------------------------------
template <int P> STAG_D float elem_absmax(typename Fmt<P>::Elem v);
template <> STAG_D float elem_absmax<P_F64>(double2 v) { return (float)fmax(fabs(v.x), fabs(v.y)); }
template <> STAG_D float elem_absmax<P_DF64>(float4 v) { return fmaxf(fabsf(v.x), fabsf(v.z)); }
template <> STAG_D float elem_absmax<P_F32>(float2 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }

template <int P> STAG_D typename Fmt<P>::Elem elem_ldexp(typename Fmt<P>::Elem v, int e);
template <> STAG_D double2 elem_ldexp<P_F64>(double2 v, int e) { return make_double2(ldexp(v.x, e), ldexp(v.y, e)); }
template <> STAG_D float4 elem_ldexp<P_DF64>(float4 v, int e) {
    return make_float4(ldexpf(v.x, e), ldexpf(v.y, e), ldexpf(v.z, e), ldexpf(v.w, e));
}
template <> STAG_D float2 elem_ldexp<P_F32>(float2 v, int e) { return make_float2(ldexpf(v.x, e), ldexpf(v.y, e)); }

template <int P>
__global__ void field_absmax_kernel(Geom g, const typename Fmt<P>::Elem *__restrict__ v, unsigned *out) {
    float m = 0.f;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < g.Vh; c += gridDim.x * blockDim.x)
#pragma unroll
        for (int a = 0; a < 3; a++)
            m = fmaxf(m, elem_absmax<P>(v[(size_t)a * g.stride + c]));  // fmaxf drops NaN
    for (int o = 16; o > 0; o >>= 1)
        m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(out, __float_as_uint(m));
}

template <int P>
__global__ void field_ldexp_kernel(Geom g, typename Fmt<P>::Elem *v, int e) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.Vh)
        return;
#pragma unroll
    for (int a = 0; a < 3; a++)
        v[(size_t)a * g.stride + c] = elem_ldexp<P>(v[(size_t)a * g.stride + c], e);
}

#define STAG_SRC_SWITCH(prec, ...)                                    \
    switch (prec) {                                                   \
    case P_F64: { constexpr int P = P_F64; __VA_ARGS__; } break;      \
    case P_DF64: { constexpr int P = P_DF64; __VA_ARGS__; } break;    \
    case P_F32: { constexpr int P = P_F32; __VA_ARGS__; } break;      \
    default: return cudaErrorInvalidValue;                            \
    }

cudaError_t launch_field_absmax(int prec, const Geom &g, const void *v, unsigned *out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned), s);
    if (e != cudaSuccess)
        return e;
    STAG_SRC_SWITCH(prec, field_absmax_kernel<P><<<512, 256, 0, s>>>(g, (const typename Fmt<P>::Elem *)v, out));
    return cudaGetLastError();
}

cudaError_t launch_field_ldexp(int prec, const Geom &g, void *v, int e, cudaStream_t s) {
    STAG_SRC_SWITCH(prec, field_ldexp_kernel<P><<<(g.Vh + 255) / 256, 256, 0, s>>>(g, (typename Fmt<P>::Elem *)v, e));
    return cudaGetLastError();
}

}  // namespace stag
