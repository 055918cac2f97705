// The stencil with one site's sixteen hops spread over the warps of a block.
//
// With one thread per site a small lattice leaves most of the chip idle: at
// 8^4 a double-float launch is 64 warps on 608 schedulers, each working
// through 16 hops (about 7000 instructions) one memory latency after the
// other, 14.6 us, and up to 46080 sites a launch costs 15-31 us whatever it
// moves.  Here NG warps share 32 sites (a warp still reads 32 consecutive
// sites, so every request is one contiguous segment), the sums meet in
// shared memory, and one launch takes 4.5 us at 8^4 (cycle-bound on the
// dependent loads), 13.8 us at 16^4 (was 26.9; its links come from L2) and
// 20 us at 46080 sites (was 31).  The hop is a loop over runtime mu, h, dir
// rather than sixteen unrolled copies: 8 KB of instructions instead of 110.
// At 896 resident threads per SM (72 registers in double float; 768 and
// 1024 measured slower at 32768 to 128000 sites) the finer blocks also fill
// the last wave better, which keeps the form ahead up to 331776 sites except
// where one thread per site takes a single, nearly full wave.  split_warps
// (kernels_dslash.cu) says where it runs.
#pragma once
#include "dslash.cuh"

namespace stag {

constexpr int SPLIT_SITES = 32;  // output sites per block, one per lane

// acc += one hop of the stencil at site c (coordinates x) of the parity of
// Gout: direction mu, h = 0 one-link, 1 three-link, dir = 0 forward, 1
// backward, all three known at run time only (warp-uniform).  q carries the
// 12-real links' constants (DslashArgs; not read on full links).
template <int P, int CM, int LD, class Q>
STAG_D void stencil_hop(const Geom &g, const void *__restrict__ Gout, const void *__restrict__ Gin,
                        const typename Fmt<P>::Elem *__restrict__ in, const Q &q, int keep, int c, const int x[4],
                        int mu, int h, int dir, cplx<typename Fmt<P>::R> acc[3]) {
    using R = typename Fmt<P>::R;
    const int S = g.stride;
    const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
    const int s = h ? 3 : 1, hop = dir ? -s : s, L = g.L[mu];
    int y = xm + hop, wraps = 0;
    // |hop| <= 3 and L >= 2: at most two wraps
#pragma unroll
    for (int k = 0; k < 2; k++) {
        if (y >= L) y -= L, wraps++;
        if (y < 0) y += L, wraps++;
    }
    const int j = mu == 0 ? c + (((x[0] & 1) + y - xm) >> 1) : c + (y - xm) * g.plane[mu];
    float inv_s = 0.f;
    if constexpr (CM != 0) {
        if ((CM >> h) & 1) {
            const int esum = (mu > 0 ? x[0] : 0) + (mu > 1 ? x[1] : 0) + (mu > 2 ? x[2] : 0);
            const int flip = (esum + (q.bc_neg[mu] ? wraps : 0)) & 1;
            inv_s = flip ? -q.inv_c[h] : q.inv_c[h];
        }
    }
    cplx<R> v[3], U[9];
    const l2pol pol = LinkPolicy<LD>(keep).of(dir ? j : c);
    load_vec<P>(in, S, j, v);
    if (dir) {
        load_link<P, CM, LD>(Gin, 4 * h + mu, S, j, 0.f, inv_s, pol, U);
#pragma unroll
        for (int b = 0; b < 3; b++)
            v[b] = cneg(v[b]);
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int b = 0; b < 3; b++)
                cmac_conj(acc[r], U[3 * b + r], v[b]);
    } else {
        load_link<P, CM, LD>(Gout, 4 * h + mu, S, c, 0.f, inv_s, pol, U);
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int b = 0; b < 3; b++)
                cmac(acc[r], U[3 * r + b], v[b]);
    }
}

STAG_D void acc_add(double &a, double b) { a += b; }
STAG_D void acc_add(float &a, float b) { a += b; }
STAG_D void acc_add(df &a, df b) {  // lo left unnormalised, as df_mac leaves it
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    a.hi = s;
    a.lo = __fadd_rn(a.lo, __fadd_rn(e, b.lo));
}

// the epilogue of one component o of D psi, at element `at` of its plane:
// store it (EPI_NONE), or m^2 p - o, or b minus that (residuals; EPI_RESID
// stores nothing); returns the component's share of the sum
template <int P, int EPI>
STAG_D red_t<typename Fmt<P>::R> split_epilogue(typename Fmt<P>::Elem *out, const typename Fmt<P>::Elem *pp,
                                                const typename Fmt<P>::Elem *bp, typename Fmt<P>::R m2, int at,
                                                cplx<typename Fmt<P>::R> o) {
    using F = Fmt<P>;
    using R = typename F::R;
    if (EPI == EPI_NONE) {
        o.re = rnorm<R>(o.re);
        o.im = rnorm<R>(o.im);
        __stcs(out + at, F::pack(o));
        return red_zero<red_t<R>>();
    }
    const cplx<R> p = F::unpack(ld_keep(pp + at));
    o = cneg(o);
    mac(o.re, m2, p.re);
    mac(o.im, m2, p.im);
    o.re = rnorm<R>(o.re);
    o.im = rnorm<R>(o.im);
    const bool resid = EPI == EPI_RESID || EPI == EPI_RESID_STORE;
    if (resid) {
        const cplx<R> b = F::unpack(ld_keep(bp + at));
        o.re = rsub(b.re, o.re);
        o.im = rsub(b.im, o.im);
    }
    if (EPI != EPI_RESID)
        __stcs(out + at, F::pack(o));
    R d = rzero<R>();
    mac(d, resid ? o.re : p.re, o.re);
    mac(d, resid ? o.im : p.im, o.im);
    return to_red(d);
}

// component w (colour) at lane `lane` of the block's NG partial sums, added
// in the warps' order
template <int P, int NG>
STAG_D cplx<typename Fmt<P>::R> split_sum(const typename Fmt<P>::Elem (&part)[NG][3][SPLIT_SITES], int w, int lane) {
    using F = Fmt<P>;
    cplx<typename F::R> o = F::unpack(part[0][w][lane]);
#pragma unroll
    for (int q = 1; q < NG; q++) {
        const cplx<typename F::R> u = F::unpack(part[q][w][lane]);
        acc_add(o.re, u.re);
        acc_add(o.im, u.im);
    }
    return o;
}

// NG warps per block; warp w takes the hops w 16/NG .. of the block's 32
// sites, the partial sums meet in shared memory and warps 0..2 finish one
// colour component each (sums over the warps in their order).
template <int P, int EPI, int NG, int CM>
__global__ void __launch_bounds__(32 * NG, 896 / (32 * NG)) dslash_split_kernel(const __grid_constant__ DslashArgs a) {
    using F = Fmt<P>;
    using R = typename F::R;
    using E = typename F::Elem;
    constexpr int BLOCK = 32 * NG;
    __shared__ double smem[32];
    __shared__ E part[NG][3][SPLIT_SITES];
    if (a.skip_if_done && a.sc->status != CG_RUNNING)
        return;
    if (a.gate && *a.gate == 0)
        return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // site i of the launch: the range c0.., then the second range c0b..
    const int i = blockIdx.x * SPLIT_SITES + lane;
    const int n1 = a.cn ? a.cn : a.g.Vh;
    const int n2 = a.cn ? a.cnb : 0;
    const int c = i < n1 ? a.c0 + i : a.c0b + (i - n1);
    const bool in_range = i < n1 + n2;
    const size_t vec = blockIdx.y * a.vec_step;  // this block's vector of a batch
    if (in_range) {
        int x[4];
        cb_coords(a.g, c, a.out_par, x);
        cplx<R> acc[3] = {czero<R>(), czero<R>(), czero<R>()};
#pragma unroll 1
        for (int q = 0; q < 16 / NG; q++) {
            const int hop = w * (16 / NG) + q;
            stencil_hop<P, CM, LD_KEEP>(a.g, a.links_out, a.links_in, (const E *)((const char *)a.in + vec), a, a.keep, c,
                                        x, hop >> 2, (hop >> 1) & 1, hop & 1, acc);
        }
#pragma unroll
        for (int k = 0; k < 3; k++)
            part[w][k][lane] = F::pack(acc[k]);
    }
    __syncthreads();
    red_t<R> dot = red_zero<red_t<R>>();
    if (w < 3 && in_range) {
        const cplx<R> o = split_sum<P, NG>(part, w, lane);
        const R m2 = EPI == EPI_NONE ? rzero<R>() : scalar_as<R>(a.m2_in_args ? a.m2 : a.sc->m2);
        dot = split_epilogue<P, EPI>((E *)((char *)a.out + vec), (const E *)((const char *)a.p + vec), (const E *)a.b, m2,
                                     w * a.g.stride + c, o);
    }
    dslash_reduce<EPI, BLOCK>(a, dot, smem);
}

}  // namespace stag
