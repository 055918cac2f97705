// Kernels of a gauge upload: the scan of the raw links (largest entry,
// deviation from SU(3)), their folding into the library's copies, and the
// three-link products.
#include "dslash.cuh"
#include "kernels.h"

#include <cfloat>
#include <cmath>

namespace stag {

STAG_D void full_coords(const Geom &g, long long i, int x[4]) {
    x[0] = (int)(i % g.L[0]);
    i /= g.L[0];
    x[1] = (int)(i % g.L[1]);
    i /= g.L[1];
    x[2] = (int)(i % g.L[2]);
    x[3] = (int)(i / g.L[2]);
}

STAG_D void copy16_async(void *smem, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(src)
                 : "memory");
}
STAG_D void copy_async_wait() { asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory"); }

// --------------------------------------------------------------------------
// double -> float without the FP64 pipe.  GB300 converts between double and
// float at the FP64 rate, 1/64 of the integer rate: a link's 18 reals cost
// 64 cycles of a scheduler per conversion and warp, and the double-float split
// takes four per real.  On the bits it is integer work.
// --------------------------------------------------------------------------
// the exact split d = hi + lo of df_from_double (both rounded to nearest even)
STAG_D df df_split(double d) {
    const long long u = __double_as_longlong(d);
    const int e = (int)((u >> 52) & 0x7ff);
    // lo's lowest bit 2^(e - 1023 - 52) and hi's exponent stay in the normal
    // float range; zero, tiny, huge and non-finite values take the conversions
    if (e < 1023 - 70 || e > 1023 + 126)
        return df_from_double(d);
    const long long m = (u & 0xfffffffffffffLL) | (1LL << 52);
    int q = (int)(m >> 29);                 // 24 bits
    int r = (int)(m & 0x1fffffff);          // 29 bits
    const int half = 1 << 28;
    if (r > half || (r == half && (q & 1))) {
        q += 1;
        r -= 1 << 29;
    }
    // d = +-(q 2^(e-1023-23) + r 2^(e-1023-52)); q and the scalings are exact,
    // r is rounded to 24 bits by its conversion
    if (u < 0) {
        q = -q;
        r = -r;
    }
    return df_make((float)q * __int_as_float((e - 1023 + 127 - 23) << 23),
                   (float)r * __int_as_float((e - 1023 + 127 - 52) << 23));
}

// --------------------------------------------------------------------------
// the scan
// --------------------------------------------------------------------------
constexpr int SCAN_BLOCK = 128;

// max(|U U^+ - 1|, entry-wise, |det U - 1|) of one link.  The nine products
// of U U^+ run in FP32 first (rounding at most 8 u sum |u||v| < 4.8e-7 for
// rows of length one); only a link that may miss 1e-6 by that repeats them in
// double-float.  The determinant's bound in FP32 would exceed 1e-6, so it is
// double-float always.  In FP64 this took 240 operations at 1/64 rate.  Where
// FP32 can tell, the products add nothing to the result, which then serves the
// decision and is not the deviation; with EXACT they run in double-float for
// every link.
template <bool EXACT> STAG_D float su3_deviation(const double2 *A) {
    df re[9], im[9];
#pragma unroll
    for (int e = 0; e < 9; e++) {
        re[e] = df_split(A[e].x);
        im[e] = df_split(A[e].y);
    }
    float dev = 0.f;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = a; b < 3; b++) {
            float sr = a == b ? -1.f : 0.f, si = 0.f;
#pragma unroll
            for (int k = 0; k < 3; k++) {  // (U U^+)_ab = sum_k U_ak conj(U_bk)
                const int p = 3 * a + k, q = 3 * b + k;
                sr = fmaf(re[p].hi, re[q].hi, sr);
                sr = fmaf(im[p].hi, im[q].hi, sr);
                if (a != b) {
                    si = fmaf(im[p].hi, re[q].hi, si);
                    si = fmaf(-re[p].hi, im[q].hi, si);
                }
            }
            const float d = fmaxf(fabsf(sr), fabsf(si));
            dev = d >= 0.f ? fmaxf(dev, d) : INFINITY;  // an overflow to NaN is no special unitary link
        }
    if (EXACT || !(dev <= 5e-7f)) {
        dev = 0.f;
        for (int a = 0; a < 3; a++)
            for (int b = a; b < 3; b++) {
                df sr = df_make(a == b ? -1.f : 0.f, 0.f), si = df_zero();
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const int p = 3 * a + k, q = 3 * b + k;
                    const double2 u = A[p], v = A[q];
                    const df ur = df_split(u.x), ui = df_split(u.y), vr = df_split(v.x), vi = df_split(v.y);
                    df_mac(sr, ur, vr);
                    df_mac(sr, ui, vi);
                    df_mac(si, ui, vr);
                    df_mac(si, -ur, vi);
                }
                const float d = fmaxf(fabsf(sr.hi + sr.lo), fabsf(si.hi + si.lo));
                dev = d >= 0.f ? fmaxf(dev, d) : INFINITY;
            }
    } else {
        dev = 0.f;
    }
    // det - 1 by the first row's cofactors
    df dr = df_make(-1.f, 0.f), di = df_zero();
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const int k = 3 + (j + 1) % 3, q = 3 + (j + 2) % 3;
        // U_1k U_2q - U_1q U_2k
        df cr = df_zero(), ci = df_zero();
        df_mac(cr, re[k], re[q + 3]);
        df_mac(cr, -im[k], im[q + 3]);
        df_mac(cr, -re[q], re[k + 3]);
        df_mac(cr, im[q], im[k + 3]);
        df_mac(ci, re[k], im[q + 3]);
        df_mac(ci, im[k], re[q + 3]);
        df_mac(ci, -re[q], im[k + 3]);
        df_mac(ci, -im[q], re[k + 3]);
        cr = df_norm(cr);
        ci = df_norm(ci);
        df_mac(dr, re[j], cr);
        df_mac(dr, -im[j], ci);
        df_mac(di, re[j], ci);
        df_mac(di, im[j], cr);
    }
    const float d = fmaxf(fabsf(dr.hi + dr.lo), fabsf(di.hi + di.lo));
    return d >= 0.f ? fmaxf(dev, d) : INFINITY;
}

// One pass over up to two link fields (blockIdx.y): the largest |entry|, as
// the largest magnitude bits of the doubles (an infinity or a NaN exceeds
// every finite value), and with su3 the deviation from SU(3) as float bits.
// Each warp stages 32 links (4608 contiguous bytes) in shared memory by
// asynchronous copies, so that every global request is one contiguous segment
// (links are 144 bytes apart), the next 32 while it works on these.  Both
// fields of 24^3x48 (764 MB) take about 257 us (3.0 TB/s), bound by the
// integer work of the splits and the determinant; 361 us with each warp waiting
// for its own loads at 4 blocks per SM, 2.2 ms as four passes in FP64.  Five
// blocks hold the registers to 96; six would spill 136 bytes a thread.
constexpr int SCAN_BLOCKS_PER_SM = 5;
static_assert(kSMs * SCAN_BLOCKS_PER_SM * SCAN_BLOCK == 97280,
              "tests/test_gpu_upload.py puts its wrong links at multiples of the links of one sweep");

template <ScanSu3 SU3>
__global__ void __launch_bounds__(SCAN_BLOCK, SCAN_BLOCKS_PER_SM)
scan_links_kernel(const double2 *__restrict__ f0, const double2 *__restrict__ f1, long long nlinks, LinkScan *out) {
    __shared__ double2 tile[SCAN_BLOCK / 32][2][288];
    const double2 *U = blockIdx.y ? f1 : f0;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long nchunk = (nlinks + 31) / 32, total = nlinks * 9;
    const long long step = gridDim.x * (SCAN_BLOCK / 32LL);
    auto stage = [&](long long c, int buf) {
        if (c < nchunk) {
#pragma unroll
            for (int k = 0; k < 9; k++)
                if (c * 288 + k * 32 + lane < total)
                    copy16_async(&tile[w][buf][k * 32 + lane], U + c * 288 + k * 32 + lane);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    long long big = 0;
    float dev = 0.f;
    int buf = 0;
    long long c = blockIdx.x * (SCAN_BLOCK / 32LL) + w;
    stage(c, 0);
    for (; c < nchunk; c += step, buf ^= 1) {
        stage(c + step, buf ^ 1);
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncwarp();
        if (c * 32 + lane < nlinks) {
            const double2 *A = &tile[w][buf][lane * 9];
#pragma unroll
            for (int e = 0; e < 9; e++) {
                big = max(big, __double_as_longlong(A[e].x) & 0x7fffffffffffffffLL);
                big = max(big, __double_as_longlong(A[e].y) & 0x7fffffffffffffffLL);
            }
            if (SU3 != SCAN_NO_SU3)
                dev = fmaxf(dev, su3_deviation<SU3 == SCAN_SU3_EXACT>(A));
        }
        __syncwarp();
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        big = max(big, __shfl_down_sync(0xffffffffu, big, o));
        dev = fmaxf(dev, __shfl_down_sync(0xffffffffu, dev, o));
    }
    if (lane == 0) {
        atomicMax((long long *)&out[blockIdx.y].maxbits, big);
        if (SU3 != SCAN_NO_SU3)
            atomicMax(&out[blockIdx.y].dev, __float_as_uint(dev));
    }
}

cudaError_t launch_scan_links(const double *f0, const double *f1, long long nlinks, ScanSu3 su3, LinkScan *out,
                              cudaStream_t s) {
    const int nf = f1 ? 2 : 1;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(LinkScan) * nf, s);
    if (e != cudaSuccess)
        return e;
    const long long blocks = (nlinks + 127) / 128;
    const int most = kSMs * SCAN_BLOCKS_PER_SM;
    const dim3 grid((unsigned)(blocks < most ? blocks : most), nf);
    const double2 *a = (const double2 *)f0, *b = (const double2 *)f1;
    switch (su3) {
    case SCAN_NO_SU3: scan_links_kernel<SCAN_NO_SU3><<<grid, SCAN_BLOCK, 0, s>>>(a, b, nlinks, out); break;
    case SCAN_SU3_LIMIT: scan_links_kernel<SCAN_SU3_LIMIT><<<grid, SCAN_BLOCK, 0, s>>>(a, b, nlinks, out); break;
    case SCAN_SU3_EXACT: scan_links_kernel<SCAN_SU3_EXACT><<<grid, SCAN_BLOCK, 0, s>>>(a, b, nlinks, out); break;
    }
    return cudaGetLastError();
}

float scan_absmax(const LinkScan &s) {
    double d;
    static_assert(sizeof d == sizeof s.maxbits, "double bits");
    memcpy(&d, &s.maxbits, sizeof d);
    const float v = (float)d;
    return v <= FLT_MAX ? v : INFINITY;
}
float scan_su3_deviation(const LinkScan &s) {
    float d;
    memcpy(&d, &s.dev, sizeof d);
    return d;
}

// --------------------------------------------------------------------------
// link folding: entry j of kind `kind` = mu (+4 long) at (par, cb) = coef * L[mu][i][j]
// (the kinds' layouts as link_kind_offset describes)
//   coef = c * eta_mu(x) * bc_mu^w,  w = floor((x_mu + s) / L_mu), s = 1 or 3
// so that the stencil applies  + G(x) psi(x+s mu)  and  - G(x-s mu)^+ psi(x-s mu).
// --------------------------------------------------------------------------
struct FoldArgs {
    Geom g;
    double bc[4];
    double c1, c3;
    float inv_scale[2];  // 16-bit links: 32767 / field max (one-link, three-link)
    FoldOut out;
};

// One launch folds a field into every copy that is asked for.  A warp takes
// 64 consecutive links of one kind (32 sites of each parity): 9216 contiguous
// bytes, staged in shared memory by 16-byte asynchronous copies, so that the
// reads are whole segments (a thread reading its own link touches 32 segments
// per request), and the 32 sites of one parity are written as whole segments
// of each plane.  Bound by HBM: 24^3x48 into DF64, FP32, 16-bit and the two
// 12-real copies moves 2.5 GB in 367 us, 6.8 TB/s (2.2 ms in one launch per
// copy with a thread reading its own link).  Plain stores: copies that fit the L2
// wait there for the first application (D_oe and D_eo on new 12-real FP32 links
// at 120960 sites 52 us, 59 with streaming stores, which move no less).
constexpr int FOLD_BLOCK = 128;
constexpr int FOLD_LINKS = 64;

__global__ void __launch_bounds__(FOLD_BLOCK)
fold_kernel(const __grid_constant__ FoldArgs fa, const double *__restrict__ fat, const double *__restrict__ lng) {
    __shared__ double2 tile[FOLD_BLOCK / 32][FOLD_LINKS * 9];
    const Geom &g = fa.g;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long V = 2LL * g.Vh;
    const int kind = blockIdx.y, mu = kind & 3;
    const bool three = kind >= 4;
    const long long i0 = (blockIdx.x * (FOLD_BLOCK / 32LL) + w) * FOLD_LINKS;
    if (i0 >= V)
        return;
    const double2 *src = (const double2 *)(three ? lng : fat) + ((size_t)mu * V + i0) * 9;
    const int nl = (int)(V - i0 < FOLD_LINKS ? V - i0 : FOLD_LINKS);
#pragma unroll
    for (int k = 0; k < FOLD_LINKS * 9 / 32; k++)
        if (k * 32 + lane < nl * 9)
            copy16_async(&tile[w][k * 32 + lane], src + k * 32 + lane);
    copy_async_wait();
    __syncwarp();
    if (2 * lane >= nl)  // V is even: links 2 lane and 2 lane + 1 exist together
        return;
    // links 2 lane and 2 lane + 1: the same checkerboard index, one site of each parity
    const size_t cb = (size_t)(i0 >> 1) + lane, S = (size_t)g.stride;
    const int s = three ? 3 : 1;
    const float inv = fa.inv_scale[three ? 1 : 0];
    const int mask = fa.out.mask;
    const bool c12 = (mask >> (three ? 1 : 0)) & 1;  // this kind's form in the copies with 12-real kinds
#pragma unroll 1
    for (int par = 0; par < 2; par++) {
        int x[4];
        cb_coords(g, (int)cb, par, x);
        const int eta_sum = (mu > 0 ? x[0] : 0) + (mu > 1 ? x[1] : 0) + (mu > 2 ? x[2] : 0);
        const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
        const int wraps = (xm + s) / g.L[mu];
        double coef = three ? fa.c3 : fa.c1;
        if (eta_sum & 1)
            coef = -coef;
        if ((wraps & 1) && fa.bc[mu] < 0)
            coef = -coef;
        const double2 *L = &tile[w][(2 * lane + (x[0] & 1)) * 9];
        const size_t half = link_parity_bytes(P_F64, 0, S);  // one parity of the FP64 copy
        const size_t at = (size_t)kind * 9 * S + cb;
        float2 f[9];
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const double2 v = L[e];
            const double re = coef * v.x, im = coef * v.y;
            if (fa.out.full[P_F64])
                *((double2 *)((char *)fa.out.full[P_F64] + par * half) + at + e * S) = make_double2(re, im);
            const df dr = df_split(re), di = df_split(im);
            if (fa.out.full[P_DF64])
                *((float4 *)((char *)fa.out.full[P_DF64] + par * half) + at + e * S) = make_float4(dr.hi, dr.lo, di.hi, di.lo);
            f[e] = make_float2(dr.hi, di.hi);
        }
        if (fa.out.full[P_F32])
#pragma unroll
            for (int e = 0; e < 9; e++)
                *((float2 *)((char *)fa.out.full[P_F32] + par * (half / 2)) + at + e * S) = f[e];
        if (fa.out.c12[P_F32]) {
            char *kb = (char *)fa.out.c12[P_F32] + par * link_parity_bytes(P_F32, mask, S) +
                       link_kind_offset(P_F32, mask, kind, S);
            if (c12) {
#pragma unroll
                for (int k = 0; k < 3; k++)
                    *((float4 *)kb + k * S + cb) = make_float4(f[2 * k].x, f[2 * k].y, f[2 * k + 1].x, f[2 * k + 1].y);
            } else {
#pragma unroll
                for (int e = 0; e < 9; e++)
                    *((float2 *)kb + e * S + cb) = f[e];
            }
        }
        if (!fa.out.full[P_F16])
            continue;
        int q[9];
#pragma unroll
        for (int e = 0; e < 9; e++)
            q[e] = q16_pair(f[e].x * inv, f[e].y * inv);
#pragma unroll
        for (int copy = 0; copy < 2; copy++) {
            char *base = (char *)(copy ? fa.out.c12[P_F16] : fa.out.full[P_F16]);
            if (!base)
                break;
            const int m = copy ? mask : 0;
            char *kb = base + par * link_parity_bytes(P_F16, m, S) + link_kind_offset(P_F16, m, kind, S);
            *((int4 *)kb + cb) = make_int4(q[0], q[1], q[2], q[3]);
            if (copy && c12) {
                *((int2 *)(kb + 16 * S) + cb) = make_int2(q[4], q[5]);
            } else {
                *((int4 *)(kb + 16 * S) + cb) = make_int4(q[4], q[5], q[6], q[7]);
                *((int *)(kb + 32 * S) + cb) = q[8];
            }
        }
    }
}

cudaError_t launch_fold_links(const Geom &g, const double bc[4], double c1, double c3, const double *fat,
                              const double *lng, const FoldOut &out, const float inv_scale[2], cudaStream_t s) {
    FoldArgs fa;
    fa.g = g;
    for (int k = 0; k < 4; k++)
        fa.bc[k] = bc[k];
    fa.c1 = c1;
    fa.c3 = c3;
    fa.inv_scale[0] = inv_scale[0];
    fa.inv_scale[1] = inv_scale[1];
    fa.out = out;
    const int per = FOLD_BLOCK / 32 * FOLD_LINKS;
    const dim3 grid((unsigned)((2LL * g.Vh + per - 1) / per), 8);
    fold_kernel<<<grid, FOLD_BLOCK, 0, s>>>(fa, fat, lng);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// three-link products (FP64): N_mu(x) = U_mu(x) U_mu(x+mu) U_mu(x+2mu)
// --------------------------------------------------------------------------
STAG_D void mat_mul_c(double2 C[9], const double2 A[9], const double2 B[9]) {
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) {
            double re = 0.0, im = 0.0;
            for (int k = 0; k < 3; k++) {
                const double2 x = A[3 * a + k], y = B[3 * k + b];
                re = fma(x.x, y.x, re);
                re = fma(-x.y, y.y, re);
                im = fma(x.x, y.y, im);
                im = fma(x.y, y.x, im);
            }
            C[3 * a + b] = make_double2(re, im);
        }
}

__global__ void long_links_kernel(Geom g, const double2 *__restrict__ U, double2 *__restrict__ N) {
    const long long V = 2LL * g.Vh;
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= 4 * V)
        return;
    const int mu = (int)(t / V);
    const long long i = t % V;
    int x[4];
    full_coords(g, i, x);
    long long step = 1;
    for (int nu = 0; nu < mu; nu++)
        step *= g.L[nu];
    const int L = g.L[mu];
    const long long i1 = i + ((x[mu] + 1) % L - x[mu]) * step;
    const long long i2 = i + ((x[mu] + 2) % L - x[mu]) * step;
    double2 A[9], B[9], T[9];
    for (int j = 0; j < 9; j++) {
        A[j] = U[((size_t)mu * V + i) * 9 + j];
        B[j] = U[((size_t)mu * V + i1) * 9 + j];
    }
    mat_mul_c(T, A, B);
    for (int j = 0; j < 9; j++)
        B[j] = U[((size_t)mu * V + i2) * 9 + j];
    mat_mul_c(A, T, B);
    for (int j = 0; j < 9; j++)
        N[((size_t)mu * V + i) * 9 + j] = A[j];
}

cudaError_t launch_long_links(const Geom &g, const double *fat, double *lng, cudaStream_t s) {
    const long long n = 8LL * g.Vh;
    const int grid = (int)((n + 127) / 128);
    long_links_kernel<<<grid, 128, 0, s>>>(g, (const double2 *)fat, (double2 *)lng);
    return cudaGetLastError();
}

}  // namespace stag
