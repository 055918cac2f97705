// Deterministic block and grid reductions.
//
// Each block reduces its threads' values with warp shuffles and shared
// memory in a fixed tree, writes one FP64 partial, and takes a ticket; the
// block that draws the last ticket sums all partials in a fixed order.  The
// result therefore does not depend on block scheduling.
//
// Inside a block the tree runs in the thread values' reduction type: FP64
// for the FP64 path, double-float (about 48 bits, FP32 pipe) for the others.
// GB300's FP64 pipe runs at 1/64 of the FP32 rate, and an FP64 shuffle tree
// in every thread of a 5M-site reduction costs tens of microseconds; in
// double-float it costs a few, and only thread 0 of each block converts its
// result to FP64.
#pragma once
#include "common.cuh"

namespace stag {

// reduction type of per-thread values computed in arithmetic type R
template <class R> struct RedType { using type = df; };
template <> struct RedType<double> { using type = double; };
template <class R> using red_t = typename RedType<R>::type;

template <class T> STAG_D T red_zero();
template <> STAG_D double red_zero<double>() { return 0.0; }
template <> STAG_D df red_zero<df>() { return df_zero(); }

STAG_D double red_add(double a, double b) { return a + b; }
STAG_D df red_add(df a, df b) { return df_add(a, b); }
STAG_D double red_to_double(double a) { return a; }
STAG_D double red_to_double(df a) { return df_to_double(a); }

STAG_D double shfl_down(double v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
STAG_D df shfl_down(df v, int o) {
    return df_make(__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o));
}

// Sum over the block; the FP64 result is valid in thread 0 only (0 elsewhere).
// smem: 32 doubles of shared memory.
template <int BLOCK, class T> STAG_D double block_sum(T v, double *smem) {
    static_assert(BLOCK % 32 == 0 && BLOCK <= 1024, "block size");
    static_assert(sizeof(T) <= sizeof(double), "reduction type");
    T *ts = reinterpret_cast<T *>(smem);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = red_add(v, shfl_down(v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        ts[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < BLOCK / 32 ? ts[lane] : red_zero<T>();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            v = red_add(v, shfl_down(v, o));
    }
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        r = red_to_double(v);
    return r;
}

// This thread's share of the sum of n partials of stride `step` that other
// blocks wrote: a fixed assignment to BLOCK threads, U loads in flight
// (one after the other, the last block of a 4096-block reduction waited 16
// L2 latencies).  A warp past n skips its adds: an FP64 add costs its
// scheduler 64 cycles also when it adds nothing.
template <int BLOCK, int U = 8> STAG_D double partials_share(const double *__restrict__ v, int n, int step = 1) {
    if (n <= BLOCK)
        return (int)threadIdx.x < n ? __ldcg(v + (size_t)threadIdx.x * step) : 0.0;
    double a = 0.0;
    for (int base = threadIdx.x & ~31; base < n; base += U * BLOCK) {
        double t[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = base + u * BLOCK + (threadIdx.x & 31);
            t[u] = i < n ? __ldcg(v + (size_t)i * step) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (base + u * BLOCK < n)
                a += t[u];
    }
    return a;
}

// Grid-wide sum.  Every thread of every block must call it.  Returns true in
// all threads of the one block that finishes last; there `total` holds the
// grid sum (in every thread).  `ticket` must be zero on entry and is reset to
// zero by the last block.
template <int BLOCK, class T>
STAG_D bool grid_sum(T v, double *partial, unsigned *ticket, double *smem, double &total) {
    __shared__ bool last;
    const double s = block_sum<BLOCK>(v, smem);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = s;
        __threadfence();
        unsigned t = atomicAdd(ticket, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last)
        return false;
    __threadfence();
    const double acc = block_sum<BLOCK>(partials_share<BLOCK, 4>(partial, (int)gridDim.x), smem);
    if (threadIdx.x == 0) {
        smem[0] = acc;
        *ticket = 0u;
    }
    __syncthreads();
    total = smem[0];
    __syncthreads();
    return true;
}

// Blocks of a vector kernel that ends in grid_sum: at most eight per SM, each
// thread then takes several sites.  With one site per thread a block spends
// as long on its fence and ticket as on its loads (16-bit update at 1048576
// sites: 25 us, now 21; a mixed solve on 48^3x96 598 -> 583 ms).  Not where
// some threads would take two sites and most one (331776 sites: 19.3 -> 20.4).
constexpr int SUM_BLOCKS = 8 * kSMs;
inline int sum_grid(int n, int block) {
    const int need = (n + block - 1) / block;
    return need <= 2 * SUM_BLOCKS ? need : SUM_BLOCKS;
}

}  // namespace stag
