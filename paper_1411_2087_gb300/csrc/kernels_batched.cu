// Dispatch of the batched CG kernels over precision, block size and group
// size (the kernels are in batched_kernels.cuh, instantiated in
// batched_<prec>.cu so that the precisions compile in parallel).
#include "batched.cuh"
#include "kernels.h"

namespace stag {

template <int P, int BLOCK, int K> cudaError_t launch_batch_pbk(int what, const BatchArgs &a, cudaStream_t s);
#define STAG_BATCH_EXTERN(P, B, K) \
    extern template cudaError_t launch_batch_pbk<P, B, K>(int, const BatchArgs &, cudaStream_t);
STAG_BATCH_EXTERN(P_F32, 128, 4)
STAG_BATCH_EXTERN(P_F32, 128, 8)
STAG_BATCH_EXTERN(P_F32, 256, 4)
STAG_BATCH_EXTERN(P_F32, 256, 8)
STAG_BATCH_EXTERN(P_DF64, 128, 4)
STAG_BATCH_EXTERN(P_DF64, 256, 4)
STAG_BATCH_EXTERN(P_F64, 128, 4)
STAG_BATCH_EXTERN(P_F64, 256, 4)
#undef STAG_BATCH_EXTERN

// right-hand sides per group: FP32 keeps K vectors per thread (kernels for
// K = 4 and 8), double float and FP64 map one thread to one (site, system)
// pair (K = 2 or 4 lanes share a link load; one kernel serves both)
int batch_max_k(int prec) { return prec == P_F32 ? 8 : 4; }
int batch_min_k(int prec) { return prec == P_F32 ? 4 : 2; }

// An iteration in split form against one thread per (site, system): double
// float 4096 items 35 / 50 us, 27648: 51 / 60, 61440: 83.8 / 86.4, 65536: 92.2
// / 92.8, 73728: 94.3 / 88.0, 98304: 117.7 / 113.3; FP64 4096: 44 / 82, 41472:
// 132 / 154, 61440: 172 / 193, 65536: 190 / 202, 73728: 204 / 196, 81920: 225 /
// 245, 98304: 264 / 284, 114688: 288 either way.  (FP64 at 73728: the split form
// is past two waves of 1064 blocks of 32 items, the other within one of 608
// blocks of 128.)
bool batch_split(int prec, long long items) {
    switch (prec) {
    case P_DF64: return items <= 70000;
    case P_F64: return items <= 2 * 7 * 32 * kSMs || (items > 4 * 128 * kSMs && items <= 100000);
    default: return false;
    }
}

cudaError_t launch_batch(int prec, int what, const BatchArgs &a, int block, cudaStream_t s) {
    if (block != 128 && block != 256)
        return cudaErrorInvalidValue;
    const bool b128 = block == 128;
    switch (prec) {
    case P_F32:
        if (a.kmax <= 4)
            return b128 ? launch_batch_pbk<P_F32, 128, 4>(what, a, s) : launch_batch_pbk<P_F32, 256, 4>(what, a, s);
        return b128 ? launch_batch_pbk<P_F32, 128, 8>(what, a, s) : launch_batch_pbk<P_F32, 256, 8>(what, a, s);
    case P_DF64:
        return b128 ? launch_batch_pbk<P_DF64, 128, 4>(what, a, s) : launch_batch_pbk<P_DF64, 256, 4>(what, a, s);
    case P_F64:
        return b128 ? launch_batch_pbk<P_F64, 128, 4>(what, a, s) : launch_batch_pbk<P_F64, 256, 4>(what, a, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace stag
