// Dispatch of the Dslash launchers over precisions.
#include "dslash_split.cuh"
#include "kernels.h"

namespace stag {

template <int P> cudaError_t launch_dslash_p(int epi, const DslashArgs &a, int block, cudaStream_t s);
extern template cudaError_t launch_dslash_p<P_F64>(int, const DslashArgs &, int, cudaStream_t);
extern template cudaError_t launch_dslash_p<P_DF64>(int, const DslashArgs &, int, cudaStream_t);
extern template cudaError_t launch_dslash_p<P_F32>(int, const DslashArgs &, int, cudaStream_t);
extern template cudaError_t launch_dslash_p<P_F16>(int, const DslashArgs &, int, cudaStream_t);

int dslash_default_block(int prec) {
    (void)prec;
    return 128;
}

// Where the split form (dslash_split.cuh) is the faster one, by measurement
// (microseconds of one plain-CG iteration, in FP32 of a mixed one; split
// against one thread per site, at sites per parity):
//   double-float  2048: 24.5 / 55, 46080: 58 / 69, 65536: 67.2 / 71.4, 73728:
//                 78.9 / 76.0, 98304: 97.2 / 93.5, 114688: 109.0 / 101.4,
//                 128000: 125 / 148, 331776: 298 / 305, 1048576: 891 / 894,
//                 3538944: 2930 / 2898; one thread per site, 768 threads per
//                 SM, takes one wave up to 116736 sites
//   FP64          2048: 34 / 60, 20736: 74 / 97, 32768: 94 / 97, 46080: 126 / 140,
//                 96000: 229 / 221, 1048576: 2230 / 2128; single calls lose 4 % at 50000
//   FP32 full     40960: 41.0 / 38.8, 49152: 43.3 / 43.8, 65536: 47.1 / 48.1,
//                 73728: 54.5 / 50.8, 81920: 59.9 / 55.6; a single D_oe or M,
//                 whose links nothing keeps in L2, 49152: 11.8 / 12.2, 22.0 /
//                 23.0, 57344: 13.0 / 13.4, 24.1 / 24.9, 65536: equal kernels,
//                 an M every 21.0 / 20.3; 81920: 18.2 / 16.9, 36.5 / 33.8; the
//                 vectors of several training pairs in one launch against one
//                 by one, a gradient of eight pairs 73728: 1007 / 1098, 81920:
//                 1187 / 1279
//   FP32 12-real  20736: 12 / 14 (all), 12 / 16 (three-link), D_oe and D_eo; 32768:
//                 16.5 / 15, 16.5 / 16.5
// Eight warps per 32 sites on the smallest lattices (double float, 2048
// sites: 24.5 against 27; 10368: 31.6 against 34; 20736: 41.6 against 39.6).
// The 16-bit stencil has no split form.
int split_warps(int prec, const DslashArgs &a) {
    const int Vh = a.g.Vh;
    bool split = false;
    switch (prec) {
    case P_DF64: split = Vh <= 70000 || (Vh > 768 * kSMs && Vh <= 400000); break;
    case P_F64: split = Vh <= 36000; break;
    case P_F32: split = Vh <= (a.compressed ? 24576 : a.nbatch > 0 ? 85000 : a.keep > 0 ? 70000 : 60000); break;
    }
    return !split ? 0 : Vh <= 16384 ? 8 : 4;
}

// Links kept in L2 from one launch to the next in a solve (each launch reads
// every link of both parities): the rest is evicted first, so that the kept
// ones and the vectors stay.  32 MB of the 129 MB L2 measured best or equal
// (an iteration of plain CG in double float at 46080 sites per parity 65 ->
// 58 us, at 80000 93.5 -> 87; of mixed CG in FP32 on 12-real links at 80000
// 59.9 -> 52.8, 128000: 69 -> 66; 64 MB and more were slower again).  A
// single call keeps none (stag_dslash_*, stag_apply_M: its caller may well be
// working on several lattices in turn; three of them at 120960 sites on
// 12-real links: 28.8 against 27.8 us a pair of Dslash calls; M in FP32 at
// 112000 sites 37.7 against 35.6 us, 331776: 112.1 against 110.1).  The
// kernels that load with LD_STREAM ignore it.
int link_keep_sites(int prec, int compressed) {
    const size_t site = 2 * link_parity_bytes(prec, compressed, 256) / 256;  // both parities' links
    return (int)((32u << 20) / site);
}

int dslash_blocks(int prec, int epi, const DslashArgs &a, int block) {
    if (pair16_used(prec, epi, a, block))
        return dslash_pair16_grid(a.g, block);
    const int n = (a.cn ? a.cn : a.g.Vh) + (a.cn ? a.cnb : 0);
    const int sites = split_warps(prec, a) > 0 ? SPLIT_SITES : block;
    return (n + sites - 1) / sites;
}

cudaError_t launch_dslash(int prec, int epi, const DslashArgs &a, int block, cudaStream_t s) {
    if (block <= 0)
        block = dslash_default_block(prec);
    switch (prec) {
    case P_F64: return launch_dslash_p<P_F64>(epi, a, block, s);
    case P_DF64: return launch_dslash_p<P_DF64>(epi, a, block, s);
    case P_F32: return launch_dslash_p<P_F32>(epi, a, block, s);
    case P_F16: return launch_dslash_p<P_F16>(epi, a, block, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace stag
