// Row-space local potential: host interface (kernels in rowspace.cuh).
#pragma once

#include "cplx.cuh"
#include "apply_common.cuh"
#include "mb_internal.h"

namespace mb {

// one k-point's disc on the (folded) plane
struct RsK {
    const void *X;
    void *Y;
    int ng, ldg;
    int gofs;             // offset of the per-G tables (plane offsets, phases)
    int pofs, npos;       // its position list: disc-free positions, or (folded) the source table
};

template <typename R> struct RsArgs {
    const typename V2<R>::T *U;       // [nb + kRsPad][3][residue][point, axis 1 fastest]: pairs U(j, j - 2t), U(j, j - 2t - 1)
    const int *gpos;                  // plane offset of each G
    const int *pos;                   // unfolded: plane offsets of the compact plane's disc-free positions
    const int4 *src;                  // folded: the up to four G of each plane position (-1: none)
    const typename V2<R>::T *phase;   // folded: [residue][G] exp(2 pi i (c1 n1 / N1 + c2 n2 / N2))
    size_t phase_stride;              // elements from one residue's phases to the next
    int nbands, nb;
    int workers;                      // equal runs of the k-points x bands x nb rows (rs_cut):
    int num, den, snap;               // num / den rows each, in lowest terms
    int s1, s2;                       // folds of the two grid sides
    int pruned;                       // the tables are those of the 3/4 x 3/4 compact plane
    RsK d[kMaxK];
};

// launch shape of one (grid, precision)
struct RsShape {
    bool ok = false;
    int id = -1;
    char name[96] = {0};
    int m1 = 0, m2 = 0, s1 = 1, s2 = 1;
    int threads = 0, rows = 0, ctas_per_sm = 1;   // rows per step
    size_t smem = 0;
};
constexpr int kMaxRsShapes = 4;
template <typename R> int rs_shapes(int n1, int n2, int order, RsShape *out, int max);
template <typename R> cudaError_t rs_launch(const RsArgs<R> &a, const RsShape &sh, cudaStream_t s);
// CTAs (clusters where the grid is folded) of a shape that the device holds at once
template <typename R> int rs_resident(const RsShape &sh, int num_sms);

// Small FP64 problems: a cluster of kRsSmallCl CTAs per (k-point, band), at most
// kRsSmallRows rows each (rowspace64.cu), up to as many CTAs as SMs.  A cluster's
// CTAs share a GPC, and 15 clusters of 8 are resident on 152 SMs: up to 15
// pairs take one round (40 rows: 46 us an apply, 59 to 86 by runs of rows), 16
// to 19 two (80 us; 20 pairs by runs 71).
constexpr int kRsSmallCl = 8, kRsSmallRows = 8;
bool rs_small_supported(const RsShape &sh, int pairs, int nb, int num_sms);
cudaError_t rs_launch_small(const RsArgs<double> &a, unsigned pairs, cudaStream_t s);

// First row of worker w: equal shares of all rows, a share's end moved to the
// next band boundary where that is at most snap rows away.
__device__ __forceinline__ int rs_cut(int w, int num, int den, int nb, int snap) {
    const unsigned long long x = (unsigned long long)w * (unsigned)num;
    const int r = x >> 32 ? (int)(x / (unsigned)den) : (int)((unsigned)x / (unsigned)den), off = r % nb;
    return off <= snap ? r - off : nb - off <= snap ? r + nb - off : r;
}

}  // namespace mb
