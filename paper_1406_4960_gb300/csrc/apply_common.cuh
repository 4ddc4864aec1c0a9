// Launch descriptors shared by the apply kernels.
#pragma once

#include "cplx.cuh"

namespace mb {

constexpr int kMaxK = 64;   // k-points per launch (descriptors travel as kernel parameters)
constexpr int kMaxChunks = 64;   // runs of knot intervals or rows per (k, band) in the plane kernels

// First knot interval (or row) of run c when nint of them are split into
// nchunks runs of balanced length (lengths differ by at most one).
__host__ __device__ inline int chunk_begin(int c, int nint, int nchunks) {
    return (int)(((long long)c * nint) / nchunks);
}

struct KDesc {
    const void *X;
    void *Y;
    void *part;      // boundary partial rows
    void *W;         // projector overlaps: Zx[b][f][G] (CUDA-core path) or W[(b, j)][p] (tensor cores)
    void *C;         // projector coefficients: c[b][p] (CUDA-core path) or C[(b, j)][p] (tensor cores)
    int ng, ldg;
    int kofs;        // offset of per-k G arrays
    int qofs;        // offset of q_p(G) table
};

template <typename R> struct PlaneArgs {
    const R *Bq;
    const R *V;       // bit-reversed layout
    const typename V2<R>::T *tw;
    const int *goff;
    int n1, n2, l1, l2, nmax;
    int order, nquad, nint, nb;
    int nbands, nchunks, np;
    KDesc d[kMaxK];
};

}  // namespace mb
