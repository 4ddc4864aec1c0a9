// FP64 instances of the row-space kernel.
#include "rowspace.cuh"

namespace mb {

// id, plane, threads, rows per step, rows per group of the band phase, CTAs per SM
#define MB_RS64_LIST(X)         \
    X(0, 16, 16, 128, 16, 2, 2) \
    X(1, 16, 32, 256, 16, 2, 1) \
    X(2, 32, 16, 256, 16, 2, 1) \
    X(3, 32, 32, 256, 8, 2, 1)

#define MB_RS_R double
#define MB_RS_NAME "double"
#define MB_RS_LIST MB_RS64_LIST
#include "rowspace_inst.inc"

}  // namespace mb
