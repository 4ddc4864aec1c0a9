// FP32 instances of the row-space kernel.
#include "rowspace.cuh"

namespace mb {

// id, plane, threads, rows per step, rows per group of the band phase, CTAs per SM
#define MB_RS32_LIST(X)         \
    X(0, 16, 16, 128, 16, 4, 4) \
    X(1, 16, 32, 256, 16, 4, 2) \
    X(2, 32, 16, 256, 16, 4, 2) \
    X(3, 32, 32, 512, 16, 4, 1)

#define MB_RS_R float
#define MB_RS_NAME "float"
#define MB_RS_LIST MB_RS32_LIST
#include "rowspace_inst.inc"

}  // namespace mb
