// Local potential through row space (§II.B.1, Eqs. (12)-(13), (19)-(20)).
//
// Per in-plane grid point r the local potential acts on the B-spline
// coefficients alone: with x_j(r) the inverse 2D transform of coefficient row
// j,
//     (V x)_i(r) = sum_q B_i(z_q) w_q V(r, z_q) sum_j B_j(z_q) x_j(r)
//                = sum_j U_ij(r) x_j(r),   U_ij(r) = sum_q w_q B_i B_j V(r, z_q),
// a symmetric band of half-width kappa - 1.  U is built once per potential
// (rs_tables_kernel in vloc.cu), so one inverse and one forward transform per
// B-spline row replace one pair per Gauss plane (nquad per knot interval,
// about six times as many).
//
// A CTA takes a run of the rows of all k-points and bands (a piece of a band,
// or the end of one, whole ones and the beginning of another, so that every
// CTA of one round has the same work) and walks each band's rows in steps of RR, on RR planes in shared memory and five more for the history:
//   A  the step's coefficient rows onto compact planes (the disc's occupied
//      rows and columns only: a cyclic shift of the frequency index along an
//      axis is a phase in real space, which commutes with the real U);
//   B  inverse transforms along axis 2, C along axis 1, one line per thread
//      in registers;
//   D  the band along z: a thread owns fixed grid points, keeps five partial
//      sums in registers, reads the five rows before the step from the
//      history (and leaves it the step's last five), and writes output row
//      m - 5 over input row m;
//   E, F  forward transforms of the finished rows, G their disc to Y.
// Runs recompute the transforms of the 5 + 5 rows that their neighbours own,
// so every output row has one writer and one summation order.
//
// Discs that fit in 3/4 of both sides of the plane (every cell's, on a grid
// of at least 2 n_max + 1 points) take the pruned instance: compact planes of
// 3/4 x 3/4 entries, with the butterflies of the zero inputs and of the
// unused outputs left out.
//
// Grid sides of 64 are folded: real-space points i = 2 m + c are split by
// residue c over the CTAs of a cluster (2 or 4), each transforming planes of
// at most 32 x 32 after multiplying the disc by the residue's phases (a
// decimation in time); the residues' outputs are added in residue order from
// the cluster's shared memory.
//
// Bounds and measurements (GB300).  FP64: the FP64 pipe (two FMAs a clock and
// SM); per grid point and row about 37 instructions of transforms and 22 of
// the band.  FP32: shared-memory traffic (the line transforms' exchanges) and
// latency at 16 warps per SM, which 128 registers a thread leave.  Against
// one transform pair per Gauss plane (the compact-plane and register-FFT
// kernels that this one replaced), per launch:
//   slab, 4 k x 32 bands     FP32 0.155 -> 0.055 ms   FP64 4.38 -> 1.00 ms
//   graphene, 80 bands       FP32 0.868 -> 0.27 ms    FP64 42 -> 4.64 ms
//   64 k x 24 bands          FP32 3.48 -> 0.81 ms
// A line in one thread's registers sets the 32-point limit (64 FP32
// registers); RR = 16 rows a step make one line per thread and keep the
// 5-row halo small; 64-bit accesses to rows padded by one entry are free of
// bank conflicts along both axes.  Two or four bands per CTA (sharing the
// loads of U) and 8-row steps with twice the CTAs measured the same or slower.
#pragma once

#include <algorithm>
#include <cstdint>
#include <cstdio>

#include "fft_reg.cuh"
#include "mb_internal.h"
#include "rowspace.h"

namespace mb {

__device__ __forceinline__ void rs_cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void rs_cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t rs_mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ float2 rs_ld_cluster(uint32_t addr, float2) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ double2 rs_ld_cluster(uint32_t addr, double2) {
    double2 v;
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr));
    return v;
}

// Plane layout: [M2 rows of axis 2][M1 points of axis 1, padded by one].
template <typename R, int M1, int M2, int RR, bool PR> struct RsGeom {
    static constexpr int N1 = PR ? M1 * 3 / 4 : M1, N2 = PR ? M2 * 3 / 4 : M2;   // compact plane
    static constexpr int LDP = M1 + 1, PS = M2 * LDP;
    static constexpr size_t smem = (size_t)(RR * PS + kRsHalo * M1 * M2) * sizeof(typename V2<R>::T);
};

// transforms along axis 1: the N2 compact lines of n planes
template <typename R, int M1, int M2, int T, int RR, bool PR, bool INV>
__device__ __forceinline__ void rs_axis1(typename V2<R>::T *planes, int n) {
    typedef typename V2<R>::T C;
    typedef RsGeom<R, M1, M2, RR, PR> G;
    for (int e = threadIdx.x; e < n * G::N2; e += T) {
        C *line = planes + e * G::LDP + (e / G::N2) * (G::PS - G::N2 * G::LDP);
        C v[M1];
#pragma unroll
        for (int r = 0; r < M1; ++r) v[r] = (!INV || r < G::N1) ? line[r] : czero<C>();
        fft_reg<M1, INV, INV ? G::N1 : M1>(v);
#pragma unroll
        for (int r = 0; r < M1; ++r)
            if (INV || r < G::N1) line[r] = v[r];
    }
}

// transforms along axis 2: the M1 lines of n planes
template <typename R, int M1, int M2, int T, int RR, bool PR, bool INV>
__device__ __forceinline__ void rs_axis2(typename V2<R>::T *planes, int n) {
    typedef typename V2<R>::T C;
    typedef RsGeom<R, M1, M2, RR, PR> G;
    for (int e = threadIdx.x; e < n * M1; e += T) {
        C *line = planes + (e / M1) * G::PS + e % M1;
        C v[M2];
#pragma unroll
        for (int p = 0; p < M2; ++p) v[p] = (!INV || p < G::N2) ? line[p * G::LDP] : czero<C>();
        fft_reg<M2, INV, INV ? G::N2 : M2>(v);
#pragma unroll
        for (int p = 0; p < M2; ++p)
            if (INV || p < G::N2) line[p * G::LDP] = v[p];
    }
}

// element of a row block at a 32-bit byte offset (the base is uniform)
template <typename C> __device__ __forceinline__ const C &rs_at(const void *base, unsigned off) {
    return *reinterpret_cast<const C *>(reinterpret_cast<const char *>(base) + off);
}
template <typename C> __device__ __forceinline__ C &rs_at(void *base, unsigned off) {
    return *reinterpret_cast<C *>(reinterpret_cast<char *>(base) + off);
}

template <typename R, int M1, int M2, int T, int RR, int GR, int CTAS, bool PR, bool FOLD>
__global__ void __launch_bounds__(T, CTAS) rowspace_kernel(const __grid_constant__ RsArgs<R> a) {
    typedef typename V2<R>::T C;
    typedef RsGeom<R, M1, M2, RR, PR> G;
    constexpr int H = kRsHalo, NP = M1 * M2, PPT = NP / T;
    static_assert(NP % T == 0 && RR % GR == 0 && RR >= H, "whole points and row groups per thread");
    extern __shared__ __align__(16) unsigned char rs_smem[];
    C *planes = reinterpret_cast<C *>(rs_smem);       // [RR][M2][LDP]
    C *hist = planes + RR * G::PS;                    // [H][NP]: x of the five rows before the step
    const int tid = threadIdx.x;
    const int S = FOLD ? a.s1 * a.s2 : 1;
    const int rank = FOLD ? (int)(blockIdx.x % (unsigned)S) : 0;
    const int w = FOLD ? (int)(blockIdx.x / (unsigned)S) : (int)blockIdx.x, nb = a.nb;
    const int rbeg = rs_cut(w, a.num, a.den, nb, a.snap), rend = rs_cut(w + 1, a.num, a.den, nb, a.snap);
    for (int r = rbeg; r < rend;) {
    const bool first = r == rbeg;
    const int kb = r / nb, b = kb % a.nbands;
    const RsK &d = a.d[kb / a.nbands];
    const int ldg = d.ldg;
    const int j0 = r - kb * nb, j1 = min(nb, j0 + rend - r);      // output rows
    const int ji = max(0, j0 - H), je = min(nb, j1 + H);          // rows transformed
    r += j1 - j0;
    if (!FOLD && !first) __syncthreads();                         // the last band's planes are read
    const C *X = reinterpret_cast<const C *>(d.X) + (size_t)b * nb * ldg;
    C *Y = reinterpret_cast<C *>(d.Y) + (size_t)b * nb * ldg;
    const unsigned xrow = (unsigned)(ldg * sizeof(C));               // bytes per coefficient row
    const unsigned urow = (unsigned)(S * NP * sizeof(C));            // bytes per pair of the potential band

    C acc[PPT][H];                    // acc[q][k]: partial sum of row m - 5 + k at point q
#pragma unroll
    for (int q = 0; q < PPT; ++q)
#pragma unroll
        for (int k = 0; k < H; ++k) {
            acc[q][k] = czero<C>();
            hist[k * NP + tid + q * T] = czero<C>();                 // read back by this thread only
        }

    C xv[FOLD ? 1 : RR];              // coefficient rows a0 .. a0 + RR - 1 of one G
    auto load_x = [&](int a0, int g) {
        if constexpr (!FOLD) {
            const int nin = min(RR, je - a0);
            const C *Xa = X + (size_t)a0 * ldg;
            unsigned off = (unsigned)(g * sizeof(C));
            if (g >= d.ng) return;
#pragma unroll
            for (int i = 0; i < RR; ++i, off += xrow)
                if (i < nin) xv[i] = rs_at<C>(Xa, off);
        }
    };
    for (int a0 = ji; a0 < j1 + H; a0 += RR) {
        const int nin = max(0, min(RR, je - a0));
        // A
        if constexpr (!FOLD) {
            if (a0 == ji) load_x(a0, tid);
            for (int g = tid; g < d.ng; g += T) {
                if (g >= T) load_x(a0, g);
                C *dst = planes + __ldg(a.gpos + d.gofs + g);
#pragma unroll
                for (int i = 0; i < RR; ++i)
                    if (i < nin) dst[i * G::PS] = xv[i];
            }
            for (int e = tid; e < d.npos; e += T) {                  // the compact plane's disc-free positions
                C *dst = planes + __ldg(a.pos + d.pofs + e);
#pragma unroll
                for (int i = 0; i < RR; ++i) dst[i * G::PS] = czero<C>();
            }
        } else {
            const C *phase = a.phase + rank * a.phase_stride + d.gofs;
            const C *Xa = X + (size_t)a0 * ldg;
#pragma unroll
            for (int u = 0; u < PPT; ++u) {
                const int e = tid + u * T;                           // axis 1 fastest
                C *dst = planes + (e / M1) * G::LDP + e % M1;
                const int4 p4 = __ldg(a.src + d.pofs + e);
                C v[RR];
#pragma unroll
                for (int i = 0; i < RR; ++i) v[i] = czero<C>();
#pragma unroll 1
                for (int s = 0; s < 4; ++s) {
                    const int g = s == 0 ? p4.x : s == 1 ? p4.y : s == 2 ? p4.z : p4.w;
                    if (g < 0) break;
                    const C ph = phase[g];
                    unsigned off = (unsigned)(g * sizeof(C));
                    if (nin == RR) {
#pragma unroll
                        for (int i = 0; i < RR; ++i, off += xrow) cfma(v[i], ph, rs_at<C>(Xa, off));
                    } else {
#pragma unroll
                        for (int i = 0; i < RR; ++i, off += xrow)
                            if (i < nin) cfma(v[i], ph, rs_at<C>(Xa, off));
                    }
                }
                if (u == 0 && !(first && a0 == ji)) rs_cluster_wait();            // the other residues have read this CTA's planes
#pragma unroll
                for (int i = 0; i < RR; ++i) dst[i * G::PS] = v[i];
            }
        }
        __syncthreads();
        rs_axis1<R, M1, M2, T, RR, PR, true>(planes, nin);
        __syncthreads();
        rs_axis2<R, M1, M2, T, RR, PR, true>(planes, nin);
        const char *ub = reinterpret_cast<const char *>(a.U) + (size_t)a0 * (3 * urow);
        C un[GR][3];                  // potential of the next GR rows at one point
        auto load_u = [&](int q, int i0) {
            unsigned uo = (unsigned)((rank * NP + tid + q * T) * sizeof(C)) + (unsigned)(3 * i0) * urow;
#pragma unroll
            for (int i = 0; i < GR; ++i)
#pragma unroll
                for (int t = 0; t < 3; ++t, uo += urow) un[i][t] = rs_at<C>(ub, uo);
        };
        load_u(0, 0);
        // rows past the basis enter the band as zeros
        for (int i = nin; je == nb && i < min(RR, nb + H - a0); ++i)
            for (int e = tid; e < G::PS; e += T) planes[i * G::PS + e] = czero<C>();
        __syncthreads();
        // D: GR rows of one point at a time, the next group's potential in flight
        // during the products (the first group's since before the barrier)
#pragma unroll
        for (int q = 0; q < PPT; ++q) {
            const int pt = tid + q * T;
            C *x = planes + (pt / M1) * G::LDP + pt % M1;
            C h[H + GR];              // h[k]: x of row a0 + i0 - 5 + k
#pragma unroll
            for (int k = 0; k < H; ++k) h[k] = hist[k * NP + pt];
#pragma unroll
            for (int i0 = 0; i0 < RR; i0 += GR) {
                if (sizeof(R) == 8 && a0 + i0 >= j1 + H) {            // the run ends inside the step
                    if (q + 1 < PPT) load_u(q + 1, 0);
                    break;
                }
                C u[GR][3];
#pragma unroll
                for (int i = 0; i < GR; ++i)
#pragma unroll
                    for (int t = 0; t < 3; ++t) u[i][t] = un[i][t];
                if (i0 + GR < RR) load_u(q, i0 + GR);
                else if (q + 1 < PPT) load_u(q + 1, 0);
#pragma unroll
                for (int i = 0; i < GR; ++i) h[H + i] = x[(i0 + i) * G::PS];
#pragma unroll
                for (int i = 0; i < GR; ++i) {
                    const C xm = h[i + H];
                    // FP64: only the products that reach a row of this run (a
                    // branch is nothing beside the FP64 pipe's 64 clocks a warp)
                    const int m = a0 + i0 + i;
                    auto live = [&](int row) { return sizeof(R) == 4 || (row >= j0 && row < j1); };
                    C y = acc[q][0];
                    if (live(m - 5)) rfma(y, u[i][2].y, xm);
                    acc[q][0] = acc[q][1];
                    if (live(m - 4)) rfma(acc[q][0], u[i][2].x, xm);
                    acc[q][1] = acc[q][2];
                    if (live(m - 3)) rfma(acc[q][1], u[i][1].y, xm);
                    acc[q][2] = acc[q][3];
                    if (live(m - 2)) rfma(acc[q][2], u[i][1].x, xm);
                    acc[q][3] = acc[q][4];
                    if (live(m - 1)) rfma(acc[q][3], u[i][0].y, xm);
                    if (live(m)) {
                        C n = rscale(u[i][2].y, h[i]);
                        rfma(n, u[i][2].x, h[i + 1]);
                        rfma(n, u[i][1].y, h[i + 2]);
                        rfma(n, u[i][1].x, h[i + 3]);
                        rfma(n, u[i][0].y, h[i + 4]);
                        rfma(n, u[i][0].x, xm);
                        acc[q][4] = n;
                    }
                    x[(i0 + i) * G::PS] = y;
                }
#pragma unroll
                for (int k = 0; k < H; ++k) h[k] = h[k + GR];
            }
#pragma unroll
            for (int k = 0; k < H; ++k) hist[k * NP + pt] = h[k];
        }
        __syncthreads();
        const int jo = max(j0, a0 - H), no = min(j1, a0 + RR - H) - jo;   // finished rows
        C *done = planes + (jo - (a0 - H)) * G::PS;
        if (no > 0) {
            rs_axis2<R, M1, M2, T, RR, PR, false>(done, no);
            __syncthreads();
            rs_axis1<R, M1, M2, T, RR, PR, false>(done, no);
        }
        C *Yo = Y + (size_t)max(jo, 0) * ldg;
        if constexpr (!FOLD) {
            load_x(a0 + RR, tid);      // the next step's rows, in flight during G
            __syncthreads();
            // G (the next step's A writes a G's entries in the thread that reads them here)
            for (int g = tid; g < ldg; g += T) {
                unsigned off = (unsigned)(g * sizeof(C));
                if (g < d.ng) {
                    const C *src = done + __ldg(a.gpos + d.gofs + g);
                    if (no == RR) {
#pragma unroll
                        for (int i = 0; i < RR; ++i, off += xrow) rs_at<C>(Yo, off) = src[i * G::PS];
                    } else {
#pragma unroll 4
                        for (int i = 0; i < no; ++i, off += xrow) rs_at<C>(Yo, off) = src[i * G::PS];
                    }
                } else {
                    for (int i = 0; i < no; ++i, off += xrow) rs_at<C>(Yo, off) = czero<C>();   // padding columns
                }
            }
        } else {
            rs_cluster_arrive();
            rs_cluster_wait();
            // G: this CTA's share of the disc, the residues' parts in order
            const int g0 = rank * ldg / S, g1 = (rank + 1) * ldg / S;
            const uint32_t mine = (uint32_t)__cvta_generic_to_shared(done);
            for (int g = g0 + tid; g < g1 && no > 0; g += T) {
                unsigned off = (unsigned)(g * sizeof(C));
                if (g >= d.ng) {
                    for (int i = 0; i < no; ++i, off += xrow) rs_at<C>(Yo, off) = czero<C>();   // padding columns
                    continue;
                }
                const uint32_t at = mine + (uint32_t)(__ldg(a.gpos + d.gofs + g) * sizeof(C));
                C ph[4];
                uint32_t rem[4];
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s < S) {
                        ph[s] = a.phase[s * a.phase_stride + d.gofs + g];
                        ph[s].y = -ph[s].y;
                        rem[s] = rs_mapa(at, s);
                    }
                if (S == 4) {
#pragma unroll 4
                    for (int i = 0; i < no; ++i, off += xrow) {
                        C y = czero<C>();
#pragma unroll
                        for (int s = 0; s < 4; ++s) cfma(y, ph[s], rs_ld_cluster(rem[s] + i * (uint32_t)(G::PS * sizeof(C)), C()));
                        rs_at<C>(Yo, off) = y;
                    }
                } else {
#pragma unroll 4
                    for (int i = 0; i < no; ++i, off += xrow) {
                        C y = czero<C>();
#pragma unroll
                        for (int s = 0; s < 2; ++s) cfma(y, ph[s], rs_ld_cluster(rem[s] + i * (uint32_t)(G::PS * sizeof(C)), C()));
                        rs_at<C>(Yo, off) = y;
                    }
                }
            }
            rs_cluster_arrive();      // waited for before the planes are written again
        }
    }
    }
    if (FOLD && rbeg < rend) rs_cluster_wait();
}

template <typename R, int M1, int M2, int T, int RR, int GR, int CTAS, bool PR, bool FOLD>
static cudaError_t rs_config(unsigned S, unsigned workers, cudaStream_t s, cudaLaunchConfig_t &cfg, cudaLaunchAttribute &at) {
    constexpr size_t smem = RsGeom<R, M1, M2, RR, PR>::smem;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaError_t e = smem_limit_once((const void *)rowspace_kernel<R, M1, M2, T, RR, GR, CTAS, PR, FOLD>, dev, (int)smem);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(workers * S);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    if (S > 1) {
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = S;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
    }
    return cudaSuccess;
}

template <typename R, int M1, int M2, int T, int RR, int GR, int CTAS, bool PR, bool FOLD>
static cudaError_t rs_launch_one(const RsArgs<R> &a, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at = {};
    const cudaError_t e = rs_config<R, M1, M2, T, RR, GR, CTAS, PR, FOLD>((unsigned)(a.s1 * a.s2), (unsigned)a.workers, s, cfg, at);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, rowspace_kernel<R, M1, M2, T, RR, GR, CTAS, PR, FOLD>, a);
}

template <typename R, int M1, int M2, int T, int RR, int GR, int CTAS>
static cudaError_t rs_launch_shape(const RsArgs<R> &a, cudaStream_t s) {
    if (a.s1 * a.s2 > 1) {
        if constexpr (M1 * M2 > 256) return rs_launch_one<R, M1, M2, T, RR, GR, CTAS, false, true>(a, s);
        else return cudaErrorInvalidValue;
    }
    return a.pruned ? rs_launch_one<R, M1, M2, T, RR, GR, CTAS, true, false>(a, s)
                    : rs_launch_one<R, M1, M2, T, RR, GR, CTAS, false, false>(a, s);
}

// (a cluster's CTAs share a GPC, whose SMs need not be a multiple of it)
template <typename R, int M1, int M2, int T, int RR, int GR, int CTAS>
static int rs_resident_shape(const RsShape &sh, int num_sms) {
    const int S = sh.s1 * sh.s2;
    if constexpr (M1 * M2 > 256) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at = {};
        int n = 0;
        if (S > 1 && rs_config<R, M1, M2, T, RR, GR, CTAS, false, true>((unsigned)S, 1, nullptr, cfg, at) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&n, rowspace_kernel<R, M1, M2, T, RR, GR, CTAS, false, true>, &cfg) == cudaSuccess && n > 0)
            return n;
        if (S > 1) cudaGetLastError();
    }
    return std::max(1, num_sms * CTAS / S);
}

}  // namespace mb
