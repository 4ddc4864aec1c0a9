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

// Small FP64 problems: a cluster of kRsSmallCl CTAs per (k-point, band), at
// most RM rows each, instead of runs that transform their neighbours' rows
// again.  A run of two rows transforms twelve, and since a line transform
// holds an FP64 pipe for 64 clocks an operation, its 144 and 192 lines take two
// rounds of the SM's four warps where 8 rows take one (six rounds a CTA
// against four).  Each CTA transforms its own rows to real space, reads the
// five rows on either side from its neighbours' shared memory, keeps the
// band's results in registers until every CTA of the cluster has read, and
// transforms them back.  The band's sums run in rowspace_kernel's order.
// 8 bands of 40 rows: 52 -> 39 us, half of it in the band.
//
// Its lines are 16 points on two neighbouring lanes (the even and the odd
// samples, joined by one exchange), so that the 60 to 128 lines of up to 8
// rows occupy all four pipes: 5.6 k clocks a pass for 9.6 k with a line per
// lane on two warps.
static __constant__ double2 c_w16[8] = {{1.0, 0.0},   {kC2, 0.38268343236508977173},   {kC4, kC4},  {0.38268343236508977173, kC2},
                                        {0.0, 1.0},   {-0.38268343236508977173, kC2},  {-kC4, kC4}, {-kC2, 0.38268343236508977173}};

// 16-point lines `line(l)` (element n at line(l)[n * stride]), l < n: the first
// NIN inputs are read (the others are zero), the first NOUT outputs written
template <int T, bool INV, int NIN, int NOUT, typename Line>
__device__ __forceinline__ void rs_lines16(int n, int stride, Line line) {
    for (int e = threadIdx.x; e < (2 * n + 31) / 32 * 32; e += T) {       // whole warps: the lanes exchange
        const int hf = e & 1;
        double2 *p = line(min(e / 2, n - 1));
        double2 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = 2 * k < NIN ? p[(2 * k + hf) * stride] : czero<double2>();
        __syncwarp();                                  // (a clamped lane reads its line before the owner writes it)
        fft_reg<8, INV, (NIN + 1) / 2>(v);
        double2 out[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            double2 m = v[k];
            if (hf && k > 0) {                         // odd half: times exp(+-2 pi i k / 16)
                const double2 w = c_w16[k];
                m = cmul(v[k], mk(w.x, INV ? w.y : -w.y));
            }
            double2 o;
            o.x = __shfl_xor_sync(0xffffffffu, m.x, 1);
            o.y = __shfl_xor_sync(0xffffffffu, m.y, 1);
            out[k] = hf ? o - m : m + o;               // outputs k and k + 8
        }
        if (e < 2 * n)
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k + 8 * hf < NOUT) p[(k + 8 * hf) * stride] = out[k];
    }
}

template <int T, bool PR>
__global__ void __launch_bounds__(T, 1) rowspace_small_kernel(const __grid_constant__ RsArgs<double> a) {
    typedef double2 C;
    constexpr int M1 = 16, M2 = 16, RM = kRsSmallRows, H = kRsHalo, NP = M1 * M2, PPT = NP / T;
    typedef RsGeom<double, M1, M2, RM, PR> G;
    extern __shared__ __align__(16) unsigned char rs_smem[];
    C *planes = reinterpret_cast<C *>(rs_smem);       // [RM][M2][LDP]
    const int tid = threadIdx.x, nb = a.nb;
    const int rank = blockIdx.x % kRsSmallCl, kb = blockIdx.x / kRsSmallCl, b = kb % a.nbands;
    const RsK &d = a.d[kb / a.nbands];
    const int ldg = d.ldg;
    const int j0 = rank * nb / kRsSmallCl, j1 = (rank + 1) * nb / kRsSmallCl, L = j1 - j0;
    auto line1 = [&](int l) { return planes + (l / G::N2) * G::PS + (l % G::N2) * G::LDP; };
    auto line2 = [&](int l) { return planes + (l / 16) * G::PS + l % 16; };
    const C *X = reinterpret_cast<const C *>(d.X) + ((size_t)b * nb + j0) * ldg;
    C *Y = reinterpret_cast<C *>(d.Y) + ((size_t)b * nb + j0) * ldg;
    for (int g = tid; g < d.ng; g += T) {
        C *dst = planes + __ldg(a.gpos + d.gofs + g);
#pragma unroll
        for (int i = 0; i < RM; ++i)
            if (i < L) dst[i * G::PS] = X[(size_t)i * ldg + g];
    }
    for (int e = tid; e < d.npos; e += T) {                          // the compact plane's disc-free positions
        C *dst = planes + __ldg(a.pos + d.pofs + e);
#pragma unroll
        for (int i = 0; i < RM; ++i) dst[i * G::PS] = czero<C>();
    }
    __syncthreads();
    rs_lines16<T, true, G::N1, 16>(L * G::N2, 1, line1);
    __syncthreads();
    rs_lines16<T, true, G::N2, 16>(L * 16, G::LDP, line2);
    rs_cluster_arrive();
    rs_cluster_wait();
    C y[PPT][RM];
#pragma unroll
    for (int q = 0; q < PPT; ++q) {
        const int pt = tid + q * T;
        const C *x = planes + (pt / M1) * G::LDP + pt % M1;
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(x);
        // row j0 + s from the CTA that owns it (zero outside the basis)
        auto remote = [&](int s) {
            const int row = j0 + s;
            if (row < 0 || row >= nb) return czero<C>();
            const int own = ((row + 1) * kRsSmallCl - 1) / nb;
            return rs_ld_cluster(rs_mapa(mine + (uint32_t)((row - own * nb / kRsSmallCl) * G::PS * sizeof(C)), own), C());
        };
        C lo[H], hi[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            lo[k] = remote(k - H);
            hi[k] = remote(L + k);
        }
        // the band's rows of the potential, two ahead
        const C *U = a.U + (size_t)j0 * 3 * NP + pt;
        const int nt = min(L + H, nb - j0);
        C un[2][3];
        auto load_u = [&](int t) {
            if (t < nt)
#pragma unroll
                for (int p = 0; p < 3; ++p) un[t & 1][p] = __ldg(U + (size_t)(3 * t + p) * NP);
        };
        load_u(0);
        load_u(1);
        C h[H];                       // x of rows t - 5 .. t - 1
#pragma unroll
        for (int k = 0; k < H; ++k) h[k] = lo[k];
#pragma unroll
        for (int t = 0; t < RM + H; ++t) {
            if (t >= nt) break;                                      // uniform in the CTA
            const double ud[6] = {un[t & 1][0].x, un[t & 1][0].y, un[t & 1][1].x,
                                  un[t & 1][1].y, un[t & 1][2].x, un[t & 1][2].y};     // U(t, t - d)
            load_u(t + 2);
            C xt = czero<C>();
            if (t < L) {
                if (t < RM) xt = x[t * G::PS];
            } else {
#pragma unroll
                for (int k = 0; k < H; ++k)
                    if (t - L == k) xt = hi[k];
            }
#pragma unroll
            for (int dd = H; dd >= 1; --dd)
                if (t - dd >= 0 && t - dd < RM && t - dd < L) rfma(y[q][t - dd < RM ? t - dd : 0], ud[dd], xt);
            if (t < RM && t < L) {
                C n = rscale(ud[5], h[0]);
#pragma unroll
                for (int dd = 4; dd >= 1; --dd) rfma(n, ud[dd], h[H - dd]);
                rfma(n, ud[0], xt);
                y[q][t < RM ? t : 0] = n;
            }
#pragma unroll
            for (int k = 0; k + 1 < H; ++k) h[k] = h[k + 1];
            h[H - 1] = xt;
        }
    }
    rs_cluster_arrive();
    rs_cluster_wait();                // every CTA has read its neighbours' rows
#pragma unroll
    for (int q = 0; q < PPT; ++q) {
        const int pt = tid + q * T;
        C *x = planes + (pt / M1) * G::LDP + pt % M1;
#pragma unroll
        for (int i = 0; i < RM; ++i)
            if (i < L) x[i * G::PS] = y[q][i];
    }
    __syncthreads();
    rs_lines16<T, false, 16, G::N2>(L * 16, G::LDP, line2);
    __syncthreads();
    rs_lines16<T, false, 16, G::N1>(L * G::N2, 1, line1);
    __syncthreads();
    for (int g = tid; g < ldg; g += T) {
        const C *src = planes + (g < d.ng ? __ldg(a.gpos + d.gofs + g) : 0);
#pragma unroll
        for (int i = 0; i < RM; ++i)
            if (i < L) Y[(size_t)i * ldg + g] = g < d.ng ? src[i * G::PS] : czero<C>();   // padding columns
    }
}

bool rs_small_supported(const RsShape &sh, int pairs, int nb, int num_sms) {
    return sh.m1 == 16 && sh.m2 == 16 && sh.s1 * sh.s2 == 1 && nb >= kRsSmallCl && nb <= kRsSmallCl * kRsSmallRows &&
           pairs * kRsSmallCl <= num_sms;
}

cudaError_t rs_launch_small(const RsArgs<double> &a, unsigned pairs, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at = {};
    cfg.gridDim = dim3(pairs * kRsSmallCl);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = RsGeom<double, 16, 16, kRsSmallRows, true>::PS * kRsSmallRows * sizeof(double2);
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kRsSmallCl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return a.pruned ? cudaLaunchKernelEx(&cfg, rowspace_small_kernel<256, true>, a)
                    : cudaLaunchKernelEx(&cfg, rowspace_small_kernel<256, false>, a);
}

}  // namespace mb
