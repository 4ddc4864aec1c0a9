// Electron density through row space: the FP64 companion of the row-space
// H apply (rowspace.cuh) for the self-consistent loop.
//
// With x_j(r) the inverse 2D transform of coefficient row j, the density on
// the Gauss planes is the quadratic form
//   rho(r, z_q) = (1/A_c) sum_kn f_kn |sum_j B_j(z_q) x_j(r)|^2
//               = (1/A_c) sum_ij B_i(z_q) B_j(z_q) P_ij(r),
//   P_ij(r) = sum_kn f_kn Re(conj(x_i) x_j),  |i - j| < kappa,
// so the bands are summed once per B-spline row (a band of kappa products per
// grid point) instead of once per Gauss plane, and the planes are formed from
// the sum.  Per (band, row, point) that is about 19 FP64 instructions of
// transforms and 14 of products, against 43 per plane (six planes a row)
// with a transform of every plane.
//
// The quadratic form's rounding is of its largest product, so where the sum of
// the bands nearly vanishes it loses twice the digits that |sum_j B_j x_j|^2
// loses (the slab's one band near its nodes: 1.4e-11 of the density there for
// 5.6e-13, and 3.2e-14 for 2.4e-15 of the largest v_xc).  Few bands therefore
// take the planes' sums of squares themselves, formed from the same
// transformed rows (SQUARES: 90 instructions a row).
//
// density_rows_kernel: one CTA per (part, run of rows or knot intervals), a
// part being a contiguous share of the (k-point, band) pairs; it walks its
// pairs one after the other and adds their products (or squares) to its own
// part in global memory (L2).  density_planes_kernel adds the parts in order
// and forms the planes (density_sum_kernel: adds them).
// FP64 bound.  Slab, 4 k x 32 bands: 0.65 ms + 0.07 ms, against 5.1 ms (both
// under ncu) with every plane of every band transformed and squared.
#include <algorithm>
#include <cmath>

#include "rowspace.cuh"

namespace mb {

namespace {

// The number of equally occupied pairs, (sum |f|)^2 / sum f^2, from which on the
// products are taken.  The smallest of a million sums of n squares of real
// amplitudes is about (n!! 1e-6)^(2/n) / n of their mean: 7e-4 for n = 4, 6e-3
// for 6, where the largest error of v_xc ~ rho^(1/3) no longer comes from such
// points (6e-16 to 8e-16 either way from 5 bands on).  The slab's 8 bands (6.1)
// take 240 us by squares and 185 by products, 3 bands 112 and 122; the 16 x 16
// cell's 3 bands 64 and 84 to 97.
constexpr double kMinPairs = 6.0;

struct DensRowsK {
    const double2 *X;     // nbands x nb x ldg coefficients of this k-point
    int ng, ldg, gofs, pofs, npos, kg;
};

struct DensRowsArgs {
    const double *occ;    // nk x nbands
    const double *Bq;     // nq x kappa
    double *part;         // [part][nb][kappa][residue][point], or [part][nq][residue][point]
    const int *gpos;
    const int *pos;
    const int4 *src;
    const double2 *phase;
    size_t phase_stride;
    int nbands, nb, nint, nquad, nk, nparts, nchunks, s1, s2;
    int accumulate;       // 0: the parts hold nothing yet
    DensRowsK d[kMaxK];
};

template <int M1, int M2, int T, int RR, int CTAS, bool PR, bool FOLD, bool SQUARES>
__global__ void __launch_bounds__(T, CTAS) density_rows_kernel(const __grid_constant__ DensRowsArgs a) {
    typedef double2 C;
    typedef RsGeom<double, M1, M2, RR, PR> G;
    constexpr int H = kRsHalo, NP = M1 * M2, PPT = NP / T, GR = 4;
    extern __shared__ __align__(16) unsigned char rs_smem[];
    C *planes = reinterpret_cast<C *>(rs_smem);       // [RR][M2][LDP]
    C *hist = planes + RR * G::PS;                    // [H][NP]: x of the five rows before the step
    const int tid = threadIdx.x;
    const int S = FOLD ? a.s1 * a.s2 : 1, rank = FOLD ? (int)blockIdx.x % S : 0, item = (int)blockIdx.x / S;
    const int c = item % a.nchunks, p = item / a.nchunks, nb = a.nb;
    // SQUARES: knot intervals j0 .. j1 - 1, whose splines are rows j0 - 1 .. j1 + 3;
    // row m completes interval m - 4 (rows outside the basis are zero)
    const int n = SQUARES ? a.nint : nb;
    const int j0 = chunk_begin(c, n, a.nchunks), j1 = chunk_begin(c + 1, n, a.nchunks);
    const int ji = max(0, j0 - (SQUARES ? 1 : H)), mend = SQUARES ? j1 + 4 : j1, je = min(nb, mend);
    const int npair = a.nk * a.nbands;
    const int q0 = (int)((long long)p * npair / a.nparts), q1 = (int)((long long)(p + 1) * npair / a.nparts);
    const size_t prow = (size_t)S * NP;               // one product of one row
    double *part = a.part + (size_t)p * (SQUARES ? a.nint * a.nquad : nb * kRsOrder) * prow + (size_t)rank * NP;
    bool fresh = !a.accumulate;
    for (int pair = q0; pair < q1; ++pair) {
        const int k = pair / a.nbands, n = pair - k * a.nbands;
        const DensRowsK &d = a.d[k];
        const double f = a.occ[(size_t)d.kg * a.nbands + n];
        if (f == 0.0) continue;                       // uniform over the CTA
        const C *X = d.X + (size_t)n * nb * d.ldg;
        for (int a0 = ji; a0 < mend; a0 += RR) {
            const int nin = max(0, min(RR, je - a0));
            const C *Xa = X + (size_t)a0 * d.ldg;
            __syncthreads();                          // the previous step's planes are consumed
            if constexpr (!FOLD) {
                for (int g = tid; g < d.ng; g += T) {
                    C *dst = planes + a.gpos[d.gofs + g];
#pragma unroll
                    for (int i = 0; i < RR; ++i)
                        if (i < nin) dst[i * G::PS] = Xa[(size_t)i * d.ldg + g];
                }
                for (int e = tid; e < d.npos; e += T) {
                    C *dst = planes + a.pos[d.pofs + e];
#pragma unroll
                    for (int i = 0; i < RR; ++i) dst[i * G::PS] = czero<C>();
                }
            } else {
                const C *phase = a.phase + rank * a.phase_stride + d.gofs;
                for (int e = tid; e < NP; e += T) {
                    C *dst = planes + (e / M1) * G::LDP + e % M1;
                    const int4 p4 = a.src[d.pofs + e];
                    C v[RR];
#pragma unroll
                    for (int i = 0; i < RR; ++i) v[i] = czero<C>();
#pragma unroll 1
                    for (int s = 0; s < 4; ++s) {
                        const int g = s == 0 ? p4.x : s == 1 ? p4.y : s == 2 ? p4.z : p4.w;
                        if (g < 0) break;
                        const C ph = phase[g];
#pragma unroll
                        for (int i = 0; i < RR; ++i)
                            if (i < nin) cfma(v[i], ph, Xa[(size_t)i * d.ldg + g]);
                    }
#pragma unroll
                    for (int i = 0; i < RR; ++i) dst[i * G::PS] = v[i];
                }
            }
            __syncthreads();
            rs_axis1<double, M1, M2, T, RR, PR, true>(planes, nin);
            __syncthreads();
            rs_axis2<double, M1, M2, T, RR, PR, true>(planes, nin);
            __syncthreads();
#pragma unroll
            for (int q = 0; q < PPT; ++q) {
                const int pt = tid + q * T;
                const C *x = planes + (pt / M1) * G::LDP + pt % M1;
                C h[H];                               // h[k]: x of row m - 5 + k
#pragma unroll
                for (int k2 = 0; k2 < H; ++k2) h[k2] = a0 > ji ? hist[k2 * NP + pt] : czero<C>();
                if constexpr (SQUARES) {
                    for (int i = 0; i < min(RR, mend - a0); ++i) {
                        const C xm = i < nin ? x[i * G::PS] : czero<C>();
                        const int t = a0 + i - 4;
                        for (int s0 = 0; t >= j0 && s0 < a.nquad; s0 += 6) {      // planes, six at a time
                            double *R = part + (size_t)(t * a.nquad + s0) * prow + pt, acc[6];
#pragma unroll
                            for (int s = 0; s < 6; ++s) acc[s] = !fresh && s0 + s < a.nquad ? R[s * prow] : 0.0;
#pragma unroll
                            for (int s = 0; s < 6; ++s) {
                                if (s0 + s >= a.nquad) break;
                                const double *b = a.Bq + (size_t)(t * a.nquad + s0 + s) * kRsOrder;
                                C psi = rscale(__ldg(b), h[0]);
#pragma unroll
                                for (int u = 1; u < H; ++u) rfma(psi, __ldg(b + u), h[u]);
                                rfma(psi, __ldg(b + H), xm);
                                R[s * prow] = fma(f, fma(psi.x, psi.x, psi.y * psi.y), acc[s]);
                            }
                        }
#pragma unroll
                        for (int k2 = 0; k2 + 1 < H; ++k2) h[k2] = h[k2 + 1];
                        h[H - 1] = xm;
                    }
                }
                double *P = part + (size_t)a0 * kRsOrder * prow + pt;
                // GR rows at a time: their sums so far are all loaded first
                for (int i0 = 0; !SQUARES && i0 < nin; i0 += GR, P += GR * kRsOrder * prow) {
                    double acc[GR][kRsOrder];
#pragma unroll
                    for (int i = 0; i < GR; ++i)
#pragma unroll
                        for (int e = 0; e < kRsOrder; ++e)
                            acc[i][e] = !fresh && i0 + i < nin && a0 + i0 + i >= j0 ? P[(i * kRsOrder + e) * prow] : 0.0;
#pragma unroll
                    for (int i = 0; i < GR; ++i) {
                        if (i0 + i >= nin) break;
                        const C xm = x[(i0 + i) * G::PS];
                        if (a0 + i0 + i >= j0) {
                            const C fx = make_double2(f * xm.x, f * xm.y);
                            acc[i][0] = fma(fx.x, xm.x, fma(fx.y, xm.y, acc[i][0]));
#pragma unroll
                            for (int e = 1; e < kRsOrder; ++e)
                                acc[i][e] = fma(fx.x, h[H - e].x, fma(fx.y, h[H - e].y, acc[i][e]));
#pragma unroll
                            for (int e = 0; e < kRsOrder; ++e) P[(i * kRsOrder + e) * prow] = acc[i][e];
                        }
#pragma unroll
                        for (int k2 = 0; k2 + 1 < H; ++k2) h[k2] = h[k2 + 1];
                        h[H - 1] = xm;
                    }
                }
#pragma unroll
                for (int k2 = 0; k2 < H; ++k2) hist[k2 * NP + pt] = h[k2];
            }
        }
        fresh = false;
    }
    const int per = SQUARES ? a.nquad : kRsOrder;
    if (fresh)                                        // no occupied pair
        for (int e = j0 * per; e < j1 * per; ++e)
            for (int pt = tid; pt < NP; pt += T) part[e * prow + pt] = 0.0;
}

// rho of the squares: the parts added in order
__global__ void __launch_bounds__(128) density_sum_kernel(const double *part, int nparts, int nq, int N1, int N2, int s1, int s2,
                                                          double scale, double *rho) {
    const int NN = N1 * N2, M1 = N1 / s1, NP = NN / (s1 * s2), e = blockIdx.x % (unsigned)(NN / 128) * 128 + threadIdx.x;
    const int q = blockIdx.x / (unsigned)(NN / 128), res = e / NP, pt = e % NP;
    const int r = (pt % M1 * s1 + res / s2) * N2 + pt / M1 * s2 + res % s2;
    double s = 0.0;
#pragma unroll 8
    for (int p = 0; p < nparts; ++p) s += part[((size_t)p * nq + q) * NN + e];
    rho[(size_t)q * NN + r] = scale * s;
}

// rho of one knot interval's planes at one grid point: the band of P that the
// interval's kappa splines touch, summed over the parts in order, then the
// quadratic form at every Gauss point.  clamp: occupations are >= 0, and so
// is rho (rounding may leave -1e-17 of the largest product where it vanishes);
// NaN and infinite sums stay what they are.
__global__ void __launch_bounds__(128) density_planes_kernel(const double *part, int nparts, int nb, int nint, int nquad,
                                                             int N1, int N2, int s1, int s2, const double *Bq,
                                                             double scale, int clamp, double *rho) {
    constexpr int K = kRsOrder;
    const int NN = N1 * N2, M1 = N1 / s1, NP = NN / (s1 * s2), e = blockIdx.x * 128 + threadIdx.x, t = blockIdx.y;
    if (e >= NN) return;
    const size_t stride = (size_t)nb * K * NN;
    double P[K * (K + 1) / 2];
    int n = 0;
#pragma unroll
    for (int u = 0; u < K; ++u)
#pragma unroll
        for (int v = 0; v <= u; ++v, ++n) {
            const int j = t - 1 + u, j2 = t - 1 + v;  // spline j is entry u of the interval
            double s = 0.0;
            if (j2 >= 0 && j < nb)
#pragma unroll 8
                for (int p = 0; p < nparts; ++p) s += part[p * stride + ((size_t)j * K + (j - j2)) * NN + e];
            P[n] = u == v ? s : 2.0 * s;
        }
    const int res = e / NP, pt = e % NP;
    const int r = (pt % M1 * s1 + res / s2) * N2 + pt / M1 * s2 + res % s2;
    for (int q = t * nquad; q < (t + 1) * nquad; ++q) {
        double B[K], s = 0.0;
#pragma unroll
        for (int u = 0; u < K; ++u) B[u] = Bq[(size_t)q * K + u];
        n = 0;
#pragma unroll
        for (int u = 0; u < K; ++u) {
            double w = 0.0;
#pragma unroll
            for (int v = 0; v <= u; ++v, ++n) w = fma(B[v], P[n], w);
            s = fma(B[u], w, s);
        }
        s *= scale;
        rho[(size_t)q * NN + r] = clamp && s < 0.0 && !isinf(s) ? 0.0 : s;
    }
}

template <int M1, int M2, int T, int RR, int CTAS, bool SQUARES>
cudaError_t launch_rows(const DensRowsArgs &a, bool pruned, int smem_limit, int device, cudaStream_t s) {
    const unsigned S = (unsigned)(a.s1 * a.s2), grid = (unsigned)(a.nparts * a.nchunks) * S;
    auto go = [&](auto kern) {
        constexpr size_t smem = RsGeom<double, M1, M2, RR, false>::smem;   // the same for pruned planes
        const cudaError_t e = smem_limit_once((const void *)kern, device, smem_limit);
        if (e != cudaSuccess) return e;
        kern<<<grid, T, smem, s>>>(a);
        return cudaGetLastError();
    };
    if constexpr (M1 * M2 > 256)
        if (S > 1) return go(density_rows_kernel<M1, M2, T, RR, CTAS, false, true, SQUARES>);
    if (S > 1) return cudaErrorInvalidValue;
    return pruned ? go(density_rows_kernel<M1, M2, T, RR, CTAS, true, false, SQUARES>)
                  : go(density_rows_kernel<M1, M2, T, RR, CTAS, false, false, SQUARES>);
}
template <bool SQUARES>
cudaError_t launch_rows(const DensRowsArgs &a, int m1, int m2, bool pruned, int smem_limit, int device, cudaStream_t s) {
    if (m1 == 16 && m2 == 16) return launch_rows<16, 16, 128, 16, 2, SQUARES>(a, pruned, smem_limit, device, s);
    if (m1 == 16) return launch_rows<16, 32, 256, 16, 1, SQUARES>(a, pruned, smem_limit, device, s);
    if (m2 == 16) return launch_rows<32, 16, 256, 16, 1, SQUARES>(a, pruned, smem_limit, device, s);
    return launch_rows<32, 32, 256, 8, 1, SQUARES>(a, pruned, smem_limit, device, s);
}

}  // namespace

// rho (device, nq x N1 x N2) on grids the row-space kernels serve; occ: the
// occupations on the host, occ_dev: their copy on the device.
int density_rows(mb_handle *h, const void *evecs, int nbands, const double *occ, const double *occ_dev, double *rho,
                 cudaStream_t s) {
    const int nk = (int)h->kp.size(), nb = h->nb, NN = h->n1 * h->n2;
    const int s1 = rs_fold(h->n1), s2 = rs_fold(h->n2), S = s1 * s2, m1 = h->n1 / s1, m2 = h->n2 / s2;
    // Parts of the pairs times runs of rows, by FP64 instructions on the
    // busiest SM sub-partition: per step of up to RR rows the line transforms
    // in whole rounds of four warps, and 14 products per output row and point
    // (runs that leave a step nearly empty pay for it: 1.03 ms with 16 parts
    // of 9 runs, 18 rows each, on the slab); a part more costs its sum.
    double sum = 0.0, sq = 0.0;
    bool nonneg = true;
    for (int i = 0; i < nk * nbands; ++i) {
        sum += std::fabs(occ[i]);
        sq += occ[i] * occ[i];
        nonneg = nonneg && occ[i] >= 0.0;
    }
    const bool squares = !(sum * sum >= kMinPairs * sq);
    const int pairs = nk * nbands, RR = m1 == 32 && m2 == 32 ? 8 : 16, N2 = h->rs_pruned ? m2 * 3 / 4 : m2;
    auto line = [](int m) { return m == 32 ? 360.0 : 140.0; };
    auto rounds4 = [](int lines) { return (double)((lines + 127) / 128); };
    int nparts = 1, nchunks = 1;
    double best = 1e300;
    const int items = squares ? h->nint : nb;
    const double per = squares ? 15.0 * h->nquad : 14.0;
    for (int c = 1; c <= std::min(items, 64); ++c) {
        // the longest run of one pair: the last, of ceil(items / c) rows and the
        // rows before them that they multiply (or intervals and their rows)
        const int L = (items + c - 1) / c, in = std::min(nb, L + std::min(kRsHalo, nb - L));
        auto lines = [&](int n) { return rounds4(n * N2) * line(m1) + rounds4(n * m1) * line(m2); };
        const double run = per * L * (m1 * m2 / 128) + in / RR * lines(RR) + lines(in % RR);
        for (int p = 1; p <= std::min(pairs, 32); ++p) {
            const double rounds = (double)(((long long)p * c * S + h->num_sms - 1) / h->num_sms);
            const double cost = rounds * ((pairs + p - 1) / p) * run + 9.0 * 14.0 * (m1 * m2 / 128) * p;
            if (cost < best) {
                best = cost;
                nparts = p;
                nchunks = c;
            }
        }
    }
    cudaMemPool_t pool = mb_pool(h->device);
    if (!pool) return MB_ECUDA;
    double *part = nullptr;
    MB_CUDA(cudaMallocFromPoolAsync((void **)&part, (size_t)nparts * (squares ? h->nq : nb * kRsOrder) * NN * sizeof(double), pool, s));
    DensRowsArgs a;
    a.occ = occ_dev;
    a.Bq = (const double *)h->t64.Bq;
    a.part = part;
    a.gpos = h->d_rsgpos;
    a.pos = reinterpret_cast<const int *>(h->d_rspos);
    a.src = reinterpret_cast<const int4 *>(h->d_rspos);
    a.phase = reinterpret_cast<const double2 *>(h->t64.phase);
    a.phase_stride = (size_t)h->total_ldg;
    a.nbands = nbands;
    a.nb = nb;
    a.nint = h->nint;
    a.nquad = h->nquad;
    a.nparts = nparts;
    a.nchunks = nchunks;
    a.s1 = s1;
    a.s2 = s2;
    size_t off = 0;
    cudaError_t e = cudaSuccess;
    for (int k0 = 0; k0 < nk && e == cudaSuccess; k0 += kMaxK) {
        a.nk = std::min(kMaxK, nk - k0);
        a.accumulate = k0 > 0;
        for (int i = 0; i < a.nk; ++i) {
            const int k = k0 + i;
            DensRowsK &d = a.d[i];
            d.X = reinterpret_cast<const double2 *>(evecs) + off;
            d.ng = h->kp[k].ng;
            d.ldg = h->kp[k].ldg;
            d.gofs = h->kofs[k];
            d.pofs = h->rs_pofs[k];
            d.npos = h->rs_npos[k];
            d.kg = k;
            off += (size_t)nbands * nb * h->kp[k].ldg;
        }
        e = squares ? launch_rows<true>(a, m1, m2, h->rs_pruned, h->smem_optin, h->device, s)
                    : launch_rows<false>(a, m1, m2, h->rs_pruned, h->smem_optin, h->device, s);
        ++h->launches;
    }
    if (e == cudaSuccess && squares) {
        density_sum_kernel<<<(unsigned)(h->nq * (NN / 128)), 128, 0, s>>>(part, nparts, h->nq, h->n1, h->n2, s1, s2, 1.0 / h->Ac, rho);
        e = cudaGetLastError();
        ++h->launches;
    } else if (e == cudaSuccess) {
        density_planes_kernel<<<dim3((NN + 127) / 128, h->nint), 128, 0, s>>>(
            part, nparts, nb, h->nint, h->nquad, h->n1, h->n2, s1, s2, (const double *)h->t64.Bq, 1.0 / h->Ac, nonneg, rho);
        e = cudaGetLastError();
        ++h->launches;
    }
    cudaFreeAsync(part, s);
    MB_CUDA(e);
    return MB_OK;
}

}  // namespace mb
