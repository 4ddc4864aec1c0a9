// The local potential V(r, z_q) on the quadrature planes, built on the device
// from the analytic in-plane components of the atoms' local pseudopotentials
// (§II.B.1, Eq. (10)):
//   Gaussian term A exp(-a r^2) (Eq. (13)):
//       (A / A_c)(pi / a) exp(-g^2 / 4a) exp(-a dz^2)
//   core term -Z erf(r / R_c) / r: the Coulomb potential of the Gaussian core
//   charge through the 2D transform of 1/r (the Coulomb integral of §II.B.1),
//   in closed form
//       -(Z / A_c)(pi / g) [T(dz) + T(-dz)],  T(z) = exp(g z) erfc(g R_c / 2 + z / R_c),
//   written exp(-g^2 R_c^2 / 4 - z^2 / R_c^2) erfcx(x) where the erfc argument
//   x is >= 0; at g = 0 the divergent constant (2 pi / g)(Z / A_c) is dropped
//   and +(2 pi Z / A_c)[dz erf(dz / R_c) + (R_c / sqrt(pi)) exp(-dz^2 / R_c^2)]
//   kept,
// each times exp(-i g . R_par), summed over the grid frequencies g_m
// (m in [-N/2, N/2) per axis) into the real table
//   V(r, z_q) = Re sum_m c(m, z_q) exp(i g_m . r),  r = (i1/N1) a1 + (i2/N2) a2.
//
// Atoms that share a profile (kind, width, height) share its z dependence,
// so their phases are summed once into a structure factor per group
// (vloc_sfac_kernel).  Per plane the components are the groups' profiles
// times their structure factors, summed along m2 (vloc_rows_kernel) and then
// along m1, keeping the real part (vloc_cols_kernel): plain O(N) sums per
// output with N <= 256, in FP64, twiddles from sincospi of exact ratios.
// The table the handle's plane kernel reads is derived from the natural
// table, which may also be one set by the caller: the row-space potential U
// (rs_tables_kernel), or, on grids without a row-space kernel, the planes
// with weight and 1/(N1 N2) folded in, bit-reversed (vloc_tables_kernel);
// each in FP64 with an FP32 copy.
#include <algorithm>
#include <vector>

#include "mb_internal.h"

namespace mb {

namespace {

constexpr double kPiD = 3.14159265358979323846;
constexpr double kInvSqrtPi = 0.56418958354775628695;
constexpr size_t kVlocChunkBytes = 64ull << 20;   // planes per pass of the two-step transform

struct VlocGeom {
    int N1, N2, nq, ngrp;
    double b1x, b1y, b2x, b2y, Ac;
};

__device__ __forceinline__ void grid_g(const VlocGeom &G, int u, int v, double &gx, double &gy) {
    const int m1 = u < G.N1 / 2 ? u : u - G.N1, m2 = v < G.N2 / 2 ? v : v - G.N2;
    gx = m1 * G.b1x + m2 * G.b2x;
    gy = m1 * G.b1y + m2 * G.b2y;
}

// z profile of one group at |g| and height dz above the group's atoms, per
// unit weight (A of a Gaussian, Z of a core term) and per unit cell area.
// mode 0: the potential; mode 1: the core charge density
// rho_c = Z exp(-r^2/R_c^2) / (pi^(3/2) R_c^3), whose components are
// exp(-g^2 R_c^2/4) exp(-dz^2/R_c^2) / (sqrt(pi) R_c A_c) (Gaussians: none).
__device__ double profile(int mode, int kind, double p, double g, double dz, double Ac) {
    if (mode == 1) {
        if (kind != 1) return 0.0;
        const double u = dz / p;
        return kInvSqrtPi / (p * Ac) * exp(-0.25 * (g * p) * (g * p) - u * u);
    }
    if (kind == 0) {   // Gaussian, p = a
        return (kPiD / p) / Ac * exp(-g * g / (4.0 * p)) * exp(-p * dz * dz);
    }
    const double Rc = p;   // core term
    if (g == 0.0) {
        const double u = dz / Rc;
        return (2.0 * kPiD / Ac) * (dz * erf(u) + Rc * kInvSqrtPi * exp(-u * u));
    }
    double t = 0.0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const double z = s ? -dz : dz;
        const double x = 0.5 * g * Rc + z / Rc;
        t += x >= 0.0 ? exp(-0.25 * (g * Rc) * (g * Rc) - (z / Rc) * (z / Rc)) * erfcx(x) : exp(g * z) * erfc(x);
    }
    return -(kPiD / g) / Ac * t;
}

// S[grp][u N2 + v] = sum_{atoms of grp} weight exp(-i g_m . R_par)
__global__ void vloc_sfac_kernel(VlocGeom G, const double *ion, const int *start, double2 *S) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x, grp = blockIdx.y;
    const int NN = G.N1 * G.N2;
    if (e >= NN) return;
    double gx, gy;
    grid_g(G, e / G.N2, e % G.N2, gx, gy);
    double re = 0.0, im = 0.0;
    for (int i = start[grp]; i < start[grp + 1]; ++i) {
        double sn, cs;
        sincos(-(gx * ion[3 * i + 1] + gy * ion[3 * i + 2]), &sn, &cs);
        re += ion[3 * i] * cs;
        im += ion[3 * i] * sn;
    }
    S[(size_t)grp * NN + e] = make_double2(re, im);
}

// One (row u, plane q) per threadIdx.y slice: c(m, z_q) for the N2
// frequencies of the row, then tmp[q][u][i2] = sum_v c(u, v) exp(2 pi i v i2 / N2).
// blockDim = (N2, planes per block).
__global__ void vloc_rows_kernel(VlocGeom G, int mode, const double *grp, const double2 *S, const double *zq, int q0,
                                 int nqc, double2 *tmp) {
    extern __shared__ double2 rs[];
    double2 *tw = rs, *c = rs + G.N2 + threadIdx.y * G.N2;
    const int u = blockIdx.x, qq = blockIdx.y * blockDim.y + threadIdx.y, v = threadIdx.x, NN = G.N1 * G.N2;
    if (threadIdx.y == 0) {
        double sn, cs;
        sincospi(2.0 * v / G.N2, &sn, &cs);
        tw[v] = make_double2(cs, sn);
    }
    const bool live = qq < nqc;
    if (live) {
        double gx, gy;
        grid_g(G, u, v, gx, gy);
        const double g = sqrt(gx * gx + gy * gy), z = zq[q0 + qq];
        double re = 0.0, im = 0.0;
        for (int k = 0; k < G.ngrp; ++k) {
            const double f = profile(mode, (int)grp[3 * k], grp[3 * k + 1], g, z - grp[3 * k + 2], G.Ac);
            const double2 s = S[(size_t)k * NN + u * G.N2 + v];
            re += f * s.x;
            im += f * s.y;
        }
        c[v] = make_double2(re, im);
    }
    __syncthreads();
    if (!live) return;
    double sr = 0.0, si = 0.0;
    for (int w = 0; w < G.N2; ++w) {
        const double2 a = c[w], t = tw[(w * v) & (G.N2 - 1)];
        sr += a.x * t.x - a.y * t.y;
        si += a.x * t.y + a.y * t.x;
    }
    tmp[((size_t)qq * G.N1 + u) * G.N2 + v] = make_double2(sr, si);
}

// One (column i2, plane q) per threadIdx.y slice:
// V[q][i1][i2] = Re sum_u tmp[q][u][i2] exp(2 pi i u i1 / N1).  blockDim = (N1, planes per block).
__global__ void vloc_cols_kernel(VlocGeom G, const double2 *tmp, int q0, int nqc, double *V) {
    extern __shared__ double2 cs_[];
    double2 *tw = cs_, *col = cs_ + G.N1 + threadIdx.y * G.N1;
    const int i2 = blockIdx.x, qq = blockIdx.y * blockDim.y + threadIdx.y, i1 = threadIdx.x;
    const bool live = qq < nqc;
    if (live) col[i1] = tmp[((size_t)qq * G.N1 + i1) * G.N2 + i2];
    if (threadIdx.y == 0) {
        double sn, cs;
        sincospi(2.0 * i1 / G.N1, &sn, &cs);
        tw[i1] = make_double2(cs, sn);
    }
    __syncthreads();
    if (!live) return;
    double s = 0.0;
    for (int u = 0; u < G.N1; ++u) {
        const double2 a = col[u], t = tw[(u * i1) & (G.N1 - 1)];
        s += a.x * t.x - a.y * t.y;
    }
    V[((size_t)(q0 + qq) * G.N1 + i1) * G.N2 + i2] = s;
}

// The radix-2 plane kernel's table from the natural table V (nq x N1 x N2):
// (w_q / (N1 N2)) V, bit-reversed on both axes.
__global__ void vloc_tables_kernel(int nq, int N1, int N2, int l1, int l2, const double *V, const double *wq,
                                   double *Vp64, float *Vp32) {
    const int NN = N1 * N2;
    const size_t total = (size_t)nq * NN;
    const double scale = 1.0 / NN;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int q = (int)(e / NN), r = (int)(e % NN), i1 = r / N2, i2 = r % N2;
        const double val = wq[q] * scale * V[e];
        const int p1 = (int)(__brev((unsigned)i1) >> (32 - l1)), p2 = (int)(__brev((unsigned)i2) >> (32 - l2));
        const size_t pe = (size_t)q * NN + (size_t)p1 * N2 + p2;
        Vp64[pe] = val;
        Vp32[pe] = (float)val;
    }
}

// The row-space potential U[j][d](r) = sum_q B_j(z_q) B_{j-d}(z_q) w_q V(r, z_q) / (N1 N2),
// d = 0 .. order - 1 (0 where j - d < 0), over the knot intervals both splines
// share.  A CTA takes blockDim.x grid points of one row j: the products of B
// values and weights of the row's planes are formed once in shared memory, and
// a thread reads every plane of the row's support once at its point, a batch
// of loads in flight together.  Stored in pairs of d, each residue of the
// folded sides contiguous: [j][d / 2][residue][point].  Bound by the FP64 pipe:
// 126 FMAs per element, 234 operations with a thread forming its own products.
// It runs once per potential.
constexpr int kMaxQuad = 16;      // setup's limit of points per interval
__global__ void __launch_bounds__(256) rs_tables_kernel(int nb, int nint, int P, int N1, int N2, int s1, int s2,
                                                        const double *V, const double *wq, const double *Bq,
                                                        double2 *U64, float2 *U32) {
    constexpr int K = kRsOrder, PF = 12;
    __shared__ double W[K * kMaxQuad][K];
    const int NN = N1 * N2, M1 = N1 / s1, NP = NN / (s1 * s2);
    const int j = (int)blockIdx.x / (NN / blockDim.x), r = (int)blockIdx.x % (NN / blockDim.x) * blockDim.x + threadIdx.x;
    // spline j is entry m = j + 1 - t of interval t's kappa splines
    const int t0 = max(0, j + 2 - K), q0 = t0 * P, np = j < nb ? (min(nint - 1, j + 1) + 1 - t0) * P : 0;
    const double scale = 1.0 / NN;
    for (int e = threadIdx.x; e < np * K; e += blockDim.x) {
        const int p = e / K, d = e % K, m = j + 1 - t0 - p / P;
        const double *b = Bq + (size_t)(q0 + p) * K;
        W[p][d] = d <= m ? b[m] * (wq[q0 + p] * scale) * b[m - d] : 0.0;
    }
    __syncthreads();
    double acc[K];
#pragma unroll
    for (int d = 0; d < K; ++d) acc[d] = 0.0;
    for (int p0 = 0; p0 < np; p0 += PF) {
        double v[PF];
#pragma unroll
        for (int i = 0; i < PF; ++i) v[i] = p0 + i < np ? V[(size_t)(q0 + p0 + i) * NN + r] : 0.0;
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            if (p0 + i >= np) break;
            const int dm = min(j, j + 1 - t0 - (p0 + i) / P);        // uniform in the CTA
#pragma unroll
            for (int d = 0; d < K; ++d)
                if (d <= dm) acc[d] = fma(W[p0 + i][d], v[i], acc[d]);
        }
    }
    const int i1 = r / N2, i2 = r % N2;
    const int res = (i1 % s1) * s2 + i2 % s2, pt = (i2 / s2) * M1 + i1 / s1;
#pragma unroll
    for (int t = 0; t < K / 2; ++t) {
        const size_t o = ((size_t)j * (K / 2) + t) * NN + (size_t)res * NP + pt;
        U64[o] = make_double2(acc[2 * t], acc[2 * t + 1]);
        U32[o] = make_float2((float)acc[2 * t], (float)acc[2 * t + 1]);
    }
}

int pool_alloc(mb_handle *h, void **p, size_t bytes) {
    if (*p) return MB_OK;
    cudaMemPool_t pool = mb_pool(h->device);
    if (!pool) return MB_ECUDA;
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, h->hs);
    return e == cudaSuccess ? MB_OK : cuda_fail(h, e);
}

}  // namespace

size_t vloc_build_scratch_bytes(const mb_handle *h) {
    const size_t NN = (size_t)h->n1 * h->n2;
    const size_t ngrp = h->lstart.empty() ? 0 : h->lstart.size() - 1;
    const size_t per_plane = NN * sizeof(double2);
    const size_t qc = std::max<size_t>(1, std::min<size_t>(h->nq, kVlocChunkBytes / per_plane));
    return qc * per_plane + ngrp * NN * sizeof(double2) + (h->lion.size() + h->lgrp.size()) * sizeof(double) +
           h->lstart.size() * sizeof(int) + 2 * (size_t)h->nq * sizeof(double);
}

// The natural table d_vloc -> the table of t64 / t32 the handle's plane kernel reads.
int vloc_derive_tables(mb_handle *h) {
    const size_t NN = (size_t)h->n1 * h->n2, n = (size_t)h->nq * NN;
    int rc;
    const bool rs = rs_supported(h->n1, h->n2, h->order);
    const size_t nu = (size_t)(h->nb + kRsPad) * kRsOrder * NN;
    if (rs) {
        if ((rc = pool_alloc(h, &h->t64.U, nu * sizeof(double)))) return rc;
        if ((rc = pool_alloc(h, &h->t32.U, nu * sizeof(float)))) return rc;
    } else {
        if ((rc = pool_alloc(h, &h->t64.V, n * sizeof(double)))) return rc;
        if ((rc = pool_alloc(h, &h->t32.V, n * sizeof(float)))) return rc;
    }
    double *wq = nullptr;
    if ((rc = dev_upload(h, (void **)&wq, h->wq.data(), h->wq.size() * sizeof(double)))) return rc;
    auto blocks = [&](size_t m) { return (int)std::min<size_t>((m + 255) / 256, (size_t)h->num_sms * 8); };
    // 64 points a CTA (256 divides NN) where 256 would leave SMs without one
    const int T = h->nb * (NN / 256) < 2 * (size_t)h->num_sms ? 64 : 256;
    if (rs)
        rs_tables_kernel<<<(unsigned)((h->nb + kRsPad) * (NN / T)), T, 0, h->hs>>>(
            h->nb, h->nint, h->nquad, h->n1, h->n2, rs_fold(h->n1), rs_fold(h->n2), h->d_vloc, wq,
            (const double *)h->t64.Bq, (double2 *)h->t64.U, (float2 *)h->t32.U);
    else
        vloc_tables_kernel<<<blocks(n), 256, 0, h->hs>>>(h->nq, h->n1, h->n2, h->l1, h->l2, h->d_vloc, wq,
                                                        (double *)h->t64.V, (float *)h->t32.V);
    cudaError_t e = cudaGetLastError();
    dev_free(h, (void **)&wq);
    if (e != cudaSuccess) return cuda_fail(h, e);
    MB_CUDA(cudaStreamSynchronize(h->hs));
    return MB_OK;
}

// The real table of the atoms' analytic terms on the planes into out (nq x
// N1 x N2, device), on stream s: mode 0 the local potential V(r, z_q),
// mode 1 the Gaussian core charge density.
int vloc_tabulate(mb_handle *h, int mode, double *out, cudaStream_t s, const std::vector<double> *lgrp_in,
                  const std::vector<double> *lion_in, const std::vector<int> *lstart_in) {
    const std::vector<double> &lgrp = lgrp_in ? *lgrp_in : h->lgrp, &lion = lion_in ? *lion_in : h->lion;
    const std::vector<int> &lstart = lstart_in ? *lstart_in : h->lstart;
    const int N1 = h->n1, N2 = h->n2, NN = N1 * N2, nq = h->nq;
    const int ngrp = lstart.empty() ? 0 : (int)lstart.size() - 1;
    if (ngrp == 0) {
        MB_CUDA(cudaMemsetAsync(out, 0, (size_t)nq * NN * sizeof(double), s));
        return MB_OK;
    }
    VlocGeom G{N1, N2, nq, ngrp, h->b1[0], h->b1[1], h->b2[0], h->b2[1], h->Ac};
    const size_t per_plane = (size_t)NN * sizeof(double2);
    const int qc = (int)std::max<size_t>(1, std::min<size_t>(nq, kVlocChunkBytes / per_plane));
    cudaMemPool_t pool = mb_pool(h->device);
    if (!pool) return MB_ECUDA;
    // one pool block: ions | groups | planes | group starts (int) | S | tmp
    const size_t nion = lion.size(), ngv = lgrp.size();
    const size_t off_grp = nion * sizeof(double), off_zq = off_grp + ngv * sizeof(double);
    const size_t off_start = off_zq + (size_t)nq * sizeof(double);
    const size_t off_S = (off_start + lstart.size() * sizeof(int) + 255) / 256 * 256;
    const size_t off_tmp = off_S + (size_t)ngrp * per_plane, bytes = off_tmp + (size_t)qc * per_plane;
    unsigned char *blk = nullptr;
    MB_CUDA(cudaMallocFromPoolAsync((void **)&blk, bytes, pool, s));
    double *ion = reinterpret_cast<double *>(blk), *grp = reinterpret_cast<double *>(blk + off_grp);
    double *zq = reinterpret_cast<double *>(blk + off_zq);
    int *start = reinterpret_cast<int *>(blk + off_start);
    double2 *S = reinterpret_cast<double2 *>(blk + off_S), *tmp = reinterpret_cast<double2 *>(blk + off_tmp);
    cudaError_t e = cudaMemcpyAsync(ion, lion.data(), nion * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(grp, lgrp.data(), ngv * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(zq, h->zq.data(), nq * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(start, lstart.data(), lstart.size() * sizeof(int), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        vloc_sfac_kernel<<<dim3((NN + 255) / 256, ngrp), 256, 0, s>>>(G, ion, start, S);
        // planes per block: blocks of about 256 threads
        const int pr = std::max(1, 256 / N2), pc = std::max(1, 256 / N1);
        for (int q0 = 0; q0 < nq; q0 += qc) {
            const int n = std::min(qc, nq - q0);
            vloc_rows_kernel<<<dim3(N1, (n + pr - 1) / pr), dim3(N2, pr), (size_t)(1 + pr) * N2 * sizeof(double2), s>>>(
                G, mode, grp, S, zq, q0, n, tmp);
            vloc_cols_kernel<<<dim3(N2, (n + pc - 1) / pc), dim3(N1, pc), (size_t)(1 + pc) * N1 * sizeof(double2), s>>>(
                G, tmp, q0, n, out);
        }
        e = cudaGetLastError();
    }
    cudaFreeAsync(blk, s);
    if (e != cudaSuccess) return cuda_fail(h, e);
    // the host vectors copied above must stay untouched until the copies ran
    MB_CUDA(cudaStreamSynchronize(s));
    return MB_OK;
}

// V(r, z_q) from the atoms' analytic terms into d_vloc, then the derived tables.
int vloc_build(mb_handle *h) {
    int rc;
    if ((rc = pool_alloc(h, (void **)&h->d_vloc, (size_t)h->nq * h->n1 * h->n2 * sizeof(double)))) return rc;
    if ((rc = vloc_tabulate(h, 0, h->d_vloc, h->hs))) return rc;
    return vloc_derive_tables(h);
}

}  // namespace mb
