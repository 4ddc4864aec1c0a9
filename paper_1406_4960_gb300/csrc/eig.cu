// Generalized Lanczos-Krylov eigensolver (§II.C) on the device.
//
// Per k-point the solver keeps M roots X with HX and SX, and runs two
// alternating grand cycles:
//   A  Rayleigh-Ritz on [X | K_A], K_A the Krylov space of the root with the
//      largest residual;
//   B  roots split into blocks of b; each block does Rayleigh-Ritz on
//      [X_b | K_b] and keeps the b Ritz pairs of maximum overlap with its
//      inputs (plus any new lower root).
// after which X is S-orthonormalized and rotated to Ritz vectors in one
// Cholesky-QR + Rayleigh-Ritz step.  Krylov vectors come from
// A = P (H - theta S), P the banded per-G solve (T(G) + c S)^-1,
// S-orthogonalized by classical Gram-Schmidt applied twice.  Every step runs
// for all k-points in one launch; from the second cycle of each phase a
// grand cycle is one CUDA graph launch.
//
// Precision.  MB_FP64: everything in FP64.  Mixed (MB_FP32 / MB_BF16): bulk
// cycles on FP32 vectors only (FP32 applies in place on the chain slots,
// Gram products on the tensor cores with a TF32 hi + lo split, FP32 S
// products, preconditioner solves, rotations, residuals, Cholesky and
// Jacobi); then finish cycles with FP64 roots: FP64 applies of the roots,
// FP64 Grams, Cholesky and Jacobi (FP32 sweeps first), and the root
// rotations in float-float arithmetic, while the chains stay FP32.  The FP64
// residual is the convergence test.
#include <algorithm>
#include <chrono>
#include <tuple>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "cplx.cuh"
#include "mb_internal.h"
#include "tc_gemm.cuh"

namespace mb {

constexpr int LD = 128;       // leading dimension of subspace matrices
constexpr int JMAX = 112;     // largest subspace the Jacobi kernel holds (matrix in shared memory)
constexpr int JPAIRS = 56;    // rotation slots per Jacobi round (JMAX / 2)

// the small matrices of consecutive problems: leading dimension ld, ld^2 apart
struct Mat {
    double2 *p;
    int ld;
    Mat(const double2 *q = nullptr, int l = LD) : p(const_cast<double2 *>(q)), ld(l) {}
    __device__ double2 *of(int prob) const { return p + (size_t)prob * ld * ld; }
};

struct EigK {
    double2 *base;            // FP64 vectors of this k-point, stride nvec
    float2 *stage;            // FP32 staging for mixed-precision applies
    float2 *v32;              // FP32 copies for the Krylov Gram-Schmidt (mixed precision)
    const double *pfac;       // preconditioner factors of this k-point
    const float *pfac32;      // the same in FP32 (the mixed-precision Krylov chains)
    long long nvec;           // nb * ldg
    int ldg, ng;
};

// vector index sets: i < c1 -> s1 + ch*cs1 + i*st1;  else s2 + ch*cs2 + (i - c1)*st2
// (st = 1: a contiguous run; st = nc: one slot of every chain, the layout of
// the FP32 Krylov chains, whose slot i of all chains is contiguous)
struct VSet {
    int s1, c1, cs1, s2, c2, cs2, st1, st2;
    __host__ __device__ int count() const { return c1 + c2; }
    __host__ __device__ int at(int i, int ch) const {
        return i < c1 ? s1 + ch * cs1 + i * st1 : s2 + ch * cs2 + (i - c1) * st2;
    }
};
static VSet vs(int s1, int c1, int cs1 = 0, int s2 = 0, int c2 = 0, int cs2 = 0, int st1 = 1, int st2 = 1) {
    VSet v;
    v.s1 = s1; v.c1 = c1; v.cs1 = cs1; v.s2 = s2; v.c2 = c2; v.cs2 = cs2; v.st1 = st1; v.st2 = st2;
    return v;
}

// ---------------------------------------------------------------------------
// Fixed-order reduction of per-chunk partial Gram products (deterministic):
// one warp per output, lane l sums chunks l, l+32, ... and a fixed shuffle
// tree combines the lanes.  lower: only entries j <= i were computed (a
// Hermitian product); the upper triangle is written as the conjugate of the
// lower one.  Grid: (outputs / 8, problems), 256 threads.
__global__ void gram_reduce_kernel(const double2 *part, int nsplit, int ma, int mb, double2 *G, int lower) {
    const int prob = blockIdx.y;
    const int nout = ma * mb;
    const int o = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (o >= nout) return;                        // whole warp leaves together
    int i = o / mb, j = o % mb;
    const bool up = lower && j > i;
    const int src = up ? j * mb + i : o;
    const double2 *p = part + (size_t)prob * nsplit * nout + src;
    double2 s = make_double2(0.0, 0.0);
    for (int sp = lane; sp < nsplit; sp += 32) s = s + p[(size_t)sp * nout];
    for (int off = 16; off > 0; off >>= 1) {
        s.x += __shfl_down_sync(0xffffffffu, s.x, off);
        s.y += __shfl_down_sync(0xffffffffu, s.y, off);
    }
    if (lane == 0) {
        if (up) s.y = -s.y;
        G[(size_t)prob * LD * LD + i * LD + j] = s;
    }
}

// dst_i = src_i for index sets (FP64 -> FP64), or into / out of the FP32 stage
__global__ void copy_kernel(const EigK *ks, int nch, VSet S, VSet D, int mode) {
    // grid: (blocks along the vector, vector of the set, problem)
    // mode 0: base -> base; 1: base -> stage (to float); 2: stage -> base (to double);
    // 3: base -> v32 (to float); 4: v32 -> base (to double); 5: v32 -> v32
    const int prob = blockIdx.z, i = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    if (i >= S.count()) return;
    const long long sb = (long long)S.at(i, ch) * d.nvec, db = (long long)D.at(i, ch) * d.nvec;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < d.nvec;
         t += (long long)gridDim.x * blockDim.x) {
        const long long si = sb + t, di = db + t;
        if (mode == 0) d.base[di] = d.base[si];
        else if (mode == 1) d.stage[di] = make_float2((float)d.base[si].x, (float)d.base[si].y);
        else if (mode == 2) d.base[di] = make_double2((double)d.stage[si].x, (double)d.stage[si].y);
        else if (mode == 3) d.v32[di] = make_float2((float)d.base[si].x, (float)d.base[si].y);
        else if (mode == 4) d.base[di] = make_double2((double)d.v32[si].x, (double)d.v32[si].y);
        else d.v32[di] = d.v32[si];
    }
}

// W_ch = H_src - theta_ch S_src   (per-(k, ch) source indices); to32: W goes
// to the FP32 Gram-Schmidt copies (slot dst + ch of v32) instead
__global__ void krylov_residual_kernel(const EigK *ks, int nch, const int *srcH, const int *srcS,
                                       const double *theta, int dst, int to32) {
    const int prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const double th = theta[prob];
    const double2 *h = d.base + (long long)srcH[prob] * d.nvec;
    const double2 *s = d.base + (long long)srcS[prob] * d.nvec;
    double2 *w = d.base + (long long)(dst + ch) * d.nvec;
    float2 *w32 = to32 ? d.v32 + (long long)(dst + ch) * d.nvec : nullptr;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < d.nvec;
         t += (long long)gridDim.x * blockDim.x) {
        const double2 r = h[t] - rscale(th, s[t]);
        if (to32) w32[t] = make_float2((float)r.x, (float)r.y);
        else w[t] = r;
    }
}

// Bulk cycles of the mixed solver, on the FP32 copies (v32):
// W_ch = HX_seed - theta SX_seed (slot 0) or HK_{slot-1} - theta SK_{slot-1}
// of chain ch, the chains' slot s of chain ch at base + s*nc + ch
__global__ void krylov_residual32_kernel(const EigK *ks, int nch, int slot, const int *seed, const double *theta,
                                         int oHX, int oSX, int oHK, int oSK, int nc, int dst) {
    const int prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    __shared__ float th_s;
    if (threadIdx.x == 0) th_s = (float)theta[prob];
    __syncthreads();
    const float th = th_s;
    const int ih = slot == 0 ? oHX + seed[prob] : oHK + (slot - 1) * nc + ch;
    const int is = slot == 0 ? oSX + seed[prob] : oSK + (slot - 1) * nc + ch;
    const float2 *h = d.v32 + (long long)ih * d.nvec;
    const float2 *s = d.v32 + (long long)is * d.nvec;
    float2 *w = d.v32 + (long long)(dst + ch) * d.nvec;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < d.nvec;
         t += (long long)gridDim.x * blockDim.x) {
        const float2 hv = h[t], sv = s[t];
        w[t] = make_float2(fmaf(-th, sv.x, hv.x), fmaf(-th, sv.y, hv.y));
    }
}

// R_i = HX_i - eps_i SX_i on the FP32 copies
__global__ void residual32_kernel(const EigK *ks, int M, int oHX, int oSX, int dst, const double *eps) {
    const int k = blockIdx.y;
    const EigK d = ks[k];
    const long long total = (long long)M * d.nvec;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / d.nvec);
        const long long t = e - (long long)i * d.nvec;
        const float ev = (float)eps[k * M + i];
        const float2 hv = d.v32[(long long)(oHX + i) * d.nvec + t], sv = d.v32[(long long)(oSX + i) * d.nvec + t];
        d.v32[(long long)(dst + i) * d.nvec + t] = make_float2(fmaf(-ev, sv.x, hv.x), fmaf(-ev, sv.y, hv.y));
    }
}

// R_i = HX_i - eps_i SX_i into dst
__global__ void residual_kernel(const EigK *ks, int M, int oX, int oHX, int oSX, int dst, const double *eps) {
    const int k = blockIdx.y;
    const EigK d = ks[k];
    const long long total = (long long)M * d.nvec;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        int i = (int)(e / d.nvec);
        long long t = e - (long long)i * d.nvec;
        double ev = eps[k * M + i];
        d.base[(long long)(dst + i) * d.nvec + t] =
            d.base[(long long)(oHX + i) * d.nvec + t] - rscale(ev, d.base[(long long)(oSX + i) * d.nvec + t]);
    }
    (void)oX;
}

// Re <A_i, B_i> over one of gridDim.z chunks of the vector into part[(prob m + i)
// chunks + chunk] (block reduction with warp shuffles); coldot_sum_kernel adds
// the chunks in order.  Bound by the read of the vectors: one CTA a vector
// (73 us for 90 vectors of 115 k elements) left half the SMs idle.
// F32: on the FP32 copies, per-thread sums in FP32 and the rest in FP64
template <bool F32>
__global__ void coldot_kernel(const EigK *ks, int nch, VSet A, VSet B, double *part) {
    typedef typename std::conditional<F32, float2, double2>::type T2;
    typedef typename std::conditional<F32, float, double>::type T;
    const int i = blockIdx.x, prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const T2 *vb = F32 ? reinterpret_cast<const T2 *>(d.v32) : reinterpret_cast<const T2 *>(d.base);
    const T2 *a = vb + (long long)A.at(i, ch) * d.nvec;
    const T2 *b = vb + (long long)B.at(i, ch) * d.nvec;
    const long long t0 = blockIdx.z * d.nvec / gridDim.z, t1 = (blockIdx.z + 1) * d.nvec / gridDim.z;
    T st = T(0);
#pragma unroll 4
    for (long long t = t0 + threadIdx.x; t < t1; t += blockDim.x) st = fma(a[t].x, b[t].x, fma(a[t].y, b[t].y, st));
    double s = (double)st;
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    __shared__ double ws[32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? ws[threadIdx.x] : 0.0;
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (threadIdx.x == 0) part[((size_t)prob * A.count() + i) * gridDim.z + blockIdx.z] = s;
    }
}
__global__ void coldot_sum_kernel(const double *part, int chunks, int n, double *out) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    double s = 0.0;
    for (int c = 0; c < chunks; ++c) s += part[(size_t)e * chunks + c];
    out[e] = s;
}

// new Krylov vector: K = W / ||W||_S, SK = SW / ||W||_S, HK slot cleared;
// a norm below the breakdown threshold marks the slot dead (zero vector).
__global__ void normalize_kernel(const EigK *ks, int nch, int oW, int oSW, int kV, int kS, int cs,
                                 int slot, const double *nrm2, int *alive, int kd, int k32, int sk32, int nc) {
    const int prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    __shared__ double inv_s;
    if (threadIdx.x == 0) {
        const double n2 = nrm2[prob];
        const bool ok = n2 > 1e-24;
        inv_s = ok ? 1.0 / sqrt(n2) : 0.0;
        if (blockIdx.x == 0) alive[prob * kd + slot] = ok ? 1 : 0;
    }
    __syncthreads();
    const double inv = inv_s;
    const double2 *w = d.base + (long long)(oW + ch) * d.nvec;
    const double2 *sw = d.base + (long long)(oSW + ch) * d.nvec;
    double2 *kv = d.base + (long long)(kV + ch * cs + slot) * d.nvec;
    double2 *ksv = d.base + (long long)(kS + ch * cs + slot) * d.nvec;
    // FP32 copies for later Gram-Schmidt steps (k32 < 0: none)
    float2 *kv32 = k32 >= 0 ? d.v32 + (long long)(k32 + slot * nc + ch) * d.nvec : nullptr;
    float2 *ks32 = k32 >= 0 ? d.v32 + (long long)(sk32 + slot * nc + ch) * d.nvec : nullptr;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < d.nvec;
         t += (long long)gridDim.x * blockDim.x) {
        const double2 a = rscale(inv, w[t]), b = rscale(inv, sw[t]);
        kv[t] = a;
        ksv[t] = b;
        if (kv32) {
            kv32[t] = make_float2((float)a.x, (float)a.y);
            ks32[t] = make_float2((float)b.x, (float)b.y);
        }
    }
}

// FP32 chain slot (bulk cycles): K[slot] = W / ||W||_S and SK[slot] (which
// holds S W) scaled in place; slot s of chain ch at base + s*nc + ch
__global__ void normalize32_kernel(const EigK *ks, int nch, int oW, int oK, int oSK, int nc, int slot,
                                   const double *nrm2, int *alive, int kd) {
    const int prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    // the scale once per block (FP64 square roots and divisions are slow)
    __shared__ float inv_s;
    if (threadIdx.x == 0) {
        const double n2 = nrm2[prob];
        const bool ok = n2 > 1e-24;
        inv_s = ok ? (float)(1.0 / sqrt(n2)) : 0.f;
        if (blockIdx.x == 0) alive[prob * kd + slot] = ok ? 1 : 0;
    }
    __syncthreads();
    const float inv = inv_s;
    const float2 *w = d.v32 + (long long)(oW + ch) * d.nvec;
    float2 *kv = d.v32 + (long long)(oK + slot * nc + ch) * d.nvec;
    float2 *sk = d.v32 + (long long)(oSK + slot * nc + ch) * d.nvec;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < d.nvec;
         t += (long long)gridDim.x * blockDim.x) {
        const float2 a = w[t], b = sk[t];
        kv[t] = make_float2(inv * a.x, inv * a.y);
        sk[t] = make_float2(inv * b.x, inv * b.y);
    }
}

// residual norms and seeds: res[k*M + i] = sqrt(max(0, dot)); seed = argmax over a range
__global__ void seed_kernel(const double *dots, int M, int mconv, int nk, int nch, int bsize, double *res,
                            const double *eps, int *seed, double *theta, int *srcH, int *srcS,
                            int oHX, int oSX) {
    const int prob = blockIdx.x * blockDim.x + threadIdx.x;
    if (prob >= nk * nch) return;
    const int k = prob / nch, ch = prob % nch;
    if (ch == 0)
        for (int i = 0; i < M; ++i) res[k * M + i] = sqrt(fmax(0.0, dots[k * M + i]));
    int lo = nch == 1 ? 0 : ch * bsize, hi = nch == 1 ? mconv : min(M, lo + bsize);
    int best = lo;
    double bv = -1.0;
    for (int i = lo; i < hi; ++i) {
        double v = sqrt(fmax(0.0, dots[k * M + i]));
        if (v > bv) { bv = v; best = i; }
    }
    seed[prob] = best;
    theta[prob] = eps[k * M + best];
    srcH[prob] = oHX + best;
    srcS[prob] = oSX + best;
}

// ---------------------------------------------------------------------------
// Jacobi diagonalization of Hermitian m x m matrices (m <= JMAX), parallel
// (round-robin) ordering: m'/2 disjoint rotations per round.
//
// A problem takes gridDim.x CTAs.  Every one of them holds all of A in shared
// memory and computes the same rotations, but only its share of the rows of
// the eigenvector matrix, which is most of the work of one CTA and needs
// nothing from the other rows: no communication, and the result does not
// depend on the number of CTAs.  Bound by instruction issue (FP32) or the
// FP64 pipe of one SM, so the index arithmetic of the 2 x 2 blocks is done
// once for all rounds and blocks whose two rotations are the identity are
// skipped.  The FP32 problems of 90 to 95 columns of a solve took 1.1 ms on the
// mean with one CTA each and take 0.5 ms with 15.

// rotation of pair (p, q): columns times diag(1, conj e) [[c, s], [-s, c]]
template <typename T> struct __align__(16) JRot {
    T c, s;
    typename std::conditional<std::is_same<T, float>::value, float2, double2>::type e;
};
constexpr int kJacobiThreads = 512;                       // at most
constexpr int kJacobiBlocks = 4;                         // 2x2 blocks per thread, at most
static_assert(JPAIRS * (JPAIRS + 1) / 2 <= kJacobiBlocks * kJacobiThreads, "a thread's blocks");
template <typename T> constexpr size_t jacobi_smem(int m, int rows) {
    return (((size_t)(m + rows) * m + 1) & ~(size_t)1) * 2 * sizeof(T) + JPAIRS * (sizeof(JRot<T>) + 2 * sizeof(T) + 2 * sizeof(int));
}

// A from the lower triangle of the problem's G (Hermitian completion: with the
// subspace ordered [roots | Krylov vectors], the coupling block comes from
// K^H (H X), which uses the roots' HX rather than the Krylov vectors' HK,
// which may come from a reduced-precision apply); dead slots become decoupled
// with a huge diagonal.  full (or null): the completed matrix, of which this
// CTA writes rows [r0, r1) (leading dimension m).  Returns the squared
// Frobenius norm of the live part (all threads).
template <typename T2>
__device__ double jacobi_load(const double2 *g, int m, const int *dead, int dead_ofs, T2 *A, double2 *full, int r0, int r1,
                              double *red) {
    double f = 0.0;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, j = e % m;
        double2 v = i >= j ? g[i * LD + j] : g[j * LD + i];
        if (i < j) v.y = -v.y;
        if (i == j) v.y = 0.0;
        const bool di = dead && dead[i] == 0 && i >= dead_ofs;
        const bool dj = dead && dead[j] == 0 && j >= dead_ofs;
        if (di || dj) v = make_double2((i == j) ? 1e30 : 0.0, 0.0);
        else f += v.x * v.x + v.y * v.y;
        A[e] = mk((decltype(A[0].x))v.x, (decltype(A[0].x))v.y);
        if (full && i >= r0 && i < r1) full[e] = v;
    }
    for (int off = 16; off > 0; off >>= 1) f += __shfl_down_sync(0xffffffffu, f, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = f;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    __syncthreads();
    return s;
}

// Sweeps until the off-diagonal Frobenius norm is <= rel_tol * that of the
// matrix.  sort: eigenvalues ascending (else column i stays near slot i, dead
// slots exactly there).  T = float: the rotations in FP32.
template <typename T>
__global__ void __launch_bounds__(kJacobiThreads) jacobi_kernel(const double2 *G, int m, const int *dead, int dead_stride,
                                                                int dead_ofs, double *evals, Mat evecs, double2 *full, int sort,
                                                                int max_sweeps, double rel_tol) {
    typedef typename std::conditional<std::is_same<T, float>::value, float2, double2>::type T2;
    extern __shared__ __align__(16) unsigned char sm[];
    const int prob = blockIdx.y, tid = threadIdx.x, nt = blockDim.x;
    const int r0 = blockIdx.x * m / gridDim.x, r1 = (blockIdx.x + 1) * m / gridDim.x, rows = r1 - r0;
    const T skip_rel = std::is_same<T, float>::value ? T(1e-7) : T(1e-15);
    T2 *A = reinterpret_cast<T2 *>(sm);
    T2 *V = A + m * m;                                    // rows r0 .. r1 - 1
    JRot<T> *rot = reinterpret_cast<JRot<T> *>(A + (((m + (m + gridDim.x - 1) / gridDim.x) * m + 1) & ~1u));
    T *diag = reinterpret_cast<T *>(rot + JPAIRS);        // per pair: the rotated diagonal
    int2 *pq = reinterpret_cast<int2 *>(diag + 2 * JPAIRS);
    __shared__ double red[32];
    __shared__ int perm[LD];
    const double fro2 = jacobi_load(G + (size_t)prob * LD * LD, m, dead ? dead + prob * dead_stride : nullptr, dead_ofs, A,
                                    full ? full + (size_t)prob * m * m : nullptr, r0, r1, red);
    for (int e = tid; e < rows * m; e += nt) V[e] = mk(T(e % m == r0 + e / m ? 1 : 0), T(0));
    const int mp = (m + 1) & ~1;      // players, padded to even
    const int npair = mp / 2;
    // this thread's 2x2 blocks (I >= J) of the pair partition
    int bI[kJacobiBlocks], bJ[kJacobiBlocks];
#pragma unroll
    for (int k = 0; k < kJacobiBlocks; ++k) {
        const int e = tid + k * nt;
        int I = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
        while (I * (I + 1) / 2 > e) --I;
        while ((I + 1) * (I + 2) / 2 <= e) ++I;
        bI[k] = I < npair ? I : -1;
        bJ[k] = e - I * (I + 1) / 2;
    }
    __syncthreads();
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        double off2 = 0.0;
        for (int e = tid; e < m * m; e += nt)
            if (e / m > e % m) off2 += (double)(A[e].x * A[e].x + A[e].y * A[e].y);
        for (int off = 16; off > 0; off >>= 1) off2 += __shfl_down_sync(0xffffffffu, off2, off);
        if ((tid & 31) == 0) red[tid >> 5] = off2;
        __syncthreads();
        off2 = 0.0;
        for (int w = 0; w < nt / 32; ++w) off2 += 2 * red[w];
        __syncthreads();                                  // red is free again, and everyone leaves together
        if (off2 <= rel_tol * rel_tol * fro2) break;
        for (int r = 0; r < mp - 1; ++r) {
            // rotation of every pair of the round (q >= m: an index left
            // alone this round, identity)
            if (tid < npair) {
                const int a = tid == 0 ? 0 : ((r + tid - 1) % (mp - 1)) + 1;
                const int b = tid == 0 ? ((r + mp - 2) % (mp - 1)) + 1 : ((r + mp - 1 - tid - 1) % (mp - 1)) + 1;
                const int p = min(a, b), q = max(a, b);
                JRot<T> w;
                w.c = 1, w.s = 0, w.e = mk(T(1), T(0));
                if (q < m) {
                    const T2 apq = A[p * m + q];
                    const T app = A[p * m + p].x, aqq = A[q * m + q].x;
                    // rotations below rounding level of the diagonal are
                    // skipped (in FP64 first by the components' bound: the
                    // square roots take 64 clocks an operation)
                    const T big = T(1.5) * max(fabs(apq.x), fabs(apq.y));
                    if (big > T(1e-30) && (sizeof(T) == 4 || big * big > skip_rel * skip_rel * fabs(app * aqq))) {
                        const T mag = hypot(apq.x, apq.y);
                        if (mag > skip_rel * sqrt(fabs(app * aqq)) && mag > T(1e-30)) {
                            w.e = mk(apq.x / mag, apq.y / mag);
                            const T th = (aqq - app) / (T(2) * mag);
                            const T t = (th >= 0 ? T(1) : T(-1)) / (fabs(th) + sqrt(th * th + T(1)));
                            w.c = T(1) / sqrt(t * t + T(1));
                            w.s = t * w.c;
                            diag[2 * tid] = app - t * mag;
                            diag[2 * tid + 1] = aqq + t * mag;
                        }
                    }
                }
                pq[tid] = make_int2(p, q);
                rot[tid] = w;
            }
            __syncthreads();
            // A <- J^H A J by 2x2 blocks (rows of pair I, columns of pair J,
            // I >= J; the block above the diagonal is written as the
            // conjugate transpose)
#pragma unroll
            for (int k = 0; k < kJacobiBlocks; ++k) {
                const int I = bI[k], J = bJ[k];
                if (I < 0) break;
                const T sI = rot[I].s, sJ = rot[J].s;
                if (sI == T(0) && sJ == T(0)) continue;
                const int pI = pq[I].x, qI = pq[I].y, pJ = pq[J].x, qJ = pq[J].y;
                const bool vI = qI < m, vJ = qJ < m;
                if (I == J) {
                    A[pI * m + pI] = mk(diag[2 * I], T(0));
                    A[qI * m + qI] = mk(diag[2 * I + 1], T(0));
                    A[pI * m + qI] = A[qI * m + pI] = czero<T2>();
                    continue;
                }
                T2 a00 = A[pI * m + pJ];
                T2 a01 = vJ ? A[pI * m + qJ] : czero<T2>();
                T2 a10 = vI ? A[qI * m + pJ] : czero<T2>();
                T2 a11 = (vI && vJ) ? A[qI * m + qJ] : czero<T2>();
                if (sJ != T(0)) {     // columns pJ, qJ
                    const JRot<T> w = rot[J];
                    const T2 ec = mk(w.e.x, -w.e.y);
                    T2 x = a00, y = cmul(ec, a01);
                    a00 = rscale(w.c, x) - rscale(w.s, y);
                    a01 = rscale(w.s, x) + rscale(w.c, y);
                    x = a10;
                    y = cmul(ec, a11);
                    a10 = rscale(w.c, x) - rscale(w.s, y);
                    a11 = rscale(w.s, x) + rscale(w.c, y);
                }
                if (sI != T(0)) {     // rows pI, qI
                    const JRot<T> w = rot[I];
                    T2 x = a00, y = cmul(w.e, a10);
                    a00 = rscale(w.c, x) - rscale(w.s, y);
                    a10 = rscale(w.s, x) + rscale(w.c, y);
                    x = a01;
                    y = cmul(w.e, a11);
                    a01 = rscale(w.c, x) - rscale(w.s, y);
                    a11 = rscale(w.s, x) + rscale(w.c, y);
                }
                A[pI * m + pJ] = a00;
                A[pJ * m + pI] = mk(a00.x, -a00.y);
                if (vJ) {
                    A[pI * m + qJ] = a01;
                    A[qJ * m + pI] = mk(a01.x, -a01.y);
                }
                if (vI) {
                    A[qI * m + pJ] = a10;
                    A[pJ * m + qI] = mk(a10.x, -a10.y);
                }
                if (vI && vJ) {
                    A[qI * m + qJ] = a11;
                    A[qJ * m + qI] = mk(a11.x, -a11.y);
                }
            }
            // V <- V J: half a warp per pair, a lane per row
            for (int pi = tid / 16; pi < npair; pi += nt / 16) {
                const JRot<T> w = rot[pi];
                if (w.s == T(0)) continue;
                const int2 c = pq[pi];
                const T2 ec = mk(w.e.x, -w.e.y);
                for (int row = tid % 16; row < rows; row += 16) {
                    T2 *v = V + row * m;
                    const T2 x = v[c.x], y = cmul(ec, v[c.y]);
                    v[c.x] = rscale(w.c, x) - rscale(w.s, y);
                    v[c.y] = rscale(w.s, x) + rscale(w.c, y);
                }
            }
            __syncthreads();
        }
    }
    // slot of every column: its rank on the diagonal (equal values, the dead
    // slots, in their order)
    if (tid < m) perm[tid] = tid;
    __syncthreads();
    if (sort && tid < m) {
        const T v = A[tid * m + tid].x;
        int rank = 0;
        for (int j = 0; j < m; ++j) {
            const T u = A[j * m + j].x;
            rank += u < v || (u == v && j < tid);
        }
        perm[rank] = tid;
    }
    __syncthreads();
    if (blockIdx.x == 0 && tid < m) evals[(size_t)prob * LD + tid] = A[perm[tid] * m + perm[tid]].x;
    double2 *out = evecs.of(prob);
    for (int e = tid; e < rows * m; e += nt) {
        const T2 v = V[e / m * m + perm[e % m]];
        out[(r0 + e / m) * evecs.ld + e % m] = make_double2(v.x, v.y);
    }
}

// FP64 result from FP32 sweeps: X0 of the FP32 sweeps is refined by steps
// of the Ogita-Aishima iteration (Iterative refinement for symmetric
// eigenvalue decomposition, Japan J. Indust. Appl. Math. 35, 2018): with
// S = X^H A X, P = X^H X, R = I - P and l_i = S_ii / P_ii,
//   X <- X + X E,  E_ij = (S_ij + l_j R_ij) / (l_j - l_i),  E_ii = R_ii / 2,
// which squares the error of the vectors and of their orthogonality.  Where
// that E_ij is above lim (neighbours that FP32 does not separate), R_ij / 2
// only makes the two orthogonal and the FP64 sweeps on X^H A X rotate them.  A
// step leaves I - P = E^H E + O(R^2), at most (m lim)^2 where all corrections
// are at lim and in phase: 1.3e-4 after the first step with lim = 1e-4, 1e-8
// after the second with 1e-8, and 1e-16 after a third that only
// orthonormalizes, E = R / 2 (without it, a cluster coupled at 1e-4 of its gaps
// lost 2e-11 of 95 vectors' orthonormality, which the FP64 sweeps, unitary
// themselves, do not restore).
__global__ void refine_kernel(Mat Sm, Mat Pm, Mat Em, int m, double lim) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m * m) return;
    const int i = t / m, j = t % m;
    if (i < j) return;
    const double2 *S = Sm.of(blockIdx.y), *P = Pm.of(blockIdx.y);
    double2 *E = Em.of(blockIdx.y);
    const double2 p = P[i * Pm.ld + j];
    if (i == j) {
        E[i * Em.ld + i] = make_double2(0.5 * (1.0 - p.x), 0.0);
        return;
    }
    // the lower triangle, and E_ji = conj(R_ij - E_ij), so that E + E^H = R
    // holds to rounding however small the gap
    const double li = S[i * Sm.ld + i].x / P[i * Pm.ld + i].x, lj = S[j * Sm.ld + j].x / P[j * Pm.ld + j].x;
    const double2 sv = S[i * Sm.ld + j];
    const double nx = sv.x - lj * p.x, ny = sv.y - lj * p.y, gap = lj - li;
    const bool far = fmax(fabs(nx), fabs(ny)) <= lim * fabs(gap) && gap != 0.0;
    const double2 v = far ? make_double2(nx / gap, ny / gap) : make_double2(-0.5 * p.x, -0.5 * p.y);
    E[i * Em.ld + j] = v;
    E[j * Em.ld + i] = make_double2(-p.x - v.x, p.y + v.y);
}

// U = L^{-H} with G = L L^H (G Hermitian positive definite, m <= JMAX), one
// CTA per problem, the matrix in shared memory throughout: right-looking
// Cholesky (a warp per row of the trailing update), then the lower triangle
// inverted in place row by row (row i of L^{-1} needs row i of L and the rows
// above it: kCholSplit threads per column share the sum).  Latency bound, two
// barriers a column: m = 90 in FP32 took 0.66 ms with one thread per column
// of the inverse reading it back from global memory; now 0.10 ms.
// T = float: the arithmetic in FP32 (the bulk cycles' S-Grams, which are the
// identity up to the FP32 Gram-Schmidt error).
constexpr int kCholThreads = 512, kCholSplit = 4;
template <typename T> constexpr size_t cholinv_smem(int m) {
    return ((size_t)m * (m + 1) + m + (size_t)kCholSplit * JMAX) * 2 * sizeof(T);
}
template <typename T>
__global__ void __launch_bounds__(kCholThreads) cholinv_kernel(const double2 *G, int m, double2 *U, int *status) {
    typedef typename std::conditional<std::is_same<T, float>::value, float2, double2>::type T2;
    extern __shared__ __align__(16) unsigned char sm[];
    const int ld = m + 1;                   // rows padded by one: columns are free of bank conflicts
    T2 *L = reinterpret_cast<T2 *>(sm);     // m x ld, lower
    T2 *row = L + m * ld;                   // m
    T2 *red = row + m;                      // kCholSplit x JMAX
    __shared__ T rpiv;
    const int prob = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const double2 *g = G + (size_t)prob * LD * LD;
    double2 *u = U + (size_t)prob * LD * LD;
    for (int i = warp; i < m; i += kCholThreads / 32)
        for (int j = lane; j <= i; j += 32) {
            const double2 v = g[i * LD + j];
            L[i * ld + j] = mk((T)v.x, (T)v.y);
        }
    __syncthreads();
    for (int j = 0; j < m; ++j) {
        if (tid == 0) {
            T d = L[j * ld + j].x;
            if (!(d > T(0))) {
                status[prob] = 1;
                d = std::is_same<T, float>::value ? T(1e-30) : T(1e-300);
            }
            const T piv = sqrt(d);
            rpiv = T(1) / piv;
            L[j * ld + j] = mk(piv, T(0));
        }
        __syncthreads();
        const T r = rpiv;
        // column j scaled into `row`, then the trailing update L[i][c] -= l_i conj(l_c), j < c <= i
        for (int i = j + 1 + tid; i < m; i += kCholThreads) {
            const T2 v = rscale(r, L[i * ld + j]);
            L[i * ld + j] = v;
            row[i] = v;
        }
        __syncthreads();
        for (int i = j + 1 + warp; i < m; i += kCholThreads / 32) {
            const T2 li = row[i];
            for (int c = j + 1 + lane; c <= i; c += 32) L[i * ld + c] = L[i * ld + c] - cmul_c(li, row[c]);
        }
        __syncthreads();
    }
    // row i of Z = L^{-1}: Z[i][c] = -(1 / L_ii) sum_{c <= q < i} L[i][q] Z[q][c]
    const int part = tid / (kCholThreads / kCholSplit), c0 = tid % (kCholThreads / kCholSplit);
    static_assert(kCholThreads / kCholSplit >= JMAX, "a thread per column and part");
    for (int i = 0; i < m; ++i) {
        const T r = T(1) / L[i * ld + i].x;
        if (c0 < i) {
            T2 s = mk(T(0), T(0));
            // an equal share of the column's terms for every part
            const int n = i - c0, q1 = c0 + (part + 1) * n / kCholSplit;
            for (int q = c0 + part * n / kCholSplit; q < q1; ++q) cfma(s, L[i * ld + q], L[q * ld + c0]);
            red[part * JMAX + c0] = s;
        }
        __syncthreads();
        if (tid < i) {
            T2 s = red[tid];
#pragma unroll
            for (int p = 1; p < kCholSplit; ++p) s = s + red[p * JMAX + tid];
            L[i * ld + tid] = rscale(-r, s);
        } else if (tid == i) {
            L[i * ld + i] = mk(r, T(0));
        }
        __syncthreads();
    }
    for (int c = warp; c < m; c += kCholThreads / 32)
        for (int i = lane; i < m; i += 32) {
            const T2 z = i >= c ? L[i * ld + c] : mk(T(0), T(0));
            u[c * LD + i] = make_double2((double)z.x, (double)-z.y);
        }
}

// Maximum-overlap selection of bsz Ritz pairs in a block (+ new roots).
__global__ void select_kernel(const double *evals, const double2 *evecs, int mB, int b, int M, int nblk,
                              int nprob, double *eps, double2 *Ysel) {
    const int prob = blockIdx.x * blockDim.x + threadIdx.x;
    if (prob >= nprob) return;
    const int k = prob / nblk, blk = prob % nblk;
    const int lo = blk * b, bsz = min(b, M - lo);
    const double *w = evals + (size_t)prob * LD;
    const double2 *Y = evecs + (size_t)prob * LD * LD;
    double ov[LD];
    int chosen[LD];
    bool used[LD];
    for (int l = 0; l < mB; ++l) {
        double s = 0.0;
        for (int i = 0; i < bsz; ++i) s += Y[i * LD + l].x * Y[i * LD + l].x + Y[i * LD + l].y * Y[i * LD + l].y;
        ov[l] = s;
        used[l] = false;
    }
    for (int c = 0; c < bsz; ++c) {     // stable top-bsz by overlap
        int best = -1;
        for (int l = 0; l < mB; ++l)
            if (!used[l] && (best < 0 || ov[l] > ov[best])) best = l;
        chosen[c] = best;
        used[best] = true;
    }
    double lowest_in = 1e300;
    for (int i = 0; i < bsz; ++i) lowest_in = fmin(lowest_in, eps[k * M + lo + i]);
    for (int l = 0; l < mB; ++l) {
        if (used[l]) continue;
        if (w[l] < lowest_in && ov[l] < 0.5) {
            int worst = 0;
            for (int c = 1; c < bsz; ++c)
                if (w[chosen[c]] > w[chosen[worst]]) worst = c;
            if (w[l] < w[chosen[worst]]) {
                used[chosen[worst]] = false;
                chosen[worst] = l;
                used[l] = true;
            }
        }
    }
    for (int i = 1; i < bsz; ++i) {     // sort chosen by Ritz value
        int x = chosen[i], j = i - 1;
        while (j >= 0 && w[chosen[j]] > w[x]) { chosen[j + 1] = chosen[j]; --j; }
        chosen[j + 1] = x;
    }
    double2 *ys = Ysel + (size_t)prob * LD * LD;
    for (int c = 0; c < bsz; ++c) {
        for (int r = 0; r < mB; ++r) ys[r * LD + c] = Y[r * LD + chosen[c]];
        eps[k * M + lo + c] = w[chosen[c]];
    }
}

__global__ void take_evals_kernel(const double *evals, int M, int nk, double *eps) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < M * nk) eps[e] = evals[(size_t)(e / M) * LD + (e % M)];
}

// Banded solves on vector ranges of every k-point: L L^T y = x, one thread per
// G column (FP64: per real component of one, since the factors are real and an
// FP64 warp instruction holds its pipe for 64 clocks: 45 -> 28 us for small
// problems) and NV vectors; the last K-1 solution values ride in registers.
// per_g: the k-point's factors L_G[j][d] stored as pfac[(j*K + d)*ldg + G]
// (coalesced over G); else the G-independent L_z.  F32: on the FP32
// Gram-Schmidt copies with FP32 factors (a preconditioner solve, whose
// rounding only changes which Krylov space is built).
// Rows go in tiles of PD: while a tile's recurrence runs, the next tile's
// right-hand sides and factors (none of which depends on it) are in flight,
// and NV vectors share every factor: with one vector per thread the factors
// were 7 of 9 bytes read, from L2, and each tile waited for its own loads.
template <int K, bool F32, int NV>
__global__ void __launch_bounds__(64) eig_banded_solve_kernel(const EigK *ks, const void *Lbv, int per_g, int nb, int src,
                                                              int dst, int nv) {
    typedef typename std::conditional<F32, float, double>::type T;
    typedef typename std::conditional<F32, float2, double>::type T2;      // a thread's element: a column, or one component
    constexpr int CP = F32 ? 1 : 2;                                        // elements per column
    const int nvt = (nv + NV - 1) / NV;
    const int k = blockIdx.z / nvt, v0 = blockIdx.z % nvt * NV, nvl = min(NV, nv - v0);
    const EigK d = ks[k];
    const int t = blockIdx.x * blockDim.x + threadIdx.x, g = t / CP;
    if (g >= d.ldg) return;
    T2 *vb = F32 ? reinterpret_cast<T2 *>(d.v32) : reinterpret_cast<T2 *>(d.base);
    const T *Lb = reinterpret_cast<const T *>(Lbv);
    const T *pf = F32 ? reinterpret_cast<const T *>(d.pfac32) : reinterpret_cast<const T *>(d.pfac);
    const int ldg = d.ldg, row = CP * ldg;
    const long long nvec = CP * d.nvec;
    // vector v of the thread (past the last one: the last one again, not written)
    const T2 *xv[NV];
    T2 *yv[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        xv[v] = vb + (src + v0 + min(v, nvl - 1)) * nvec + t;
        yv[v] = vb + (dst + v0 + min(v, nvl - 1)) * nvec + t;
    }
    if (g >= d.ng) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
            for (int j = 0; j < nb; ++j) yv[v][j * row] = T2{};
        return;
    }
    // factors hold L[j][j-d] for d >= 1 (0 where j < d) and 1 / L[j][j] at
    // d = 0; fd: entry (j, d) is fp[j * fr + d * fd]
    const T *fp = per_g ? pf + g : Lb;
    const int fd = per_g ? ldg : 1, fr = K * fd;
    constexpr int PD = F32 ? 4 : 2;
    struct Tile {
        T2 x[NV][PD];
        T f[PD][K];
    };
    T2 win[NV][K];                                  // win[v][i]: solution i + 1 rows back
    auto clear = [&]() {
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int i = 0; i < K; ++i) win[v][i] = T2{};
    };
    // one row: s - sum_d f_d win_d, the newest solution last (only its FMA waits for the previous row)
    auto solve = [&](int v, T2 s, const T(&f)[K]) {
#pragma unroll
        for (int dd = K - 1; dd >= 1; --dd) rfma(s, -f[dd], win[v][dd - 1]);
        s = rscale(f[0], s);
#pragma unroll
        for (int i = K - 1; i > 0; --i) win[v][i] = win[v][i - 1];
        win[v][0] = s;
        return s;
    };
    auto load_f = [&](Tile &t, int j0) {
#pragma unroll
        for (int u = 0; u < PD; ++u) {
            const int j = min(j0 + u, nb - 1), o = j * fr;
#pragma unroll
            for (int dd = 0; dd < K; ++dd) t.f[u][dd] = fp[o + dd * fd];
#pragma unroll
            for (int v = 0; v < NV; ++v) t.x[v][u] = xv[v][j * row];
        }
    };
    auto load_b = [&](Tile &t, int j1) {
#pragma unroll
        for (int u = 0; u < PD; ++u) {
            // (past the last row the solutions are still zero: any finite factor will do)
            const int j = max(j1 - u, 0), o = j * fr;
#pragma unroll
            for (int dd = 0; dd < K; ++dd) t.f[u][dd] = fp[j + dd < nb ? o + dd * (fr + fd) : o];
#pragma unroll
            for (int v = 0; v < NV; ++v) t.x[v][u] = yv[v][j * row];
        }
    };
    auto run_f = [&](const Tile &t, int j0) {
#pragma unroll
        for (int u = 0; u < PD; ++u) {
            if (j0 + u >= nb) break;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const T2 r = solve(v, t.x[v][u], t.f[u]);
                if (NV == 1 || v < nvl) yv[v][(j0 + u) * row] = r;
            }
        }
    };
    auto run_b = [&](const Tile &t, int j1) {
#pragma unroll
        for (int u = 0; u < PD; ++u) {
            if (j1 - u < 0) break;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const T2 r = solve(v, t.x[v][u], t.f[u]);
                if (NV == 1 || v < nvl) yv[v][(j1 - u) * row] = r;
            }
        }
    };
    Tile ta, tb;
    clear();
    load_f(ta, 0);
    for (int j0 = 0; j0 < nb; j0 += 2 * PD) {
        if (j0 + PD < nb) load_f(tb, j0 + PD);
        run_f(ta, j0);
        if (j0 + 2 * PD < nb) load_f(ta, j0 + 2 * PD);
        if (j0 + PD < nb) run_f(tb, j0 + PD);
    }
    clear();
    load_b(ta, nb - 1);
    for (int j1 = nb - 1; j1 >= 0; j1 -= 2 * PD) {
        if (j1 - PD >= 0) load_b(tb, j1 - PD);
        run_b(ta, j1);
        if (j1 - 2 * PD >= 0) load_b(ta, j1 - 2 * PD);
        if (j1 - PD >= 0) run_b(tb, j1 - PD);
    }
}

// A^H B, one warp per row i and up to GJ columns: the lanes stride over an
// n-chunk with coalesced loads, each holding GJ complex partial sums in
// registers, then reduce them by warp shuffles.  Grid: (n-chunks, problems,
// row groups of 8 x column groups of GJ).
// GJ, the column-group width, is picked per call so that predicated-off
// column slots (which still occupy the FP64 pipe) are few.
// F32: the vectors are the FP32 Gram-Schmidt copies (v32) and the partial
// sums are FP32 (the reduction over chunks stays FP64).
template <bool F32, int GJ>
__global__ void __launch_bounds__(256) gram_rows_kernel(const EigK *ks, int nch, VSet A, VSet B, int nsplit,
                                                        int colgroups, double2 *part, int lower) {
    typedef typename std::conditional<F32, float2, double2>::type T2;
    typedef typename std::conditional<F32, float, double>::type T;
    const int split = blockIdx.x, prob = blockIdx.y;
    const int rg = blockIdx.z / colgroups, cg = blockIdx.z % colgroups;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const int ma = A.count(), mb = B.count();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = rg * 8 + warp;
    const int j0 = cg * GJ, nj = min(GJ, mb - j0);
    if (i >= ma || nj <= 0) return;                     // whole warp leaves together
    if (lower && j0 > i) return;                        // tile above the diagonal
    const long long n = d.nvec;
    const long long chunk = (n + nsplit - 1) / nsplit;
    const long long t0 = split * chunk, t1 = min(n, t0 + chunk);
    const T2 *vb = F32 ? reinterpret_cast<const T2 *>(d.v32) : reinterpret_cast<const T2 *>(d.base);
    const T2 *a = vb + (long long)A.at(i, ch) * n;
    const T2 *bp[GJ];
#pragma unroll
    for (int jj = 0; jj < GJ; ++jj) bp[jj] = vb + (long long)B.at(j0 + (jj < nj ? jj : 0), ch) * n;
    T sx[GJ], sy[GJ];
#pragma unroll
    for (int jj = 0; jj < GJ; ++jj) sx[jj] = sy[jj] = T(0);
    for (long long t = t0 + lane; t < t1; t += 32) {
        const T2 av = a[t];
#pragma unroll
        for (int jj = 0; jj < GJ; ++jj) {
            if (jj < nj) {
                const T2 bv = bp[jj][t];
                sx[jj] = fma(av.x, bv.x, fma(av.y, bv.y, sx[jj]));
                sy[jj] = fma(av.x, bv.y, fma(-av.y, bv.x, sy[jj]));
            }
        }
    }
#pragma unroll
    for (int jj = 0; jj < GJ; ++jj) {
        if (jj >= nj) break;
        T x = sx[jj], y = sy[jj];
        for (int off = 16; off > 0; off >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, off);
            y += __shfl_down_sync(0xffffffffu, y, off);
        }
        if (lane == 0) part[((size_t)prob * nsplit + split) * ma * mb + (size_t)i * mb + j0 + jj] = make_double2(x, y);
    }
}

// A^H b for one vector b and up to eight rows on the FP32 copies (the
// Gram-Schmidt products within many chains): every thread of a CTA takes 16
// bytes of b and of every row at a time, and the sums meet once at the end of
// the CTA's chunk.  Bound by the read of the vectors.  (gram_rows_kernel's
// warp per row leaves most warps without one in the first chain steps: 90
// chains of 115 k elements 136 -> 87 us, 144 of 23 k 45 -> 34 us; for few
// problems or more rows its smaller chunks are faster, 26 us against 31 for 90
// rows.)
constexpr int kGram1Rows = 8;
__global__ void __launch_bounds__(256) gram1_kernel(const EigK *ks, int nch, VSet A, VSet B, int nsplit, double2 *part) {
    constexpr int VE = 2, NR = kGram1Rows;                // elements per load (nvec is a multiple of 32)
    struct __align__(16) Pack { float2 v[VE]; };
    const int split = blockIdx.x, prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const int ma = A.count();
    const long long np = d.nvec / VE;
    const long long t0 = split * np / nsplit, t1 = (split + 1) * np / nsplit;
    const Pack *b = reinterpret_cast<const Pack *>(d.v32 + (long long)B.at(0, ch) * d.nvec);
    const Pack *a[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) a[r] = reinterpret_cast<const Pack *>(d.v32 + (long long)A.at(min(r, ma - 1), ch) * d.nvec);
    float sx[NR], sy[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) sx[r] = sy[r] = 0.f;
#pragma unroll 2
    for (long long t = t0 + threadIdx.x; t < t1; t += 256) {
        Pack av[NR];
        const Pack bv = b[t];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (r < ma) av[r] = a[r][t];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (r < ma)
#pragma unroll
                for (int u = 0; u < VE; ++u) {
                    sx[r] = fma(av[r].v[u].x, bv.v[u].x, fma(av[r].v[u].y, bv.v[u].y, sx[r]));
                    sy[r] = fma(av[r].v[u].x, bv.v[u].y, fma(-av[r].v[u].y, bv.v[u].x, sy[r]));
                }
    }
    __shared__ double2 red[8][NR];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        if (r >= ma) break;
        float x = sx[r], y = sy[r];
        for (int off = 16; off > 0; off >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, off);
            y += __shfl_down_sync(0xffffffffu, y, off);
        }
        if (lane == 0) red[warp][r] = make_double2(x, y);
    }
    __syncthreads();
    if (threadIdx.x < ma) {
        double2 s = red[0][threadIdx.x];
        for (int w = 1; w < 8; ++w) s = s + red[w][threadIdx.x];
        part[((size_t)prob * nsplit + split) * ma + threadIdx.x] = s;
    }
}

// A^H B on the FP32 copies for products wider than the tensor-core kernel's
// tile: a CTA takes one chunk of the vector length for a 96 x 96 tile of the
// product, 6 x 6 complex outputs per thread (rows ti + 16 i, columns tj + 16 j:
// 144 FMAs for 12 shared-memory reads), the next KC elements of every vector
// copied to shared memory (cp.async) while the staged ones are used.  Bound by the FMA pipe.
// Partial sums per chunk go to `part` (FP64) and are reduced in a fixed order
// by gram_reduce_kernel; larger products are covered by tiles (blockIdx.z).
// (With 3 x 3 outputs per thread on 48 x 48 tiles and no loads in flight:
// 418 us for 90 x 90 over 115 k elements.)
constexpr int GT_KC = 16, GT_MAX = 96, GT_R = GT_MAX / 16;
__global__ void __launch_bounds__(256, 2) gram_tile32_kernel(const EigK *ks, int nch, VSet A, VSet B, int nsplit,
                                                             double2 *part) {
    extern __shared__ __align__(16) unsigned char gtsm[];
    typedef float2 Stage[GT_KC][GT_MAX + 1];
    Stage *As = reinterpret_cast<Stage *>(gtsm), *Bs = As + 2;     // two buffers each
    const int split = blockIdx.x, prob = blockIdx.y, tid = threadIdx.x;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const int MA = A.count(), MB = B.count();
    const int ncb = (MB + GT_MAX - 1) / GT_MAX;
    const int r0 = (blockIdx.z / ncb) * GT_MAX, c0 = (blockIdx.z % ncb) * GT_MAX;
    const int ma = min(GT_MAX, MA - r0), mb = min(GT_MAX, MB - c0);
    const long long n = d.nvec;
    const long long chunk = (n + nsplit - 1) / nsplit;
    const long long t0 = split * chunk, t1 = min(n, t0 + chunk);
    const int ti = tid / 16, tj = tid % 16;
    // staging: element kk = tid % KC of vectors tid / KC + 16 u
    const int kk = tid % GT_KC, v0 = tid / GT_KC;
    auto fetch = [&](long long tb, int buf) {
        const int in = tb + kk < t1 ? 8 : 0;              // bytes read; the rest is zero
#pragma unroll
        for (int u = 0; u < GT_R; ++u) {
            const int v = v0 + 16 * u;
            const float2 *a = d.v32 + (long long)A.at(r0 + min(v, ma - 1), ch) * n + (in ? tb + kk : 0);
            const float2 *b = d.v32 + (long long)B.at(c0 + min(v, mb - 1), ch) * n + (in ? tb + kk : 0);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(tc::smem_u32(&As[buf][kk][v])), "l"(a),
                         "r"(v < ma ? in : 0)
                         : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(tc::smem_u32(&Bs[buf][kk][v])), "l"(b),
                         "r"(v < mb ? in : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 acc[GT_R][GT_R];
#pragma unroll
    for (int i = 0; i < GT_R; ++i)
#pragma unroll
        for (int j = 0; j < GT_R; ++j) acc[i][j] = make_float2(0.f, 0.f);
    int buf = 0;
    if (t0 < t1) fetch(t0, 0);
    for (long long tb = t0; tb < t1; tb += GT_KC, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                // this buffer is complete, and the other one's readers have passed
        if (tb + GT_KC < t1) fetch(tb + GT_KC, buf ^ 1);
#pragma unroll 2
        for (int q = 0; q < GT_KC; ++q) {
            float2 a[GT_R], b[GT_R];
#pragma unroll
            for (int i = 0; i < GT_R; ++i) a[i] = As[buf][q][ti + 16 * i];
#pragma unroll
            for (int j = 0; j < GT_R; ++j) b[j] = Bs[buf][q][tj + 16 * j];
#pragma unroll
            for (int i = 0; i < GT_R; ++i)
#pragma unroll
                for (int j = 0; j < GT_R; ++j) {
                    acc[i][j].x = fmaf(a[i].x, b[j].x, fmaf(a[i].y, b[j].y, acc[i][j].x));
                    acc[i][j].y = fmaf(a[i].x, b[j].y, fmaf(-a[i].y, b[j].x, acc[i][j].y));
                }
        }
    }
#pragma unroll
    for (int i = 0; i < GT_R; ++i)
#pragma unroll
        for (int j = 0; j < GT_R; ++j) {
            const int r = ti + 16 * i, c = tj + 16 * j;
            if (r < ma && c < mb)
                part[((size_t)prob * nsplit + split) * MA * MB + (size_t)(r0 + r) * MB + c0 + c] =
                    make_double2(acc[i][j].x, acc[i][j].y);
        }
}

// Both Grams of a small pencil, V^H HV and V^H SV (lower triangles, m = M
// <= 8), on the FP32 copies: every thread reads the 3M vectors once per
// element and keeps all M(M+1) partial sums in registers; the CTA reduces
// them (FP64 across warps) into per-chunk partials for gram_reduce_kernel.
template <int M>
__global__ void __launch_bounds__(128) pencil_gram32_kernel(const EigK *ks, int nch, VSet V, VSet HV, VSet SV,
                                                           int nsplit, double2 *partH, double2 *partS) {
    constexpr int NL = M * (M + 1) / 2;
    constexpr int NW = 128 / 32;
    __shared__ float2 red[NW][2 * NL];
    const int split = blockIdx.x, prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const long long n = d.nvec;
    const long long chunk = (n + nsplit - 1) / nsplit;
    const long long t0 = (long long)split * chunk, t1 = min(n, t0 + chunk);
    const float2 *vp[M], *hp[M], *sp[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        vp[i] = d.v32 + (long long)V.at(i, ch) * n;
        hp[i] = d.v32 + (long long)HV.at(i, ch) * n;
        sp[i] = d.v32 + (long long)SV.at(i, ch) * n;
    }
    float2 aH[NL], aS[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) aH[l] = aS[l] = make_float2(0.f, 0.f);
    for (long long t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
        float2 v[M], hv[M], sv[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            v[i] = vp[i][t];
            hv[i] = hp[i][t];
            sv[i] = sp[i][t];
        }
        int l = 0;
#pragma unroll
        for (int i = 0; i < M; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j, ++l) {      // G[i][j] = conj(v_i) x_j
                aH[l].x = fmaf(v[i].x, hv[j].x, fmaf(v[i].y, hv[j].y, aH[l].x));
                aH[l].y = fmaf(v[i].x, hv[j].y, fmaf(-v[i].y, hv[j].x, aH[l].y));
                aS[l].x = fmaf(v[i].x, sv[j].x, fmaf(v[i].y, sv[j].y, aS[l].x));
                aS[l].y = fmaf(v[i].x, sv[j].y, fmaf(-v[i].y, sv[j].x, aS[l].y));
            }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        float hx = aH[l].x, hy = aH[l].y, sx = aS[l].x, sy = aS[l].y;
        for (int off = 16; off > 0; off >>= 1) {
            hx += __shfl_down_sync(0xffffffffu, hx, off);
            hy += __shfl_down_sync(0xffffffffu, hy, off);
            sx += __shfl_down_sync(0xffffffffu, sx, off);
            sy += __shfl_down_sync(0xffffffffu, sy, off);
        }
        if (lane == 0) {
            red[warp][l] = make_float2(hx, hy);
            red[warp][NL + l] = make_float2(sx, sy);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 2 * NL; e += blockDim.x) {
        double x = 0.0, y = 0.0;
        for (int w = 0; w < NW; ++w) {
            x += (double)red[w][e].x;
            y += (double)red[w][e].y;
        }
        const int l = e % NL;
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= l) ++i;
        const int j = l - i * (i + 1) / 2;
        double2 *part = e < NL ? partH : partS;
        part[((size_t)prob * nsplit + split) * M * M + (size_t)i * M + j] = make_double2(x, y);
    }
}

// A^H B on the tensor cores (tcgen05, TF32 inputs, FP32 accumulation in
// tensor memory) for the FP32 copies, to FP32 accuracy by splitting every
// value into x = hi + lo (hi = x rounded to TF32) and summing hi*hi + hi*lo +
// lo*hi.  Complex products become one real product over interleaved (re, im)
// rows: with the MMA's M side holding B_j and B'_j = (im, -re) of B_j, and its
// N side holding A_i,
//   D[j][i]      = sum (ar br + ai bi) = Re (A_i^H B_j)
//   D[mb + j][i] = sum (ar bi - ai br) = Im (A_i^H B_j).
// One CTA (128 threads, TMEM lane = row) takes one chunk of the vector length
// of one problem, in steps of GTC_KC complex elements staged in shared
// memory (canonical K-major layout without swizzle: 8-row x 16-byte core
// matrices, element (r, k) at (r/8)*SBO + (k/4)*LBO + (r%8)*16 + (k%4)*4).
// Requires 2 mb <= 128 and ma <= GTC_NMAX.  Partials go to `part` like the
// CUDA-core Gram kernels' (reduced by gram_reduce_kernel); a wait on the MMA
// barrier that runs out sets *err and skips the rest.
constexpr int GTC_KC = 16;                    // complex elements per step (32 TF32 values per row)
constexpr int GTC_NMAX = 64;
constexpr int GTC_LBO = 128, GTC_SBO = (2 * GTC_KC / 4) * 128;
__host__ __device__ constexpr size_t gtc_smem_bytes(int ntile) {
    return (size_t)2 * 128 * 2 * GTC_KC * 4 + (size_t)2 * ntile * 2 * GTC_KC * 4;
}
__device__ __forceinline__ float tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}
__device__ __forceinline__ uint32_t gtc_off(int r, int k) {
    return (uint32_t)((r >> 3) * GTC_SBO + (k >> 2) * GTC_LBO + (r & 7) * 16 + (k & 3) * 4);
}
__global__ void __launch_bounds__(128) gram_tc32_kernel(const EigK *ks, int nch, VSet A, VSet B, int nsplit, int ntile,
                                                        double2 *part, int *err) {
    extern __shared__ __align__(1024) unsigned char gsm[];
    unsigned char *Mhi = gsm, *Mlo = gsm + 128 * 2 * GTC_KC * 4;
    unsigned char *Nhi = Mlo + 128 * 2 * GTC_KC * 4, *Nlo = Nhi + ntile * 2 * GTC_KC * 4;
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    const int split = blockIdx.x, prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const int ma = A.count(), mb = B.count();
    const long long n = d.nvec;
    const long long chunk = (n + nsplit - 1) / nsplit;
    const long long t0 = (long long)split * chunk, t1 = min(n, t0 + chunk);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int ncols = 32;
    while (ncols < ntile) ncols <<= 1;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&tmem_base)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        tc::mbar_init(&mbar, 1);
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    // rows that no step writes (M side beyond 2 mb, N side beyond ma) stay zero
    for (int e = tid; e < (128 - 2 * mb) * 2 * GTC_KC; e += blockDim.x) {
        const int r = 2 * mb + e / (2 * GTC_KC), kk = e % (2 * GTC_KC);
        *reinterpret_cast<float *>(Mhi + gtc_off(r, kk)) = 0.f;
        *reinterpret_cast<float *>(Mlo + gtc_off(r, kk)) = 0.f;
    }
    for (int e = tid; e < (ntile - ma) * 2 * GTC_KC; e += blockDim.x) {
        const int r = ma + e / (2 * GTC_KC), kk = e % (2 * GTC_KC);
        *reinterpret_cast<float *>(Nhi + gtc_off(r, kk)) = 0.f;
        *reinterpret_cast<float *>(Nlo + gtc_off(r, kk)) = 0.f;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_base;
    // kind::tf32 instruction descriptor: D F32, A and B TF32, both K-major, M = 128, N = ntile
    const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(ntile >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    uint32_t phase = 0;
    bool any = false;
    // staging: element e = tid + 128 u of a side maps to row (e/8/KC)*8 + e%8
    // and element (e/8) % KC (a warp reads 8 rows x 4 consecutive elements);
    // each thread holds its elements of one step in registers, loaded while
    // the previous step's products run
    constexpr int UMAX = GTC_NMAX * GTC_KC / 128;     // 8
    const int nem = ((mb + 7) / 8) * 8 * GTC_KC, nea = ((ma + 7) / 8) * 8 * GTC_KC;
    float2 bv[UMAX], av[UMAX];
    auto fetch = [&](long long tb) {
#pragma unroll
        for (int u = 0; u < UMAX; ++u) {
            const int e = tid + 128 * u;
            const int rl = e & 7, c = (e >> 3) % GTC_KC, r = ((e >> 3) / GTC_KC) * 8 + rl;
            const long long t = tb + c;
            bv[u] = (e < nem && r < mb && t < t1) ? d.v32[(long long)B.at(r, ch) * n + t] : make_float2(0.f, 0.f);
            av[u] = (e < nea && r < ma && t < t1) ? d.v32[(long long)A.at(r, ch) * n + t] : make_float2(0.f, 0.f);
        }
    };
    if (t0 < t1) fetch(t0);
    for (long long tb = t0; tb < t1; tb += GTC_KC) {
#pragma unroll
        for (int u = 0; u < UMAX; ++u) {
            const int e = tid + 128 * u;
            const int rl = e & 7, c = (e >> 3) % GTC_KC, r = ((e >> 3) / GTC_KC) * 8 + rl;
            if (e < nem && r < mb) {
                const float2 v = bv[u];
                const float hx = tf32_rna(v.x), hy = tf32_rna(v.y);
                const float lx = v.x - hx, ly = v.y - hy;
                *reinterpret_cast<float2 *>(Mhi + gtc_off(r, 2 * c)) = make_float2(hx, hy);
                *reinterpret_cast<float2 *>(Mlo + gtc_off(r, 2 * c)) = make_float2(lx, ly);
                *reinterpret_cast<float2 *>(Mhi + gtc_off(mb + r, 2 * c)) = make_float2(hy, -hx);
                *reinterpret_cast<float2 *>(Mlo + gtc_off(mb + r, 2 * c)) = make_float2(ly, -lx);
            }
            if (e < nea && r < ma) {
                const float2 v = av[u];
                const float hx = tf32_rna(v.x), hy = tf32_rna(v.y);
                *reinterpret_cast<float2 *>(Nhi + gtc_off(r, 2 * c)) = make_float2(hx, hy);
                *reinterpret_cast<float2 *>(Nlo + gtc_off(r, 2 * c)) = make_float2(v.x - hx, v.y - hy);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (tid == 0) {
            const uint32_t mh = tc::smem_u32(Mhi), ml = tc::smem_u32(Mlo), nh = tc::smem_u32(Nhi), nl = tc::smem_u32(Nlo);
            for (int kk = 0; kk < 2 * GTC_KC / 8; ++kk) {
                const uint32_t o = kk * 2 * GTC_LBO;
                const uint64_t dmh = tc::smem_desc(mh + o, GTC_LBO, GTC_SBO), dml = tc::smem_desc(ml + o, GTC_LBO, GTC_SBO);
                const uint64_t dnh = tc::smem_desc(nh + o, GTC_LBO, GTC_SBO), dnl = tc::smem_desc(nl + o, GTC_LBO, GTC_SBO);
                const uint64_t da[3] = {dmh, dmh, dml}, db[3] = {dnh, dnl, dnh};
                for (int q = 0; q < 3; ++q) {
                    const uint32_t acc = (any || kk > 0 || q > 0) ? 1u : 0u;
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
                        "l"(da[q]), "l"(db[q]), "r"(idesc), "r"(acc));
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                tc::smem_u32(&mbar)));
        }
        any = true;
        if (tb + GTC_KC < t1) fetch(tb + GTC_KC);        // next step's loads overlap the products
        if (!tc::mbar_wait(&mbar, phase, 1ll << 24)) {
            if (tid == 0) {
                failed = 1;
                atomicExch(err, 1);
            }
        }
        phase ^= 1;
        asm volatile("tcgen05.fence::after_thread_sync;");
        __syncthreads();
        if (failed) break;
    }
    if (!failed) {
        // warp w holds rows (TMEM lanes) 32w .. 32w+31; 8 columns (A vectors) per load
        double *pd = reinterpret_cast<double *>(part + ((size_t)prob * nsplit + split) * ma * mb);
        const int r = 32 * warp + lane;
        for (int c0 = 0; c0 < ntile; c0 += 8) {
            uint32_t v[8];
            if (any) {
                const uint32_t taddr = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                             : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                               "=r"(v[7])
                             : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;");
            } else {
                for (int j = 0; j < 8; ++j) v[j] = 0u;
            }
            for (int j = 0; j < 8; ++j) {
                const int c = c0 + j;
                if (c >= ma) break;
                if (r < mb) pd[2 * ((size_t)c * mb + r)] = (double)__uint_as_float(v[j]);
                else if (r < 2 * mb) pd[2 * ((size_t)c * mb + (r - mb)) + 1] = (double)__uint_as_float(v[j]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

// Float-float arithmetic (a value is hi + lo, two FP32 numbers with
// |lo| <= ulp(hi)/2): Knuth's two-sum and the FMA two-product give the
// rounding error of a sum or product exactly, so sums of products carry
// about 48 significant bits on the FP32 pipe.
struct FF {
    float h, l;
};
__device__ __forceinline__ FF ff_from(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
// (the _rn intrinsics are never contracted into FMAs, which would break the
// exact error terms)
__device__ __forceinline__ void ff_two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// acc += u v (u, v float-float; the lo*lo term is below the result's precision)
__device__ __forceinline__ void ff_mac(FF &acc, FF u, FF v) {
    const float ph = __fmul_rn(u.h, v.h);
    const float pl = fmaf(u.h, v.h, -ph) + fmaf(u.h, v.l, u.l * v.h);
    float s, e;
    ff_two_sum(acc.h, ph, s, e);
    acc.h = s;
    acc.l += e + pl;
}
__device__ __forceinline__ FF ff_neg(FF a) { return {-a.h, -a.l}; }

// The combine kernels' tiles of te elements x tc columns lie on blockIdx.x
// (the only grid axis without a 65535 limit), the column groups of one run of
// elements side by side, so that they share its reads through L2.
static unsigned tile_grid(long long n, int te, int mc, int tc) {
    return (unsigned)((n + te - 1) / te * ((mc + tc - 1) / tc));
}
__device__ __forceinline__ int tile_col(int mc, int tc) { return (int)(blockIdx.x % ((mc + tc - 1) / tc)) * tc; }
__device__ __forceinline__ long long tile_elem(int mc, int tc, int te) {
    return (long long)(blockIdx.x / ((mc + tc - 1) / tc)) * te;
}

// C_j = beta C_j + alpha sum_i A_i Y[i][j] on FP64 vectors with the products
// and sums in float-float arithmetic (the mixed solver's FP64 root rotations:
// FP64-level results at the FP32 rate).  Tiles of 64 elements x 48 columns,
// 4 x 3 outputs per thread (elements tx + 16 i, columns ty + 16 j), so that an
// element of A is read and split into float-float once for 48 columns: the
// split runs at the FP64 rate.  Stages of CF_KC vectors go from registers into
// two buffers, the next one loaded during the products.  Bound by the FP32
// pipe (13 operations a real product): 90 x 90 over 115 k elements 2.04 ms,
// 2.94 ms with 12 columns per pass and a split for each.
constexpr int CF_T = 64, CF_KC = 8, CF_RI = 4, CF_RJ = 3, CF_C = 16 * CF_RJ;
__global__ void __launch_bounds__(256, 2) combine_ff_kernel(const EigK *ks, int nch, VSet A, VSet C,
                                                            const double2 *Y, double alpha, double beta) {
    __shared__ float4 As[2][CF_KC][CF_T], Ys[2][CF_KC][CF_C];        // (re.h, re.l, im.h, im.l)
    const int ma = A.count(), mc = C.count(), prob = blockIdx.y, tid = threadIdx.x;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const int j0 = tile_col(mc, CF_C);
    const long long t0 = tile_elem(mc, CF_C, CF_T);
    if (t0 >= d.nvec) return;                                        // the batch's longest vectors size the grid
    const int nt = (int)min((long long)CF_T, d.nvec - t0);
    const double2 *y = Y + (size_t)prob * LD * LD;
    constexpr int NA = CF_KC * CF_T / 256, NY = (CF_KC * CF_C + 255) / 256;
    double2 ra[NA], ry[NY];
    auto load = [&](int i0) {
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const int q = (tid + u * 256) / CF_T, t = (tid + u * 256) % CF_T;
            ra[u] = i0 + q < ma && t < nt ? d.base[(long long)A.at(i0 + q, ch) * d.nvec + t0 + t] : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < NY; ++u) {
            const int q = (tid + u * 256) / CF_C, j = (tid + u * 256) % CF_C;
            ry[u] = q < CF_KC && i0 + q < ma && j0 + j < mc ? y[(i0 + q) * LD + j0 + j] : make_double2(0.0, 0.0);
        }
    };
    auto split = [](double2 v) {
        const FF re = ff_from(v.x), im = ff_from(v.y);
        return make_float4(re.h, re.l, im.h, im.l);
    };
    auto stage = [&](int buf) {
#pragma unroll
        for (int u = 0; u < NA; ++u) As[buf][(tid + u * 256) / CF_T][(tid + u * 256) % CF_T] = split(ra[u]);
#pragma unroll
        for (int u = 0; u < NY; ++u) {
            const int q = (tid + u * 256) / CF_C;
            if (q < CF_KC) Ys[buf][q][(tid + u * 256) % CF_C] = split(ry[u]);
        }
    };
    const int tx = tid % 16, ty = tid / 16;
    FF ar[CF_RI][CF_RJ], ai[CF_RI][CF_RJ];
#pragma unroll
    for (int i = 0; i < CF_RI; ++i)
#pragma unroll
        for (int j = 0; j < CF_RJ; ++j) ar[i][j] = ai[i][j] = FF{0.f, 0.f};
    int buf = 0;
    load(0);
    for (int i0 = 0; i0 < ma; i0 += CF_KC, buf ^= 1) {
        stage(buf);                     // its readers passed the barrier of the stage between
        __syncthreads();
        if (i0 + CF_KC < ma) load(i0 + CF_KC);
        const int nq = min(CF_KC, ma - i0);
        for (int q = 0; q < nq; ++q) {
            float4 av[CF_RI];
#pragma unroll
            for (int i = 0; i < CF_RI; ++i) av[i] = As[buf][q][tx + 16 * i];
#pragma unroll
            for (int j = 0; j < CF_RJ; ++j) {
                if (j0 + 16 * j + (ty & ~1) >= mc) continue;          // uniform in the warp
                const float4 w = Ys[buf][q][ty + 16 * j];
                const FF yr{w.x, w.y}, yi{w.z, w.w};
#pragma unroll
                for (int i = 0; i < CF_RI; ++i) {
                    const FF xr{av[i].x, av[i].y}, xi{av[i].z, av[i].w};
                    ff_mac(ar[i][j], xr, yr);          // re += xr yr - xi yi
                    ff_mac(ar[i][j], ff_neg(xi), yi);
                    ff_mac(ai[i][j], xr, yi);          // im += xr yi + xi yr
                    ff_mac(ai[i][j], xi, yr);
                }
            }
        }
    }
    // C is read before any of the stores, which could alias the loads
    auto col = [&](int j) { return d.base + (long long)C.at(j0 + ty + 16 * j, ch) * d.nvec + t0 + tx; };
#pragma unroll
    for (int j = 0; j < CF_RJ; ++j) {
        if (j0 + ty + 16 * j >= mc) continue;
        double2 cv[CF_RI];
#pragma unroll
        for (int i = 0; i < CF_RI; ++i)
            cv[i] = beta != 0.0 && tx + 16 * i < nt ? col(j)[16 * i] : make_double2(0.0, 0.0);
#pragma unroll
        for (int i = 0; i < CF_RI; ++i)
            if (tx + 16 * i < nt)
                col(j)[16 * i] = make_double2(beta * cv[i].x + alpha * ((double)ar[i][j].h + (double)ar[i][j].l),
                                              beta * cv[i].y + alpha * ((double)ai[i][j].h + (double)ai[i][j].l));
    }
}

// C_j = beta C_j + alpha sum_i A_i Y[i][j]: TE elements per thread (blockDim.x
// apart) and JC output columns per CTA (blockIdx.x: the column group, so that
// the groups that read one piece of A run together and share it in L2), their
// coefficients staged in shared memory and read two columns at a time, so that
// a pair of 16-byte loads serves 4 TE complex products.  FP64: bound by the
// FP64 pipe, so small problems take narrow groups to reach every SM (15 x 5
// over 1.5 k elements 41.7 -> 8.9 us); FP32 (F32) for at most 8 columns.
constexpr int kCombThreads = 128;
template <int JC, int TE, bool F32>
__global__ void __launch_bounds__(kCombThreads) combine2_kernel(const EigK *ks, int nch, VSet A, VSet C,
                                                                const double2 *Y, double alpha, double beta) {
    typedef typename std::conditional<F32, float2, double2>::type T2;
    typedef typename std::conditional<F32, float, double>::type T;
    __shared__ __align__(16) T2 Ys[JMAX][JC];
    const int ma = A.count(), mc = C.count(), prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const int j0 = tile_col(mc, JC);
    const long long t0 = tile_elem(mc, JC, kCombThreads * TE) + threadIdx.x;
    if (t0 - threadIdx.x >= d.nvec) return;               // the batch's longest vectors size the grid
    const double2 *y = Y + (size_t)prob * LD * LD;
    for (int e = threadIdx.x; e < ma * JC; e += kCombThreads) {
        const int i = e / JC, jj = e % JC;
        const double2 yv = j0 + jj < mc ? y[i * LD + j0 + jj] : make_double2(0.0, 0.0);
        Ys[i][jj] = mk((T)yv.x, (T)yv.y);
    }
    __syncthreads();
    T2 *vb = F32 ? reinterpret_cast<T2 *>(d.v32) : reinterpret_cast<T2 *>(d.base);
    T2 acc[TE][JC];
#pragma unroll
    for (int u = 0; u < TE; ++u)
#pragma unroll
        for (int jj = 0; jj < JC; ++jj) acc[u][jj] = czero<T2>();
    auto step = [&](int i, const T2(&av)[TE]) {
#pragma unroll
        for (int jj = 0; jj < JC; jj += 2) {
            T2 w0, w1;
            if constexpr (F32) {
                const float4 w = *reinterpret_cast<const float4 *>(&Ys[i][jj]);
                w0 = make_float2(w.x, w.y);
                w1 = make_float2(w.z, w.w);
            } else {
                w0 = Ys[i][jj];
                w1 = Ys[i][jj + 1];
            }
#pragma unroll
            for (int u = 0; u < TE; ++u) {
                cfma(acc[u][jj], av[u], w0);
                cfma(acc[u][jj + 1], av[u], w1);
            }
        }
    };
    auto load = [&](int i, T2(&av)[TE]) {
        const T2 *v = vb + (long long)A.at(i, ch) * d.nvec + t0;
#pragma unroll
        for (int u = 0; u < TE; ++u) av[u] = t0 + u * kCombThreads < d.nvec ? v[u * kCombThreads] : czero<T2>();
    };
    constexpr int PF = 6;                                 // vectors in flight
    for (int i = 0; i < ma; i += PF) {
        T2 av[PF][TE];
#pragma unroll
        for (int p = 0; p < PF; ++p)
            if (i + p < ma) load(i + p, av[p]);
#pragma unroll
        for (int p = 0; p < PF; ++p)
            if (i + p < ma) step(i + p, av[p]);
    }
    // C is read before any of the stores, which could alias the loads
    auto col = [&](int jj) { return vb + (long long)C.at(j0 + jj, ch) * d.nvec + t0; };
    T2 cv[TE][JC];
#pragma unroll
    for (int jj = 0; jj < JC; ++jj)
#pragma unroll
        for (int u = 0; u < TE; ++u)
            cv[u][jj] = beta != 0.0 && j0 + jj < mc && t0 + u * kCombThreads < d.nvec ? col(jj)[u * kCombThreads] : czero<T2>();
#pragma unroll
    for (int jj = 0; jj < JC; ++jj)
#pragma unroll
        for (int u = 0; u < TE; ++u)
            if (j0 + jj < mc && t0 + u * kCombThreads < d.nvec)
                col(jj)[u * kCombThreads] = rscale((T)beta, cv[u][jj]) + rscale((T)alpha, acc[u][jj]);
}

// The same for many columns of the FP32 copies, as a matrix product in tiles
// of 128 elements x 48 columns: 8 x 3 complex outputs per thread (elements
// tx + 16 i, columns ty + 16 j), A staged KC vectors at a time by cp.async,
// so that every element of A is read once for all its columns.  Yf: the
// coefficients in FP32 (to_float_kernel; FP64 conversions run at the FP64
// rate and would cost every CTA a quarter of its time).  Bound by the FMA
// pipe: 90 x 90 over 115 k elements 341 -> 173 us, four problems of 36 x 36
// over 23 k 54 -> 39 us against combine2_kernel's 12 columns per CTA.  (96
// columns and one CTA an SM: 188 us.)
constexpr int CT_T = 128, CT_KC = 8, CT_RJ = 3, CT_C = 16 * CT_RJ;
__global__ void __launch_bounds__(256, 2) combine_tile_kernel(const EigK *ks, int nch, VSet A, VSet C, const float2 *Yf,
                                                              float alpha, float beta) {
    constexpr int RJ = CT_RJ;
    __shared__ __align__(16) float2 As[2][CT_KC][CT_T], Ys[2][CT_KC][CT_C];
    const int ma = A.count(), mc = C.count(), prob = blockIdx.y, tid = threadIdx.x;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const int j0 = tile_col(mc, CT_C);
    const long long t0 = tile_elem(mc, CT_C, CT_T);
    if (t0 >= d.nvec) return;                                      // the batch's longest vectors size the grid
    const int nt = (int)min((long long)CT_T, d.nvec - t0);         // a multiple of 32
    const float2 *y = Yf + (size_t)prob * LD * LD;
    // staging: 16 bytes (two elements) of A per copy, one coefficient per copy
    auto fetch = [&](int i0, int buf) {
#pragma unroll
        for (int e = tid; e < CT_KC * CT_T / 2; e += 256) {
            const int q = e / (CT_T / 2), t = e % (CT_T / 2) * 2;
            const bool in = i0 + q < ma && t < nt;
            const float2 *a = d.v32 + (long long)A.at(in ? i0 + q : 0, ch) * d.nvec + (in ? t0 + t : 0);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(&As[buf][q][t])), "l"(a),
                         "r"(in ? 16 : 0)
                         : "memory");
        }
#pragma unroll
        for (int e = tid; e < CT_KC * CT_C; e += 256) {
            const int q = e / CT_C, j = e % CT_C;
            const bool in = i0 + q < ma && j0 + j < mc;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(tc::smem_u32(&Ys[buf][q][j])),
                         "l"(y + (in ? (i0 + q) * LD + j0 + j : 0)), "r"(in ? 8 : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int tx = tid % 16, ty = tid / 16;
    float2 acc[8][RJ];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < RJ; ++j) acc[i][j] = make_float2(0.f, 0.f);
    int buf = 0;
    fetch(0, 0);
    for (int i0 = 0; i0 < ma; i0 += CT_KC, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                // this buffer is complete, and the other one's readers have passed
        if (i0 + CT_KC < ma) fetch(i0 + CT_KC, buf ^ 1);
#pragma unroll 2
        for (int q = 0; q < CT_KC; ++q) {
            float2 av[8], w[RJ];
#pragma unroll
            for (int i = 0; i < 8; ++i) av[i] = As[buf][q][tx + 16 * i];
#pragma unroll
            for (int j = 0; j < RJ; ++j) w[j] = Ys[buf][q][ty + 16 * j];
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < RJ; ++j) cfma(acc[i][j], av[i], w[j]);
        }
    }
    // C is read a column ahead of its stores, which could alias the loads
    auto col = [&](int j) { return d.v32 + (long long)C.at(j0 + ty + 16 * j, ch) * d.nvec + t0 + tx; };
    auto old = [&](int j, float2(&cv)[8]) {
        const bool in = beta != 0.f && j < RJ && j0 + ty + 16 * j < mc;
#pragma unroll
        for (int i = 0; i < 8; ++i) cv[i] = in && tx + 16 * i < nt ? col(j)[16 * i] : make_float2(0.f, 0.f);
    };
    float2 cv[2][8];
    old(0, cv[0]);
#pragma unroll
    for (int j = 0; j < RJ; ++j) {
        old(j + 1, cv[(j + 1) & 1]);
        if (j0 + ty + 16 * j >= mc) continue;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (tx + 16 * i < nt) col(j)[16 * i] = rscale(beta, cv[j & 1][i]) + rscale(alpha, acc[i][j]);
    }
}

// rows i < ma, columns j < mc of every problem's matrix in FP32
__global__ void to_float_kernel(const double2 *Y, float2 *Yf, int ma, int mc) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ma * mc) return;
    const size_t o = (size_t)blockIdx.y * LD * LD + (e / mc) * LD + e % mc;
    Yf[o] = make_float2((float)Y[o].x, (float)Y[o].y);
}

// The same for one output column (a chain's Gram-Schmidt update): 16 bytes
// of every vector per thread, eight vectors in flight.  Bound by the read of
// the vectors.
template <bool F32>
__global__ void __launch_bounds__(kCombThreads) combine1_kernel(const EigK *ks, int nch, VSet A, VSet C,
                                                                const double2 *Y, double alpha, double beta) {
    typedef typename std::conditional<F32, float2, double2>::type T2;
    typedef typename std::conditional<F32, float, double>::type T;
    constexpr int VE = F32 ? 2 : 1;                       // elements per thread (nvec is a multiple of 32)
    __shared__ T2 Ys[JMAX];
    const int prob = blockIdx.y;
    const int k = prob / nch, ch = prob % nch;
    const EigK d = ks[k];
    const long long t = ((long long)blockIdx.x * kCombThreads + threadIdx.x) * VE;
    const int ma = A.count();
    const double2 *y = Y + (size_t)prob * LD * LD;
    for (int i = threadIdx.x; i < ma; i += kCombThreads) Ys[i] = mk((T)(alpha * y[i * LD].x), (T)(alpha * y[i * LD].y));
    __syncthreads();
    if (t >= d.nvec) return;
    T2 *vb = F32 ? reinterpret_cast<T2 *>(d.v32) : reinterpret_cast<T2 *>(d.base);
    struct __align__(16) Pack { T2 v[VE]; };
    Pack *c = reinterpret_cast<Pack *>(vb + (long long)C.at(0, ch) * d.nvec + t);
    Pack acc;
    if (beta == 0.0) {
#pragma unroll
        for (int u = 0; u < VE; ++u) acc.v[u] = czero<T2>();
    } else {
        acc = *c;
#pragma unroll
        for (int u = 0; u < VE; ++u) acc.v[u] = rscale((T)beta, acc.v[u]);
    }
    for (int i0 = 0; i0 < ma; i0 += 8) {
        Pack a[8];
#pragma unroll
        for (int p = 0; p < 8; ++p)
            if (i0 + p < ma) a[p] = *reinterpret_cast<const Pack *>(vb + (long long)A.at(i0 + p, ch) * d.nvec + t);
#pragma unroll
        for (int p = 0; p < 8; ++p)
            if (i0 + p < ma)
#pragma unroll
                for (int u = 0; u < VE; ++u) cfma(acc.v[u], a[p].v[u], Ys[i0 + p]);
    }
    *c = acc;
}

// [X|K]^H H [X|K] (and the S counterpart) when X holds Ritz vectors of the
// last Rayleigh-Ritz (X^H H X = diag(eps), X^H S X = I): rows i >= M come
// from the products KH = K^H H [X|K], KS = K^H S [X|K] (row i - M), the
// upper triangle is their conjugate.  GS may be null (no S matrix).
__global__ void assemble_rr_kernel(const double2 *KH, const double2 *KS, const double *eps, int M, int m,
                                   double2 *GH, double2 *GS) {
    const int k = blockIdx.y;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m * m) return;
    const int i = e / m, j = e % m;
    const size_t o = (size_t)k * LD * LD;
    double2 h, sv;
    if (i < M && j < M) {
        h = make_double2(i == j ? eps[k * M + i] : 0.0, 0.0);
        sv = make_double2(i == j ? 1.0 : 0.0, 0.0);
    } else if (i >= j) {
        h = KH[o + (i - M) * LD + j];
        sv = KS ? KS[o + (i - M) * LD + j] : make_double2(0.0, 0.0);
    } else {
        h = KH[o + (j - M) * LD + i];
        h.y = -h.y;
        sv = KS ? KS[o + (j - M) * LD + i] : make_double2(0.0, 0.0);
        sv.y = -sv.y;
    }
    if (i == j) { h.y = 0.0; sv.y = 0.0; }
    GH[o + i * LD + j] = h;
    if (GS) GS[o + i * LD + j] = sv;
}

// dead slots (mask 0) of an S-Gram matrix become identity rows and columns,
// so that its Cholesky factor exists and leaves them decoupled
__global__ void mask_sgram_kernel(double2 *G, const int *mask, int m) {
    const int prob = blockIdx.y;
    double2 *g = G + (size_t)prob * LD * LD;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m * m) return;
    const int i = e / m, j = e % m;
    const bool di = mask[prob * LD + i] == 0, dj = mask[prob * LD + j] == 0;
    if (di || dj) g[i * LD + j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
}

// C = op(A) B, or alpha op(A) B + delta D where D is given, for small m x m
// matrices, op = conjugate transpose when conjA; a second product op(A) B2 into
// C2 where B2 is given.
// Bound by the FP64 pipe and the latency of the operands: 8 x 8 outputs per
// CTA, so that 90 x 90 reaches every SM, the sum split over the warps of all
// four FP64 pipes, all of A's and B's share in shared memory behind one
// barrier.  (One thread per output on 128-thread CTAs reading both operands
// through L2: 30 us for m = 95, now 12.)
__global__ void __launch_bounds__(256) small_zgemm_kernel(Mat A, Mat B, Mat C, int m, int conjA, Mat D, double alpha,
                                                          double delta, Mat B2, Mat C2) {
    __shared__ double2 As[JMAX][9], Bs[JMAX][8], sum[3][64];
    const int prob = blockIdx.z;
    const double2 *a = A.of(prob);
    const int i0 = blockIdx.y * 8, j0 = blockIdx.x * 8, tid = threadIdx.x, part = tid / 64, t = tid % 64, ti = t / 8, tj = t % 8;
#pragma unroll 4
    for (int e = tid; e < 8 * m; e += 256) {
        const int q = conjA ? e / 8 : e % m, i = conjA ? e % 8 : e / m;      // along the rows of memory
        double2 v = i0 + i < m ? (conjA ? a[q * A.ld + i0 + i] : a[(i0 + i) * A.ld + q]) : make_double2(0.0, 0.0);
        if (conjA) v.y = -v.y;
        As[q][i] = v;
    }
    const int i = i0 + ti, j = j0 + tj;
    const bool in = part == 0 && i < m && j < m;
    for (int pass = 0; pass < (B2.p ? 2 : 1); ++pass) {
        const Mat &Bm = pass ? B2 : B, &Cm = pass ? C2 : C;
        const double2 *b = Bm.of(prob);
#pragma unroll 4
        for (int e = tid; e < 8 * m; e += 256) Bs[e / 8][tj] = j < m ? b[(e / 8) * Bm.ld + j] : make_double2(0.0, 0.0);
        __syncthreads();
        double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
        for (int q = part; q < m; q += 4) cfma(s, As[q][ti], Bs[q][tj]);
        if (part > 0) sum[part - 1][t] = s;
        __syncthreads();
        if (in) {
            s = (s + sum[0][t]) + (sum[1][t] + sum[2][t]);
            if (D.p) s = rscale(alpha, s) + rscale(delta, D.of(prob)[i * D.ld + j]);
            Cm.of(prob)[i * Cm.ld + j] = s;
        }
        __syncthreads();
    }
}

// dead-slot mask of a subspace: columns < ofs are the block's inputs (the
// first bsz live), columns >= ofs are Krylov slots with their alive flags
__global__ void alive_mask_kernel(const int *alive, int kd, int ofs, int M, int b, int nch, int m,
                                  int nprob, int *mask) {
    const int prob = blockIdx.x * blockDim.x + threadIdx.x;
    if (prob >= nprob) return;
    const int ch = prob % nch;
    const int bsz = nch == 1 ? M : min(b, M - ch * b);
    for (int c = 0; c < m; ++c)
        mask[prob * LD + c] = c < ofs ? (c < bsz ? 1 : 0) : alive[prob * kd + (c - ofs)];
}

__global__ void fill_int_kernel(int *p, int n, int v) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

__global__ void set_src_kernel(int *srcH, int *srcS, int nprob, int nch, int kH, int kS, int cs, int slot) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nprob) return;
    srcH[p] = kH + (p % nch) * cs + slot;
    srcS[p] = kS + (p % nch) * cs + slot;
}

// ---------------------------------------------------------------------------
// host driver
#define MB_LAUNCH_E(kid, ...)            \
    do {                                 \
        if (rc) break;                   \
        cudaEvent_t ev_;                 \
        prof_begin(h, s, kid, &ev_);     \
        __VA_ARGS__;                     \
        prof_end(h, s, kid, ev_);        \
        launched();                      \
    } while (0)

namespace {

// real symmetric Jacobi (host, small): z-modes of the initial guess
void host_jacobi_sym(int n, std::vector<double> &A, std::vector<double> &w, std::vector<double> &V) {
    V.assign((size_t)n * n, 0.0);
    for (int i = 0; i < n; ++i) V[(size_t)i * n + i] = 1.0;
    for (int sweep = 0; sweep < 100; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) {
                tot += A[(size_t)i * n + j] * A[(size_t)i * n + j];
                if (i != j) off += A[(size_t)i * n + j] * A[(size_t)i * n + j];
            }
        if (off <= 1e-30 * tot) break;
        for (int p = 0; p < n - 1; ++p)
            for (int q = p + 1; q < n; ++q) {
                double apq = A[(size_t)p * n + q];
                if (apq == 0.0) continue;
                double th = (A[(size_t)q * n + q] - A[(size_t)p * n + p]) / (2 * apq);
                double t = (th >= 0 ? 1.0 : -1.0) / (std::fabs(th) + std::sqrt(th * th + 1));
                double c = 1 / std::sqrt(t * t + 1), s = t * c;
                for (int r = 0; r < n; ++r) {
                    double xp = A[(size_t)r * n + p], xq = A[(size_t)r * n + q];
                    A[(size_t)r * n + p] = c * xp - s * xq;
                    A[(size_t)r * n + q] = s * xp + c * xq;
                }
                for (int r = 0; r < n; ++r) {
                    double xp = A[(size_t)p * n + r], xq = A[(size_t)q * n + r];
                    A[(size_t)p * n + r] = c * xp - s * xq;
                    A[(size_t)q * n + r] = s * xp + c * xq;
                }
                for (int r = 0; r < n; ++r) {
                    double vp = V[(size_t)r * n + p], vq = V[(size_t)r * n + q];
                    V[(size_t)r * n + p] = c * vp - s * vq;
                    V[(size_t)r * n + q] = s * vp + c * vq;
                }
            }
    }
    w.resize(n);
    for (int i = 0; i < n; ++i) w[i] = A[(size_t)i * n + i];
}

// Lowest M free-electron states (|k+G|^2/2 + z-mode n): pure plane wave times
// an S-normalized eigenvector of (D/2) c = e S c.  S-orthonormal by construction.
// The z modes of the free-electron start: eigenvectors c of (D/2) c = w S c,
// S-normalized (c = L^{-T} y with S = L L^T), ascending in w.  They do not
// depend on k, so they are computed once per handle.
static void zmodes(mb_handle *h) {
    if (!h->zmode_w.empty()) return;
    const int nb = h->nb, K = h->order, W = 2 * K - 1;
    std::vector<double> L((size_t)nb * nb, 0.0), D((size_t)nb * nb, 0.0);
    for (int j = 0; j < nb; ++j)
        for (int d = 0; d < K && j - d >= 0; ++d) L[(size_t)j * nb + (j - d)] = h->Lb[(size_t)j * K + d];
    for (int j = 0; j < nb; ++j)
        for (int dd = 0; dd < W; ++dd) {
            int jj = j + dd - (K - 1);
            if (jj >= 0 && jj < nb) D[(size_t)j * nb + jj] = 0.5 * h->Db[(size_t)j * W + dd];
        }
    // Linv by forward substitution
    std::vector<double> Li((size_t)nb * nb, 0.0);
    for (int c = 0; c < nb; ++c)
        for (int i = c; i < nb; ++i) {
            double s = (i == c) ? 1.0 : 0.0;
            for (int q = c; q < i; ++q) s -= L[(size_t)i * nb + q] * Li[(size_t)q * nb + c];
            Li[(size_t)i * nb + c] = s / L[(size_t)i * nb + i];
        }
    std::vector<double> T1((size_t)nb * nb, 0.0), A((size_t)nb * nb, 0.0);
    for (int i = 0; i < nb; ++i)
        for (int j = 0; j < nb; ++j) {
            double s = 0;
            for (int q = 0; q < nb; ++q) s += Li[(size_t)i * nb + q] * D[(size_t)q * nb + j];
            T1[(size_t)i * nb + j] = s;
        }
    for (int i = 0; i < nb; ++i)
        for (int j = 0; j < nb; ++j) {
            double s = 0;
            for (int q = 0; q < nb; ++q) s += T1[(size_t)i * nb + q] * Li[(size_t)j * nb + q];
            A[(size_t)i * nb + j] = s;
        }
    std::vector<double> w, V;
    host_jacobi_sym(nb, A, w, V);
    std::vector<int> ord(nb);
    for (int i = 0; i < nb; ++i) ord[i] = i;
    std::sort(ord.begin(), ord.end(), [&](int a, int b) { return w[a] < w[b]; });
    h->zmode_w.resize(nb);
    h->zmode_c.assign((size_t)nb * nb, 0.0);   // [mode][j]
    for (int n = 0; n < nb; ++n) {
        h->zmode_w[n] = w[ord[n]];
        for (int j = 0; j < nb; ++j) {   // c_z = L^{-T} y
            double s = 0;
            for (int q = j; q < nb; ++q) s += Li[(size_t)q * nb + j] * V[(size_t)q * nb + ord[n]];
            h->zmode_c[(size_t)n * nb + j] = s;
        }
    }
}

// Lowest M free-electron states at k-point ik: plane wave G times z mode n,
// energy |k+G|^2/2 + w_n.
void free_electron_start(mb_handle *h, int ik, int M, std::vector<double2> &X) {
    zmodes(h);
    const int nb = h->nb;
    const KPoint &kp = h->kp[ik];
    std::vector<std::tuple<double, int, int>> cand;
    const int nmode = std::min(nb, M);
    cand.reserve((size_t)kp.ng * nmode);
    for (int g = 0; g < kp.ng; ++g)
        for (int n = 0; n < nmode; ++n) cand.emplace_back(0.5 * kp.q2[g] + h->zmode_w[n], g, n);
    std::partial_sort(cand.begin(), cand.begin() + std::min<size_t>(M, cand.size()), cand.end());
    X.assign((size_t)M * nb * kp.ldg, make_double2(0.0, 0.0));
    for (int c = 0; c < M; ++c) {
        const int g = std::get<1>(cand[c]), n = std::get<2>(cand[c]);
        for (int j = 0; j < nb; ++j) X[((size_t)c * nb + j) * kp.ldg + g] = make_double2(h->zmode_c[(size_t)n * nb + j], 0.0);
    }
}

struct Solver {
    mb_handle *h;
    cudaStream_t s;
    int nk, M, kd, b, nblk, mA, mB, nc;
    int Mconv;          // roots tested for convergence and returned (M includes guards)
    int prec;           // precision of the H applies that build Krylov vectors
    bool fp64_roots = false;   // finish phase: HX of the roots recomputed in FP64 every cycle
    // mixed precision: the Krylov Gram-Schmidt runs on FP32 copies (v32), and
    // the small Rayleigh-Ritz problems of cycles A and B use the S-Gram of
    // their basis (a pencil; FP32 in the bulk cycles, FP64 in the finish
    // phase), so that their result does not depend on how orthogonal the
    // Krylov vectors came out
    bool gs32 = false;
    // bulk cycles (lowp()): X, HX and SX live only in the FP32 copies, and
    // the chains' slot s of chain ch is at o32K + s*nc + ch (likewise SK, HK),
    // so that one slot of every chain is a contiguous block for the applies
    int o32X = 0, o32SX = 0, o32HX = 0, o32W = 0, o32K = 0, o32SK = 0, o32HK = 0, o32T = 0, o32T2 = 0, n32 = 0;
    double2 *d_Sg = nullptr, *d_Ub = nullptr, *d_Tb = nullptr;
    int *d_statb = nullptr;
    int oV, oHV, oSV, oVB, oHVB, oSVB, oQ, oHQ, oW, oSW, oT;
    int nvecs;
    std::vector<EigK> kd_host;
    EigK *d_k = nullptr;
    std::vector<void *> allocs;
    double2 *d_G = nullptr, *d_part = nullptr, *d_Y = nullptr, *d_Ysel = nullptr;
    double2 *d_U = nullptr, *d_G2 = nullptr, *d_T = nullptr;
    double *d_evals = nullptr, *d_eps = nullptr, *d_res = nullptr, *d_dots = nullptr, *d_theta = nullptr;
    int *d_seed = nullptr, *d_srcH = nullptr, *d_srcS = nullptr, *d_alive = nullptr, *d_status = nullptr;
    int *d_mask = nullptr;
    int *d_tcerr = nullptr;   // set by a tensor-core kernel whose bounded wait ran out
    size_t part_cap = 0;
    long long nmax = 0;
    int maxldg = 0;
    int applies = 0;
    int rc = MB_OK;

    ~Solver() {
        for (void *p : allocs) cudaFreeAsync(p, s);   // stream-ordered: no device-wide synchronization
    }
    int cuda(cudaError_t e) {
        if (e != cudaSuccess && rc == MB_OK) rc = cuda_fail(h, e);
        return rc;
    }
    int launched() { return cuda(cudaGetLastError()); }
    template <typename T> T *alloc(size_t n) {
        void *p = nullptr;
        if (rc) return nullptr;
        if (cuda(cudaMallocFromPoolAsync(&p, std::max<size_t>(n, 1) * sizeof(T), mb_pool(h->device), s))) return nullptr;
        allocs.push_back(p);
        return reinterpret_cast<T *>(p);
    }

    // G = A^H B per problem; lower: A^H B is Hermitian (A and B span the same
    // vectors in the same order), only j <= i is computed
    void gram(int nch, VSet A, VSet B, double2 *G, bool f32 = false, bool lower = false) {
        const int mbc = B.count();
        if (f32 && mbc == 1 && A.count() <= kGram1Rows && nk * nch >= 32) {
            // chunks of at least 512 loads, eight CTAs per SM over the grid
            const int ma = A.count(), np = nk * nch;
            int nsplit = std::max(1, std::min(512, (8 * h->num_sms + np - 1) / np));
            nsplit = (int)std::min<long long>(nsplit, std::max<long long>(1, nmax / 1024));
            while ((size_t)np * nsplit * ma > part_cap && nsplit > 1) --nsplit;
            MB_LAUNCH_E(KN_GRAM32, gram1_kernel<<<dim3(nsplit, np), 256, 0, s>>>(d_k, nch, A, B, nsplit, d_part));
            MB_LAUNCH_E(KN_GRAM32,
                        gram_reduce_kernel<<<dim3((ma + 7) / 8, np), 256, 0, s>>>(d_part, nsplit, ma, 1, G, lower ? 1 : 0));
            return;
        }
        // narrowest column group that covers mbc in the fewest slots
        static const int widths[] = {1, 2, 3, 4, 5, 6, 7, 8, 12, 16};
        int gj = 16;
        long long best = 1ll << 40;
        for (int w : widths) {
            const long long slots = (long long)((mbc + w - 1) / w) * w;
            const long long cost = slots * 64 + (mbc + w - 1) / w;   // column slots, then fewer groups
            if (cost < best) { best = cost; gj = w; }
        }
        switch (gj) {
#define MB_GJ(W) case W: gram_t<W>(nch, A, B, G, f32, lower); break;
            MB_GJ(1) MB_GJ(2) MB_GJ(3) MB_GJ(4) MB_GJ(5) MB_GJ(6) MB_GJ(7) MB_GJ(8) MB_GJ(12) MB_GJ(16)
#undef MB_GJ
        }
    }
    template <int GJ> void gram_t(int nch, VSet A, VSet B, double2 *G, bool f32, bool lower) {
        const int nprob = nk * nch;
        const int ma = A.count(), mbc = B.count();
        if (f32 && mbc >= 4 && 2 * mbc <= 128 && ma <= GTC_NMAX && ma * mbc >= 64) {
            // tensor cores: four resident CTAs per SM over the whole grid
            const int ntile = std::max(16, (ma + 15) / 16 * 16);
            int nsplit = std::max(1, std::min(1024, (4 * h->num_sms + nprob - 1) / nprob));
            nsplit = std::min<long long>(nsplit, std::max<long long>(1, nmax / (2 * GTC_KC)));
            while ((size_t)nprob * nsplit * ma * mbc > part_cap && nsplit > 1) --nsplit;
            const size_t smem = gtc_smem_bytes(ntile);
            cuda(smem_limit_once((const void *)gram_tc32_kernel, h->device, h->smem_optin));
            MB_LAUNCH_E(KN_GRAM32, gram_tc32_kernel<<<dim3(nsplit, nprob), 128, smem, s>>>(d_k, nch, A, B, nsplit, ntile,
                                                                                        d_part, d_tcerr));
            MB_LAUNCH_E(KN_GRAM32,
                        gram_reduce_kernel<<<dim3((ma * mbc + 7) / 8, nprob), 256, 0, s>>>(d_part, nsplit, ma, mbc, G,
                                                                                           lower ? 1 : 0));
            return;
        }
        if (f32 && ma * mbc >= 64 && mbc >= 4) {
            // tile kernel: about two resident CTAs per SM over the whole grid
            const int tiles = ((ma + GT_MAX - 1) / GT_MAX) * ((mbc + GT_MAX - 1) / GT_MAX);
            int nsplit = std::max(1, std::min(1024, (2 * h->num_sms + nprob * tiles - 1) / (nprob * tiles)));
            nsplit = std::min<long long>(nsplit, std::max<long long>(1, nmax / (4 * GT_KC)));
            while ((size_t)nprob * nsplit * ma * mbc > part_cap && nsplit > 1) --nsplit;
            const size_t smem = (size_t)4 * GT_KC * (GT_MAX + 1) * sizeof(float2);
            cuda(smem_limit_once((const void *)gram_tile32_kernel, h->device, h->smem_optin));
            MB_LAUNCH_E(KN_GRAM32, gram_tile32_kernel<<<dim3(nsplit, nprob, tiles), 256, smem, s>>>(d_k, nch, A, B, nsplit,
                                                                                                  d_part));
            MB_LAUNCH_E(KN_GRAM32,
                        gram_reduce_kernel<<<dim3((ma * mbc + 7) / 8, nprob), 256, 0, s>>>(d_part, nsplit, ma, mbc, G,
                                                                                           lower ? 1 : 0));
            return;
        }
        const int rowgroups = (ma + 7) / 8, colgroups = (mbc + GJ - 1) / GJ;
        const int per_split = nprob * rowgroups * colgroups;
        int nsplit = std::max(1, std::min(512, (8 * h->num_sms + per_split - 1) / per_split));
        nsplit = std::min<long long>(nsplit, std::max<long long>(1, nmax / 256));   // >= 256 elements per chunk
        while ((size_t)nprob * nsplit * ma * mbc > part_cap && nsplit > 1) --nsplit;
        if (f32)
            MB_LAUNCH_E(KN_GRAM32, (gram_rows_kernel<true, GJ><<<dim3(nsplit, nprob, rowgroups * colgroups), 256, 0, s>>>(
                                       d_k, nch, A, B, nsplit, colgroups, d_part, lower ? 1 : 0)));
        else
            MB_LAUNCH_E(KN_GRAM, (gram_rows_kernel<false, GJ><<<dim3(nsplit, nprob, rowgroups * colgroups), 256, 0, s>>>(
                                     d_k, nch, A, B, nsplit, colgroups, d_part, lower ? 1 : 0)));
        MB_LAUNCH_E(f32 ? KN_GRAM32 : KN_GRAM,
                    gram_reduce_kernel<<<dim3((ma * mbc + 7) / 8, nprob), 256, 0, s>>>(d_part, nsplit, ma, mbc, G,
                                                                                           lower ? 1 : 0));
    }
    void combine(int nch, VSet A, VSet C, const double2 *Y, double alpha, double beta, bool f32 = false) {
        if (f32) {
            combine_t<true>(nch, A, C, Y, alpha, beta);
        } else if (gs32 && C.count() > 8) {
            // mixed solver, FP64 vectors: the root rotations in float-float
            const dim3 grid(tile_grid(nmax, CF_T, C.count(), CF_C), nk * nch);
            MB_LAUNCH_E(KN_COMBINE, combine_ff_kernel<<<grid, 256, 0, s>>>(d_k, nch, A, C, Y, alpha, beta));
        } else {
            combine_t<false>(nch, A, C, Y, alpha, beta);
        }
    }
    template <int JC, int TE, bool F32> void combine_j(int nch, VSet A, VSet C, const double2 *Y, double alpha, double beta) {
        const dim3 grid(tile_grid(nmax, kCombThreads * TE, C.count(), JC), nk * nch);
        MB_LAUNCH_E(F32 ? KN_COMBINE32 : KN_COMBINE,
                    (combine2_kernel<JC, TE, F32><<<grid, kCombThreads, 0, s>>>(d_k, nch, A, C, Y, alpha, beta)));
    }
    template <bool F32> void combine_t(int nch, VSet A, VSet C, const double2 *Y, double alpha, double beta) {
        const int mc = C.count();
        if (mc == 1) {
            const int per = kCombThreads * (F32 ? 2 : 1);
            MB_LAUNCH_E(F32 ? KN_COMBINE32 : KN_COMBINE,
                        (combine1_kernel<F32><<<dim3((unsigned)((nmax + per - 1) / per), nk * nch), kCombThreads, 0, s>>>(
                            d_k, nch, A, C, Y, alpha, beta)));
            return;
        }
        if (F32 && mc > 8) {
            const int np = nk * nch;
            // (in the Gram products' buffer, which is free here: 2 JMAX^2 >= LD^2)
            float2 *Yf = reinterpret_cast<float2 *>(d_part);
            MB_LAUNCH_E(KN_COMBINE32, to_float_kernel<<<dim3((A.count() * mc + 127) / 128, np), 128, 0, s>>>(Y, Yf, A.count(), mc));
            MB_LAUNCH_E(KN_COMBINE32, combine_tile_kernel<<<dim3(tile_grid(nmax, CT_T, mc, CT_C), np), 256, 0, s>>>(
                                          d_k, nch, A, C, Yf, (float)alpha, (float)beta));
            return;
        }
        // the widest column group (least re-reading of A) among those with the
        // least padding, narrow ones where wide ones would leave SMs idle
        const long long ctas = (nmax + kCombThreads - 1) / kCombThreads * nk * nch;
        auto waste = [&](int jc) { return (mc + jc - 1) / jc * jc - mc; };
        if (mc <= 2 || (!F32 && ctas * ((mc + 11) / 12) < 2 * h->num_sms)) {
            combine_j<2, 1, F32>(nch, A, C, Y, alpha, beta);
        } else if (mc <= 4) {
            combine_j<4, 1, F32>(nch, A, C, Y, alpha, beta);
        } else if (mc <= 8) {
            combine_j<8, 1, F32>(nch, A, C, Y, alpha, beta);
        } else if (waste(10) < waste(12)) {
            combine_j<10, 1, false>(nch, A, C, Y, alpha, beta);
        } else {
            combine_j<12, 1, false>(nch, A, C, Y, alpha, beta);
        }
    }
    // U = L^{-H} of np problems (FP32 arithmetic in the bulk cycles)
    void cholinv(int np, int m, const double2 *G, double2 *U, int *status, bool f32) {
        if (f32) {
            cuda(smem_limit_once((const void *)cholinv_kernel<float>, h->device, h->smem_optin));
            MB_LAUNCH_E(KN_SMALL, cholinv_kernel<float><<<np, kCholThreads, cholinv_smem<float>(m), s>>>(G, m, U, status));
        } else {
            cuda(smem_limit_once((const void *)cholinv_kernel<double>, h->device, h->smem_optin));
            MB_LAUNCH_E(KN_SMALL, cholinv_kernel<double><<<np, kCholThreads, cholinv_smem<double>(m), s>>>(G, m, U, status));
        }
    }
    void small_gemm(Mat A, Mat B, Mat C, int m, int conjA, int np = 0, Mat D = Mat(), Mat B2 = Mat(), Mat C2 = Mat(),
                    double alpha = 1.0, double delta = 1.0) {
        const unsigned t = (unsigned)(m + 7) / 8;
        MB_LAUNCH_E(KN_SMALL, small_zgemm_kernel<<<dim3(t, t, np > 0 ? np : nk), 256, 0, s>>>(A, B, C, m, conjA, D, alpha, delta, B2, C2));
    }
    void copy(int nch, VSet S, VSet D, int mode) {
        const unsigned bx = (unsigned)std::min<long long>(64, (nmax + 255) / 256);
        MB_LAUNCH_E(KN_VEC, copy_kernel<<<dim3(bx, S.count(), nk * nch), 256, 0, s>>>(d_k, nch, S, D, mode));
    }
    // S X: the banded S_0 of Eqs. (7)-(8) and, for ultrasoft atoms, the
    // augmentation term sum q |beta><beta| X (§II.B.2)
    void bandS(int src, int dst, int nv, bool f32 = false) {
        if (rc) return;
        std::vector<int> iks(nk);
        std::vector<const void *> xs(nk);
        std::vector<void *> ys(nk);
        for (int k = 0; k < nk; ++k) {
            iks[k] = k;
            if (f32) {
                xs[k] = kd_host[k].v32 + (long long)src * kd_host[k].nvec;
                ys[k] = kd_host[k].v32 + (long long)dst * kd_host[k].nvec;
            } else {
                xs[k] = kd_host[k].base + (long long)src * kd_host[k].nvec;
                ys[k] = kd_host[k].base + (long long)dst * kd_host[k].nvec;
            }
        }
        const int prec = f32 ? MB_FP32 : MB_FP64;
        int r = banded_block_apply(h, false, nk, iks.data(), xs.data(), ys.data(), nv, prec, s);
        if (r == MB_OK && h->uspp) r = uspp_S_add(h, nk, iks.data(), xs.data(), ys.data(), nv, prec, s);
        if (r && rc == MB_OK) rc = r;
    }
    void coldot(int nch, VSet A, VSet B, double *out, bool f32 = false) {
        // chunks of at least 2048 elements, until there are about four CTAs per SM
        const int n = A.count() * nk * nch;
        const int chunks = (int)std::max<long long>(1, std::min<long long>((4 * h->num_sms + n - 1) / n, nmax / 2048));
        double *part = chunks > 1 ? reinterpret_cast<double *>(d_part) : out;
        const dim3 grid(A.count(), nk * nch, chunks);
        if (f32) MB_LAUNCH_E(KN_SMALL, coldot_kernel<true><<<grid, 256, 0, s>>>(d_k, nch, A, B, part));
        else MB_LAUNCH_E(KN_SMALL, coldot_kernel<false><<<grid, 256, 0, s>>>(d_k, nch, A, B, part));
        if (chunks > 1)
            MB_LAUNCH_E(KN_SMALL, coldot_sum_kernel<<<(n + 127) / 128, 128, 0, s>>>(part, chunks, n, out));
    }
    // Y = H X on the FP32 copies (bulk cycles): nv vectors from src32 to dst32
    void apply32(int src32, int dst32, int nv) {
        if (rc) return;
        std::vector<int> iks(nk);
        std::vector<const void *> xs(nk);
        std::vector<void *> ys(nk);
        for (int k = 0; k < nk; ++k) {
            iks[k] = k;
            xs[k] = kd_host[k].v32 + (long long)src32 * kd_host[k].nvec;
            ys[k] = kd_host[k].v32 + (long long)dst32 * kd_host[k].nvec;
        }
        int r = apply_H_batch(h, nk, iks.data(), xs.data(), ys.data(), nv, prec, s);
        if (r && rc == MB_OK) rc = r;
        applies += nv * nk;
    }
    void bandSolve(int per_g, int src, int dst, int nv, bool f32 = false) {
        const void *Lb = f32 ? h->t32.Lrecip : h->t64.Lrecip;
        // four (two) vectors per thread where that leaves at least 96 threads an SM
        const long long cols = (long long)nk * nv * maxldg;
        const int nvt = !f32 ? 1 : cols >= 4ll * 96 * h->num_sms ? 4 : cols >= 2ll * 96 * h->num_sms ? 2 : 1;
        const dim3 grid(((f32 ? 1 : 2) * maxldg + 63) / 64, 1, nk * ((nv + nvt - 1) / nvt));
        switch (h->order) {
#define MB_BLV(KK, F, NVV)                                                                              \
    MB_LAUNCH_E(KN_BANDED, (eig_banded_solve_kernel<KK, F, NVV><<<grid, 64, 0, s>>>(d_k, Lb, per_g, h->nb, src, dst, nv)))
#define MB_BL(KK)                              \
    case KK:                                   \
        if (!f32) MB_BLV(KK, false, 1);        \
        else if (nvt == 4) MB_BLV(KK, true, 4); \
        else if (nvt == 2) MB_BLV(KK, true, 2); \
        else MB_BLV(KK, true, 1);              \
        break;
            MB_BL(3) MB_BL(4) MB_BL(5) MB_BL(6) MB_BL(7) MB_BL(8)
#undef MB_BL
#undef MB_BLV
        }
    }
    int nc_stage() const { return std::max(M, nc); }
    void applyH(int src, int dst, int nv, int p) {
        if (rc) return;
        std::vector<int> iks(nk);
        std::vector<const void *> xs(nk);
        std::vector<void *> ys(nk);
        for (int k = 0; k < nk; ++k) {
            iks[k] = k;
            if (p == MB_FP64) {
                xs[k] = kd_host[k].base + (long long)src * kd_host[k].nvec;
                ys[k] = kd_host[k].base + (long long)dst * kd_host[k].nvec;
            } else {
                xs[k] = kd_host[k].stage;
                ys[k] = kd_host[k].stage + (long long)nc_stage() * kd_host[k].nvec;
            }
        }
        if (p != MB_FP64) copy(1, vs(src, nv), vs(0, nv), 1);
        if (rc) return;
        int r = apply_H_batch(h, nk, iks.data(), xs.data(), ys.data(), nv, p, s);
        if (r && rc == MB_OK) rc = r;
        if (p != MB_FP64) copy(1, vs(nc_stage(), nv), vs(dst, nv), 2);
        applies += nv * nk;
    }
    void residuals_and_seeds(int nch) {
        if (lowp()) {
            MB_LAUNCH_E(KN_VEC, residual32_kernel<<<dim3(256, nk), 256, 0, s>>>(d_k, M, o32HX, o32SX, o32T, d_eps));
            bandSolve(0, o32T, o32T2, M, true);
            coldot(1, vs(o32T, M), vs(o32T2, M), d_dots, true);
        } else {
            MB_LAUNCH_E(KN_VEC, residual_kernel<<<dim3(256, nk), 256, 0, s>>>(d_k, M, oV, oHV, oSV, oT, d_eps));
            bandSolve(0, oT, oT + M, M);
            coldot(1, vs(oT, M), vs(oT + M, M), d_dots);
        }
        int np = nk * nch;
        MB_LAUNCH_E(KN_SMALL, seed_kernel<<<(np + 63) / 64, 64, 0, s>>>(d_dots, M, Mconv, nk, nch, b, d_res, d_eps, d_seed,
                                                                        d_theta, d_srcH, d_srcS, oHV, oSV));
    }
    // H K[slot] of every chain into HK[slot]; reduced-precision applies go
    // straight from the chain slots through the FP32 stage
    void applyH_chain(int nch, int slot, int kV, int kH, int cs) {
        if (prec == MB_FP64) {
            copy(nch, vs(kV + slot, 1, cs), vs(oQ, 1, 1), 0);
            applyH(oQ, oHQ, nch, prec);
            copy(nch, vs(oHQ, 1, 1), vs(kH + slot, 1, cs), 0);
            return;
        }
        if (rc) return;
        std::vector<int> iks(nk);
        std::vector<const void *> xs(nk);
        std::vector<void *> ys(nk);
        for (int k = 0; k < nk; ++k) {
            iks[k] = k;
            xs[k] = kd_host[k].stage;
            ys[k] = kd_host[k].stage + (long long)nc_stage() * kd_host[k].nvec;
        }
        copy(nch, vs(kV + slot, 1, cs), vs(0, 1, 1), 1);
        if (rc) return;
        int r = apply_H_batch(h, nk, iks.data(), xs.data(), ys.data(), nch, prec, s);
        if (r && rc == MB_OK) rc = r;
        copy(nch, vs(nc_stage(), 1, 1), vs(kH + slot, 1, cs), 2);
        applies += nch * nk;
    }
    // classical Gram-Schmidt, twice, in the S inner product, of the chain
    // inputs W (one per chain) on the FP32 copies: all coefficients of a pass
    // come from the same (pre-update) vector.  The roots X are common to
    // every chain of a k-point, so their part is one product with a column
    // per chain.
    void gs32_passes(int nch, int i) {
        for (int pass = 0; pass < 2; ++pass) {
            gram(1, vs(o32SX, M), vs(o32W, nch), d_G2, true);                              // SX^H [W_0 .. W_nch-1]
            if (i > 0) gram(nch, vs(o32SK, i, 1, 0, 0, 0, nc), vs(o32W, 1, 1), d_G, true);  // SK_ch^H W_ch
            combine(1, vs(o32X, M), vs(o32W, nch), d_G2, -1.0, 1.0, true);
            if (i > 0) combine(nch, vs(o32K, i, 1, 0, 0, 0, nc), vs(o32W, 1, 1), d_G, -1.0, 1.0, true);
        }
    }
    void krylov(int nch, int kV, int kS, int kH, int cs) {
        int np = nk * nch;
        MB_LAUNCH_E(KN_SMALL, fill_int_kernel<<<(np * kd + 127) / 128, 128, 0, s>>>(d_alive, np * kd, 1));
        const unsigned rbx = (unsigned)std::min<long long>(1024, (nmax + 255) / 256);
        if (lowp()) {
            // bulk cycles: every step on the FP32 copies; the applies read
            // and write the chain slots in place
            for (int i = 0; i < kd && !rc; ++i) {
                if (i > 0) apply32(o32K + (i - 1) * nc, o32HK + (i - 1) * nc, nch);
                MB_LAUNCH_E(KN_VEC, krylov_residual32_kernel<<<dim3(rbx, np), 256, 0, s>>>(
                                        d_k, nch, i, d_seed, d_theta, o32HX, o32SX, o32HK, o32SK, nc, o32W));
                bandSolve(1, o32W, o32W, nch, true);
                gs32_passes(nch, i);
                bandS(o32W, o32SK + i * nc, nch, true);
                coldot(nch, vs(o32W, 1, 1), vs(o32SK + i * nc, 1, 1), d_dots, true);
                MB_LAUNCH_E(KN_VEC, normalize32_kernel<<<dim3(128, np), 256, 0, s>>>(d_k, nch, o32W, o32K, o32SK, nc, i,
                                                                                     d_dots, d_alive, kd));
            }
            apply32(o32K + (kd - 1) * nc, o32HK + (kd - 1) * nc, nch);
            return;
        }
        if (gs32) {
            copy(1, vs(oV, M), vs(o32X, M), 3);
            copy(1, vs(oSV, M), vs(o32SX, M), 3);
        }
        for (int i = 0; i < kd && !rc; ++i) {
            if (i > 0) {
                applyH_chain(nch, i - 1, kV, kH, cs);
                MB_LAUNCH_E(KN_SMALL, set_src_kernel<<<(np + 63) / 64, 64, 0, s>>>(d_srcH, d_srcS, np, nch, kH, kS, cs, i - 1));
            }
            MB_LAUNCH_E(KN_VEC, krylov_residual_kernel<<<dim3(rbx, np), 256, 0, s>>>(
                                    d_k, nch, d_srcH, d_srcS, d_theta, gs32 ? o32W : oW, gs32 ? 1 : 0));
            if (gs32) {
                bandSolve(1, o32W, o32W, nch, true);
                gs32_passes(nch, i);
                copy(nch, vs(o32W, 1, 1), vs(oW, 1, 1), 4);
            } else {
                bandSolve(1, oW, oW, nch);
                for (int pass = 0; pass < 2; ++pass) {
                    gram(1, vs(oSV, M), vs(oW, nch), d_G2);                    // SX^H [W_0 .. W_nch-1]
                    if (i > 0) gram(nch, vs(kS, i, cs), vs(oW, 1, 1), d_G);     // SK_ch^H W_ch
                    combine(1, vs(oV, M), vs(oW, nch), d_G2, -1.0, 1.0);
                    if (i > 0) combine(nch, vs(kV, i, cs), vs(oW, 1, 1), d_G, -1.0, 1.0);
                }
            }
            bandS(oW, oSW, nch);
            coldot(nch, vs(oW, 1, 1), vs(oSW, 1, 1), d_dots);
            const bool need32 = gs32 && i + 1 < kd;
            MB_LAUNCH_E(KN_VEC, normalize_kernel<<<dim3(128, np), 256, 0, s>>>(d_k, nch, oW, oSW, kV, kS, cs, i,
                                                                               d_dots, d_alive, kd,
                                                                               need32 ? o32K : -1, o32SK, nc));
        }
        applyH_chain(nch, kd - 1, kV, kH, cs);
    }
    // eigenpairs of d_G (overwritten unless f32) into d_evals, d_Y
    void jacobi(int nch, int m, bool masked, int ofs, bool f32 = false) {
        const int np = nk * nch;
        if (masked)
            MB_LAUNCH_E(KN_SMALL, alive_mask_kernel<<<(np + 63) / 64, 64, 0, s>>>(d_alive, kd, ofs, M, b, nch, m, np, d_mask));
        if (f32) {
            jacobi_t<float>(np, m, masked, d_G, d_Y, nullptr, true, 1e-6);
            return;
        }
        // FP32 sweeps, two refinement steps and an orthonormalization, FP64
        // sweeps on what they leave (m = 95: 0.15 to 1.5 ms in all, 6.8 ms with
        // FP64 sweeps throughout, which the FP64 pipe of one SM bounds at 3 ms
        // a sweep).  Four matrices of every problem in the Gram products'
        // buffer, which is free here; it is too small only for more than
        // num_sms / 2 problems of over JMAX / 2 columns (blocks of over 50).
        const size_t one = (size_t)np * m * m;
        if (4 * one > part_cap) {
            jacobi_t<double>(np, m, masked, d_G, d_Y, nullptr, true, 1e-13);
            return;
        }
        const Mat b0(d_part, m), b1(b0.p + one, m), b2(b1.p + one, m), A(b2.p + one, m);
        const dim3 ge((m * m + 127) / 128, np);
        jacobi_t<float>(np, m, masked, d_G, d_Y, A.p, false, 1e-6);
        small_gemm(A, d_Y, b0, m, 0, np);                          // A X0
        small_gemm(d_Y, b0, b1, m, 1, np, Mat(), d_Y, b2);          // S, P
        MB_LAUNCH_E(KN_JACOBI, refine_kernel<<<ge, 128, 0, s>>>(b1, b2, b0, m, 1e-4));
        small_gemm(d_Y, b0, b1, m, 0, np, d_Y);                    // X1 = X0 + X0 E
        small_gemm(A, b1, b0, m, 0, np);
        small_gemm(b1, b0, b2, m, 1, np, Mat(), b1, d_Y);
        MB_LAUNCH_E(KN_JACOBI, refine_kernel<<<ge, 128, 0, s>>>(b2, d_Y, b0, m, 1e-8));
        small_gemm(b1, b0, b2, m, 0, np, b1);                      // X2
        small_gemm(b2, b2, b0, m, 1, np);
        small_gemm(b2, b0, b1, m, 0, np, b2, Mat(), Mat(), -0.5, 1.5);   // X3 = X2 + X2 (I - P) / 2
        small_gemm(A, b1, b0, m, 0, np);
        small_gemm(b1, b0, d_G, m, 1, np);                         // X3^H A X3
        jacobi_t<double>(np, m, masked, d_G, b0, nullptr, true, 1e-13);
        small_gemm(b1, b0, d_Y, m, 0, np);
    }
    // CTAs per problem: as many as give each 6 rows of eigenvectors (fewer
    // would not shorten a round) and fit on the SMs, and enough for the
    // matrix and the rows to fit in shared memory
    template <typename T>
    void jacobi_t(int np, int m, bool masked, const double2 *G, Mat Y, double2 *full, bool sort, double tol) {
        const size_t stat = 32 * sizeof(double) + LD * sizeof(int) + 256;
        int nc = std::max(1, std::min(h->num_sms / np, m / 6));
        while (nc < m && jacobi_smem<T>(m, (m + nc - 1) / nc) + stat > (size_t)h->smem_optin) ++nc;
        // a thread per 2x2 block up to 512: a round of a small problem is a few
        // latencies and two barriers, which more warps only lengthen (m = 10:
        // 50 us with 512 threads, 32 with 128)
        const int npair = (m + 1) / 2, blocks = npair * (npair + 1) / 2;
        const int nt = blocks <= 128 ? 128 : blocks <= 256 ? 256 : kJacobiThreads;
        cuda(smem_limit_once((const void *)jacobi_kernel<T>, h->device, h->smem_optin));
        MB_LAUNCH_E(KN_JACOBI, (jacobi_kernel<T><<<dim3(nc, np), nt, jacobi_smem<T>(m, (m + nc - 1) / nc), s>>>(
                                   G, m, masked ? d_mask : nullptr, LD, 0, d_evals, Y, full, sort ? 1 : 0, 30, tol)));
    }
    // bulk cycles of the mixed solver (before the FP64 finish phase)
    bool lowp() const { return gs32 && !fp64_roots; }
    // Rayleigh-Ritz of the pencil (V^H H V, V^H S V) of nch problems of size m
    // per k-point: U = L^{-H} from V^H S V = L L^H (dead Krylov slots made
    // identity), Ritz pairs of U^H (V^H H V) U; returns the Ritz vectors'
    // coordinates in the V basis (U Y) and leaves the values in d_evals.
    const double2 *rr_pencil(int nch, VSet V, VSet HV, VSet SV, int m, int ofs, bool f32 = false) {
        if (f32 && m >= 2 && m <= 8) {
            pencil_grams32(nch, V, HV, SV, m);
        } else {
            gram(nch, V, HV, d_G, f32, true);
            gram(nch, V, SV, d_Sg, f32, true);
        }
        return pencil_solve(nch, m, ofs);
    }
    // V^H HV into d_G and V^H SV into d_Sg (lower triangles completed), FP32 copies
    void pencil_grams32(int nch, VSet V, VSet HV, VSet SV, int m) {
        const int nprob = nk * nch;
        int nsplit = std::max(1, std::min(32, (4 * h->num_sms + nprob - 1) / nprob));
        while ((size_t)2 * nprob * nsplit * m * m > part_cap && nsplit > 1) --nsplit;
        double2 *pH = d_part, *pS = d_part + (size_t)nprob * nsplit * m * m;
        const dim3 grid(nsplit, nprob);
        switch (m) {
#define MB_PG(MM) case MM: MB_LAUNCH_E(KN_GRAM32, (pencil_gram32_kernel<MM><<<grid, 128, 0, s>>>(d_k, nch, V, HV, SV, nsplit, pH, pS))); break;
            MB_PG(2) MB_PG(3) MB_PG(4) MB_PG(5) MB_PG(6) MB_PG(7) MB_PG(8)
#undef MB_PG
        }
        const dim3 gr((m * m + 7) / 8, nprob);
        MB_LAUNCH_E(KN_GRAM32, gram_reduce_kernel<<<gr, 256, 0, s>>>(pH, nsplit, m, m, d_G, 1));
        MB_LAUNCH_E(KN_GRAM32, gram_reduce_kernel<<<gr, 256, 0, s>>>(pS, nsplit, m, m, d_Sg, 1));
    }
    // the pencil (d_G, d_Sg) of nch problems per k-point
    const double2 *pencil_solve(int nch, int m, int ofs) {
        const int np = nk * nch;
        const dim3 gs((m * m + 127) / 128, np);
        MB_LAUNCH_E(KN_SMALL, alive_mask_kernel<<<(np + 63) / 64, 64, 0, s>>>(d_alive, kd, ofs, M, b, nch, m, np, d_mask));
        MB_LAUNCH_E(KN_SMALL, mask_sgram_kernel<<<gs, 128, 0, s>>>(d_Sg, d_mask, m));
        cholinv(np, m, d_Sg, d_Ub, d_statb, lowp());
        small_gemm(d_G, d_Ub, d_Tb, m, 0, np);    // (V^H H V) U
        small_gemm(d_Ub, d_Tb, d_G, m, 1, np);    // U^H (V^H H V) U
        jacobi(nch, m, true, ofs, lowp());
        small_gemm(d_Ub, d_Y, d_Tb, m, 0, np);    // U Y
        return d_Tb;
    }
    // X, HX <- [V|..](m) Y[:, :M] and SX = S X (S is banded: recomputing it is
    // cheaper than rotating it).  Bulk cycles (lowp): the rotation of the
    // FP32 copies V32 in FP32, and HX from a fresh FP32 apply instead of a
    // rotation (cheaper, and no less accurate than HK from FP32 applies).
    void rotate_set(const double2 *Y, int m, const VSet *V32 = nullptr) {
        if (lowp()) {
            combine(1, *V32, vs(o32T, M), Y, 1.0, 0.0, true);
            copy(1, vs(o32T, M), vs(o32X, M), 5);
            apply32(o32X, o32HX, M);
            bandS(o32X, o32SX, M, true);
            return;
        }
        combine(1, vs(oV, m), vs(oT, M), Y, 1.0, 0.0);
        combine(1, vs(oHV, m), vs(oT + M, M), Y, 1.0, 0.0);
        copy(1, vs(oT, M), vs(oV, M), 0);
        copy(1, vs(oT + M, M), vs(oHV, M), 0);
        bandS(oV, oSV, M);
    }
    // Rayleigh-Ritz on [X | K_A] (withK) or on X.  With K_A, X holds the Ritz
    // vectors of the last Rayleigh-Ritz, so only the Krylov rows of the
    // projected matrices are computed.
    void rr_full(bool withK) {
        int m = withK ? mA : M;
        if (withK && lowp()) {
            // bulk cycles: the Krylov rows from the FP32 copies
            gram(1, vs(o32K, kd, 0, 0, 0, 0, nc), vs(o32HX, M, 0, o32HK, kd, 0, 1, nc), d_G2, true);
            gram(1, vs(o32K, kd, 0, 0, 0, 0, nc), vs(o32SX, M, 0, o32SK, kd, 0, 1, nc), d_T, true);
        } else if (withK) {
            gram(1, vs(oV + M, kd), vs(oHV, m), d_G2);
            if (gs32) gram(1, vs(oV + M, kd), vs(oSV, m), d_T);
        }
        if (withK) {
            MB_LAUNCH_E(KN_SMALL, assemble_rr_kernel<<<dim3((m * m + 127) / 128, nk), 128, 0, s>>>(
                                      d_G2, gs32 ? d_T : nullptr, d_eps, M, m, d_G, gs32 ? d_Sg : nullptr));
            if (gs32) {
                const VSet v32 = vs(o32X, M, 0, o32K, kd, 0, 1, nc);
                rotate_set(pencil_solve(1, m, M), m, &v32);
            } else {
                jacobi(1, m, true, M);
                rotate_set(d_Y, m);
            }
        } else {
            gram(1, vs(oV, m), vs(oHV, m), d_G, false, true);
            jacobi(1, m, false, M);
            rotate_set(d_Y, m);
        }
        MB_LAUNCH_E(KN_SMALL, take_evals_kernel<<<(M * nk + 127) / 128, 128, 0, s>>>(d_evals, M, nk, d_eps));
    }
    // S-orthonormalization and Rayleigh-Ritz in one rotation: U = L^{-H} from
    // X^H S X = L L^H, Ritz pairs of U^H (X^H H X) U, then X <- X U Y.
    void orth_rr() {
        const bool f32 = lowp();
        if (f32) {
            gram(1, vs(o32X, M), vs(o32SX, M), d_G, true, true);
        } else {
            gram(1, vs(oV, M), vs(oSV, M), d_G, false, true);
        }
        cholinv(nk, M, d_G, d_U, d_status, f32);
        if (f32) gram(1, vs(o32X, M), vs(o32HX, M), d_G2, true, true);
        else gram(1, vs(oV, M), vs(oHV, M), d_G2, false, true);
        small_gemm(d_G2, d_U, d_T, M, 0);     // (X^H H X) U
        small_gemm(d_U, d_T, d_G, M, 1);      // U^H (X^H H X) U
        jacobi(1, M, false, M, lowp());
        small_gemm(d_U, d_Y, d_T, M, 0);      // U Y
        const VSet x32 = vs(o32X, M);
        rotate_set(d_T, M, &x32);
        MB_LAUNCH_E(KN_SMALL, take_evals_kernel<<<(M * nk + 127) / 128, 128, 0, s>>>(d_evals, M, nk, d_eps));
    }
    void cycle_B() {
        residuals_and_seeds(nblk);
        if (!lowp()) {
            copy(nblk, vs(oV, b, b), vs(oVB, b, mB), 0);
            copy(nblk, vs(oHV, b, b), vs(oHVB, b, mB), 0);
            if (gs32) copy(nblk, vs(oSV, b, b), vs(oSVB, b, mB), 0);
        }
        krylov(nblk, oVB + b, oSVB + b, oHVB + b, mB);
        const double2 *Yc = d_Y;
        // block ch: [X_b | K_ch] (in the bulk cycles from the FP32 copies)
        const VSet x32 = vs(o32X, b, b, o32K, kd, 1, 1, nc);
        const VSet hx32 = vs(o32HX, b, b, o32HK, kd, 1, 1, nc);
        if (lowp()) {
            Yc = rr_pencil(nblk, x32, hx32, vs(o32SX, b, b, o32SK, kd, 1, 1, nc), mB, b, true);
        } else if (gs32) {
            Yc = rr_pencil(nblk, vs(oVB, mB, mB), vs(oHVB, mB, mB), vs(oSVB, mB, mB), mB, b);
        } else {
            gram(nblk, vs(oVB, mB, mB), vs(oHVB, mB, mB), d_G, false, true);
            jacobi(nblk, mB, true, b);
        }
        int np = nk * nblk;
        MB_LAUNCH_E(KN_SMALL, select_kernel<<<(np + 31) / 32, 32, 0, s>>>(d_evals, Yc, mB, b, M, nblk, np, d_eps, d_Ysel));
        if (lowp()) {
            // the new X and HX of every block land in scratch (nblk*b vectors
            // each) first: the rotation reads the old X
            combine(nblk, x32, vs(o32T, b, b), d_Ysel, 1.0, 0.0, true);
            combine(nblk, hx32, vs(o32T2, b, b), d_Ysel, 1.0, 0.0, true);
            copy(1, vs(o32T, M), vs(o32X, M), 5);
            copy(1, vs(o32T2, M), vs(o32HX, M), 5);
            bandS(o32X, o32SX, M, true);
        } else {
            combine(nblk, vs(oVB, mB, mB), vs(oV, b, b), d_Ysel, 1.0, 0.0);
            combine(nblk, vs(oHVB, mB, mB), vs(oHV, b, b), d_Ysel, 1.0, 0.0);
            bandS(oV, oSV, M);
        }
    }
};

}  // namespace

namespace {
// The solve runs on a private non-blocking stream (capturable, unlike the
// legacy default stream) that first waits for the caller's stream.
// a mixed-precision warm start whose FP64 residuals are all below this (Ha)
// goes straight to the finish phase
constexpr double kWarmFinishResidual = 1e-4;

struct SolveStream {
    cudaStream_t s = nullptr;
    cudaError_t err = cudaSuccess;
    SolveStream(cudaStream_t caller) {
        err = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        if (err != cudaSuccess) return;
        cudaEvent_t ev;
        err = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (err != cudaSuccess) return;
        err = cudaEventRecord(ev, caller);
        if (err == cudaSuccess) err = cudaStreamWaitEvent(s, ev, 0);
        cudaEventDestroy(ev);
    }
    ~SolveStream() {
        if (s) {
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
        }
    }
};
}  // namespace

int eigsolve(mb_handle *h, int nbands, double tol, int prec, double *evals, void *evecs,
             const mb_solve_opts *so, mb_solve_info *info, cudaStream_t caller) {
    auto t0 = std::chrono::steady_clock::now();
    if (!evals || nbands < 1 || !(tol > 0.0)) return MB_EINVAL;
    if (prec != MB_FP64 && prec != MB_FP32 && prec != MB_BF16) return MB_EINVAL;
    if (cudaSetDevice(h->device) != cudaSuccess) return MB_ECUDA;
    SolveStream stream(caller);       // declared before the solver: its workspace is freed on it first
    if (stream.err != cudaSuccess) return cuda_fail(h, stream.err);
    cudaStream_t s = stream.s;
    Solver S;
    S.h = h;
    S.s = s;
    S.nk = (int)h->kp.size();
    int guard = so && so->guard != 0 ? std::max(0, so->guard) : std::max(2, (nbands + 7) / 8);
    S.Mconv = nbands;
    S.M = nbands + guard;
    S.kd = so && so->krylov_depth > 0 ? so->krylov_depth : kDefaultKrylovDepth;
    S.b = so && so->block > 0 ? so->block : kDefaultBlock;
    int max_cycles = so && so->max_cycles > 0 ? so->max_cycles : 200;
    if (S.b > S.M) S.b = S.M;
    S.nblk = (S.M + S.b - 1) / S.b;
    S.mA = S.M + S.kd;
    S.mB = S.b + S.kd;
    S.nc = std::max(1, S.nblk);
    if (S.mA > JMAX || S.mB > JMAX || S.M > LD) return MB_EUNSUPPORTED;
    if (S.nc_stage() > h->max_bands) return MB_EUNSUPPORTED;
    for (auto &k : h->kp)
        if ((long long)k.ng * h->nb < S.mA) return MB_EINVAL;
    if (cudaSetDevice(h->device) != cudaSuccess) return MB_ECUDA;
    int rc = ensure_precond(h);
    if (rc) return rc;
    // vector regions
    // [X | K_A] regions are sized so that the last block of cycle B, when M is
    // not a multiple of b, writes its unused columns into K_A (scratch then)
    const int mAr = std::max(S.mA, S.nblk * S.b);
    S.oV = 0;
    S.oHV = mAr;
    S.oSV = 2 * mAr;
    S.oVB = 3 * mAr;
    S.oHVB = S.oVB + S.nblk * S.mB;
    S.oSVB = S.oHVB + S.nblk * S.mB;
    S.oQ = S.oSVB + S.nblk * S.mB;
    S.oHQ = S.oQ + S.nc;
    S.oW = S.oHQ + S.nc;
    S.oSW = S.oW + S.nc;
    S.oT = S.oSW + S.nc;
    S.nvecs = S.oT + 3 * S.mA;
    // FP32 Gram-Schmidt workspace (mixed precision): X, SX, the chain inputs W,
    // then K and SK of every chain (chain ch, depth i at + ch*kd + i)
    S.gs32 = prec != MB_FP64;
    S.o32X = 0;
    S.o32SX = S.M;
    S.o32HX = 2 * S.M;
    S.o32W = 3 * S.M;
    S.o32K = S.o32W + S.nc;
    S.o32SK = S.o32K + S.nc * S.kd;
    S.o32HK = S.o32SK + S.nc * S.kd;
    S.o32T = S.o32HK + S.nc * S.kd;
    S.o32T2 = S.o32T + std::max(S.M, S.nblk * S.b);
    S.n32 = S.o32T2 + std::max(S.M, S.nblk * S.b);
    // per-k memory
    S.kd_host.resize(S.nk);
    size_t pofs = 0;
    for (int k = 0; k < S.nk; ++k) {
        EigK &e = S.kd_host[k];
        e.ldg = h->kp[k].ldg;
        e.ng = h->kp[k].ng;
        e.nvec = (long long)h->nb * e.ldg;
        e.base = S.alloc<double2>((size_t)S.nvecs * e.nvec);
        e.stage = S.alloc<float2>((size_t)2 * S.nc_stage() * e.nvec);
        e.v32 = S.gs32 ? S.alloc<float2>((size_t)S.n32 * e.nvec) : nullptr;
        e.pfac = (const double *)h->t64.Pfac + pofs;
        e.pfac32 = (const float *)h->t32.Pfac + pofs;
        pofs += (size_t)e.ldg * h->nb * h->order;
        if (S.rc) return S.rc;
        S.cuda(cudaMemsetAsync(e.base, 0, sizeof(double2) * (size_t)S.nvecs * e.nvec, s));
        S.nmax = std::max(S.nmax, e.nvec);
        S.maxldg = std::max(S.maxldg, e.ldg);
    }
    int nprob = S.nk * S.nc;
    S.d_k = S.alloc<EigK>(S.nk);
    S.d_G = S.alloc<double2>((size_t)nprob * LD * LD);
    S.d_Y = S.alloc<double2>((size_t)nprob * LD * LD);
    S.d_Ysel = S.alloc<double2>((size_t)nprob * LD * LD);
    S.d_U = S.alloc<double2>((size_t)S.nk * LD * LD);
    S.d_G2 = S.alloc<double2>((size_t)S.nk * LD * LD);
    S.d_T = S.alloc<double2>((size_t)S.nk * LD * LD);
    // partial products; what else is kept in it is gone before the next ones
    S.part_cap = (size_t)std::max(2 * h->num_sms, nprob) * JMAX * JMAX;
    S.d_part = S.alloc<double2>(S.part_cap);
    S.d_evals = S.alloc<double>((size_t)nprob * LD);
    S.d_eps = S.alloc<double>((size_t)S.nk * S.M);
    S.d_res = S.alloc<double>((size_t)S.nk * S.M);
    S.d_dots = S.alloc<double>((size_t)S.nk * std::max(S.M, S.nc));
    S.d_theta = S.alloc<double>(nprob);
    S.d_seed = S.alloc<int>(nprob);
    S.d_srcH = S.alloc<int>(nprob);
    S.d_srcS = S.alloc<int>(nprob);
    S.d_alive = S.alloc<int>((size_t)nprob * S.kd);
    S.d_mask = S.alloc<int>((size_t)nprob * LD);
    S.d_status = S.alloc<int>(S.nk);
    S.d_tcerr = S.alloc<int>(1);
    if (S.gs32) {
        S.d_Sg = S.alloc<double2>((size_t)nprob * LD * LD);
        S.d_Ub = S.alloc<double2>((size_t)nprob * LD * LD);
        S.d_Tb = S.alloc<double2>((size_t)nprob * LD * LD);
        S.d_statb = S.alloc<int>(nprob);
    }
    if (S.rc) return S.rc;
    S.cuda(cudaMemcpyAsync(S.d_k, S.kd_host.data(), sizeof(EigK) * S.nk, cudaMemcpyHostToDevice, s));
    S.cuda(cudaMemsetAsync(S.d_Ysel, 0, sizeof(double2) * (size_t)nprob * LD * LD, s));
    S.cuda(cudaMemsetAsync(S.d_status, 0, sizeof(int) * S.nk, s));
    S.cuda(cudaMemsetAsync(S.d_tcerr, 0, sizeof(int), s));
    // initial trial vectors: the lowest free-electron states, or (warm
    // start) the caller's vectors in place of the first nbands of them
    const bool warm = so && so->warm_start && evecs;
    size_t woff = 0;
    for (int k = 0; k < S.nk && !S.rc; ++k) {
        std::vector<double2> X0;
        free_electron_start(h, k, S.M, X0);
        S.cuda(cudaMemcpyAsync(S.kd_host[k].base, X0.data(), sizeof(double2) * X0.size(), cudaMemcpyHostToDevice, s));
        const size_t nwarm = (size_t)nbands * h->nb * h->kp[k].ldg;
        if (warm)
            S.cuda(cudaMemcpyAsync(S.kd_host[k].base, reinterpret_cast<const double2 *>(evecs) + woff,
                                   sizeof(double2) * nwarm, cudaMemcpyDeviceToDevice, s));
        woff += nwarm;
        S.cuda(cudaStreamSynchronize(s));
    }
    S.prec = prec;
    // the apply scratch is sized up front for every batch this solve issues,
    // so that nothing allocates while a grand cycle is being captured
    {
        size_t need = 0;
        const int sizes[3] = {1, S.nc, S.nc_stage()};
        for (int pi = 0; pi < 2; ++pi)
            for (int bi = 0; bi < 3; ++bi) {
                need = std::max(need, apply_scratch_bytes(h, S.nk, sizes[bi], pi == 0 ? MB_FP64 : MB_FP32));
                if (h->uspp) need = std::max(need, uspp_scratch_bytes(h, S.nk, sizes[bi], pi == 0 ? MB_FP64 : MB_FP32));
            }
        S.cuda(cudaStreamSynchronize(s));
        if (S.rc == MB_OK) {
            int r2 = ensure_scratch(h, need, s);
            if (r2) return r2;
        }
    }
    bool started = false;
    if (S.lowp() && warm) {
        // a warm start already near convergence skips the FP32 bulk cycles
        // (whose rounding would first undo its accuracy): the start vectors'
        // FP64 residuals decide
        S.fp64_roots = true;
        S.applyH(S.oV, S.oHV, S.M, MB_FP64);
        S.bandS(S.oV, S.oSV, S.M);
        S.orth_rr();
        S.residuals_and_seeds(1);
        std::vector<double> r0((size_t)S.nk * S.M);
        S.cuda(cudaMemcpyAsync(r0.data(), S.d_res, sizeof(double) * r0.size(), cudaMemcpyDeviceToHost, s));
        S.cuda(cudaStreamSynchronize(s));
        double mx = 0.0;
        for (int k = 0; k < S.nk; ++k)
            for (int i = 0; i < S.Mconv; ++i) {
                const double r = r0[(size_t)k * S.M + i];
                mx = std::max(mx, r == r ? r : 1e300);
            }
        if (mx < kWarmFinishResidual) started = true;
        else S.fp64_roots = false;
    }
    if (!started) {
        if (S.lowp()) {
            // mixed precision: the bulk cycles start from FP32 copies of the
            // (S-orthonormal) start vectors
            S.copy(1, vs(S.oV, S.M), vs(S.o32X, S.M), 3);
            S.apply32(S.o32X, S.o32HX, S.M);
            S.bandS(S.o32X, S.o32SX, S.M, true);
            S.orth_rr();
        } else {
            S.applyH(S.oV, S.oHV, S.M, S.prec);
            S.bandS(S.oV, S.oSV, S.M);
            // the caller's vectors next to free-electron guards, or free-electron
            // states that the ultrasoft S does not keep orthonormal: S-orthonormalize
            if (warm || h->uspp) S.orth_rr();
            else S.rr_full(false);
        }
        S.residuals_and_seeds(1);
    }
    std::vector<double> res((size_t)S.nk * S.M);
    double last = 1e300, prev = 1e300, maxres = 1e300, bulk_best = 1e300;
    int bulk_idle = 0;
    int cycles = 0;
    bool converged = false;
    // One grand cycle: A (Krylov space of the worst root + Rayleigh-Ritz on
    // all roots), B (per-block Krylov spaces, Rayleigh-Ritz, maximum-overlap
    // selection), S-orthonormalization + Rayleigh-Ritz, residuals and seeds.
    auto cycle_body = [&]() {
        S.krylov(1, S.oV + S.M, S.oSV + S.M, S.oHV + S.M, 0);
        S.rr_full(true);
        S.cycle_B();
        // Krylov vectors may come from reduced-precision applies: in the
        // finish phase the roots' HX is recomputed in FP64 first, so the
        // Rayleigh-Ritz values and the residual test below are FP64
        if (S.fp64_roots) S.applyH(S.oV, S.oHV, S.M, MB_FP64);
        S.orth_rr();
        S.residuals_and_seeds(1);
    };
    // From the second cycle of each apply precision on, a cycle is one CUDA
    // graph launch (captured once); the host only reads the residuals.
    const bool use_graphs = !h->profiling;
    cudaGraphExec_t gexec[2] = {nullptr, nullptr};
    int applies_per_cycle[2] = {0, 0};
    int cur_gi = -1, plain_left = 0;
    auto conv_max = [&]() {
        double mx = 0.0;
        for (int k = 0; k < S.nk; ++k)
            for (int i = 0; i < S.Mconv; ++i) {
                double r = res[(size_t)k * S.M + i];
                mx = std::max(mx, r == r ? r : 1e300);
            }
        return mx;
    };
    int finish_cycles = 0;
    for (cycles = 1; cycles <= max_cycles && !S.rc; ++cycles) {
        const int gi = (S.prec == MB_FP64 || S.fp64_roots) ? 1 : 0;
        finish_cycles += gi;
        if (gi != cur_gi) {
            cur_gi = gi;
            plain_left = 1;
        }
        if (!use_graphs || plain_left > 0) {
            cycle_body();
            --plain_left;
        } else {
            if (!gexec[gi]) {
                cudaGraph_t graph = nullptr;
                const int before = S.applies;
                S.cuda(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
                cycle_body();
                applies_per_cycle[gi] = S.applies - before;
                S.applies = before;
                cudaError_t e = cudaStreamEndCapture(s, &graph);
                S.cuda(e);
                if (S.rc == MB_OK) S.cuda(cudaGraphInstantiate(&gexec[gi], graph, 0));
                if (graph) cudaGraphDestroy(graph);
            }
            if (S.rc == MB_OK) S.cuda(cudaGraphLaunch(gexec[gi], s));
            S.applies += applies_per_cycle[gi];
        }
        S.cuda(cudaMemcpyAsync(res.data(), S.d_res, sizeof(double) * res.size(), cudaMemcpyDeviceToHost, s));
        int tcerr = 0, tcerr_apply = 0;
        S.cuda(cudaMemcpyAsync(&tcerr, S.d_tcerr, sizeof(int), cudaMemcpyDeviceToHost, s));
        if (h->d_tcerr)        // the projector contractions of MB_BF16 applies
            S.cuda(cudaMemcpyAsync(&tcerr_apply, h->d_tcerr, sizeof(int), cudaMemcpyDeviceToHost, s));
        S.cuda(cudaStreamSynchronize(s));
        if (S.rc) break;
        if (tcerr || tcerr_apply) {   // a tensor-core kernel's bounded wait ran out: its products are not valid
            S.rc = MB_ETIMEOUT;
            break;
        }
        maxres = conv_max();
        if (S.prec != MB_FP64 && !S.fp64_roots) {
            // stalled: two bulk cycles in a row without a 30 % gain on the best
            // residual so far (the FP32 arithmetic of the bulk cycles has a
            // floor, and its residuals need not decrease monotonically there)
            if (maxres < 0.7 * bulk_best) {
                bulk_best = maxres;
                bulk_idle = 0;
            } else {
                ++bulk_idle;
            }
            // a stall counts only near the FP32 floor (~1e-5 of the spectrum's
            // width): far above it the largest residual belongs to roots still
            // converging, which the cheaper bulk cycles handle as well; past
            // half the cycle budget the finish phase starts regardless
            bool stalled = (cycles > 3 && maxres < 1e-3 && (maxres > 0.7 * prev || bulk_idle >= 2)) ||
                           cycles >= max_cycles / 2;
            if (maxres < 30.0 * tol || stalled) {
                // finish phase: the roots get FP64 HX from here on
                S.fp64_roots = true;
                S.copy(1, vs(S.o32X, S.M), vs(S.oV, S.M), 4);
                S.applyH(S.oV, S.oHV, S.M, MB_FP64);
                S.bandS(S.oV, S.oSV, S.M);
                S.orth_rr();
                S.residuals_and_seeds(1);
                S.cuda(cudaMemcpyAsync(res.data(), S.d_res, sizeof(double) * res.size(), cudaMemcpyDeviceToHost, s));
                S.cuda(cudaStreamSynchronize(s));
                maxres = conv_max();
            }
        }
        prev = last;
        last = maxres;
        if ((S.prec == MB_FP64 || S.fp64_roots) && maxres < tol) {
            converged = true;
            break;
        }
    }
    for (auto &g : gexec)
        if (g) cudaGraphExecDestroy(g);
    if (S.rc) return S.rc;
    if (S.lowp()) S.copy(1, vs(S.o32X, S.M), vs(S.oV, S.M), 4);   // stopped in the bulk phase
    std::vector<double> eps((size_t)S.nk * S.M);
    S.cuda(cudaMemcpyAsync(eps.data(), S.d_eps, sizeof(double) * eps.size(), cudaMemcpyDeviceToHost, s));
    if (evecs) {
        char *dst = reinterpret_cast<char *>(evecs);
        for (int k = 0; k < S.nk; ++k) {
            size_t bytes = sizeof(double2) * (size_t)S.Mconv * S.kd_host[k].nvec;
            S.cuda(cudaMemcpyAsync(dst, S.kd_host[k].base, bytes, cudaMemcpyDeviceToDevice, s));
            dst += bytes;
        }
    }
    S.cuda(cudaStreamSynchronize(s));
    if (S.rc) return S.rc;
    for (int k = 0; k < S.nk; ++k)
        std::memcpy(evals + (size_t)k * S.Mconv, eps.data() + (size_t)k * S.M, sizeof(double) * S.Mconv);
    if (info) {
        info->cycles = std::min(cycles, max_cycles);
        info->applies = S.applies;
        info->max_residual = maxres;
        info->finish_cycles = std::min(finish_cycles, max_cycles);
        info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    return converged ? MB_OK : MB_ENOTCONV;
}

}  // namespace mb

// Self-test hook for the tensor-core Gram kernel: G = A^H B (FP64 host
// output, row-major ma x mb interleaved complex) for ma + mb FP32 complex
// vectors of length n stored contiguously on the device (A first), split
// into nsplit chunks.
extern "C" int mb_debug_gram_tc32(const void *V, long long n, int ma, int mb, int nsplit, double *G, void *stream) {
    using namespace mb;
    if (!V || !G || n < 1 || ma < 1 || mb < 1 || 2 * mb > 128 || ma > GTC_NMAX || nsplit < 1 || nsplit > 4096)
        return MB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    EigK hk{};
    hk.v32 = reinterpret_cast<float2 *>(const_cast<void *>(V));
    hk.nvec = n;
    const int ntile = std::max(16, (ma + 15) / 16 * 16);
    EigK *dk = nullptr;
    double2 *part = nullptr, *Gd = nullptr;
    int *err = nullptr;
    cudaError_t e = cudaMalloc(&dk, sizeof(EigK));
    if (e == cudaSuccess) e = cudaMalloc(&part, sizeof(double2) * (size_t)nsplit * ma * mb);
    if (e == cudaSuccess) e = cudaMalloc(&Gd, sizeof(double2) * LD * LD);
    if (e == cudaSuccess) e = cudaMalloc(&err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemcpyAsync(dk, &hk, sizeof(EigK), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), s);
    const size_t smem = gtc_smem_bytes(ntile);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gram_tc32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) {
        gram_tc32_kernel<<<dim3(nsplit, 1), 128, smem, s>>>(dk, 1, vs(0, ma), vs(ma, mb), nsplit, ntile, part, err);
        gram_reduce_kernel<<<dim3((ma * mb + 7) / 8, 1), 256, 0, s>>>(part, nsplit, ma, mb, Gd, 0);
        e = cudaGetLastError();
    }
    std::vector<double2> hG((size_t)LD * LD);
    int herr = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(hG.data(), Gd, sizeof(double2) * LD * LD, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(dk);
    cudaFree(part);
    cudaFree(Gd);
    cudaFree(err);
    if (e != cudaSuccess) return MB_ECUDA;
    for (int i = 0; i < ma; ++i)
        for (int j = 0; j < mb; ++j) {
            G[2 * ((size_t)i * mb + j)] = hG[(size_t)i * LD + j].x;
            G[2 * ((size_t)i * mb + j) + 1] = hG[(size_t)i * LD + j].y;
        }
    return herr ? MB_ETIMEOUT : MB_OK;
}

// Self-test hook for the float-float rotation kernel: C = A Y for ma FP64
// complex device vectors A of length n (stored one after another) and a host
// ma x mc complex matrix Y (interleaved doubles, row i = coefficients of
// A_i); C: mc device vectors of length n, overwritten.
extern "C" int mb_debug_combine_ff(const void *A, const double *Y, long long n, int ma, int mc, void *C,
                                   void *stream) {
    using namespace mb;
    if (!A || !Y || !C || n < 1 || ma < 1 || mc < 1 || ma > JMAX || mc > LD) return MB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    // one work array holding A then C, addressed through index sets
    double2 *base = nullptr, *Yd = nullptr;
    EigK *dk = nullptr;
    cudaError_t e = cudaMalloc(&base, sizeof(double2) * (size_t)(ma + mc) * n);
    if (e == cudaSuccess) e = cudaMalloc(&Yd, sizeof(double2) * LD * LD);
    if (e == cudaSuccess) e = cudaMalloc(&dk, sizeof(EigK));
    std::vector<double2> hY((size_t)LD * LD, make_double2(0.0, 0.0));
    for (int i = 0; i < ma; ++i)
        for (int j = 0; j < mc; ++j)
            hY[(size_t)i * LD + j] = make_double2(Y[2 * ((size_t)i * mc + j)], Y[2 * ((size_t)i * mc + j) + 1]);
    EigK hk{};
    hk.base = base;
    hk.nvec = n;
    if (e == cudaSuccess) e = cudaMemcpyAsync(base, A, sizeof(double2) * (size_t)ma * n, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(Yd, hY.data(), sizeof(double2) * LD * LD, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dk, &hk, sizeof(EigK), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        const dim3 grid(tile_grid(n, CF_T, mc, CF_C), 1);
        combine_ff_kernel<<<grid, 256, 0, s>>>(dk, 1, vs(0, ma), vs(ma, mc), Yd, 1.0, 0.0);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(C, base + (size_t)ma * n, sizeof(double2) * (size_t)mc * n, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(base);
    cudaFree(Yd);
    cudaFree(dk);
    return e == cudaSuccess ? MB_OK : MB_ECUDA;
}

// Self-test hook for the Rayleigh-Ritz problems: eigenpairs of nprob Hermitian
// m x m matrices A (host, row-major interleaved doubles, one after another).
// refined: as the solver treats its FP64 problems; 0: FP64 sweeps alone.
// evals: nprob x m ascending; Y: nprob x m x m, column i the vector of value i.
extern "C" int mb_debug_rayleigh_ritz(mb_handle *h, const double *A, int m, int nprob, int refined, double *evals,
                                      double *Y) {
    using namespace mb;
    if (!h || !A || !evals || !Y || m < 1 || m > JMAX || nprob < 1 || nprob > 4096) return MB_EINVAL;
    if (cudaSetDevice(h->device) != cudaSuccess) return MB_ECUDA;
    SolveStream stream(nullptr);
    if (stream.err != cudaSuccess) return cuda_fail(h, stream.err);
    Solver S;
    S.h = h;
    S.s = stream.s;
    S.nk = nprob;
    const size_t one = (size_t)LD * LD;
    S.part_cap = (size_t)std::max(2 * h->num_sms, nprob) * JMAX * JMAX;
    S.d_G = S.alloc<double2>(nprob * one);
    S.d_Y = S.alloc<double2>(nprob * one);
    S.d_part = S.alloc<double2>(S.part_cap);
    S.d_evals = S.alloc<double>((size_t)nprob * LD);
    std::vector<double2> g(nprob * one, make_double2(0.0, 0.0));
    std::vector<double> ev((size_t)nprob * LD);
    for (int p = 0; p < nprob; ++p)
        for (int i = 0; i < m; ++i)
            for (int j = 0; j < m; ++j) {
                const size_t e = 2 * (((size_t)p * m + i) * m + j);
                g[p * one + (size_t)i * LD + j] = make_double2(A[e], A[e + 1]);
            }
    if (S.rc == MB_OK) S.cuda(cudaMemcpyAsync(S.d_G, g.data(), sizeof(double2) * g.size(), cudaMemcpyHostToDevice, S.s));
    if (S.rc == MB_OK) {
        if (refined) S.jacobi(1, m, false, 0);
        else S.jacobi_t<double>(nprob, m, false, S.d_G, S.d_Y, nullptr, true, 1e-13);
    }
    if (S.rc == MB_OK) S.cuda(cudaMemcpyAsync(g.data(), S.d_Y, sizeof(double2) * g.size(), cudaMemcpyDeviceToHost, S.s));
    if (S.rc == MB_OK) S.cuda(cudaMemcpyAsync(ev.data(), S.d_evals, sizeof(double) * ev.size(), cudaMemcpyDeviceToHost, S.s));
    cudaStreamSynchronize(S.s);
    if (S.rc) return S.rc;
    for (int p = 0; p < nprob; ++p)
        for (int i = 0; i < m; ++i) {
            evals[(size_t)p * m + i] = ev[(size_t)p * LD + i];
            for (int j = 0; j < m; ++j) {
                const size_t e = 2 * (((size_t)p * m + i) * m + j);
                Y[e] = g[p * one + (size_t)i * LD + j].x;
                Y[e + 1] = g[p * one + (size_t)i * LD + j].y;
            }
        }
    return MB_OK;
}
