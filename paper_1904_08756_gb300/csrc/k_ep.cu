// k_ep.cu -- empirical-potential update (Sec. 2.1 and Eq. 2): the differences Delta S_i(Q)
// between measured and simulated structure factors are resolved into pair terms with the
// (pseudo-)inverse of the Eq. (1) weight matrix, fitted by a series of Poisson-shaped
// functions whose Q-space transform is known in closed form, and the fitted real-space
// series is added to the tabulated empirical potential:
//   U_EP[p][k] += -alpha kT sum_n C[p][n] p_n(r_k),  p_n(r) = (r/(n s))^n exp(n - r/s).
// The Poisson basis is nearly collinear (condition number ~1e10 for 20 functions), so the
// least-squares fit uses Householder QR in FP64, never normal equations.
//
// Two launches. ep_basis_kernel evaluates the basis over the whole GPU (FP64 transcendentals on
// GB300's narrow FP64 unit; what depends on n or Q alone once). ep_fit_kernel is one cluster of
// eight CTAs, each holding an eighth of the Q rows of the basis and of the right-hand sides in shared
// memory: a reflection's norm and its products with all later columns are formed together, a warp
// per column, and meet in one exchange over distributed shared memory, so a step costs one cluster
// barrier instead of three block sums per column. 1000 Q, 20 functions, 3 pairs: 2735 us (one CTA,
// transcendentals included) -> 144 us (17 basis, 127 fit); bound by the cluster barrier and FP64 latency of the 20
// dependent steps.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "epsr_device.cuh"
#include "epsr_internal.h"

namespace epsr {

constexpr int kEpThreads = 512;

__device__ double block_sum_chi(double v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x / 32); ++i) t += red[i];
    return t;
}

// 4 pi rho int_0^inf r^2 p_n(r) sin(Qr)/(Qr) dr in closed form:
// (4 pi rho / Q) e^n (n s)^-n Gamma(n+2) s^(n+2) sin((n+2) atan(Q s)) (1 + Q^2 s^2)^-((n+2)/2)
// as exp(logc(n)) and the factors of log1p(Q^2 s^2) and atan(Q s).
__device__ __forceinline__ double poisson_logc(int n, double s)
{
    const double m = n + 2.0;
    return n - n * log(n * s) + lgamma(m) + m * log(s);
}

__device__ __forceinline__ double poisson_value(int n, double logc, double l1, double th, double Q, double rho)
{
    const double m = n + 2.0;
    return 4.0 * 3.14159265358979323846 * rho / Q * exp(logc - 0.5 * m * l1) * sin(m * th);
}

// Basis values of the two spaces: F[n][i] = F_{n+1}(Q_i) (n_basis rows of nQ), then B[n][k] =
// p_{n+1}((k + 1/2) dr) (rows of n_bins); one block per 32 columns, a warp per row.
constexpr int kBasisThreads = 256;

__global__ void __launch_bounds__(kBasisThreads) ep_basis_kernel(const float *Q, int nQ, int n_basis, double s, double rho,
                                                                 double dr, int n_bins, double *F, double *B, double *change)
{
    __shared__ double s_th[32], s_l1[32], s_logc[kEpMaxBasis];
    const int nqb = (nQ + 31) / 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (change && blockIdx.x == 0 && threadIdx.x == 0) *change = 0.0;
    if ((int)blockIdx.x < nqb) {
        const int i0 = blockIdx.x * 32;
        if (threadIdx.x < 32 && i0 + (int)threadIdx.x < nQ) s_th[threadIdx.x] = atan((double)Q[i0 + threadIdx.x] * s);
        if (threadIdx.x >= 32 && threadIdx.x < 64 && i0 + lane < nQ) {
            const double q = (double)Q[i0 + lane];
            s_l1[lane] = log1p(q * s * q * s);
        }
        if (threadIdx.x >= 64 && threadIdx.x < 64 + n_basis) {
            const int n = threadIdx.x - 64 + 1;
            s_logc[n - 1] = poisson_logc(n, s);
        }
        __syncthreads();
        if (i0 + lane < nQ)
            for (int n = w + 1; n <= n_basis; n += kBasisThreads / 32)
                F[(long long)(n - 1) * nQ + i0 + lane] =
                    poisson_value(n, s_logc[n - 1], s_l1[lane], s_th[lane], (double)Q[i0 + lane], rho);
    } else {
        const int k = (blockIdx.x - nqb) * 32 + lane;
        if (k >= n_bins) return;
        const double r = (k + 0.5) * dr;
        for (int n = w + 1; n <= n_basis; n += kBasisThreads / 32)
            B[(long long)(n - 1) * n_bins + k] = exp(n * log(r / (n * s)) + n - r / s);
    }
}

// Pair-resolving matrix M = (A^T A)^-1 A^T restricted to the data rows, A = [w; gamma I] (P columns),
// by one thread.
__device__ __noinline__ void pair_matrix(const EpArgs &A, double *M)
{
    const int P = A.n_pairs, nd = A.n_data;
    double G[kEpMaxPairs][2 * kEpMaxPairs];
    for (int a = 0; a < P; ++a)
        for (int b = 0; b < P; ++b) {
            double v = a == b ? A.gamma * A.gamma : 0.0;
            for (int d = 0; d < nd; ++d) v += A.w[d * P + a] * A.w[d * P + b];
            G[a][b] = v;
            G[a][P + b] = a == b ? 1.0 : 0.0;
        }
    for (int c = 0; c < P; ++c) {               // Gauss-Jordan with partial pivoting
        int piv = c;
        for (int r = c + 1; r < P; ++r)
            if (fabs(G[r][c]) > fabs(G[piv][c])) piv = r;
        for (int k = 0; k < 2 * P; ++k) { double t = G[c][k]; G[c][k] = G[piv][k]; G[piv][k] = t; }
        const double inv = 1.0 / G[c][c];
        for (int k = 0; k < 2 * P; ++k) G[c][k] *= inv;
        for (int r = 0; r < P; ++r)
            if (r != c) {
                const double f = G[r][c];
                for (int k = 0; k < 2 * P; ++k) G[r][k] -= f * G[c][k];
            }
    }
    for (int p = 0; p < P; ++p)
        for (int d = 0; d < nd; ++d) {
            double v = 0.0;
            for (int b = 0; b < P; ++b) v += G[p][P + b] * A.w[d * P + b];
            M[p * nd + d] = v;
        }
}

constexpr int kEpCtas = 8;                       // one portable cluster

// Doubles of shared memory besides the columns: M, R, Q^T y, C, and per parity the partial products
// of every CTA and the pivot row.
__host__ __device__ inline int ep_fixed_doubles(int nb, int P, int nd)
{
    return P * nd + nb * nb + 2 * P * nb + 2 * (kEpCtas + 1) * (nb + P);
}

__global__ void __cluster_dims__(kEpCtas, 1, 1) __launch_bounds__(kEpThreads, 1) ep_fit_kernel(EpArgs A, int in_smem)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ double sm[];
    __shared__ double s_alpha, s_v0, s_beta;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = (int)cluster.block_rank();
    const int nQ = A.nQ, nb = A.n_basis, P = A.n_pairs, nd = A.n_data, nc = nb + P;
    double *M = sm, *Rm = M + P * nd, *yq = Rm + nb * nb, *Cf = yq + P * nb;
    double *part = Cf + P * nb;                  // [2][kEpCtas][nc]
    double *piv = part + 2 * kEpCtas * nc;       // [2][nc]
    double *cols = piv + 2 * nc;                 // [nc][rows]
    // rows of this CTA, and its columns (F then Y) in shared memory or in place in global memory
    const int per = (nQ + kEpCtas - 1) / kEpCtas, r0 = min(nQ, rank * per), rows = min(nQ, r0 + per) - r0;
    auto column = [&](int k) {
        return in_smem ? cols + (long long)k * per : (k < nb ? A.F + (long long)k * nQ : A.Y + (long long)(k - nb) * nQ) + r0;
    };
    if (tid == 0) pair_matrix(A, M);
    if (in_smem)
        for (int e = tid; e < nb * rows; e += kEpThreads) {
            const int k = e / rows, i = e - k * rows;
            cols[(long long)k * per + i] = A.F[(long long)k * nQ + r0 + i];
        }
    __syncthreads();
    // pair-resolved differences
    for (int e = tid; e < P * rows; e += kEpThreads) {
        const int p = e / rows, i = e - p * rows;
        double v = 0.0;
        for (int d = 0; d < nd; ++d) v += M[p * nd + d] * (double)A.dS[(long long)d * nQ + r0 + i];
        column(nb + p)[i] = v;
    }
    __syncthreads();
    cluster.sync();                              // every CTA of the cluster runs: its shared memory may be written
    // Householder QR of F, the reflections applied to the P right-hand sides: f_j . c_k over the rows
    // i >= j of every column k >= j (k = j: the norm), one warp per column
    for (int j = 0; j < nb; ++j) {
        const int par = j & 1, i0 = max(0, j - r0);
        const double *fj = column(j);
        for (int k = j + warp; k < nc; k += kEpThreads / 32) {
            const double *c = column(k);
            double dot = 0.0;
            for (int i = i0 + lane; i < rows; i += 32) dot += fj[i] * c[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
            if (lane < kEpCtas) {
                cluster.map_shared_rank(part, lane)[(par * kEpCtas + rank) * nc + k] = dot;
                if (j >= r0 && j < r0 + rows) cluster.map_shared_rank(piv, lane)[par * nc + k] = c[j - r0];
            }
        }
        cluster.sync();
        // FP64 runs two lanes a cycle here, so the step's scalars are formed by one warp, and a column's
        // eight partial products by eight lanes (a fixed tree)
        const double *pt = part + par * kEpCtas * nc, *pr = piv + par * nc;
        auto total = [&](int k) {
            double t = lane < kEpCtas ? pt[lane * nc + k] : 0.0;
#pragma unroll
            for (int o = kEpCtas / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            return __shfl_sync(0xffffffffu, t, 0);
        };
        if (warp == 0) {
            const double nn = total(j);
            if (lane == 0) {
                const double norm = sqrt(nn), x0 = pr[j];
                const double alpha = x0 > 0 ? -norm : norm;
                const double v0 = x0 - alpha;
                const double vtv = norm * norm - x0 * x0 + v0 * v0;
                s_alpha = alpha;
                s_v0 = v0;
                s_beta = vtv > 0 ? 2.0 / vtv : 0.0;
                Rm[j * nb + j] = alpha;
            }
        }
        __syncthreads();
        const double alpha = s_alpha, v0 = s_v0, beta = s_beta;
        for (int k = j + 1 + warp; k < nc; k += kEpThreads / 32) {
            const double f = beta * (total(k) - alpha * pr[k]);        // v = f_j - alpha e_j
            double *c = column(k);
            for (int i = i0 + lane; i < rows; i += 32) c[i] -= f * (r0 + i == j ? v0 : fj[i]);
            if (lane == 0) {
                const double t = pr[k] - f * v0;
                if (k < nb) Rm[j * nb + k] = t;
                else yq[(k - nb) * nb + j] = t;
            }
        }
        __syncthreads();
    }
    // back substitution R C_p = (Q^T y_p)[0:nb], in every CTA
    if (tid < P) {
        for (int j = nb - 1; j >= 0; --j) {
            double v = yq[tid * nb + j];
            for (int k = j + 1; k < nb; ++k) v -= Rm[j * nb + k] * Cf[tid * nb + k];
            Cf[tid * nb + j] = v / Rm[j * nb + j];
        }
    }
    __syncthreads();
    if (rank == 0)
        for (int e = tid; e < P * nb; e += kEpThreads) A.C_out[e] = Cf[e];
    // table: U_EP[p][k] += -alpha kT sum_n C[p][n] p_n(r_k), and the largest change
    double most = 0.0;
    for (int e = rank * kEpThreads + tid; e < P * A.n_bins; e += kEpCtas * kEpThreads) {
        const int p = e / A.n_bins, k = e % A.n_bins;
        double v = 0.0;
        for (int n = 0; n < nb; ++n) v += Cf[p * nb + n] * A.B[(long long)n * A.n_bins + k];
        A.ep[e] = (float)((double)A.ep[e] - A.alpha * A.kT * v);
        most = fmax(most, fabs(A.alpha * A.kT * v));
    }
    if (most > 0.0) atomicMax(reinterpret_cast<unsigned long long *>(A.change), (unsigned long long)__double_as_longlong(most));
    cluster.sync();                              // no CTA leaves while another may still write to it
}

// ---- chi^2 of the differentiable form: chi2 = sum_Q [S(Q) + sum_p W_p sum_n C_pn F_n(Q) - T(Q)]^2
// One CTA forms the residuals and the sums in a fixed FP64 order (deterministic): dS = 2 res,
// dC_pn = 2 W_p sum_Q res F_n(Q), a warp per function (the sum is shared by the pairs).
constexpr int kChiThreads = 1024;
constexpr int kChiMaxQ = 8192;

__global__ void __launch_bounds__(kChiThreads, 1)
chi2_kernel(const float *S, const float *T, int nQ, ChiParams prm, const double *C, const double *F,
            double *chi2, float *dS, double *dC)
{
    __shared__ double red[kChiThreads / 32];
    __shared__ double wc[kEpMaxBasis];           // sum_p W_p C_pn
    if (C)
        for (int n = threadIdx.x; n < prm.n_basis; n += kChiThreads) {
            double v = 0.0;
            for (int p = 0; p < prm.P; ++p) v += prm.W[p] * C[p * prm.n_basis + n];
            wc[n] = v;
        }
    __syncthreads();
    double part = 0.0;
    for (int i = threadIdx.x; i < nQ; i += kChiThreads) {
        double img = 0.0;
        if (C)
            for (int n = 0; n < prm.n_basis; ++n) img += wc[n] * F[(long long)n * nQ + i];
        const double res = (double)S[i] + img - (double)T[i];
        dS[i] = (float)(2.0 * res);
        prm.res_scratch[i] = res;
        part += res * res;
    }
    const double tot = block_sum_chi(part, red);
    if (threadIdx.x == 0) *chi2 = tot;
    __syncthreads();
    if (dC) {
        const int lane = threadIdx.x & 31;
        for (int n = threadIdx.x >> 5; n < prm.n_basis; n += kChiThreads / 32) {
            double v = 0.0;
            for (int i = lane; i < nQ; i += 32) v += prm.res_scratch[i] * F[(long long)n * nQ + i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            for (int p = lane; p < prm.P; p += 32) dC[p * prm.n_basis + n] = 2.0 * prm.W[p] * v;
        }
    }
}

int launch_ep_update(const EpArgs &a, cudaStream_t stream)
{
    ep_basis_kernel<<<(a.nQ + 31) / 32 + (a.n_bins + 31) / 32, kBasisThreads, 0, stream>>>(
        a.Q, a.nQ, a.n_basis, a.s, a.rho, a.dr, a.n_bins, a.F, a.B, a.change);
    note_launch();
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(ep_fit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kClMaxSmem);
        if (e != cudaSuccess) return set_cuda_error(e, "cudaFuncSetAttribute(ep fit)");
        attr = true;
    }
    const size_t fixed = (size_t)ep_fixed_doubles(a.n_basis, a.n_pairs, a.n_data) * sizeof(double);
    const size_t cols = (size_t)((a.nQ + kEpCtas - 1) / kEpCtas) * (a.n_basis + a.n_pairs) * sizeof(double);
    const bool in_smem = fixed + cols <= (size_t)kClMaxSmem;         // else the columns stay in global memory
    ep_fit_kernel<<<kEpCtas, kEpThreads, in_smem ? fixed + cols : fixed, stream>>>(a, in_smem ? 1 : 0);
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EPSR_OK : set_cuda_error(e, "ep_update");
}

int launch_chi2(const float *S, const float *target, const float *Q, int nQ, const ChiParams &prm,
                const double *C, double *chi2, float *dS, double *dC, cudaStream_t stream)
{
    if (nQ > kChiMaxQ) return set_error(EPSR_EINVAL, "chi2: nQ above %d", kChiMaxQ);
    if (C) {
        ep_basis_kernel<<<(nQ + 31) / 32, kBasisThreads, 0, stream>>>(Q, nQ, prm.n_basis, prm.s, prm.rho, 0.0, 0,
                                                                     prm.F_scratch, nullptr, nullptr);
        note_launch();
    }
    chi2_kernel<<<1, kChiThreads, 0, stream>>>(S, target, nQ, prm, C, prm.F_scratch, chi2, dS, dC);
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EPSR_OK : set_cuda_error(e, "chi2");
}

}  // namespace epsr
