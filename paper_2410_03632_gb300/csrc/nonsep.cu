// Non-separable spectra (Eqs. cheb_pk and pmd with a general c_n(chi1, chi2)):
// the caller samples P(k_j, chi_a, R_r chi_a) at the N Chebyshev k-nodes of
// every chi-R node q = a n_R + r (scale-dependent growth, massive neutrinos),
// and per node
//   c_n(q)    = (c / N) sum_j P(k_j, q) cos(n (2j+1) pi / 2N),  c = 1 (n = 0), 2
//   w_l(t, q) = sum_n c_n(q) T~^t_{n;l}(q)
// replaces D(chi_a) D(R_r chi_a) sum_n a_n T~; the R sum and the chi sum are
// those of the separable FP64 path.  FP64 on CUDA cores: the coefficient table
// is as large as one ell of the basis per cosmology, so the contraction is a
// batched dot product over n bound by reading the basis.
#include "blast_internal.h"

namespace {

// Per-node Chebyshev coefficients c[n][q], 32 nodes a block.  The transform's
// cosines are even (odd) in j about (N - 1) / 2 for even (odd) n, so the samples
// are folded to sums and differences first and a coefficient takes N / 2
// multiply-adds.  Lanes are nodes (their samples come in as whole rows and lie
// transposed in shared memory), warps and their steps are the orders n.
// Bound by the FP64 pipe: 16,384 nodes of order 64 take 0.09 ms (one thread per
// node, N^2 multiply-adds on strided rows: 0.81 ms).
constexpr int kFitNodes = 32, kFitWarps = 8;

__global__ void __launch_bounds__(32 * kFitWarps)
k_fit_nodes(const double *__restrict__ Pq, int Q, int N, const double *__restrict__ cos_tab, double *__restrict__ c)
{
    extern __shared__ double sm[];
    double *ct = sm;                   // [4N] cos(pi p / 2N)
    double *S = ct + 4 * N;            // [N][33]: rows j < H sums, rows N - 1 - j differences
    const int q0 = blockIdx.x * kFitNodes, cnt = min(kFitNodes, Q - q0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, H = N / 2;
    for (int i = threadIdx.x; i < 4 * N; i += blockDim.x) ct[i] = cos_tab[i];
    for (int i = threadIdx.x; i < cnt * N; i += blockDim.x) {
        const int q = i / N, j = i - q * N;
        S[j * 33 + q] = Pq[(size_t)q0 * N + i];
    }
    __syncthreads();
    for (int j = warp; j < H; j += kFitWarps) {
        const double x = S[j * 33 + lane], y = S[(N - 1 - j) * 33 + lane];
        S[j * 33 + lane] = x + y;
        S[(N - 1 - j) * 33 + lane] = x - y;
    }
    __syncthreads();
    const double mid = (N & 1) ? S[H * 33 + lane] : 0.0;  // cos(n pi / 2): 1, 0, -1, 0
    for (int n = warp; n < N; n += kFitWarps) {
        const double *row = S + ((n & 1) ? (N - 1) * 33 : 0) + lane;
        const int step = (n & 1) ? -33 : 33, mod = 4 * N, inc = 2 * n;
        double a0 = 0.0, a1 = 0.0;
        int idx = n;
        auto cosine = [&]() {
            const double v = ct[idx];
            idx += inc;
            if (idx >= mod) idx -= mod;
            return v;
        };
        for (int j = 0; j + 1 < H; j += 2) {
            a0 = fma(row[j * step], cosine(), a0);
            a1 = fma(row[(j + 1) * step], cosine(), a1);
        }
        if (H & 1) a0 = fma(row[(H - 1) * step], cosine(), a0);
        double a = a0 + a1;
        if (!(n & 1)) a += (n & 2) ? -mid : mid;
        if (lane < cnt) c[(size_t)n * Q + q0 + lane] = (n == 0 ? 1.0 : 2.0) * a / (double)N;
    }
}

// Sum over the 32 lanes of x[0..4]: the width halves with the lanes (8 additions
// a lane instead of 25).  Lanes return one value each; `mine` is its number, -1 none.
__device__ __forceinline__ double lane_sums5(const double (&x)[5], int lane, int &mine)
{
    const unsigned all = 0xffffffffu;
    const bool u16 = lane & 16, u8 = lane & 8;
    const double a = (u16 ? x[3] : x[0]) + __shfl_xor_sync(all, u16 ? x[0] : x[3], 16);
    const double b = (u16 ? x[4] : x[1]) + __shfl_xor_sync(all, u16 ? x[1] : x[4], 16);
    const double e = x[2] + __shfl_xor_sync(all, x[2], 16);
    double f = (u8 ? b : a) + __shfl_xor_sync(all, u8 ? a : b, 8);
    // the third value rides on the upper lanes from here: lanes with bit 2 set
    double g = e + __shfl_xor_sync(all, e, 8);
    const bool u4 = lane & 4;
    double h = (u4 ? g : f) + __shfl_xor_sync(all, u4 ? f : g, 4);
    h += __shfl_xor_sync(all, h, 2);
    h += __shfl_xor_sync(all, h, 1);
    mine = (lane & 3) ? -1 : u4 ? (lane == 4 ? 2 : -1) : (u16 ? 3 : 0) + (u8 ? 1 : 0);
    return h;
}

// w = sum_n c[n][q] T[t][e][n][q] and Y[t][es][a][j] = sum_r V_j(a, r) w, one
// CTA per (chi node a, type t and selected ell) of one request (the layout of
// the separable path's partials).  FP64 multiply-adds bound it (n_cheb + tracers
// per node; reading the basis takes 0.6 of that): 64 ells, 128 x 128 nodes,
// order 64, 5+5 tracers 0.43 ms, with five shuffles a tracer 0.59 ms.
__global__ void __launch_bounds__(128)
k_contract_ns(const ReqDev *__restrict__ rq, const double *__restrict__ c, const double *__restrict__ T, int L,
              int N, int X, int Rn, const int *__restrict__ esel, int n_esel, int MT, double *__restrict__ Y)
{
    constexpr int kG = 5;
    __shared__ double red[4][BLAST_MAX_TRACERS / 2 + kG];
    const int a = blockIdx.x;
    const int t = blockIdx.y / n_esel, es = blockIdx.y % n_esel;
    const int e = esel[es];
    const int ng = rq->n_clust, ns = rq->n_lens;
    const int nB = (t == 0) ? ng : ns, offB = (t == 0) ? 0 : ng;
    const int Q = X * Rn;
    const double *Tb = T + ((size_t)t * L + e) * N * Q + (size_t)a * Rn;
    const double *cb = c + (size_t)a * Rn;
    const double *V = rq->V64 + (size_t)offB * Q + (size_t)a * Rn;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double w[BLAST_MAX_NR / 128];
#pragma unroll
    for (int i = 0; i < BLAST_MAX_NR / 128; i++) {
        w[i] = 0.0;
        const int r = threadIdx.x + 128 * i;
        if (r < Rn) {
            double w0 = 0.0, w1 = 0.0;
#pragma unroll 4
            for (int n = 0; n + 1 < N; n += 2) {
                w0 = fma(cb[(size_t)n * Q + r], Tb[(size_t)n * Q + r], w0);
                w1 = fma(cb[(size_t)(n + 1) * Q + r], Tb[(size_t)(n + 1) * Q + r], w1);
            }
            if (N & 1) w0 = fma(cb[(size_t)(N - 1) * Q + r], Tb[(size_t)(N - 1) * Q + r], w0);
            w[i] = w0 + w1;
        }
    }
    for (int j0 = 0; j0 < nB; j0 += kG) {
        double part[kG];
#pragma unroll
        for (int k = 0; k < kG; k++) part[k] = 0.0;
#pragma unroll
        for (int i = 0; i < BLAST_MAX_NR / 128; i++) {
            const int r = threadIdx.x + 128 * i;
            if (r < Rn)
#pragma unroll
                for (int k = 0; k < kG; k++)
                    if (j0 + k < nB) part[k] = fma(V[(size_t)(j0 + k) * Q + r], w[i], part[k]);
        }
        int mine;
        const double s = lane_sums5(part, lane, mine);
        if (mine >= 0) red[warp][j0 + mine] = s;
    }
    __syncthreads();
    if (threadIdx.x < nB) {
        double s = 0.0;
        for (int v = 0; v < 4; v++) s += red[v][threadIdx.x];
        Y[(((size_t)t * n_esel + es) * X + a) * MT + threadIdx.x] = s;
    }
}

}  // namespace

int launch_fit_nodes(blast_plan *p, const double *Pq, double *c, cudaStream_t s)
{
    const size_t smem = sizeof(double) * (4 * (size_t)p->N + (size_t)p->N * 33);  // 38 KB at order 128
    k_fit_nodes<<<(p->Q + kFitNodes - 1) / kFitNodes, 32 * kFitWarps, smem, s>>>(Pq, p->Q, p->N, p->d_cos_tab, c);
    BL_CUDA(cudaGetLastError());
    return BLAST_OK;
}

int launch_contract_ns(blast_plan *p, const ReqDev *dreq, const double *c, const int *d_esel, int n_esel, double *Y,
                       cudaStream_t s)
{
    dim3 grid(p->X, 3 * n_esel);
    k_contract_ns<<<grid, 128, 0, s>>>(dreq, c, p->T64, p->L, p->N, p->X, p->Rn, d_esel, n_esel, p->max_tr, Y);
    BL_CUDA(cudaGetLastError());
    return BLAST_OK;
}
