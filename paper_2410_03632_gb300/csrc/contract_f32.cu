// FP32 contraction (a) with the R sum of quadrature (b), on CUDA cores:
//
//   w_b(q) = sum_n a_b[n] T~[t][l][n][q],  Y_b(t, l, a, j) = sum_r V_bj(a, r) w_b(a n_R + r).
//
// A block of two warps owns one chi node, eight (type, ell) pairs in turn and
// BB cosmologies.  A thread keeps w of NQ R nodes for all of them, so a basis
// value is loaded once per BB multiply-adds and a coefficient (a broadcast from
// shared memory) once per NQ, and the sums over lanes are halved in width at
// every step: BB values cost BB shuffles, not 5 BB.  Two cosmologies share a
// packed multiply-add.  Blocks run over the cosmology groups first (they share
// the basis tile in L2), then over (type, ell) (they share the weights), then
// over chi nodes.
//
// Order of the sums: n ascending, then the R nodes of a lane (r = lane + 32 v +
// 128 k, v = 0..3) in ascending k, the lanes of each v in the tree 16, 8, 4, 2,
// 1, and v = 0..3 in turn.  It depends on nothing but n_R, so a cosmology's
// bits are the same in every batch and for every BB and NQ.
//
// Bound by issue and L2 latency (128 registers leave 16 warps an SM).  48
// cosmologies (64 ells, 128 x 128 nodes, order 64, 5+5 tracers) take 1.07 ms;
// one block per cosmology and node, which re-read the basis from L2 for each
// and shuffled five times per tracer, took 19 ms; without the packed pairs and
// the shared coefficients it was 1.22 ms.
#include <climits>

#include "blast_internal.h"

namespace {

constexpr int kThreads = 64;
constexpr int kSpan = 8;   // (type, ell) pairs of a block, which share its coefficients

// Sum over the 32 lanes of each of the BB values x[0..BB): the width halves
// while more than one value is left.  Returns the sum of value `mine`.
template <int BB>
__device__ __forceinline__ float lane_sums(float (&x)[BB], int lane, int &mine)
{
    mine = 0;
    int o = 16;
#pragma unroll
    for (int wdt = BB / 2; wdt >= 1; wdt /= 2, o /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < BB / 2; k++) {
            if (k >= wdt) break;
            const float keep = up ? x[k + wdt] : x[k], send = up ? x[k] : x[k + wdt];
            x[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        if (up) mine += wdt;
    }
    for (; o >= 1; o /= 2) x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
    return x[0];
}

// Two cosmologies in one 64-bit register pair: one instruction multiplies and
// adds for both, each rounded as alone.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pair(float x, float y)
{
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Off: type of an offset in floats from the weights of the block's first
// cosmology.  The work spaces of a group span 45 (max_clust + max_lens) (n_chi + Q)
// floats at BB = 16, past 2^31 from 1.5 million nodes of 16+16 tracers; 64-bit
// offsets everywhere cost 2 % (48 cosmologies 1.28 ms a call instead of 1.26).
template <int BB, int NQ, class Off>
__global__ void __launch_bounds__(kThreads)
k_contract_f32(const ReqDev *__restrict__ reqs, int n, const float *__restrict__ basis, int L, int N, int X, int Rn,
               const int *__restrict__ esel, int n_esel, int MT, int sym, int ngr, float *__restrict__ Y)
{
    extern __shared__ float4 sm4[];
    float *as = reinterpret_cast<float *>(sm4);  // [N][BB]
    float *red = as + (size_t)N * BB;            // [parity][tracer][v][BB]
    constexpr int PB = BB / 2;                   // pairs of cosmologies
    struct alignas(2 * sizeof(Off)) Off2 { Off x, y; };
    __shared__ __align__(16) Off sV[3][BB];  // a cosmology's list of a type, in floats from the first one's weights
    __shared__ int sB[3][BB], sE[kSpan];
    __shared__ const float *sA[BB];
    const int g = blockIdx.x % ngr, rest = blockIdx.x / ngr, ntl = 3 * n_esel;
    const int nspan = (ntl + kSpan - 1) / kSpan, a = rest / nspan, tl0 = (rest - a * nspan) * kSpan;
    const int b0 = g * BB, nb = min(BB, n - b0), Q = X * Rn;
    const int tid = threadIdx.x, lane = tid & 31, pw = tid >> 5;
    const float *V0 = reqs[b0].V32 + (size_t)a * Rn;
    if (tid < BB) {
        const bool live = tid < nb;
        const ReqDev &rq = reqs[b0 + (live ? tid : 0)];
        const int ng = rq.n_clust, ns = rq.n_lens;
        const Off off = (Off)(rq.V32 + (size_t)a * Rn - V0);
        sA[tid] = rq.a32;
        for (int t = 0; t < 3; t++) {
            const bool both = sym && t == 1;
            sV[t][tid] = off + (t == 0 || both ? 0 : (Off)ng * Q);
            sB[t][tid] = !live ? 0 : t == 0 ? ng : both ? ng + ns : ns;
        }
    }
    if (tid < kSpan && tl0 + tid < ntl) sE[tid] = esel[(tl0 + tid) % n_esel];
    __syncthreads();
    for (int i = tid; i < N * BB; i += kThreads) {
        const int b = i / N, k = i - b * N;
        as[k * BB + b] = b < nb ? __ldg(sA[b] + k) : 0.f;
    }
    __syncthreads();
    int at[NQ];  // past the end: the last node again, not used
#pragma unroll
    for (int i = 0; i < NQ; i++) at[i] = min(32 * (pw + 2 * i) + lane, Rn - 1);
    for (int x = 0; x < kSpan && tl0 + x < ntl; x++) {
        const int tl = tl0 + x, t = tl / n_esel, es = tl - t * n_esel, e = sE[x];
        float *redx = red + (x & 1) * (MT * 4 * BB);
        int most = 0;
#pragma unroll
        for (int b = 0; b < BB; b++) most = max(most, sB[t][b]);
        f32x2 w[PB][NQ];
#pragma unroll
        for (int b = 0; b < PB; b++)
#pragma unroll
            for (int i = 0; i < NQ; i++) w[b][i] = 0;
        const float *Tb = basis + ((size_t)t * L + e) * N * Q + (size_t)a * Rn;
#pragma unroll 4
        for (int k = 0; k < N; k++) {
            f32x2 tv[NQ], av[PB];
#pragma unroll
            for (int i = 0; i < NQ; i++) {
                const float x = __ldg(Tb + (size_t)k * Q + at[i]);
                tv[i] = pair(x, x);
            }
#pragma unroll
            for (int b = 0; b < PB; b += 2) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(as + (size_t)k * BB + 2 * b);
                av[b] = v.x;
                av[b + 1] = v.y;
            }
#pragma unroll
            for (int b = 0; b < PB; b++)
#pragma unroll
                for (int i = 0; i < NQ; i++) w[b][i] = fma2(av[b], tv[i], w[b][i]);
        }
        // Rows past a cosmology's own tracers lie in its work space (sized for the plan's
        // counts); what comes of them is not written.
        for (int j = 0; j < most; j++) {
            f32x2 v[PB][NQ];
            const float *Vj = V0 + (size_t)j * Q;
#pragma unroll
            for (int b = 0; b < PB; b++) {
                const Off2 off = *reinterpret_cast<const Off2 *>(&sV[t][2 * b]);
#pragma unroll
                for (int i = 0; i < NQ; i++)
                    v[b][i] = pair(__ldg(Vj + (off.x + at[i])), __ldg(Vj + (off.y + at[i])));
            }
#pragma unroll
            for (int p = 0; p < 2 && p < NQ; p++) {
                const int vw = pw + 2 * p;
                if (32 * vw >= Rn) break;
                f32x2 part[PB];
#pragma unroll
                for (int b = 0; b < PB; b++) {
                    part[b] = 0;
#pragma unroll
                    for (int i = p; i < NQ; i += 2)
                        if (32 * (pw + 2 * i) + lane < Rn) part[b] = fma2(v[b][i], w[b][i], part[b]);
                }
                float x[BB];
#pragma unroll
                for (int b = 0; b < BB; b++) x[b] = __uint_as_float((uint32_t)(part[b / 2] >> (32 * (b & 1))));
                int mine;
                const float s = lane_sums<BB>(x, lane, mine);
                if (lane % (32 / BB) == 0) redx[(j * 4 + vw) * BB + mine] = s;
            }
        }
        __syncthreads();
        const int nv = min(4, (Rn + 31) / 32);
        for (int i = tid; i < most * BB; i += kThreads) {
            const int j = i / BB, b = i % BB;
            if (j >= sB[t][b]) continue;
            float s = 0.f;
            for (int v = 0; v < nv; v++) s += redx[(j * 4 + v) * BB + b];
            Y[((((size_t)(b0 + b) * 3 + t) * n_esel + es) * X + a) * MT + j] = s;
        }
    }
}

template <int BB, int NQ>
int launch(blast_plan *p, const ReqDev *dreq, int n, const int *d_esel, int n_esel, float *Y, cudaStream_t s)
{
    const int ngr = (n + BB - 1) / BB;
    const size_t smem = sizeof(float) * ((size_t)p->N * BB + (size_t)p->max_tr * 8 * BB);  // at most 24 KB
    const int nspan = (3 * n_esel + kSpan - 1) / kSpan;
    const bool near = request_weights_bytes(p) / sizeof(float) * BB <= INT_MAX;
    (near ? k_contract_f32<BB, NQ, int> : k_contract_f32<BB, NQ, long long>)<<<(unsigned)ngr * p->X * nspan, kThreads,
                                                                               smem, s>>>(
        dreq, n, p->T32, p->L, p->N, p->X, p->Rn, d_esel, n_esel, p->max_tr, p->r_form == 1, ngr, Y);
    BL_CUDA(cudaGetLastError());
    return BLAST_OK;
}

}  // namespace

// NQ R nodes a thread (64 NQ >= n_R), BB cosmologies a block.  Places without a
// cosmology are multiplied all the same, but a larger BB has more loads of the
// basis in flight, so no grid has a variant for one cosmology: 128 R nodes of
// order 64, one cosmology 0.31 ms with BB = 1, 0.29 with 4, 0.40 with 16; 192 of
// order 96 1.04, 0.87 and (BB = 8) 0.70 ms.  Lines, in ms:
//   NQ = 2, BB = 4 / 16: four cosmologies 0.32 / 0.42, eight 0.44 / 0.42 (on a
//     grid of 16 ells and 64 x 64 nodes 0.028 / 0.035), twelve 0.57 / 0.42;
//   NQ = 4, BB = 4 / 8: one 0.52 / 0.42, eight of order 96 1.38 / 0.80;
//   NQ = 8, BB = 4 / 8: four 0.23 / 0.31 (320 nodes), 0.37 / 0.30 (512 nodes of
//     order 96), eight 0.41 / 0.32 and 0.39 / 0.32.
int launch_contract_f32(blast_plan *p, const ReqDev *dreq, int n, const int *d_esel, int n_esel, float *Y,
                        cudaStream_t s)
{
    if (p->Rn <= 128)
        return n <= 8 ? launch<4, 2>(p, dreq, n, d_esel, n_esel, Y, s) : launch<16, 2>(p, dreq, n, d_esel, n_esel, Y, s);
    if (p->Rn <= 256) return launch<8, 4>(p, dreq, n, d_esel, n_esel, Y, s);
    return n <= 4 ? launch<4, 8>(p, dreq, n, d_esel, n_esel, Y, s) : launch<8, 8>(p, dreq, n, d_esel, n_esel, Y, s);
}
