// Step (pre): the cosmology-independent basis integrals of Eq. t_tilde,
//   T~^{AB}_{n;l}(chi_a, R_r chi_a) = int_{kmin}^{kmax} dk f^{AB}(k) T_n(x(k)) j_l(k chi_a) j_l(k R_r chi_a),
// f^gg = k^2, f^gs = 1, f^ss = 1/k^2, by the Clenshaw-Curtis rule of Sec. 3.2:
// a GEMM over the k nodes m,
//   T~[t n][l, q] = sum_m A[m][t n] B_l[m][q],  A = w_m f_t(k_m) T_n(x_m),
//   B_l[m][q]    = j_l(k_m chi_a) j_l(k_m R_r chi_a),
// with B generated on chip from spherical Bessel recurrences in FP64.
//
// The GEMM runs as exact integer products on the FP16 tensor cores (eight 8-bit
// digits an operand, eight exact levels; contract_fx.cu states the arithmetic),
// over windows of at most 56 k nodes: in a window every row of A and every column
// of B has its own exponent, the window's sum is exact in the levels up to the
// dropped ones (about 2^-58 of the row's largest entry times the column's), and
// windows add in FP64.  The two largest entries can lie at different nodes (1/k^2
// falls where j_l j_l rises), so a window also ends where the spreads of w_m and k^2
// multiply to more than 2^6: what is dropped then stays under 2^-52 of the
// window's largest product up to T_n.  Few nodes on a wide k range need it (k over
// [1e-4, 10], 17 nodes, l = 2, type ss: 7e-11 of the sum of magnitudes with one
// window, 1.5e-16 with five); 65,537 nodes get 1173 windows instead of 1171.  What is
// left on the FP64 pipe (two multiply-adds a clock and SM) are the recurrences,
// a product per entry of B and an addition per output and window.  Infinities and
// NaN (the integer recurrences leave the FP64 range below x of about 1e-24) make
// their integrals NaN; entries under 2^-953 count as zero.
//
// Bound by the recurrences.  16 ells to 200, 38 x 64 nodes, order 32, 65,537 k
// nodes: 0.31 s (with the GEMM in FP64 multiply-adds and 2l + 1 counted up in
// FP64 0.81 s); error against an independent FP64 evaluation 2e-15 (9e-15).
#include <algorithm>
#include <cmath>

#include "blast_internal.h"
#include "fx.h"
#include "tc_ptx.h"

namespace {

constexpr int kG = 8;     // plan ells per CTA (one group)
constexpr int kRT = 8;    // R nodes per CTA
constexpr int kMC = 56;   // most k nodes of a window: (1 + kRT) * kMC = 504 Bessel chains
constexpr double kSpread = 64.0;  // largest product of the spreads of w_m and k^2 in a window
constexpr int kKS = kMC / 8;              // MMA K steps of a window (8 k nodes, two digits each)
constexpr int kWork = 512;                // worker threads; then the A loader and the MMA issuer
constexpr int kThreads = kWork + 64;
constexpr int kCols = kG * kRT;           // columns of a CTA, in groups of 16
constexpr int kRows = 16 * kLev;          // rows of a column group's operand, TMEM columns of its levels
constexpr uint32_t kGroupBytes = (kMC / 4) * kRows * 16;  // a column group's digits: [k-group of 4][row][16 B]
constexpr uint32_t kAStep = 4 * 2 * 128 * 16;  // A's digits of a K step: [pair][k-group][128 rows][16 B]
constexpr int kARing = 3;
constexpr size_t kPartBytes = (size_t)256 << 20;  // digits of A in memory at a time

struct BasisCtl {
    uint64_t afull[kARing], aempty[kARing], bready, dfull, dempty, mdone;
    uint64_t never;  // no thread ever arrives on it (test hook)
    uint32_t tmem;
    int abort;
    int colmax[2][kCols];  // biased exponent of a column's largest entry, by parity of the window
    int lg[kG];
    double lgr[kG];
};
constexpr size_t kBasisSmem = 1024 + (kCols / 16) * kGroupBytes + kARing * kAStep +
                              sizeof(double) * (1 + kRT) * kMC * kG + sizeof(BasisCtl);

// k as FP64, 0 < k < 2^31, without the FP64 pipe (a conversion costs a
// recurrence step as much as its multiply-add).
__device__ __forceinline__ double fp64_of(int k)
{
    const int z = __clz(k);
    const uint32_t m = (uint32_t)k << z;
    return __hiloint2double((int)(((uint32_t)(1054 - z) << 20) | ((m >> 11) & 0xfffffu)), (int)(m << 21));
}

// |f| > 1e200 (up to the low 32 bits of the limit), without the FP64 pipe.
__device__ __forceinline__ bool is_huge(double f) { return (__double2hiint(f) & 0x7fffffff) > 0x6974e718; }

// A[m][t*N + n] = w_m f_t(k_m) T_n(x(k_m)); T_n by the three-term recurrence.
__global__ void k_basis_A(const double *__restrict__ kq, const double *__restrict__ wq, int Nk, int N,
                          int kmap, double kmin, double kmax, double *__restrict__ A)
{
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= Nk) return;
    double k = kq[m];
    double x = (kmap == 0) ? (2.0 * k - kmin - kmax) / (kmax - kmin)
                           : 2.0 * (log(k) - log(kmin)) / (log(kmax) - log(kmin)) - 1.0;
    x = fmin(1.0, fmax(-1.0, x));
    double f0 = wq[m] * k * k, f1 = wq[m], f2 = wq[m] / (k * k);
    double *row = A + (size_t)m * 3 * N;
    double tprev = 1.0, tcur = x;
    for (int n = 0; n < N; n++) {
        double Tn;
        if (n == 0) Tn = 1.0;
        else if (n == 1) Tn = x;
        else { Tn = 2.0 * x * tcur - tprev; tprev = tcur; tcur = Tn; }
        row[n] = f0 * Tn;
        row[N + n] = f1 * Tn;
        row[2 * N + n] = f2 * Tn;
    }
}

// j_l(x) for the (at most kG) ascending multipoles lg[0..ng) of one group.
// x > lhi: forward recurrence from j_0, j_1 (stable for l < x).
// x <= lhi: Miller's backward recurrence from lhi + 20 + 10 lhi^(1/3), scaled
// by the least-squares match of the recurrence's two lowest orders to the
// closed forms of j_0 and j_1.  Values below 1e-323 (j_l(x) <= (e x / 2l)^l)
// are returned as zero without a recurrence.
__device__ void jl_group(double x, const int *lg, int ng, double *out)
{
#pragma unroll
    for (int g = 0; g < kG; g++) out[g] = 0.0;
    if (ng <= 0 || !(x > 0.0)) return;
    const int llo = lg[0], lhi = lg[ng - 1];
    if ((double)llo * log(2.718281828459045 * x / (2.0 * llo)) < -744.0) return;
    double s, c;
    sincos(x, &s, &c);
    const double inv = 1.0 / x;
    double j0 = s * inv;
    double j1 = (x < 1e-2) ? x * (1.0 / 3.0 - x * x / 30.0 + x * x * x * x / 840.0) : (j0 - c) * inv;
    if (x > (double)lhi) {
        double jm = j0, jc = j1;
        int gi = 0;
        while (gi < ng && lg[gi] <= 1) { out[gi] = (lg[gi] == 0) ? j0 : j1; gi++; }
        for (int l = 1; l < lhi; l++) {
            double jn = (fp64_of(2 * l + 1) * inv) * jc - jm;  // j_{l+1}
            jm = jc;
            jc = jn;
            if (gi < ng && l + 1 == lg[gi]) { out[gi] = jc; gi++; }
        }
        return;
    }
    const int l0 = lhi + 20 + (int)(10.0 * cbrt((double)lhi));
    double fp = 0.0, f = 1e-200;
    int gi = ng - 1;
    for (int l = l0; l > 0; l--) {
        if (gi >= 0 && l == lg[gi]) { out[gi] = f; gi--; }
        double fm = (fp64_of(2 * l + 1) * inv) * f - fp;  // f_{l-1}
        fp = f;
        f = fm;
        if ((l & 3) == 0 && is_huge(f)) {
            f *= 1e-200;
            fp *= 1e-200;
#pragma unroll
            for (int g = 0; g < kG; g++)
                if (g > gi) out[g] *= 1e-200;
        }
    }
    // f = f_0, fp = f_1 (arbitrary scale): normalise before squaring
    const double mx = fmax(fabs(f), fabs(fp));
    f /= mx;
    fp /= mx;
    double scale = (j0 * f + j1 * fp) / ((f * f + fp * fp) * mx);
#pragma unroll
    for (int g = 0; g < kG; g++) out[g] *= scale;
}

// j_v0(x) and j_v0+1(x) for a fractional order v0 in [0, 1) (non-integer
// multipoles), j_v = sqrt(pi / 2x) J_{v+1/2}:
// x >= 30: Hankel's asymptotic expansion, j_v = (P cos w - Q sin w) / x with
//   w = x - (v + 1) pi / 2 (formed by angle addition from sincos(x), which
//   keeps the phase exact for large x), P and Q the even and odd terms of
//   a_k = (m - 1)(m - 9)...(m - (2k-1)^2) / (k! (8x)^k), m = 4 (v + 1/2)^2;
// 1e-3 <= x < 30: Miller's backward recurrence on J_{mu0 + k}, mu0 =
//   frac(v0 + 1/2), normalised by Neumann's expansion
//   (x/2)^mu0 = sum_i (mu0 + 2i) Gamma(mu0 + i) / i! J_{mu0 + 2i};
// x < 1e-3: the first three terms of the power series.
__device__ void jnu_start(double v0, double x, double &j0, double &j1)
{
    const double mu = v0 + 0.5;
    if (x >= 30.0) {
        double sx, cx;
        sincos(x, &sx, &cx);
        double out[2];
#pragma unroll
        for (int o = 0; o < 2; o++) {
            const double v = v0 + o, m = 4.0 * (v + 0.5) * (v + 0.5);
            double P = 1.0, Qs = 0.0, t = 1.0;
            for (int k = 1; k < 60; k++) {
                const double c = (double)(2 * k - 1);
                const double tn = t * (m - c * c) / ((double)k * 8.0 * x);
                if (fabs(tn) > fabs(t) && k > 2) break;  // the asymptotic terms start to grow
                t = tn;
                const int r = k & 3;  // signs: k = 1 +Q, 2 -P, 3 -Q, 4 +P
                if (r == 1) Qs += t;
                else if (r == 2) P -= t;
                else if (r == 3) Qs -= t;
                else P += t;
                if (fabs(t) < 1e-18) break;
            }
            double sp, cp;  // phase (v + 1) pi / 2
            sincospi(0.5 * (v + 1.0), &sp, &cp);
            const double cw = cx * cp + sx * sp, sw = sx * cp - cx * sp;
            out[o] = (P * cw - Qs * sw) / x;
        }
        j0 = out[0];
        j1 = out[1];
        return;
    }
    const double pre = sqrt(0.5 * 3.14159265358979323846 / x);
    if (x < 1e-3) {
#pragma unroll
        for (int o = 0; o < 2; o++) {
            const double m = mu + o, h = 0.25 * x * x;
            const double J = pow(0.5 * x, m) / tgamma(m + 1.0) * (1.0 - h / (m + 1.0) + h * h / (2.0 * (m + 1.0) * (m + 2.0)));
            (o ? j1 : j0) = pre * J;
        }
        return;
    }
    const int nb = (int)floor(mu);
    const double mu0 = mu - nb;
    const int K = (int)x + 40;  // <= 69
    double c[36];               // Neumann weights for k = 2i <= K
    double g = tgamma(mu0 + 1.0);
    c[0] = g;
    for (int i = 1; i <= K / 2; i++) {
        c[i] = (mu0 + 2.0 * i) * g;
        g *= (mu0 + i) / (i + 1.0);
    }
    double fp = 0.0, f = 1e-250, S = 0.0, r0 = 0.0, r1 = 0.0;
    for (int k = K; k >= 0; k--) {
        if (k == nb) r0 = f;
        if (k == nb + 1) r1 = f;
        if ((k & 1) == 0) S += c[k / 2] * f;
        if (k == 0) break;
        const double fm = 2.0 * (mu0 + k) / x * f - fp;
        fp = f;
        f = fm;
        if (fabs(f) > 1e200) { f *= 1e-200; fp *= 1e-200; S *= 1e-200; r0 *= 1e-200; r1 *= 1e-200; }
    }
    const double nrm = pow(0.5 * x, mu0) / S;
    j0 = pre * r0 * nrm;
    j1 = pre * r1 * nrm;
}

// j_nu(x) for a real multipole nu >= 2: from j_v0 and j_v0+1 (v0 = frac(nu))
// forward to nu when x > nu, else Miller's backward recurrence from
// nu + 20 + 10 nu^(1/3) down to v0 matched to them (least squares, as for
// integer orders).  Values below 1e-323 are zero.
__device__ double jnu_real(double nu, double x)
{
    if (!(x > 0.0)) return 0.0;
    if (nu * log(2.718281828459045 * x / (2.0 * nu)) < -744.0) return 0.0;
    const int n = (int)floor(nu);
    const double v0 = nu - n;
    double j0, j1;
    jnu_start(v0, x, j0, j1);
    if (n == 0) return j0;
    if (x > nu) {
        double jm = j0, jc = j1, v = v0 + 1.0;
        for (int k = 1; k < n; k++) {
            const double jn = (2.0 * v + 1.0) / x * jc - jm;
            jm = jc;
            jc = jn;
            v += 1.0;
        }
        return jc;
    }
    const int top = n + 20 + (int)(10.0 * cbrt((double)n));
    double fp = 0.0, f = 1e-200, rec = 0.0, v = v0 + top;
    for (int k = top; k > 0; k--) {
        if (k == n) rec = f;
        const double fm = (2.0 * v + 1.0) / x * f - fp;  // order v - 1
        fp = f;
        f = fm;
        v -= 1.0;
        if (fabs(f) > 1e200) { f *= 1e-200; fp *= 1e-200; rec *= 1e-200; }
    }
    const double mx = fmax(fabs(f), fabs(fp));
    f /= mx;
    fp /= mx;
    return rec * (j0 * f + j1 * fp) / ((f * f + fp * fp) * mx);
}

// Digits of A: rows t N + n of 128-row tiles, window by window, each row with
// its own exponent in a window; the layout is the MMA operand's, one 16 KB block
// per (row tile, window, K step).  wstart lists the part's windows, A starts at its
// first node.
__global__ void __launch_bounds__(128)
k_basis_A_digits(const double *__restrict__ A, const int *__restrict__ wstart, int rows3, int nwin,
                 uint4 *__restrict__ dig, uint16_t *__restrict__ ea)
{
    const int win = blockIdx.x, mt = blockIdx.y, row = mt * 128 + threadIdx.x;
    const int m0 = wstart[win] - wstart[0], m1 = wstart[win + 1] - wstart[0];
    const bool live = row < rows3;
    int mx = 0;
    for (int i = 0; i < kMC; i++)
        if (live && m0 + i < m1) mx = max(mx, (__double2hiint(A[(size_t)(m0 + i) * rows3 + row]) >> 20) & 0x7ff);
    const int M = mx < 70 ? kNone : mx;
    ea[((size_t)mt * nwin + win) * 128 + threadIdx.x] = (uint16_t)M;
    const uint32_t top = fx_top(M);
    uint4 *dst = dig + ((size_t)mt * nwin + win) * kKS * (kAStep / 16) + threadIdx.x;
    for (int kg = 0; kg < kMC / 4; kg++) {
        uint32_t w[4][4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int m = m0 + kg * 4 + i;
            fx_pairs<false>(live && m < m1 ? A[(size_t)m * rows3 + row] : 0.0, top, w[0][i], w[1][i], w[2][i], w[3][i]);
        }
#pragma unroll
        for (int p = 0; p < 4; p++)
            dst[(size_t)(kg >> 1) * (kAStep / 16) + (p * 2 + (kg & 1)) * 128] =
                make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
    }
}

// MMA with both operands in shared memory.
__device__ __forceinline__ void umma_f16_ss(uint32_t d_tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        ::"r"(d_tmem), "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

// A CTA owns eight R nodes of a chi node and a group of eight ells: 64 columns,
// 128-row tiles of A in turn.  Per window the workers run the recurrences, then
// take the previous window's sums out of TMEM, then write the digits of the
// products j j for the MMAs, which run beside the next window's recurrences.
// A launch takes the windows of one part of the k nodes; all but the first add to T.
__global__ void __launch_bounds__(kThreads, 1)
k_basis_fx(const uint4 *__restrict__ dig, const uint16_t *__restrict__ ea, int Mt, int nwin,
           const double *__restrict__ kq, const int *__restrict__ wstart, int add, int N,
           const double *__restrict__ ell, int real_ell, int L, const double *__restrict__ chi,
           const double *__restrict__ R, int Rn, int Q, double *__restrict__ T, int *err,
           long long limit, int trip)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sB = (unsigned char *)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);  // [group][k-group][row][16 B]
    unsigned char *sA = sB + (kCols / 16) * kGroupBytes;                                  // [ring][K step block]
    double *Jv = reinterpret_cast<double *>(sA + kARing * kAStep);                        // [(1 + kRT) kMC][kG]
    BasisCtl *ctl = reinterpret_cast<BasisCtl *>(Jv + (1 + kRT) * kMC * kG);
    volatile int *abort_flag = &ctl->abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r0 = blockIdx.x * kRT, a = blockIdx.y, e0 = blockIdx.z * kG, ng = min(kG, L - e0);

    if (tid == 0) {
        for (int i = 0; i < kARing; i++) { mbar_init(&ctl->afull[i], 1); mbar_init(&ctl->aempty[i], 1); }
        mbar_init(&ctl->bready, kWork);
        mbar_init(&ctl->dfull, 1);
        mbar_init(&ctl->dempty, kWork);
        mbar_init(&ctl->mdone, 1);
        mbar_init(&ctl->never, 1);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < kG) {
        ctl->lgr[tid] = (tid < ng) ? ell[e0 + tid] : 0.0;
        ctl->lg[tid] = (int)ctl->lgr[tid];
    }
    if (warp == kWork / 32 + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem)),
                     "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem;

    if (warp == kWork / 32) {
        // ---------------------------------------------- A loader: blocks in the order of the MMAs
        Ring ring;
        uint32_t k = 0;
        const int stop = blockIdx.x + blockIdx.y + blockIdx.z == 0 ? min(trip, nwin - 1) : -1;  // test hook's window
        bool ok = true;
        for (int win = 0; ok && win < nwin; win++)
            for (int mt = 0; ok && mt < Mt; mt++)
                for (int ks = 0; ks < kKS; ks++, k++, ring.next(kARing)) {
                    const bool bad = (win == stop && !mbar_wait(&ctl->never, 0, 32, kTripLimit, abort_flag)) ||
                                     !mbar_wait(&ctl->aempty[ring.st], ring.ph ^ 1, 32, limit, abort_flag);
                    if (__any_sync(0xffffffffu, bad)) {
                        if (lane == 0) { atomicExch(err, 21); *abort_flag = 1; }
                        ok = false;
                        break;
                    }
                    if (elect_one()) {
                        mbar_expect_tx(&ctl->afull[ring.st], kAStep);
                        bulk_g2s(sA + (size_t)ring.st * kAStep,
                                 dig + (((size_t)mt * nwin + win) * kKS + ks) * (kAStep / 16), kAStep,
                                 &ctl->afull[ring.st]);
                    }
                    __syncwarp();
                }
        for (uint32_t h = (k > (uint32_t)kARing ? k - kARing : 0); h < k; h++)  // every load has landed before the exit
            mbar_wait(&ctl->afull[h % kARing], (h / kARing) & 1, 32);
        __syncwarp();
    } else if (warp == kWork / 32 + 1) {
        // ---------------------------------------------- MMA issuer
        const uint32_t ab = __shfl_sync(0xffffffffu, smem_u32(sA), 0), bb = __shfl_sync(0xffffffffu, smem_u32(sB), 0);
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        Ring ring;
        uint32_t fills = 0;  // accumulator fills so far
        bool ok = true;
        for (int win = 0; ok && win < nwin; win++)
            for (int mt = 0; ok && mt < Mt; mt++, fills++)
                for (int ks = 0; ks < kKS; ks++, ring.next(kARing)) {
                    const bool bad =
                        (ks == 0 && mt == 0 && !mbar_wait(&ctl->bready, win & 1, 32, limit, abort_flag)) ||
                        (ks == 0 && !mbar_wait(&ctl->dempty, (fills & 1) ^ 1, 32, limit, abort_flag)) ||
                        !mbar_wait(&ctl->afull[ring.st], ring.ph, 32, limit, abort_flag);
                    if (__any_sync(0xffffffffu, bad)) {
                        if (lane == 0) { atomicExch(err, 22); *abort_flag = 1; }
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t ad = sdesc_plain(ab + ring.st * kAStep, 128 * 16);
                        const uint64_t bd = sdesc_plain(bb + ks * 2 * kRows * 16, kRows * 16);
#pragma unroll
                        for (int p = 0; p < 4; p++) {
                            const int s = p < 2 ? p : p + 2;  // digit pairs (s, s + 2): levels from s on
                            const uint32_t idesc = (1u << 4) | ((uint32_t)((kLev - s) * 16 >> 3) << 17) | (8u << 24);
#pragma unroll
                            for (int cg = 0; cg < kCols / 16; cg++)
                                umma_f16_ss(tm + cg * kRows + s * 16, ad + ((p * 2 * 128 * 16) >> 4),
                                            bd + ((cg * kGroupBytes) >> 4), idesc, (ks | p) != 0);
                        }
                        umma_commit(&ctl->aempty[ring.st]);
                        if (ks == kKS - 1) umma_commit(&ctl->dfull);
                    }
                    __syncwarp();
                }
        if (elect_one()) umma_commit(&ctl->mdone);  // every MMA has completed before TMEM is released
        __syncwarp();
        mbar_wait(&ctl->mdone, 0, 32);
        __syncwarp();
    } else {
        // ---------------------------------------------- workers
        const double chia = chi[a];
        const int mi = tid % kMC, side = tid / kMC, rr = r0 + side - 1;  // chain: k node of the window, distance
        const double dist = side == 0 ? chia : (side <= kRT && rr < Rn) ? R[rr] * chia : 0.0;
        const int quad = warp & 3, cg = warp >> 2;  // TMEM lanes and column group taken out
        uint32_t fills = 0;
        bool dead = false;
        auto take = [&](int win) {  // the window's sums join the output
            for (int mt = 0; mt < Mt; mt++, fills++) {
                if (!dead) {
                    const bool bad = !mbar_wait(&ctl->dfull, fills & 1, 0, limit, abort_flag);
                    if (__any_sync(0xffffffffu, bad)) {
                        if (lane == 0) { atomicExch(err, 23); *abort_flag = 1; }
                        dead = true;
                    }
                }
                if (dead) continue;
                tc_fence_after();
                const int row = mt * 128 + quad * 32 + lane;
                const int me = ea[((size_t)mt * nwin + win) * 128 + quad * 32 + lane] - 994;
                const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + cg * kRows;
                const int t = row / N, n = row - t * N;
#pragma unroll 1
                for (int c4 = 0; c4 < 16; c4 += 4) {
                    uint32_t D[kLev][4];
#pragma unroll
                    for (int l = 0; l < kLev; l++) tmem_ld4(tl + l * 16 + c4, D[l]);
                    tmem_wait_ld4(D[0]);
#pragma unroll
                    for (int l = 1; l < kLev; l++) reg_fence4(D[l]);
                    const int col = cg * 16 + c4, g = col / kRT, r = r0 + col % kRT;
                    if (t < 3 && g < ng) {
                        double *out = T + (((size_t)t * L + e0 + g) * N + n) * Q + (size_t)a * Rn + r;
#pragma unroll
                        for (int i = 0; i < 4; i++) {
                            int d[kLev];
#pragma unroll
                            for (int l = 0; l < kLev; l++) {
                                const float f = __uint_as_float(D[l][i]);
                                d[l] = __float2int_rn(f + f);
                            }
                            const int mc = ctl->colmax[win & 1][col + i];
                            double v = fx_join(d, me + mc);
                            // an infinity or NaN has no digits: the sum is what a product with it is
                            if (mc == 2047 || me == 2047 - 994) v = __longlong_as_double(0x7ff8000000000000ll);
                            if (r + i < Rn) out[i] = add | win ? out[i] + v : v;
                        }
                    }
                    __syncwarp();
                }
                tc_fence_before();
                mbar_arrive(&ctl->dempty);
            }
        };
        // the window's nodes and this chain's k; the next ones are fetched a window ahead
        int m0 = wstart[0], m1 = wstart[1];
        const int kend = wstart[nwin] - 1;
        double kx = kq[min(m0 + mi, kend)];
        for (int win = 0; win < nwin; win++) {
            const int m2 = wstart[min(win + 2, nwin)], mcnt = m1 - m0;
            const double k = kx;
            kx = kq[min(m1 + mi, kend)];
            if (side <= kRT) {
                double *out = Jv + (side * kMC + mi) * kG;
                const bool ok = !dead && mi < mcnt && dist > 0.0;
                if (ok && !real_ell) {
                    jl_group(k * dist, ctl->lg, ng, out);
                } else if (ok) {  // each non-integer multipole has its own recurrence
#pragma unroll
                    for (int g = 0; g < kG; g++) out[g] = (g < ng) ? jnu_real(ctl->lgr[g], k * dist) : 0.0;
                } else {
#pragma unroll
                    for (int g = 0; g < kG; g++) out[g] = 0.0;
                }
            }
            if (tid < kCols) ctl->colmax[win & 1][tid] = 0;
            if (win > 0) take(win - 1);  // its MMAs have read their digits
            named_bar_sync(1, kWork);
            // products j j of column (g, r) and of the k nodes of k-groups kg0 and kg0 + 8
            const int col = tid % kCols, kg0 = tid / kCols, g = col / kRT, rc = col % kRT;
            double p[2][4];
            int mx = 0;
#pragma unroll
            for (int h = 0; h < 2; h++)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int m = (kg0 + 8 * h) * 4 + i;
                    p[h][i] = m < kMC ? Jv[m * kG + g] * Jv[((1 + rc) * kMC + m) * kG + g] : 0.0;
                    mx = max(mx, (__double2hiint(p[h][i]) >> 20) & 0x7ff);
                }
            atomicMax(&ctl->colmax[win & 1][col], mx);
            named_bar_sync(1, kWork);
            const int M = ctl->colmax[win & 1][col];
            const uint32_t top = fx_top(M < 70 ? kNone : M);
            unsigned char *dst = sB + (col / 16) * kGroupBytes + (col % 16) * 16;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int kg = kg0 + 8 * h;
                if (kg >= kMC / 4) break;
                uint64_t y[4];
#pragma unroll
                for (int i = 0; i < 4; i++) y[i] = fx_digits(p[h][i], top);
                uint32_t prev[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};  // digits j - 2 and j - 1
#pragma unroll
                for (int j = 0; j < kLev; j++) {
                    uint32_t w[4];
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const uint32_t d =
                            __half_as_ushort(__int2half_rn(((int)((y[i] >> (8 * (7 - j))) & 255) - 128) * 256));
                        w[i] = (d << 16) | prev[0][i];
                        prev[0][i] = prev[1][i];
                        prev[1][i] = d;
                    }
                    *reinterpret_cast<uint4 *>(dst + (size_t)(kg * kRows + j * 16) * 16) =
                        make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            fence_proxy_async();
            mbar_arrive(&ctl->bready);
            m0 = m1;
            m1 = m2;
        }
        take(nwin - 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWork / 32 + 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    }
}

// FP64 basis -> FP32 copy (same layout) for the CUDA-core FP32 path.
__global__ void k_basis_to_f32(const double *__restrict__ T, float *__restrict__ T32, size_t n)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t stride = (size_t)gridDim.x * blockDim.x;
    for (; i < n; i += stride) T32[i] = (float)T[i];
}

}  // namespace

std::vector<int> basis_windows(const std::vector<double> &k, const std::vector<double> &w)
{
    const int n = (int)k.size();
    std::vector<int> start(1, 0);
    double lo = w[0], hi = w[0], k0 = k[0] * k[0];  // k falls
    for (int m = 1, first = 0; m < n; m++) {
        const double l = std::min(lo, w[m]), h = std::max(hi, w[m]);
        if (m - first < kMC && h * k0 <= kSpread * l * (k[m] * k[m])) {
            lo = l;
            hi = h;
        } else {
            start.push_back(first = m);
            lo = hi = w[m];
            k0 = k[m] * k[m];
        }
    }
    start.push_back(n);
    return start;
}

int launch_basis(blast_plan *p, cudaStream_t s)
{
    const int rows3 = 3 * p->N;
    const std::vector<int> &wstart = p->kwin;
    const int Mt = (rows3 + 127) / 128, nwin = (int)wstart.size() - 1;
    uint4 *dig = nullptr;
    uint16_t *ea = nullptr;
    double *A = nullptr, *tab = nullptr;
    int gave_up = 0;
    const int trip = p->test_trip;
    p->test_trip = -1;  // one call only
    int rc = BLAST_OK;
    const size_t ntab = 2 * (size_t)p->Nk + p->Rn + p->L;
    if (cudaMalloc(&tab, sizeof(double) * ntab + sizeof(int) * (wstart.size() + 1))) {
        cudaGetLastError();
        return BLAST_ENOMEM;
    }
    double *kq = tab, *wq = kq + p->Nk, *R = wq + p->Nk, *ell = R + p->Rn;
    int *ws = reinterpret_cast<int *>(tab + ntab);
    int *err = ws + wstart.size();  // the build's own error word: the plan's may hold an earlier call's
    // A and its digits take three times (rows padded to 128: up to 43 times) the memory of A
    // alone, so they are made for a part of the windows at a time, and for smaller parts
    // where even that is not to be had.  The sums do not depend on the parts.
    const size_t wbytes = (size_t)Mt * kKS * kAStep;
    const int parts = (int)((nwin * wbytes + kPartBytes - 1) / kPartBytes);
    int per = (nwin + parts - 1) / parts;  // windows of a part
    while (!rc) {
        if (!cudaMalloc(&A, sizeof(double) * per * kMC * rows3) && !cudaMalloc(&dig, per * wbytes) &&
            !cudaMalloc(&ea, sizeof(uint16_t) * Mt * per * 128))
            break;
        cudaGetLastError();
        cudaFree(A); cudaFree(dig); cudaFree(ea);
        A = nullptr; dig = nullptr; ea = nullptr;
        if (per == 1) rc = BLAST_ENOMEM;
        per = (per + 1) / 2;
    }
    if (!rc && (cudaMemcpyAsync(kq, p->kq.data(), sizeof(double) * p->Nk, cudaMemcpyHostToDevice, s) ||
                cudaMemcpyAsync(wq, p->wq.data(), sizeof(double) * p->Nk, cudaMemcpyHostToDevice, s) ||
                cudaMemcpyAsync(R, p->R.data(), sizeof(double) * p->Rn, cudaMemcpyHostToDevice, s) ||
                cudaMemcpyAsync(ell, p->ell.data(), sizeof(double) * p->L, cudaMemcpyHostToDevice, s) ||
                cudaMemcpyAsync(ws, wstart.data(), sizeof(int) * wstart.size(), cudaMemcpyHostToDevice, s) ||
                cudaMemsetAsync(err, 0, sizeof(int), s)))
        rc = BLAST_EDEVICE;
    // The waits cover the recurrences of a window, 512 chains at two FP64 lanes a clock: an
    // operation of every chain takes 256 cycles, a step about 14 of them with a division,
    // real orders have a recurrence each, and a warp may run both directions.  Eight times
    // that: a full window of eight real multipoles near 1e5 takes 4e9 cycles, where a fixed
    // limit of 4e9 ran out.
    const double top = p->ell.back(), steps = (top + 20.0 + 10.0 * cbrt(top)) * (p->real_ell ? kG : 1);
    const long long limit = kWaitLimit + (long long)(steps * (8 * 2 * 14 * 256));
    if (!rc && allow_opt_in_smem(k_basis_fx, p->device) != cudaSuccess) rc = BLAST_EDEVICE;
    for (int w0 = 0; w0 < nwin && !rc; w0 += per) {
        const int nw = std::min(per, nwin - w0), m0 = wstart[w0], nk = wstart[w0 + nw] - m0;
        k_basis_A<<<(nk + 255) / 256, 256, 0, s>>>(kq + m0, wq + m0, nk, p->N, p->kmap, p->k_min, p->k_max, A);
        if (cudaGetLastError() != cudaSuccess) rc = BLAST_EDEVICE;
        k_basis_A_digits<<<dim3(nw, Mt), 128, 0, s>>>(A, ws + w0, rows3, nw, dig, ea);
        const dim3 grid((p->Rn + kRT - 1) / kRT, p->X, (p->L + kG - 1) / kG);
        k_basis_fx<<<grid, kThreads, kBasisSmem, s>>>(dig, ea, Mt, nw, kq, ws + w0, w0 > 0, p->N, ell,
                                                      p->real_ell ? 1 : 0, p->L, p->d_chi, R, p->Rn, p->Q, p->T64, err,
                                                      limit, w0 ? -1 : trip);
        if (cudaGetLastError() != cudaSuccess) rc = BLAST_EDEVICE;
    }
    if (!rc && cudaMemcpyAsync(&gave_up, err, sizeof(int), cudaMemcpyDeviceToHost, s)) rc = BLAST_EDEVICE;
    if (cudaStreamSynchronize(s) != cudaSuccess && !rc) rc = BLAST_EDEVICE;
    cudaFree(tab); cudaFree(A); cudaFree(dig); cudaFree(ea);
    if (!rc && gave_up) rc = BLAST_ETIMEOUT;
    if (!rc && cudaGetLastError() != cudaSuccess) rc = BLAST_EDEVICE;
    return rc;
}

int launch_basis_convert(blast_plan *p, unsigned mask, cudaStream_t s)
{
    size_t n = (size_t)3 * p->L * p->N * p->Q;
    int rc = fx_prepare(p, s);
    if (rc) return rc;
    if ((mask & BLAST_BASIS_FP32) && p->T32) {
        k_basis_to_f32<<<152 * 8, 256, 0, s>>>(p->T64, p->T32, n);
        BL_CUDA(cudaGetLastError());
        p->have32 = true;
    }
    if ((mask & BLAST_BASIS_BF16S) && p->Tsl) {
        if ((rc = launch_basis_slices(p, s))) return rc;
        p->havebf = true;
    }
    return BLAST_OK;
}
