// FP64 contraction (a) with the R sum of quadrature (b), on the tensor cores:
//
//   w_b(t, l, q) = sum_n a_b[n] T~[t][l][n][q]                       (Eq. pmd)
//   Y_b(t, l, a, j) = sum_r V_bj(a, r) w_b(t, l, a n_R + r)
//
// An SM retires two FP64 multiply-adds per clock and 4096 FP16 ones, so the
// Chebyshev sum is done in exact integer arithmetic on the FP16 pipe.  Both
// operands are cut to 62 fractional bits below their largest entry (basis: the
// largest over n of the column; coefficients: the largest of the cosmology)
// and written as eight balanced base-256 digits,
//
//   T~[n][q] = 2^(eT(q) - 62) sum_p 256^(7-p) t_p,   a[n] = 2^(ea - 62) sum_p 256^(7-p) a_p,
//
// |digit| <= 128 (64 for p = 0).  A digit is exact in FP16, a product below
// 2^14, and level k, D_k = sum_{p+q=k} sum_n a_p t_q, below 2^24 for n_cheb <=
// 128 and k <= 7, so the FP32 accumulation of levels 0..7 is exact in any
// order.  What is cut off and the dropped levels are relative to max_n |a_n|
// max_n |T~[n][q]|: under n_cheb 2^-56 of it in the worst case, about 2^-59 for
// digits of random sign.  A multiply-add chain rounds its partial sums, so where
// T~ rises as a falls the chain keeps more of sum_n |a_n T~[n][q]|: tables rising by
// 10^3, 10^6 and 10^9 with n, under coefficients falling to nothing, put 8e-16,
// 7e-13 and 4e-11 of that sum between the two.  The spectra do not see it: every a_n
// comes from the fit with a rounding of about 2^-53 max |a| of its own, and against
// quad precision the same calls are off by 5.1e-14, 1.7e-11 and 1.1e-9 by either
// path.  Tables of Bessel integrals have max |a| max |T~| <= 1.3 sum_n |a_n T~| over the
// R nodes of a chi (orders 20 to 96, ells to 120; single columns far from R = 1 reach
// 1.4e3).  The epilogue joins the eight integers into one FP64 number with a single
// rounding, in integer arithmetic, and the R sum runs in FP64 multiply-adds.
//
// Because every level is exact and the R sum has one fixed order, a
// cosmology's result is the same in every batch.
//
// Layout of one tile: M = 128 chi-R nodes (TMEM lanes), N = 16 cosmologies x
// 8 levels (TMEM columns, column = 16 level + cosmology), K = n_cheb.  The
// nodes are the M side because a batch of one then fills the tile (a batch on
// the M side would leave 127 of 128 lanes empty), and level = a-digit +
// t-digit becomes a column offset of the accumulator: one MMA per basis digit
// covers all its pairs.  Two basis digits share an MMA: the K positions of
// order n hold digits s + 2 and s of T~ (they lie two bytes apart in a 32-bit
// word, so one byte permute unpacks both), against rows holding a-digits
// j - 2 and j.
//
// Warp roles: TMA producer (FP64 basis tiles as they stand in memory, no
// second table), MMA issuer, eight slicer warps (FP64 -> digits, integer and
// half2 arithmetic) with two warps that fetch the column exponents, two epilogue
// warpgroups that take turns: while one joins levels (integer pipe) the other
// sums over R (FP64 pipe).  Slicers that fetched the exponents themselves waited
// for them (one cosmology 0.380 ms, with the two warps 0.365 ms).
//
// What bounds it, and what it measured (64 ells, 128 x 128 nodes, order 64, 5+5
// tracers; the multiply-add kernel of eval.cu in brackets): one cosmology is
// near the reading of the basis (1.61 GB: 0.24 ms) and bound by the slicers'
// integer pipe, 0.37 ms (0.64 ms); 24 cosmologies 1.74 ms (14.0 ms), bound by
// the FP64 multiply-adds of the R sum, five per node instead of 69, and by the
// L2 latency of their weights.
#include <cmath>
#include <cstring>

#include "blast_internal.h"
#include "fx.h"
#include "tc_ptx.h"

namespace {

constexpr int kNB = 16;                  // cosmologies per group
constexpr int kRows = kNB * kLev;        // rows of the coefficient operand, columns of an accumulator
constexpr int kM = 128;                  // chi-R nodes per tile
constexpr int kKC = 32;                  // Chebyshev orders per chunk, in steps of 8 (one MMA K step)
constexpr int kUnsigned = 76;            // largest n_cheb for unsigned basis digits
constexpr int kThreads = 640;            // TMA, MMA, 2 exponent, 8 epilogue and 8 slicer warps
constexpr int kEpi0 = 4, kSli0 = 12;     // first epilogue and slicer warp
constexpr int kWP = kM + 8;              // row pitch of w in shared memory (8 chains x 2 rows without conflicts)
constexpr int kJC = 5;                   // tracers summed together
constexpr uint32_t kStageBytes = kKC * kM * 8;   // basis chunk as FP64
constexpr uint32_t kChunkCols = 128;             // TMEM columns of a chunk's digits: 4 pairs x 4 K steps x 8
constexpr int kChunks = 2;                       // chunks of digits in TMEM
constexpr uint32_t kTmemCols = 512;              // two accumulators and the digits
constexpr int kMaxRing = 4;
constexpr int kBad = 1 << 20;            // exponent of coefficients that are not all finite

constexpr int kTops = 4;                         // items whose column exponents are at hand

struct FxCtl {
    uint32_t top[kTops][kM];  // fx_top of the columns' exponents
    uint64_t efull[kTops], eempty[kTops];
    uint64_t tfull[kMaxRing], tempty[kMaxRing], sfull[kChunks], sempty[kChunks], dfull[2], dempty[2], mdone;
    uint64_t never;  // no thread ever arrives on it (test hook)
    uint32_t tmem;
    int abort;
    const double *V[kNB];
    int ng[kNB], ns[kNB], ea[kNB];
    int most[3];           // largest clustering, lensing and total tracer count of the group
    uint32_t inv[3], invb; // floor(2^32 / d) + 1 of those and of the group's size
    int esel[BLAST_MAX_ELL];
};

struct FxArgs {
    const ReqDev *reqs;
    int n, ngr, gs;        // requests, groups, requests per group
    int L, N, Q, Rn, X, n_esel, MT, sym;
    int span, rtq, apt;    // nodes per tile, tiles per chi node (or 1), chi nodes per tile (or 1)
    int nqt;               // node groups: ceil(X / apt)
    int q_fast;            // unit order: node groups fastest, or (type, ell) fastest
    int inner;             // units of the fast index: nqt (q_fast) or 3 n_esel
    int kT;                // ring depth of the FP64 chunks
    const int *esel;
    const uint16_t *cexp;  // [3 L Q] biased exponent of the largest entry of a basis column
    double *Y;             // [n][3][n_esel][X][MT]
    int *err;
    int trip;              // test hook: item before which CTA 0 waits on a barrier nothing completes (-1 off)
};

// MMA with A from tensor memory (128 lanes x 16 FP16 in 8 columns), B from shared memory.
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bd), "r"(idesc), "r"(acc));
}

// Items of a CTA: its units (chi nodes of one type and ell) two by two, R tile
// by R tile, so that consecutive items belong to units of different parity: a
// unit's parity names its accumulator and its epilogue warpgroup.  A last
// single unit runs alone.  Stepping costs a few additions (every role steps
// through every item, and a division by a run-time number costs them more than
// reading the item's basis column).
struct FxItem {
    int left;                      // units of this CTA from this pair on
    int h, rt;                     // parity, R tile
    int out[2], in[2];             // slow and fast index of the pair's units

    __device__ __forceinline__ FxItem(const FxArgs &A, int u0, int ustep, int n_mine) : left(n_mine), h(0), rt(0)
    {
        const int u1 = u0 + ustep;
        out[0] = u0 / A.inner;
        in[0] = u0 - out[0] * A.inner;
        out[1] = u1 / A.inner;
        in[1] = u1 - out[1] * A.inner;
        dout = 2 * ustep / A.inner;
        din = 2 * ustep - dout * A.inner;
    }
    __device__ __forceinline__ void next(const FxArgs &A)
    {
        if (h == 0 && left > 1) { h = 1; return; }
        h = 0;
        if (++rt < A.rtq) return;
        rt = 0;
        left -= 2;
#pragma unroll
        for (int k = 0; k < 2; k++) {
            out[k] += dout;
            in[k] += din;
            if (in[k] >= A.inner) { in[k] -= A.inner; out[k]++; }
        }
    }
    __device__ __forceinline__ bool done() const { return left <= 0; }
    __device__ __forceinline__ int qt(const FxArgs &A) const { return A.q_fast ? (h ? in[1] : in[0]) : (h ? out[1] : out[0]); }
    __device__ __forceinline__ int tl(const FxArgs &A) const { return A.q_fast ? (h ? out[1] : out[0]) : (h ? in[1] : in[0]); }

private:
    int dout, din;
};

// Where an item lies: type, selected ell, ell, first chi node, first node,
// chi nodes, valid nodes.
struct FxPlace {
    int t, es, e, a0, q0, nodes, cnt;

    __device__ __forceinline__ FxPlace(const FxArgs &A, const int *esel, const FxItem &it)
    {
        const int tl = it.tl(A);
        t = (tl >= A.n_esel) + (tl >= 2 * A.n_esel);
        es = tl - t * A.n_esel;
        e = esel[es];
        a0 = it.qt(A) * A.apt;
        q0 = a0 * A.Rn + it.rt * A.span;
        nodes = min(A.apt, A.X - a0);
        cnt = A.apt > 1 ? nodes * A.Rn : min(A.span, A.Rn - it.rt * A.span);
    }
    __device__ __forceinline__ size_t slab(const FxArgs &A) const { return (size_t)t * A.L + e; }
};

// Sum over the R nodes of a chi node for NJ <= 5 rows (tracers of one or two
// cosmologies) by the eight lanes of a group: lane c sums r = c, c + 8, .. and
// the lanes meet in the tree (c, c + 4), (c, c + 2), (c, c + 1).  The tree
// halves the rows a lane carries at each step, so five rows cost 7 additions
// per lane, not 15.  The weights come from L2: H steps of r are multiplied
// while the next H are on their way.  The lane that ends up with a row's sum
// returns its number in `mine` (-1: none).
template <int NJ, int H>
__device__ __forceinline__ double fx_rsum(const double *const (&V)[5], const double *w, const int (&wo)[5], int len, int c,
                                          unsigned mask, int &mine)
{
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, v[2][NJ][H];
    auto load = [&](double (&x)[NJ][H], int r) {  // past the end: the last node again, not used
#pragma unroll
        for (int h = 0; h < H; h++) {
            const int at = min(c + r + 8 * h, len - 1);
#pragma unroll
            for (int j = 0; j < NJ; j++) x[j][h] = __ldg(V[j] + at);
        }
    };
    auto sum = [&](const double (&x)[NJ][H], int r) {
#pragma unroll
        for (int h = 0; h < H; h++)
            if (c + r + 8 * h < len) {
#pragma unroll
                for (int j = 0; j < NJ; j++) acc[j] = fma(x[j][h], w[wo[j] + c + r + 8 * h], acc[j]);
            }
    };
    load(v[0], 0);
    for (int r = 0; r < len; r += 16 * H) {
        load(v[1], r + 8 * H);
        sum(v[0], r);
        load(v[0], r + 16 * H);
        sum(v[1], r + 8 * H);
    }
    if constexpr (NJ == 1) {
        double s = acc[0];
        s += __shfl_xor_sync(mask, s, 4);
        s += __shfl_xor_sync(mask, s, 2);
        s += __shfl_xor_sync(mask, s, 1);
        mine = c == 0 ? 0 : -1;
        return s;
    } else {
        const bool u4 = c & 4, u2 = c & 2;
        const double k0 = (u4 ? acc[3] : acc[0]) + __shfl_xor_sync(mask, u4 ? acc[0] : acc[3], 4);
        const double k1 = (u4 ? acc[4] : acc[1]) + __shfl_xor_sync(mask, u4 ? acc[1] : acc[4], 4);
        double m0 = 0.0, m1 = 0.0;
        if constexpr (NJ > 2) {
            const double k2 = acc[2] + __shfl_xor_sync(mask, acc[2], 4);
            m1 = k2 + __shfl_xor_sync(mask, k2, 2);
            m1 += __shfl_xor_sync(mask, m1, 1);
        }
        m0 = (u2 ? k1 : k0) + __shfl_xor_sync(mask, u2 ? k0 : k1, 2);
        m0 += __shfl_xor_sync(mask, m0, 1);
        // lanes 0, 2, 4, 6 hold rows 0, 1, 3, 4 in m0; every lane holds row 2 in m1
        mine = c == 0 ? 0 : c == 2 ? 1 : c == 4 ? 3 : c == 6 ? 4 : c == 1 ? 2 : -1;
        return c == 1 ? m1 : m0;
    }
}

template <bool BAL>
__global__ void __launch_bounds__(kThreads, 1)
k_contract_fx(const __grid_constant__ CUtensorMap mapT, const FxArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    const int nk8 = (A.N + 7) / 8, nch = (nk8 + 3) / 4;  // K steps and chunks of an item
    unsigned char *sT = smem;                                   // [kT][16][span] FP64
    unsigned char *sB = sT + (size_t)A.kT * kStageBytes;        // [k-group][128 rows][16 B]
    double *sW = reinterpret_cast<double *>(sB + (size_t)nk8 * 2 * kRows * 16);  // [2][16][kWP]
    FxCtl *ctl = reinterpret_cast<FxCtl *>(sW + 2 * kNB * kWP);
    volatile int *abort_flag = &ctl->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x % A.ngr, u0 = blockIdx.x / A.ngr, ustep = gridDim.x / A.ngr;
    const int b0 = g * A.gs, nbl = min(A.gs, A.n - b0);
    const int n_units = A.nqt * 3 * A.n_esel;
    const int n_mine = u0 < n_units ? (n_units - u0 + ustep - 1) / ustep : 0, n_items = n_mine * A.rtq;
    const FxItem first(A, u0, ustep, n_mine);

    if (threadIdx.x == 0) {
        for (int i = 0; i < A.kT; i++) { mbar_init(&ctl->tfull[i], 1); mbar_init(&ctl->tempty[i], 4); }
        for (int i = 0; i < kTops; i++) { mbar_init(&ctl->efull[i], 64); mbar_init(&ctl->eempty[i], 8); }
        for (int i = 0; i < kChunks; i++) { mbar_init(&ctl->sfull[i], 4); mbar_init(&ctl->sempty[i], 1); }
        for (int i = 0; i < 2; i++) { mbar_init(&ctl->dfull[i], 1); mbar_init(&ctl->dempty[i], 128); }
        mbar_init(&ctl->mdone, 1);
        mbar_init(&ctl->never, 1);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < A.n_esel; i += blockDim.x) ctl->esel[i] = A.esel[i];
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // coefficient operand of this CTA's group, a warp per cosmology: row 16 j + b,
    // K positions 2n, 2n + 1 = digits j - 2 and j of a_b[n], times 2^8
    if (warp < kNB) {
        const int b = warp;
        const ReqDev *rq = b < nbl ? &A.reqs[b0 + b] : nullptr;
        const double *a = rq ? rq->a64 : nullptr;
        int mx = 0, down = 0;
        for (int n = lane; n < A.N; n += 32) mx = max(mx, a ? (__double2hiint(a[n]) >> 20) & 0x7ff : 0);
        for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        double up = 1.0;  // tiny coefficients are scaled up (exact) so that all have an exponent of their own
        if (mx < 400) {
            up = 0x1p400;
            down = 400;
            for (int n = lane; n < A.N; n += 32) mx = max(mx, a ? (__double2hiint(a[n] * up) >> 20) & 0x7ff : 0);
            for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (lane == 0) {
            ctl->V[b] = rq ? rq->V64 : nullptr;
            ctl->ng[b] = rq ? rq->n_clust : 0;
            ctl->ns[b] = rq ? rq->n_lens : 0;
            ctl->ea[b] = mx == 2047 ? kBad : mx - down;
        }
        const uint32_t top = fx_top(mx < 70 || mx == 2047 ? kNone : mx);
        for (int n = lane; n < nk8 * 8; n += 32) {
            const uint64_t y = fx_digits((a && n < A.N) ? a[n] * up : 0.0, top);
            uint32_t *dst = reinterpret_cast<uint32_t *>(sB + (size_t)(n >> 2) * (kRows * 16) + (n & 3) * 4);
            uint32_t d[kLev];
#pragma unroll
            for (int p = 0; p < kLev; p++)
                d[p] = __half_as_ushort(__int2half_rn(((int)((y >> (8 * (7 - p))) & 255) - 128) * 256));
#pragma unroll
            for (int j = 0; j < kLev; j++) dst[(j * kNB + b) * 4] = (d[j] << 16) | (j >= 2 ? d[j - 2] : 0u);
        }
    }
    fence_proxy_async();  // the coefficient operand is read by the MMAs
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x < 3) {
        int m = 0;
        for (int b = 0; b < nbl; b++)
            m = max(m, threadIdx.x == 0 ? ctl->ng[b] : threadIdx.x == 1 ? ctl->ns[b] : ctl->ng[b] + ctl->ns[b]);
        ctl->most[threadIdx.x] = m;
        ctl->inv[threadIdx.x] = m > 1 ? 0xffffffffu / (uint32_t)m + 1 : 0;
        if (threadIdx.x == 0) ctl->invb = nbl > 1 ? 0xffffffffu / (uint32_t)nbl + 1 : 0;
    }
    __syncthreads();
    const uint32_t tmem = ctl->tmem;

    if (warp == 0) {
        // ---------------------------------------------- TMA producer
        Ring T;
        uint32_t k = 0;
        bool ok = true;
        for (FxItem it = first; ok && !it.done(); it.next(A)) {
            const FxPlace at(A, ctl->esel, it);
            const int row = (int)at.slab(A) * A.N;
            for (int c = 0; c < nch; c++, k++, T.next(A.kT)) {
                const int st = T.st;
                const bool bad = !mbar_wait(&ctl->tempty[st], T.ph ^ 1, 32, kWaitLimit, abort_flag);
                if (__any_sync(0xffffffffu, bad)) {
                    if (lane == 0) { atomicExch(A.err, 11); *abort_flag = 1; }
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    const int nks = min(4, nk8 - 4 * c);
                    const uint32_t part = (uint32_t)A.span * 8 * 8;  // eight orders
                    mbar_expect_tx(&ctl->tfull[st], part * nks);
                    for (int ks = 0; ks < nks; ks++)
                        tma_load_2d(sT + (size_t)st * kStageBytes + ks * part, &mapT, &ctl->tfull[st], at.q0,
                                    row + c * kKC + ks * 8);
                }
                __syncwarp();
            }
        }
        for (uint32_t h = (k > (uint32_t)A.kT ? k - A.kT : 0); h < k; h++)  // every load has landed before the exit
            mbar_wait(&ctl->tfull[h % A.kT], (h / A.kT) & 1, 32);
        __syncwarp();
    } else if (warp == 1) {
        // ---------------------------------------------- MMA issuer
        const uint32_t bb = __shfl_sync(0xffffffffu, smem_u32(sB), 0);
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        Ring S;
        uint32_t uses = 0;  // bit per accumulator: parity of its uses so far
        bool ok = true;
        for (FxItem it = first; ok && !it.done(); it.next(A)) {
            const int buf = it.h;
            const uint32_t dpar = ((uses >> buf) & 1) ^ 1;
            uses ^= 1u << buf;
            for (int c = 0; c < nch; c++, S.next(kChunks)) {
                const int st = S.st;
                const bool bad = (c == 0 && !mbar_wait(&ctl->dempty[buf], dpar, 32, kWaitLimit, abort_flag)) ||
                                 !mbar_wait(&ctl->sfull[st], S.ph, 32, kWaitLimit, abort_flag);
                if (__any_sync(0xffffffffu, bad)) {
                    if (lane == 0) { atomicExch(A.err, 12); *abort_flag = 1; }
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t bd = sdesc_plain(bb + c * 8 * kRows * 16, kRows * 16);
                    const int nks = min(4, nk8 - 4 * c);
                    // digit pairs (s, s + 2), s = 0, 1, 4, 5: columns from level s on
                    for (int ks = 0; ks < nks; ks++) {
#pragma unroll
                        for (int p = 0; p < 4; p++) {
                            const int s = p < 2 ? p : p + 2;
                            const uint32_t nn = (kLev - s) * kNB;
                            const uint32_t idesc = (1u << 4) | ((nn >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
                            umma_f16_ts(tm + buf * kRows + s * kNB, tm + 2 * kRows + st * kChunkCols + p * 32 + ks * 8,
                                        bd + ((ks * 2 * kRows * 16) >> 4), idesc, (c | ks | p) != 0);
                        }
                    }
                    umma_commit(&ctl->sempty[st]);
                    if (c == nch - 1) umma_commit(&ctl->dfull[buf]);
                }
                __syncwarp();
            }
        }
        if (elect_one()) umma_commit(&ctl->mdone);  // every MMA has completed before TMEM is released
        __syncwarp();
        mbar_wait(&ctl->mdone, 0, 32);
        __syncwarp();
    } else if (warp < kEpi0) {
        // ---------------------------------------------- column exponents, a few items ahead of the slicers:
        // stepping through the items and the table's latency cost those a fifth of their time
        Ring E;
        const int q0 = (warp - 2) * 64 + lane;
        int trip = blockIdx.x == 0 ? min(A.trip, n_items - 1) : -1;  // items until the test hook's wait
        for (FxItem it = first; !it.done(); it.next(A), E.next(kTops), trip--) {
            const FxPlace at(A, ctl->esel, it);
            const uint16_t *row = A.cexp + at.slab(A) * A.Q + at.q0;
            const int m0 = row[min(q0, at.cnt - 1)], m1 = row[min(q0 + 32, at.cnt - 1)];
            const bool bad = (trip == 0 && !mbar_wait(&ctl->never, 0, 32, kTripLimit, abort_flag)) ||
                             !mbar_wait(&ctl->eempty[E.st], E.ph ^ 1, 0, kWaitLimit, abort_flag);
            if (__any_sync(0xffffffffu, bad)) {
                if (lane == 0) { atomicExch(A.err, 15); *abort_flag = 1; }
                break;
            }
            ctl->top[E.st][q0] = fx_top(m0);
            ctl->top[E.st][q0 + 32] = fx_top(m1);
            mbar_arrive(&ctl->efull[E.st]);
        }
    } else if (warp >= kSli0) {
        // ---------------------------------------------- slicers: two sets of four warps take every other chunk;
        // a thread owns one node (its TMEM lane), all orders of the chunk
        const int quad = warp & 3, q = quad * 32 + lane, set = (warp - kSli0) >> 2;
        const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + 2 * kRows;
        Ring T, S, E;
        bool ok = true;
        int mine = set;  // chunks until the next one of this set
        for (int i = 0; ok && i < n_items; i++, E.next(kTops)) {
            bool bad = !mbar_wait(&ctl->efull[E.st], E.ph, 0, kWaitLimit, abort_flag);
            const uint32_t top = ctl->top[E.st][q];
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->eempty[E.st]);
            for (int c = 0; c < nch; c++, T.next(A.kT), S.next(kChunks)) {
                if (mine--) continue;
                mine = 1;
                const int ts = T.st, ss = S.st;
                bad = bad || !mbar_wait(&ctl->tfull[ts], T.ph, 0, kWaitLimit, abort_flag) ||
                      !mbar_wait(&ctl->sempty[ss], S.ph ^ 1, 0, kWaitLimit, abort_flag);
                if (__any_sync(0xffffffffu, bad)) {
                    if (lane == 0) { atomicExch(A.err, 13); *abort_flag = 1; }
                    ok = false;
                    break;
                }
                tc_fence_after();
                const double *src = reinterpret_cast<const double *>(sT + (size_t)ts * kStageBytes) +
                                    min(q, A.span - 1);
                const int nks = min(4, nk8 - 4 * c);
#pragma unroll 1
                for (int ks = 0; ks < nks; ks++) {
                    uint32_t w[4][8];
#pragma unroll
                    for (int n = 0; n < 8; n++)
                        fx_pairs<BAL>(src[(ks * 8 + n) * A.span], top, w[0][n], w[1][n], w[2][n], w[3][n]);
#pragma unroll
                    for (int p = 0; p < 4; p++) tmem_st8(ta + ss * kChunkCols + p * 32 + ks * 8, w[p]);
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&ctl->tempty[ts]);
                    mbar_arrive(&ctl->sfull[ss]);
                }
            }
        }
    } else if (warp >= kEpi0) {
        // ---------------------------------------------- epilogue: warpgroup wg takes every other unit
        const int wg = (warp - kEpi0) >> 2, tid = (threadIdx.x - kEpi0 * 32) & 127;
        const int quad = warp & 3, q = quad * 32 + lane;  // TMEM lanes of this warp: quad 32 ..
        const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
        double *wb = sW + (size_t)wg * kNB * kWP;
        const int c = tid & 7, slot = tid >> 3;
        const unsigned mask = 0xffu << (lane & 24);
        uint32_t use = 0;
        bool dead = false;
        for (FxItem step = first; !step.done(); step.next(A)) {
            if (step.h != wg) continue;
            const FxPlace it(A, ctl->esel, step);
            const int buf = wg, rt = step.rt;
            const int mt = A.cexp[it.slab(A) * A.Q + it.q0 + min(q, it.cnt - 1)];
            if (!dead) {
                const bool bad = !mbar_wait(&ctl->dfull[buf], use & 1, 0, kWaitLimit, abort_flag);
                if (__any_sync(0xffffffffu, bad)) {
                    if (lane == 0) { atomicExch(A.err, 14); *abort_flag = 1; }
                    dead = true;
                }
            }
            use++;
            if (!dead) {
                tc_fence_after();
                const bool live = quad * 32 < it.cnt;
                for (int bq = 0; live && bq < nbl; bq += 4) {
                    uint32_t D[kLev][4];
#pragma unroll
                    for (int l = 0; l < kLev; l++) tmem_ld4(tl + buf * kRows + l * kNB + bq, D[l]);
                    tmem_wait_ld4(D[0]);
#pragma unroll
                    for (int l = 1; l < kLev; l++) reg_fence4(D[l]);
#pragma unroll
                    for (int bb = 0; bb < 4; bb++) {
                        if (bq + bb >= nbl) break;
                        int d[kLev];
#pragma unroll
                        for (int l = 0; l < kLev; l++) {
                            const float f = __uint_as_float(D[l][bb]);
                            d[l] = __float2int_rn(f + f);  // digits were scaled by 2^8 and 2^-9
                        }
                        const int ea = ctl->ea[bq + bb];
                        double w = fx_join(d, ea + mt - 994);
                        if (ea == kBad) w = __longlong_as_double(0x7ff8000000000000ll);
                        wb[(bq + bb) * kWP + q] = w;
                    }
                }
                tc_fence_before();
                mbar_arrive(&ctl->dempty[buf]);
            }
            named_bar_sync(1 + wg, 128);
            if (!dead) {
                const int len = A.apt > 1 ? A.Rn : it.cnt;
                const bool both = A.sym && it.t == 1;
                const int per = it.nodes * nbl;
                const int kind = it.t == 0 ? 0 : both ? 2 : 1, most = ctl->most[kind];
                const uint32_t inv = ctl->inv[kind], invb = ctl->invb;
                // rows (chi node, cosmology, tracer) in runs of up to five per lane group, of
                // even length: the 16 groups, and with them the four FP64 pipes, share the work
                const int rows = per * most, passes = (rows + 16 * kJC - 1) / (16 * kJC);
                const int jc = passes ? (rows + 16 * passes - 1) / (16 * passes) : 1;
                // quotients of small numbers (row < 2^16, divisors <= 32) by multiplication
                auto decode = [&](int row, int &node, int &b, int &j) {
                    const int nb = inv ? (int)__umulhi(row, inv) : row;
                    j = row - nb * most;
                    node = invb ? (int)__umulhi(nb, invb) : nb;
                    b = nb - node * nbl;
                };
                auto count = [&](int b) { return it.t == 0 ? ctl->ng[b] : both ? ctl->ng[b] + ctl->ns[b] : ctl->ns[b]; };
                auto weights = [&](int row, int &wo) {  // a row's weights and its place in w
                    int node, b, j;
                    decode(row, node, b, j);
                    wo = b * kWP + node * A.Rn;
                    return ctl->V[b] + (size_t)(j < count(b) ? (it.t == 0 || both ? j : ctl->ng[b] + j) : 0) * A.Q +
                           it.q0 + node * A.Rn;
                };
                auto put = [&](int row, double s) {
                    int node, b, j;
                    decode(row, node, b, j);
                    if (j >= count(b)) return;
                    double *y = A.Y + ((((size_t)(b0 + b) * 3 + it.t) * A.n_esel + it.es) * A.X + it.a0 + node) * A.MT + j;
                    *y = rt > 0 ? *y + s : s;
                };
                int mine;
                if (jc == 1) {
                    for (int r0 = slot; r0 < rows; r0 += 16) {
                        const double *V[5];
                        int wo[5];
                        V[0] = weights(r0, wo[0]);
                        const double s = fx_rsum<1, 8>(V, wb, wo, len, c, mask, mine);
                        if (mine == 0) put(r0, s);
                    }
                } else {
                    for (int r0 = slot * jc; r0 < rows; r0 += 16 * jc) {
                        const double *V[5];
                        int wo[5];
#pragma unroll
                        for (int k = 0; k < kJC; k++) V[k] = weights(min(r0 + k, rows - 1), wo[k]);
                        const double s = jc == 5   ? fx_rsum<5, 2>(V, wb, wo, len, c, mask, mine)
                                         : jc == 4 ? fx_rsum<4, 2>(V, wb, wo, len, c, mask, mine)
                                         : jc == 3 ? fx_rsum<3, 2>(V, wb, wo, len, c, mask, mine)
                                                   : fx_rsum<2, 4>(V, wb, wo, len, c, mask, mine);
                        if (mine >= 0 && mine < jc && r0 + mine < rows) put(r0 + mine, s);
                    }
                }
            }
            named_bar_sync(1 + wg, 128);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
    }
}

// Exponent of the largest entry of every basis column, and per (type, ell) the
// largest of those.  Entries of exponent 0 count as 1 unless they are zero.
__global__ void k_column_exp(const double *__restrict__ T, int N, int Q, uint16_t *__restrict__ cexp, int *slab)
{
    const size_t tl = blockIdx.y;
    int top = 0;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < Q; q += gridDim.x * blockDim.x) {
        const double *src = T + tl * (size_t)N * Q + q;
        int mx = 0;
        for (int n = 0; n < N; n++) {
            const double x = src[(size_t)n * Q];
            const int e = (__double2hiint(x) >> 20) & 0x7ff;
            mx = max(mx, max(e, x != 0.0 ? 1 : 0));
        }
        top = max(top, mx);
        cexp[tl * Q + q] = (uint16_t)(mx < 70 || mx == 2047 ? kNone : mx);
    }
    for (int o = 16; o; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((threadIdx.x & 31) == 0 && top) atomicMax(&slab[tl], top);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

}  // namespace

// Column exponents of the FP64 basis; p->fx_ok says whether the digits hold
// every entry that can matter: all entries finite, and no (type, ell) whose
// largest entry is under 2^-700 (columns under 2^-953 are taken as zero; a
// whole table that small keeps the CUDA-core kernel, as does a table with
// infinities or NaN, whose sums follow the rules of FP64 there), and the memory
// for the exponents (2 bytes a column beside 8 n_cheb of the table) is to be had.
int fx_prepare(blast_plan *p, cudaStream_t s)
{
    p->fx_ok = false;
    const size_t nslab = (size_t)3 * p->L;
    if (!p->colexp && cudaMalloc(&p->colexp, nslab * p->Q * sizeof(uint16_t)) != cudaSuccess) {
        cudaGetLastError();
        p->colexp = nullptr;
        return BLAST_OK;
    }
    if (!p->d_slab && cudaMalloc(&p->d_slab, nslab * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        p->d_slab = nullptr;
        return BLAST_OK;
    }
    BL_CUDA(cudaMemsetAsync(p->d_slab, 0, nslab * sizeof(int), s));
    k_column_exp<<<dim3((p->Q + 255) / 256, (unsigned)nslab), 256, 0, s>>>(p->T64, p->N, p->Q, p->colexp, p->d_slab);
    BL_CUDA(cudaGetLastError());
    std::vector<int> slab(nslab);
    BL_CUDA(cudaMemcpyAsync(slab.data(), p->d_slab, nslab * sizeof(int), cudaMemcpyDeviceToHost, s));
    BL_CUDA(cudaStreamSynchronize(s));
    p->fx_ok = true;
    for (int m : slab)
        if (m == 2047 || (m > 0 && m < 1023 - 700)) p->fx_ok = false;
    return BLAST_OK;
}

int fx_kernels(int device)
{
    BL_CUDA(allow_opt_in_smem(k_contract_fx<false>, device));
    BL_CUDA(allow_opt_in_smem(k_contract_fx<true>, device));
    return BLAST_OK;
}

int launch_contract_fx(blast_plan *p, const ReqDev *dreq, int n, const int *d_esel, int n_esel, double *Y,
                       cudaStream_t s)
{
    static const EncodeTiledFn encode = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess || q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return (EncodeTiledFn)f;
    }();
    if (!encode) return BLAST_EDEVICE;
    FxArgs A;
    A.reqs = dreq;
    A.n = n;
    A.ngr = (n + kNB - 1) / kNB;
    A.gs = (n + A.ngr - 1) / A.ngr;
    A.ngr = (n + A.gs - 1) / A.gs;
    A.L = p->L; A.N = p->N; A.Q = p->Q; A.Rn = p->Rn; A.X = p->X;
    A.n_esel = n_esel;
    A.MT = p->max_tr;
    A.sym = p->r_form == 1;
    // tiles: whole chi nodes where several fit into 128 rows, else even parts of one
    A.apt = A.Rn <= kM / 2 ? (kM / A.Rn < A.X ? kM / A.Rn : A.X) : 1;
    A.rtq = (A.Rn + kM - 1) / kM;
    A.span = A.rtq > 1 ? ((A.Rn + A.rtq - 1) / A.rtq + 7) / 8 * 8 : A.apt * A.Rn;
    A.nqt = (A.X + A.apt - 1) / A.apt;
    // one group: neighbouring CTAs read neighbouring nodes of the basis; several
    // groups: they share the weights of the same nodes in L2.  Nodes fastest and (type, ell)
    // fastest, 64 ells, 128 x 128 nodes: 4 cosmologies 0.512 / 0.537 ms, 24 1.75 / 1.70, 64
    // 4.30 / 4.09; 24 of 10+10 tracers on 256 x 192 nodes 5.65 / 4.88
    A.q_fast = A.ngr == 1;
    A.inner = A.q_fast ? A.nqt : 3 * n_esel;
    A.esel = d_esel;
    A.cexp = p->colexp;
    A.Y = Y;
    A.err = p->d_err;
    A.trip = p->test_trip;
    p->test_trip = -1;  // one call only
    const int nk8 = (A.N + 7) / 8;
    const int optin = p->smem_optin, sms = p->sms;
    const size_t fixed = 128 + (size_t)nk8 * 2 * kRows * 16 + sizeof(double) * 2 * kNB * kWP + sizeof(FxCtl);
    A.kT = (int)(((size_t)optin - fixed) / kStageBytes);
    // even, so that a slot belongs to one set of slicers: with three, a set that comes back to
    // a slot may find the phase of the other set's chunk still open and take it for its own
    A.kT = A.kT >= kMaxRing ? kMaxRing : 2;
    const size_t smem = fixed + A.kT * kStageBytes;

    CUtensorMap map;
    cuuint64_t dims[2] = {(cuuint64_t)p->Q, (cuuint64_t)3 * p->L * p->N};
    cuuint64_t strides[1] = {(cuuint64_t)p->Q * 8};
    cuuint32_t box[2] = {(cuuint32_t)A.span, 8};
    cuuint32_t es[2] = {1, 1};
    if (encode(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, p->T64, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
        blast_last_error(__FILE__, __LINE__, "cuTensorMapEncodeTiled failed");
        return BLAST_EDEVICE;
    }
    const int units = A.nqt * 3 * n_esel;
    int per = sms / A.ngr < 1 ? 1 : sms / A.ngr;  // CTAs per group
    if (per > units) per = units;
    (A.N <= kUnsigned ? k_contract_fx<false> : k_contract_fx<true>)<<<per * A.ngr, kThreads, smem, s>>>(map, A);
    BL_CUDA(cudaGetLastError());
    return BLAST_OK;
}
