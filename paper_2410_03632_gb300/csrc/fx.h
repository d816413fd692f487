// Fixed-point digits of FP64 numbers for exact products on the FP16 tensor
// cores, and the joining of the digit levels: shared by the FP64 contraction
// and the basis integrals.
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

namespace {

constexpr int kLev = 8;                  // digits per operand = level accumulators
constexpr int kNone = 2040;              // exponent of a column without usable entries: every digit 0

// Magnitude of x / 2^(M + 1 - 1023) truncated to 62 fractional bits, M the biased
// exponent of the largest entry, given as top = fx_top(M).  M = kNone gives 0.
__device__ __forceinline__ uint32_t fx_top(int M) { return ((uint32_t)M << 21) + 0x1fffffu; }

__device__ __forceinline__ uint64_t fx_mag(uint32_t hi, uint32_t lo, uint32_t top)
{
    const uint32_t sh = (top - hi - hi) >> 21;  // M - exponent: twice hi drops the sign
    const uint32_t mh = (__funnelshift_l(lo, hi, 9) & 0x1fffffffu) | 0x20000000u;  // mantissa, leading bit at 61
    uint64_t m = (uint64_t)mh << 32 | lo << 9;
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(sh));  // amounts past 63 give 0
    return m;
}

// Balanced digits of x as the bytes of the result plus 128 each, most
// significant digit in the top byte.
__device__ __forceinline__ uint64_t fx_digits(double x, uint32_t top)
{
    const uint32_t hi = __double2hiint(x), lo = __double2loint(x);
    const uint64_t s = (uint64_t)(int64_t)((int32_t)hi >> 31);
    return (fx_mag(hi, lo, top) ^ s) + (0x8080808080808080ull - s);
}

// Two bytes (0 and 2, or 1 and 3) of w as FP16 times 2^-9: a byte in the low
// half of FP16 is the subnormal y 2^-24.
__device__ __forceinline__ half2 fx_bytes(uint32_t w, uint32_t sel)
{
    const uint32_t b = __byte_perm(w, 0, sel);
    return *reinterpret_cast<const half2 *>(&b);
}
__device__ __forceinline__ uint32_t fx_word(half2 h) { return *reinterpret_cast<const uint32_t *>(&h); }

// FP16 digit pairs of a basis entry, (2, 0), (3, 1), (6, 4), (7, 5), each times
// 2^-9.  Balanced digits need four integer operations more per entry (sign and
// carry through the word) than the bytes of the magnitude with the sign put on
// by the multiply that scales them; the bytes go up to 255, which keeps the
// levels under 2^24 for n_cheb <= 76 only.
template <bool BAL>
__device__ __forceinline__ void fx_pairs(double x, uint32_t top, uint32_t &w0, uint32_t &w1, uint32_t &w2, uint32_t &w3)
{
    if constexpr (BAL) {
        const uint64_t y = fx_digits(x, top);
        const half2 m = __half2half2(__ushort_as_half(0x7800)), a = __half2half2(__ushort_as_half(0xB400));  // 2^15, -1/4
        w0 = fx_word(__hfma2(fx_bytes((uint32_t)(y >> 32), 0x4341), m, a));
        w1 = fx_word(__hfma2(fx_bytes((uint32_t)(y >> 32), 0x4240), m, a));
        w2 = fx_word(__hfma2(fx_bytes((uint32_t)y, 0x4341), m, a));
        w3 = fx_word(__hfma2(fx_bytes((uint32_t)y, 0x4240), m, a));
    } else {
        const uint32_t hi = __double2hiint(x);
        const uint64_t y = fx_mag(hi, __double2loint(x), top);
        const uint32_t mb = ((uint32_t)((int32_t)hi >> 31) & 0x80008000u) | 0x78007800u;  // +-2^15
        const half2 m = *reinterpret_cast<const half2 *>(&mb);
        w0 = fx_word(__hmul2(fx_bytes((uint32_t)(y >> 32), 0x4341), m));
        w1 = fx_word(__hmul2(fx_bytes((uint32_t)(y >> 32), 0x4240), m));
        w2 = fx_word(__hmul2(fx_bytes((uint32_t)y, 0x4341), m));
        w3 = fx_word(__hmul2(fx_bytes((uint32_t)y, 0x4240), m));
    }
}

// The FP64 number nearest to S = sum_k i[k] 256^(7-k) in the scale of the
// operands; me is the biased exponent that a sum with its leading bit at
// position 95 would have (an operand's 2^61 stands for 2^(M - 1023), and S
// counts units of 2^56: me = Ma + MT - 994).
__device__ __forceinline__ double fx_join(const int (&i)[kLev], int me)
{
    int64_t hi = (int64_t)(i[0] * 256 + i[1]) * 65536 + (i[2] * 256 + i[3]);
    const int64_t lo = (int64_t)i[4] * 16777216 + (int64_t)i[5] * 65536 + ((int64_t)i[6] * 256 + i[7]);
    hi += lo >> 32;
    // sign and magnitude h1 : h0 : l (96 bits)
    const uint32_t sg = (uint32_t)(hi >> 63);
    const uint64_t ul = (uint64_t)((uint32_t)lo ^ sg) + (sg & 1);
    const uint64_t uh = ((uint64_t)hi ^ (uint64_t)(int64_t)(int32_t)sg) + (ul >> 32);
    uint32_t h1 = (uint32_t)(uh >> 32), h0 = (uint32_t)uh, l = (uint32_t)ul;
    // leading bit to the top of h1 : h0, whole words first
    if (h1 == 0) { h1 = h0; h0 = l; l = 0; me -= 32; }
    if (h1 == 0) { h1 = h0; h0 = l; l = 0; me -= 32; }
    const int z = __clz(h1);
    const uint32_t m1 = __funnelshift_l(h0, h1, z), m0 = __funnelshift_l(l, h0, z);
    const int be = me - z;
    uint64_t bits = ((uint64_t)(m1 >> 11) << 32 | __funnelshift_r(m0, m1, 11)) + ((m0 >> 10) & 1);
    bits += (uint64_t)(uint32_t)(be - 1) << 52;
    if ((uint32_t)(be - 1) >= 2046u) bits = be <= 0 ? 0 : 0x7ff0000000000000ull;
    if (h1 == 0) bits = 0;
    return __longlong_as_double(bits | (uint64_t)(sg & 0x80000000u) << 32);
}

// K-major operand without swizzle: 8-row groups of 128 B, k-groups of 8 (16 B
// wide) kLbo bytes apart.
__device__ __forceinline__ uint64_t sdesc_plain(uint32_t saddr, uint32_t kgroup_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(kgroup_bytes >> 4) << 16;  // leading byte offset: next k-group
    d |= (uint64_t)(128 >> 4) << 32;           // stride byte offset: next eight rows
    d |= (uint64_t)1 << 46;                    // descriptor version
    return d;
}

// Position in a ring of n stages and the parity of its current lap.
struct Ring {
    int st = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next(int n)
    {
        if (++st == n) { st = 0; ph ^= 1; }
    }
};

}  // namespace
