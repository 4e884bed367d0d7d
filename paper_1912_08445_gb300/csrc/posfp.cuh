// Arithmetic on non-negative numbers with 64-bit significands on the integer pipe.
//
// GB300 issues one warp-wide FP64 instruction per SM sub-partition about every 80 cycles
// (measured: 0.50 T DFMA/s on 152 SMs), so a double-precision operation costs as much as
// 80 integer or FP32 instructions. The transfer sweep works on non-negative quantities
// only: without signs and cancellation a multiplication is one 64-bit high product and a
// normalisation by at most two bits (about 15 instructions). Significands keep 64
// bits, 11 more than a double, and results are rounded once when they are packed.
//
// - 2^(-t) is table driven (Tang 1989: a table of 2^(-i/256) and a short polynomial), in
//   fixed point: the error is below 2^-58 of the result, against 2^-53 of a rounded
//   double.
// - The reciprocal is Newton's iteration y <- y + y (1 - D y) from a single-precision
//   reciprocal (24 -> 46 -> 62 bits).
#pragma once
#include <cstdint>

namespace mg {

// High 64 bits of a product, short of it by at most two units (the low halves' product is
// left out: three 32-bit multiplications instead of four and no carries).
__device__ __forceinline__ uint64_t mulhi_near(uint64_t a, uint64_t b) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}

// A number m 2^e >= 0: m has its top bit set, or is 0.
struct PosFp {
    uint64_t m;
    int e;
};

// From the magnitude of a double (subnormals count as zero, whose exponent is below every other;
// infinities and NaN as numbers of 2^1024 and more: callers that can meet them ask `not_finite`).
__device__ __forceinline__ PosFp pos_from(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    if (ex == 0) return PosFp{0, -(1 << 20)};
    return PosFp{((b << 11) | 0x8000000000000000ull), ex - 1086};   // 1086 = 1023 + 63
}

// (a constant: FP64 instructions under a predicate cost as much as executed ones)
__device__ __forceinline__ double nan64() { return __longlong_as_double(0x7ff8000000000000ll); }
__device__ __forceinline__ bool not_finite(double x) { return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000; }

// m 2^e rounded to a double; m may have up to two leading zero bits. Below the smallest
// normal double the result is 0, beyond the largest it is infinity.
__device__ __forceinline__ double pos_pack(uint64_t m, int e) {
    const int z = (m >> 63) ? 0 : ((m >> 62) & 1 ? 1 : 2);
    m <<= z;
    const int E = e - z + 1086;
    // the rounded significand carries its leading bit (and a carry) into the exponent
    const uint64_t r = (m >> 11) + ((m >> 10) & 1);
    uint64_t b = ((uint64_t)(uint32_t)(E - 1) << 52) + r;
    if (E >= 0x7ff) b = 0x7ff0000000000000ull;
    if (E < 1 || !(m >> 63)) b = 0;
    return __longlong_as_double((long long)b);
}
__device__ __forceinline__ double pos_pack(const PosFp &a) { return pos_pack(a.m, a.e); }

__device__ __forceinline__ PosFp pos_mul(const PosFp &a, const PosFp &b) {
    uint64_t h = mulhi_near(a.m, b.m);
    int e = a.e + b.e + 64;
    if (!(h >> 63)) {
        h <<= 1;
        e--;
    }
    return PosFp{h, e};
}

// a + b. Both normalised; a zero has m = 0 and an exponent below every other.
__device__ __forceinline__ PosFp pos_add(const PosFp &a, const PosFp &b) {
    const bool sw = a.e < b.e;
    const uint64_t hm = sw ? b.m : a.m, lm = sw ? a.m : b.m;
    const int he = sw ? b.e : a.e, d = sw ? b.e - a.e : a.e - b.e;
    uint64_t m = hm + (d < 64 ? lm >> d : 0);
    const bool carry = m < hm;
    m = carry ? (m >> 1) | 0x8000000000000000ull : m;
    return PosFp{m, he + (carry ? 1 : 0)};
}

// Normalised from a significand with up to two leading zero bits.
__device__ __forceinline__ PosFp pos_norm(uint64_t m, int e) {
    const int z = (m >> 63) ? 0 : ((m >> 62) & 1 ? 1 : 2);
    return PosFp{m << z, e - z};
}

// 1/a, a > 0.
__device__ __forceinline__ PosFp pos_rcp(const PosFp &a) {
    const float d = (float)(uint32_t)(a.m >> 40);            // D 2^24, exact; D = m/2^64 in [1/2, 1)
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    // y = 1/D in units of 2^-62, in (1, 2]: 1/D = r 2^24, so y 2^62 = r 2^86
    const uint32_t rb = __float_as_uint(r);
    uint64_t y = (uint64_t)((rb & 0x7fffffu) | 0x800000u) << ((int)(rb >> 23) - 127 - 23 + 86);
#pragma unroll
    for (int it = 0; it < 2; it++) {
        const int64_t err = (int64_t)((1ull << 62) - mulhi_near(a.m, y));   // (1 - D y) 2^62
        y += (uint64_t)__mul64hi((int64_t)(y >> 1), err << 3);
    }
    // 1/a = (1/D) 2^(-64 - e) = y 2^(-62 - 64 - e)
    PosFp q{y, -126 - a.e};
    if (!(q.m >> 63)) {
        q.m <<= 1;
        q.e--;
    }
    return q;
}

// ---------------------------------------------------------------- 2^(-t)
// 2^(-2^-k), k = 1 .. 8, in units of 2^-64.
constexpr uint64_t kExp2Half[8] = {
    0xb504f333f9de6484ull,
    0xd744fccad69d6af4ull,
    0xeac0c6e7dd24392eull,
    0xf5257d152486cc2cull,
    0xfa83b2db722a033aull,
    0xfd3e0c0cf486c174ull,
    0xfe9e115c7b8f884bull,
    0xff4ecb59511ec8a5ull};

struct Exp2Table {
    uint64_t t[256];   // 2^(-i/256) in units of 2^-63
};
constexpr uint64_t mulhi_u64(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
constexpr Exp2Table make_exp2_table() {
    Exp2Table T{};
    T.t[0] = 1ull << 63;
    for (int i = 1; i < 256; i++) {
        uint64_t p = 0;
        for (int k = 0; k < 8; k++)
            if (i & (128 >> k)) p = p ? mulhi_u64(p, kExp2Half[k]) : kExp2Half[k];
        T.t[i] = p >> 1;
    }
    return T;
}
__device__ constexpr Exp2Table kExp2Table = make_exp2_table();

// c_k = ln(2)^k / k!: c1, c2 in units of 2^-64, c3 .. c5 in units of 2^-32
constexpr uint64_t kExpC1 = 0xb17217f7d1cf79abull;
constexpr uint64_t kExpC2 = 0x3d7f7bff058b1d50ull;
constexpr uint32_t kExpC3 = 0x0e35846bu;
constexpr uint32_t kExpC4 = 0x0276556du;
constexpr uint32_t kExpC5 = 0x005761ffu;

// sqrt(log2 e) and log2 e in units of 2^-63
constexpr uint64_t kSqrtLog2eFix = 0x99be610c1d827eefull, kLog2eFix = 0xb8aa3b295c17f0bbull;

// 2^(-f 2^-64) in units of 2^-63, in [2^62, 2^63] (t: the table in shared memory).
__device__ __forceinline__ uint64_t exp2_neg_frac(uint64_t f, const uint64_t *t) {
    const uint64_t T = t[f >> 56];
    const uint64_t r = f << 8;                                // remainder / 2^-8, in units of 2^-64
    const uint32_t r32 = (uint32_t)(r >> 32);
    // 2^(-r') = 1 - r' (c1 - r' (c2 - r' (c3 - r' (c4 - r' c5)))), c_k = ln(2)^k / k!,
    // r' = r 2^-8; the inner terms need 32 bits only
    const uint32_t a4 = kExpC4 - (__umulhi(kExpC5, r32) >> 8);
    const uint32_t a3 = kExpC3 - (__umulhi(a4, r32) >> 8);
    const uint64_t a2 = kExpC2 - (((uint64_t)a3 * (uint32_t)(r >> 32) + (((uint64_t)a3 * (uint32_t)r) >> 32)) >> 8);
    const uint64_t a1 = kExpC1 - (mulhi_near(a2, r) >> 8);
    const uint64_t d = mulhi_near(a1, r) >> 8;                // 1 - 2^(-r'), in units of 2^-64
    const uint64_t s = T - mulhi_near(T, d);
    return s < (1ull << 62) ? (1ull << 62) : s;               // (one unit below 1/2 by truncation)
}

// Significand (in units of 2^-63, in [2^62, 2^63]) and integer exponent n of
// exp(-x^2) = sig 2^(-n), for |x| < 53. The factor sqrt(log2 e) is applied in fixed point:
// folded into a double-precision x it would carry a rounding that is the same at every point.
__device__ __forceinline__ uint64_t exp_neg_sq(double x, const uint64_t *t, int &n) {
    // U = sqrt(log2 e) |x| 2^57
    const uint64_t b = (uint64_t)__double_as_longlong(x) & 0x7fffffffffffffffull;
    const int sh = (int)(b >> 52) - 1023 + 5;                 // exponent + 57 - 52
    const uint64_t mant = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
    const uint64_t U = mulhi_near(sh >= 0 ? mant << sh : (sh > -64 ? mant >> -sh : 0), kSqrtLog2eFix) << 1;
    // U^2 = log2(e) x^2 2^114: integer part, fraction of 64 bits
    const uint32_t ua = (uint32_t)(U >> 32), ub = (uint32_t)U;
    const uint64_t mid = 2 * ((uint64_t)ua * ub) + __umulhi(ub, ub);   // (below 2^64: U < 2^63)
    const uint64_t hi = (uint64_t)ua * ua + (mid >> 32);
    n = (int)(hi >> 50);
    return exp2_neg_frac((hi << 14) | ((uint32_t)mid >> 18), t);
}

// The same for exp(-d), 0 <= d < 2^12, d as significand and exponent.
__device__ __forceinline__ uint64_t exp_neg(const PosFp &d, const uint64_t *t, int &n) {
    // log2(e) d = m 2^(e + 1): m in units of 2^(e + 1) = 2^-k
    const uint64_t m = mulhi_near(d.m, kLog2eFix);
    const int k = -(d.e + 1);                                 // 52 .. (d < 2^12)
    n = k >= 64 ? 0 : (int)(m >> k);
    const uint64_t f = k >= 64 ? (k - 64 < 64 ? m >> (k - 64) : 0) : m << (64 - k);
    return exp2_neg_frac(f, t);
}

}  // namespace mg
