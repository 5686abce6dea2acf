// FP64 exponentials on the integer pipe.
//
// GB300 does 1.9 FP64 operations per clock and SM against 116 FP32 or integer
// ones (26 32 x 32 -> 64-bit multiplies), so CUDA's exp(double), about 20 FP64
// operations, takes the time of 1,400 integer operations.  Here the exponent is
// a 64-bit fixed-point number and the FP64 pipe does nothing: Tang's
// table-driven method (P. T. P. Tang, ACM TOMS 15 (1989) 144) in fixed point,
//   2^-t = 2^-n T[j] 2^-r,  t = n + j / 1024 + r,  0 <= r < 2^-10,
//   2^-r = 1 - q,  q = r (L - r (L^2/2 - r (L^3/6 - r L^4/24))),  L = ln 2,
// with T[j] = 2^(-j/1024) to 64 bits from shared memory, the last product of
// q and the product with T in 64 bits, the inner ones in 32 bits (they are
// scaled by 2^-10 each).  About 95 integer operations; 14 times the rate of
// exp(double).  Relative error below 0.9 2^-53 for a given t (20,000 random t
// against 160-bit arithmetic, mean -0.18 2^-53), below 2.2 2^-53 for
// exp_fix(x), where t is x log2(e) to 2^-54.
#pragma once

#include <cstdint>

constexpr int EXPFIX_N = 1024;   // table entries (8 KB of shared memory)

struct ExpFixTable { uint64_t v[EXPFIX_N]; };

namespace expfix_detail {
// floor(a b / 2^64)
constexpr uint64_t mulhi(uint64_t a, uint64_t b) {
    const uint64_t al = a & 0xffffffffu, ah = a >> 32, bl = b & 0xffffffffu, bh = b >> 32;
    const uint64_t m1 = ah * bl, m2 = al * bh, ll = al * bl;
    const uint64_t c = ((ll >> 32) + (m1 & 0xffffffffu) + (m2 & 0xffffffffu)) >> 32;
    return ah * bh + (m1 >> 32) + (m2 >> 32) + c;
}
// floor(sqrt(x 2^64)) for x in [2^62, 2^64): bit by bit
constexpr uint64_t sqrt_frac(uint64_t x) {
    uint64_t r = 0;
    for (int b = 63; b >= 0; --b) {
        const uint64_t t = r | (uint64_t(1) << b);
        // t^2 <= x 2^64: high word below x, or equal to it with a zero low word
        const uint64_t hi = mulhi(t, t), lo = t * t;
        if (hi < x || (hi == x && lo == 0)) r = t;
    }
    return r;
}
constexpr ExpFixTable make_table() {
    ExpFixTable t{};
    uint64_t root[10] = {};
    uint64_t x = uint64_t(1) << 63;   // 2^-1, then its square roots 2^-1/2, 2^-1/4, ...
    for (int k = 0; k < 10; ++k) { x = sqrt_frac(x); root[k] = x; }
    t.v[0] = ~uint64_t(0);
    for (int j = 1; j < EXPFIX_N; ++j) {
        uint64_t v = 0;
        for (int k = 0; k < 10; ++k)
            if ((j >> (9 - k)) & 1) v = v == 0 ? root[k] : mulhi(v, root[k]);
        t.v[j] = v;
    }
    return t;
}
}  // namespace expfix_detail

#ifdef __CUDACC__

// one copy a translation unit
static __device__ const ExpFixTable d_expfix_table = expfix_detail::make_table();

// The block's copy of the table; a __syncthreads() must follow.
__device__ __forceinline__ void expfix_load(uint64_t* tab) {
    for (int i = threadIdx.x; i < EXPFIX_N; i += blockDim.x) tab[i] = d_expfix_table.v[i];
}

// 2^-(frac / 2^64) in units of 2^-64, in [2^63, 2^64).
__device__ __forceinline__ uint64_t expfix_frac(uint64_t frac, const uint64_t* tab) {
    const uint64_t T = tab[(uint32_t)(frac >> 54)];
    const uint64_t R = frac << 10;
    const uint32_t rho = (uint32_t)(R >> 32);
    const uint32_t k3 = 0xe35846b8u - (__umulhi(0x276556dfu, rho) >> 10);   // 16 L^3/6, 16 L^4/24
    const uint32_t h = 0xf5fdeffcu - (__umulhi(k3, rho) >> 12);             // 4 L^2/2
    const uint64_t G = 0xb17217f7d1cf79acull - ((uint64_t)__umulhi(h, rho) << 20);
    const uint64_t q = __umul64hi(R, G) >> 10;
    const uint64_t v = T - __umul64hi(T, q);
    return v | (uint64_t(1) << 63);   // a value a rounding below 2^63 stays in range
}

// v 2^(-64 - n) as a double, for |n| <= 1000.
__device__ __forceinline__ double expfix_double(uint64_t v, int n) {
    const uint64_t m = (v >> 11) + ((v >> 10) & 1);   // 53 bits, rounded (2^53 carries into the exponent)
    return __longlong_as_double((long long)(((uint64_t)(uint32_t)(1021 - n) << 52) + m));
}

// log2(e) 2^63
constexpr uint64_t EXPFIX_LOG2E = 0xb8aa3b295c17f0bcull;

// out of line: the rare path's FP64 operations stay out of the callers' loops
static __device__ __noinline__ double expfix_slow(double x) { return exp(x); }
// e^x for any x: the fixed-point form for |x| < 690, exp(x) otherwise.
__device__ __forceinline__ double exp_fix(double x, const uint64_t* tab) {
    const uint64_t bits = (uint64_t)__double_as_longlong(x);
    const int ex = (int)(bits >> 52) & 0x7ff;
    const int hi = __double2hiint(x) & 0x7fffffff;
    if (hi >= 0x40859000) return expfix_slow(x);   // |x| >= 690, inf or NaN
    const uint64_t B = ((bits << 11) | (uint64_t(1) << 63));   // |x| = B 2^(ex - 1086)
    const uint64_t P = __umul64hi(B, EXPFIX_LOG2E);            // |x| log2(e) = P 2^(ex - 1085)
    const int sh = 1032 - ex;                                   // to 53 fraction bits; > 0 for |x| < 2^9.. 690
    int64_t t = 0;
    if (sh <= 63) t = sh > 0 ? (int64_t)((P >> sh) + ((P >> (sh - 1)) & 1)) : (int64_t)(P << -sh);
    if ((int64_t)bits >= 0) t = -t;   // 2^-t
    return expfix_double(expfix_frac((uint64_t)t << 11, tab), (int)(t >> 53));
}

// e^{-b E} for many E >= 0 and a few b > 0 (Boltzmann factors, b = c2 / T):
// E as 64-bit fixed point with 44 fraction bits, b log2(e) as a normalised
// 64-bit mantissa, t their product.  For b < 2^-10 (T above 1,473 K) E's last
// bit is worth b 2^-45 < 2^-55 of the result and t's less than 0.7 2^-53, so
// the error is below 1.8 2^-53 for any E, while the rounding of a double b E
// alone is b E 2^-53 or less.  With a larger b the fixed point would hold
// less than a double (b 2^-45: 1e-14 at 3 K), and the product is formed in
// FP64: exp_fix(-b E).
constexpr uint64_t EXPFIX_BAD = ~uint64_t(0);
// E in [0, 2^20) in units of 2^-44, else EXPFIX_BAD
__device__ __forceinline__ uint64_t expfix_energy(double E) {
    const uint64_t bits = (uint64_t)__double_as_longlong(E);
    const int sh = (int)(bits >> 52) - 1031;   // the sign bit makes it large
    const uint64_t m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
    if (sh > 11) return EXPFIX_BAD;
    if (sh >= 0) return m << sh;
    return sh < -54 ? 0 : (m + (uint64_t(1) << (-sh - 1))) >> -sh;
}
struct ExpFixScale {
    uint64_t m;   // b log2(e) = m 2^(-64 - (F - 44))
    int F;        // fraction bits of the products; 0: b outside (2^-1022, 2^-10), exp_fix(-b E)
};
__device__ __forceinline__ ExpFixScale expfix_scale(double b) {
    ExpFixScale r;
    r.m = 0; r.F = 0;
    const uint64_t bits = (uint64_t)__double_as_longlong(b);
    const int ex = (int)(bits >> 52);
    if (ex == 0 || ex >= 1013) return r;   // zero, negative, inf, NaN or 2^-10 and above
    uint64_t m = __umul64hi((bits << 11) | (uint64_t(1) << 63), EXPFIX_LOG2E);
    int e = ex;
    if (!(m >> 63)) { m <<= 1; --e; }     // b log2(e) = m 2^(e - 1085)
    int s = 1021 - e;                     // 9 or more
    if (s > 19) { m = s - 19 < 64 ? m >> (s - 19) : 0; s = 19; }
    r.m = m;
    r.F = 44 + s;
    return r;
}
// (out of line, so that its product is not formed ahead of the test: an FP64
// operation a term)
static __device__ __noinline__ double expfix_far(double E, double b, const uint64_t* tab) {
    return exp_fix(-b * E, tab);
}
// e^{-b E}: Ef from expfix_energy(E), sc from expfix_scale(b)
__device__ __forceinline__ double expfix_boltzmann(uint64_t Ef, const ExpFixScale& sc, double E, double b,
                                                   const uint64_t* tab) {
    const uint64_t P = __umul64hi(Ef, sc.m);
    const int n = (int)(P >> sc.F);
    if (sc.F == 0 || Ef == EXPFIX_BAD || (P >> sc.F) > 1000) return expfix_far(E, b, tab);
    return expfix_double(expfix_frac(P << (64 - sc.F), tab), n);
}

#endif
