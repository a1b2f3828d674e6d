// FP64 evaluation of F_0..F_K at one argument (the paper's Algorithm 1, Section
// II.E): the region's approximant gives F_K, then for every lane of the warp,
// whatever its region, one downward recurrence
//     F_l = (2x F_{l+1} + e^{-x}) / (2l+1)            (e^{-x} := 0 in region C).
//
//   A = [0, x_0):   F_K = r_{A,K}(x), as in the paper.
//   B = [x_0, x_1): the paper takes F_0 = r_B(x) and recurs upward; the table here
//                   holds the F_K of that recurrence, and the downward one returns
//                   the same F_{K-1}..F_0 = r_B(x).
//   C = [x_1, 2^28]: F_K = (sqrt(pi)/2) (2K-1)!!/2^K x^{-K-1/2}, which is where the
//                   paper's F_0 = (sqrt(pi)/2) x^{-1/2} and F_{l+1} = (2l+1)/(2x) F_l lead.
//   Everything else (larger x, +inf, x < 0, NaN) is rare and handled apart.
//
// What bounds it: the integer multiply pipe, which takes a 32 x 32 -> 64-bit
// product every clock and SM (and also most moves and adds), at small K; the
// stores at K = 32 (2^26 arguments of all regions: 2.68 ms, 1.02 of the measured
// copy bandwidth).  All terms of the downward step are positive: it never
// cancels, one scaling per order serves every lane, and since every lane
// produces the orders in the same sequence a warp stores whole rows as it goes
// and keeps no values back.  The step it replaced served the upward recurrence
// as well, with per-lane operands, aligned signed sums and half of the values
// held back for the row order: 59 instructions an order against 26, 4.55 ms.
// Sorting the arguments of a tile by region (one region's code per warp, rows
// staged in shared memory) was slower than either: 6.8 ms, its warps waiting for
// the ones at the region boundaries.
//
// A value depends on x and K alone, so every kernel gives the same bits.
#pragma once

#include <cstdint>
#include <type_traits>
#include <utility>

#include "boys_coeffs_fp64.h"
#include "boys_local_tables.h"
#include "boys_xf.cuh"

namespace boys {
namespace region {

using u64 = unsigned long long;

// f(0), f(1), ..., f(N-1) with the index as a type, so that everything derived
// from it is a constant in the source (an unrolled loop left the constant
// functions below to run time: 60 instructions an order instead of 26).
template <class F, int... I>
__device__ __forceinline__ void unrolled(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void unrolled(F&& f) {
    unrolled(f, std::make_integer_sequence<int, N>{});
}

// Bit patterns: for non-negative doubles the IEEE order equals the integer order,
// so the region tests run on the integer pipes.
constexpr u64 kBitsX0 = BOYS_FP64_X0_BITS;
constexpr u64 kBitsX1 = BOYS_FP64_X1_BITS;
constexpr u64 kBitsTwo28 = 0x41B0000000000000ULL;
constexpr long long kBitsInf = 0x7FF0000000000000LL;
constexpr long long kBits1e300 = 0x7E37E43C8800759CLL;

// One 64-byte entry of the expansion tables (gen_local.py).
struct __align__(16) Local {
    u64 b0, b1, b2, b3, b4;
    unsigned b5, b6, b7;
    unsigned exps;  // n (low half) and eb (high half, signed) of the state below
    u64 w;
};
static_assert(sizeof(Local) == 64, "table entries are four 16-byte words");

template <int K>
__device__ __forceinline__ const Local* local_table() {
#define BOYS_LOCAL_ROW(k) if constexpr (K == k) return reinterpret_cast<const Local*>(&g_local_##k[0][0]);
    BOYS_LOCAL_ROW(0) BOYS_LOCAL_ROW(1) BOYS_LOCAL_ROW(2) BOYS_LOCAL_ROW(3) BOYS_LOCAL_ROW(4) BOYS_LOCAL_ROW(5)
    BOYS_LOCAL_ROW(6) BOYS_LOCAL_ROW(7) BOYS_LOCAL_ROW(8) BOYS_LOCAL_ROW(9) BOYS_LOCAL_ROW(10) BOYS_LOCAL_ROW(11)
    BOYS_LOCAL_ROW(12) BOYS_LOCAL_ROW(13) BOYS_LOCAL_ROW(14) BOYS_LOCAL_ROW(15) BOYS_LOCAL_ROW(16) BOYS_LOCAL_ROW(17)
    BOYS_LOCAL_ROW(18) BOYS_LOCAL_ROW(19) BOYS_LOCAL_ROW(20) BOYS_LOCAL_ROW(21) BOYS_LOCAL_ROW(22) BOYS_LOCAL_ROW(23)
    BOYS_LOCAL_ROW(24) BOYS_LOCAL_ROW(25) BOYS_LOCAL_ROW(26) BOYS_LOCAL_ROW(27) BOYS_LOCAL_ROW(28) BOYS_LOCAL_ROW(29)
    BOYS_LOCAL_ROW(30) BOYS_LOCAL_ROW(31) BOYS_LOCAL_ROW(32)
#undef BOYS_LOCAL_ROW
}

// e^{t/16} on [0, 1]: Q63 (the last three terms, literals, are Q58).  In constant
// memory the products take them as operands; as 64-bit literals each costs two moves.
static __constant__ u64 c_exp[5] = {BOYS_LOCAL_EXP_C0, BOYS_LOCAL_EXP_C1, BOYS_LOCAL_EXP_C2, BOYS_LOCAL_EXP_C3,
                                    BOYS_LOCAL_EXP_C4};

// add + the high half of a b from three partial products, as xf::mulhi3 (at most
// 2 below the exact high half).  The 32-bit halves are added with the carry flag: plain
// 64-bit adds go to the multiply pipe, at the price of a product each (K = 4, 2^25
// arguments: 351 us; halves first 356; as 64-bit adds K = 8 3% slower).
__device__ __forceinline__ u64 mulhi(u64 a, u64 b, u64 add = 0) {
    const unsigned a0 = (unsigned)a, a1 = (unsigned)(a >> 32), b0 = (unsigned)b, b1 = (unsigned)(b >> 32);
    const u64 p = (u64)a1 * b1 + add;
    unsigned lo = (unsigned)p, hi = (unsigned)(p >> 32);
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;\n\tadd.cc.u32 %0, %0, %3;\n\taddc.u32 %1, %1, 0;"
        : "+r"(lo), "+r"(hi)
        : "r"(__umulhi(a1, b0)), "r"(__umulhi(a0, b1)));
    return (u64)hi << 32 | lo;
}

// The same where the two halves sum to less than 2^32.
__device__ __forceinline__ u64 mulhi_nocarry(u64 a, u64 b) {
    const unsigned a0 = (unsigned)a, a1 = (unsigned)(a >> 32), b0 = (unsigned)b, b1 = (unsigned)(b >> 32);
    unsigned s = __umulhi(a1, b0);
    asm("mad.hi.u32 %0, %1, %2, %0;" : "+r"(s) : "r"(a0), "r"(b1));
    return (u64)a1 * b1 + s;
}

__host__ __device__ constexpr int ilog2(int v) { return v < 2 ? 0 : 1 + ilog2(v >> 1); }
// floor(2^(63 + s) / (2l+1)), s = ilog2(2l+1), l >= 1, by long division on 32-bit halves
__host__ __device__ constexpr u64 kappa(int l) {
    const u64 d = 2 * l + 1, top = 1ULL << (31 + ilog2(2 * l + 1));
    return ((top / d) << 32) + ((top % d) << 32) / d;
}

// T kappa_l / 2^64 for T < 0.56 2^64 (the recurrence's sums, see eval_regular).
template <int L>
__device__ __forceinline__ u64 times_kappa(u64 T) {
    constexpr u64 k = kappa(L);
    if constexpr (0.57 * (double)(k & 0xFFFFFFFF) + (double)(k >> 32) < 4294967295.0) return mulhi_nocarry(T, k);
    else return mulhi(T, k);
}

// The state of the recurrence.  F_l = y 2^-62 2^(f+1-1023) with f = eb + n and y in
// [2^62, 2^63): f is the exponent field of F_l less the hidden bit.
struct State {
    u64 y, X, Em;  // X = x 2^(59-q) (q = 0 below 32), Em = e^{-x} in its own scale (0 in C)
    int n, eb, q;  // Em >> n is e^{-x} in the scale of the next sum
};

// (hi : lo) >> n, its low word, n <= 32
__device__ __forceinline__ unsigned shift_right(unsigned lo, unsigned hi, unsigned n) {
    unsigned r;
    asm("shf.r.clamp.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(n));
    return r;
}

// 2^32 <= y < 2^63 moved up to [2^62, 2^63), its exponent along (C: what it gains
// on the way), and its value as a double (truncated).
template <int C>
__device__ __forceinline__ double normalise(State& S) {
    const unsigned lo = (unsigned)S.y, hi = (unsigned)(S.y >> 32);
    int b;  // leading bit of the high word, to become bit 30
    asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(hi));
    const unsigned h = shift_right(lo, hi, b + 2), l = shift_right(0, lo, b + 2);
    S.y = (u64)h << 32 | l;
    S.n += b + (C - 30);
    return __hiloint2double((int)((h >> 10) + ((unsigned)(S.n + S.eb) << 20)), (int)shift_right(l, h, 10));
}

// The state at order K for 0 <= x <= 2^28 (bit pattern xb): the anchor and e^{-x}
// from one table entry, seven and eight products (the last terms in 32 bits)
// and the same instructions in every region.  Rationals evaluated at x, with their
// inverse square root, the exponential and region C's inverse square root took
// about thirty products and the selects of their operands (K = 0, 2^24
// arguments: 275 us against 84).
template <int K>
__device__ __forceinline__ State start(u64 xb, const Local* __restrict__ tab) {
    constexpr int kBitsC = K <= 12 ? 9 : 10;  // index bits of region C: one for the factor of two, log2 of its intervals
    const bool inC = xb >= kBitsX1;
    const u64 m = (xb << 11) | 0x8000000000000000ULL;
    const int be = (int)(xb >> 52);
    State S;
    S.X = xf::shr_u64(m, max(1027 - be, 0));  // x 2^59 below 32 (0 below 2^-59), the significand above
    S.q = max(be - 1027, 0);
    // Index and variable: the leading bits of x 2^59 in A and B; in C those of the
    // significand under the exponent's parity, x = M 4^h.
    unsigned vh = (unsigned)(S.X >> 32);
    if (inC) vh &= 0x7FFFFFFFu | ((unsigned)be << 31);
    const u64 v = (u64)vh << 32 | (unsigned)S.X;
    const int bits = inC ? kBitsC : 9;
    const int h = inC ? (be - 1023) >> 1 : 0;
    const int first = inC ? BOYS_LOCAL_FIRST_C : xb >= kBitsX0 ? 1 : 0;
    const Local* __restrict__ e = tab + (first + (int)(vh >> (32 - bits)));
    const u64 t = ~(v << bits);
    const unsigned t32 = (unsigned)(t >> 32);
    const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(&e->b0);
    const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(&e->b2);
    const ulonglong2 w2 = *reinterpret_cast<const ulonglong2*>(&e->b4);
    const ulonglong2 w3 = *reinterpret_cast<const ulonglong2*>(&e->b7);
    const unsigned u5 = (unsigned)w2.y + __umulhi(t32, (unsigned)(w2.y >> 32) + __umulhi(t32, (unsigned)w3.x));
    u64 y = w2.x + ((u64)__umulhi(t32, u5) << 5);
    y = mulhi(t, y, w1.y);
    y = mulhi(t, y, w1.x);
    y = mulhi(t, y, w0.y);
    S.y = mulhi(t, y, w0.x);
    S.n = (int)((w3.x >> 32) & 0xFFFF) - h * (2 * K + 1);
    S.eb = (int)((long long)w3.x >> 48);
    S.Em = 0;
    if (K > 0) {
        const unsigned e5 = (unsigned)BOYS_LOCAL_EXP_C5 +
                            __umulhi(t32, (unsigned)BOYS_LOCAL_EXP_C6 + __umulhi(t32, (unsigned)BOYS_LOCAL_EXP_C7));
        u64 E = c_exp[4] + ((u64)__umulhi(t32, e5) << 5);
        E = mulhi(t, E, c_exp[3]);
        E = mulhi(t, E, c_exp[2]);
        E = mulhi(t, E, c_exp[1]);
        E = mulhi(t, E, c_exp[0]);
        S.Em = mulhi(w3.y, E);
    }
    return S;
}

// e^{-x} of a state as a double (0 in region C).
__device__ __forceinline__ double exponential(const State& S) {
    const int b = 31 - __clz((int)(S.Em >> 32));
    const u64 m = S.Em >> ((b - 20) & 63);
    const double e = __hiloint2double((int)((unsigned)(m >> 32) + ((unsigned)(S.eb + b - 24) << 20)), (int)(unsigned)m);
    return S.Em == 0 ? 0.0 : e;
}

// x and -0.0 as 0; whether its bit pattern is one that start() takes, 0 <= x <= 2^28.
// (The test for -0.0 by halves: as one 64-bit comparison it becomes an FP64 one.)
__device__ __forceinline__ u64 bits_of(double x) {
    const unsigned lo = (unsigned)__double2loint(x), hi = (unsigned)__double2hiint(x);
    const unsigned h = (lo | (hi ^ 0x80000000u)) == 0 ? 0 : hi;
    return (u64)h << 32 | lo;
}
__device__ __forceinline__ bool regular(u64 xb) { return xb <= kBitsTwo28; }  // negative numbers and NaN lie above

// Large, infinite and invalid arguments: rare, so a rolled loop, upward: to
// out(k, value) with a run-time k.  F_k below the normal range becomes subnormal (every
// order alike: the former FP64 steps gave these values, the integer ones 0), +inf gives
// 0, an invalid argument NaN.
template <class Out>
__device__ __forceinline__ void eval_other(int K, double x, Out&& out) {
    const long long xb = __double_as_longlong(x);
    const bool valid = xb >= 0 && xb <= kBitsInf;
    const xf::Xf r = xf::rsqrt(xf::from_double(!valid || xb > kBits1e300 ? 1e300 : x));
    xf::Xf y = xb == kBitsInf ? xf::zero() : xf::mul(xf::sqrt_pi_over_2(), r);
    const xf::Xf R = xf::mul(xf::Xf{r.m, r.e - 1}, r);
#pragma unroll 1
    for (int j = 0; j <= K; ++j) {
        out(j, valid ? xf::to_double_gradual(y) : __longlong_as_double(0x7FF8000000000000LL));
        y = xf::mul_norm(xf::mul_raw(xf::odd(j), y), R);
    }
}
// Stores the orders of one argument: column `col` of rows `ld` apart.  The
// address moves down a row at a time (addresses formed as col + k ld were all
// kept in registers), with the carry flag (see mulhi; K = 16: 795 to 750 us for
// 2^25 arguments).
struct Column {
    double* row;
    int64_t ld;
    template <int K>
    static __device__ __forceinline__ Column of(double* col, int64_t ld) { return Column{col + K * ld, ld}; }
    template <int L>
    __device__ __forceinline__ void operator()(std::integral_constant<int, L>, double v) {
        __stcs(row, v);
        const u64 r = (u64)row, d = (u64)ld * (u64)-8;
        unsigned lo = (unsigned)r, hi = (unsigned)(r >> 32);
        asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;"
            : "+r"(lo), "+r"(hi)
            : "r"((unsigned)d), "r"((unsigned)(d >> 32)));
        row = (double*)((u64)hi << 32 | lo);
    }
};

// Recurrence steps in FP64, the first ones: two instructions and a ready value
// for 26 on the integer pipes, but at 2 a clock and SM.  Swept on GB300 (2^25
// arguments, us): about a quarter of the orders, rounded up, to K = 16 (K = 7: 430
// with 2, 455 with 1; K = 10: 518 with 3, 541 with 2; K = 13: 619 with 4, 627 with 3;
// K = 16: 731 with 4, 738 with 3, 734 with 5), a fifth above, where the stores take
// over (K = 24: 1038 with 4, 1044 with 6; K = 32, 2^26: 2692 with 6, 2698 with 8).
// None below K = 6: one would give 1 % at K = 4 (347 for 352), and the results there
// are those of the exact integer arithmetic to the last bit.
constexpr int fp64_steps(int K) { return K < 6 ? 0 : K <= 16 ? (K + 3) / 4 : K < 20 ? 4 : K / 5; }

// F_K, F_{K-1}, ..., F_LAST at a regular x, to out(integral_constant k, value);
// `tab` is the order's table.
//
// A step, with u the scale of y: T = X y / 2^64 + (Em >> n) is (2l+1) F_l 2^(u-6), its
// second term free in the product's accumulator, and y = T kappa_l / 2^64.  T / 2^64 is
// below (2x + e^{-x} / F_{l+1}) / 128, at most 0.556 in A and B (l = 31, x -> x_1), and
// below a half in C; it is above 2^56.  A value of the integer steps is within 2^-53
// of itself before it is cut to a double (the tests' integer model: 2^-53.6 at most,
// order 0 of K = 31 just above x = 32); an FP64 step adds two roundings of 2^-53.
template <int K, int NF = fp64_steps(K), int LAST = 0, class Out>
__device__ __forceinline__ void eval_regular(u64 xb, const Local* __restrict__ tab, Out&& out) {
    const double x = __longlong_as_double((long long)xb);
    State S = start<K>(xb, tab);
    double yd = normalise<0>(S);
    out(std::integral_constant<int, K>{}, yd);
    if constexpr (NF > 0) {
        const double two_x = x + x, e = exponential(S);
        unrolled<NF>([&](auto p) {
            constexpr int l = K - 1 - decltype(p)::value;
            yd = fma(two_x, yd, e) * (1.0 / (2 * l + 1));
            out(std::integral_constant<int, l>{}, yd);
        });
        const u64 yb = (u64)__double_as_longlong(yd);
        S.y = ((yb & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL) << 10;
        S.n = (int)(yb >> 52) - 1 - S.eb;
    }
    unrolled<K - NF - LAST>([&](auto p) {
        constexpr int l = K - 1 - NF - decltype(p)::value;
        const u64 T = mulhi(S.X, S.y, xf::shr_u64(S.Em, S.n));
        S.n += S.q;
        if constexpr (l == 0) {
            S.y = T;  // below 2^63
            out(std::integral_constant<int, 0>{}, normalise<6>(S));
        } else {
            S.y = times_kappa<l>(T);
            constexpr int gain = 7 - ilog2(2 * l + 1);
            out(std::integral_constant<int, l>{}, normalise<gain>(S));
        }
    });
}

static __device__ __noinline__ void store_other(int K, double x, double* col, int64_t ld) {
    eval_other(K, x, [col, ld](int k, double v) { col[k * ld] = v; });
}

// All orders of one argument, to column `col` of rows `ld` apart.  A kernel of many
// orders keeps one copy of the loop for irregular arguments (kShared), out of line.
template <int K, bool kShared = false>
__device__ __forceinline__ void eval_store(double x, double* col, int64_t ld) {
    const u64 xb = bits_of(x);
    if (regular(xb)) {
        eval_regular<K>(xb, local_table<K>(), Column::of<K>(col, ld));
    } else if (kShared) {
        store_other(K, x, col, ld);
    } else {
        eval_other(K, x, [col, ld](int k, double v) { col[k * ld] = v; });
    }
}

}  // namespace region
}  // namespace boys
