// The paper's benchmark workload (Section III, Algorithm 2):
//     z_i = sum_{l=0}^{k} c_l sum_{j=0}^{n-1} F_l(x_i + x_j) y_j.
// (Algorithm 2 as printed has no region C although x_i + x_j reaches 60.)
//
// The weights are the same for all n^2 pairs, so a pair needs one function of one
// variable, w(X) = sum_l c_l F_l(X).  Since dF_l/dX = -F_{l+1}, its Taylor
// coefficients at a point are sums of Boys functions there: every block takes F_0..
// F_{k+8} at the 1024 multiples of 1/16 up to 64 (a table of the definition's values,
// to the last bit of a double), forms the expansions of w to degree 8 about them in
// shared memory (64 KB, in integers), and a pair is then an index, eight products
// of a Horner sum and one FMA.  The truncation is below 2^-54 sum |c_l| F_l; the
// coefficients carry the FP64 rounding that the sum over l had pair by pair.  A block
// whose j have few pairs there expands w at those alone.  Bound by
// the multiply pipe (17 products and as many other instructions that run there, 31
// of 52 SM cycles for the 32 pairs of a warp); evaluating the orders for each pair took
// 255 cycles where x is sorted and the chip full (k = 12: n = 65536 156 to 21 ms,
// n = 2^17 530 to 73 ms).
//
// Pairs with X >= 64, with a negative, invalid or infinite argument, and all pairs where
// the weights are not finite (or near the largest double), are evaluated order by order: in region C w = F_0 sum_l e_l t^l, e_l = c_l
// (2l-1)!! / 32^l, t = 16 / X, as a fixed-point Horner sum (its partial sums are bounded
// by sum|e_l|); elsewhere by the downward recurrence of boys_region.cuh and FP64 FMAs.
//
// One thread per i; (x_j, y_j) go through shared memory in tiles.  The blocks of a
// cluster share their i and split the j, and sum their parts in a fixed order, so that
// a batch with few i still fills the chip.
#include <array>
#include <utility>

#include <cooperative_groups.h>

#include "boys_grid_table.h"
#include "boys_internal.h"
#include "boys_region.cuh"

namespace boys {
namespace {

namespace cg = cooperative_groups;
using region::u64;

constexpr int kBlock = 256;
constexpr int kEntries = BOYS_GRID;  // right edges 1/16, 2/16, ..., 64
static_assert(kEntries == 1024 && BOYS_GRID_ORDERS == 41, "the grid covers X < 64 and orders up to 32 + 8");
constexpr int kMaxCluster = 8;
constexpr int kNotFinite = -100000;

// Expansion of w about the right edge in t = 4 (edge - X), t in [0, 1/4]: signed
// integers, a0..a4 in units of 2^(ex - 62), a5..a8 in 2^14 of those.  The unit follows
// the interval's own sum |c_l| F_l, so that w keeps its relative accuracy where it is
// small; it holds the weights' scale too, so that y_j meets w itself (a sum of y_j w
// over the scale overflowed, or ran out of bits, where y and the weights offset each
// other).
struct __align__(16) Entry {
    long long a0, a1, a2, a3, a4;
    int a5, a6, a7, a8;
    int ex, pad;
};
static_assert(sizeof(Entry) == 64, "table entries are four 16-byte words");

// v 2^-f as a double (v a signed fixed-point integer), by integer assembly.
__device__ __forceinline__ double fixed_to_double(long long v, int f) {
    if (v == 0) return 0.0;
    const xf::Xf a = xf::from_fixed(v, f);
    const double m = xf::to_double(a);
    return v < 0 ? -m : m;
}

// Binary point f of a fixed-point sum bounded by M: M 2^f < 2^61 (f = 0 for M = 0).
__device__ __forceinline__ int fixed_point_for(double M) { return M > 0.0 ? 60 - ilogb(M) : 0; }

// t u + add for t = t1 2^-32 + t0 2^-64 (t1 >= 0, t0 signed) and a signed u.
__device__ __forceinline__ long long level(int t1, int t0, long long u, long long add) {
    const int u1 = (int)(u >> 32);
    const unsigned u0 = (unsigned)u;
    const u64 p = (u64)((long long)t1 * u1 + add);
    const int s = __mulhi(t0, u1);
    unsigned lo = (unsigned)p, hi = (unsigned)(p >> 32);
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;\n\tadd.cc.u32 %0, %0, %4;\n\taddc.u32 %1, %1, 0;"
        : "+r"(lo), "+r"(hi)
        : "r"((unsigned)s), "r"((unsigned)(s >> 31)), "r"(__umulhi((unsigned)t1, u0)));
    return (long long)((u64)hi << 32 | lo);
}

// Weights below this are taken up to it in the table and back in the sum: the unit's
// exponent stays above it less 84 (F_32 at X = 64) and a double's exponent has room.
constexpr int kMinScale = -900;

// v 2^(ex - 62) as a double (truncated); ex >= kMinScale - 84, the value below 2^1021.
__device__ __forceinline__ double unit_double(long long v, int ex) {
    const long long sign = v >> 63;
    const u64 a = (u64)(v ^ sign);
    const unsigned lo = (unsigned)a, hi = (unsigned)(a >> 32);
    if (hi == 0) return (sign ? -1.0 : 1.0) * ldexp((double)lo, ex - 62);
    int b;
    asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(hi));
    const unsigned h = region::shift_right(lo, hi, b + 2), l = region::shift_right(0, lo, b + 2);
    // leading bit 62, of weight 2^(b + 32 - 62 + ex); the hidden bit adds the last 1 to the exponent
    const unsigned top = (h >> 10) + ((unsigned)(b + ex + (1022 - 30)) << 20);
    return __hiloint2double((int)(top | ((unsigned)(sign >> 32) & 0x80000000u)), (int)region::shift_right(l, h, 10));
}

// (2l-1)!! / 32^l
struct Closed {
    double v[33];
    constexpr Closed() : v{} {
        double f = 1.0, p = 1.0;
        for (int l = 0; l <= 32; ++l, p /= 32.0) {
            v[l] = f * p;
            f *= (double)(2 * l + 1);
        }
    }
};
static __constant__ Closed c_closed;

constexpr u64 kOutside = 1ULL << 62;  // 64 in units of 2^-56

// w at X = U 2^-56 < 64 from its interval's expansion.
__device__ __forceinline__ double w_entry(const Entry* __restrict__ e, u64 U) {
    // edge - X = (2^52 - d) 2^-56 with d = U mod 2^52, and t is four of it
    const u64 tq = ~(U << 12) >> 2;  // t in Q64
    const int t0 = (int)(unsigned)tq, t1 = (int)((unsigned)(tq >> 32) + ((unsigned)tq >> 31));
    const int u5 = e->a5 + __mulhi(t1, e->a6 + __mulhi(t1, e->a7 + __mulhi(t1, e->a8)));
    long long u = e->a4 + ((long long)__mulhi(t1, u5) << 14);
    u = level(t1, t0, u, e->a3);
    u = level(t1, t0, u, e->a2);
    u = level(t1, t0, u, e->a1);
    u = level(t1, t0, u, e->a0);
    return unit_double(u, e->ex);
}

// x in units of 2^-56 (to nearest), below 2^62; 2^63 - 1 if x is not in [0, 64), so
// that the sum of two of these is at least 2^62 exactly where the pair is not in
// the table, and never wraps.
__device__ __forceinline__ u64 to_units(double x) {
    return x >= 0.0 && x < 64.0 ? (u64)__double2ll_rn(x * 0x1p56) : 0x7FFFFFFFFFFFFFFFULL;
}

// sum_l c_l F_l, the orders as they come.
struct Weighted {
    const double* c;  // shared memory
    double s;
    template <int L>
    __device__ __forceinline__ void operator()(std::integral_constant<int, L>, double v) { s = fma(c[L], v, s); }
};

// w(X) order by order.  efx holds the region-C sum's coefficients in units of 2^-fe.
template <int K>
__device__ __noinline__ double w_direct(double X, const double* c, const long long* efx, int fe) {
    const u64 xb = region::bits_of(X);
    Weighted w{c, 0.0};
    if (!region::regular(xb)) {
        region::eval_other(K, X, [&](int k, double v) { w.s = fma(c[k], v, w.s); });
        return w.s;
    }
    if (xb < region::kBitsX1 || fe == kNotFinite) {
        region::eval_regular<K, 0>(xb, region::local_table<K>(), w);
        return w.s;
    }
    const xf::Xf r = xf::rsqrt(xf::from_double(X));
    const xf::Xf R = xf::mul(xf::Xf{r.m, r.e - 1}, r);  // 1/(2X)
    const u64 T = R.m >> min(max(-(R.e + 6), 0), 63);   // 16/X in Q64
    const u64 Th = T >> 1;
    long long h = efx[K];
#pragma unroll
    for (int l = K - 1; l >= 0; --l) h = xf::mulhi_s(h, T, Th) + efx[l];
    return xf::to_double(xf::mul(xf::sqrt_pi_over_2(), r)) * fixed_to_double(h, fe);
}

// The entry of the interval that ends at x = (e + 1) / 16, for weights c 2^scale, c
// with sum |c_l| in [1/2, 1] (or all zero), from S_i = sum_l c_l F_{l+i}(x), i = 0..8.  The
// sums run from the highest order down, the smallest values first: from 0 up, the sums'
// rounding reached 10 units of 2^-53 sum |c_l| F_l (K = 32, X > 36).
// kLanes > 1: that many neighbouring lanes share an entry, every kLanes-th order each.
template <int K, int kLanes>
__device__ __noinline__ void expand(int e, const double* c, int scale, Entry& E) {
    double S[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, bound = 0.0;
#pragma unroll 1
    for (int l = K - (int)(threadIdx.x & (kLanes - 1)); l >= 0; l -= kLanes) {
        const double cl = c[l];
        const double* f = &g_grid_f[l][e];
        bound = fma(fabs(cl), __ldg(f), bound);
#pragma unroll
        for (int i = 0; i <= 8; ++i) S[i] = fma(cl, __ldg(f + i * kEntries), S[i]);
    }
#pragma unroll
    for (int d = 1; d < kLanes; d <<= 1) {
        const unsigned group = ((1u << kLanes) - 1) << (threadIdx.x & 31 & ~(kLanes - 1));
        bound += __shfl_xor_sync(group, bound, d);
#pragma unroll
        for (int i = 0; i <= 8; ++i) S[i] += __shfl_xor_sync(group, S[i], d);
    }
    // on the whole interval sum |c_l| F_l <= e^{1/16} bound; its unit keeps |w| below 2^61
    const int s = bound > 0.0 ? 59 - ilogb(bound) : 62;
    // Half of what the cut to a double drops at this size goes in, so that w is
    // rounded to nearest instead (where the interval stays within a factor of two).
    const long long a0 = __double2ll_rn(ldexp(S[0], s));
    const int lead = 63 - __clzll(llabs(a0) | 1);
    const long long half = lead < 53 ? 0 : 1LL << (lead - 53);
    E.a0 = a0 < 0 ? a0 - half : a0 + half;
    E.a1 = __double2ll_rn(ldexp(S[1], s - 2));
    E.a2 = __double2ll_rn(ldexp(S[2] * (1.0 / 2), s - 4));
    E.a3 = __double2ll_rn(ldexp(S[3] * (1.0 / 6), s - 6));
    E.a4 = __double2ll_rn(ldexp(S[4] * (1.0 / 24), s - 8));
    E.a5 = (int)__double2ll_rn(ldexp(S[5] * (1.0 / 120), s - 10 - 14));
    E.a6 = (int)__double2ll_rn(ldexp(S[6] * (1.0 / 720), s - 12 - 14));
    E.a7 = (int)__double2ll_rn(ldexp(S[7] * (1.0 / 5040), s - 14 - 14));
    E.a8 = (int)__double2ll_rn(ldexp(S[8] * (1.0 / 40320), s - 16 - 14));
    E.ex = 62 - s + scale;
}

// w at X = U 2^-56 < 64 without the table: the interval's entry for this pair alone.
template <int K, int kLanes>
__device__ __noinline__ double w_alone(u64 U, const double* c, int scale) {
    Entry E;
    expand<K, kLanes>((int)(U >> 52), c, scale, E);
    return w_entry(&E, U);
}

constexpr int kTileJ = kBlock;
// A block forms the table if more than this many of its j have pairs in it; the pairs
// of fewer j are expanded one by one.  Every block used to form it: a call of one pair
// took 55 us at k = 12 and 110 at k = 32 (10 and 14 now), and one whose pairs all
// lie beyond it, n = 256 with x on [32, 300], 275 at k = 12 (35 now).  n = 32, 48, 64
// (4, 6, 8 j a block) by the table and by pairs, us: k = 0 27, 28, 29 and 19, 25, 29;
// k = 12 57, 59, 59 and 43, 62, 80; k = 32 112, 113, 113 and 88, 127, 165.
#ifndef BOYS_PAIRWISE_TABLE_J
#define BOYS_PAIRWISE_TABLE_J 5
#endif
// Up to kFewRows rows, kFewLanes threads serve one row (an FP64 instruction of a warp
// costs 64 clocks of its quarter of the SM however few of its lanes are in use: n = 8, k
// = 32: 47 us with one, 16 with four), and the table is never formed.
constexpr int kFewRows = 8, kFewLanes = 4;
static_assert(kFewRows * kFewLanes <= 32 && BOYS_PAIRWISE_TABLE_J >= 2, "few rows share a warp, at most two j a block");

// The sum of a warp's values, in every lane.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

template <int K>
__global__ void __launch_bounds__(kBlock, 3) k_pairwise(const double* __restrict__ x, const double* __restrict__ y,
                                                        int64_t n, const double* __restrict__ c, double* __restrict__ z) {
    extern __shared__ __align__(64) unsigned char smem[];
    Entry* const s_tab = reinterpret_cast<Entry*>(smem);
    __shared__ double s_x[kTileJ], s_y[kTileJ], s_c[K + 1], s_cn[K + 1], s_z[kBlock];
    __shared__ u64 s_u[kTileJ];
    __shared__ long long s_efx[K + 1];
    __shared__ int s_fe, s_scale;
    __shared__ unsigned s_low[kBlock / 32];
    const cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part = (int)cluster.block_rank();
    const int t = threadIdx.x;
    if (t <= K) s_c[t] = __ldg(c + t);
    __syncthreads();
    if (t < 32) {
        // The exponent of sum |c_l|, by which the weights are scaled, and the binary
        // point of the region-C sum over e_l = c_l (2l-1)!! / 32^l of the scaled ones;
        // lane t has the orders t and t + 32
        double sc = 0.0, se = 0.0, e[2] = {0.0, 0.0};
        for (int l = t; l <= K; l += 32) sc += fabs(s_c[l]);
        sc = warp_sum(sc);
        const bool finite = sc < 0x1p1020;
        const int scale = finite ? (sc > 0.0 ? ilogb(sc) + 1 : 0) : kNotFinite;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int l = t + 32 * q;
            if (l > K) break;
            const double cn = finite ? ldexp(s_c[l], -scale) : 0.0;
            s_cn[l] = cn;
            e[q] = cn * c_closed.v[l];
            se += fabs(e[q]);
        }
        se = warp_sum(se);
        const int fe = fixed_point_for(se);
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (t + 32 * q <= K) s_efx[t + 32 * q] = __double2ll_rn(ldexp(e[q], fe));
        if (t == 0) {
            s_fe = finite ? fe - scale : kNotFinite;
            s_scale = scale;
        }
    }
    const bool few = n <= kFewRows;
    const int64_t i = few ? t / kFewLanes : (int64_t)(blockIdx.x / parts) * kBlock + t;
    const bool row = i < n, writes = row && !(few && t % kFewLanes);
    const double xi = row ? __ldg(x + i) : INFINITY;
    const int64_t first = n * part / parts, last = n * (part + 1) / parts;
    // Whether to form the table: j that have a pair in it are those with x_j below 64
    // less the smallest x_i (by the high words of both, so some just above count too).
    const unsigned low = __reduce_min_sync(0xffffffffu, (unsigned)(to_units(xi) >> 32));
    if ((t & 31) == 0) s_low[t / 32] = low;
    __syncthreads();
    const int scale = s_scale, held = max(scale, kMinScale);
    unsigned lowest = s_low[0];
#pragma unroll
    for (int w = 1; w < kBlock / 32; ++w) lowest = min(lowest, s_low[w]);
    int inside = 0;
    for (int64_t j0 = first; j0 < last && inside <= BOYS_PAIRWISE_TABLE_J && scale != kNotFinite; j0 += kBlock)
        inside += __syncthreads_count(j0 + t < last && lowest + (unsigned)(to_units(__ldg(x + j0 + t)) >> 32) < (unsigned)(kOutside >> 32));
    const bool table = inside > BOYS_PAIRWISE_TABLE_J;
    if (table)
        for (int e = t; e < kEntries; e += kBlock) expand<K, 1>(e, s_cn, held, s_tab[e]);
    const u64 ui = scale != kNotFinite ? to_units(xi) : 0x7FFFFFFFFFFFFFFFULL;
    double zt = 0.0, zd = 0.0;  // the table's pairs, in units of 2^(scale - held), and the others
    for (int64_t j0 = first; j0 < last; j0 += kTileJ) {
        __syncthreads();
        if (j0 + t < last) {
            const double xj = __ldg(x + j0 + t);
            s_x[t] = xj;
            s_u[t] = to_units(xj);
            s_y[t] = __ldg(y + j0 + t);
        }
        __syncthreads();
        const int jn = row ? (int)min((int64_t)kTileJ, last - j0) : 0;
        // Two pairs at a time, the products of one filling the waits of the other (n =
        // 65536, k = 12: 22.4 ms with one, 21.1 with two, 20.9 with four).
        int jj = 0;
        for (; table && jj + 2 <= jn; jj += 2) {
            u64 U[2], all = 0;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                U[q] = ui + s_u[jj + q];
                all |= U[q];
            }
            if (all < kOutside) {
                double w[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) w[q] = w_entry(s_tab + (int)(U[q] >> 52), U[q]);
#pragma unroll
                for (int q = 0; q < 2; ++q) zt = fma(s_y[jj + q], w[q], zt);
            } else {
#pragma unroll 1
                for (int q = 0; q < 2; ++q) {
                    const u64 V = ui + s_u[jj + q];
                    if (V < kOutside) zt = fma(s_y[jj + q], w_entry(s_tab + (int)(V >> 52), V), zt);
                    else zd = fma(s_y[jj + q], w_direct<K>(xi + s_x[jj + q], s_c, s_efx, s_fe), zd);
                }
            }
        }
        for (; jj < jn; ++jj) {
            const u64 V = ui + s_u[jj];
            if (V < kOutside)
                zt = fma(s_y[jj], table ? w_entry(s_tab + (int)(V >> 52), V) : few ? w_alone<K, kFewLanes>(V, s_cn, held)
                                                                                 : w_alone<K, 1>(V, s_cn, held), zt);
            else zd = fma(s_y[jj], w_direct<K>(xi + s_x[jj], s_c, s_efx, s_fe), zd);
        }
    }
    const double zi = scale < held ? ldexp(zt, scale - held) + zd : zt + zd;
    if (parts == 1) {
        if (writes) z[i] = zi;
        return;
    }
    s_z[t] = zi;
    cluster.sync();
    if (part == 0 && writes) {
        double sum = zi;
        for (int r = 1; r < parts; ++r) sum += cluster.map_shared_rank(s_z, r)[t];
        z[i] = sum;
    }
    cluster.sync();  // the parts stay readable until they are summed
}

template <int... K>
constexpr auto pairwise_table(std::integer_sequence<int, K...>) {
    using Fn = void (*)(const double*, const double*, int64_t, const double*, double*);
    return std::array<Fn, sizeof...(K)>{&k_pairwise<K>...};
}

}  // namespace
}  // namespace boys

BOYS_API boys_status boys_pairwise(const double* x, const double* y, int64_t n, const double* c, int k, double* z,
                                   void* stream) {
    using namespace boys;
    if (k < 0 || k > 32) return fail(BOYS_ERR_KMAX, "boys_pairwise: k=%d outside [0, 32]", k);
    if (n < 0) return fail(BOYS_ERR_INVALID_ARG, "boys_pairwise: n=%lld < 0", (long long)n);
    if (n == 0) return BOYS_OK;
    if (!x || !y || !c || !z) return fail(BOYS_ERR_INVALID_ARG, "boys_pairwise: NULL pointer");
    if (!aligned(x, 8) || !aligned(y, 8) || !aligned(c, 8) || !aligned(z, 8))
        return fail(BOYS_ERR_ALIGNMENT, "boys_pairwise: pointers not 8-byte aligned");
    if (n > ((int64_t)1 << 40)) return fail(BOYS_ERR_INVALID_ARG, "boys_pairwise: n=%lld too large", (long long)n);
    static constexpr auto t = pairwise_table(std::make_integer_sequence<int, 33>{});
    const int64_t rows = (n + kBlock - 1) / kBlock;
    // As many parts (a power of two) as bring the grid to eight blocks per SM, as long
    // as each keeps one j.
    int parts = 1;
    while (parts < kMaxCluster && rows * parts < (int64_t)sm_count() * 8 && 2 * parts <= n) parts *= 2;
    if (rows * parts > 0x7fffffff) return fail(BOYS_ERR_INVALID_ARG, "boys_pairwise: grid too large");
    const size_t smem = sizeof(Entry) * kEntries;
    boys_status st = check_cuda(cudaFuncSetAttribute((const void*)t[k], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                                "boys_pairwise shared memory");
    if (st != BOYS_OK) return st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)parts;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(rows * parts));
    lc.blockDim = dim3(kBlock);
    lc.dynamicSmemBytes = smem;
    lc.stream = (cudaStream_t)stream;
    lc.attrs = &attr;
    lc.numAttrs = 1;
    return check_cuda(cudaLaunchKernelEx(&lc, t[k], x, y, n, c, z), "boys_pairwise launch");
}
