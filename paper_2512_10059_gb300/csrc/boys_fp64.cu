// FP64 stored mode (boys_eval, boys_eval_host) and fused consumer
// (boys_eval_fused).
//
// Stored mode: one thread per argument (grid-stride loop); KMAX is a template
// parameter, the recurrence is unrolled, and each step writes one whole row of the
// warp (256 bytes).
#include <array>
#include <utility>

#include "boys_internal.h"
#include "boys_region.cuh"

namespace boys {
namespace {

constexpr int kBlock = 128;

// Full occupancy (16 blocks of 128 threads per SM, 32 registers): the recurrence
// keeps a dozen values, so the cap costs at most a few spills (kmax 8, 2^25
// arguments: 478 us against 492 with 12 blocks and 492 with 10).
// BOYS_STORED_MIN_BLOCKS forces another value.
#ifndef BOYS_STORED_MIN_BLOCKS
#define BOYS_STORED_MIN_BLOCKS 16
#endif
template <int KMAX>
__global__ void __launch_bounds__(kBlock, BOYS_STORED_MIN_BLOCKS) k_eval_f64(const double* __restrict__ x, int64_t n,
                                                     double* __restrict__ out, int64_t ld) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        region::eval_store<KMAX>(__ldcs(x + i), out + i, ld);
}

// The fused consumer is bound by the FP64 pipe: kmax FMAs an argument at 2 a clock
// and SM (kmax 32, 2^24 arguments: 853 us of the 880), so every step of the recurrence
// stays on the integer pipes, and so does everything else (with two more FP64
// instructions an argument, the factor -2 and a comparison, 964 us).  8 blocks per SM
// suffice (8, 10, 12, 16 blocks: within 1%).
#ifndef BOYS_FUSED_MIN_BLOCKS
#define BOYS_FUSED_MIN_BLOCKS 8
#endif

// Horner sum in a, the orders as they come, from the highest down (order K first).
template <int K>
struct Horner {
    double a, s;
    template <int L>
    __device__ __forceinline__ void operator()(std::integral_constant<int, L>, double v) {
        s = L == K ? v : fma(s, a, v);
    }
};

// -2 v without the FP64 pipe where that is an exponent's increment (the product in
// the same function would be computed every time and selected).
static __device__ __noinline__ double minus_twice_special(double v) { return -2.0 * v; }
__device__ __forceinline__ double minus_twice(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), e = (hi >> 20) & 0x7FF;
    if (e - 1 < 0x7FD) return __hiloint2double((int)((hi ^ 0x80000000u) + 0x100000u), __double2loint(v));
    return minus_twice_special(v);  // zero, subnormal, 2^1023 and above, NaN
}

// The same for the arguments that eval_other takes, whose orders come upward.
template <int KMAX>
__device__ __noinline__ double fused_other(double x, double a) {
    double f[KMAX + 1];
    region::eval_other(KMAX, x, [&](int k, double v) { f[k] = v; });
    double s = f[KMAX];
#pragma unroll 1
    for (int k = KMAX - 1; k >= 0; --k) s = fma(s, a, f[k]);
    return s;
}

// out[i] = sum_k a^k F_k(x_i), a = -2 rho_i.
template <int KMAX>
__global__ void __launch_bounds__(kBlock, BOYS_FUSED_MIN_BLOCKS) k_fused_f64(const double* __restrict__ x,
                                                      const double* __restrict__ rho, int64_t n,
                                                      double* __restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const double xi = __ldcs(x + i), a = minus_twice(__ldcs(rho + i));
        const region::u64 xb = region::bits_of(xi);
        Horner<KMAX> h{a, 0.0};
        if (region::regular(xb)) {
            region::eval_regular<KMAX, 0>(xb, region::local_table<KMAX>(), h);
        } else {
            h.s = fused_other<KMAX>(xi, a);
        }
        __stcs(out + i, h.s);
    }
}

template <int... K>
constexpr auto eval_table(std::integer_sequence<int, K...>) {
    using Fn = void (*)(const double*, int64_t, double*, int64_t);
    return std::array<Fn, sizeof...(K)>{&k_eval_f64<K>...};
}

template <int... K>
constexpr auto fused_table(std::integer_sequence<int, K...>) {
    using Fn = void (*)(const double*, const double*, int64_t, double*);
    return std::array<Fn, sizeof...(K)>{&k_fused_f64<K>...};
}

}  // namespace
}  // namespace boys


namespace boys {
// Checks and launches stored mode.
static boys_status eval_launch(const char* name, const double* x, int64_t n, int kmax, double* out, int64_t ld,
                               void* stream) {
    if (kmax < 0 || kmax > 32) return fail(BOYS_ERR_KMAX, "%s: kmax=%d outside [0, 32]", name, kmax);
    if (n < 0) return fail(BOYS_ERR_INVALID_ARG, "%s: n=%lld < 0", name, (long long)n);
    if (ld < n) return fail(BOYS_ERR_INVALID_ARG, "%s: ld=%lld < n=%lld", name, (long long)ld, (long long)n);
    if (n == 0) return BOYS_OK;
    if (!x || !out) return fail(BOYS_ERR_INVALID_ARG, "%s: NULL pointer", name);
    if (ld > INT64_MAX / (kmax + 1)) return fail(BOYS_ERR_INVALID_ARG, "%s: (kmax+1)*ld overflows", name);
    if (!aligned(x, 8) || !aligned(out, 8)) return fail(BOYS_ERR_ALIGNMENT, "%s: x/out not 8-byte aligned", name);
    static constexpr auto t = eval_table(std::make_integer_sequence<int, 33>{});
    const auto fn = t[kmax];
    // A block of a small order is over so soon that its launch shows: at most 8
    // waves of resident blocks up to kmax 10 (kmax 0, 2^24 arguments: 83 us
    // against 99 with 64 waves; kmax 8, 2^25: 478 against 483), the default 64
    // above, where finer blocks balance the stores better (kmax 32, 2^26: 2.70 ms
    // against 2.77 with 8).
    const int64_t grid = grid_for((const void*)fn, kBlock, n, (int64_t)kBlock, kmax <= 10 ? 8 : BOYS_GRID_WAVES);
    fn<<<(unsigned)grid, kBlock, 0, (cudaStream_t)stream>>>(x, n, out, ld);
    return check_cuda(cudaGetLastError(), "boys_eval launch");
}
}  // namespace boys

BOYS_API boys_status boys_eval(const double* x, int64_t n, int kmax, double* out, int64_t ld,
                               void* stream) {
    return boys::eval_launch("boys_eval", x, n, kmax, out, ld, stream);
}

BOYS_API boys_status boys_eval_fused(const double* x, const double* rho, int64_t n, int kmax,
                                     double* out, void* stream) {
    using namespace boys;
    if (kmax < 0 || kmax > 32) return fail(BOYS_ERR_KMAX, "boys_eval_fused: kmax=%d outside [0, 32]", kmax);
    if (n < 0) return fail(BOYS_ERR_INVALID_ARG, "boys_eval_fused: n=%lld < 0", (long long)n);
    if (n == 0) return BOYS_OK;
    if (!x || !rho || !out) return fail(BOYS_ERR_INVALID_ARG, "boys_eval_fused: NULL pointer");
    if (!aligned(x, 8) || !aligned(rho, 8) || !aligned(out, 8))
        return fail(BOYS_ERR_ALIGNMENT, "boys_eval_fused: pointers not 8-byte aligned");
    static constexpr auto t = fused_table(std::make_integer_sequence<int, 33>{});
    const auto fn = t[kmax];
    const int64_t grid = grid_for((const void*)fn, kBlock, n, kBlock);
    fn<<<(unsigned)grid, kBlock, 0, (cudaStream_t)stream>>>(x, rho, n, out);
    return check_cuda(cudaGetLastError(), "boys_eval_fused launch");
}

// Host buffers (pinned, or pageable where the GPU can address pageable memory):
// the evaluation kernel itself reads x and writes F over the host link.
namespace boys {
static boys_status host_view(const void* p, void** dev, const char* what) {
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) return check_cuda(e, "boys_eval_host: cudaPointerGetAttributes");
    if (a.type == cudaMemoryTypeHost && a.devicePointer) {
        *dev = a.devicePointer;
        return BOYS_OK;
    }
    if (a.type == cudaMemoryTypeUnregistered) {
        int device = 0, pageable = 0;
        cudaGetDevice(&device);
        cudaDeviceGetAttribute(&pageable, cudaDevAttrPageableMemoryAccess, device);
        if (pageable) {
            *dev = const_cast<void*>(p);
            return BOYS_OK;
        }
    }
    return fail(BOYS_ERR_INVALID_ARG,
                "boys_eval_host: %s is not host memory the GPU can address (pin it with cudaHostAlloc/cudaHostRegister)",
                what);
}
}  // namespace boys

BOYS_API boys_status boys_eval_host(const double* x, int64_t n, int kmax, double* out, int64_t ld, void* stream) {
    using namespace boys;
    if (kmax < 0 || kmax > 32) return fail(BOYS_ERR_KMAX, "boys_eval_host: kmax=%d outside [0, 32]", kmax);
    if (n < 0) return fail(BOYS_ERR_INVALID_ARG, "boys_eval_host: n=%lld < 0", (long long)n);
    if (ld < n) return fail(BOYS_ERR_INVALID_ARG, "boys_eval_host: ld=%lld < n=%lld", (long long)ld, (long long)n);
    if (n == 0) return BOYS_OK;
    if (!x || !out) return fail(BOYS_ERR_INVALID_ARG, "boys_eval_host: NULL pointer");
    void *xd = nullptr, *od = nullptr;
    boys_status st = host_view(x, &xd, "x");
    if (st != BOYS_OK) return st;
    st = host_view(out, &od, "out");
    if (st != BOYS_OK) return st;
    return eval_launch("boys_eval_host", (const double*)xd, n, kmax, (double*)od, ld, stream);
}
