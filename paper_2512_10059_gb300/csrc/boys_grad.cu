// Backward of F_0..F_kmax with respect to x (boys_grad).
//
// Differentiating the definition (Eq. 3) under the integral sign gives
// dF_k/dx = -F_{k+1}, so for upstream gradients g_k:
//     dL/dx_i = -sum_{k=0}^{kmax} g[k*ldg + i] * F_{k+1}(x_i).
// The kernel re-evaluates F_{kmax+1}..F_1 with the forward method at order
// kmax+1 (nothing but x is saved by the forward), so kmax <= 31.
#include <array>
#include <utility>

#include "boys_internal.h"
#include "boys_region.cuh"

namespace boys {
namespace {

constexpr int kBlock = 128;

// The sum is kmax + 1 FMAs an argument on the FP64 pipe, at 2 a clock and SM (kmax
// 16, 2^24 arguments: 453 us of the 486; 561 with two more FP64 instructions, 958 with
// the recurrence that served all regions), so every step of the recurrence stays on
// the integer pipes.  8 to 16 blocks per SM are within 1%.
#ifndef BOYS_GRAD_MIN_BLOCKS
#define BOYS_GRAD_MIN_BLOCKS 8
#endif

// Subtracts g_k F_{k+1} as the orders come, from the highest down.
struct Dot {
    const double* g;  // the next order's row
    int64_t ldg;
    double s;
    template <int L>
    __device__ __forceinline__ void operator()(std::integral_constant<int, L>, double v) {
        s = fma(-__ldcs(g), v, s);
        g -= ldg;
    }
};

template <int KMAX>
__global__ void __launch_bounds__(kBlock, BOYS_GRAD_MIN_BLOCKS) k_grad_f64(const double* __restrict__ x, int64_t n,
                                                     const double* __restrict__ g, int64_t ldg,
                                                     double* __restrict__ dx) {
    constexpr int K = KMAX + 1;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const double xi = __ldcs(x + i);
        const region::u64 xb = region::bits_of(xi);
        Dot d{g + KMAX * ldg + i, ldg, 0.0};
        if (region::regular(xb)) {
            region::eval_regular<K, 0, 1>(xb, region::local_table<K>(), d);
        } else {
            const double* gi = g + i;
            region::eval_other(K, xi, [&](int k, double v) {
                if (k > 0) d.s = fma(-__ldcs(gi + (k - 1) * ldg), v, d.s);
            });
        }
        __stcs(dx + i, d.s);
    }
}

template <int... K>
constexpr auto grad_table(std::integer_sequence<int, K...>) {
    using Fn = void (*)(const double*, int64_t, const double*, int64_t, double*);
    return std::array<Fn, sizeof...(K)>{&k_grad_f64<K>...};
}

}  // namespace
}  // namespace boys

BOYS_API boys_status boys_grad(const double* x, int64_t n, int kmax, const double* g, int64_t ldg,
                               double* dx, void* stream) {
    using namespace boys;
    if (kmax < 0 || kmax > 31) return fail(BOYS_ERR_KMAX, "boys_grad: kmax=%d outside [0, 31]", kmax);
    if (n < 0) return fail(BOYS_ERR_INVALID_ARG, "boys_grad: n=%lld < 0", (long long)n);
    if (ldg < n) return fail(BOYS_ERR_INVALID_ARG, "boys_grad: ldg=%lld < n=%lld", (long long)ldg, (long long)n);
    if (n == 0) return BOYS_OK;
    if (!x || !g || !dx) return fail(BOYS_ERR_INVALID_ARG, "boys_grad: NULL pointer");
    if (ldg > INT64_MAX / (kmax + 1)) return fail(BOYS_ERR_INVALID_ARG, "boys_grad: (kmax+1)*ldg overflows");
    if (!aligned(x, 8) || !aligned(g, 8) || !aligned(dx, 8))
        return fail(BOYS_ERR_ALIGNMENT, "boys_grad: pointers not 8-byte aligned");
    static constexpr auto t = grad_table(std::make_integer_sequence<int, 32>{});
    const auto fn = t[kmax];
    const int64_t grid = grid_for((const void*)fn, kBlock, n, kBlock);
    fn<<<(unsigned)grid, kBlock, 0, (cudaStream_t)stream>>>(x, n, g, ldg, dx);
    return check_cuda(cudaGetLastError(), "boys_grad launch");
}
