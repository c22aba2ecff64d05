// xmath_probe.cu -- the plain form's scalar arithmetic (xmath.cuh) beside CUDA's
// own operations, for tests/test_gpu_xmath.py: every pair of operands through
// both, results compared as bit patterns (any NaN equals any other).
#include <cuda_runtime.h>

#include "integrators.cuh"
#include "rhs.cuh"
#include "xmath.cuh"

using namespace bode;

namespace {

__device__ bool same(double x, double y) {
    return __double_as_longlong(x) == __double_as_longlong(y) || (isnan(x) && isnan(y));
}

__device__ bool check(int what, double a, double b) {
    switch (what) {
    case 0: {  // reciprocal: 1 / b in its range, 0 outside (and for what is not positive)
        const double r = xm::reciprocal(b);
        return same(r, b >= 0x1p-100 && b <= 0x1p100 ? 1.0 / b : 0.0);
    }
    case 1: return same(xm::div_by(a, b, xm::reciprocal(b)), a / b);
    case 2: {  // products on the integer pipe, in the range their users test
        const xm::Multiplier m = xm::multiplier(b);
        return !m.ok || !(fabs(a) >= 0x1p-600 && fabs(a) <= 0x1p600) || same(xm::mul_int(a, m), a * b);
    }
    case 3: {  // two exponentials side by side, one, and the general one
        const double x[2] = {a, b};
        double out[2];
        xm::exp_series2(x, out);
        return same(out[0], xm::exp_general(a)) && same(out[1], xm::exp_general(b)) && same(xm::exp_series(a), out[0]);
    }
    case 4: return same(xm::log_series(a), xm::log_general(a));
    case 5:  // comparisons of numbers that are not negative
        a = fabs(a);
        b = fabs(b);
        return xm::lt_nn(a, b) == (a < b) && xm::le_nn(a, b) == (a <= b) && xm::is_nan(a) == (bool)isnan(a) &&
               xm::is_finite(a) == (bool)isfinite(a) && xm::is_pos(a) == (a > 0.0) && xm::is_pos(-a) == (-a > 0.0) &&
               (isnan(a) || (same(xm::max_nn(a, b), fmax(a, b)) && same(xm::min_nn(a, b), fmin(a, b))));
    default:  // (int)sqrt(v) of a stage count
        a = fabs(a) + 1.0;
        return !(a < 4.0e18) || RkcF64<VdpModel>::floor_sqrt(a) == (int)sqrt(a);
    }
}

__global__ void k_check(int what, const double* a, const double* b, long long n, unsigned long long* bad, double* first) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || check(what, a[i], b[i])) return;
    if (atomicAdd(bad, 1ull) == 0ull) {
        first[0] = a[i];
        first[1] = b[i];
    }
}

}  // namespace

// host arrays a, b [n]; the number of pairs that differ, and one of them
extern "C" long long xmath_check(int what, const double* a, const double* b, long long n, double* first) {
    double *da = nullptr, *db = nullptr, *df = nullptr;
    unsigned long long* bad = nullptr;
    unsigned long long count = ~0ull;
    const size_t bytes = sizeof(double) * (size_t)n;
    if (n > 0 && cudaMalloc(&da, bytes) == cudaSuccess && cudaMalloc(&db, bytes) == cudaSuccess &&
        cudaMalloc(&df, 2 * sizeof(double)) == cudaSuccess && cudaMalloc(&bad, sizeof(*bad)) == cudaSuccess &&
        cudaMemcpy(da, a, bytes, cudaMemcpyHostToDevice) == cudaSuccess &&
        cudaMemcpy(db, b, bytes, cudaMemcpyHostToDevice) == cudaSuccess &&
        cudaMemset(bad, 0, sizeof(*bad)) == cudaSuccess && cudaMemset(df, 0, 2 * sizeof(double)) == cudaSuccess) {
        k_check<<<(unsigned)((n + 255) / 256), 256>>>(what, da, db, n, bad, df);
        if (cudaGetLastError() != cudaSuccess || cudaMemcpy(&count, bad, sizeof(count), cudaMemcpyDeviceToHost) != cudaSuccess ||
            cudaMemcpy(first, df, 2 * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess)
            count = ~0ull;
    }
    cudaFree(da);
    cudaFree(db);
    cudaFree(df);
    cudaFree(bad);
    return (long long)count;
}
