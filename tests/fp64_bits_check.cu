// The FP64 comparisons by bits and the FP64 square root of the kernels (fp_convert.cuh) against plain
// comparisons and CUDA's sqrt, over random values (both signs, exponents in [-300, 300], pairs of equal
// magnitude) and special ones (zeros, infinities, NaN, subnormals, neighbours of 1): prints the number of
// differences and the square root's largest distance in units in the last place.  Built and run by
// tests/test_gpu_fp64_bits.py.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
#include <vector>

#include "fp_convert.cuh"

__global__ void check_kernel(const double* x, const double* y, double* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[5 * i] = rhd::max0_d(x[i], y[i]);
    out[5 * i + 1] = rhd::min0_d(x[i], y[i]);
    out[5 * i + 2] = rhd::minmod_d(x[i], y[i]);
    out[5 * i + 3] = rhd::reaches1_d(x[i]) ? 1.0 : 0.0;
    out[5 * i + 4] = rhd::sqrt3(x[i]);
}

static int64_t bits(double v)
{
    int64_t b;
    std::memcpy(&b, &v, sizeof b);
    return b;
}

int main()
{
    const double inf = std::numeric_limits<double>::infinity(), nan = std::nan("");
    const double special[] = {0.0, -0.0, inf, -inf, nan, 1.0, -1.0, 5e-324, -5e-324, 2.3e-308, 1e308, 1.0 - 1e-15,
                              1.0 - 8.8817841970012523e-16, 1.0 - 7.7715611723760958e-16, 1.0 + 2.2204460492503131e-16};
    const int ns = sizeof special / sizeof special[0], nr = 1 << 18, n = ns * ns + nr;
    std::vector<double> x(n), y(n), o(5 * n);
    for (int i = 0; i < ns * ns; ++i) {
        x[i] = special[i / ns];
        y[i] = special[i % ns];
    }
    std::mt19937_64 rng(64);
    std::uniform_real_distribution<double> m(-2.0, 2.0);
    std::uniform_int_distribution<int> ex(-300, 300);
    for (int i = ns * ns; i < n; ++i) {
        x[i] = std::ldexp(m(rng), ex(rng));
        y[i] = i % 3 == 0 ? x[i] * (1.0 + 1e-15 * m(rng)) : (i % 3 == 1 ? -x[i] : std::ldexp(m(rng), ex(rng)));
    }
    double *dx, *dy, *d;
    if (cudaMalloc(&dx, 8 * n) || cudaMalloc(&dy, 8 * n) || cudaMalloc(&d, 40 * n)) return 2;
    cudaMemcpy(dx, x.data(), 8 * n, cudaMemcpyHostToDevice);
    cudaMemcpy(dy, y.data(), 8 * n, cudaMemcpyHostToDevice);
    check_kernel<<<(n + 255) / 256, 256>>>(dx, dy, d, n);
    if (cudaMemcpy(o.data(), d, 40 * n, cudaMemcpyDeviceToHost)) return 3;
    long long off[4] = {0, 0, 0, 0}, sqrt_special = 0;
    int64_t worst = 0;
    for (int i = 0; i < n; ++i) {
        const double a = x[i], b = y[i];
        const bool nn = std::isnan(a) || std::isnan(b);
        const double hi = std::fmax(std::fmax(a, b), 0.0), lo = std::fmin(std::fmin(a, b), 0.0);
        const bool same = (a > 0 && b > 0) || (a < 0 && b < 0);
        const double mm = !same ? 0.0 : (std::fabs(a) < std::fabs(b) ? a : b);
        if (!nn) {  // maxima and minima carry a positive NaN on; the kernels' other values then do as well
            off[0] += !(o[5 * i] == hi);
            off[1] += !(o[5 * i + 1] == lo);
        }
        off[2] += !(o[5 * i + 2] == mm);
        off[3] += (o[5 * i + 3] == 1.0) != (a > 1.0 - 8.8817841970012523e-16);
        const double s = o[5 * i + 4];
        if (a >= 2.2250738585072014e-308 && a < inf) {
            const int64_t dd = std::llabs(bits(s) - bits(std::sqrt(a)));
            if (dd > worst) worst = dd;
        } else if (std::isnan(a) || a < -2.2250738585072014e-308) sqrt_special += !std::isnan(s);
        else sqrt_special += !(s == (a == inf ? inf : 0.0));
    }
    std::printf("max0 %lld min0 %lld minmod %lld reaches1 %lld sqrt_special %lld sqrt_ulp %lld\n", off[0], off[1], off[2],
                off[3], sqrt_special, (long long)worst);
    return 0;
}
