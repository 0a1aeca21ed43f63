// div_by (k_aux.cu), the division of fluxes by the speed of light as a multiplication and a correction, against the
// division: on the quotients nearest to a halfway point between two doubles (both sides, for random divisors and ones
// next to a power of two, at several scales), on random operands, and on zeros, subnormals, infinities, NaN and
// operands near the ends of the range.  Also, on the host, the same three operations in p-bit arithmetic over all
// operands, p = 4 .. 11.  Prints "<halfway cases> <differences> <other cases> <differences> <p-bit differences>".
// Built and run by tests/test_gpu_div_by.py.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
#include <vector>

#include "k_aux.cu"

__global__ void check_kernel(const double* x, const double* c, const double* y, double* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = rhd::div_by(x[i], c[i], y[i]);
}

typedef unsigned __int128 u128;

static uint64_t inverse(uint64_t a, uint64_t m)
{
    __int128 t = 0, nt = 1, r = m, nr = a % m;
    while (nr) {
        const __int128 q = r / nr, t2 = t - q * nt, r2 = r - q * nr;
        t = nt, nt = t2, r = nr, nr = r2;
    }
    return (uint64_t)(t < 0 ? t + m : t);
}

// x / c with x 2^s = +-k mod c: the quotient is k / (c 2^s) from a multiple of 2^-s, which for these s are the halfway points
static void halfway(std::vector<double>& x, std::vector<double>& c, std::mt19937_64& rng)
{
    std::uniform_int_distribution<int> scale(-190, 190);
    for (int it = 0; it < 200000; ++it) {
        uint64_t C = (1ull << 52) | (rng() & ((1ull << 52) - 1)) | 1;
        if (it % 3 == 0) C = (1ull << 53) - 1 - 2 * (rng() % 100000);
        for (int big = 0; big < 2; ++big) {
            const uint64_t inv = inverse((uint64_t)(((u128)1 << (54 - big)) % C), C);
            for (int k = -3; k <= 3; ++k) {
                if (!k) continue;
                uint64_t X = (uint64_t)((u128)(k > 0 ? (uint64_t)k : C + k) * inv % C);
                if (big) X += C;
                if (X < (1ull << 52) || X >= (1ull << 53)) continue;
                x.push_back((rng() & 1 ? -1.0 : 1.0) * std::ldexp((double)X, scale(rng) - 52));
                c.push_back(std::ldexp((double)C, scale(rng) - 52));
            }
        }
    }
}

static long long differences(const std::vector<double>& x, const std::vector<double>& c)
{
    const int n = (int)x.size();
    std::vector<double> y(n), o(n);
    for (int i = 0; i < n; ++i) y[i] = 1.0 / c[i];
    double* d[4];
    for (auto& p : d)
        if (cudaMalloc(&p, 8 * (size_t)n)) return -1;
    cudaMemcpy(d[0], x.data(), 8 * (size_t)n, cudaMemcpyHostToDevice);
    cudaMemcpy(d[1], c.data(), 8 * (size_t)n, cudaMemcpyHostToDevice);
    cudaMemcpy(d[2], y.data(), 8 * (size_t)n, cudaMemcpyHostToDevice);
    check_kernel<<<(n + 255) / 256, 256>>>(d[0], d[1], d[2], d[3], n);
    if (cudaMemcpy(o.data(), d[3], 8 * (size_t)n, cudaMemcpyDeviceToHost)) return -2;
    for (auto& p : d) cudaFree(p);
    long long bad = 0;
    for (int i = 0; i < n; ++i) {
        const double ref = x[i] / c[i];
        bad += std::isnan(ref) ? !std::isnan(o[i]) : std::memcmp(&ref, &o[i], 8) != 0;
    }
    return bad;
}

// v rounded to p bits (v exact in a double: p <= 11)
static double rn(double v, int p)
{
    if (v == 0.0) return 0.0;
    int e;
    std::frexp(v, &e);
    return std::ldexp(std::nearbyint(std::ldexp(v, p - e)), e - p);
}

int main()
{
    std::mt19937_64 rng(3);
    std::vector<double> x, c;
    halfway(x, c, rng);
    const size_t n_half = x.size();
    const long long bad_half = differences(x, c);
    x.clear(), c.clear();
    std::uniform_real_distribution<double> m(-2.0, 2.0);
    std::uniform_int_distribution<int> ex(-1070, 1020), ec(-199, 199);
    for (int i = 0; i < 1 << 20; ++i) {
        x.push_back(std::ldexp(m(rng), ex(rng)));
        c.push_back(std::ldexp(1.0 + std::fabs(m(rng)) / 2.0, ec(rng)));
    }
    const double inf = std::numeric_limits<double>::infinity();
    for (double s : {0.0, -0.0, inf, -inf, std::nan(""), 5e-324, -5e-324, 2.2e-308, 1.7e308, -1.7e308, 1.0})
        for (double t : {1.0, 10.0, 2.99792458e10, 1e-59, 1e59}) x.push_back(s), c.push_back(t);
    const size_t n_other = x.size();
    const long long bad_other = differences(x, c);
    long long bad_p = 0;
    for (int p = 4; p <= 11; ++p)
        for (int C = 1 << (p - 1); C < 1 << p; ++C) {
            const double y = rn(1.0 / C, p);
            for (int X = 1 << (p - 1); X < 1 << p; ++X) {
                const double q = rn(X * y, p), r = rn(X - q * C, p);
                bad_p += rn(q + r * y, p) != rn((double)X / C, p);
            }
        }
    std::printf("%zu %lld %zu %lld %lld\n", n_half, bad_half, n_other, bad_other, bad_p);
    return 0;
}
