// fp_convert.cuh -- FP64 <-> FP32 conversions by integer bit operations, and the square roots and
// reciprocals of the kernels (shared by the kernel translation units).
#pragma once
#include <cuda_runtime.h>

namespace rhd {

// FP64 <-> FP32 conversions without the FP64 pipe (which runs at a small fraction of the FP32 rate
// on this part): truncation of the FP64 value to FP32 (normal range; underflow to 0, overflow to
// inf), and the exact widening of an FP32 value (denormals flushed), by integer bit operations.
__device__ __forceinline__ float d2f_trunc(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned sign = hi & 0x80000000u, a = hi & 0x7fffffffu;
    // (hi:lo) << 3 puts the exponent's low 8 bits above the 23 leading mantissa bits; in the FP32
    // normal range the rebias (exponent - 896) mod 256 is those 8 bits with the top one flipped
    unsigned r = ((__funnelshift_l(lo, hi, 3) & 0x7fffffffu) ^ 0x40000000u) | sign;
    r = a < 0x38100000u ? sign : r;                   // below the FP32 normal range: signed zero
    r = a >= 0x47f00000u ? (sign | 0x7f800000u) : r;  // beyond it: signed infinity
    return __uint_as_float(r);
}
__device__ __forceinline__ double f2d_exact(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned sign = b & 0x80000000u, a = b & 0x7fffffffu;
    // exponent and mantissa shifted into place with the exponent rebiased by 896 (1023 - 127)
    unsigned hi = ((a >> 3) + 0x38000000u) | sign, lo = b << 29;
    hi = a < 0x00800000u ? sign : hi;  // zero and denormals: signed zero
    lo = a < 0x00800000u ? 0u : lo;
    hi = a >= 0x7f800000u ? ((a >> 3) | 0x7ff00000u | sign) : hi;
    return __hiloint2double((int)hi, (int)lo);
}

// Square root and reciprocal.  Split path: the hardware approximations (MUFU, about 1-2 ulp), well
// inside the FP32 error budget of the fluxes.  FP64, 1D grids and the gas step (2D and 3D grids: rcp3,
// rsqrt3 and sqrt3 below): IEEE square root; the reciprocal is the hardware FP64 approximation refined by
// two Newton-Raphson steps r <- r + r (1 - x r), each of which squares the relative error (from below
// 2^-20 to below 2^-40, then to rounding): within an ulp or two of 1/x, not the correctly rounded
// quotient, which the FP64 path does not need (its bound against the oracle is 1e-12) and which costs
// several more FP64 operations.  x = 0, +-inf and FP64 denormals (flushed) give NaN.
__device__ __forceinline__ double sqrt_fast(double x) { return sqrt(x); }
__device__ __forceinline__ float sqrt_fast(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double rcp(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double e = fma(-x, r, 1.0);
    r = fma(r, e, r);
    e = fma(-x, r, 1.0);
    return fma(r, e, r);
}
// 1/sqrt(x) for normal x > 0, FP64: the hardware approximation refined by two Newton-Raphson steps for
// f(y) = y^-2 - x, y <- y + (y/2)(1 - x y^2), each of which squares the relative error (within an ulp or
// two of 1/sqrt(x); tested against CUDA's 1/sqrt).  x sqrt(x)^-1 is then the square root as well.
__device__ __forceinline__ double rsqrt_nr(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double r = __fma_rn(-__dmul_rn(x, y), y, 1.0);
    y = __fma_rn(__dmul_rn(0.5, y), r, y);
    r = __fma_rn(-__dmul_rn(x, y), y, 1.0);
    return __fma_rn(__dmul_rn(0.5, y), r, y);
}
// The FP64 kernels of two- and three-dimensional grids are bound by the FP64 pipe (one warp instruction per
// 64 cycles and SM sub-partition), so they refine the same hardware approximations (MUFU pipe, relative
// error below 2^-19) by one third-order step: r <- r (1 + e + e^2), e = 1 - x r, for the reciprocal (the
// error becomes e^3; three FP64 instructions against four for two Newton-Raphson steps), and
// y <- y + y r (1/2 + 3/8 r), r = 1 - x y^2, for the inverse square root (the dropped term is 5/16 r^3; five
// against eight).  Within an ulp or two; the special cases of rcp.
__device__ __forceinline__ double rcp3(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = __fma_rn(-x, r, 1.0);
    return __fma_rn(r, __fma_rn(e, e, e), r);
}
__device__ __forceinline__ double rsqrt3(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double r = __fma_rn(-__dmul_rn(x, y), y, 1.0);
    return __fma_rn(__dmul_rn(y, r), __fma_rn(r, 0.375, 0.5), y);
}
// sqrt(x) by the same step on x y ~ sqrt(x) (five instructions; CUDA's correctly rounded sqrt takes about
// twice as many and a slow path).  Zero and subnormal x give 0, +inf gives +inf, negative x NaN.
__device__ __forceinline__ double sqrt3(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double g = __dmul_rn(x, y);
    const double r = __fma_rn(-g, y, 1.0);
    const double s = __fma_rn(__dmul_rn(g, r), __fma_rn(r, 0.375, 0.5), g);
    const int hi = __double2hiint(x);
    return (hi & 0x7fffffff) < 0x00100000 ? 0.0 : (hi == 0x7ff00000 ? x : s);
}

// Comparisons of FP64 values by their bits, on the integer pipes (an FP64 comparison, minimum or maximum
// occupies the FP64 pipe like an addition).  Values of one sign are ordered as the integers their bits
// make; a NaN counts as larger than any number.
__device__ __forceinline__ unsigned long long mag_bits(double x)
{
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
// max(a, b, 0) and min(a, b, 0)
__device__ __forceinline__ double max0_d(double a, double b)
{
    const long long x = max(__double_as_longlong(a), 0ll), y = max(__double_as_longlong(b), 0ll);
    return __longlong_as_double(max(x, y));
}
__device__ __forceinline__ double min0_d(double a, double b)
{
    const unsigned long long s = 0x8000000000000000ull;
    const unsigned long long x = (unsigned long long)__double_as_longlong(a), y = (unsigned long long)__double_as_longlong(b);
    return __longlong_as_double((long long)max(x >= s ? x : 0ull, y >= s ? y : 0ull));
}
// x > 0 (false for NaN)
__device__ __forceinline__ bool pos_d(double x)
{
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool is_one_d(double x) { return __double_as_longlong(x) == 0x3ff0000000000000ll; }
// x > 1, and x > 1 - 2^-50 (true for +inf, false for NaN)
__device__ __forceinline__ bool above1_d(double x)
{
    const long long b = __double_as_longlong(x);
    return b > 0x3ff0000000000000ll && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool reaches1_d(double x)
{
    const long long b = __double_as_longlong(x);
    return b > 0x3ff0000000000000ll - 8 && b <= 0x7ff0000000000000ll;
}
// a < b (neither NaN)
__device__ __forceinline__ bool less_d(double a, double b)
{
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return (x ^ ((x >> 63) & 0x7fffffffffffffffll)) < (y ^ ((y >> 63) & 0x7fffffffffffffffll));
}
// minmod(a, b): the one nearer zero if both have the same sign, else 0 (and 0 if either is NaN)
__device__ __forceinline__ double minmod_d(double a, double b)
{
    const unsigned long long x = mag_bits(a), y = mag_bits(b);
    const bool none = (__double2hiint(a) ^ __double2hiint(b)) < 0 || max(x, y) > 0x7ff0000000000000ull;
    return none ? 0.0 : (x < y ? a : b);
}
__device__ __forceinline__ float rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Explicitly rounded arithmetic: never contracted into FMAs or reassociated by the compiler, so every
// inlined copy of an expression written with these rounds the same way.  Quantities that two tiles (or a
// tile's own cells and its halo) compute separately use them, so that both copies get the same bits
// (a face flux shared by two tiles, a uniform state that must stay uniform).
__device__ __forceinline__ float xmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double xmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float xadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double xadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float xfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double xfma(double a, double b, double c) { return __fma_rn(a, b, c); }

}  // namespace rhd
