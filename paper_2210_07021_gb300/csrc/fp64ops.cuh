// FP64 building blocks of the pair loops.  This GPU's FP64 pipe takes one warp
// instruction in about 19 cycles per SM (1.05 TFLOP/s measured), 64 times the
// FP32 and integer pipes' cost, so a pair loop in FP64 costs what its FP64
// instructions cost: everything that does not need the FP64 pipe (range tests,
// exponents, seeds, small correction terms) runs on the other pipes here.
//
// Reciprocal: the MUFU seed r0 of rcp.approx.ftz.f64 (relative error below
// 2^-19) and e = 1 - d r0, so 1/d = r0 (1 + e + e^2 + ...) with the series cut
// after e^2 (error e^3 < 2^-57): three FP64 instructions after the seed.
//
// Logarithm: sums of q log d^2 run over products.  The mantissas of consecutive
// d^2 of equal mass are multiplied, their exponents summed as integers, and one
// logarithm is taken where the mass changes or the run ends: one FP64 multiply
// per pair of equal masses.  The logarithm of the product is table-driven (Tang,
// ACM TOMS 16, 1990): m in [1, 2), c_j the midpoint of m's 1/128 interval,
// r = m / c_j - 1, |r| < 2^-7.9, log m = log c_j + r - r^2/2 + r^3/3 + r^4 g(r); g is
// a polynomial in FP32 (r^4/4 < 2^-33, so its rounding stays below 2^-56).
//
// Errors.  A term q/d^2 has about 1.5 units in the last place where a division had 1/2, but
// the sums it goes into have fewer roundings: the logarithms of a run are one, and the mass
// is not summed pair by pair.  Near fields alone (40, 300 and 2000 sources; wide and arcminute
// skies; equal, lognormal and signed masses; half of the targets on sources) against 80-bit
// sums, before -> now: psi, rms 1.5e-16 .. 4.8e-14 -> 1.1e-16 .. 3.9e-15 (0.03 to 1.00 of
// before), alpha 2.0e-16 .. 1.0e-14 -> 1.6e-16 .. 1.3e-15 (0.12 to 0.83).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace sfmm {

constexpr int LOG64_N = 128;                 // table: (1/c_j, log c_j) for j < 128
constexpr int F64_HI_MIN = (1023 - 900) << 20;     // high word of 2^-900: the fast paths' smallest d^2
constexpr int F64_HI_INF = 0x7ff00000;

// 2^-900 <= d < infinity (and not a NaN), on the integer pipe
__device__ __forceinline__ bool f64_plain(double d)
{
    return (unsigned)(__double2hiint(d) - F64_HI_MIN) < (unsigned)(F64_HI_INF - F64_HI_MIN);
}
__device__ __forceinline__ bool f64_same(double a, double b)
{
    return __double_as_longlong(a) == __double_as_longlong(b);
}
__device__ __forceinline__ double rcp_seed(double d)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    return r;
}
// r0 and u = e + e^2 with 1/d = r0 (1 + u)
__device__ __forceinline__ double rcp_series(double d, double* u)
{
    const double r0 = rcp_seed(d);
    const double e = fma(-d, r0, 1.0);
    *u = fma(e, e, e);
    return r0;
}

// conversions of values in the normal FP32 range on the integer pipe (truncating)
__device__ __forceinline__ float f64_to_f32_bits(double d)
{
    const int hi = __double2hiint(d), lo = __double2loint(d);
    const int ex = (hi >> 20) & 0x7ff;
    const unsigned f = ((unsigned)(ex - 896) << 23) | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)lo >> 29);
    return ex > 896 ? __uint_as_float(f | ((unsigned)hi & 0x80000000u)) : 0.f;
}
__device__ __forceinline__ double f32_to_f64_bits(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned ex = (b >> 23) & 0xffu;
    const unsigned hi = (b & 0x80000000u) | ((ex + 896u) << 20) | ((b >> 3) & 0xfffffu);
    return ex ? __hiloint2double((int)hi, (int)(b << 29)) : 0.0;
}

// log(m 2^k) for m in [1, 2)
__device__ __forceinline__ double log_mk(double m, int k, const double2* __restrict__ tab)
{
    const double2 t = tab[(__double2hiint(m) >> 13) & (LOG64_N - 1)];     // the leading seven fraction bits
    const double r = fma(m, t.x, -1.0);
    const float x = f64_to_f32_bits(r);
    const float x2 = x * x;
    const float g = (x2 * x2) * (-0.25f + x * (0.2f + x * (-1.f / 6.f + x * (1.f / 7.f))));
    const double a = fma(r, 1.0 / 3.0, -0.5);
    const double p = fma(r * r, a, f32_to_f64_bits(g));
    // k as a double: 2^52 + 2^31 + k has k's bits in its low word
    const double kd = __hiloint2double(0x43300000, (int)(0x80000000u + (unsigned)k)) - 4503601774854144.0;
    return fma(kd, 0.69314718055994530942, t.y) + (r + p);
}

// sum of q log d^2 over pairs taken one after another
struct LogSum {
    double sum, prod, q;      // finished runs; mantissa product in [1, 2) of the open run and its mass
    int k;                    // its exponent
    __device__ __forceinline__ void init() { sum = 0.0; prod = 1.0; q = 0.0; k = 0; }
    __device__ __forceinline__ void flush(const double2* __restrict__ tab)
    {
        sum = fma(q, log_mk(prod, k, tab), sum);
        prod = 1.0;
        k = 0;
    }
    // d2: plain (f64_plain), positive
    __device__ __forceinline__ void add(double qj, double d2, const double2* __restrict__ tab)
    {
        if (!f64_same(qj, q)) {
            flush(tab);
            q = qj;
        }
        const int hi = __double2hiint(d2);
        prod *= __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(d2));
        const int ph = __double2hiint(prod);                  // product in [1, 4): back to [1, 2)
        k += (hi >> 20) + (ph >> 20) - 2046;
        prod = __hiloint2double((ph & 0xfffff) | 0x3ff00000, __double2loint(prod));
    }
};

}  // namespace sfmm
