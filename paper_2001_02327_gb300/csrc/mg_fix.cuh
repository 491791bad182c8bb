// mg_fix.cuh -- sums of doubles on the integer pipe.
//
// The part issues one FP64 instruction per sub-partition every 64 to 77 cycles,
// a 64-bit integer addition every 2.3 (measured: DADD 76, DFMA 65, 64-bit add
// 2.3, 64-bit shift 5, count of leading zeros 11 cycles a warp).  A sum of n
// doubles with small integer weights is therefore formed from their mantissas,
// aligned to the largest exponent with P bits below its last place, and rounded
// once: about 16 integer instructions a term and 25 for the result, against 64
// cycles an FP64 addition.  The sum is exact but for bits more than P places
// below the last place of the largest term, so its error is below that of the
// additions it replaces, each of which rounds.  Terms outside the plain range
// of exponents (fx_ok: zero, denormal, huge, infinite or NaN as the largest)
// take the FP64 instructions.
#pragma once

#include <cuda_runtime.h>

// The FP64 instructions of the rare branches sit in functions of their own: a
// short branch is otherwise predicated, and an instruction that no lane
// executes still takes its 64 cycles of the FP64 pipe (measured: 7 instead of
// 2 of them an update).
static __device__ __noinline__ double fx_rare_add(double a, double b) { return a + b; }
static __device__ __noinline__ double fx_rare_mul(double a, double b) { return a * b; }
static __device__ __noinline__ double fx_rare_nsum2(double a, double b, double c, double d) { return (a + b) + (c + d); }
static __device__ __noinline__ double fx_rare_nsum3(double a, double b, double c, double d, double e, double f)
{
    return ((a + b) + (c + d)) + (e + f);
}
static __device__ __noinline__ double fx_rare_diff4(double a, double b, double c, double d)
{
    return 8.0 * (a - b) - (c - d);
}
static __device__ __noinline__ float fx_rare_float(double x) { return (float)x; }

__device__ __forceinline__ int fx_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// largest exponent for which the integer sums and the rounding below hold
__device__ __forceinline__ bool fx_ok(int emax) { return (unsigned)(emax - 128) < 1792u; }

// x as an integer multiple of 2^(emax - 1023 - 52 - P), truncated; |x| < 2^(53 + P)
template <int P>
__device__ __forceinline__ long long fx_align(double x, int emax)
{
    const int hi = __double2hiint(x);
    const unsigned long long m =
        ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
    const long long t = (long long)((m << P) >> min(emax - ((hi >> 20) & 0x7ff), 63));
    const long long s = hi >> 31;
    return (t ^ s) - s;
}

// s * 2^(emax - 1023 - 52 - P) rounded to nearest (ties away from zero); emax as fx_ok
template <int P>
__device__ __forceinline__ double fx_round(long long s, int emax)
{
    const unsigned long long a = s < 0 ? 0ull - (unsigned long long)s : (unsigned long long)s;
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << (lz & 63);
    const unsigned long long q = (n >> 11) + ((n >> 10) & 1);      // 2^52 .. 2^53
    const int e = 63 - lz + emax - 52 - P;
    unsigned long long bits = ((unsigned long long)(unsigned)(e - 1) << 52) + q;   // the carry of 2^53 reaches the exponent
    bits |= (unsigned long long)s & 0x8000000000000000ull;
    return a ? __longlong_as_double((long long)bits) : 0.0;
}

// (float)x, round to nearest even, without the FP64 pipe where x and the result are normal numbers
__device__ __forceinline__ float fx_to_float(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    if ((unsigned)(e - 898) >= 250u)
        return fx_rare_float(x);
    unsigned long long v = (b & 0x7fffffffffffffffull) - (896ull << 52);
    v += 0x0fffffffull + ((v >> 29) & 1);
    return __uint_as_float((unsigned)(v >> 29) | ((unsigned)(b >> 32) & 0x80000000u));
}

// Neighbour sum of the 5/7-point Laplacian: v[0..2 DIM)
template <int DIM>
__device__ __forceinline__ double fx_nsum(const double (&v)[2 * DIM])
{
    int e = fx_exp(v[0]);
#pragma unroll
    for (int q = 1; q < 2 * DIM; q++)
        e = max(e, fx_exp(v[q]));
    if (!fx_ok(e))
        return DIM == 3 ? fx_rare_nsum3(v[0], v[1], v[2], v[3], v[2 * DIM - 2], v[2 * DIM - 1])
                        : fx_rare_nsum2(v[0], v[1], v[2], v[3]);
    long long s = 0;
#pragma unroll
    for (int q = 0; q < 2 * DIM; q++)
        s += fx_align<7>(v[q], e);
    return fx_round<7>(s, e);
}

// Neighbour sum minus 2 DIM times the centre
template <int DIM>
__device__ __forceinline__ double fx_lap(const double (&v)[2 * DIM], double c)
{
    int e = fx_exp(c);
#pragma unroll
    for (int q = 0; q < 2 * DIM; q++)
        e = max(e, fx_exp(v[q]));
    if (!fx_ok(e))
        return fx_rare_add(DIM == 3 ? fx_rare_nsum3(v[0], v[1], v[2], v[3], v[2 * DIM - 2], v[2 * DIM - 1])
                                    : fx_rare_nsum2(v[0], v[1], v[2], v[3]),
                           fx_rare_mul(-2.0 * DIM, c));
    long long s = -(2 * DIM) * fx_align<6>(c, e);
#pragma unroll
    for (int q = 0; q < 2 * DIM; q++)
        s += fx_align<6>(v[q], e);
    return fx_round<6>(s, e);
}

// sum of 2^DIM values with weights w[axis][0 / 1], one axis at a time (x first)
static __device__ __noinline__ double fx_rare_mix2(double v0, double v1, double v2, double v3, double w0, double w1,
                                                   double y0, double y1)
{
    const double a = w0 * v0 + w1 * v1, b = w0 * v2 + w1 * v3;
    return y0 * a + y1 * b;
}

// Linear interpolation between 2^DIM values (x lowest bit): per axis weights 3/4
// and 1/4, the larger to the second value where far[a]
template <int DIM>
__device__ __forceinline__ double fx_interp(const double (&v)[1 << DIM], const bool (&far)[3])
{
    int e = 0;
#pragma unroll
    for (int m = 0; m < (1 << DIM); m++)
        e = max(e, fx_exp(v[m]));
    if (fx_ok(e)) {
        long long s[1 << DIM];
#pragma unroll
        for (int m = 0; m < (1 << DIM); m++)
            s[m] = fx_align<4>(v[m], e);   // weights of 4^DIM in all: below 2^(6 + 57)
        int a = 0;
#pragma unroll
        for (int n = (1 << DIM) / 2; n >= 1; n /= 2, a++)
#pragma unroll
            for (int m = 0; m < n; m++) {
                const long long x = s[2 * m], y = s[2 * m + 1];
                s[m] = x + y + 2 * (far[a] ? y : x);
            }
        return fx_round<4 + 2 * DIM>(s[0], e);
    }
    double z[2] = {};
#pragma unroll
    for (int k = 0; k < (DIM == 3 ? 2 : 1); k++)
        z[k] = fx_rare_mix2(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3], far[0] ? 0.25 : 0.75,
                            far[0] ? 0.75 : 0.25, far[1] ? 0.25 : 0.75, far[1] ? 0.75 : 0.25);
    return DIM == 3 ? fx_rare_add(fx_rare_mul(far[2] ? 0.25 : 0.75, z[0]), fx_rare_mul(far[2] ? 0.75 : 0.25, z[1])) : z[0];
}

// 8 (a - b) - (c - d), the numerator of the fourth-order difference: exact and
// rounded once where no term loses bits, else by the FP64 instructions (the
// terms may cancel, so a bound by the largest of them would not do)
__device__ __forceinline__ double fx_diff4(double a, double b, double c, double d)
{
    const int ea = fx_exp(a), eb = fx_exp(b), ec = fx_exp(c), ed = fx_exp(d);
    const int e = max(max(ea, eb), max(ec, ed));
    if (!fx_ok(e) || min(min(ea, eb), min(ec, ed)) < e - 5)
        return fx_rare_diff4(a, b, c, d);
    return fx_round<5>(8 * (fx_align<5>(a, e) - fx_align<5>(b, e)) - (fx_align<5>(c, e) - fx_align<5>(d, e)), e);
}
