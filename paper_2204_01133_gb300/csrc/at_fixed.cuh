// at_fixed.cuh -- central differences of FP64 rows in 64-bit integers.
//
// GB300 issues one FP64 warp instruction per SM sub-partition every 64 cycles
// and an integer one every one to two (measured: DFMA, DADD, DMUL and every
// conversion from or to double 64, add or logic 1.1-1.4, shift or multiply 2,
// 64-bit add 2.3).  A 6th-order first and second derivative of one row took 13
// FP64 instructions, 832 cycles.  Here the taps are what they are, small
// integers over a common denominator: the values of one stencil are aligned to
// the largest exponent among them as signed integers, the integer combination
// is formed exactly, and one normalisation turns it into a double, to be
// scaled by one FP64 multiply: a few hundred issue cycles a derivative pair
// that the FP64 unit does not see.
//
// Accuracy: a value keeps all its bits while its exponent is within 3 of the
// largest one and is cut below 2^-55 of the largest value otherwise; the sum
// itself is exact and rounded once.  So the result is within half an ulp plus
// (sum of taps) 2^-55 max|F| of the exact combination, less than the roundings
// of a chain of FMAs over the same taps (each half an ulp of a partial sum).
//
// The result is a function of the stencil's values alone, the same on every
// path whatever window or strip the stencil is part of.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define AT_HD __host__ __device__ __forceinline__
#else
#define AT_HD inline
#endif

namespace atk {

AT_HD uint32_t fx_hi(double x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2hiint(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return (uint32_t)(b >> 32);
#endif
}

AT_HD uint32_t fx_lo(double x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2loint(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return (uint32_t)b;
#endif
}

AT_HD double fx_double(uint32_t hi, uint32_t lo)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = (uint64_t)hi << 32 | lo;
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}

AT_HD uint32_t fx_max(uint32_t a, uint32_t b) { return a > b ? a : b; }
AT_HD uint32_t fx_min(uint32_t a, uint32_t b) { return a < b ? a : b; }

// leading zeros of a nonzero 64-bit integer
AT_HD int fx_clz(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}

constexpr uint32_t FX_EXP = 0x7ff00000u;
constexpr int FX_GUARD = 3;  // bits kept below the last bit of the largest value

// x as a signed integer in units of 2^-FX_GUARD ulp at the exponent field
// emax (>= x's own; in place, bits 20..30 of the high word), cut towards zero;
// a zero or subnormal has no implicit bit
AT_HD int64_t fx_align(double x, uint32_t emax)
{
    const uint32_t hi = fx_hi(x), t = hi & FX_EXP;
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | fx_min(t, 0x100000u)) << 32 | fx_lo(x)) << FX_GUARD;
    const uint64_t v = m >> fx_min((emax - t) >> 20, 63u);
    const int64_t s = (int32_t)hi >> 31;
    return (int64_t)(v ^ (uint64_t)s) - s;
}

// the integer x in fx_align's units as a double, rounded to nearest; *ok is
// cleared where the result is not a normal number or zero
AT_HD double fx_result(int64_t x, uint32_t emax, bool* ok)
{
    const uint32_t s = (uint32_t)((uint64_t)x >> 32) & 0x80000000u;
    const uint64_t a = x < 0 ? 0u - (uint64_t)x : (uint64_t)x;
    const int lz = fx_clz(a | 1u);
    const uint64_t v = a << lz;  // bit 63 set unless x = 0
    const int e = (int)(emax >> 20) - lz + (63 - 52 - FX_GUARD);  // exponent field of the result
    if (a != 0 && (unsigned)(e - 1) >= 0x7fdu) *ok = false;
    const uint64_t r = (v >> 11) + ((v >> 10) & 1u);  // implicit bit at 52; a carry moves into the exponent
    const uint32_t hi = a == 0 ? 0u : ((uint32_t)(r >> 32) + ((uint32_t)(e - 1) << 20)) | s;
    return fx_double(hi, (uint32_t)r);
}

// the taps: first derivative sum_o t1(o) (F_o - F_-o) / D1, second derivative
// sum_o t2(o) (F_o - 2 F_0 + F_-o) / D2, o = 1..H
template <int H>
AT_HD constexpr int fx_t1(int o)
{
    return H == 3 ? (o == 1 ? 45 : (o == 2 ? -9 : 1)) : (H == 2 ? (o == 1 ? 8 : -1) : 1);
}
template <int H>
AT_HD constexpr int fx_t2(int o)
{
    return H == 3 ? (o == 1 ? 270 : (o == 2 ? -27 : 2)) : (H == 2 ? (o == 1 ? 16 : -1) : 1);
}

// Where the integers do not apply (Inf or NaN among the values, results next
// to the ends of the exponent range, second differences that could overflow),
// the combination by FMAs.  Loops that stay loops: straight-line code could be
// predicated, and FP64 instructions take their issue slots also when off.
template <int H, int ORDER>
AT_HD double fx_chain(const double* F)
{
    double x = 0.0;
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
    for (int o = -H; o <= H; ++o) {
        double t;
        if (ORDER == 1) {
            if (o == 0) continue;
            t = o > 0 ? (double)fx_t1<H>(o) : -(double)fx_t1<H>(-o);
        } else {
            t = o == 0 ? (H == 3 ? -490.0 : (H == 2 ? -30.0 : -2.0)) : (double)fx_t2<H>(o > 0 ? o : -o);
        }
        x = ::fma(t, F[o], x);
    }
    return x;
}

// D1 times the first difference at F[0]
template <int H>
AT_HD double fx_d1(const double* F)
{
    double f[2 * H];
    uint32_t emax = 0;
#pragma unroll
    for (int o = 0; o < H; ++o) {
        f[2 * o] = F[o + 1];
        f[2 * o + 1] = F[-o - 1];
        emax = fx_max(emax, fx_max(fx_hi(f[2 * o]) & FX_EXP, fx_hi(f[2 * o + 1]) & FX_EXP));
    }
    int64_t x = 0;
#pragma unroll
    for (int o = 0; o < H; ++o)
        x += fx_t1<H>(o + 1) * (fx_align(f[2 * o], emax) - fx_align(f[2 * o + 1], emax));
    bool ok = emax != FX_EXP;
    double r = fx_result(x, emax, &ok);
    if (!ok) r = fx_chain<H, 1>(F);
    return r;
}

// D2 times the second difference at F[0]
template <int H>
AT_HD double fx_d2(const double* F)
{
    const double f0 = F[0];
    double f[2 * H];
    uint32_t emax = fx_hi(f0) & FX_EXP;
#pragma unroll
    for (int o = 0; o < H; ++o) {
        f[2 * o] = F[o + 1];
        f[2 * o + 1] = F[-o - 1];
        emax = fx_max(emax, fx_max(fx_hi(f[2 * o]) & FX_EXP, fx_hi(f[2 * o + 1]) & FX_EXP));
    }
    const int64_t two0 = 2 * fx_align(f0, emax);
    bool ok = emax != FX_EXP;
    int64_t x = 0;
#pragma unroll
    for (int o = 0; o < H; ++o) {
        const int64_t s = fx_align(f[2 * o], emax) + fx_align(f[2 * o + 1], emax) - two0;
        // |s| < 2^58; with the taps of H = 3 the sum stays below 2^63 when
        // |s_1| < 2^53 (an eighth of the largest value) and |s_2| < 2^57
        if (H == 3 && o < 2) {
            const int32_t sh = (int32_t)((uint64_t)s >> 32);
            if ((uint32_t)(sh ^ (sh >> 31)) >= (o == 0 ? 1u << 21 : 1u << 25)) ok = false;
        }
        x += fx_t2<H>(o + 1) * s;
    }
    double r = fx_result(x, emax, &ok);
    if (!ok) r = fx_chain<H, 2>(F);
    return r;
}

} // namespace atk
