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
// largest one and is otherwise cut, downwards, below 2^-55 of the largest value;
// the sum itself is exact and rounded once.  So the result is within half an ulp
// plus (sum of taps) 2^-55 max|F| of the exact combination.  Where the values
// share a few binades, as those of a resolved field do, that is far less than the
// roundings of a chain of FMAs over the same taps (each half an ulp of a partial
// sum): mean error below 1e-4 of the chain's on ripples of a per cent, 0.02 to 0.6
// on sines of 60 to 3 points, 0.7 on values doubling from point to point.  Where
// the values with the large taps lie binades below the others it is more: values
// growing e times a point 1.3 (first) and 2.2 times the chain's mean error (second
// difference, H = 3), 4 times a point 2.6 and 5.3, 16 times 11 and 44; that is 3
// and 28 times 2^-53 of the largest value.  Exact
// sums there (in 128 bits, on a branch of their own) were measured and left out:
// burnt gas whose fuel is rounding noise takes the branch in every window (flame
// of 16,384 points 949 -> 1,067 us for 50 steps, batched 20.2 -> 21.9 ms).
// The cut being downwards, a mirrored stencil need not give mirrored bits (nor
// does a chain of FMAs).
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

// x cut to FP32 (|x| < 2^128; below 2^-127 zero or a subnormal)
AT_HD float fx_float(double x)
{
    const uint32_t hi = fx_hi(x), ah = hi & 0x7fffffffu;
    const uint32_t b = ((fx_max(ah, 0x38000000u) - 0x38000000u) << 3) | (fx_lo(x) >> 29) | (hi & 0x80000000u);
    float f;
#ifdef __CUDA_ARCH__
    f = __uint_as_float(b);
#else
    std::memcpy(&f, &b, 4);
#endif
    return f;
}

AT_HD uint64_t fx_mulhi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)((unsigned __int128)a * b >> 64);
#endif
}

AT_HD int64_t fx_smulhi(int64_t a, int64_t b)
{
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (int64_t)((__int128)a * b >> 64);
#endif
}

AT_HD uint32_t fx_mulhi32(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }

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

// A double as a signed integer in units of 2^-FX_GUARD of its last place and its
// exponent field (in place, bits 20..30 of the high word).  A zero or subnormal
// has no implicit bit and the field of the smallest normal numbers, whose unit
// is its own.  Inf and NaN are their bits with an implicit one, marked by the field;
// fx_join gives them back like any other number.
struct FxV {
    int64_t m;
    uint32_t e;
};

template <int GUARD = FX_GUARD>
AT_HD FxV fx_split(double x)
{
    const uint32_t hi = fx_hi(x), t = hi & FX_EXP;
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | fx_min(t, 0x100000u)) << 32 | fx_lo(x)) << GUARD;
    const int64_t s = (int32_t)hi >> 31;
    return FxV{(int64_t)(m ^ (uint64_t)s) - s, fx_max(t, 0x100000u)};
}

// the double that fx_split took apart (the sign of a zero aside)
AT_HD double fx_join(FxV v)
{
    const uint64_t a = (v.m < 0 ? 0u - (uint64_t)v.m : (uint64_t)v.m) >> FX_GUARD;
    const uint32_t s = (uint32_t)((uint64_t)v.m >> 32) & 0x80000000u;
    const uint64_t x = a + ((uint64_t)((v.e - 0x100000u) | s) << 32);  // the implicit bit, if any, adds one to the field
    return fx_double((uint32_t)(x >> 32), (uint32_t)x);
}

// its integer at the exponent field emax (at least its own), cut downwards
AT_HD int64_t fx_at(FxV v, uint32_t emax) { return v.m >> fx_min((emax - v.e) >> 20, 63u); }

// fx_at of fx_split in fewer instructions, for values read once: i is the implicit
// bit, 0 for a subnormal, whose field then counts as 1
template <int GUARD>
AT_HD int64_t fx_align(double x, uint32_t emax)
{
    const uint32_t hi = fx_hi(x), t = hi & FX_EXP, i = fx_min(t, 0x100000u);
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | i) << 32 | fx_lo(x)) << GUARD;
    const int64_t s = (int32_t)hi >> 31;
    return ((int64_t)(m ^ (uint64_t)s) - s) >> fx_min((emax - 0x100000u - t + i) >> 20, 63u);
}

// the integer x in fx_at's units as a double, rounded to nearest; *ok is
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
// to the ends of the exponent range), the combination by FMAs.  Loops that stay
// loops: straight-line code could be predicated, and FP64 instructions take
// their issue slots also when off.
template <int H, int ORDER, class ROW>
AT_HD double fx_chain(const ROW& F)
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
        x = ::fma(t, fx_join(F[o]), x);
    }
    return x;
}

// A row around a point: F[o] the split value o points on.  Of doubles, split
// where they are read; or of values split once where they were formed (a
// mantissa and an exponent row), which leaves 8 of the 24 issue cycles a tap
// (the flame of 2^22 points 2.13 -> 1.99 ms per step, of 2,048 points 16.6 -> 15.7 us).
struct FxDoubles {
    const double* f;
    AT_HD FxV operator[](int o) const { return fx_split(f[o]); }
};
struct FxRow {
    const int64_t* m;
    const uint32_t* e;
    AT_HD FxV operator[](int o) const { return FxV{m[o], e[o]}; }
};

// D1 times the first difference at F[0]
template <int H, class ROW>
AT_HD double fx_d1(const ROW& F)
{
    FxV f[2 * H];
    uint32_t emax = 0;
#pragma unroll
    for (int o = 0; o < H; ++o) {
        f[2 * o] = F[o + 1];
        f[2 * o + 1] = F[-o - 1];
        emax = fx_max(emax, fx_max(f[2 * o].e, f[2 * o + 1].e));
    }
    int64_t x = 0;
#pragma unroll
    for (int o = 0; o < H; ++o) x += fx_t1<H>(o + 1) * (fx_at(f[2 * o], emax) - fx_at(f[2 * o + 1], emax));
    bool ok = emax != FX_EXP;
    double r = fx_result(x, emax, &ok);
    if (!ok) r = fx_chain<H, 1>(F);
    return r;
}

// D2 times the second difference at F[0]
template <int H, class ROW>
AT_HD double fx_d2(const ROW& F)
{
    const FxV f0 = F[0];
    FxV f[2 * H];
    uint32_t emax = f0.e;
#pragma unroll
    for (int o = 0; o < H; ++o) {
        f[2 * o] = F[o + 1];
        f[2 * o + 1] = F[-o - 1];
        emax = fx_max(emax, fx_max(f[2 * o].e, f[2 * o + 1].e));
    }
    const int64_t two0 = 2 * fx_at(f0, emax);
    int64_t x = 0, s[H];
    bool wide = false;
#pragma unroll
    for (int o = 0; o < H; ++o) {
        s[o] = fx_at(f[2 * o], emax) + fx_at(f[2 * o + 1], emax) - two0;
        // |s| <= 2^58; with the taps of H = 3 the sum stays below 2^63 when
        // |s_1| < 2^53 (an eighth of the largest value) and |s_2| < 2^57
        if (H == 3 && o < 2) {
            const int32_t sh = (int32_t)((uint64_t)s[o] >> 32);
            if ((uint32_t)(sh ^ (sh >> 31)) >= (o == 0 ? 1u << 21 : 1u << 25)) wide = true;
        }
        x += fx_t2<H>(o + 1) * s[o];
    }
    // beyond that (fronts of a point or two, noise) the sum, below 2^67, by halves
    // of 32 bits and in units of 2^5, 2^-50 of the largest value (the FMA chain in
    // its place: rows of noise 1.51 -> 0.94 ms per step of 2^21 points, 28.2 -> 22.9
    // us of 16,384, where FP64 throughout took 1.56 ms and 26.7 us)
    uint32_t ex = emax;
    if (H == 3 && wide) {
        int64_t xh = 0, xl = 0;
#pragma unroll
        for (int o = 0; o < H; ++o) {
            xh += fx_t2<H>(o + 1) * (s[o] >> 32);
            xl += (int64_t)fx_t2<H>(o + 1) * (uint32_t)s[o];
        }
        x = (xh << 27) + (xl >> 5);
        ex += 5u << 20;
    }
    bool ok = emax != FX_EXP;
    double r = fx_result(x, ex, &ok);
    if (!ok) r = fx_chain<H, 2>(F);
    return r;
}

// ---------------------------------------------------------------------------
// Products, sums and reciprocals of numbers with 64-bit mantissas: about 18 to
// 25 issue cycles each against 64 for an FP64 instruction.  m 2^e, cut towards
// zero; a zero's exponent lies below every other, so that nothing is shifted
// out beside it.
// ---------------------------------------------------------------------------
struct FxU {
    uint64_t m;
    int e;
};
struct FxS {
    int64_t m;
    int e;
};

constexpr int FX_TINY = -(1 << 20), FX_HUGE = 1 << 20;

AT_HD FxU fx_mul(FxU a, FxU b) { return FxU{fx_mulhi(a.m, b.m), a.e + b.e + 64}; }

AT_HD FxU fx_add(FxU a, FxU b)
{
    const int e = (a.e > b.e ? a.e : b.e) + 1;
    return FxU{(a.m >> fx_min((uint32_t)(e - a.e), 63u)) + (b.m >> fx_min((uint32_t)(e - b.e), 63u)), e};
}

AT_HD FxU fx_normal(FxU a)
{
    const int lz = fx_clz(a.m | 1u);
    return FxU{a.m << lz, a.e - lz};
}

// a nonnegative double; Inf and NaN have an exponent above every other, beside
// which nothing is left
AT_HD FxU fx_unpack(double x)
{
    const uint32_t hi = fx_hi(x), t = hi & FX_EXP;
    const uint64_t m = (uint64_t)((hi & 0xfffffu) | fx_min(t, 0x100000u)) << 32 | fx_lo(x);
    const FxU v = fx_normal(FxU{m << 11, (int)(fx_max(t, 0x100000u) >> 20) - 1086});
    return t == FX_EXP ? FxU{0, FX_HUGE} : (m == 0 ? FxU{0, FX_TINY} : v);
}

AT_HD double fx_pack(FxS a)
{
    const uint32_t s = (uint32_t)((uint64_t)a.m >> 32) & 0x80000000u;
    const uint64_t u = a.m < 0 ? 0u - (uint64_t)a.m : (uint64_t)a.m;
    const int lz = fx_clz(u | 1u);
    const uint64_t v = u << lz;
    const int e = a.e - lz + 1086;  // exponent field
    const uint64_t r = (v >> 11) + ((v >> 10) & 1u);
    uint32_t hi = (uint32_t)(r >> 32) + ((uint32_t)(e - 1) << 20), lo = (uint32_t)r;
    if (u == 0 || e < 1) hi = lo = 0u;         // below the normal range: zero
    if (e > 0x7fe) hi = 0x7ff00000u, lo = 0u;  // above it: infinity
    return fx_double(hi | s, lo);
}

// the bits of an FP32 number of about 1/2 to 1 in units of 2^-32
AT_HD uint32_t fx_seed(uint32_t rb)
{
    return rb >= 0x3f800000u ? 0xffffffffu : (fx_max(rb, 0x3f000000u) << 8) | 0x80000000u;
}

// 2^126 / m for a mantissa with bit 63 set, in [2^62, 2^63], relative error
// below 2^-60: two Newton steps r <- r + r (1 - m r) in integers from the
// hardware's approximate FP32 reciprocal (22 bits, then 43, then 60)
AT_HD uint64_t fx_recip(uint64_t m)
{
    const uint32_t mh = (uint32_t)(m >> 32);
    const uint32_t fb = 0x3f800000u | ((mh >> 8) & 0x7fffffu);
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(fb)));
    const uint32_t rb = __float_as_uint(r);
#else
    float f;
    std::memcpy(&f, &fb, 4);
    f = 1.0f / f;
    uint32_t rb;
    std::memcpy(&rb, &f, 4);
#endif
    const uint32_t r0 = fx_seed(rb);                                                 // units of 2^-32
    const uint64_t t = (uint64_t)mh * r0 + fx_mulhi32((uint32_t)m, r0);              // m r in units of 2^-63
    const int32_t e1 = (int32_t)((int64_t)(0x8000000000000000ull - t) >> 11);        // 1 - m r in units of 2^-52
    const int64_t c1 = (int64_t)e1 * (int32_t)(r0 >> 1);                             // units of 2^-83
    const uint64_t r1 = ((uint64_t)r0 << 31) + (uint64_t)(c1 >> 20);                 // units of 2^-63
    const int32_t e2 = (int32_t)(0x4000000000000000ll - (int64_t)fx_mulhi(m, r1));   // units of 2^-62
    const int64_t c2 = (int64_t)e2 * (int32_t)(r1 >> 33);                            // units of 2^-92
    return r1 + (uint64_t)(c2 >> 29);
}

// 1/x of a normal x whose reciprocal is normal, within half an ulp and 2^-60;
// *ok is cleared for every other x
AT_HD double fx_rcp(double x, bool* ok)
{
    const uint32_t hi = fx_hi(x), t = hi & FX_EXP;
    *ok = t - 0x100000u < 0x7fc00000u;  // exponent fields 1..2044
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | fx_lo(x)) << 11;
    const uint64_t r = fx_recip(m);  // 2^62 (x nearly twice a power of two) .. 2^63 (a power of two)
    const uint64_t v = (r >> 10) + ((r >> 9) & 1u);
    return fx_double((uint32_t)(v >> 32) + (0x7fc00000u - t) + (hi & 0x80000000u), (uint32_t)v);
}

// sqrt(x) of a positive normal x, within half an ulp and 2^-58: two Newton
// steps s <- s + (x - s^2) y / 2 in integers, y the hardware's approximate
// FP32 reciprocal root; *ok is cleared for every other x
AT_HD double fx_sqrt(double x, bool* ok)
{
    const uint32_t hi = fx_hi(x);
    *ok = hi - 0x100000u < 0x7fe00000u;
    // x = X 4^k, X in [1, 4) in units of 2^-62
    const uint32_t odd = 1u - ((hi >> 20) & 1u);  // 1: the unbiased exponent is odd
    const uint64_t X = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | fx_lo(x)) << (10 + odd);
    const uint32_t xh = (uint32_t)(X >> 32);
    const uint32_t fb = (0x3f800000u + (odd << 23)) | ((hi << 3) & 0x7fffffu) | (fx_lo(x) >> 29);
#ifdef __CUDA_ARCH__
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(fb)));
    const uint32_t rb = __float_as_uint(r);
#else
    float f;
    std::memcpy(&f, &fb, 4);
    f = 1.0f / std::sqrt(f);
    uint32_t rb;
    std::memcpy(&rb, &f, 4);
#endif
    const uint32_t y = fx_seed(rb);                                                     // units of 2^-32
    const uint64_t s1 = (uint64_t)xh * y + fx_mulhi32((uint32_t)X, y);                  // units of 2^-62
    const int32_t e1 = (int32_t)((int64_t)((X >> 2) - fx_mulhi(s1, s1)) >> 12);         // units of 2^-48
    const uint64_t s2 = s1 + (uint64_t)((int64_t)e1 * (int32_t)(y >> 1) >> 18);
    const int32_t e2 = (int32_t)((X >> 2) - fx_mulhi(s2, s2));                          // units of 2^-60
    const uint64_t s3 = s2 + (uint64_t)((int64_t)e2 * (int32_t)(y >> 1) >> 30);
    const uint64_t v = (s3 >> 10) + ((s3 >> 9) & 1u);  // implicit bit at 52
    return fx_double((uint32_t)(v >> 32) + ((((hi >> 20) + 1021u - odd) >> 1) << 20), (uint32_t)v);
}

// x / 2 (exact; what would be subnormal is zero)
AT_HD double fx_half(double x)
{
    const uint32_t hi = fx_hi(x), t = hi & FX_EXP;
    const bool in = t - 0x200000u < FX_EXP - 0x200000u;
    const bool keep = t == FX_EXP;
    return fx_double(in ? hi - 0x100000u : (keep ? hi : hi & 0x80000000u), in || keep ? fx_lo(x) : 0u);
}

// fmax of two numbers that are not negative (or not a number)
AT_HD double fx_fmax(double a, double b)
{
    const uint64_t inf = (uint64_t)FX_EXP << 32;
    const uint64_t ka = ((uint64_t)fx_hi(a) << 32 | fx_lo(a)) & 0x7fffffffffffffffull;
    const uint64_t kb = ((uint64_t)fx_hi(b) << 32 | fx_lo(b)) & 0x7fffffffffffffffull;
    return (kb > inf || (ka <= inf && ka >= kb)) ? a : b;
}

// the 64 leading bits of the nonnegative integer hi 2^64 + lo, times 2^e
AT_HD FxU fx_leading(uint64_t hi, uint64_t lo, int e)
{
    uint32_t w3 = (uint32_t)(hi >> 32), w2 = (uint32_t)hi, w1 = (uint32_t)(lo >> 32), w0 = (uint32_t)lo;
    e += 64;
#pragma unroll
    for (int i = 0; i < 3; ++i) {  // past leading zero words
        const bool z = w3 == 0;
        w3 = z ? w2 : w3;
        w2 = z ? w1 : w2;
        w1 = z ? w0 : w1;
        w0 = z ? 0u : w0;
        e -= z ? 32 : 0;
    }
#ifdef __CUDA_ARCH__
    const int lz = __clz((int)w3);  // 32 for zero
    const uint64_t m = (uint64_t)__funnelshift_l(w2, w3, lz) << 32 | __funnelshift_l(w1, w2, lz);
#else
    const int lz = w3 ? __builtin_clz(w3) : 32;
    const uint64_t m = (((uint64_t)w3 << 32 | w2) << lz) | (lz ? w1 >> (32 - lz) : 0u);
#endif
    return FxU{m, e - lz - ((lz & 32) << 15)};  // zero: 2^20 further down
}

// a in units of 2^e, less than 2^64 of them
AT_HD uint64_t fx_fixed(FxU a, int e)
{
    const int r = e - a.e;  // right shift
    return (a.m >> fx_min((uint32_t)(r > 0 ? r : 0), 63u)) << (r < 0 ? -r & 63 : 0);
}

// The sum of the corrections of the two WENO5 reconstructions of an edge, six
// times (sum of corrections) - (s_1+ + s_1-) of weno_flux, at_device.cuh,
// from the first differences c of C and q of hl Q at the columns c-2..c+2.
// With the ten differences aligned to their largest exponent (58 bits), the
// split differences q + c and q - c, the second and third differences and
// 3 beta_i = s (4 s + 3 a) + 3 a^2 are exact integers; 3 (eps + beta_i) then has
// a 64-bit mantissa of its own (62 bits or more of it used, also where beta_i is
// zero and eps alone is left), and with E_i its square, A = 3 E_0 and
// den = E_1 (A + E_2) + 2 A E_2 the correction is
//   (2 E_1 E_2 / den) (s_0 - s_1) + (E_1 A / den) (s_1 - s_2)
// (the threes cancel), the two weights as fixed-point numbers.  The products are
// not normalised: E_i keeps 60 bits or more, a product of two 55, a weight 53.
// About 1,600 issue cycles of integer work for an edge and variable stand beside
// seven FP64 instructions (448 cycles), in place of 66 of those (4,224).  Measured
// on GB300: the detonation of 2^23 points 10.77 -> 6.83 ms per RK3 step (16.3 with
// all of it in FP64), of 61,440 points 123 -> 91 us (168).  eps3 = 3 eps.  Not a
// number where a difference or eps is not (or is infinite), or where a
// denominator vanishes (eps = 0 and two indicators that are zero).
AT_HD double fx_weno_sum(const double* c, const double* q, FxU eps3)
{
    constexpr int G = 5;
    uint32_t emax = 0x100000u;
#pragma unroll
    for (int j = 0; j < 5; ++j) emax = fx_max(emax, fx_max(fx_hi(c[j]) & FX_EXP, fx_hi(q[j]) & FX_EXP));
    const int unit = (int)(emax >> 20) - 1075 - G;
    int64_t C[5], Q[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        C[j] = fx_align<G>(c[j], emax);  // below 2^58
        Q[j] = fx_align<G>(q[j], emax);
    }
    bool bad = emax == FX_EXP;
    int64_t sum = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        // f+ from the left, f- mirrored: a_1..a_4, below 2^59
        const int64_t a1 = s ? Q[4] - C[4] : Q[0] + C[0], a2 = s ? Q[3] - C[3] : Q[1] + C[1];
        const int64_t a3 = s ? Q[2] - C[2] : Q[2] + C[2], a4 = s ? Q[1] - C[1] : Q[3] + C[3];
        const int64_t s0 = a2 - a1, s1 = a3 - a2, s2 = a4 - a3;  // below 2^60
        const int64_t a2x3 = 3 * a2, a3x3 = 3 * a3;
        const uint64_t l2 = (uint64_t)a2 * (uint64_t)a2x3, l3 = (uint64_t)a3 * (uint64_t)a3x3;
        const int64_t h2 = fx_smulhi(a2, a2x3), h3 = fx_smulhi(a3, a3x3);
        FxU d[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int64_t si = i == 0 ? s0 : (i == 1 ? s1 : s2);
            const int64_t ti = 4 * si + (i < 2 ? a2x3 : -a3x3);  // below 2^63
            const uint64_t l = (uint64_t)si * (uint64_t)ti, lo = l + (i < 2 ? l2 : l3);
            const int64_t hi = fx_smulhi(si, ti) + (i < 2 ? h2 : h3) + (lo < l ? 1 : 0);
            d[i] = fx_add(fx_leading((uint64_t)hi, lo, 2 * unit), eps3);
        }
        const FxU e0 = fx_mul(d[0], d[0]), e1 = fx_mul(d[1], d[1]), e2 = fx_mul(d[2], d[2]);
        const FxU A{(e0.m >> 2) * 3u, e0.e + 2};
        const FxU we = fx_mul(e1, e2), wa = fx_mul(e1, A);  // E_1 E_2, E_1 A
        FxU den = fx_mul(A, e2);
        den.e += 1;  // A B
        den = fx_normal(fx_add(fx_add(we, wa), den));
        bad |= den.m == 0;
        const FxU r{fx_recip(den.m | 0x8000000000000000ull), -126 - den.e};
        // the weights 2 E_1 E_2 / den (at most 2) and E_1 A / den (at most 1) in
        // units of 2^-61, times the third differences in units of 1/4: halves
        const uint64_t w0 = fx_fixed(fx_mul(we, r), -62), w2 = fx_fixed(fx_mul(wa, r), -61);
        const int64_t h = fx_smulhi((s0 - s1) * 4, (int64_t)w0) + fx_smulhi((s1 - s2) * 4, (int64_t)w2);
        sum += 2 * h - s1;
    }
    const double v = fx_pack(FxS{sum, unit});
    return bad ? fx_double(0x7ff80000u, 0u) : v;
}

} // namespace atk
