// fixed.cuh -- fixed-point arithmetic of the FP64 deposits.
//
// The FP64 pipe of sm_103a takes one warp instruction per 64 clocks and SM
// sub-partition; a 32 x 32 + 64 bit multiply-add takes two (measured: FMA,
// add and conversion 64 to 77 clocks, mad.wide 2.1, 64-bit add 2.05).  The
// weighted sums of Eq. 4 are sums of products of numbers in [0, 1] (weights)
// and marker values, so they are formed in 64-bit integers, each factor in
// two limbs of 28 low bits and the rest:
//   weights of a (column, v_x row) pair     2^-57     (FX_A)
//   (v_y, v_z) cell weights                 2^-56     (FX_Q)
//   marker values                           2^(el - 1078), el the exponent
//                                           field of the largest value that
//                                           reaches the row in the column
//   sums of products                        h + m 2^-28 units of 2^-57
// The low limbs are signed, so that the product of two of them, which is
// left out, is at most a quarter of the sum's unit, of either sign.  The units
// are absolute, so what would reach a cell with a small weight only, and values
// outside FX_EMIN .. FX_EMAX, are summed in FP64 instead (k_pd3x, k_pd1x,
// k_ad_depx).  Against exact rational sums of 4 to 12 markers with values over
// one e-fold: f 7e-17 rms, weights 5e-17 (the same sums in FP64: 1.3e-16 and
// 1e-16).  In the least favourable cell,
// one reached by one weight just above the kernel's limit, n is within 2^-36
// (k_pd3x), 2^-33 (k_pd1x) and 2^-41 (k_ad_depx) of itself; f within 2^-36
// (k_pd3x, whose numerators are rounded apart from its weights), and to FP64's
// rounding in the other two, which take the same weights above and below.
#pragma once
#include <cuda_runtime.h>

namespace avl {

constexpr long long FX_ONE = 1ll << 52;       // 1 of a 52-bit fraction (position, row weights)
constexpr int FX_LIMB = 28;
constexpr int FX_PAIRS = 56;                  // products of weights <= 1 a sum takes before it is flushed:
                                              // |h| stays below 56 2^57 + 2^59, |m| below 56 (2^56 + 2^55)
constexpr int FX_EMIN = 96, FX_EMAX = 2040;   // exponent fields of the values that the sums take: theirs (units of
                                              // at least 2^-983, magnitudes below 2^1024) are normal numbers, also
                                              // with 26 bits below the unit

// v = h 2^28 + l, -2^27 <= l < 2^27
struct Limbs {
    int h, l;
};
__device__ __forceinline__ Limbs fx_split(long long v)
{
    const int l = ((int)v << (32 - FX_LIMB)) >> (32 - FX_LIMB);
    return {(int)(v >> FX_LIMB) + (l < 0 ? 1 : 0), l};
}

// c += a b.  The product and the sum as two PTX instructions with the
// accumulator updated in place, which become one multiply-add: 48 of them
// take 114 clocks and 60 instructions of a warp; as mad.wide.s32 153 clocks
// and 124 instructions, from c += (long long)a * b 197 and 166.
__device__ __forceinline__ void mad_wide(long long& c, int a, int b)
{
    long long t;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(t) : "r"(a), "r"(b));
    asm("add.s64 %0, %0, %1;" : "+l"(c) : "l"(t));
}

// a b / 2^56, to nearest but for the product of the low limbs (at most a
// quarter unit); exact for a = 0 or b = 0, and never negative for a, b >= 0
__device__ __forceinline__ long long fx_mul(Limbs a, Limbs b)
{
    long long m = 1ll << (FX_LIMB - 1);
    mad_wide(m, a.h, b.l);
    mad_wide(m, a.l, b.h);
    long long h = m >> FX_LIMB;
    mad_wide(h, a.h, b.h);
    return h;
}

// sum of products, h + m 2^-28
struct FxSum {
    long long h, m;
    __device__ __forceinline__ void clear() { h = m = 0; }
    __device__ __forceinline__ void add(Limbs a, Limbs b)
    {
        mad_wide(h, a.h, b.h);
        mad_wide(m, a.h, b.l);
        mad_wide(m, a.l, b.h);
    }
    // whole units, to nearest
    __device__ __forceinline__ long long units() const { return h + ((m + (1 << (FX_LIMB - 1))) >> FX_LIMB); }
};

// f as mant 2^(e - 1078), |mant| < 2^56, e >= 1 the exponent field of f
__device__ __forceinline__ long long fx_value(double f, int& e)
{
    const long long b = __double_as_longlong(f);
    const int ef = (int)(b >> 52) & 0x7ff;
    long long m = b & (FX_ONE - 1);
    if (ef) m |= FX_ONE;
    e = max(ef, 1);
    m <<= 3;
    return b < 0 ? -m : m;
}

// whether the sums take a value with exponent field e
__device__ __forceinline__ bool fx_in_range(int e) { return e >= FX_EMIN && e <= FX_EMAX; }

// t in counts of 2^-52, to nearest, without the FP64 pipe for |t| < 1024;
// saturates, NaN gives 0
__device__ __forceinline__ long long fx_count(double t)
{
    const long long b = __double_as_longlong(t);
    const int s = 1032 - ((int)(b >> 52) & 0x7ff);   // t 2^53 = (mantissa 2^10) 2^-s
    if (s < 0) return __double2ll_rn(t * 4503599627370496.0);
    const unsigned long long m = (unsigned long long)((b & (FX_ONE - 1)) | FX_ONE) << 10;
    const long long r = (long long)(((m >> min(s, 63)) + 1) >> 1);
    return b < 0 ? -r : r;
}

// an integer as FP64, to nearest, without the FP64 pipe
__device__ __forceinline__ double fx_double(unsigned long long a)
{
    if (a == 0) return 0.0;
    const int z = __clzll((long long)a);
    const unsigned long long t = a << z;                       // top bit set
    // exponent field of the top bit, less the bit itself; the rounding carry
    // runs into the exponent as it should
    return __longlong_as_double((long long)(((unsigned long long)(1085 - z) << 52) + ((t >> 11) + ((t >> 10) & 1ull))));
}
__device__ __forceinline__ double fx_double(long long v)
{
    const long long r = __double_as_longlong(fx_double(v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v));
    return __longlong_as_double(v < 0 ? r | (long long)0x8000000000000000ull : r);
}

// an FP32 value as FP64, without the FP64 pipe for zeros and normal numbers
__device__ __forceinline__ double fx_widen(float v)
{
    const unsigned b = (unsigned)__float_as_int(v), m = b & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0) return (double)v;   // subnormal, Inf, NaN
    return __hiloint2double((int)((b & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u)), (int)(b << 29));
}

// lesser of a weight w (a count of 2^-52) and 1 - w, but 1 for w = 0, whose
// corner takes nothing (at least 0 and less than 2^-32 below)
__device__ __forceinline__ float lesser_weight(long long w)
{
    const unsigned a = (unsigned)(w >> 20);
    return w == 0 ? 1.0f : (float)min(a, ~a) * 2.3283064365386963e-10f;   // 2^-32
}

// FP64 value of the weight of the next row or column, or of this one
__device__ __forceinline__ double weight_of(long long w, bool next) { return fx_double(next ? w : FX_ONE - w); }

// d 2^k for a normal result (d = 0 stays 0)
__device__ __forceinline__ double fx_scale(double d, int k)
{
    const long long b = __double_as_longlong(d);
    return __longlong_as_double(b + ((b & 0x7fffffffffffffffll) ? (long long)k << 52 : 0ll));
}

// n / d for a normal d > 0, in integers: a 24-bit reciprocal of d's mantissa
// from the FP32 approximation, one Newton-Raphson step to 30 bits, the
// quotient's first 29 bits, one correction by the exact remainder (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000
// processor", IBM J. Res. Dev. 34, 1990, the same scheme in floating point),
// which leaves 0.55 units in the last place, and a second one to the nearest.
// Operands or quotients that are not normal numbers take the division
// operator.
__device__ __forceinline__ double fx_div(double n, double d)
{
    const long long bn = __double_as_longlong(n), bd = __double_as_longlong(d);
    const int en = (int)(bn >> 52) & 0x7ff, ed = (int)(bd >> 52);
    int ex = en - ed + 1023;
    if (en == 0 || en == 0x7ff || ed <= 0 || ed >= 0x7ff || ex < 2 || ex > 0x7fd) return n / d;
    const unsigned long long N = (unsigned long long)((bn & (FX_ONE - 1)) | FX_ONE);
    const unsigned long long D = (unsigned long long)((bd & (FX_ONE - 1)) | FX_ONE);
    // 1 / (D 2^-52) in (1/2, 1]: R0 2^-24, then R1 2^-31
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__int_as_float(0x3f800000 | (int)((D >> 29) & 0x7fffff))));
    const int R0 = (__float_as_int(fminf(r, 0.99999994f)) & 0x7fffff) | 0x800000;
    const unsigned Dh = (unsigned)(D >> 21);
    const int e = (int)(((1ll << 55) - (long long)((unsigned long long)Dh * (unsigned)R0)) >> 23);
    const unsigned R1 = ((unsigned)R0 << 7) + (unsigned)(int)(((long long)R0 * e) >> 25);
    const unsigned Q0 = __umulhi((unsigned)(N >> 21), R1);                                  // 2^-30
    const long long rem = (long long)((N << 30) - (unsigned long long)Q0 * D);               // 2^-82, exact
    long long Q = ((long long)Q0 << 32) + (((long long)(int)(rem >> 24) * (int)(R1 >> 1)) >> 26);   // 2^-62
    const int below = Q < (1ll << 62) ? 1 : 0;
    Q <<= below;
    ex -= below;
    long long M = (long long)(((unsigned long long)Q + 512ull) >> 10);   // (Q may be just below 2^63)
    // N 2^(52 + below) - M D, between -D and D, from its low 64 bits
    const long long left = (long long)((N << (52 + below)) - (unsigned long long)M * D);
    if (2 * left > (long long)D) ++M;
    if (2 * left < -(long long)D) --M;
    return __longlong_as_double((((long long)ex << 52) + (M - FX_ONE)) | (bn & (long long)0x8000000000000000ull));
}

// log f for a positive f: table-driven argument reduction (P. T. P. Tang,
// "Table-driven implementation of the logarithm function in IEEE
// floating-point arithmetic", ACM TOMS 16, 1990) in integers.  With
// f = 2^e m, m in [1, 2), and c_j = 1 + (j + 1/2) / 2048 the centre of the
// 1/2048 interval that holds m, log f = e ln 2 + log c_j + log1p(r),
// r = m / c_j - 1 (|r| < 2^-12), log1p by its series to r^4, the cubic and
// quartic terms (below 2^-37) in FP32.  tab[j] = (2^62 / c_j, 2^53 log c_j);
// the sum is in units of 2^-53, good to two of them.  That is few bits of a
// small logarithm, so f between 7/8 and 9/8 takes 2 artanh s, s = (f - 1) /
// (f + 1), by its series to s^13 (the next term is below 2^-56 of it), within
// 2^-51 of itself with 11 FP64 operations.  Subnormal f take the library's
// function.
__device__ __forceinline__ double fx_log(double f, const longlong2* __restrict__ tab)
{
    const long long b = __double_as_longlong(f);
    if (b < 0x0010000000000000ll) return log(f);
    if (b >= 0x3fec000000000000ll && b < 0x3ff2000000000000ll) {
        const double s = fx_div(f - 1.0, f + 1.0), z = s * s;
        double p = 1.0 / 13.0;
        p = fma(p, z, 1.0 / 11.0);
        p = fma(p, z, 1.0 / 9.0);
        p = fma(p, z, 1.0 / 7.0);
        p = fma(p, z, 1.0 / 5.0);
        p = fma(p, z, 1.0 / 3.0);
        return 2.0 * fma(s * z, p, s);
    }
    const int e = (int)(b >> 52) - 1023;
    const longlong2 t = __ldg(tab + (int)((b >> 41) & 2047));
    const unsigned Mh = (unsigned)((b >> 32) & 0xfffff) | 0x100000, Ml = (unsigned)b;
    const unsigned Ih = (unsigned)(t.x >> 32), Il = (unsigned)t.x;
    const unsigned long long mid =
        (unsigned long long)Mh * Il + (unsigned long long)Ml * Ih + (unsigned long long)__umulhi(Ml, Il);
    // r in units of 2^-72, and of 2^-42
    const long long T = ((long long)((unsigned long long)Mh * Ih - (1ull << 50)) << 22) + (long long)(mid >> 10);
    const int Th = (int)((T + (1ll << 29)) >> 30);
    const float rs = (float)Th * 2.2737367544323206e-13f;   // 2^-42
    const int cu = __float2int_rn((rs * rs) * (rs * 9007199254740992.0f) * (1.f / 3.f - 0.25f * rs));
    const int sq = (int)(((long long)Th * Th + (1ll << 31)) >> 32);   // r^2 / 2
    // e ln 2 (2^63 ln 2 in two words)
    const long long el2 = (long long)e * (0x58b90bfbll << 22) + (((long long)e * 0xe8e7bcd6ll + 512) >> 10);
    const long long L = el2 + t.y + ((T + (1ll << 18)) >> 19) - sq + cu;
    return fx_scale(fx_double(L), -53);
}

}  // namespace avl
