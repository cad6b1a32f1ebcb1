// Block fixed-point arithmetic on the integer pipe, for sums of products
// that need double-precision accuracy.
//
// Measured on GB300 (one SM, 32 warps): a double multiply-add takes 19
// cycles per warp instruction, a 32 x 32 + 64 bit integer multiply-add 1.3.
// Three of the latter give a product of two 58-bit numbers to 2^-56, so a
// sum of products over operands brought to a common exponent is formed at
// about a fifth of the FP64 pipe's cost, with no more error than a chain
// of fused multiply-adds: the operands keep all 53 bits down to 2^-5 of the
// largest one, and the sum is rounded once.
#pragma once

#include "lbm_internal.h"

namespace {

// x as a value the compiler knows nothing about.  A 32-bit factor that it has
// seen cut out of a 64-bit integer makes it form products of two such
// factors in 64 bits: 12 instructions for the three multiply-adds of
// fma_limbs58 instead of 4.
__device__ __forceinline__ int opaque(int x)
{
#ifdef __CUDA_ARCH__
    asm("" : "+r"(x));
#endif
    return x;
}

// A signed 59-bit integer as two limbs: value = h 2^29 + l, 0 <= l < 2^29.
struct Limbs58 {
    int h, l;
};

__device__ __forceinline__ Limbs58 limbs_of(long long v)
{
    return Limbs58{opaque((int)(v >> 29)), opaque((int)((unsigned)v & 0x1fffffffu))};
}

__device__ __forceinline__ int biased_exponent(double d) { return (__double2hiint(d) >> 20) & 0x7ff; }

// d in units of 2^(e - 1080), for e at least d's biased exponent: the
// largest operand of a block keeps its leading bit at 2^57; bits below
// the unit are dropped.
__device__ __forceinline__ long long to_fixed58(double d, int e)
{
    const int hi = __double2hiint(d), ed = (hi >> 20) & 0x7ff;
    const unsigned mh = ((unsigned)hi & 0xfffffu) | (ed ? 0x100000u : 0u);
    const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(d)) << 5;
    const int sh = e - ed < 63 ? e - ed : 63;                 // m < 2^58
    const long long v = (long long)(m >> sh);
    return hi < 0 ? -v : v;
}

__device__ __forceinline__ Limbs58 to_limbs58(double d, int e)
{
    return limbs_of(to_fixed58(d, e));
}

// Adds x (limbs) times the constant c < 2^58 to a running sum kept
// as hi + mid 2^-29 in units of 2^58; the low x low product, less than
// one of those units, is left out.  Eight terms stay within 63 bits.
__device__ __forceinline__ void fma_limbs58(long long &hi, long long &mid, Limbs58 c, Limbs58 x)
{
    hi += (long long)c.h * x.h;
    mid += (long long)c.h * x.l;
    mid += (long long)c.l * x.h;
}

// Entry of MechConst::mix.
__device__ __forceinline__ Limbs58 limbs_of(const MixLimbs &m) { return Limbs58{m.h, m.l}; }

// Exponents of up to ten operands, by how far each lies below the largest, at
// most 15, in fields of 6 bits: the sum of two is a shift of a 32-bit word.
typedef unsigned long long Below;
__device__ __forceinline__ Below below_field(int s, int top, int e) { return (Below)(unsigned)min(top - e, 15) << (6 * s); }
__device__ __forceinline__ int below_of(Below b, int s) { return (int)(unsigned)(b >> (6 * s)) & 63; }

// The differences D_b = pe_b xe_b - ps_b xs_b of M pairs of products, as limbs
// at one exponent; le, -ls and xs as limbs at the exponents er - dr and ex - dx
// of their b (er, ex: the largest, dr, dx: below_field).  Each pair keeps its
// own exponent (down to 2^-15 of the largest factor) and is then brought to
// the exponent er + ex - (returned number) of the largest, rounded to
// nearest, with signed low limbs, so that what the sums over b leave out has
// no mean; equal products give zero.  The sums over b have a root mean square
// error of 0.015 to 0.019 units of 2^-53 of the largest product, 0.05 to 0.07 in
// double (tests/test_limb_differences.py).  With one exponent for all factors
// of a row and one for all x factors, whose largest belong to different
// species (heavy, abundant ones and light ones), it was 0.13 to 2.8, and the
// populations of heavy species were off by 2.3 to 5 units of 2^-53 of
// themselves where they now are by 1.0 to 2.1, and by 1.1 to 2.3 with the
// collision all in double (median over the nodes of a flame after one step).
// 128^3 double k_step: 8.00 -> 8.17 ms.
template <int M, class XE, class XS>
__device__ __forceinline__ int limb_differences(const Limbs58 *le, const Limbs58 *ls, Below dr, Below dx, int ex,
                                                XE &&xe, XS &&xs, Limbs58 *D)
{
    const Below d = dr + dx;
    int least = below_of(d, 0);
#pragma unroll
    for (int b = 1; b < M; ++b) least = min(least, below_of(d, b));
#pragma unroll
    for (int b = 0; b < M; ++b) {
        const Limbs58 l = to_limbs58(xe(b), ex - below_of(dx, b)), m = xs(b);
        const int sh = below_of(d, b) - least;
        long long hi = 0, mid = 0;
        fma_limbs58(hi, mid, le[b], l);
        fma_limbs58(hi, mid, ls[b], m);
        const long long v = (hi + (mid >> 29) + (0x40000000u >> (31 - sh))) >> sh;  // below 2^59
        const int h = (int)((v + (1 << 28)) >> 29);
        D[b] = Limbs58{opaque(h), opaque((int)((unsigned)v - ((unsigned)h << 29)))};
    }
    return least;
}

// s 2^e rounded to nearest (results below the normal range become zero).
__device__ __forceinline__ double double_of_int64(long long s, int e)
{
    const unsigned long long mag = s < 0 ? 0ull - (unsigned long long)s : (unsigned long long)s;
    const int lz = __clzll((long long)mag);
    const int be = e + 1086 - lz;                             // biased exponent: e + 63 - lz + 1023
    const unsigned long long nrm = mag << (lz & 63);
    unsigned long long bits = ((unsigned long long)(unsigned)(be - 1) << 52) + (nrm >> 11) + ((nrm >> 10) & 1ull);
    if (mag == 0 || be <= 0) bits = 0;
    if (be >= 2047) bits = 0x7ff0000000000000ull;
    if (s < 0) bits |= 0x8000000000000000ull;
    return __longlong_as_double((long long)bits);
}

// a + b as a rounded sum and its error (Knuth).
__device__ __forceinline__ float two_sum(float a, float b, float &err)
{
    const float s = a + b, bb = s - a;
    err = (a - (s - bb)) + (b - bb);
    return s;
}

// The leading 24 and the next 23 bits of d as floats; d rounded to float and 0
// outside the range where both are normal (and not zero).
__device__ __forceinline__ void split2(double d, float &h, float &l)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const int ed = (int)((hi >> 20) & 0x7ffu) - 896;                 // float exponent field
    const unsigned sign = hi & 0x80000000u;
    if (ed > 24 && ed < 255) {
        h = __uint_as_float(sign | ((unsigned)ed << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
        // 23 of the low 29 bits as a float of exponent ed - 23, less its implicit one
        const unsigned e2 = sign | ((unsigned)(ed - 23) << 23);
        l = __uint_as_float(e2 | ((lo & 0x1fffffffu) >> 6)) - __uint_as_float(e2);
    } else {
        h = (hi << 1 | lo) == 0u ? 0.0f : __double2float_rn(d);
        l = 0.0f;
    }
}

// 2^k, clamped to the normal floats.
__device__ __forceinline__ float pow2f(int k)
{
    return __int_as_float((min(max(k, -126), 127) + 127) << 23);
}

// d 2^k; 0 below the normal doubles, infinite above the largest.
__device__ __forceinline__ double scale2(double d, int k)
{
    const long long v = ((long long)__double2hiint(d) << 32) | (unsigned)__double2loint(d);
    const int e = (int)(v >> 52) & 0x7ff, s = e + k;
    if (e == 0x7ff) return d;                                        // infinite, NaN
    const long long inf = (v < 0 ? (long long)(1ull << 63) : 0ll) | 0x7ffll << 52;
    return __longlong_as_double(e == 0 || s <= 0 ? 0ll : (s >= 0x7ff ? inf : v + ((long long)k << 52)));
}

// Sums of the molar production rates of a node, one 8-byte column per
// species: in double, or (PAIR) in pairs of floats, for callers that store
// the rates as floats: a sum and the sum of its rounding errors (two_sum), 48
// bits.  The pairs hold the terms 2^scale times larger (rate_scale): rates of
// cold gas are below the floats' range, and without the scale terms below
// 2^-102 had 24 bits (nine terms of ten in a 300 K box; root mean square
// error of the stored rates 0.37 units in the last place, now 0.29, that of
// exact sums).
template <bool PAIR>
struct RateSums {
    double *col;
    int stride, scale;
    __device__ __forceinline__ void clear(int s) { col[s * stride] = 0.0; }
    struct Term {
        double q;
        float h, l;
    };
    __device__ __forceinline__ Term term(double q) const
    {
        Term t{q, 0.0f, 0.0f};
        if (PAIR) split2(scale2(q, scale), t.h, t.l);
        return t;
    }
    template <int SIGN>
    __device__ __forceinline__ void add(int s, const Term &t)
    {
        if (PAIR) {
            float2 *p = reinterpret_cast<float2 *>(col + s * stride);
            float2 v = *p;
            float e;
            v.x = two_sum(v.x, SIGN * t.h, e);
            v.y += e + SIGN * t.l;
            *p = v;
        } else {
            col[s * stride] += SIGN * t.q;
        }
    }
    // w_s times the molar mass (PAIR)
    __device__ __forceinline__ float mass_float(int s, double W) const
    {
        const float2 v = *reinterpret_cast<const float2 *>(col + s * stride);
        float wh, wl;
        split2(W, wh, wl);
        const float p = wh * v.x;
        return (p + (fma(wh, v.x, -p) + fma(wh, v.y, wl * v.x))) * pow2f(-scale);
    }
};

// The scale of the pairs for density rho: a rate as large as the density
// becomes 2^64, so that sums stay in range and terms down to 2^-166 of the
// density, below the smallest float for densities of order one, keep their 48
// bits.
__device__ __forceinline__ int rate_scale(float rho)
{
    return min(191 - ((__float_as_int(rho) >> 23) & 0xff), 126);
}

}  // namespace
