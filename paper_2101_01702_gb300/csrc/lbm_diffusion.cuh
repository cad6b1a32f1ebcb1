// Stefan-Maxwell diffusion velocities (Eq. (transform1)) almost without the
// FP64 pipe: a float factorisation and one step of iterative refinement whose
// residual is formed in fixed point (lbm_fixed.cuh).  For the mixed unit,
// where the velocities are stored as floats.
//
// The system of a node, with h = kappa/2 = m R_U T/2, A_ab = 1/(W_a W_b D_ab),
//   x_a + h sum_b A_ab Y_b (x_a - x_b) = V_a,   V_a = j_a/rho_a - u,
// is diagonally dominant by rows with excess 1, and A is symmetric.
// Eliminating species k leaves a system of the same form with
//   A_ij += A_ik A_kj Y_k / d_k,   e_i += A_ik Y_k e_k / d_k,
//   d_k = e_k + sum_{j>k} A_kj Y_j            (e = 1/h at the start),
// sums of positive terms only (Grassmann, Taksar and Heyman's elimination),
// so the float factors carry a few units of 2^-24 in every entry, however
// small the mass fractions.  The float solution x0 is an exact operand of the
// residual
//   r_a = V_a - x_a - (h/W_a) (x_a S_a - sum_b K_ab n_b x_b),
//   S_a = sum_b K_ab n_b,  K_ab = 1/D_ab,  n_b = Y_b/W_b,
// whose sums over b run in 58-bit limbs, the products n_b x_b brought to the
// largest one's exponent, and whose other terms are pairs of floats (2^-46 of
// each); the correction is solved with the same factors and x0 plus it rounded
// to float once.  A velocity is the exact one to 2^-40 of the largest
// n_b |x_b| over the largest n_b and 2^-53 of |u|, rounded to float
// (tests/test_diffusion_traces.py measures it against a 113-bit solution).
// That is no further from the exact velocity than a double LDL^T solve
// rounded to float.  Root mean square error in units of the last place, each
// over 540,000 velocities of nine species (exact rounding: 0.289): ordinary
// mixtures 0.289 (LDL^T 0.289), traces down to 1e-14 0.289 (4.2), down to
// 1e-10 with absent species 0.289 (0.59), rounding-level traces of either
// sign 0.289 (0.289), one species nearly pure 0.289 (5e6: its j_a/rho and
// Y_a u cancel).
//
// A double LDL^T solve costs 740 FP64 instructions per warp at nine species,
// 56 thousand cycles of a scheduler; this one about 9 thousand
// instructions, 36 of them FP64.
#pragma once

#include "lbm_fixed.cuh"

namespace {

// 1/x for normal x (the instruction takes subnormal operands for zero).
__device__ __forceinline__ float rcp_approx(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / (((__float_as_int(x) >> 23) & 0xff) == 0 ? 0.0f * x : x);
#endif
}

// |d| 2^-k in [1, 2) with d's sign as a float of its leading 24 bits and one
// of the next 23, and k; false for d = 0 or below the normal doubles.
__device__ __forceinline__ bool mantissa2(double d, float &h, float &l, int &k)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d), sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned e2 = sign | (104u << 23);                         // 2^-23
    h = __uint_as_float(sign | (127u << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    l = __uint_as_float(e2 | ((lo & 0x1fffffffu) >> 6)) - __uint_as_float(e2);
    if (e == 0x7ff) h = __int_as_float(0x7fc00000);                  // infinite, NaN
    k = e - 1023;
    return e != 0;
}

// x as a double, on the integer pipe; subnormals by way of 2^64 times them.
__device__ __forceinline__ double widen(float x)
{
    const bool small = ((__float_as_int(x) >> 23) & 0xff) == 0;
    const unsigned b = (unsigned)__float_as_int(small ? x * 18446744073709551616.0f : x), mag = b & 0x7fffffffu;
    const unsigned bias = (mag >> 23) == 255u ? 1792u : (small ? 832u : 896u);
    const unsigned hi = (b & 0x80000000u) | (mag == 0u ? 0u : (mag >> 3) + (bias << 20));
    return __longlong_as_double((long long)((unsigned long long)hi << 32 | (unsigned long long)(b << 29)));
}

// V = j/r - u as a pair of floats, 0 for r = 0 or below the normal doubles:
// the numerator j - r u in one double operation, which rounds once however
// much of the two cancels, of r's mantissa and j scaled by r's exponent (r may
// be far below the floats while j is not: a trace's rest population is a
// double), and its quotient by the mantissa.  |V| below 2^-126 or above 2^127
// counts as that.
__device__ __forceinline__ void slip_velocity(double r, float j, double u, float &h, float &l)
{
    float dh, dl, rh, rl;
    int kd, kr;
    const bool here = mantissa2(r, rh, rl, kr);
    const unsigned m = ((unsigned)__double2hiint(r) & 0x800fffffu) | 0x3ff00000u;
    const double rm = __longlong_as_double((long long)((unsigned long long)m << 32 | (unsigned)__double2loint(r)));
    const bool moves = mantissa2(fma(-rm, u, scale2(widen(j), -kr)), dh, dl, kd);
    const float ri = rcp_approx(rh), v = dh * ri;
    const float w = (fma(-v, rl, fma(-v, rh, dh)) + dl) * ri;
    const float g = moves && here ? pow2f(kd) : 0.0f;
    h = v * g;
    l = w * g;
}

// du[M][3], and ita = 1/tau_a [M], of a node, from the rows (stride N) of
// its species densities ra, velocity ud and momenta J, and hk = h/rho.  All
// quantities are scale-free in the densities: with rho_b in place of Y_b, h
// becomes h/rho.  sh: 2 M columns of this thread's shared memory, stride
// bs, or 5 M with KEEP, as the kernel has it: the V_a of all three components
// are then formed before the factorisation and kept in the last 3 M, so that
// their loads overlap and the loop over the components fits the registers
// (moments and diffusion, 256^3: 22.1 ms; formed in that loop 24.9, and 25.3
// with j - r u in integers there; 23.1 with V from j/r and u as pairs of
// floats, 2^-46 of each and up to 160 times the double solve's error where
// they cancel).  Sets *bad for a non-finite pivot.
template <int M, bool KEEP = false>
__device__ __forceinline__ void diffusion_refined(const MechConst &mc, const double *ra, const double *ud,
                                                  const float *J, size_t N, double hk, double *sh, int bs,
                                                  float (*du)[3], float *ita, bool *bad)
{
    float2 *sV = reinterpret_cast<float2 *>(sh + 2 * M * bs);
    if (KEEP) {
        const double u0 = ud[0], u1 = ud[N], u2 = ud[2 * N];
#pragma unroll
        for (int s = 0; s < M; ++s)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                float2 v;
                slip_velocity(ra[(size_t)s * N], J[(size_t)(3 * s + d) * N], d == 0 ? u0 : (d == 1 ? u1 : u2), v.x, v.y);
                sV[(3 * s + d) * bs] = v;
            }
    }
    // n_b = rho_b / W_b
    long long *ln = reinterpret_cast<long long *>(sh), *lS = ln + M * bs;
    float y[M], nh[M], nl[M];
    int top = 0;                                           // exponent of the largest
#pragma unroll
    for (int b = 0; b < M; ++b) {
        const double nb = ra[(size_t)b * N] * mc.invW[b];
        top = max(top, biased_exponent(nb));
        ln[b * bs] = ((long long)__double2hiint(nb) << 32) | (unsigned)__double2loint(nb);
    }
    // the floats take all densities 2^k times larger, of order one
    const int k = 1023 - top;
#pragma unroll
    for (int b = 0; b < M; ++b) {
        float lo;
        split2(scale2(ra[(size_t)b * N], k), y[b], lo);
        y[b] += lo;
        split2(scale2(__longlong_as_double(ln[b * bs]), k), nh[b], nl[b]);
    }
    float hh, hl;
    split2(scale2(hk, -k), hh, hl);

    // S_a as pairs of floats, summed with their errors (all terms have one
    // sign, so each S_a keeps its relative accuracy), and 1/tau_a = 2 (h/W_a) S_a
#pragma unroll
    for (int s = 0; s < M; ++s) {
        float Sh = 0.0f, Sl = 0.0f;
#pragma unroll
        for (int b = 0; b < M; ++b)
            if (b != s) {
                const float kh = mc.invD_h[s][b], p = kh * nh[b];
                const float pe = fma(kh, nh[b], -p) + fma(kh, nl[b], mc.invD_l[s][b] * nh[b]);
                float e;
                Sh = two_sum(Sh, p, e);
                Sl += e + pe;
            }
        const float S = Sh + Sl;
        Sl = (Sh - S) + Sl;
        lS[s * bs] = ((long long)__float_as_int(S) << 32) | (unsigned)__float_as_int(Sl);
        const float wh = mc.invW_h[s], wl = mc.invW_l[s];
        const float th = hh * wh, tl = fma(hh, wh, -th) + fma(hh, wl, hl * wh);
        const float p = th * S;
        ita[s] = 2.0f * (p + (fma(th, S, -p) + fma(th, Sl, tl * S)));
    }

    // factors: K[i][j], i < j, and 1/d_k
    float K[M][M], dinv[M];
    const float ex0 = rcp_approx(hh);
    {
        float ex[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            ex[i] = ex0;
#pragma unroll
            for (int j = i + 1; j < M; ++j) K[i][j] = mc.inv_WWD_f[i][j];
        }
#pragma unroll
        for (int k = 0; k < M; ++k) {
            float d = ex[k];
#pragma unroll
            for (int j = k + 1; j < M; ++j) d = fma(K[k][j], y[j], d);
            if (!finite_bits(d)) *bad = true;
            dinv[k] = rcp_approx(d);
            const float m = y[k] * dinv[k];
#pragma unroll
            for (int i = k + 1; i < M; ++i) {
                const float l = K[k][i] * m;
                ex[i] = fma(l, ex[k], ex[i]);
#pragma unroll
                for (int j = i + 1; j < M; ++j) K[i][j] = fma(l, K[k][j], K[i][j]);
            }
        }
    }
    // x <- solution for the right-hand side x (in units of V)
    auto solve = [&](float *x) {
#pragma unroll
        for (int k = 0; k < M; ++k) x[k] *= ex0;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const float mk = y[k] * dinv[k] * x[k];
#pragma unroll
            for (int i = k + 1; i < M; ++i) x[i] = fma(K[k][i], mk, x[i]);
        }
        float z[M];
#pragma unroll
        for (int k = M - 1; k >= 0; --k) {
            float s = x[k];
#pragma unroll
            for (int j = k + 1; j < M; ++j) s = fma(K[k][j], z[j], s);
            x[k] = s * dinv[k];
            z[k] = y[k] * x[k];
        }
    };

#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
        float Vh[M], Vl[M], x[M];
        {
            const double u = KEEP ? 0.0 : ud[d * N];
#pragma unroll
            for (int s = 0; s < M; ++s) {
                if (KEEP) {
                    const float2 v = sV[(3 * s + d) * bs];
                    Vh[s] = v.x;
                    Vl[s] = v.y;
                } else {
                    slip_velocity(ra[(size_t)s * N], J[(size_t)(3 * s + d) * N], u, Vh[s], Vl[s]);
                }
                x[s] = Vh[s] + Vl[s];
            }
        }
        solve(x);
        // w_b = n_b x0_b as integers below 2^58, in units of 2^(ew - 1206), of
        // which the largest keeps at least 57 bits: from the 53 bits of n_b and
        // the 24 of x0_b, so that a trace whose momentum balances that of all
        // others counts in full (subnormal floats x0 count as zero)
        int ew = 1022 - mc.mix_exp - k;                                        // sums in units of at least 2^-126
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const int ex = (__float_as_int(x[s]) >> 23) & 0xff, en = (int)(ln[s * bs] >> 52) & 0x7ff;
            if (ex == 0) x[s] = 0.0f;
            if (ex != 0 && en != 0) ew = max(ew, ex + en);
        }
        const int c = mc.mix_exp + ew + k - 1148;                                // the sums are integers times 2^c
        const float g1 = pow2f(41 + c), g2 = pow2f(18 + c), g3 = pow2f(c);
        Limbs58 w[M];
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const int xi = __float_as_int(x[s]), hi = opaque((int)(ln[s * bs] >> 32)), lo = opaque((int)ln[s * bs]);
            const int ex = (xi >> 23) & 0xff, en = (hi >> 20) & 0x7ff;
            const unsigned mx = ((unsigned)xi & 0x7fffffu) | 0x800000u;
            const unsigned mh = (((unsigned)hi & 0xfffffu) | 0x100000u) << 8 | (unsigned)lo >> 24, ml = (unsigned)lo & 0xffffffu;
            const unsigned long long v = ((unsigned long long)mh * mx << 5) + ((unsigned long long)ml * mx >> 19);
            const long long p = ex != 0 && en != 0 ? (long long)(v >> min(ew - ex - en, 63)) : 0ll;
            w[s] = limbs_of((hi ^ xi) < 0 ? -p : p);
        }
        float r[M];
#pragma unroll
        for (int s = 0; s < M; ++s) {
            long long hi = 0, mid = 0;
#pragma unroll
            for (int b = 0; b < M; ++b)
                if (b != s) fma_limbs58(hi, mid, limbs_of(mc.mix[s][b]), w[b]);
            const long long G = hi + (mid >> 29);
            // G as a pair of floats, from pieces of 22, 23 and 18 bits
            const float G1 = (__int_as_float(0x4b400000 + (int)(G >> 41)) - 12582912.0f) * g1;
            const float G2 = (__int_as_float(0x4b000000 | (int)((G >> 18) & 0x7fffff)) - 8388608.0f) * g2;
            const float G3 = (__int_as_float(0x4b000000 | (int)(G & 0x3ffff)) - 8388608.0f) * g3;
            const float Gh = G1 + G2, Gl = (G2 - (Gh - G1)) + G3;
            const long long S = lS[s * bs];
            const float x0 = x[s];
            // H = x_a S_a - G_a
            const float Sh = __int_as_float((int)(S >> 32)), xS = x0 * Sh;
            float He;
            const float Hh = two_sum(xS, -Gh, He);
            const float Hl = He + (fma(x0, Sh, -xS) + fma(x0, __int_as_float((int)S), -Gl));
            const float wh = mc.invW_h[s], wl = mc.invW_l[s];
            const float th = hh * wh, tl = fma(hh, wh, -th) + fma(hh, wl, hl * wh);
            const float p = th * Hh, pe = fma(th, Hh, -p) + fma(th, Hl, tl * Hh);
            float e1, e2;
            const float s1 = two_sum(Vh[s], -x0, e1);
            const float s2 = two_sum(s1, -p, e2);
            r[s] = s2 + (e2 + ((e1 + Vl[s]) - pe));
        }
        solve(r);
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const float v = Vh[s] == 0.0f && Vl[s] == 0.0f && y[s] == 0.0f ? 0.0f : x[s] + r[s];
            if (d == 0) du[s][0] = v;
            else if (d == 1) du[s][1] = v;
            else du[s][2] = v;
        }
    }
}

}  // namespace
