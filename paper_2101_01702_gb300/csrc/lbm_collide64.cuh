// Collisions of the species and mixture sets in double precision (pass 3b
// of lbm_kernels.cuh, which includes this file in the double units).
//
// The kernel is bound by the FP64 pipe.  With
//   e_b = psi_x psi_y psi_z at u,  s_b the same at u + du_b (Eq. (phis)),
//   D_b = R_b (e_b - s_b),  R_b = rho Y_b / W_b,  K_ab = 1/D_ab,
//   f_a <- (1 - 2 beta_a) f_a + (2 beta_a rho_a + rho_dot_a) e_a
//          + (beta_a - 1) kappa Y_a / W_a sum_b K_ab D_b,
// which is Eq. (finalNumericalEquations) with Eq. (fStar) and the factors that
// do not depend on the direction taken out of it, three FP64 operations
// per direction and species remain (the product e_a from the y-z part of
// its row, two multiply-adds).  The differences D_b and the sums over the
// partner species -- (M-1)^2 terms per direction -- run on the integer pipe
// (lbm_fixed.cuh): the y-z parts of a row and the x factors of a direction as
// limbs at each species' own exponent, the D_b brought to the largest one's,
// and K to that of its largest entry.
//
// Measured, 128^3 with nine species: with the production rates in the kernel
// 33.2 ms with every term formed per direction in floating point, 15.4 with
// the D_b in double and only the sums over b in integers, 13.1 with both in
// integers, 11.1 after the exponentials and exponents of the rates left the
// FP64 pipe; without the rates (a kernel of 1.5 ms of its own) 8.0 ms,
// 8.2 with each species' own exponents (limb_differences).
#pragma once

#include "lbm_fixed.cuh"

namespace {

// Columns of shared memory per thread: the y factors of e and s and the x
// factors of e as doubles, the x factors of s as limbs (FX) or doubles, for
// c = -1, 0, 1 (12 per species).
template <int M>
constexpr int step_cols() { return 12 * M; }

// psi_c(v, v^2 + z) = A + B z with the coefficients of an axis and c.
struct PsiCoef {
    double A, B;
};
__device__ __forceinline__ PsiCoef psi_coef(int c, double v)
{
    return PsiCoef{c == 0 ? fma(-v, v, 1.0) : 0.5 * fma(v, v, c > 0 ? v : -v), c == 0 ? -1.0 : 0.5};
}

// FX: the tables are in the range of the fixed-point sums (MechConst::
// mix_fixed; from four species on, below there are at most four products
// per direction, fewer than the conversions cost).
template <int M, bool FX>
__device__ __forceinline__ void step_node(const StepArgs &a, const Node &nd, double *sh, int bs)
{
    const MechConst &mc = c_mech[a.slot];
    const int n = nd.n, t = threadIdx.x;
    const size_t N = a.N;
    const RecRows rr = rec_rows(M);
    const double *R = rec(a);
    auto ld = [&](int row) { return R[(size_t)row * N + n]; };

    const double rho = ld(rr.rho), T = a.macro[(size_t)DR_T * N + n];
    // per species: R_b, and the factors of f_a, R_a e_a and the cross term
    double Rw[M], kf[M - 1], kE[M - 1], kF[M - 1];
    {
        const double kappa = ld(rr.kappa);
        const double *wd = R + (size_t)rr.wd * N + n;
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const double Y = ld(rr.y + s), ra = rho * Y, wscale = FX ? mc.invW[s] : 1.0;
            // e is scaled by R_b; a species that is absent keeps a scale far
            // below every population, so that its source term survives
            double r = FX ? ra * mc.invW[s] : ra;
            r = fabs(r) < 1e-150 ? (r < 0.0 ? -1e-150 : 1e-150) : r;
            Rw[s] = r;
            if (s < M - 1) {
                const double be = ld(rr.beta + s);
                kf[s] = fma(-2.0, be, 1.0);
                kE[s] = fma(2.0 * be, ra, wd[(size_t)s * N]) / r;
                kF[s] = (be - 1.0) * kappa * Y * wscale;
            }
        }
    }
    const double u[3] = {ld(rr.u), ld(rr.u + 1), ld(rr.u + 2)};
    const double om = ld(rr.om), omf = 1.0 - om, omr = om * rho, RT = ld(rr.rt);
    int ex[3] = {0, 0, 0};                                  // exponents of the x factors, per c
    Below dx[3] = {0, 0, 0};
    double fx[3];                                           // x factors of the mixture set
    {
        PsiCoef q[2][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            q[0][c] = psi_coef(c - 1, u[1]);
            q[1][c] = psi_coef(c - 1, u[0]);
            fx[c] = fma(q[1][c].B, RT, q[1][c].A);
        }
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const double z = mc.Ra[s] * T;
            double *col = sh + (size_t)(12 * s) * bs + t;
#pragma unroll
            for (int d = 0; d < 2; ++d) {                      // d = 0: y factors, d = 1: x factors
                const int ax = 1 - d;
                const double x = u[ax] + ld(rr.du + 3 * s + ax);
                const double sq = fma(x, x, z), hs = 0.5 * sq;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double e = fma(q[d][c].B, z, q[d][c].A);
                    const double g = c == 1 ? 1.0 - sq : fma(0.5 * (c - 1), x, hs);
                    col[(6 * d + c) * bs] = e;
                    col[(6 * d + 3 + c) * bs] = g;
                    if (d == 1) ex[c] = max(ex[c], max(biased_exponent(e), biased_exponent(g)));
                }
            }
        }
        if constexpr (FX) {
#pragma unroll
            for (int s = 0; s < M; ++s)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    double *x = sh + (size_t)(12 * s + 9 + c) * bs + t;
                    const int e = max(biased_exponent(x[-3 * bs]), biased_exponent(*x));
                    dx[c] |= below_field(s, ex[c], e);
                    const Limbs58 v = to_limbs58(*x, ex[c] - below_of(dx[c], s));
                    *x = __hiloint2double(v.h, v.l);
                }
        }
    }

    // X = -d_alpha G_alpha (Eq. (Xalpha))
    double X[3] = {0, 0, 0};
    {
        StencilIdx st;
        make_stencil(st, nd, a);
        const double *G = R + (size_t)rr.g * N;
        for_dirs<0, LBMK_Q>([&](auto dd) {
            constexpr int I = decltype(dd)::value;
            if constexpr (I != REST) {
                const size_t nb = nb_of<I>(st, a);
                if (CX(I)) X[0] = fma(WI(I) * CX(I), G[nb], X[0]);
                if (CY(I)) X[1] = fma(WI(I) * CY(I), G[N + nb], X[1]);
                if (CZ(I)) X[2] = fma(WI(I) * CZ(I), G[2 * N + nb], X[2]);
            }
        });
#pragma unroll
        for (int k = 0; k < 3; ++k) X[k] *= -1.5;              // A_i . X = c_i . X / 2 on the axes
    }

    const PopView v = view(a.src, a);
    PullIdx p;
    make_pull(p, nd, a);
    const size_t set = (size_t)LBMK_Q * N;
    int bad = 0;                                               // a non-finite result (exponent bits)
#pragma unroll 1
    for (int cz = -1; cz <= 1; ++cz) {
        double zE[M], zS[M];
        const PsiCoef qz = psi_coef(cz, u[2]);
        const double sA = cz == 0 ? 1.0 : 0.0, sC = cz == 0 ? 0.0 : (cz > 0 ? 0.5 : -0.5);
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const double z = mc.Ra[s] * T;
            zE[s] = Rw[s] * fma(qz.B, z, qz.A);
            const double x = u[2] + ld(rr.du + 3 * s + 2);
            zS[s] = Rw[s] * fma(sC, x, fma(qz.B, fma(x, x, z), sA));
        }
        const double fz = omr * fma(qz.B, RT, qz.A);
#pragma unroll 1
        for (int cy = -1; cy <= 1; ++cy) {
            double pe[M], ps[M];                               // R_b psi_y psi_z of e and s
            int er = 0;
#pragma unroll
            for (int s = 0; s < M; ++s) {
                pe[s] = zE[s] * sh[(12 * s + cy + 1) * bs + t];
                ps[s] = zS[s] * sh[(12 * s + 3 + cy + 1) * bs + t];
                er = max(er, max(biased_exponent(pe[s]), biased_exponent(ps[s])));
            }
            Limbs58 le[M], ls[M];
            Below dr = 0;
            if constexpr (FX) {
#pragma unroll
                for (int s = 0; s < M; ++s) {
                    dr |= below_field(s, er, max(biased_exponent(pe[s]), biased_exponent(ps[s])));
                    const int e = er - below_of(dr, s);
                    le[s] = to_limbs58(pe[s], e);
                    const Limbs58 x = to_limbs58(ps[s], e);
                    ls[s] = Limbs58{opaque(-x.h), opaque(-x.l)};
                    if (s < M - 1) pe[s] *= kE[s];
                }
            }
            const PsiCoef qy = psi_coef(cy, u[1]);
            const double fyz = fz * fma(qy.B, RT, qy.A);
#pragma unroll 1
            for (int cx = -1; cx <= 1; ++cx) {
                const int i = (cx + 1) + 3 * (cy + 1) + 9 * (cz + 1);
                double f[M];
                const Src sr = src_of(i, p, a);
                if (sr.ghost) {
#pragma unroll
                    for (int s = 0; s < M; ++s) f[s] = load_ghost(a, sr.side, s, i, sr.idx);
                } else {
                    const double *src = static_cast<const double *>(v.buf) + (size_t)i * N + sr.idx;
#pragma unroll
                    for (int s = 0; s < M; ++s) f[s] = LBMK_LDG(src + s * set);
                }
                double E[M], F[M - 1];
                if constexpr (FX) {
                    const int exc = cx < 0 ? ex[0] : (cx == 0 ? ex[1] : ex[2]);
                    Limbs58 D[M];
                    const int least = limb_differences<M>(
                        le, ls, dr, cx < 0 ? dx[0] : (cx == 0 ? dx[1] : dx[2]), exc,
                        [&](int s) {
                            const double xe = sh[(12 * s + 6 + cx + 1) * bs + t];
                            E[s] = pe[s] * xe;                 // (2 beta_a rho_a + rho_dot_a) e_a; not used for the last
                            return xe;
                        },
                        [&](int s) {
                            const double xs = sh[(12 * s + 9 + cx + 1) * bs + t];
                            return Limbs58{__double2hiint(xs), __double2loint(xs)};
                        }, D);
                    const int e = er + exc - least - 2044 + mc.mix_exp;
                    const bool nan = er == 0x7ff || exc == 0x7ff;      // an infinite or NaN factor
#pragma unroll
                    for (int s = 0; s < M - 1; ++s) {
                        long long hi = 0, mid = 0;
#pragma unroll
                        for (int b = 0; b < M; ++b)
                            if (b != s) fma_limbs58(hi, mid, limbs_of(mc.mix[s][b]), D[b]);
                        F[s] = double_of_int64(hi + (mid >> 29), e);
                        if (nan) F[s] = __longlong_as_double(0x7ff8000000000000ll);
                    }
                } else {
                    double D[M];
#pragma unroll
                    for (int s = 0; s < M; ++s) {
                        E[s] = pe[s] * sh[(12 * s + 6 + cx + 1) * bs + t];
                        D[s] = fma(-ps[s], sh[(12 * s + 9 + cx + 1) * bs + t], E[s]);
                    }
#pragma unroll
                    for (int s = 0; s < M - 1; ++s) {
                        F[s] = 0.0;
#pragma unroll
                        for (int b = 0; b < M; ++b)
                            if (b != s) F[s] = fma(mc.inv_WWD[s][b], D[b], F[s]);
                        E[s] *= kE[s];
                    }
                }
                double *dst = static_cast<double *>(a.dst) + (size_t)i * N + n;
#pragma unroll
                for (int s = 0; s < M - 1; ++s) {
                    const double val = fma(kf[s], f[s], fma(kF[s], F[s], E[s]));
                    dst[s * set] = val;
                    bad |= !finite_bits(val);
                }
                // mixture f: Eq. (f) with the isotropy correction A_i . X (Eq. (Ai))
                double val = fma(omf, f[M - 1], fyz * (cx < 0 ? fx[0] : (cx == 0 ? fx[1] : fx[2])));
                if ((cx != 0) + (cy != 0) + (cz != 0) == 1) {
                    const double ax = cx ? X[0] : (cy ? X[1] : X[2]);
                    val += cx + cy + cz < 0 ? -ax : ax;
                }
                dst[(M - 1) * set] = val;
                bad |= !finite_bits(val);
            }
        }
    }
    if (bad) flag(a.status, LBMK_BIT_NONFINITE);
}

}  // namespace
