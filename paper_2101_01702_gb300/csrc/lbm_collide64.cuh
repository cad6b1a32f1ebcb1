// Collisions of the species and mixture sets in double precision (pass 3b
// of lbm_kernels.cuh, which includes this file in the double units).
//
// The kernel is bound by the FP64 pipe.  Per node, direction and species it
// spends five FP64 operations:
//   E_b = R_b psi_x(u) psi_y(u) psi_z(u)      (one product; the y-z part of
//   D_b = E_b - R_b psi_x psi_y psi_z(u+du_b)  a row and the x factors are
//                                              kept per species)
//   f_a <- (1 - 2 beta_a) f_a + c_a E_a + g_a sum_b K_ab D_b,
// R_b = rho Y_b / W_b, c_a = (2 beta_a rho_a + rho_dot_a) / R_a,
// g_a = (beta_a - 1) kappa Y_a / W_a and K_ab = 1/D_ab, which is Eq.
// (finalNumericalEquations) with Eq. (fStar) and the factors that do not
// depend on the direction taken out of it.  The sum over the partner species
// b -- (M-1)^2 terms per direction, three quarters of what remains at
// nine species -- runs on the integer pipe (lbm_fixed.cuh): the D_b of a
// direction are brought to the largest one's exponent, and K to that of
// its largest entry.
//
// Measured, 128^3 with nine species, rates included: 33.2 ms with every
// term formed per direction in floating point, 15.4 ms so (3115 FP64
// instructions per warp, 86 % of the rate a plain chain of multiply-adds
// reaches); 1024 nodes with three species: 101 -> 53 us.
#pragma once

#include "lbm_fixed.cuh"

namespace {

// Doubles of shared memory per thread: the y and x factors of E and of the
// quasi-equilibrium for c = -1, 0, 1 (12 per species); before the
// collision the same columns are the scratch of the production rates.
template <int M>
constexpr int step_cols() { return 12 * M; }

// Whether the cross terms use fixed point: below four species there are at
// most four products per direction, fewer than the conversions cost.
template <int M>
constexpr bool kMixFixed = M >= 4;

template <int M>
__device__ __forceinline__ void step_node(const StepArgs &a, const Node &nd, double *sh, int bs)
{
    const MechConst &mc = c_mech[a.slot];
    const int n = nd.n, t = threadIdx.x;
    const size_t N = a.N;
    const RecRows rr = rec_rows(M, LBMK_MIXED);
    const double *R = rec(a);
    auto ld = [&](int row) { return R[(size_t)row * N + n]; };

    const double rho = ld(rr.rho), T = a.macro[(size_t)DR_T * N + n];
    const bool fixed = kMixFixed<M> && mc.mix_fixed;
    // per species: R_b, and the factors of f_a, E_a and the cross term
    double Rw[M], kf[M - 1], kE[M - 1], kF[M - 1];
    {
        double conc[M];
#pragma unroll
        for (int s = 0; s < M; ++s) {
            Rw[s] = rho * ld(rr.y + s);
            conc[s] = Rw[s] * mc.invW[s];
        }
        molar_production<M>(mc, T, conc, sh, sh + M * bs, sh + 2 * M * bs, t, bs);
        const double kappa = ld(rr.kappa);
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const double wscale = fixed ? mc.invW[s] : 1.0;
            const double ra = Rw[s];
            // E is scaled by R_b; a species that is absent keeps a scale far
            // below every population, so that its source term survives
            double r = ra * wscale;
            r = fabs(r) < 1e-150 ? (r < 0.0 ? -1e-150 : 1e-150) : r;
            Rw[s] = r;
            if (s < M - 1) {
                const double be = ld(rr.beta + s);
                kf[s] = fma(-2.0, be, 1.0);
                kE[s] = fma(2.0 * be, ra, mc.W[s] * sh[(2 * M + s) * bs + t]) / r;
                kF[s] = (be - 1.0) * kappa * ld(rr.y + s) * wscale;
            }
        }
    }
    const double u[3] = {ld(rr.u), ld(rr.u + 1), ld(rr.u + 2)};
    // psi_c(u, u^2 + z) = eA + eB z per axis and c
    auto e_factor = [&](int d, int c, double z) {
        const double usq = u[d] * u[d];
        return c == 0 ? (1.0 - usq) - z : fma(0.5, z, 0.5 * (usq + (double)c * u[d]));
    };
    auto s_factor = [&](int c, double x, double z) {
        const double sq = fma(x, x, z);
        return c == 0 ? 1.0 - sq : 0.5 * (sq + (double)c * x);
    };
#pragma unroll
    for (int s = 0; s < M; ++s) {
        const double z = mc.Ra[s] * T;
        double *col = sh + (size_t)(12 * s) * bs + t;
#pragma unroll
        for (int d = 0; d < 2; ++d) {                          // d = 0: y factors, d = 1: x factors
            const int ax = 1 - d;
            const double x = u[ax] + ld(rr.du + 3 * s + ax);
            const double sq = fma(x, x, z), hs = 0.5 * sq;
#pragma unroll
            for (int c = -1; c <= 1; ++c) {
                col[(6 * d + c + 1) * bs] = e_factor(ax, c, z);
                col[(6 * d + 3 + c + 1) * bs] = c == 0 ? 1.0 - sq : fma(0.5 * c, x, hs);
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
    const double om = ld(rr.om), omf = 1.0 - om, omr = om * rho, RT = ld(rr.rt);

    const PopView v = view(a.src, a);
    PullIdx p;
    make_pull(p, nd, a);
    int bad = 0;                                               // a non-finite result (exponent bits)
#pragma unroll 1
    for (int cz = -1; cz <= 1; ++cz) {
        double zE[M], zS[M];
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const double z = mc.Ra[s] * T;
            zE[s] = Rw[s] * e_factor(2, cz, z);
            zS[s] = Rw[s] * s_factor(cz, u[2] + ld(rr.du + 3 * s + 2), z);
        }
        const double fz = omr * e_factor(2, cz, RT);
#pragma unroll 1
        for (int cy = -1; cy <= 1; ++cy) {
            double pe[M], ps[M];
#pragma unroll
            for (int s = 0; s < M; ++s) {
                pe[s] = zE[s] * sh[(12 * s + cy + 1) * bs + t];
                ps[s] = zS[s] * sh[(12 * s + 3 + cy + 1) * bs + t];
            }
            const double fyz = fz * e_factor(1, cy, RT);
#pragma unroll 1
            for (int cx = -1; cx <= 1; ++cx) {
                const int i = (cx + 1) + 3 * (cy + 1) + 9 * (cz + 1);
                double f[M];
                const Src sr = src_of(i, p, a);
#pragma unroll
                for (int s = 0; s < M; ++s)
                    f[s] = sr.ghost ? load_ghost(a, sr.side, s, i, sr.idx) : load_raw_sf(v, s, i, sr.idx);
                double E[M], D[M];
#pragma unroll
                for (int s = 0; s < M; ++s) {
                    E[s] = pe[s] * sh[(12 * s + 6 + cx + 1) * bs + t];
                    D[s] = fma(-ps[s], sh[(12 * s + 9 + cx + 1) * bs + t], E[s]);
                }
                double F[M - 1];
                if (fixed) {
                    int e = 0;
#pragma unroll
                    for (int b = 0; b < M; ++b) e = max(e, biased_exponent(D[b]));
                    Limbs58 x[M];
#pragma unroll
                    for (int b = 0; b < M; ++b) x[b] = to_limbs58(D[b], e);
#pragma unroll
                    for (int s = 0; s < M - 1; ++s) {
                        long long hi = 0, mid = 0;
#pragma unroll
                        for (int b = 0; b < M; ++b)
                            if (b != s) fma_limbs58(hi, mid, mc.mixh[s][b], mc.mixl[s][b], x[b]);
                        F[s] = double_of_int64(hi + (mid >> 29), e - 1022 + mc.mix_exp);
                        if (e == 0x7ff) F[s] = __longlong_as_double(0x7ff8000000000000ll);   // as D is
                    }
                } else {
#pragma unroll
                    for (int s = 0; s < M - 1; ++s) {
                        F[s] = 0.0;
#pragma unroll
                        for (int b = 0; b < M; ++b)
                            if (b != s) F[s] = fma(mc.inv_WWD[s][b], D[b], F[s]);
                    }
                }
#pragma unroll
                for (int s = 0; s < M - 1; ++s) {
                    const double val = fma(kf[s], f[s], fma(kE[s], E[s], kF[s] * F[s]));
                    store_raw(a.dst, a, s, i, n, val);
                    bad |= !finite_bits(val);
                }
                // mixture f: Eq. (f) with the isotropy correction A_i . X (Eq. (Ai))
                double val = fma(omf, f[M - 1], fyz * e_factor(0, cx, RT));
                if ((cx != 0) + (cy != 0) + (cz != 0) == 1) val += cx * X[0] + cy * X[1] + cz * X[2];
                store_raw(a.dst, a, M - 1, i, n, val);
                bad |= !finite_bits(val);
            }
        }
    }
    if (bad) flag(a.status, LBMK_BIT_NONFINITE);
}

}  // namespace
