// Host-side packing of an lbm_species / lbm_mechanism description into the
// constant-memory record the kernels read (MechConst), with validation.
#pragma once

#include <math.h>
#include <string.h>

#include "../../include/lbm.h"
#include "lbm_internal.h"

// v[0..n) (elements `step` doubles apart) as integers below 2^58 in units of
// 2^*e, the largest with its leading bit at 2^57.
static inline bool lbm_pack_limbs(const double *v, int step, int n, MixLimbs *out, int out_step, size_t out_bytes,
                                  int *e)
{
    double top = 0.0;
    for (int i = 0; i < n; ++i) {
        if (!isfinite(v[(size_t)i * step])) return false;
        top = fmax(top, fabs(v[(size_t)i * step]));
    }
    *e = (top > 0.0 ? ilogb(top) : 0) - 57;
    for (int i = 0; i < n; ++i) {
        const long long x = (long long)ldexp(v[(size_t)i * step], -*e);
        MixLimbs *o = (MixLimbs *)((char *)out + (size_t)i * out_step * out_bytes);
        o->h = (int)(x >> 29);
        o->l = (int)(x & 0x1fffffff);
    }
    return *e > -900 && *e < 900;
}

// The fixed-point exponents of the rates (MechConst::chem_fixed says whether
// the tables are in range: constants below 2^9, so that sums of a few terms
// stay within the 2^10 that the unit 2^-53 leaves).
static inline void lbm_pack_exponents(MechConst &mc)
{
    bool ok = true;
    mc.gx_mask = 0;
    for (int j = 0; j < 6; ++j) {
        ok &= lbm_pack_limbs(&mc.gco[0][j], 7, mc.M, &mc.gx[0][j], 6, sizeof(MixLimbs), &mc.gx_exp[j]);
        for (int s = 0; s < mc.M; ++s)
            if (mc.gco[s][j] != 0.0) mc.gx_mask |= 1 << j;
    }
    for (int s = 0; s < mc.M; ++s) {
        ok &= fabs(mc.gco[s][6]) < 512.0;
        mc.gx0[s] = ok ? (long long)ldexp(mc.gco[s][6], 53) : 0;
        for (int j = 0; j < 7; ++j) mc.gxf[s][j] = (float)mc.gco[s][j];
    }
    if (mc.R > 0) {
        ok &= lbm_pack_limbs(mc.b, 1, mc.R, &mc.rx[0].b, 1, sizeof(RateLimbs), &mc.bx_exp);
        ok &= lbm_pack_limbs(mc.theta, 1, mc.R, &mc.rx[0].theta, 1, sizeof(RateLimbs), &mc.tx_exp);
    }
    for (int k = 0; k < mc.R; ++k) {
        ok &= fabs(mc.log_A[k]) < 512.0;
        mc.rx[k].log_A = ok ? (long long)ldexp(mc.log_A[k], 53) : 0;
        mc.rx[k].log_Af = (float)mc.log_A[k];
        mc.rx[k].bf = (float)mc.b[k];
        mc.rx[k].thetaf = (float)mc.theta[k];
    }
    mc.chem_fixed = ok;
}

// Returns LBM_OK or LBM_ERR_ARG; fills mc (refs are left zero).
static inline int lbm_pack_tables(const lbm_species *sp, const lbm_mechanism *mech, MechConst &mc)
{
    memset(&mc, 0, sizeof(mc));
    if (!sp || !mech) return LBM_ERR_ARG;
    const int M = sp->M;
    if (M < 2 || M > LBMK_MAXM || !sp->W || !sp->D) return LBM_ERR_ARG;
    if (M > LBMK_MIXM) return LBM_ERR_UNSUPPORTED;      // the tables below; no kernel takes more
    if (sp->thermo == LBM_THERMO_CONST_CP && (!sp->cp_R || !sp->h_form)) return LBM_ERR_ARG;
    if (sp->thermo == LBM_THERMO_POLY7 && !sp->poly7) return LBM_ERR_ARG;
    if (sp->thermo != LBM_THERMO_CONST_CP && sp->thermo != LBM_THERMO_POLY7) return LBM_ERR_ARG;
    if (sp->visc_model != LBM_VISC_KINEMATIC && sp->visc_model != LBM_VISC_RELAXATION) return LBM_ERR_ARG;
    if (!(sp->r_lat > 0) || !(sp->nu > 0) || !(sp->Pr > 0)) return LBM_ERR_ARG;
    if (sp->transport != LBM_TRANSPORT_CONSTANT && sp->transport != LBM_TRANSPORT_MIXTURE_AVERAGED) return LBM_ERR_ARG;
    if (sp->transport == LBM_TRANSPORT_MIXTURE_AVERAGED &&
        (!sp->mu0 || !sp->mu_exp || !(sp->T_tr > 0) || !(sp->P_tr > 0) || !isfinite(sp->D_exp)))
        return LBM_ERR_ARG;
    if (sp->thermo == LBM_THERMO_CONST_CP && !(sp->T0 > 0)) return LBM_ERR_ARG;
    if (mech->R < 0 || mech->R > LBMK_MAXR) return LBM_ERR_ARG;
    if (mech->R > 0 && (!mech->nu_f || !mech->nu_r || !mech->log_A || !mech->b || !mech->theta || !mech->rtype ||
                        !mech->reversible || !(mech->T_ref > 0)))
        return LBM_ERR_ARG;
    mc.M = M;
    mc.R = mech->R;
    mc.visc_model = sp->visc_model;
    mc.T0 = sp->T0;
    mc.nu = sp->nu;
    mc.Pr = sp->Pr;
    mc.r_lat = sp->r_lat;
    for (int a = 0; a < M; ++a) {
        if (!(sp->W[a] > 0)) return LBM_ERR_ARG;
        const double R = sp->r_lat / sp->W[a];
        mc.W[a] = sp->W[a];
        mc.invW[a] = 1.0 / sp->W[a];
        mc.Ra[a] = R;
        mc.Ra_f[a] = (float)R;
        if (sp->thermo == LBM_THERMO_CONST_CP) {
            // U_a = U0 + cv (T - T0), U0 = H0 - R T0, H_a = U_a + R T (Eq. (specHa))
            const double cpR = sp->cp_R[a], cv = (cpR - 1.0) * R, U0 = sp->h_form[a] - R * sp->T0;
            const double c0 = U0 - cv * sp->T0;
            const double h[6] = {cv + R, 0, 0, 0, 0, c0};
            const double u[6] = {c0, cv, 0, 0, 0, 0};
            const double g[7] = {cpR, 0, 0, 0, 0, c0 / R, cpR * log(sp->T0)};
            memcpy(mc.hco[a], h, sizeof h);
            memcpy(mc.uco[a], u, sizeof u);
            memcpy(mc.gco[a], g, sizeof g);
        } else {
            const double *p = sp->poly7 + 7 * a;
            const double h[6] = {R * p[0], R * p[1] / 2, R * p[2] / 3, R * p[3] / 4, R * p[4] / 5, R * p[5]};
            const double u[6] = {R * p[5], R * p[0] - R, R * p[1] / 2, R * p[2] / 3, R * p[3] / 4, R * p[4] / 5};
            const double g[7] = {p[0], -p[1] / 2, -p[2] / 6, -p[3] / 12, -p[4] / 20, p[5], -p[6]};
            memcpy(mc.hco[a], h, sizeof h);
            memcpy(mc.uco[a], u, sizeof u);
            memcpy(mc.gco[a], g, sizeof g);
        }
        for (int b = 0; b < M; ++b) {
            if (a == b) continue;
            const double D = sp->D[M * a + b];
            if (!(D > 0) || D != sp->D[M * b + a]) return LBM_ERR_ARG;
            mc.inv_WWD[a][b] = 1.0 / (sp->W[a] * sp->W[b] * D);
            mc.inv_WWD_f[a][b] = (float)mc.inv_WWD[a][b];
        }
    }
    // Fixed-point 1/D_ab for the sums over the species: the largest entry
    // keeps its leading bit at 2^57, so that entries down to 1/32 of it keep
    // all 53 bits.  Wider ranges, and magnitudes of 1/D and W so far from
    // one that the float scales of lbm_diffusion.cuh could leave their
    // normal range, take the floating sums.
    {
        double top = 0.0, low = INFINITY;
        for (int a = 0; a < M; ++a)
            for (int b = 0; b < M; ++b)
                if (a != b) {
                    top = fmax(top, 1.0 / sp->D[M * a + b]);
                    low = fmin(low, 1.0 / sp->D[M * a + b]);
                }
        const int e = isfinite(top) && top > 0.0 ? ilogb(top) : 0;
        mc.mix_fixed = isfinite(top) && top <= 32.0 * low && top >= 0x1p-12 && e <= 20;
        for (int a = 0; a < M; ++a) {
            if (sp->W[a] < 0x1p-12 || sp->W[a] > 0x1p+12) mc.mix_fixed = 0;
            mc.invW_h[a] = (float)mc.invW[a];
            mc.invW_l[a] = (float)(mc.invW[a] - (double)mc.invW_h[a]);
        }
        mc.mix_exp = e - 57;
        for (int a = 0; a < M && mc.mix_fixed; ++a)
            for (int b = 0; b < M; ++b)
                if (a != b) {
                    const long long v = (long long)ldexp(1.0 / sp->D[M * a + b], 57 - e);
                    mc.mix[a][b].h = (int)(v >> 29);
                    mc.mix[a][b].l = (int)(v & 0x1fffffff);
                    mc.invD_h[a][b] = (float)(1.0 / sp->D[M * a + b]);
                    mc.invD_l[a][b] = (float)(1.0 / sp->D[M * a + b] - (double)mc.invD_h[a][b]);
                }
    }
    mc.transport = sp->transport;
    if (sp->transport == LBM_TRANSPORT_MIXTURE_AVERAGED) {
        for (int a = 0; a < M; ++a) {
            if (!(sp->mu0[a] > 0) || !isfinite(sp->mu_exp[a])) return LBM_ERR_ARG;
            mc.mu0[a] = sp->mu0[a];
            mc.mu_exp[a] = sp->mu_exp[a];
            mc.eucken[a] = 1.25 * mc.Ra[a];
            for (int b = 0; b < M; ++b) {
                mc.wq[a][b] = pow(sp->W[b] / sp->W[a], 0.25);
                mc.wd[a][b] = 1.0 / sqrt(8.0 * (1.0 + sp->W[a] / sp->W[b]));
            }
        }
        mc.log_T_tr = log(sp->T_tr);
        mc.D_exp = sp->D_exp;
        mc.P_tr = sp->P_tr;
    }
    mc.log_T_ref = mech->R > 0 ? log(mech->T_ref) : 0.0;
    bool need_P0 = false;
    for (int k = 0; k < mech->R; ++k) {
        const int t = mech->rtype[k];
        if (t < 0 || t > 2 || (t != 0 && !mech->eff) || (t == 2 && !mech->low)) return LBM_ERR_ARG;
        mc.rtype[k] = t;
        mc.rev[k] = mech->reversible[k] ? 1 : 0;
        need_P0 |= mc.rev[k] != 0;
        mc.log_A[k] = mech->log_A[k];
        mc.b[k] = mech->b[k];
        mc.theta[k] = mech->theta[k];
        if (t == 2) {
            mc.dlow[k][0] = mech->low[3 * k] - mech->log_A[k];
            mc.dlow[k][1] = mech->low[3 * k + 1] - mech->b[k];
            mc.dlow[k][2] = mech->low[3 * k + 2] - mech->theta[k];
        }
        int nr = 0, np = 0, dn = 0;
        for (int a = 0; a < M; ++a) {
            const int f = mech->nu_f[M * k + a], g = mech->nu_r[M * k + a];
            if (f < 0 || g < 0) return LBM_ERR_ARG;
            for (int j = 0; j < f; ++j) { if (nr >= 3) return LBM_ERR_ARG; mc.reac[k][nr++] = a; }
            for (int j = 0; j < g; ++j) { if (np >= 3) return LBM_ERR_ARG; mc.prod[k][np++] = a; }
            dn += g - f;
            if (t != 0) mc.eff[k][a] = mech->eff[M * k + a];
        }
        if (nr == 0) return LBM_ERR_ARG;
        mc.nreac[k] = nr;
        mc.nprod[k] = np;
        mc.dn[k] = dn;
    }
    if (need_P0 && !(mech->P0 > 0)) return LBM_ERR_ARG;
    mc.P0_over_r = need_P0 ? mech->P0 / sp->r_lat : 1.0;
    mc.r_over_P0 = 1.0 / mc.P0_over_r;
    lbm_pack_exponents(mc);
    return LBM_OK;
}

// Host value of U_a(T) from the packed coefficients.
static inline double lbm_host_U(const MechConst &mc, int a, double T)
{
    const double *u = mc.uco[a];
    return ((((u[5] * T + u[4]) * T + u[3]) * T + u[2]) * T + u[1]) * T + u[0];
}
