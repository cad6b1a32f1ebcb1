// The refined solve of csrc/lbm_diffusion.cuh, compiled for the host, for
// species far below the others: densities down to the subnormal doubles, one
// trace that alone carries the momentum, and all densities scaled by a power
// of two.  Arguments: mode (see below), count, seed.  Prints the number of
// velocities that are not finite, and the largest |error| against a solve in
// 113-bit arithmetic in units of 2^-24 |x| + 2^-40 max_b(n_b |x_b|)/max_b n_b
// + 2^-53 |u| + 2^-100, n = rho/W.  The stand-ins for the device's intrinsics are those
// of diffusion_host.cpp.
#define main diffusion_host_main
#include "diffusion_host.cpp"
#undef main

int main(int argc, char **argv)
{
    const int mode = atoi(argv[1]), count = atoi(argv[2]);
    std::mt19937_64 g((unsigned)atoi(argv[3]));
    auto U = [&](double a, double b) { return a + (b - a) * ((g() >> 11) * 0x1p-53); };
    const double W[M] = {2, 32, 18, 1, 16, 17, 33, 34, 28};
    double D[M * M], poly[7 * M] = {0};
    for (int a = 0; a < M; ++a)
        for (int b = 0; b < M; ++b) D[M * a + b] = 0.02 * sqrt(14 * (1 / W[a] + 1 / W[b]));
    for (int a = 0; a < M; ++a) poly[7 * a] = 3.5;
    lbm_species sp;
    memset(&sp, 0, sizeof sp);
    sp.M = M;
    sp.W = W;
    sp.thermo = LBM_THERMO_POLY7;
    sp.poly7 = poly;
    sp.D = D;
    sp.nu = 0.8;
    sp.Pr = 0.71;
    sp.r_lat = 0.5 / 3000;
    sp.visc_model = LBM_VISC_RELAXATION;
    sp.T0 = 298;
    lbm_mechanism me;
    memset(&me, 0, sizeof me);
    static MechConst mc;
    if (lbm_pack_tables(&sp, &me, mc) != LBM_OK || !mc.mix_fixed) return 2;
    double worst = 0;
    long nonfinite = 0;
    for (int it = 0; it < count; ++it) {
        double ra[M], u[3], r = 0, jsum[3] = {0, 0, 0};
        float j[M][3];
        const double scale = mode == 2 ? ldexp(1.0, (int)U(-70, 70)) : 1.0;
        const int trace = it % M;
        for (int a = 0; a < M; ++a) {
            const bool major = a == 0 || a == 1 || a == 2 || a == 8;
            switch (mode) {
            case 0: ra[a] = major ? U(0.05, 1) : pow(10, U(-320, -20)); break;             // down to subnormal doubles
            case 1: ra[a] = a == trace ? pow(10, U(-13, -6)) : U(0.05, 1); break;          // one trace, see j below
            case 2: ra[a] = scale * pow(10, U(-12, 0)); break;                             // another unit of density
            default: ra[a] = (a + it) % 3 ? U(0.05, 1) : pow(10, U(-46, -36));             // about the smallest float
            }
            r += ra[a];
        }
        for (int a = 0; a < M; ++a)
            for (int d = 0; d < 3; ++d) {
                const double V = mode == 1 ? (a == trace ? U(-0.5, 0.5) : 0.0)
                                           : (g() % 4 == 0 ? 0.0 : U(-1, 1) * pow(10, U(-7, -2)));
                j[a][d] = (float)(ra[a] * V);
                jsum[d] += j[a][d];
            }
        for (int d = 0; d < 3; ++d) u[d] = jsum[d] / r;
        double im = 0;
        for (int a = 0; a < M; ++a) im += ra[a] / r / W[a];
        const double kappa = sp.r_lat * U(280, 2500) / im;
        double sh[5 * M];
        float du[M][3], ita[M];
        bool bad = false;
        diffusion_refined<M, true>(mc, ra, u, &j[0][0], 1, 0.5 * kappa / r, sh, 1, du, ita, &bad);
        if (bad) return 3;
        Q B[M][M], b[M][3], x[M][3];
        for (int a = 0; a < M; ++a) {
            Q ia = 0;
            for (int c = 0; c < M; ++c)
                if (c != a) {
                    const Q k = (Q)kappa / ((Q)W[a] * W[c] * D[M * a + c]);
                    ia += k * ra[c] / r;
                    B[a][c] = -k * ra[c] / r / 2;
                }
            B[a][a] = 1 + ia / 2;
            for (int d = 0; d < 3; ++d) b[a][d] = (Q)j[a][d] / ra[a] - u[d];
        }
        for (int k = 0; k < M; ++k)
            for (int i = k + 1; i < M; ++i) {
                const Q f = B[i][k] / B[k][k];
                for (int c = k; c < M; ++c) B[i][c] -= f * B[k][c];
                for (int d = 0; d < 3; ++d) b[i][d] -= f * b[k][d];
            }
        for (int d = 0; d < 3; ++d) {
            for (int k = M - 1; k >= 0; --k) {
                Q s = b[k][d];
                for (int c = k + 1; c < M; ++c) s -= B[k][c] * x[c][d];
                x[k][d] = s / B[k][k];
            }
            double flux = 0, top = 0;
            for (int a = 0; a < M; ++a) {
                top = max(top, ra[a] / W[a]);
                flux = max(flux, fabs((double)(x[a][d] * (ra[a] / W[a]))));
            }
            for (int a = 0; a < M; ++a) {
                if (!std::isfinite(du[a][d])) {
                    ++nonfinite;
                    continue;
                }
                // a subnormal double counts as an absent species: velocity zero or the mean of the others
                if (ra[a] < 0x1p-1022) continue;
                const double e = fabs((double)((Q)du[a][d] - x[a][d])), ex = fabs((double)x[a][d]);
                worst = max(worst, e / (0x1p-24 * ex + 0x1p-40 * (flux / top) + 0x1p-53 * fabs(u[d]) + 0x1p-100));
            }
        }
    }
    printf("%ld %.17g\n", nonfinite, worst);
    return 0;
}
