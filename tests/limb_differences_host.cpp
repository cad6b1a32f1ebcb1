// The differences and sums of the double collision in 58-bit limbs
// (limb_differences and fma_limbs58 of csrc/lbm_fixed.cuh), compiled for the
// host, against 113-bit arithmetic.  Arguments: mode (see below), count,
// seed.  Prints the largest |error| of sum_b K_ab (pe_b xe_b - ps_b xs_b) in
// units of 2^-53 max_b(|pe_b xe_b|, |ps_b xs_b|) sum_b K_ab, its root mean
// square, that of the floating form of the same sum (lbm_collide64.cuh), and
// the number of sums other than zero where every pair of products is equal.
// The stand-ins for the device's intrinsics are those of diffusion_host.cpp.
#define main diffusion_host_main
#include "diffusion_host.cpp"
#undef main

int main(int argc, char **argv)
{
    const int mode = atoi(argv[1]), count = atoi(argv[2]);
    std::mt19937_64 g((unsigned)atoi(argv[3]));
    auto U = [&](double a, double b) { return a + (b - a) * ((g() >> 11) * 0x1p-53); };
    const double W[M] = {2, 32, 18, 1, 16, 17, 33, 34, 28};
    double K[M * M];
    for (int a = 0; a < M; ++a)
        for (int b = 0; b < M; ++b) K[M * a + b] = a == b ? 0.0 : 1.0 / (0.02 * sqrt(14 * (1 / W[a] + 1 / W[b])));
    static MixLimbs k[M * M];
    int kx;
    if (!lbm_pack_limbs(K, 1, M * M, k, 1, sizeof(MixLimbs), &kx)) return 2;
    double worst = 0, sq = 0, sqf = 0;
    long off = 0;
    for (int it = 0; it < count; ++it) {
        // equilibrium factors of gases at rest or moving, at temperature T
        const double T = U(280, 2600), u[3] = {U(-0.1, 0.1), U(-0.1, 0.1), U(-0.1, 0.1)};
        const int cx = (int)(g() % 3) - 1, cy = (int)(g() % 3) - 1, cz = (int)(g() % 3) - 1;
        double pe[M], ps[M], xe[M], xs[M];
        auto psi = [](int c, double v, double z) { return c == 0 ? 1 - v * v - z : 0.5 * (v * v + z + c * v); };
        for (int b = 0; b < M; ++b) {
            double n;
            switch (mode) {
            case 0: n = U(0.01, 1); break;                                           // every species
            case 1: n = b == 1 || b == 8 ? U(0.1, 1) : pow(10, U(-14, -5)); break;   // heavy ones, traces of light ones
            default: n = b == 0 || b == 1 || b == 8 ? U(0.1, 1) : (it & 1 ? 0.0 : 1e-150); break;    // absent ones
            }
            const double z = 0.5 / 3000 * T / W[b];
            double du[3];
            for (double &d : du) d = U(-1, 1) * pow(10, U(-6, -2));
            if (it % 5 == 0) du[0] = du[1] = du[2] = 0.0;
            pe[b] = n * psi(cy, u[1], z) * psi(cz, u[2], z);
            ps[b] = n * psi(cy, u[1] + du[1], z) * psi(cz, u[2] + du[2], z);
            xe[b] = psi(cx, u[0], z);
            xs[b] = psi(cx, u[0] + du[0], z);
        }
        int er = 0, ex = 0;
        for (int b = 0; b < M; ++b) {
            er = max(er, max(biased_exponent(pe[b]), biased_exponent(ps[b])));
            ex = max(ex, max(biased_exponent(xe[b]), biased_exponent(xs[b])));
        }
        Below dr = 0, dx = 0;
        Limbs58 le[M], ls[M], lx[M], D[M];
        for (int b = 0; b < M; ++b) {
            dr |= below_field(b, er, max(biased_exponent(pe[b]), biased_exponent(ps[b])));
            dx |= below_field(b, ex, max(biased_exponent(xe[b]), biased_exponent(xs[b])));
            le[b] = to_limbs58(pe[b], er - below_of(dr, b));
            const Limbs58 v = to_limbs58(ps[b], er - below_of(dr, b));
            ls[b] = Limbs58{-v.h, -v.l};
            lx[b] = to_limbs58(xs[b], ex - below_of(dx, b));
        }
        const int least = limb_differences<M>(le, ls, dr, dx, ex, [&](int b) { return xe[b]; }, [&](int b) { return lx[b]; }, D);
        for (int a = 0; a < M; ++a) {
            long long hi = 0, mid = 0;
            Q sum = 0;
            double top = 0, kk = 0, Ff = 0;
            for (int b = 0; b < M; ++b) {
                top = max(top, max(fabs(pe[b] * xe[b]), fabs(ps[b] * xs[b])));
                if (b == a) continue;
                fma_limbs58(hi, mid, limbs_of(k[M * a + b]), D[b]);
                sum += (Q)K[M * a + b] * ((Q)pe[b] * xe[b] - (Q)ps[b] * xs[b]);
                Ff = fma(K[M * a + b], fma(-ps[b], xs[b], pe[b] * xe[b]), Ff);
                kk += K[M * a + b];
            }
            const double F = double_of_int64(hi + (mid >> 29), er + ex - least - 2044 + kx);
            const double unit = 0x1p-53 * top * kk + 1e-300, e = (double)((Q)F - sum) / unit, f = (double)((Q)Ff - sum) / unit;
            worst = max(worst, fabs(e));
            sq += e * e;
            sqf += f * f;
            off += it % 5 == 0 && F != 0.0;
        }
    }
    printf("%.17g %.17g %.17g %ld\n", worst, sqrt(sq / (count * M)), sqrt(sqf / (count * M)), off);
    return 0;
}
