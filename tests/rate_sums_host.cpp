// Sums of production rates in pairs of floats (RateSums<true> of
// csrc/lbm_fixed.cuh), compiled for the host, against 113-bit arithmetic.
// Arguments: count, seed.  Prints the largest |error| of the float result in
// units of 2^-24 |w| + n 2^-45 max|W q| + 2^-149 over sums of n terms q, and
// the number of results that are not the float nearest to the exact sum,
// over those whose terms cancel to no less than 1/64 of the largest.  The
// stand-ins for the device's intrinsics are those of diffusion_host.cpp.
#define main diffusion_host_main
#include "diffusion_host.cpp"
#undef main

int main(int argc, char **argv)
{
    const int count = atoi(argv[1]);
    std::mt19937_64 g((unsigned)atoi(argv[2]));
    auto U = [&](double a, double b) { return a + (b - a) * ((g() >> 11) * 0x1p-53); };
    double worst = 0;
    long off = 0;
    for (int it = 0; it < count; ++it) {
        // rates of cold to burnt gas, in units of density from 2^-60 to 2^60
        const double rho = U(0.1, 1.2) * ldexp(1.0, it % 4 ? 0 : (int)U(-60, 60)), base = rho * pow(10, U(-44, -3)), W = U(1, 34);
        const int n = 1 + (int)(g() % 24);
        double col[1];
        RateSums<true> w{col, 1, rate_scale((float)rho)};
        w.clear(0);
        Q sum = 0, top = 0;
        for (int k = 0; k < n; ++k) {
            const double q = base * U(-1, 1) * pow(10, U(-4, 0));
            if (k & 1) w.add<1>(0, w.term(q));
            else w.add<-1>(0, w.term(q));
            sum += k & 1 ? (Q)q : -(Q)q;
            top = max((double)top, fabs(q));
        }
        const Q ex = sum * W;
        const float got = w.mass_float(0, W);
        const double size = fabs((double)ex), big = (double)top * W;
        worst = max(worst, fabs((double)((Q)got - ex)) / (0x1p-24 * size + n * 0x1p-45 * big + 0x1p-149));
        if (size > big / 64 && size > 1.2e-38) off += got != (float)ex;
    }
    printf("%.17g %ld\n", worst, off);
    return 0;
}
