// Host build of csrc/lbm_diffusion.cuh and lbm_fixed.cuh (plain C++ stand-ins
// for the device intrinsics): the refined solve of seeded node states against
// a solve in 113-bit arithmetic, and the fixed-point sums against the same.
// Arguments: mode (see states below), count, seed.  Prints, over all
// velocities: the largest |error| in units of 2^-24 |x| + 2^-40 max|x| +
// 2^-45 |u|, the same for 1/tau_a in units of 2^-24, the root mean square error relative to
// the largest velocity divided by that of the 113-bit solution rounded to
// float, the number of absent species with a velocity other than zero, and
// the largest error of the sums in units of 2^-53 (|sum| + 1.7 times the
// largest operand times the largest constant).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include <cuda_runtime.h>
using std::max;
using std::min;
template <class To, class From> static To bits(From v) { To o; memcpy(&o, &v, sizeof o); return o; }
static inline int __double2hiint(double d) { return (int)(bits<uint64_t>(d) >> 32); }
static inline int __double2loint(double d) { return (int)bits<uint64_t>(d); }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline double __longlong_as_double(long long v) { return bits<double>(v); }
static inline float __uint_as_float(unsigned v) { return bits<float>(v); }
static inline float __int_as_float(int v) { return bits<float>(v); }
static inline int __float_as_int(float v) { return bits<int>(v); }
static inline float __double2float_rn(double v) { return (float)v; }
static inline int __float2int_rn(float v) { return (int)nearbyintf(v); }
static inline bool finite_bits(float x) { return (bits<int>(x) & 0x7f800000) != 0x7f800000; }

#include "../paper_2101_01702_gb300/csrc/lbm_pack.h"
#include "../paper_2101_01702_gb300/csrc/lbm_diffusion.cuh"

typedef __float128 Q;
constexpr int M = 9;

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
    double worst = 0, worst_tau = 0, se = 0, sr = 0;
    long wrong = 0;
    for (int it = 0; it < count; ++it) {
        double Y[M], ra[M], u[3], sum = 0;
        float j[M][3];
        for (int a = 0; a < M; ++a) {
            switch (mode) {
            case 0: Y[a] = pow(10, U(-6, 0)); break;                                     // ordinary mixtures
            case 1: Y[a] = pow(10, U(-14, 0)); break;                                    // down to traces
            case 2: Y[a] = a == 0 || a == 1 || a == 8 ? U(0.1, 1) : 1e-13 * U(-0.5, 1); break;   // rounding-level traces
            case 3: Y[a] = a == it % M ? 1.0 : pow(10, U(-16, -8)); break;               // one species nearly pure
            default: Y[a] = U(0, 1) < 0.2 ? 0.0 : pow(10, U(-10, 0));                    // absent species
            }
            sum += Y[a];
        }
        if (!(sum > 1e-9)) { Y[8] += 1; sum += 1; }
        const double rho = U(0.15, 1.2);
        for (int a = 0; a < M; ++a) ra[a] = rho * (Y[a] /= sum);
        for (int d = 0; d < 3; ++d) u[d] = U(-1e-2, 1e-2);
        for (int a = 0; a < M; ++a)
            for (int d = 0; d < 3; ++d)
                j[a][d] = (float)(ra[a] * (u[d] + U(-1, 1) * pow(10, U(-7, -2)) * (mode == 2 && Y[a] < 1e-10 ? 1e3 : 1)));
        double im = 0, r = 0;
        for (int a = 0; a < M; ++a) {
            im += Y[a] / W[a];
            r += ra[a];
        }
        const double kappa = sp.r_lat * U(280, 2500) / im;
        double sh[2 * M];
        float du[M][3], ita[M];
        bool bad = false;
        diffusion_refined<M>(mc, ra, u, &j[0][0], 1, 0.5 * kappa / r, sh, 1, du, ita, &bad);
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
            worst_tau = max(worst_tau, fabs((double)(ita[a] / ia - 1)) * 0x1p24);
            for (int d = 0; d < 3; ++d) b[a][d] = ra[a] != 0 ? (Q)j[a][d] / ra[a] - u[d] : (Q)0;
        }
        for (int k = 0; k < M; ++k)
            for (int i = k + 1; i < M; ++i) {
                const Q f = B[i][k] / B[k][k];
                for (int c = k; c < M; ++c) B[i][c] -= f * B[k][c];
                for (int d = 0; d < 3; ++d) b[i][d] -= f * b[k][d];
            }
        for (int d = 0; d < 3; ++d) {
            double top = 0;
            for (int k = M - 1; k >= 0; --k) {
                Q s = b[k][d];
                for (int c = k + 1; c < M; ++c) s -= B[k][c] * x[c][d];
                x[k][d] = s / B[k][k];
            }
            for (int a = 0; a < M; ++a)
                if (ra[a] != 0) top = max(top, fabs((double)x[a][d]));
            for (int a = 0; a < M; ++a) {
                if (ra[a] == 0) {
                    wrong += du[a][d] != 0;
                    continue;
                }
                const double e = fabs((double)((Q)du[a][d] - x[a][d])), ex = fabs((double)x[a][d]);
                worst = max(worst, e / (0x1p-24 * ex + 0x1p-40 * top + 0x1p-45 * fabs(u[d])));
                se += e * e / (top * top);
                const double er = fabs((double)((Q)(float)(double)x[a][d] - x[a][d]));
                sr += er * er / (top * top);
            }
        }
    }
    // sums of eight products, operands over seven decades, against 113 bits
    double ws = 0;
    for (int it = 0; it < count; ++it) {
        double v[M];
        int e = 0;
        for (int b = 0; b < M; ++b) {
            v[b] = U(-1, 1) * pow(10, U(-7, 0)) * pow(2, U(-300, 300) * (mode == 1));
            e = max(e, biased_exponent(v[b]));
        }
        long long hi = 0, mid = 0;
        Q ref = 0, big = 0;
        for (int b = 1; b < M; ++b) {
            fma_limbs58(hi, mid, limbs_of(mc.mix[0][b]), to_limbs58(v[b], e));
            const double k = 1.0 / D[b];
            ref += (Q)k * v[b];
            big = max((double)big, 0.0) > fabs((double)(k * v[b])) ? big : (Q)fabs((double)(k * v[b]));
        }
        const double got = double_of_int64(hi + (mid >> 29), e - 1022 + mc.mix_exp);
        if (v[0] != 0 && big != 0) {
            double top = 0;
            for (int b = 0; b < M; ++b) top = max(top, fabs(v[b]));
            double kmax = 0;
            for (int b = 1; b < M; ++b) kmax = max(kmax, 1.0 / D[b]);
            ws = max(ws, fabs((double)((Q)got - ref)) / (fabs((double)ref) + 1.7 * top * kmax) * 0x1p53);
        }
    }
    printf("%.17g %.17g %.17g %ld %.17g\n", worst, worst_tau, sqrt(se / sr), wrong, ws);
    return 0;
}
