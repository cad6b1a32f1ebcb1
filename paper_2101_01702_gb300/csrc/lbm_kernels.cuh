// Kernels of the fused reactive-mixture lattice Boltzmann step.
//
// Included once by each precision translation unit after it defines
//   LBMK_MIXED 0 : every population stored and collided in double;
//   LBMK_MIXED 1 : the moving populations of the species and mixture sets
//                  stored as float deviations from per-set rest states and
//                  collided in float; their rest populations and the whole
//                  energy set in double (see pop_bytes_for);
//   LBMK_FAST 1  : (with LBMK_MIXED 1) also the relaxation rates, the
//                  Stefan-Maxwell solve and the 2^f of the rate
//                  exponentials in float (see SReal, WReal, exp_rate).
// Otherwise the moments, the temperature iteration (Eq. (temperature)),
// the Stefan-Maxwell system (Eq. (transform1)) and the reaction rates with
// their equilibrium constants have double precision in every unit.  The FP64
// pipe is the scarce resource of this GPU (two multiply-adds per SM and
// cycle): what does not need its range runs in fixed point on the integer pipe
// or in pairs of floats (lbm_fixed.cuh), to the same accuracy.
//
// One time step is six launches on one stream (seven with x ghosts; two fewer
// with two or three species, see kFewSpecies):
//   k_ghost  x-face ghost nodes (Sec. 5a; only for non-periodic x)
//   k_pre    pull, all moments, Newton temperature, relaxation rates, the
//            local part of the energy-flux correction and the energy
//            equilibrium moments; writes the per-node record
//   k_diff   Stefan-Maxwell diffusion velocities, beta_a
//   k_chem   production rates of the reaction mechanism
//   k_grad   G_alpha = (1/omega - 1/2) d_alpha Phi_alpha (Eq. (Xalpha))
//   k_step_g pull of the energy set, sum_a H_a grad Y_a from the neighbours'
//            records, and the collision of Eq. (g) (double)
//   k_step   pull of the species and mixture sets, X = -d_alpha G_alpha from
//            the neighbours' records, and the collisions of Eqs.
//            (finalNumericalEquations), (f), direction by direction
// One thread owns one lattice node; populations are structure-of-arrays
// [set][direction][node] so that a warp's pulls are coalesced rows.
#pragma once

#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "lbm_internal.h"
#include "lbm_fixed.cuh"

#ifndef LBMK_FAST
#define LBMK_FAST 0
#endif
// LBMK_CHECKED 1: every index the kernels derive from the lattice geometry
// (pulls from neighbours and ghost planes, stencil neighbours, ghost-node
// sources, batch ranges) is checked against its buffer before use; a bad one
// sets LBMK_BIT_BOUNDS in the status word and is replaced by 0, so that
// nothing traps and no access leaves its buffer.  A testing build.
#ifndef LBMK_CHECKED
#define LBMK_CHECKED 0
#endif

#if LBMK_MIXED
typedef float Real;
#else
typedef double Real;
#endif
// SReal: the relaxation rates, the Stefan-Maxwell factorisation and solve
// and the diffusion part of the energy-flux correction; WReal: the
// accumulation of the reaction contributions.  Double except in the fast
// mixed unit (LBMK_FAST), where these results, stored as floats, are also
// computed in float.
#if LBMK_MIXED && LBMK_FAST
typedef float SReal;
typedef float WReal;
#define INVWWD_S(a_, b_) (mc.inv_WWD_f[a_][b_])
#else
typedef double SReal;
typedef double WReal;
#define INVWWD_S(a_, b_) (mc.inv_WWD[a_][b_])
#endif

// Minimum resident blocks per SM asked of the compiler for the large
// kernels (register budget 65536 / (LBMK_BLOCK * minB)).  Measured, nine
// species: the moment pass with the diffusion pass, 256^3 mixed, at 3 + 3
// blocks 33.8 ms, 4 + 3 33.3, 3 + 4 32.2, 5 + 2 30.0 (6 + 2 and 5 + 1 the
// same); 160^3 fast mixed 5.62 ms at 5 + 3, 5.43 at 5 + 5, 5.88 at 6 + 2;
// 128^3 double 6.71 ms at 5 + 2, 6.75 at 4 + 4, 7.21 at 2 + 3.  The species and mixture
// collision runs fastest at 3 blocks in the mixed units (168 registers); the
// double one (lbm_collide64.cuh) takes the registers it can get, its shared
// memory holds it to 8 warps per SM;
// 256^3 mixed: 15.3 ms at 2 blocks, 12.1 ms at 3, 13.6 ms at 4.
#ifndef LBMK_PRE_MINB
#define LBMK_PRE_MINB 5
#endif
#ifndef LBMK_CHEM_MINB
#define LBMK_CHEM_MINB 4
#endif
#ifndef LBMK_DIFF_MINB
#define LBMK_DIFF_MINB (LBMK_FAST ? 5 : 2)
#endif
// The persistent kernel takes the budget of its heaviest phase, the species
// collision (the double one's shared memory allows two blocks).
#ifndef LBMK_PERSIST_MINB
#define LBMK_PERSIST_MINB (LBMK_MIXED ? 3 : 2)
#endif
#ifndef LBMK_STEP_MINB
#define LBMK_STEP_MINB (LBMK_MIXED ? 3 : 1)
#endif
// The moments of lbm_moments (outside the step), 256^3 mixed, T and Y:
// 44.0 ms at 178 registers (2 blocks per SM), 29.3 ms at 4 blocks, 23.8 ms
// at 5 (96 registers, ~200 B spilled); the double unit stays unconstrained
// (a cap of 128 registers spills 600 B there).
#ifndef LBMK_MOM_MINB
#define LBMK_MOM_MINB (LBMK_MIXED ? 5 : 1)
#endif
// Initialisation (equilibria of every set, outside the step; FP64-bound and
// insensitive to occupancy: 43.1-43.5 ms at 4 or 6 blocks per SM): 6 blocks
// (80 registers, ~30 B spilled).
// The energy collision is a kernel of its own (k_step_g): inside k_step it was
// slower (29.5 + 4.0 ms -> 47.0 ms, more spills at k_step's 168 registers).
#ifndef LBMK_INIT_MINB
#define LBMK_INIT_MINB 6
#endif
#if LBMK_MIXED
#define INVWWD(a_, b_) (mc.inv_WWD_f[a_][b_])
#define RA(a_) (mc.Ra_f[a_])
#else
#define INVWWD(a_, b_) (mc.inv_WWD[a_][b_])
#define RA(a_) (mc.Ra[a_])
#endif

static __constant__ MechConst c_mech[LBMK_SLOTS];

namespace {

// ---------------------------------------------------------------------
// Lattice helpers.  Direction i = (cx+1) + 3 (cy+1) + 9 (cz+1); 13 = rest.
// ---------------------------------------------------------------------
__host__ __device__ constexpr int CX(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int CY(int i) { return (i / 3) % 3 - 1; }
__host__ __device__ constexpr int CZ(int i) { return i / 9 - 1; }
__host__ __device__ constexpr double W1(int c) { return c == 0 ? 2.0 / 3.0 : 1.0 / 6.0; }
__host__ __device__ constexpr double WI(int i) { return W1(CX(i)) * W1(CY(i)) * W1(CZ(i)); }
constexpr int REST = 13;

// A lattice node and the x range [x0, x1) of the lattice it belongs to
// (lattice k of a batch placed side by side in x).
struct Node {
    int n, x, y, z;
    int x0, x1, k;
};

template <int I>
struct Dir {
    static constexpr int value = I;
};

// Compile-time loop over directions: f(Dir<I>{}), ..., f(Dir<N-1>{}).
template <int I, int N, class F>
__device__ __forceinline__ void for_dirs(F &&f)
{
    if constexpr (I < N) {
        f(Dir<I>{});
        for_dirs<I + 1, N>(f);
    }
}

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

__device__ __forceinline__ void flag(unsigned *status, unsigned bit) { atomicOr(status, bit); }

// Tests on the bit pattern (integer pipe; the FP64 pipe is the step's
// bottleneck): not Inf or NaN, and of a magnitude whose reciprocal is finite
// (above 2^-1024 and 2^-128; true for NaN).
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool finite_bits(float x) { return (__float_as_int(x) & 0x7f800000) != 0x7f800000; }
__device__ __forceinline__ bool invertible_bits(double x) { return (__double2hiint(x) & 0x7fffffff) > 0x00040000; }
__device__ __forceinline__ bool invertible_bits(float x) { return (__float_as_int(x) & 0x7fffffff) > 0x00200000; }

// Conversions between float and double on the integer pipe.  A hardware
// conversion between the two issues on the FP64 pipe, which bounds the
// moment pass; these give the same IEEE 754 result (binary32 <-> binary64,
// double -> float rounded to nearest, ties to even) with integer
// operations for zeros and normal results.  A warp with a lane outside
// that range (subnormals, overflow, Inf, NaN: rare here) takes the
// hardware conversion for all its lanes; the test is a warp vote, so the
// branch is uniform and the common path issues no FP64 instruction.
__device__ __forceinline__ double f2d(float f)
{
    const unsigned b = __float_as_uint(f), mag = b & 0x7fffffffu;
    const bool rare = (mag >> 23) - 1u >= 254u && mag != 0u;            // subnormal, Inf, NaN
    if (__builtin_expect(__any_sync(__activemask(), rare), 0)) return (double)f;
    // exponent rebiased by 1023 - 127 = 896; the low 3 mantissa bits move to the low word
    const unsigned hi = (b & 0x80000000u) | (mag ? (mag >> 3) + (896u << 20) : 0u);
    return __hiloint2double((int)hi, (int)(mag << 29));
}

__device__ __forceinline__ float d2f(double d)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned hm = hi & 0x7fffffffu;
    const bool zero = (hm | lo) == 0u;
    // normal float results: biased double exponent in [897, 1150]
    const bool rare = (hm >> 20) - 897u > 253u && !zero;
    if (__builtin_expect(__any_sync(__activemask(), rare), 0)) return __double2float_rn(d);
    const unsigned m = ((hm - (896u << 20)) << 3) | (lo >> 29);     // float exponent and mantissa, truncated
    const unsigned rem = lo & 0x1fffffffu;                          // the 29 bits dropped
    const unsigned up = (rem > 0x10000000u) | ((rem == 0x10000000u) & m);
    return __uint_as_float((hi & 0x80000000u) | (zero ? 0u : m + up));   // a carry rounds into the exponent
}

// x converted to To (a plain copy when the types agree).
template <class To, class From>
__device__ __forceinline__ To cvt(From x)
{
    if constexpr (std::is_same<To, From>::value) return x;
    else if constexpr (std::is_same<To, double>::value && std::is_same<From, float>::value) return f2d(x);
    else if constexpr (std::is_same<To, float>::value && std::is_same<From, double>::value) return d2f(x);
    else return (To)x;
}

// Checked builds: records a failed index check; always true otherwise.
__device__ __forceinline__ bool index_ok(bool ok, unsigned *status)
{
#if LBMK_CHECKED
    if (!ok) flag(status, LBMK_BIT_BOUNDS);
    return ok;
#else
    (void)ok;
    (void)status;
    return true;
#endif
}

// Populations and ghost planes are read through the read-only data path
// (__ldg) in the per-phase kernels, none of which reads what it writes.
// The persistent kernel writes, within its one launch, what its later
// phases read, so its units build with LBMK_COHERENT_LOADS=1: plain loads,
// ordered by the grid barrier's fences.
#ifndef LBMK_COHERENT_LOADS
#define LBMK_COHERENT_LOADS 0
#endif
#if LBMK_COHERENT_LOADS
#define LBMK_LDG(p_) (*(p_))
#else
#define LBMK_LDG(p_) __ldg(p_)
#endif

// ---------------------------------------------------------------------
// Population storage (see pop_bytes_for).
// ---------------------------------------------------------------------
struct PopView {
    const void *buf;
    int N, M;
#if LBMK_MIXED
    __device__ const float *mov() const { return static_cast<const float *>(buf); }
    __device__ const double *rest() const
    {
        return reinterpret_cast<const double *>(static_cast<const char *>(buf) + pop_float_bytes(M, N));
    }
    __device__ const double *g() const { return rest() + (size_t)M * N; }
#endif
};

__device__ __forceinline__ PopView view(const void *buf, const StepArgs &a) { return PopView{buf, a.N, a.M}; }

// Value of species/mixture set s (< M), direction i, at buffer node idx;
// absolute (the rest state is added back in mixed precision).
__device__ __forceinline__ Real load_sf(const MechConst &mc, const PopView &v, int s, int i, size_t idx)
{
#if LBMK_MIXED
    if (i == REST) return (Real)v.rest()[(size_t)s * v.N + idx];
    return LBMK_LDG(v.mov() + ((size_t)s * LBMK_Q + i) * v.N + idx) + mc.ref[s][i];
#else
    return LBMK_LDG(static_cast<const double *>(v.buf) + ((size_t)s * LBMK_Q + i) * v.N + idx);
#endif
}

// Stored value of species/mixture set s (< M), moving direction i, at
// buffer node idx: in mixed precision the deviation from the rest state
// RAWREF(s, i); the population is the stored value + RAWREF(s, i).
__device__ __forceinline__ Real load_raw_sf(const PopView &v, int s, int i, size_t idx)
{
#if LBMK_MIXED
    return LBMK_LDG(v.mov() + ((size_t)s * LBMK_Q + i) * v.N + idx);
#else
    return LBMK_LDG(static_cast<const double *>(v.buf) + ((size_t)s * LBMK_Q + i) * v.N + idx);
#endif
}
#if LBMK_MIXED
#define RAWREF(s_, i_) (mc.ref[s_][i_])
#else
#define RAWREF(s_, i_) ((Real)0)
#endif

// The same in double, keeping the double rest population exact.
__device__ __forceinline__ double load_sf_d(const MechConst &mc, const PopView &v, int s, int i, size_t idx)
{
#if LBMK_MIXED
    if (i == REST) return v.rest()[(size_t)s * v.N + idx];
#endif
    return (double)load_sf(mc, v, s, i, idx);
}

// Energy-set value, direction i, at buffer node idx (double in both precisions).
__device__ __forceinline__ double load_g(const PopView &v, int i, size_t idx)
{
#if LBMK_MIXED
    return LBMK_LDG(v.g() + (size_t)i * v.N + idx);
#else
    return LBMK_LDG(static_cast<const double *>(v.buf) + ((size_t)v.M * LBMK_Q + i) * v.N + idx);
#endif
}

// Where a pulled population comes from: s(x) = s_post(x - c).
struct PullIdx {
    int xs[3];    // x - c for c = -1, 0, 1
    int gp[3];    // ghost plane of x - c (2k left, 2k+1 right face of lattice k), -1 inside
    int yz[9];    // y' + ny z' for (cy, cz)
};

__device__ __forceinline__ void make_pull(PullIdx &p, const Node &nd, const StepArgs &a)
{
    for (int c = -1; c <= 1; ++c) {
        int xs = nd.x - c, gp = -1;
        if (a.bc_x == 0) xs = wrapi(xs, a.nx);
        else if (xs < nd.x0) gp = 2 * nd.k;
        else if (xs >= nd.x1) gp = 2 * nd.k + 1;
        p.xs[c + 1] = xs;
        p.gp[c + 1] = gp;
    }
    for (int cz = -1; cz <= 1; ++cz)
        for (int cy = -1; cy <= 1; ++cy)
            p.yz[(cy + 1) + 3 * (cz + 1)] = wrapi(nd.y - cy, a.ny) + a.ny * wrapi(nd.z - cz, a.nz);
}

// Source of direction i: a buffer node, or (ghost plane, index in the plane).
struct Src {
    bool ghost;
    int side;     // ghost plane (see PullIdx::gp)
    size_t idx;
};

// GH false: for a node none of whose pulls reaches a ghost plane.
template <bool GH = true>
__device__ __forceinline__ Src src_of(int i, const PullIdx &p, const StepArgs &a)
{
    const int xs = p.xs[CX(i) + 1];
    const int gp = GH ? p.gp[CX(i) + 1] : -1;
    const int yz = p.yz[(CY(i) + 1) + 3 * (CZ(i) + 1)];
    if (gp >= 0) {
        const int nlat = a.nseg > 1 ? a.nseg : 1;
        if (!index_ok(gp < 2 * nlat && yz >= 0 && yz < a.ny * a.nz, a.status)) return Src{false, 0, 0};
        return Src{true, gp, (size_t)yz};
    }
    const size_t idx = (size_t)xs + (size_t)a.nx * yz;
    if (!index_ok(xs >= 0 && xs < a.nx && yz >= 0 && idx < (size_t)a.N, a.status)) return Src{false, 0, 0};
    return Src{false, 0, idx};
}

__device__ __forceinline__ double load_ghost(const StepArgs &a, int plane_idx, int s, int i, size_t yz)
{
    const size_t plane = (size_t)a.ny * a.nz;
    return LBMK_LDG(static_cast<const double *>(a.ghost) + ((size_t)(plane_idx * (a.M + 1) + s) * LBMK_Q + i) * plane +
                 yz);
}

template <bool GH = true>
__device__ __forceinline__ Real pull_sf(const MechConst &mc, const PopView &v, const StepArgs &a, int s, int i,
                                        const PullIdx &p)
{
    const Src sr = src_of<GH>(i, p, a);
    return sr.ghost ? (Real)load_ghost(a, sr.side, s, i, sr.idx) : load_sf(mc, v, s, i, sr.idx);
}

template <bool GH = true>
__device__ __forceinline__ double pull_g(const PopView &v, const StepArgs &a, int i, const PullIdx &p)
{
    const Src sr = src_of<GH>(i, p, a);
    return sr.ghost ? load_ghost(a, sr.side, a.M, i, sr.idx) : load_g(v, i, sr.idx);
}

// Writers of the post-collision state at node n.  store_raw writes the
// stored value of a moving population of a species/mixture set: in the
// mixed units its deviation from the rest state RAWREF(s, i), in double
// the population; store_sf takes an absolute double value, any direction.
__device__ __forceinline__ void store_raw(void *buf, const StepArgs &a, int s, int i, size_t n, Real v)
{
    static_cast<Real *>(buf)[((size_t)s * LBMK_Q + i) * a.N + n] = v;
}

__device__ __forceinline__ void store_sf(const MechConst &mc, void *buf, const StepArgs &a, int s, int i, size_t n,
                                         double v)
{
#if LBMK_MIXED
    const size_t N = a.N;
    if (i == REST) {
        reinterpret_cast<double *>(static_cast<char *>(buf) + pop_float_bytes(a.M, N))[(size_t)s * N + n] = v;
    } else {
        static_cast<float *>(buf)[((size_t)s * LBMK_Q + i) * N + n] = cvt<float>(v) - mc.ref[s][i];
    }
#else
    static_cast<double *>(buf)[((size_t)s * LBMK_Q + i) * a.N + n] = v;
#endif
}

__device__ __forceinline__ void store_g(void *buf, const StepArgs &a, int i, size_t n, double v)
{
#if LBMK_MIXED
    const size_t N = a.N;
    reinterpret_cast<double *>(static_cast<char *>(buf) + pop_float_bytes(a.M, N))[(size_t)a.M * N + (size_t)i * N + n] = v;
#else
    static_cast<double *>(buf)[((size_t)a.M * LBMK_Q + i) * a.N + n] = v;
#endif
}

// Stencil neighbours x + c (periodic, or clamped to the node's own lattice
// for zero-gradient x faces).
struct StencilIdx {
    int xs[3];
    int row[9];
};

__device__ __forceinline__ void make_stencil(StencilIdx &t, const Node &nd, const StepArgs &a)
{
    for (int c = -1; c <= 1; ++c) {
        int xn = nd.x + c;
        if (a.bc_x == 0) xn = wrapi(xn, a.nx);
        else xn = xn < nd.x0 ? nd.x0 : (xn >= nd.x1 ? nd.x1 - 1 : xn);
        t.xs[c + 1] = xn;
    }
    for (int cz = -1; cz <= 1; ++cz)
        for (int cy = -1; cy <= 1; ++cy)
            t.row[(cy + 1) + 3 * (cz + 1)] = a.nx * (wrapi(nd.y + cy, a.ny) + a.ny * wrapi(nd.z + cz, a.nz));
}

template <int I>
__device__ __forceinline__ size_t nb_of(const StencilIdx &t, const StepArgs &a)
{
    const size_t nb = (size_t)t.xs[CX(I) + 1] + t.row[(CY(I) + 1) + 3 * (CZ(I) + 1)];
    return index_ok(nb < (size_t)a.N, a.status) ? nb : 0;
}

__device__ __forceinline__ Real *rec(const StepArgs &a)
{
    return reinterpret_cast<Real *>(a.macro + (size_t)macro_double_rows(a.M) * a.N);
}

// ---------------------------------------------------------------------
// Thermodynamics (Eqs. (specHa), (Umix), (temperature)).
// ---------------------------------------------------------------------
template <int M>
__device__ __forceinline__ void mixture_energy_poly(const MechConst &mc, const double *Y, double u[6])
{
#pragma unroll
    for (int k = 0; k < 6; ++k) u[k] = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a)
#pragma unroll
        for (int k = 0; k < 6; ++k) u[k] = fma(Y[a], mc.uco[a][k], u[k]);
}

__device__ __forceinline__ double poly5(const double u[6], double T)
{
    return fma(fma(fma(fma(fma(u[5], T, u[4]), T, u[3]), T, u[2]), T, u[1]), T, u[0]);
}

__device__ __forceinline__ double dpoly5(const double u[6], double T)
{
    return fma(fma(fma(fma(5.0 * u[5], T, 4.0 * u[4]), T, 3.0 * u[3]), T, 2.0 * u[2]), T, u[1]);
}

// Newton iteration on U(T) = e from T.  The residual is formed in double;
// the derivative and the quotient, which only scale the correction, in float
// (a float division and conversions on the integer pipe in place of 13
// FP64 operations per iteration).  It stops once a correction is at most
// 5e-10 T: the error left is then the correction's relative error, 2e-7, of
// that and Newton's quadratic term, (C_v'/2C_v) dT^2: 1e-16 T in all.
__device__ __forceinline__ double solve_T(const double u[6], double e, double T, unsigned *status)
{
    const float d5 = 5.0f * d2f(u[5]), d4 = 4.0f * d2f(u[4]), d3 = 3.0f * d2f(u[3]), d2 = 2.0f * d2f(u[2]),
                d1 = d2f(u[1]);                               // C_v's coefficients
    for (int it = 0; it < 50; ++it) {
        const float t = d2f(T);
        const float dT = d2f(poly5(u, T) - e) / fma(fma(fma(fma(d5, t, d4), t, d3), t, d2), t, d1);
        T -= f2d(dT);
        if (!finite_bits(T)) { flag(status, LBMK_BIT_NONFINITE); return T; }
        if (fabsf(dT) <= 5e-10f * fabsf(t)) return T;
    }
    flag(status, LBMK_BIT_NEWTON);
    return T;
}

// Species specific enthalpy H_a(T).
__device__ __forceinline__ double H_spec(const MechConst &mc, int a, double T)
{
    const double *h = mc.hco[a];
    return fma(fma(fma(fma(fma(h[4], T, h[3]), T, h[2]), T, h[1]), T, h[0]), T, h[5]);
}

// Specific heat C_p,a(T) = dH_a/dT.
__device__ __forceinline__ double cp_spec(const MechConst &mc, int a, double T)
{
    const double *h = mc.hco[a];
    return fma(fma(fma(fma(5.0 * h[4], T, 4.0 * h[3]), T, 3.0 * h[2]), T, 2.0 * h[1]), T, h[0]);
}

__device__ __forceinline__ double nu_prime(const MechConst &mc, double Rm, double T)
{
    return mc.visc_model == 0 ? mc.nu / (Rm * T) : mc.nu;
}

// Mixture-averaged transport of a node state (mc.transport = 1; Sec. 3
// after Eq. (lambda), where the paper takes the coefficients from Cantera):
// species viscosities mu_a = mu0_a (T/T_tr)^s_a, Wilke's mixing rule
//   mu = sum_a X_a mu_a / sum_b X_b Phi_ab,
//   Phi_ab = (1 + (mu_a/mu_b)^(1/2) (W_b/W_a)^(1/4))^2 / (8 (1 + W_a/W_b))^(1/2),
// Eucken's lambda_a = mu_a (C_p,a + 5/4 R_a) with the average of Mathur,
// Tondon and Saxena lambda = (sum X_a lambda_a + 1/sum X_a/lambda_a)/2;
// returns 1/omega - 1/2 = mu/P (Eq. (mu)), 1/omega_1 - 1/2 = lambda/(P C_p)
// (Eq. (lambda)) in the storage type, and the factor dfac =
// (T/T_tr)^D_exp P_tr/P of every binary diffusivity (Eq. (tauab)).
template <int M>
__device__ void mixture_transport(const MechConst &mc, const double *Y, double inv_m, double T, double P,
                                  double Cp, Real &nup, Real &nup1, double &dfac)
{
    const double lnT = log(T) - mc.log_T_tr;
    const Real iim = (Real)(1.0 / inv_m);
    Real X[M], mu[M], r[M], ir[M];
#pragma unroll
    for (int a = 0; a < M; ++a) {
        X[a] = (Real)(Y[a] * mc.invW[a]) * iim;
        mu[a] = (Real)mc.mu0[a] * exp((Real)(mc.mu_exp[a] * lnT));
        r[a] = sqrt(mu[a]);
        ir[a] = (Real)1 / r[a];
    }
    Real num = 0, ls = 0, lr = 0;
#pragma unroll
    for (int a = 0; a < M; ++a) {
        Real den = 0;
#pragma unroll
        for (int b = 0; b < M; ++b) {
            const Real t = fma(r[a] * ir[b], (Real)mc.wq[a][b], (Real)1);
            den = fma(X[b], t * t * (Real)mc.wd[a][b], den);
        }
        num += X[a] * mu[a] / den;
        const Real lam = mu[a] * (Real)(cp_spec(mc, a, T) + mc.eucken[a]);
        ls = fma(X[a], lam, ls);
        lr += X[a] / lam;
    }
    const Real lambda = (Real)0.5 * (ls + (Real)1 / lr);
    nup = num / (Real)P;
    nup1 = lambda / (Real)(P * Cp);
    dfac = exp(mc.D_exp * lnT) * mc.P_tr / P;
}

// Product-form factor Psi_c(xi, zeta) of Eq. (phis) with s = xi^2 + zeta.
template <class V>
__device__ __forceinline__ V psi_c(int c, V xi, V s)
{
    return c == 0 ? (V)1 - s : (V)0.5 * (s + (V)c * xi);
}

// Energy equilibrium moments (Eqs. (geq1mom), (geq2mom)): q^eq, R^eq -
// rhoE theta I (xx yy zz xy xz yz) and a third of its trace.
__device__ __forceinline__ void energy_moments(double rho, const double *u, double P, double hk, double rhoE,
                                               double qeq[3], double Rt[6], double &tr3)
{
    const double hP = fma(hk, rho, P), third = rhoE / 3.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        qeq[d] = hk * rho * u[d];
        Rt[d] = fma(hk, P, fma(hP * u[d], u[d], -third));
    }
    Rt[3] = hP * u[0] * u[1];
    Rt[4] = hP * u[0] * u[2];
    Rt[5] = hP * u[1] * u[2];
    tr3 = (Rt[0] + Rt[1] + Rt[2]) * (1.0 / 3.0);
}

// Sums of products in the double passes are written with fma throughout: left
// to the compiler, which products it fuses differs between builds (the
// bounds-checked one, the persistent kernel), and so do the last bits.
__device__ __forceinline__ double dot3(const double *a, const double *b)
{
    return fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0]));
}

// Grad population of direction i (Eqs. (gieq), (giqeq)) for given moments.
__device__ __forceinline__ double grad_dir(int i, double rhoE, const double q[3], const double Rt[6], double tr3)
{
    const int cx = CX(i), cy = CY(i), cz = CZ(i);
    double qc = 0.0, rcc = 0.0;
    if (cx) { qc += cx * q[0]; rcc += Rt[0]; }
    if (cy) { qc += cy * q[1]; rcc += Rt[1]; }
    if (cz) { qc += cz * q[2]; rcc += Rt[2]; }
    if (cx && cy) rcc += 2.0 * (cx * cy) * Rt[3];
    if (cx && cz) rcc += 2.0 * (cx * cz) * Rt[4];
    if (cy && cz) rcc += 2.0 * (cy * cz) * Rt[5];
    return WI(i) * fma(4.5, rcc - tr3, fma(3.0, qc, rhoE));
}

// Equilibrium of every set at (rho_a, u, T), in double, handed to put(s, i, v).
template <int M, class Put>
__device__ void equilibria(const MechConst &mc, const double *rho_a, const double *u, double T, Put &&put)
{
    double rho = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) rho += rho_a[a];
    double Y[M], inv_m = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) { Y[a] = rho_a[a] / rho; inv_m += Y[a] * mc.invW[a]; }
    const double Rm = mc.r_lat * inv_m;
    const double usq = dot3(u, u);
#pragma unroll
    for (int s = 0; s < M; ++s) {
        const double zeta = (s < M - 1 ? mc.Ra[s] : Rm) * T;
        const double r = s < M - 1 ? rho_a[s] : rho;
        double P3[3][3];
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int c = -1; c <= 1; ++c) P3[d][c + 1] = psi_c(c, u[d], u[d] * u[d] + zeta);
#pragma unroll
        for (int i = 0; i < LBMK_Q; ++i) put(s, i, r * P3[0][CX(i) + 1] * P3[1][CY(i) + 1] * P3[2][CZ(i) + 1]);
    }
    double eu[6];
    mixture_energy_poly<M>(mc, Y, eu);
    const double U = poly5(eu, T);
    double H = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) H = fma(Y[a], H_spec(mc, a, T), H);
    const double rhoE = rho * (U + 0.5 * usq);
    const double P = rho * Rm * T;
    double q[3], Rt[6], tr3;
    energy_moments(rho, u, P, H + 0.5 * usq, rhoE, q, Rt, tr3);
#pragma unroll
    for (int i = 0; i < LBMK_Q; ++i) put(M, i, grad_dir(i, rhoE, q, Rt, tr3));
}

// Coordinates and lattice range of node nd.n (0 <= nd.n < a.N).
__device__ __forceinline__ void node_at(Node &nd, const StepArgs &a)
{
    nd.x = nd.n % a.nx;
    const int r = nd.n / a.nx;
    nd.y = r % a.ny;
    nd.z = r / a.ny;
    if (a.xseg) {
        const int4 e = __ldg(a.xseg + nd.x);
        nd.x0 = e.x;
        nd.x1 = e.y;
        nd.k = e.z;
        if (!index_ok(e.x <= nd.x && nd.x < e.y && e.y <= a.nx && e.z >= 0 && e.z < a.nseg, a.status)) {
            nd.x0 = nd.x;
            nd.x1 = nd.x + 1;
            nd.k = 0;
        }
    } else {
        nd.x0 = 0;
        nd.x1 = a.nx;
        nd.k = 0;
    }
}

__device__ __forceinline__ bool node_of(Node &nd, const StepArgs &a)
{
    nd.n = blockIdx.x * blockDim.x + threadIdx.x;
    if (nd.n >= a.N) return false;
    node_at(nd, a);
    return true;
}

// Moments of one set from its 27 populations, row by row: the directions
// come in 9 rows (cy, cz) of three (cx = -1, 0, 1); per row t = f- + f0 + f+
// and dx = f+ - f-, so that
//   sum f = sum t,  sum c_x f = sum dx,  sum c_y f = sum cy t,  sum c_z f = sum cz t,
//   P_xx = sum (f- + f+), P_yy = sum_{cy != 0} t, P_zz = sum_{cz != 0} t,
//   P_xy = sum cy dx, P_xz = sum cz dx, P_yz = sum cy cz t
// (57 additions for the first four instead of 81 direction by direction).
// ld(Dir<I>{}) returns the population of direction I.
template <bool WITH_P, class V, class LD>
__device__ __forceinline__ void row_moments(LD &&ld, V &s0, V &sx, V &sy, V &sz, V *P6)
{
    for_dirs<0, 9>([&](auto dj) {
        constexpr int j = decltype(dj)::value, cy = j % 3 - 1, cz = j / 3 - 1;
        const V fm = ld(Dir<3 * j>{}), f0 = ld(Dir<3 * j + 1>{}), fp = ld(Dir<3 * j + 2>{});
        const V ac = fm + fp, t = ac + f0, dx = fp - fm;
        if constexpr (j == 0) {                           // cy = cz = -1
            s0 = t;
            sx = dx;
            sy = -t;
            sz = -t;
            if constexpr (WITH_P) {
                P6[0] = ac;
                P6[1] = t;
                P6[2] = t;
                P6[3] = -dx;
                P6[4] = -dx;
                P6[5] = t;
            }
        } else {
            s0 += t;
            sx += dx;
            if constexpr (cy == 1) sy += t;
            if constexpr (cy == -1) sy -= t;
            if constexpr (cz == 1) sz += t;
            if constexpr (cz == -1) sz -= t;
            if constexpr (WITH_P) {
                P6[0] += ac;
                if constexpr (cy != 0) P6[1] += t;
                if constexpr (cz != 0) P6[2] += t;
                if constexpr (cy == 1) P6[3] += dx;
                if constexpr (cy == -1) P6[3] -= dx;
                if constexpr (cz == 1) P6[4] += dx;
                if constexpr (cz == -1) P6[4] -= dx;
                if constexpr (cy * cz == 1) P6[5] += t;
                if constexpr (cy * cz == -1) P6[5] -= t;
            }
        }
    });
}

// The same sums of 27 doubles on the integer pipe: the moving populations are
// brought to the largest one's exponent (to 2^-57 of it) and added as
// integers, each sum rounded once; the rest population, up to a thousand
// times larger and part of the zeroth moment alone, is added in double.  57
// (94 with WITH_P) FP64 additions, 76 cycles of a scheduler each, become
// about 600 (700) integer instructions.  What is dropped is below 2^-57 of
// the largest moving population from each, downwards from all of one sign,
// so that most of it cancels in the first moments.
template <bool WITH_P, class LD>
__device__ __forceinline__ void fixed_row_moments(LD &&ld, double &s0, double &sx, double &sy, double &sz, double *P6)
{
    double v[LBMK_Q];
    int e = 0;
    for_dirs<0, LBMK_Q>([&](auto d) {
        constexpr int I = decltype(d)::value;
        v[I] = ld(d);
        if constexpr (I != REST) e = max(e, biased_exponent(v[I]));
    });
    long long t0, tx, ty, tz, tP[6];
    row_moments<WITH_P, long long>([&](auto d) {
        constexpr int I = decltype(d)::value;
        return I == REST ? 0ll : to_fixed58(v[I], e);
    }, t0, tx, ty, tz, tP);
    const bool nan = e == 0x7ff;                           // an infinite or NaN population
    auto out = [&](long long x) {
        return nan ? __longlong_as_double(0x7ff8000000000000ll) : double_of_int64(x, e - 1080);
    };
    s0 = out(t0) + v[REST];
    sx = out(tx);
    sy = out(ty);
    sz = out(tz);
    if constexpr (WITH_P)
#pragma unroll
        for (int k = 0; k < 6; ++k) P6[k] = out(tP[k]);
}

// In the mixed units the moving populations are summed as the stored float
// deviations from the set's rest state; its moments (ref0, refP: double,
// the first moments vanish) and the double rest population are added once.
#if LBMK_MIXED
template <bool GH>
__device__ __forceinline__ Real pull_dev(const MechConst &mc, const PopView &v, const StepArgs &a, int s, int i,
                                         const PullIdx &p)
{
    const Src sr = src_of<GH>(i, p, a);
    return sr.ghost ? (Real)load_ghost(a, sr.side, s, i, sr.idx) - RAWREF(s, i) : load_raw_sf(v, s, i, sr.idx);
}
#endif

// Zeroth and first moments (and with WITH_P the second) of species or
// mixture set s < M; the first as summed, in the storage type.
template <bool WITH_P, bool GH>
__device__ __forceinline__ void set_moments(const MechConst &mc, const PopView &v, const StepArgs &a, const PullIdx &p,
                                            int n, int s, double &r, Real *j, double *P)
{
#if LBMK_MIXED
    Real a0, P6[6];
    row_moments<WITH_P, Real>([&](auto d) {
        constexpr int I = decltype(d)::value;
        return I == REST ? (Real)0 : pull_dev<GH>(mc, v, a, s, I, p);           // the double rest population: below
    }, a0, j[0], j[1], j[2], P6);
    r = cvt<double>(a0) + (mc.ref0[s] + v.rest()[(size_t)s * v.N + n]);
    if constexpr (WITH_P)
#pragma unroll
        for (int k = 0; k < 6; ++k) P[k] = cvt<double>(P6[k]) + (k < 3 ? mc.refP[s][k] : 0.0);
#else
    (void)n;
    fixed_row_moments<WITH_P>([&](auto d) { return pull_sf<GH>(mc, v, a, s, decltype(d)::value, p); }, r, j[0], j[1], j[2],
                              P);
#endif
}

// Moments of the pulled populations of a node: the mixture set gives rho,
// rho u and (WITH_P) the pressure tensor, the energy set rho E and q, and
// each species its density and momentum, the last one slaved (Eq.
// (strongest)), handed to put(s, rho_a, j_a) in order after rho and rho u
// are known (in sm).  The loop over the species is not unrolled, see
// pre_node.
struct Sums {
    double rho, j[3], P[6], rhoE, q[3];   // P: xx, yy, zz, xy, xz, yz
};

template <int M, bool WITH_P, class Put>
__device__ __forceinline__ void pull_moments(const MechConst &mc, const StepArgs &a, const PullIdx &p, int n, Sums &sm,
                                             Put &&put)
{
    const PopView v = view(a.src, a);
    // nodes away from the x faces of a lattice take code without the ghost
    // planes (whole warps of them, for all but the shortest lattices)
    const bool inside = p.gp[0] < 0 && p.gp[2] < 0;
    Real js[3];
    if (inside) set_moments<WITH_P, false>(mc, v, a, p, n, M - 1, sm.rho, js, sm.P);
    else set_moments<WITH_P, true>(mc, v, a, p, n, M - 1, sm.rho, js, sm.P);
#pragma unroll
    for (int d = 0; d < 3; ++d) sm.j[d] = cvt<double>(js[d]);
    double rest = 0.0;
#pragma unroll 1
    for (int s = 0; s < M; ++s) {
        double ra;
        Real j[3];
        if (s < M - 1) {
            if (inside) set_moments<false, false>(mc, v, a, p, n, s, ra, j, nullptr);
            else set_moments<false, true>(mc, v, a, p, n, s, ra, j, nullptr);
            rest += ra;
#pragma unroll
            for (int d = 0; d < 3; ++d) js[d] -= j[d];
        } else {
            ra = sm.rho - rest;
#pragma unroll
            for (int d = 0; d < 3; ++d) j[d] = js[d];
        }
        put(s, ra, j);
    }
    if (inside)
        fixed_row_moments<false>([&](auto d) { return pull_g<false>(v, a, decltype(d)::value, p); }, sm.rhoE, sm.q[0],
                                 sm.q[1], sm.q[2], nullptr);
    else
        fixed_row_moments<false>([&](auto d) { return pull_g<true>(v, a, decltype(d)::value, p); }, sm.rhoE, sm.q[0],
                                 sm.q[1], sm.q[2], nullptr);
}

// ---------------------------------------------------------------------
// Initialisation: every set at equilibrium for X, T, u and pressure P.
// ---------------------------------------------------------------------
template <int M>
__global__ void __launch_bounds__(LBMK_BLOCK, LBMK_INIT_MINB) k_init(StepArgs a, const double *X, const double *Tf,
                                                     const double *uf, double P)
{
    const MechConst &mc = c_mech[a.slot];
    Node nd;
    if (!node_of(nd, a)) return;
    const int n = nd.n;
    double m = 0.0;
#pragma unroll
    for (int s = 0; s < M; ++s) m += X[(size_t)s * a.N + n] * mc.W[s];
    const double T = Tf[n];
    const double rho = P / (mc.r_lat / m * T);
    double rho_a[M];
#pragma unroll
    for (int s = 0; s < M; ++s) rho_a[s] = rho * X[(size_t)s * a.N + n] * mc.W[s] / m;
    double u[3] = {0.0, 0.0, 0.0};
    if (uf)
        for (int d = 0; d < 3; ++d) u[d] = uf[(size_t)d * a.N + n];
    equilibria<M>(mc, rho_a, u, T, [&](int s, int i, double v) {
        if (s < M) store_sf(mc, a.dst, a, s, i, n, v);
        else store_g(a.dst, a, i, n, v);
    });
    a.macro[(size_t)DR_T * a.N + n] = T;
}

// ---------------------------------------------------------------------
// Ghost nodes beyond the x faces (Sec. 5a): equilibria at the
// post-collision moments of the adjacent boundary node, u = 0 on the left.
//
// One lane per set: a group of M + 1 lanes forms a ghost node, each lane the
// sums, then the equilibrium populations, of its set (the energy set's are
// dealt out over the group).  There are few ghost nodes (32 in a 4 x 4
// tube), so the kernel's time is the serial chain of one thread, 64 cycles
// per double operation: 86 us in a 4 x 4 tube with one thread per node, 19
// (double) and 25 us (mixed) with a group; 34 instead of 125 us for 48 tubes.
// ---------------------------------------------------------------------
template <int M>
constexpr int ghost_groups() { return 32 / (M + 1); }      // ghost nodes per warp

__host__ __device__ inline int ghost_count(const StepArgs &a) { return 2 * (a.nseg > 1 ? a.nseg : 1) * a.ny * a.nz; }

// The ghost nodes of warp w (whole warps only).
template <int M>
__device__ __forceinline__ void ghost_warp(const StepArgs &a, int w)
{
    constexpr int S = M + 1;
    const MechConst &mc = c_mech[a.slot];
    const int lane = threadIdx.x & 31, plane = a.ny * a.nz;
    int grp = lane / S;
    const int s = lane % S;
    int t = w * ghost_groups<M>() + grp;
    const bool live = grp < ghost_groups<M>() && t < ghost_count(a);
    if (!live) {                                       // idle lanes follow the first node
        t = w * ghost_groups<M>();
        grp = 0;
    }
    const int base = grp * S;
    const int gp = t / plane, yz = t % plane;          // ghost plane 2k + side of lattice k
    const int side = gp & 1, k = gp >> 1;
    int x0 = 0, x1 = a.nx;
    if (a.segs) {
        const int2 r = __ldg(a.segs + k);
        x0 = r.x;
        x1 = r.y;
    }
    size_t n = (size_t)(side ? x1 - 1 : x0) + (size_t)a.nx * yz;
    if (!index_ok(x0 >= 0 && x0 < x1 && x1 <= a.nx && n < (size_t)a.N, a.status)) n = 0;
    const PopView v = view(a.src, a);
    double m0, mx, my, mz;
    row_moments<false, double>([&](auto d) {
        constexpr int I = decltype(d)::value;
        return s < M ? load_sf_d(mc, v, s, I, n) : load_g(v, I, n);
    }, m0, mx, my, mz, nullptr);
    auto from = [&](double x, int set) { return __shfl_sync(0xffffffffu, x, base + set); };
    const double rho = from(m0, M - 1), rhoE = from(m0, M), ir = 1.0 / rho;
    double u[3] = {from(mx, M - 1) * ir, from(my, M - 1) * ir, from(mz, M - 1) * ir};
    double Y[M], rest = 0.0, inv_m = 0.0;
#pragma unroll
    for (int b = 0; b < M - 1; ++b) {
        const double ra = from(m0, b);
        rest += ra;
        Y[b] = ra * ir;
    }
    Y[M - 1] = (rho - rest) * ir;
#pragma unroll
    for (int b = 0; b < M; ++b) inv_m = fma(Y[b], mc.invW[b], inv_m);
    // coefficients of the mixture energy, dealt out over the group
    double eu[6];
    {
        constexpr int NK = (6 + S - 1) / S;
        double part[NK];
#pragma unroll
        for (int j = 0; j < NK; ++j) {
            const int kk = s + j * S < 6 ? s + j * S : 0;
            part[j] = 0.0;
#pragma unroll
            for (int b = 0; b < M; ++b) part[j] = fma(Y[b], mc.uco[b][kk], part[j]);
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) eu[q] = from(part[q / S], q % S);
    }
    const double e = fma(rhoE, ir, -0.5 * dot3(u, u));
    const double T = solve_T(eu, e, a.macro[(size_t)DR_T * a.N + n], a.status);
    if (side == 0) u[0] = u[1] = u[2] = 0.0;
    const double Rm = mc.r_lat * inv_m;
    double *gh = static_cast<double *>(a.ghost) + (size_t)gp * S * LBMK_Q * plane + yz;
    if (s < M) {
        const double zeta = __dmul_rn(s < M - 1 ? mc.Ra[s] : Rm, T);
        const double r = s < M - 1 ? m0 : rho;
        double P3[3][3];
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int c = -1; c <= 1; ++c) P3[d][c + 1] = psi_c(c, u[d], fma(u[d], u[d], zeta));
#pragma unroll
        for (int cz = 0; cz < 3; ++cz)
#pragma unroll
            for (int cy = 0; cy < 3; ++cy) {
                const double ryz = r * P3[2][cz] * P3[1][cy];
#pragma unroll
                for (int cx = 0; cx < 3; ++cx)
                    if (live) gh[((size_t)s * LBMK_Q + cx + 3 * cy + 9 * cz) * plane] = ryz * P3[0][cx];
            }
    }
    // energy set: rho E and H of the state with the ghost's velocity
    const double U = poly5(eu, T), usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const double rE = rho * fma(0.5, usq, U), P = rho * Rm * T;
    double q[3], Rt[6], tr3;
    energy_moments(rho, u, P, fma(0.5, usq, fma(Rm, T, U)), rE, q, Rt, tr3);
    for (int i = s; i < LBMK_Q; i += S)
        if (live) gh[((size_t)M * LBMK_Q + i) * plane] = grad_dir(i, rE, q, Rt, tr3);
}

template <int M>
__global__ void __launch_bounds__(32) k_ghost(StepArgs a)
{
    ghost_warp<M>(a, blockIdx.x);
}

template <int M>
void launch_ghost(const StepArgs &a)
{
    const int nb = (ghost_count(a) + ghost_groups<M>() - 1) / ghost_groups<M>();
    k_ghost<M><<<nb, 32, 0, a.stream>>>(a);
}

// ---------------------------------------------------------------------
// Production rates rho_dot_a (Eq. (sumRhoDot)) of the mass-action
// mechanism.  With E_a = exp(g_a/(R_U T))
// and act_a = c_a E_a, the rate of progress of a reaction is
//   q = k_f / prod_reac E * (prod_reac act - (P0/(r T))^(-dn) prod_prod act),
// which equals k_f prod_reac c - (k_f / K_c) prod_prod c.
// ---------------------------------------------------------------------

// 2^(j/256), j = 0..255, each the double nearest to the exact value
// (60-digit evaluation of 2^(j/256), rounded once).
__device__ const double c_exp2_256[256] = {
    0x1.0000000000000p+0, 0x1.00b1afa5abcbfp+0, 0x1.0163da9fb3335p+0, 0x1.02168143b0281p+0,
    0x1.02c9a3e778061p+0, 0x1.037d42e11bbccp+0, 0x1.04315e86e7f85p+0, 0x1.04e5f72f654b1p+0,
    0x1.059b0d3158574p+0, 0x1.0650a0e3c1f89p+0, 0x1.0706b29ddf6dep+0, 0x1.07bd42b72a836p+0,
    0x1.0874518759bc8p+0, 0x1.092bdf66607e0p+0, 0x1.09e3ecac6f383p+0, 0x1.0a9c79b1f3919p+0,
    0x1.0b5586cf9890fp+0, 0x1.0c0f145e46c85p+0, 0x1.0cc922b7247f7p+0, 0x1.0d83b23395decp+0,
    0x1.0e3ec32d3d1a2p+0, 0x1.0efa55fdfa9c5p+0, 0x1.0fb66affed31bp+0, 0x1.1073028d7233ep+0,
    0x1.11301d0125b51p+0, 0x1.11edbab5e2ab6p+0, 0x1.12abdc06c31ccp+0, 0x1.136a814f204abp+0,
    0x1.1429aaea92de0p+0, 0x1.14e95934f312ep+0, 0x1.15a98c8a58e51p+0, 0x1.166a45471c3c2p+0,
    0x1.172b83c7d517bp+0, 0x1.17ed48695bbc0p+0, 0x1.18af9388c8deap+0, 0x1.1972658375d2fp+0,
    0x1.1a35beb6fcb75p+0, 0x1.1af99f8138a1cp+0, 0x1.1bbe084045cd4p+0, 0x1.1c82f95281c6bp+0,
    0x1.1d4873168b9aap+0, 0x1.1e0e75eb44027p+0, 0x1.1ed5022fcd91dp+0, 0x1.1f9c18438ce4dp+0,
    0x1.2063b88628cd6p+0, 0x1.212be3578a819p+0, 0x1.21f49917ddc96p+0, 0x1.22bdda27912d1p+0,
    0x1.2387a6e756238p+0, 0x1.2451ffb82140ap+0, 0x1.251ce4fb2a63fp+0, 0x1.25e85711ece75p+0,
    0x1.26b4565e27cddp+0, 0x1.2780e341ddf29p+0, 0x1.284dfe1f56381p+0, 0x1.291ba7591bb70p+0,
    0x1.29e9df51fdee1p+0, 0x1.2ab8a66d10f13p+0, 0x1.2b87fd0dad990p+0, 0x1.2c57e39771b2fp+0,
    0x1.2d285a6e4030bp+0, 0x1.2df961f641589p+0, 0x1.2ecafa93e2f56p+0, 0x1.2f9d24abd886bp+0,
    0x1.306fe0a31b715p+0, 0x1.31432edeeb2fdp+0, 0x1.32170fc4cd831p+0, 0x1.32eb83ba8ea32p+0,
    0x1.33c08b26416ffp+0, 0x1.3496266e3fa2dp+0, 0x1.356c55f929ff1p+0, 0x1.36431a2de883bp+0,
    0x1.371a7373aa9cbp+0, 0x1.37f26231e754ap+0, 0x1.38cae6d05d866p+0, 0x1.39a401b7140efp+0,
    0x1.3a7db34e59ff7p+0, 0x1.3b57fbfec6cf4p+0, 0x1.3c32dc313a8e5p+0, 0x1.3d0e544ede173p+0,
    0x1.3dea64c123422p+0, 0x1.3ec70df1c5175p+0, 0x1.3fa4504ac801cp+0, 0x1.40822c367a024p+0,
    0x1.4160a21f72e2ap+0, 0x1.423fb2709468ap+0, 0x1.431f5d950a897p+0, 0x1.43ffa3f84b9d4p+0,
    0x1.44e086061892dp+0, 0x1.45c2042a7d232p+0, 0x1.46a41ed1d0057p+0, 0x1.4786d668b3237p+0,
    0x1.486a2b5c13cd0p+0, 0x1.494e1e192aed2p+0, 0x1.4a32af0d7d3dep+0, 0x1.4b17dea6db7d7p+0,
    0x1.4bfdad5362a27p+0, 0x1.4ce41b817c114p+0, 0x1.4dcb299fddd0dp+0, 0x1.4eb2d81d8abffp+0,
    0x1.4f9b2769d2ca7p+0, 0x1.508417f4531eep+0, 0x1.516daa2cf6642p+0, 0x1.5257de83f4eefp+0,
    0x1.5342b569d4f82p+0, 0x1.542e2f4f6ad27p+0, 0x1.551a4ca5d920fp+0, 0x1.56070dde910d2p+0,
    0x1.56f4736b527dap+0, 0x1.57e27dbe2c4cfp+0, 0x1.58d12d497c7fdp+0, 0x1.59c0827ff07ccp+0,
    0x1.5ab07dd485429p+0, 0x1.5ba11fba87a03p+0, 0x1.5c9268a5946b7p+0, 0x1.5d84590998b93p+0,
    0x1.5e76f15ad2148p+0, 0x1.5f6a320dceb71p+0, 0x1.605e1b976dc09p+0, 0x1.6152ae6cdf6f4p+0,
    0x1.6247eb03a5585p+0, 0x1.633dd1d1929fdp+0, 0x1.6434634ccc320p+0, 0x1.652b9febc8fb7p+0,
    0x1.6623882552225p+0, 0x1.671c1c70833f6p+0, 0x1.68155d44ca973p+0, 0x1.690f4b19e9538p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6b052fa75173ep+0, 0x1.6c012750bdabfp+0, 0x1.6cfdcddd47645p+0,
    0x1.6dfb23c651a2fp+0, 0x1.6ef9298593ae5p+0, 0x1.6ff7df9519484p+0, 0x1.70f7466f42e87p+0,
    0x1.71f75e8ec5f74p+0, 0x1.72f8286ead08ap+0, 0x1.73f9a48a58174p+0, 0x1.74fbd35d7cbfdp+0,
    0x1.75feb564267c9p+0, 0x1.77024b1ab6e09p+0, 0x1.780694fde5d3fp+0, 0x1.790b938ac1cf6p+0,
    0x1.7a11473eb0187p+0, 0x1.7b17b0976cfdbp+0, 0x1.7c1ed0130c132p+0, 0x1.7d26a62ff86f0p+0,
    0x1.7e2f336cf4e62p+0, 0x1.7f3878491c491p+0, 0x1.80427543e1a12p+0, 0x1.814d2add106d9p+0,
    0x1.82589994cce13p+0, 0x1.8364c1eb941f7p+0, 0x1.8471a4623c7adp+0, 0x1.857f4179f5b21p+0,
    0x1.868d99b4492edp+0, 0x1.879cad931a436p+0, 0x1.88ac7d98a6699p+0, 0x1.89bd0a478580fp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8be05bad61778p+0, 0x1.8cf3216b5448cp+0, 0x1.8e06a5e0866d9p+0,
    0x1.8f1ae99157736p+0, 0x1.902fed0282c8ap+0, 0x1.9145b0b91ffc6p+0, 0x1.925c353aa2fe2p+0,
    0x1.93737b0cdc5e5p+0, 0x1.948b82b5f98e5p+0, 0x1.95a44cbc8520fp+0, 0x1.96bdd9a7670b3p+0,
    0x1.97d829fde4e50p+0, 0x1.98f33e47a22a2p+0, 0x1.9a0f170ca07bap+0, 0x1.9b2bb4d53fe0dp+0,
    0x1.9c49182a3f090p+0, 0x1.9d674194bb8d5p+0, 0x1.9e86319e32323p+0, 0x1.9fa5e8d07f29ep+0,
    0x1.a0c667b5de565p+0, 0x1.a1e7aed8eb8bbp+0, 0x1.a309bec4a2d33p+0, 0x1.a42c980460ad8p+0,
    0x1.a5503b23e255dp+0, 0x1.a674a8af46052p+0, 0x1.a799e1330b358p+0, 0x1.a8bfe53c12e59p+0,
    0x1.a9e6b5579fdbfp+0, 0x1.ab0e521356ebap+0, 0x1.ac36bbfd3f37ap+0, 0x1.ad5ff3a3c2774p+0,
    0x1.ae89f995ad3adp+0, 0x1.afb4ce622f2ffp+0, 0x1.b0e07298db666p+0, 0x1.b20ce6c9a8952p+0,
    0x1.b33a2b84f15fbp+0, 0x1.b468415b749b1p+0, 0x1.b59728de5593ap+0, 0x1.b6c6e29f1c52ap+0,
    0x1.b7f76f2fb5e47p+0, 0x1.b928cf22749e4p+0, 0x1.ba5b030a1064ap+0, 0x1.bb8e0b79a6f1fp+0,
    0x1.bcc1e904bc1d2p+0, 0x1.bdf69c3f3a207p+0, 0x1.bf2c25bd71e09p+0, 0x1.c06286141b33dp+0,
    0x1.c199bdd85529cp+0, 0x1.c2d1cd9fa652cp+0, 0x1.c40ab5fffd07ap+0, 0x1.c544778fafb22p+0,
    0x1.c67f12e57d14bp+0, 0x1.c7ba88988c933p+0, 0x1.c8f6d9406e7b5p+0, 0x1.ca3405751c4dbp+0,
    0x1.cb720dcef9069p+0, 0x1.ccb0f2e6d1675p+0, 0x1.cdf0b555dc3fap+0, 0x1.cf3155b5bab74p+0,
    0x1.d072d4a07897cp+0, 0x1.d1b532b08c968p+0, 0x1.d2f87080d89f2p+0, 0x1.d43c8eacaa1d6p+0,
    0x1.d5818dcfba487p+0, 0x1.d6c76e862e6d3p+0, 0x1.d80e316c98398p+0, 0x1.d955d71ff6075p+0,
    0x1.da9e603db3285p+0, 0x1.dbe7cd63a8315p+0, 0x1.dd321f301b460p+0, 0x1.de7d5641c0658p+0,
    0x1.dfc97337b9b5fp+0, 0x1.e11676b197d17p+0, 0x1.e264614f5a129p+0, 0x1.e3b333b16ee12p+0,
    0x1.e502ee78b3ff6p+0, 0x1.e653924676d76p+0, 0x1.e7a51fbc74c83p+0, 0x1.e8f7977cdb740p+0,
    0x1.ea4afa2a490dap+0, 0x1.eb9f4867cca6ep+0, 0x1.ecf482d8e67f1p+0, 0x1.ee4aaa2188510p+0,
    0x1.efa1bee615a27p+0, 0x1.f0f9c1cb6412ap+0, 0x1.f252b376bba97p+0, 0x1.f3ac948dd7274p+0,
    0x1.f50765b6e4540p+0, 0x1.f6632798844f8p+0, 0x1.f7bfdad9cbe14p+0, 0x1.f91d802243c89p+0,
    0x1.fa7c1819e90d8p+0, 0x1.fbdba3692d514p+0, 0x1.fd3c22b8f71f1p+0, 0x1.fe9d96b2a23d9p+0,
};

// e^(x - N ln2/256) 2^(N/256) for x in units of 2^-70, modulo 2^64, and N = n
// (see exp_table; ln2/256 as L1 2^-70 + L2 2^-88).
__device__ __forceinline__ double exp_reduced(unsigned long long xs, int n, long long L1, long long L2)
{
    typedef long long i64;
    typedef unsigned long long u64;
    const i64 r = (i64)(xs - (u64)(i64)n * (u64)L1 - (u64)(((i64)n * L2) >> 18));
    const int rh = opaque((int)(r >> 32)), rl = opaque((int)((unsigned)r >> 1));
    const i64 r2 = (i64)rh * rh + (((i64)rh * rl) >> 30);                   // units of 2^-76
    const int t = opaque((int)(2147483648.0 / 6) + (int)(((i64)rh * (int)(2147483648.0 / 24)) >> 38) +
                         (int)(((i64)opaque((int)(r2 >> 32)) * (int)(2147483648.0 / 120)) >> 44));
    const int rt = opaque((int)(((i64)rh * t) >> 27));                      // r t, units of 2^-42
    // e^r - 1, units of 2^-70
    const i64 p = r + (r2 >> 7) + (((i64)opaque((int)(r2 >> 27)) * rt) >> 21);
    const u64 tb = (u64)__double_as_longlong(__ldg(&c_exp2_256[n & 255]));
    const u64 tm = (tb & 0xfffffffffffffull) | 0x10000000000000ull;         // 2^(j/256), units of 2^-52
    const int th = opaque((int)(tm >> 22)), tl = opaque((int)(tm & 0x3fffffull));
    const int ph = opaque((int)(p >> 32)), pl = opaque((int)((unsigned)p >> 1));
    const i64 tp = (i64)th * ph + (((i64)th * pl) >> 31) + (((i64)tl * ph) >> 22);
    u64 y = (tm << 10) + (u64)(tp >> 6);                                    // units of 2^-62
    const int lead = (int)(y >> 62), d = (lead >= 2) - (lead == 0);         // y in [1/2, 4): one place up or down
    y >>= 9 + d;
    return __longlong_as_double((i64)(((u64)(unsigned)(1022 + (n >> 8) + d) << 52) + (y >> 1) + (y & 1)));
}

// exp(x) by the table-driven method of P. T. P. Tang (ACM Trans. Math.
// Softw. 15(2), 1989): x = (256 m + j) ln2/256 + r with |r| <= 1.04 ln2/512,
// so exp(x) = 2^m 2^(j/256) e^r, and e^r - 1 is its degree-5 Taylor
// polynomial.  ln2/256 = L1 + L2 with L1 rounded to 35 significant bits.
//
// Everything runs on the integer and float pipes, in fixed point: the FP64
// pipe, which bounds the kernels that call this, takes 76 cycles of a
// scheduler per warp instruction, an integer instruction 1 to 4.
//   N = 256 m + j from the float x 256/ln2, rounded (off by at most 0.02);
//   r = x - N (L1 + L2) in units of 2^-70, exact modulo 2^64 up to the last
//   unit (|r| < 2^61: what the products lose above 64 bits cancels);
//   e^r - 1 = r + r^2/2 + r^2 (r t), t = 1/6 + r/24 + r^2/120, r^2 to 2^-76,
//   the rest in 32-bit factors (errors below 2^-60);
//   2^(j/256) (e^r - 1) to 2^-68, added and rounded once.
// |x| >= 707 (where 2^m would leave the normal range) and NaN go to exp().
// Largest error 1.02 ulp, mean 0.338 (4 million arguments in +-60 against
// 64-bit-mantissa expl; with a degree-4 polynomial in double: 1.32, 0.343).
// 9 double operations before, about 80 others now; 128^3 nodes, nine
// species, the double collision with the rates in it: 15.4 -> 14.3 ms.
__device__ __forceinline__ double exp_table(double x)
{
    constexpr double kInv = 0x1.71547652b82fep+8, kL1 = 0x1.62e42fefc0000p-9, kL2 = -0x1.c610ca86c3899p-45;
    constexpr long long L1 = (long long)(kL1 * 0x1p+70), L2 = (long long)(kL2 * 0x1p+88);
    typedef unsigned long long u64;
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x), mag = (unsigned)hi & 0x7fffffffu;
    if (mag >= 0x40861800u) return exp(x);                                  // |x| >= 707, inf, NaN
    const int ed = (int)(mag >> 20);
    // x truncated to float (0 below 2^-126), and N
    const unsigned fb = ((unsigned)hi & 0x80000000u) | ((mag - (896u << 20)) << 3) | (lo >> 29);
    const float fx = ed <= 896 ? 0.0f : __uint_as_float(fb);
    const int n = __float_as_int(fmaf(fx, (float)kInv, 12582912.0f)) - 0x4b400000;
    // x in units of 2^-70, modulo 2^64
    const u64 m = ((u64)((mag & 0xfffffu) | 0x100000u) << 32) | lo;
    const int sh = ed - 1005;
    const u64 xm = sh >= 0 ? m << sh : m >> (sh < -63 ? 63 : -sh);
    return exp_reduced(hi < 0 ? 0ull - xm : xm, n, L1, L2);
}

// Exponential of the rate expressions: exp_table(), except in the fast mixed
// unit, where the rates are stored in float: a base-2 range reduction
// done exactly in double (t = x log2(e) = k + f, k integer, |f| <= 1/2, in
// the manner of Cody and Waite), 2^f from the hardware base-2 exponential
// in float (ex2.approx, relative error about 2^-22), and 2^k added to the
// binary exponent of the result; relative error below 5e-7.
__device__ __forceinline__ double exp_rate(double x)
{
#if LBMK_MIXED && LBMK_FAST
    const double t = x * 1.4426950408889634074;          // log2(e)
    if (!(fabs(t) < 1020.0)) return t > 0.0 ? (double)INFINITY : (t < 0.0 ? 0.0 : t);
    const double k = rint(t);
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((float)(t - k)));
    const double r = (double)y;                          // in [2^-1/2, 2^1/2]
    return __hiloint2double(__double2hiint(r) + (int)k * (1 << 20), __double2loint(r));
#else
    return exp_table(x);
#endif
}

// exp(x) for x in units of 2^-53 (modulo 2^64) and a float within 1e-4 of it.
// Beyond +-707 exp() itself, of x as far as the unit holds it (e^x is 0 or
// infinite beyond).
__device__ __forceinline__ double exp_fixed(long long x, float xf)
{
    constexpr double kInv = 0x1.71547652b82fep+8, kL1 = 0x1.62e42fefc0000p-9, kL2 = -0x1.c610ca86c3899p-45;
    constexpr long long L1 = (long long)(kL1 * 0x1p+70), L2 = (long long)(kL2 * 0x1p+88);
    if (!(fabsf(xf) < 707.0f)) return exp(fabsf(xf) < 1000.0f ? (double)x * 0x1p-53 : (double)xf);
    const int n = __float_as_int(fmaf(xf, (float)kInv, 12582912.0f)) - 0x4b400000;
    return exp_reduced((unsigned long long)x << 17, n, L1, L2);
}

// v 2^sh modulo 2^64 (sh within +-63; smaller gives the sign).
__device__ __forceinline__ long long shift_by(long long v, int sh)
{
    return sh >= 0 ? (long long)((unsigned long long)v << (sh & 63)) : v >> (sh < -63 ? 63 : -sh);
}

// Molar production rates as molar_production below forms them, with every
// exponent an integer sum in units of 2^-53: the Gibbs functions
//   g_a/(R_U T) = sum_j gco_aj phi_j,  phi = 1 - ln T, T .. T^4, 1/T, 1,
// and ln k_f - sum_reac g, from products of 58-bit limbs (each phi_j with
// its leading bit at 2^57, the coefficients of a j relative to the largest)
// brought to that unit, and a float beside each exponent for exp_fixed's
// range reduction.  A sum of these is good to a few units of 2^-52; in
// double it carried half a unit of the largest partial sum, 2^-47 at the
// exponents of 300 K.  146 FP64 operations per node of nine species and 21
// reactions leave the FP64 pipe, and 80 more where the rates are summed in
// pairs of floats (RateSums).  For tables in range (MechConst::chem_fixed).
template <int M, bool PAIR>
__device__ __forceinline__ void molar_production_fixed(const MechConst &mc, double T, const double *conc,
                                                       double *sh_act, double *sh_g, RateSums<PAIR> w, int t,
                                                       int stride)
{
    typedef long long i64;
    const double invT = 1.0 / T, lnT = log(T), lnTr = lnT - mc.log_T_ref;
    Limbs58 P[6], Ll, Il;
    int sp[6], sb, st;
    float pf[6];
    {
        const double T2 = T * T;
        const double phi[6] = {1.0 - lnT, T, T2, T2 * T, T2 * T2, invT};
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int e = biased_exponent(phi[j]);
            P[j] = to_limbs58(phi[j], e);
            sp[j] = mc.gx_exp[j] + e - 969;
            pf[j] = d2f(phi[j]);
        }
        const int eL = biased_exponent(lnTr), eI = biased_exponent(invT);
        Ll = to_limbs58(lnTr, eL);
        Il = P[5];
        sb = mc.bx_exp + eL - 969;
        st = mc.tx_exp + eI - 969;
    }
    const float lf = d2f(lnTr);
    i64 *gx = reinterpret_cast<i64 *>(sh_g);
#pragma unroll 1
    for (int s = 0; s < M; ++s) {
        i64 g = mc.gx0[s];
        float gf = mc.gxf[s][6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (!(mc.gx_mask >> j & 1)) continue;          // no species has the term
            i64 hi = 0, mid = 0;
            fma_limbs58(hi, mid, limbs_of(mc.gx[s][j]), P[j]);
            g += shift_by(hi + (mid >> 29), sp[j]);
            gf = fmaf(mc.gxf[s][j], pf[j], gf);
        }
        // beyond the range of the unit: e^g is 0 or infinite either way
        if (!(fabsf(gf) < 1000.0f)) g = gf < 0.0f ? -(1000ll << 53) : 1000ll << 53;
        gx[s * stride + t] = g;
        sh_act[s * stride + t] = conc[s] * exp_fixed(g, gf);
        w.clear(s);
    }
    const double c0 = mc.P0_over_r * invT, ic0 = T * mc.r_over_P0;   // P0/(r T) and its inverse
#pragma unroll 1
    for (int k = 0; k < mc.R; ++k) {
        const int nr = mc.nreac[k], np = mc.nprod[k];     // nr >= 1 (checked at packing)
        // exponent ln k_f - sum_reac g
        const RateLimbs &rx = mc.rx[k];
        i64 bh = 0, bm = 0, th = 0, tm = 0;
        fma_limbs58(bh, bm, limbs_of(rx.b), Ll);
        fma_limbs58(th, tm, limbs_of(rx.theta), Il);
        i64 arg = rx.log_A + shift_by(bh + (bm >> 29), sb) - shift_by(th + (tm >> 29), st);
        float af = fmaf(rx.bf, lf, fmaf(-rx.thetaf, pf[5], rx.log_Af));
        double p = 1.0;
        for (int j = 0; j < nr; ++j) {
            const int sidx = mc.reac[k][j] * stride + t;
            const i64 g = gx[sidx];
            arg -= g;
            af -= (float)(int)(g >> 32) * 0x1p-21f;
            p = j == 0 ? sh_act[sidx] : p * sh_act[sidx];
        }
        if (mc.rev[k]) {
            double pr = np > 0 ? sh_act[mc.prod[k][0] * stride + t] : 1.0;
            for (int j = 1; j < np; ++j) pr *= sh_act[mc.prod[k][j] * stride + t];
            const int dn = mc.dn[k];
            for (int j = 0; j < dn; ++j) pr *= ic0;
            for (int j = 0; j < -dn; ++j) pr *= c0;
            p -= pr;
        }
        double q = p * exp_fixed(arg, af);
        const int type = mc.rtype[k];
        if (type != 0) {
            double cM = 0.0;
#pragma unroll
            for (int s = 0; s < M; ++s) cM = fma(mc.eff[k][s], conc[s], cM);
            if (type == 1) {
                q *= cM;
            } else {
                const double Pr = exp_table(fma(mc.dlow[k][1], lnTr, fma(-mc.dlow[k][2], invT, mc.dlow[k][0]))) * cM;
                q *= Pr / (1.0 + Pr);
            }
        }
        const typename RateSums<PAIR>::Term qt = w.term(q);
        for (int j = 0; j < nr; ++j) w.template add<-1>(mc.reac[k][j], qt);
        for (int j = 0; j < np; ++j) w.template add<1>(mc.prod[k][j], qt);
    }
}

// Molar production rates sum_k (nu''_ak - nu'_ak) q_k at temperature T and
// concentrations conc, left in sh_w[a * stride + t]; sh_act and sh_g are
// this thread's scratch columns (stride: the block's thread count).
template <int M>
__device__ __forceinline__ void molar_production(const MechConst &mc, double T, const double *conc, double *sh_act,
                                                 double *sh_g, WReal *sh_w, int t, int stride)
{
    const double invT = 1.0 / T, lnT = log(T);
    const double lnTr = lnT - mc.log_T_ref;
    const double om_lnT = 1.0 - lnT;
#pragma unroll
    for (int s = 0; s < M; ++s) {
        const double *gc = mc.gco[s];
        const double g = fma(gc[0], om_lnT,
                             fma(fma(fma(fma(gc[4], T, gc[3]), T, gc[2]), T, gc[1]), T, fma(gc[5], invT, gc[6])));
        sh_g[s * stride + t] = g;
        sh_act[s * stride + t] = conc[s] * exp_rate(g);
        sh_w[s * stride + t] = 0;
    }
    const double c0 = mc.P0_over_r * invT, ic0 = T / mc.P0_over_r;   // P0/(r T) and its inverse
    for (int k = 0; k < mc.R; ++k) {
        const int nr = mc.nreac[k], np = mc.nprod[k];     // nr >= 1 (checked at packing)
        const int s0 = mc.reac[k][0] * stride + t;
        double arg = fma(mc.b[k], lnTr, fma(-mc.theta[k], invT, mc.log_A[k])) - sh_g[s0];
        double pf = sh_act[s0];
        for (int j = 1; j < nr; ++j) {
            const int sidx = mc.reac[k][j] * stride + t;
            arg -= sh_g[sidx];
            pf *= sh_act[sidx];
        }
        double q = pf;
        if (mc.rev[k]) {
            double pr = np > 0 ? sh_act[mc.prod[k][0] * stride + t] : 1.0;
            for (int j = 1; j < np; ++j) pr *= sh_act[mc.prod[k][j] * stride + t];
            const int dn = mc.dn[k];
            for (int j = 0; j < dn; ++j) pr *= ic0;
            for (int j = 0; j < -dn; ++j) pr *= c0;
            q -= pr;
        }
        q *= exp_rate(arg);
        const int type = mc.rtype[k];
        if (type != 0) {
            double cM = 0.0;
#pragma unroll
            for (int s = 0; s < M; ++s) cM = fma(mc.eff[k][s], conc[s], cM);
            if (type == 1) {
                q *= cM;
            } else {
                const double Pr = exp_rate(fma(mc.dlow[k][1], lnTr, fma(-mc.dlow[k][2], invT, mc.dlow[k][0]))) * cM;
                q *= Pr / (1.0 + Pr);
            }
        }
        const WReal qr = cvt<WReal>(q);
        for (int j = 0; j < nr; ++j) sh_w[mc.reac[k][j] * stride + t] -= qr;
        for (int j = 0; j < np; ++j) sh_w[mc.prod[k][j] * stride + t] += qr;
    }
}

// The rates in sh_w by either form (the fast mixed unit's reported rates keep
// the hardware exponential; its step takes the integer one, which is both
// more accurate and faster: k_chem, 160^3, 2.4 ms against 5.4).
template <int M>
__device__ __forceinline__ void production_rates(const MechConst &mc, double T, const double *conc, double *sh_act,
                                                 double *sh_g, WReal *sh_w, int t, int stride)
{
#if !LBMK_FAST
    if (mc.chem_fixed) {
        molar_production_fixed<M, false>(mc, T, conc, sh_act, sh_g, RateSums<false>{sh_w + t, stride, 0}, t, stride);
        return;
    }
#endif
    molar_production<M>(mc, T, conc, sh_act, sh_g, sh_w, t, stride);
}

// The temperature of a node from its pulled populations, with the moments in
// sm and the densities rho_a in M columns of shared memory (this thread's,
// stride bs); eu: the coefficients of the mixture energy, when asked for.
template <int M>
__device__ __forceinline__ double node_temperature(const MechConst &mc, const StepArgs &a, const PullIdx &p, int n,
                                                   Sums &sm, double *sh_ra, int bs, double *eu_out = nullptr)
{
    double ir = 0.0, eu[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) eu[k] = 0.0;
    pull_moments<M, false>(mc, a, p, n, sm, [&](int s, double ra, const Real *) {
        if (s == 0) ir = 1.0 / sm.rho;
        const double Y = ra * ir;
#pragma unroll
        for (int k = 0; k < 6; ++k) eu[k] = fma(Y, mc.uco[s][k], eu[k]);
        sh_ra[s * bs] = ra;
    });
    const double u[3] = {sm.j[0] * ir, sm.j[1] * ir, sm.j[2] * ir};
    const double usq = dot3(u, u);
    if (eu_out)
#pragma unroll
        for (int k = 0; k < 6; ++k) eu_out[k] = eu[k];
    return solve_T(eu, fma(sm.rhoE, ir, -0.5 * usq), a.macro[(size_t)DR_T * a.N + n], a.status);
}

// ---------------------------------------------------------------------
// Moments for lbm_moments: the fields of the state in src (no record).
// ---------------------------------------------------------------------
template <int M>
__global__ void __launch_bounds__(LBMK_BLOCK, LBMK_MOM_MINB) k_moments(StepArgs a, unsigned mask, double *out)
{
    __shared__ double sh_act[M * LBMK_BLOCK];
    __shared__ double sh_g[M * LBMK_BLOCK];
    __shared__ WReal sh_w[M * LBMK_BLOCK];
    const MechConst &mc = c_mech[a.slot];
    Node nd;
    if (!node_of(nd, a)) return;
    PullIdx p;
    make_pull(p, nd, a);
    const int n = nd.n;
    const size_t N = a.N;
    // rows of out: the fields of the mask in bit order
    size_t row = 0;
    auto rows = [&](unsigned bit, int count) {
        const size_t r = row;
        if (mask & bit) row += count;
        return out + r * N + n;
    };
    double *o_ra = rows(1u, M), *o_j = rows(2u, 3), *o_E = rows(4u, 1), *o_T = rows(8u, 1), *o_P = rows(16u, 1),
           *o_Y = rows(32u, M), *o_ja = rows(64u, 3 * M);
    Sums sm = {};
    double ir = 0.0, inv_m = 0.0, eu[6], jM[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 6; ++k) eu[k] = 0.0;
    pull_moments<M, false>(mc, a, p, n, sm, [&](int s, double ra, const Real *j) {
        if (s == 0) {
            ir = 1.0 / sm.rho;
#pragma unroll
            for (int d = 0; d < 3; ++d) jM[d] = sm.j[d];
        }
        const double Y = ra * ir;
        inv_m = fma(Y, mc.invW[s], inv_m);
#pragma unroll
        for (int k = 0; k < 6; ++k) eu[k] = fma(Y, mc.uco[s][k], eu[k]);
        sh_act[s * LBMK_BLOCK + threadIdx.x] = ra;
        if (mask & 1u) o_ra[(size_t)s * N] = ra;
        if (mask & 32u) o_Y[(size_t)s * N] = Y;
        if (mask & 64u)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double jd = s < M - 1 ? cvt<double>(j[d]) : jM[d];
                o_ja[(size_t)(3 * s + d) * N] = jd;
                jM[d] -= jd;
            }
    });
    const double rho = sm.rho;
    const double u[3] = {sm.j[0] * ir, sm.j[1] * ir, sm.j[2] * ir};
    const double usq = dot3(u, u);
    const double T = solve_T(eu, fma(sm.rhoE, ir, -0.5 * usq), a.macro[DR_T * N + n], a.status);
    const double Rm = mc.r_lat * inv_m;
    if (mask & 2u)
#pragma unroll
        for (int d = 0; d < 3; ++d) o_j[(size_t)d * N] = sm.j[d];
    if (mask & 4u) *o_E = sm.rhoE;
    if (mask & 8u) *o_T = T;
    if (mask & 16u) *o_P = rho * Rm * T;
    if (mask & (128u | 256u)) {
        double conc[M];
#pragma unroll
        for (int s = 0; s < M; ++s) conc[s] = sh_act[s * LBMK_BLOCK + threadIdx.x] * mc.invW[s];
        production_rates<M>(mc, T, conc, sh_act, sh_g, sh_w, threadIdx.x, LBMK_BLOCK);
        if (mask & 128u) {
            for (int s = 0; s < M; ++s) out[(row + s) * N + n] = mc.W[s] * (double)sh_w[s * LBMK_BLOCK + threadIdx.x];
            row += M;
        }
        if (mask & 256u) {      // heat release rate, -sum_a H_a rho_dot_a
            double h = 0.0;
            for (int s = 0; s < M; ++s)
                h = fma(-H_spec(mc, s, T), mc.W[s] * (double)sh_w[s * LBMK_BLOCK + threadIdx.x], h);
            out[row * N + n] = h;
        }
    }
}

#if LBMK_MIXED && !LBMK_FAST
}  // namespace
#include "lbm_diffusion.cuh"
namespace {
#endif

// ---------------------------------------------------------------------
// Pass 1: pull, moments, temperature, relaxation, energy equilibrium
// moments; writes the per-node record but for the diffusion velocities
// (momenta j_a in their place), beta_a and the part of Dq that needs them.
//
// The loops over the species are not unrolled: fully unrolled, this pass
// and the solve of pass 1b were 19,500 instructions run once per
// warp, more than the instruction caches hold, and a quarter of every
// warp's time went to fetching them.
// sh: this thread's shared memory, pre_cols<M>() columns of bs doubles
// (rho_a, then Y_a).
// ---------------------------------------------------------------------
template <int M>
constexpr int pre_cols() { return 2 * M; }

template <int M>
__device__ __forceinline__ void pre_node(const StepArgs &a, const Node &nd, double *sh, int bs)
{
    const MechConst &mc = c_mech[a.slot];
    const int n = nd.n;
    const size_t N = a.N;
    const RecRows rr = rec_rows(M);
    Real *R = rec(a);
    PullIdx p;
    make_pull(p, nd, a);
#if LBMK_MIXED
    double *dr = static_cast<double *>(a.dst) + n;          // DiffRows
#endif
    Sums sm = {};
    double ir = 0.0, inv_m = 0.0, eu[6];
    bool neg = false;
#pragma unroll
    for (int k = 0; k < 6; ++k) eu[k] = 0.0;
    pull_moments<M, true>(mc, a, p, n, sm, [&](int s, double ra, const Real *j) {
        if (s == 0) ir = 1.0 / sm.rho;
        Real *J = R + (size_t)(rr.du + 3 * s) * N + n;
        J[0] = j[0];
        J[N] = j[1];
        J[2 * N] = j[2];
        const double Y = ra * ir;
        inv_m = fma(Y, mc.invW[s], inv_m);
        if (__double2hiint(ra) < 0)             // sign bit first: the compare only for negative values
            neg |= ra < -1e-10 * sm.rho;        // below rounding noise of trace species
#pragma unroll
        for (int k = 0; k < 6; ++k) eu[k] = fma(Y, mc.uco[s][k], eu[k]);
        sh[s * bs] = ra;
        sh[(M + s) * bs] = Y;
        R[(size_t)(rr.y + s) * N + n] = cvt<Real>(Y);
#if LBMK_MIXED
        dr[(size_t)(diff_rows(M).ra + s) * N] = ra;
#else
        R[(size_t)(rr.wd + s) * N + n] = ra;
#endif
    });
    const double rho = sm.rho, rhoE = sm.rhoE;
    const double u[3] = {sm.j[0] * ir, sm.j[1] * ir, sm.j[2] * ir};
    const double usq = dot3(u, u);
    if (!(rho > 0.0) || !isfinite(rhoE)) flag(a.status, LBMK_BIT_NONFINITE);
    if (neg) flag(a.status, LBMK_BIT_NEGATIVE);

    // temperature, Eq. (temperature)
    const double T = solve_T(eu, fma(rhoE, ir, -0.5 * usq), a.macro[DR_T * N + n], a.status);
    const double Rm = mc.r_lat * inv_m;
    const double P = rho * Rm * T;
    // enthalpies, Eq. (specHa); rest-direction equilibria of the species and
    // mixture sets (Eqs. (feq), (feqmix))
    double H = 0.0;
#if LBMK_MIXED
    const double c2[3] = {fma(-u[0], u[0], 1.0), fma(-u[1], u[1], 1.0), fma(-u[2], u[2], 1.0)};
#endif
#pragma unroll 1
    for (int s = 0; s < M; ++s) {
        const double Ha = H_spec(mc, s, T);
        H = fma(sh[(M + s) * bs], Ha, H);
        R[(size_t)(rr.h + s) * N + n] = cvt<Real>(Ha);
#if LBMK_MIXED
        const double z = __dmul_rn(s < M - 1 ? mc.Ra[s] : Rm, T);
        const double r = s < M - 1 ? sh[s * bs] : rho;
        a.macro[(size_t)(DR_FEQ0 + s) * N + n] = r * (c2[0] - z) * (c2[1] - z) * (c2[2] - z);
#endif
    }
    // relaxation rates (Eqs. (mu), (lambda)) in the storage type: in the
    // mixed units they are stored and used as floats only; dfac scales the
    // binary diffusivities of mixture-averaged transport
    Real nup, nup1;
    double kappa = mc.r_lat * T / inv_m;        // Eq. (tauab): 1/tau_ab = kappa / (W_a W_b D_ab), kappa = m R_U T
    if (mc.transport) {
        double Y[M], dfac;
#pragma unroll
        for (int s = 0; s < M; ++s) Y[s] = sh[(M + s) * bs];
        mixture_transport<M>(mc, Y, inv_m, T, P, dpoly5(eu, T) + Rm, nup, nup1, dfac);
        kappa /= dfac;
    } else {
        nup = cvt<Real>(nu_prime(mc, Rm, T));
        nup1 = nup / cvt<Real>(mc.Pr);
    }
    const Real omega = (Real)1 / ((Real)0.5 + nup);
    const Real omega1 = (Real)1 / ((Real)0.5 + nup1);

    // energy: equilibrium moments and the local part of
    // Dq = (omega - omega_1)(q^* - q^eq) (Eqs. (gstareq1mom), (qdiff)) but
    // for the diffusion velocities, added in k_diff; the grad-Y part
    // (Eq. (corrFourier)) needs the neighbours and is added in k_step_g.
    double qeq[3], Rt[6], tr3;
    energy_moments(rho, u, P, fma(0.5, usq, H), rhoE, qeq, Rt, tr3);
    const double ru[3] = {rho * u[0], rho * u[1], rho * u[2]};
    const double dP[6] = {sm.P[0] - fma(ru[0], u[0], P), sm.P[1] - fma(ru[1], u[1], P), sm.P[2] - fma(ru[2], u[2], P),
                          fma(-ru[0], u[1], sm.P[3]),    fma(-ru[0], u[2], sm.P[4]),    fma(-ru[1], u[2], sm.P[5])};
    const double row0[3] = {dP[0], dP[3], dP[4]}, row1[3] = {dP[3], dP[1], dP[5]}, row2[3] = {dP[4], dP[5], dP[2]};
    const double uP[3] = {dot3(u, row0), dot3(u, row1), dot3(u, row2)};

    // the record: double rows
    a.macro[DR_T * N + n] = T;
    a.macro[(size_t)dr_ge(M) * N + n] = rhoE;
#pragma unroll
    for (int d = 0; d < 3; ++d) a.macro[(size_t)(dr_gq(M) + d) * N + n] = qeq[d];
#pragma unroll
    for (int d = 0; d < 6; ++d) a.macro[(size_t)(dr_gr(M) + d) * N + n] = Rt[d];
    a.macro[(size_t)dr_gtr(M) * N + n] = tr3;
#if LBMK_MIXED
#pragma unroll
    for (int d = 0; d < 3; ++d) dr[(size_t)(diff_rows(M).u + d) * N] = u[d];
    dr[(size_t)diff_rows(M).hk * N] = LBMK_FAST ? ir : 0.5 * kappa * ir;
#endif
    // storage-type rows
    R[(size_t)rr.nup * N + n] = nup;
    // Phi (Eq. (Xalpha)), stored in the storage type and formed in it
    const Real rhoR = cvt<Real>(rho), rtR = cvt<Real>(Rm * T), ph = fma((Real)-3, rtR, (Real)1);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const Real ud = cvt<Real>(u[d]);
        R[(size_t)(rr.phi + d) * N + n] = rhoR * ud * fma(-ud, ud, ph);
        R[(size_t)(rr.u + d) * N + n] = ud;
        // the difference is formed in double (it cancels), the product in the storage type
        R[(size_t)(rr.dq + d) * N + n] = (omega - omega1) * cvt<Real>(sm.q[d] - uP[d] - qeq[d]);
    }
    R[(size_t)rr.rho * N + n] = rhoR;
    R[(size_t)rr.kappa * N + n] = cvt<Real>(kappa);
    R[(size_t)rr.rt * N + n] = rtR;
    R[(size_t)rr.om * N + n] = omega;
    R[(size_t)rr.om1 * N + n] = omega1;
    R[(size_t)rr.p * N + n] = cvt<Real>(P);
}

extern __shared__ double sh_pre[];

// With two or three species the step has two launches fewer: the diffusion
// velocities follow the moments in k_pre, the production rates precede the
// energy collision in k_step_g.  A kernel's launch and tail, 3 to 4 us, is a
// twentieth of such a step on a small lattice, and their code is short enough
// to share a register budget.  Three species, us per step, four kernels / six:
// 1024 nodes mixed 64.3 / 72.4, fast mixed 59.6 / 68.0, double 94.6 / 99.3
// (65.0, 61.9 and 152 before the velocities and the rates became kernels of
// their own); 128^3 mixed 2841 / 2848, fast mixed 2468 / 2501, double 6212 / 6401.
template <int M>
constexpr bool kFewSpecies = M < 4;

template <int M, bool FX>
__device__ __forceinline__ void diff_node(const StepArgs &a, const Node &nd, double *sh, int bs);

template <int M>
__global__ void __launch_bounds__(LBMK_BLOCK, LBMK_PRE_MINB) k_pre(StepArgs a)
{
    Node nd;
    if (!node_of(nd, a)) return;
    pre_node<M>(a, nd, sh_pre + threadIdx.x, blockDim.x);
    if constexpr (kFewSpecies<M>) diff_node<M, false>(a, nd, nullptr, 0);
}

// ---------------------------------------------------------------------
// Pass 1b: Stefan-Maxwell diffusion velocities (Eq. (transform1)), beta_a
// and their part of Dq.
// FX: the tables are in the range of the fixed-point sums (MechConst::
// mix_fixed); sh: this thread's shared memory, diff_cols<M, FX>() columns
// of bs doubles.
// ---------------------------------------------------------------------

// Whether the Stefan-Maxwell solve refines a float factorisation
// (lbm_diffusion.cuh): in the mixed unit, whose velocities are stored as
// floats, from four species on.  (In the fast mixed unit the whole solve is
// in float; with two or three species the LDL^T solve is cheaper.)
template <int M, bool FX>
constexpr bool kRefined = FX && M >= 4 && LBMK_MIXED && !LBMK_FAST;

template <int M, bool FX>
constexpr int diff_cols() { return kRefined<M, FX> ? 5 * M : 0; }

template <int M, bool FX>
__device__ __forceinline__ void diff_node(const StepArgs &a, const Node &nd, double *sh, int bs)
{
    const MechConst &mc = c_mech[a.slot];
    const int n = nd.n;
    const size_t N = a.N;
    const RecRows rr = rec_rows(M);
    Real *R = rec(a);
    auto ld = [&](int row) { return R[(size_t)row * N + n]; };
    Real duR[M][3], itaR[M];
#if LBMK_MIXED
    const double *dr = static_cast<const double *>(a.dst) + n;
#endif
#if LBMK_MIXED && !LBMK_FAST
    if constexpr (kRefined<M, FX>) {
        bool bad = false;
        diffusion_refined<M, true>(mc, dr + (size_t)diff_rows(M).ra * N, dr + (size_t)diff_rows(M).u * N,
                                   R + (size_t)rr.du * N + n, N, dr[(size_t)diff_rows(M).hk * N], sh, bs, duR, itaR,
                                   &bad);
        if (bad) flag(a.status, LBMK_BIT_PIVOT);
    } else
#endif
    {
    // The arithmetic is in SReal: double, or float in the fast mixed unit
    // (the results are stored as floats there, and the solve below is well
    // conditioned: B is diagonally dominant after the symmetric scaling by Y).
    SReal Yr[M], ur[3], irr, kap;
    Real ja[M][3];
    {
#if LBMK_MIXED
        const double *ra = dr + (size_t)diff_rows(M).ra * N;
#pragma unroll
        for (int d = 0; d < 3; ++d) ur[d] = cvt<SReal>(dr[(size_t)(diff_rows(M).u + d) * N]);
#else
        const double *ra = R + (size_t)rr.wd * N + n;
#pragma unroll
        for (int d = 0; d < 3; ++d) ur[d] = ld(rr.u + d);
#endif
#if LBMK_FAST
        irr = cvt<SReal>(dr[(size_t)diff_rows(M).hk * N]);
        kap = ld(rr.kappa);
#pragma unroll
        for (int s = 0; s < M; ++s) Yr[s] = ld(rr.y + s);
        (void)ra;
#else
        double rho = 0.0;
#pragma unroll
        for (int s = 0; s < M; ++s) rho += ra[(size_t)s * N];
        irr = 1.0 / rho;
#if LBMK_MIXED
        kap = 2.0 * dr[(size_t)diff_rows(M).hk * N] * rho;
#else
        kap = ld(rr.kappa);
#endif
#pragma unroll
        for (int s = 0; s < M; ++s) Yr[s] = ra[(size_t)s * N] * irr;
#endif
#pragma unroll
        for (int s = 0; s < M; ++s)
#pragma unroll
            for (int d = 0; d < 3; ++d) ja[s][d] = ld(rr.du + 3 * s + d);
    }
    // 1/tau_a = sum_b Y_b / tau_ab
    SReal ita[M];
#pragma unroll
    for (int s = 0; s < M; ++s) {
        SReal acc = 0;
#pragma unroll
        for (int b = 0; b < M; ++b)
            if (b != s) acc = fma(Yr[b], INVWWD_S(s, b), acc);
        ita[s] = kap * acc;
    }

    // Eq. (transform1), multiplied by Y_a so that the matrix is symmetric:
    //   B_aa = Y_a (1 + 1/(2 tau_a)),  B_ab = -(1/2) Y_a Y_b / tau_ab,
    //   rhs_a = Y_a (u_a - u) = j_a / rho - Y_a u.
    // B is symmetric positive definite; L D L^T without pivoting, L unit
    // lower triangular (stored below the diagonal of Ln).
    SReal du[M][3];
    {
        SReal Ln[M][M], D[M], Dinv[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const SReal hy = (SReal)-0.5 * kap * Yr[i];
#pragma unroll
            for (int k = 0; k < i; ++k) Ln[i][k] = hy * INVWWD_S(i, k) * Yr[k];
            Ln[i][i] = Yr[i] * fma((SReal)0.5, ita[i], (SReal)1);
        }
#pragma unroll
        for (int k = 0; k < M; ++k) {
            SReal tk[M];
#pragma unroll
            for (int j = 0; j < k; ++j) tk[j] = D[j] * Ln[k][j];
#pragma unroll
            for (int i = k; i < M; ++i) {
                SReal sacc = Ln[i][k];
#pragma unroll
                for (int j = 0; j < k; ++j) sacc = fma(-Ln[i][j], tk[j], sacc);
                Ln[i][k] = sacc;
            }
            // D_k = Y_k times the pivot of the unscaled system, which is
            // diagonally dominant: negative where a trace species has dipped
            // to a rounding-level negative density, zero only for an absent
            // species (Y_k = 0), whose row and column vanish and whose
            // diffusion velocity is multiplied by Y_k = 0 wherever it is used.
            // A species so far below the others that 1/D_k would be infinite
            // counts as absent.
            D[k] = Ln[k][k];
            if (!finite_bits(D[k])) flag(a.status, LBMK_BIT_PIVOT);
            Dinv[k] = invertible_bits(D[k]) ? (SReal)1 / D[k] : (SReal)0;
#pragma unroll
            for (int i = k + 1; i < M; ++i) Ln[i][k] *= Dinv[k];
        }
        // L z = rhs, z /= D, L^T x = z
#pragma unroll
        for (int i = 0; i < M; ++i)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                SReal sacc = fma(cvt<SReal>(ja[i][d]), irr, -Yr[i] * ur[d]);
#pragma unroll
                for (int j = 0; j < i; ++j) sacc = fma(-Ln[i][j], du[j][d], sacc);
                du[i][d] = sacc;
            }
#pragma unroll
        for (int i = 0; i < M; ++i)
#pragma unroll
            for (int d = 0; d < 3; ++d) du[i][d] *= Dinv[i];
#pragma unroll
        for (int i = M - 1; i >= 0; --i)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                SReal sacc = du[i][d];
#pragma unroll
                for (int j = i + 1; j < M; ++j) sacc = fma(-Ln[j][i], du[j][d], sacc);
                du[i][d] = sacc;
            }
    }
#pragma unroll
    for (int s = 0; s < M; ++s) {
        itaR[s] = cvt<Real>(ita[s]);
#pragma unroll
        for (int d = 0; d < 3; ++d) duR[s][d] = cvt<Real>(du[s][d]);
    }
    }
    // Dq: + omega_1 rho sum_a H_a Y_a du_a, in the storage type
    Real hyd[3] = {0, 0, 0};
#pragma unroll
    for (int s = 0; s < M; ++s) {
        const Real HY = ld(rr.h + s) * ld(rr.y + s);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            hyd[d] = fma(HY, duR[s][d], hyd[d]);
            R[(size_t)(rr.du + 3 * s + d) * N + n] = duR[s][d];
        }
        // beta_a = 1/(2 tau_a + 1), Eq. (fStar): a parameter of the species
        // collision, formed in the storage type it is used in
        R[(size_t)(rr.beta + s) * N + n] = itaR[s] / ((Real)2 + itaR[s]);
    }
    const Real orho = ld(rr.om1) * ld(rr.rho);
#pragma unroll
    for (int d = 0; d < 3; ++d) R[(size_t)(rr.dq + d) * N + n] = fma(orho, hyd[d], ld(rr.dq + d));
}

template <int M, bool FX>
__global__ void __launch_bounds__(LBMK_BLOCK, LBMK_DIFF_MINB) k_diff(StepArgs a)
{
    Node nd;
    nd.n = blockIdx.x * blockDim.x + threadIdx.x;
    if (nd.n >= a.N) return;
    diff_node<M, FX>(a, nd, sh_pre + threadIdx.x, blockDim.x);
}

// ---------------------------------------------------------------------
// Pass 1c: production rates rho_dot_a of the record's state, in the storage
// type (in double, into the rows that held rho_a for k_diff).  A kernel of
// its own: inside the collision its double operations, a serial chain of 64
// cycles each, ran at the collision's 8 to 12 warps per SM and barely
// overlapped it (256^3 mixed: 25.2 ms in one kernel, 9.9 + 12.1 ms in two;
// 128^3 double: 11.1 ms, 1.4 + 8.0 ms).  64 registers, 256-thread blocks at 4
// per SM: 9.9 ms; 3 per SM 10.0, 2 per SM 10.3.
// sh: shared memory, chem_cols<M>() columns of bs doubles.
// ---------------------------------------------------------------------
template <int M>
constexpr int chem_cols() { return 3 * M; }

template <int M>
__device__ __forceinline__ void chem_node(const StepArgs &a, int n, double *sh, int bs)
{
    const MechConst &mc = c_mech[a.slot];
    const int t = threadIdx.x;
    const size_t N = a.N;
    const RecRows rr = rec_rows(M);
    Real *R = rec(a);
    const double T = a.macro[(size_t)DR_T * N + n];
    const Real rho = R[(size_t)rr.rho * N + n];
    double *sh_act = sh, *sh_g = sh + M * bs;
    WReal *sh_w = reinterpret_cast<WReal *>(sh + 2 * M * bs);
    double conc[M];
#pragma unroll
    for (int s = 0; s < M; ++s) {
#if LBMK_MIXED
        conc[s] = cvt<double>(rho) * cvt<double>(R[(size_t)(rr.y + s) * N + n]) * mc.invW[s];
#else
        conc[s] = rho * R[(size_t)(rr.y + s) * N + n] * mc.invW[s];
#endif
    }
    Real *wd = R + (size_t)rr.wd * N + n;
#if LBMK_MIXED
    if (mc.chem_fixed) {
        const RateSums<true> w{sh + 2 * M * bs + t, bs, rate_scale(rho)};
        molar_production_fixed<M, true>(mc, T, conc, sh_act, sh_g, w, t, bs);
#pragma unroll
        for (int s = 0; s < M; ++s) wd[(size_t)s * N] = w.mass_float(s, mc.W[s]);
        return;
    }
#endif
    production_rates<M>(mc, T, conc, sh_act, sh_g, sh_w, t, bs);
#pragma unroll
    for (int s = 0; s < M; ++s) wd[(size_t)s * N] = cvt<Real>(mc.W[s] * sh_w[s * bs + t]);
}

extern __shared__ double sh_chem[];

template <int M>
__global__ void __launch_bounds__(LBMK_MAXBLOCK, LBMK_CHEM_MINB) k_chem(StepArgs a)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= a.N) return;
    chem_node<M>(a, n, sh_chem, blockDim.x);
}

// ---------------------------------------------------------------------
// Pass 2: G_alpha = (1/omega - 1/2) d_alpha Phi_alpha with the isotropic
// gradient d_alpha phi = (1/theta) sum_i w_i c_ia phi(x + c_i).
// ---------------------------------------------------------------------
template <int M>
__device__ __forceinline__ void grad_node(const StepArgs &a, const Node &nd)
{
    const size_t N = a.N;
    const RecRows rr = rec_rows(M);
    Real *R = rec(a);
    const Real *Phi = R + (size_t)rr.phi * N;
    StencilIdx st;
    make_stencil(st, nd, a);
    Real d[3] = {0, 0, 0};
    for_dirs<0, LBMK_Q>([&](auto dd) {
        constexpr int I = decltype(dd)::value;
        const size_t nb = nb_of<I>(st, a);
        if (CX(I)) d[0] += (Real)(WI(I) * CX(I)) * Phi[nb];
        if (CY(I)) d[1] += (Real)(WI(I) * CY(I)) * Phi[N + nb];
        if (CZ(I)) d[2] += (Real)(WI(I) * CZ(I)) * Phi[2 * N + nb];
    });
    const Real nup = R[(size_t)rr.nup * N + nd.n];
    Real *G = R + (size_t)rr.g * N;
#pragma unroll
    for (int k = 0; k < 3; ++k) G[k * N + nd.n] = nup * (Real)3 * d[k];
}

template <int M>
__global__ void __launch_bounds__(LBMK_MAXBLOCK) k_grad(StepArgs a)
{
    Node nd;
    if (!node_of(nd, a)) return;
    grad_node<M>(a, nd);
}

// ---------------------------------------------------------------------
// Pass 3a: collision of the energy set g, Eq. (g) in the regularised form
//   g + omega (g^eq - g) + w_i (Dq . c_i) / theta,
// with the grad-Y part of Dq (Eq. (corrFourier)) from the neighbours'
// records.  The post-collision value is (1 - omega) g_i + B_i with
//   B_i = omega g_i^eq + 3 w_i c_i . Dq
//       = w_i [A0 + c_i . A1 + sum_d c_id^2 A2_d + sum_{d<e} c_id c_ie A3_de],
//   A0 = omega (rho E - (9/2) tr3),  A1 = 3 (omega q^eq + Dq),
//   A2_d = (9/2) omega R_dd,         A3_de = 9 omega R_de,
// R = R^eq - rho E theta I (Eq. (gieq) expanded in c_i).  Double precision.
// ---------------------------------------------------------------------
template <int M>
__device__ __forceinline__ void collide_energy(const StepArgs &a, const Node &nd)
{
    const int n = nd.n;
    const size_t N = a.N;
    const RecRows rr = rec_rows(M);
    const Real *R = rec(a);
    auto ld = [&](int row) { return R[(size_t)row * N + n]; };
    auto ldd = [&](int row) { return a.macro[(size_t)row * N + n]; };

    // sum_a H_a grad Y_a (Eq. (corrFourier)), H_a of this node
    Real Hl[M];
#pragma unroll
    for (int s = 0; s < M; ++s) Hl[s] = ld(rr.h + s);
    Real HgY[3] = {0, 0, 0};
    {
        StencilIdx st;
        make_stencil(st, nd, a);
        const Real *Yf = R + (size_t)rr.y * N;
        for_dirs<0, LBMK_Q>([&](auto dd) {
            constexpr int I = decltype(dd)::value;
            if constexpr (I != REST) {
                const size_t nb = nb_of<I>(st, a);
                Real hy = 0;
#pragma unroll
                for (int s = 0; s < M; ++s) hy += Hl[s] * Yf[s * N + nb];
                constexpr Real wx = (Real)(WI(I) * CX(I)), wy = (Real)(WI(I) * CY(I)), wz = (Real)(WI(I) * CZ(I));
                if (CX(I)) HgY[0] += wx * hy;
                if (CY(I)) HgY[1] += wy * hy;
                if (CZ(I)) HgY[2] += wz * hy;
            }
        });
    }
    const Real om1 = ld(rr.om1), P = ld(rr.p);
    const double omd = (double)ld(rr.om), om1m = 1.0 - omd;
    double gD[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) gD[d] = (double)(ld(rr.dq + d) + (Real)1.5 * ((Real)2 - om1) * P * HgY[d]);
    // energy equilibrium moments (Eqs. (geq1mom), (geq2mom))
    const double gE = ldd(dr_ge(M));
    double gq[3], gR[6];
#pragma unroll
    for (int d = 0; d < 3; ++d) gq[d] = ldd(dr_gq(M) + d);
#pragma unroll
    for (int d = 0; d < 6; ++d) gR[d] = ldd(dr_gr(M) + d);
    const double gtr = ldd(dr_gtr(M));
    const double A0 = omd * (gE - 4.5 * gtr);
    double A1[3], A2[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        A1[d] = 3.0 * fma(omd, gq[d], gD[d]);
        A2[d] = 4.5 * omd * gR[d];
    }
    const double A3xy = 9.0 * omd * gR[3], A3xz = 9.0 * omd * gR[4], A3yz = 9.0 * omd * gR[5];

    const PopView v = view(a.src, a);
    PullIdx p;
    make_pull(p, nd, a);
    int bad = 0;     // a non-finite result: all exponent bits set (integer test, no FP64 work)
    // row by row: j = (cy+1) + 3 (cz+1), then cx = -1, 0, 1 (i = (cx+1) + 3 j)
    for_dirs<0, 9>([&](auto dj) {
        constexpr int j = decltype(dj)::value, cy = j % 3 - 1, cz = j / 3 - 1;
        constexpr int nnz = (cy != 0) + (cz != 0);
        double base = A0, lin = A1[0];
        if (cy) { base += cy * A1[1] + A2[1]; lin += cy * A3xy; }
        if (cz) { base += cz * A1[2] + A2[2]; lin += cz * A3xz; }
        if (cy && cz) base += (cy * cz) * A3yz;
        // w_i = w(cx) w(cy) w(cz) with w(0) = 2/3, w(+-1) = 1/6
        constexpr double w0 = nnz == 0 ? 8.0 / 27.0 : (nnz == 1 ? 2.0 / 27.0 : 1.0 / 54.0);
        constexpr double w1 = nnz == 0 ? 2.0 / 27.0 : (nnz == 1 ? 1.0 / 54.0 : 1.0 / 216.0);
        const double bq = base + A2[0];
        const double B[3] = {w1 * (bq - lin), w0 * base, w1 * (bq + lin)};
        for_dirs<0, 3>([&](auto dx) {
            constexpr int k = decltype(dx)::value, I = k + 3 * j;
            const double val = fma(om1m, pull_g(v, a, I, p), B[k]);
            store_g(a.dst, a, I, n, val);
            bad |= (__double2hiint(val) & 0x7ff00000) == 0x7ff00000;
        });
    });
    if (bad) flag(a.status, LBMK_BIT_NONFINITE);
}

template <int M>
__global__ void __launch_bounds__(LBMK_MAXBLOCK) k_step_g(StepArgs a)
{
    Node nd;
    if (!node_of(nd, a)) return;
    if constexpr (kFewSpecies<M>) chem_node<M>(a, nd.n, sh_chem, blockDim.x);
    collide_energy<M>(a, nd);
}

// ---------------------------------------------------------------------
// Pass 3b: collisions of the species sets (Eq. (finalNumericalEquations)
// with the quasi-equilibria of Eq. (fStar)) and of the mixture set f
// (Eq. (f) with the isotropy correction of Eq. (Ai)), direction by
// direction, in the storage precision (the double unit's: lbm_collide64.cuh).
// sh: shared memory, step_cols<M>() columns of bs doubles.
// ---------------------------------------------------------------------
#if LBMK_MIXED
template <int M>
constexpr int step_cols() { return 0; }

template <int M, bool FX>
__device__ __forceinline__ void step_node(const StepArgs &a, const Node &nd, double *sh, int bs)
{
    (void)sh;
    (void)bs;
    const MechConst &mc = c_mech[a.slot];
    const int n = nd.n;
    const size_t N = a.N;
    const RecRows rr = rec_rows(M);
    const Real *R = rec(a);
    auto ld = [&](int row) { return R[(size_t)row * N + n]; };
    auto ldd = [&](int row) { return a.macro[(size_t)row * N + n]; };

    // X = -d_alpha G_alpha (Eq. (Xalpha))
    Real X[3] = {0, 0, 0};
    {
        StencilIdx st;
        make_stencil(st, nd, a);
        const Real *G = R + (size_t)rr.g * N;
        for_dirs<0, LBMK_Q>([&](auto dd) {
            constexpr int I = decltype(dd)::value;
            if constexpr (I != REST) {
                const size_t nb = nb_of<I>(st, a);
                constexpr Real wx = (Real)(WI(I) * CX(I)), wy = (Real)(WI(I) * CY(I)), wz = (Real)(WI(I) * CZ(I));
                if (CX(I)) X[0] += wx * G[nb];
                if (CY(I)) X[1] += wy * G[N + nb];
                if (CZ(I)) X[2] += wz * G[2 * N + nb];
            }
        });
#pragma unroll
        for (int k = 0; k < 3; ++k) X[k] *= (Real)-3;
    }

    const Real rho = ld(rr.rho), om = ld(rr.om);
    const Real kappa = ld(rr.kappa), RT = ld(rr.rt);
    const Real u[3] = {ld(rr.u), ld(rr.u + 1), ld(rr.u + 2)};
    const Real T = cvt<Real>(ldd(DR_T));

    // per-species data: mass fraction, quasi-equilibrium velocity u + du_b,
    // beta_b and rho_dot_b (densities, zeta and the products are formed per
    // direction to keep the register footprint small)
    Real Yl[M], xs[M][3], bt[M], wd[M];
#pragma unroll
    for (int s = 0; s < M; ++s) {
        Yl[s] = ld(rr.y + s);
#pragma unroll
        for (int d = 0; d < 3; ++d) xs[s][d] = u[d] + ld(rr.du + 3 * s + d);
        bt[s] = ld(rr.beta + s);
        wd[s] = ld(rr.wd + s);
    }
    const Real u2[3] = {u[0] * u[0], u[1] * u[1], u[2] * u[2]};

    const PopView v = view(a.src, a);
    PullIdx p;
    make_pull(p, nd, a);
    Real check = 0;

    // Directions row by row: j = (cy+1) + 3 (cz+1), then cx = -1, 0, 1
    // (direction i = (cx+1) + 3 j, i.e. i = 0..26 in order).  The y-z
    // factors of the product-form equilibria are formed once per row.  The
    // populations of direction i+1 are loaded while direction i is collided
    // (raw stored values; the rest state is added where they are used).
    Real fraw[M];
    auto load_raw = [&](int i) {
        const Src sr = src_of(i, p, a);
        if (sr.ghost) {
#pragma unroll
            for (int s = 0; s < M; ++s) fraw[s] = (Real)load_ghost(a, sr.side, s, i, sr.idx) - RAWREF(s, i);
        } else {
            if (i == REST) return;
#pragma unroll
            for (int s = 0; s < M; ++s) fraw[s] = load_raw_sf(v, s, i, sr.idx);
        }
    };
    load_raw(0);

    Real pe_yz[M], ps_yz[M];
    Real fe_yz = 0, AXyz = 0;
    int cy = 0, cz = 0;
    auto yz_factors = [&](int s, Real z, Real &pe, Real &ps) {
        pe = psi_c(cy, u[1], u2[1] + z) * psi_c(cz, u[2], u2[2] + z);
        ps = psi_c(cy, xs[s][1], xs[s][1] * xs[s][1] + z) * psi_c(cz, xs[s][2], xs[s][2] * xs[s][2] + z);
    };
#pragma unroll 1
    for (int i = 0; i < LBMK_Q; ++i) {
        const int cx = i % 3 - 1, j = i / 3;
        if (cx < 0) {
            cy = j % 3 - 1;
            cz = j / 3 - 1;
            const int nnz = (cy != 0) + (cz != 0);
            // y-z factors of the species equilibria, shared by the row's three
            // directions
#pragma unroll
            for (int s = 0; s < M; ++s) {
                yz_factors(s, RA(s) * T, pe_yz[s], ps_yz[s]);
            }
            fe_yz = rho * psi_c(cy, u[1], u2[1] + RT) * psi_c(cz, u[2], u2[2] + RT);
            // isotropy correction A_i . X (Eq. (Ai)): only |c_i| = 1
            AXyz = nnz == 1 ? (Real)0.5 * ((Real)cy * X[1] + (Real)cz * X[2]) : (Real)0;
        }
        Real fc[M];
#pragma unroll
        for (int s = 0; s < M; ++s) fc[s] = fraw[s];
        if (i + 1 < LBMK_Q) load_raw(i + 1);
        if (i == REST) continue;   // rest of the species and mixture sets: below
        Real eqp[M], Dl[M];
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const Real z = RA(s) * T;
            const Real pyz = pe_yz[s], syz = ps_yz[s];
            const Real pe = psi_c(cx, u[0], u2[0] + z) * pyz;
            const Real pst = psi_c(cx, xs[s][0], xs[s][0] * xs[s][0] + z) * syz;
            eqp[s] = pe;
            Dl[s] = rho * Yl[s] * (pe - pst);
        }
        // species a < M-1: Eq. (finalNumericalEquations) with F_ai of Eq. (fStar)
#pragma unroll
        for (int s = 0; s < M - 1; ++s) {
            Real F = 0;
#pragma unroll
            for (int b = 0; b < M; ++b)
                if (b != s) F += INVWWD(s, b) * Dl[b];
            F *= kappa * Yl[s];
            // in deviations from the rest state (the stored values; the
            // moments of k_pre are summed from them too): f - r relaxes to
            // feq - r, and the result is stored as it is
            // (explicit fma: the same roundings in every kernel this is inlined into)
            const Real feq = fma(rho * Yl[s], eqp[s], -RAWREF(s, i));
            const Real fd = fc[s];
            const Real val = fma(wd[s], eqp[s], fma(bt[s] - (Real)1, F, fma((Real)2 * bt[s], feq - fd, fd)));
            store_raw(a.dst, a, s, i, n, val);
            check += val;
        }
        // mixture f: Eq. (f) with the isotropy correction A_i . X (Eq. (Ai))
        {
            const Real feq = fma(psi_c(cx, u[0], u2[0] + RT), fe_yz, -RAWREF(M - 1, i));
            const Real AX = cx == 0 ? AXyz : (j == 4 ? (Real)0.5 * (Real)cx * X[0] : (Real)0);
            const Real fd = fc[M - 1];
            const Real val = fma(om, feq - fd, fd) + AX;
            store_raw(a.dst, a, M - 1, i, n, val);
            check += val;
        }
    }
    // Rest direction of the species and mixture sets: populations and
    // equilibria in double, the collision increment (small near
    // equilibrium) in float.
    {
        const double *rs = v.rest();
        Real eqp[M], Dl[M];
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const Real z = RA(s) * T;
            const Real pe = ((Real)1 - (u2[0] + z)) * ((Real)1 - (u2[1] + z)) * ((Real)1 - (u2[2] + z));
            const Real pst = ((Real)1 - (xs[s][0] * xs[s][0] + z)) * ((Real)1 - (xs[s][1] * xs[s][1] + z)) *
                             ((Real)1 - (xs[s][2] * xs[s][2] + z));
            eqp[s] = pe;
            Dl[s] = rho * Yl[s] * (pe - pst);
        }
#pragma unroll
        for (int s = 0; s < M - 1; ++s) {
            Real F = 0;
#pragma unroll
            for (int b = 0; b < M; ++b)
                if (b != s) F += INVWWD(s, b) * Dl[b];
            F *= kappa * Yl[s];
            const double f0 = rs[(size_t)s * N + n];
            const Real diff = cvt<Real>(ldd(DR_FEQ0 + s) - f0);
            const double val = f0 + cvt<double>((Real)2 * bt[s] * diff + (bt[s] - (Real)1) * F + wd[s] * eqp[s]);
            store_sf(mc, a.dst, a, s, REST, n, val);
            check += cvt<Real>(val);
        }
        const double f0 = rs[(size_t)(M - 1) * N + n];
        const double val = f0 + cvt<double>(om * cvt<Real>(ldd(DR_FEQ0 + M - 1) - f0));
        store_sf(mc, a.dst, a, M - 1, REST, n, val);
        check += cvt<Real>(val);
    }
    if (!isfinite(check)) flag(a.status, LBMK_BIT_NONFINITE);
}
#else
}  // namespace
#include "lbm_collide64.cuh"
namespace {
#endif

// Whether the collision has a variant with fixed-point sums: the double one,
// from four species on.
template <int M>
constexpr bool kFixedStep = M >= 4 && !LBMK_MIXED;

// Shared memory of a block of bs threads for step_node, and for all phases of
// the persistent kernel.
template <int M>
constexpr size_t step_smem(int bs) { return (size_t)step_cols<M>() * bs * sizeof(double); }
template <int M>
constexpr size_t persist_smem(int bs)
{
    constexpr int d = diff_cols<M, true>(), c = chem_cols<M>(), s = step_cols<M>();
    return (size_t)(d > c ? (d > s ? d : s) : (c > s ? c : s)) * bs * sizeof(double);
}

extern __shared__ double sh_step[];

template <int M, bool FX>
__global__ void __launch_bounds__(LBMK_BLOCK, LBMK_STEP_MINB) k_step(StepArgs a)
{
    Node nd;
    if (!node_of(nd, a)) return;
    step_node<M, FX>(a, nd, sh_step, blockDim.x);
}

// Opts kernel f in to dynamic shared memory above 48 KB, once per device
// (done: a word of the caller's, bit d: device d has opted in).
// Idempotent, so two threads racing here both succeed.
template <class F>
int opt_in_smem(F *f, size_t bytes, std::atomic<unsigned long long> &done)
{
    if (bytes <= 48 * 1024) return 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
    if (done.load() >> dev & 1ull) return 0;
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return (int)e;
    done.fetch_or(1ull << dev);
    return 0;
}

// ---------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------
inline dim3 grid_for(int n, int bs = LBMK_BLOCK) { return dim3((unsigned)((n + bs - 1) / bs)); }

// Threads per block of kernel k: the context's choice, or (0) the default,
// halved down to one warp while the grid has fewer than 16 blocks per SM.
// Below that the blocks do not spread evenly over the 152 SMs, and with
// fewer warps than schedulers, warps of one block share an SM's FP64 unit
// (76 cycles per instruction for four warps, 64 for one) while others are
// idle.  us per step, all kernels: 1024 nodes with three species in double
// 112.5 -> 109.5, 4096 x 4 x 4 double 773 -> 761.
inline int block_of(const StepArgs &a, int k)
{
    int bs = a.bs[k];
    if (bs > 0) return bs;
    bs = k == LBMK_K_STEP && !LBMK_MIXED ? LBMK_BLOCK / 2 : LBMK_BLOCK;
    while (bs > 32 && (a.N + bs - 1) / bs < 16 * 152) bs /= 2;
    return bs;
}

template <int M, bool FX>
int launch_step(const StepArgs &a, int bs)
{
    static std::atomic<unsigned long long> opted{0};
    const int e = opt_in_smem(k_step<M, FX>, step_smem<M>(LBMK_BLOCK), opted);
    if (e) return e;
    k_step<M, FX><<<grid_for(a.N, bs), bs, step_smem<M>(bs), a.stream>>>(a);
    return 0;
}

// Launch of one kernel of the step with the context's block size for it
// (LBMK_K_*; the autotuner times them one at a time).
template <int M>
int launch_one(const StepArgs &a, int k)
{
    const int bs = block_of(a, k);
    switch (k) {
    case LBMK_K_GHOST:
        if (a.bc_x == 1) launch_ghost<M>(a);
        break;
    case LBMK_K_PRE: {
        k_pre<M><<<grid_for(a.N, bs), bs, pre_cols<M>() * bs * sizeof(double), a.stream>>>(a);
        constexpr bool FX = kRefined<M, true>;
        static_assert(diff_cols<M, true>() * LBMK_BLOCK * sizeof(double) <= 48 * 1024, "more needs an opt-in");
        if (kFewSpecies<M>) break;                  // k_pre went on
        if (FX && a.fixed)
            k_diff<M, FX><<<grid_for(a.N, bs), bs, diff_cols<M, FX>() * bs * sizeof(double), a.stream>>>(a);
        else
            k_diff<M, false><<<grid_for(a.N, bs), bs, 0, a.stream>>>(a);
        break;
    }
    case LBMK_K_CHEM: {
        if (kFewSpecies<M>) break;                  // in k_step_g
        static std::atomic<unsigned long long> opted{0};
        const int e = opt_in_smem(k_chem<M>, chem_cols<M>() * LBMK_MAXBLOCK * sizeof(double), opted);
        if (e) return e;
        k_chem<M><<<grid_for(a.N, bs), bs, chem_cols<M>() * bs * sizeof(double), a.stream>>>(a);
        break;
    }
    case LBMK_K_GRAD: k_grad<M><<<grid_for(a.N, bs), bs, 0, a.stream>>>(a); break;
    case LBMK_K_STEPG:
        k_step_g<M><<<grid_for(a.N, bs), bs, kFewSpecies<M> ? chem_cols<M>() * bs * sizeof(double) : 0, a.stream>>>(a);
        break;
    case LBMK_K_STEP: {
        constexpr bool FX = kFixedStep<M>;
        const int e = FX && a.fixed ? launch_step<M, FX>(a, bs) : launch_step<M, false>(a, bs);
        if (e) return e;
        break;
    }
    default: return (int)cudaErrorInvalidValue;
    }
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------
// Persistent step: nsteps time steps of every node in one cooperative
// launch.  Within a phase each warp takes chunks of `chunk` consecutive
// nodes from a queue (one atomic per chunk), so that SMs whose nodes cost
// less (fewer Newton iterations, no flame) take more of them; the phases
// that read a neighbour's value of the same time level -- ghost planes,
// the record (k_pre), G (k_grad), then both collisions -- are separated by
// grid barriers, whose last arrival also resets the queue, and the two
// population buffers swap every step.  A barrier polls at most `cap`
// times: a block that runs out sets LBMK_BIT_BARRIER and returns, and the
// others then run out at the next barrier, so the launch always ends.
// Built only in the units with coherent loads (LBMK_COHERENT_LOADS).
// ---------------------------------------------------------------------
#if LBMK_COHERENT_LOADS
__device__ __forceinline__ bool grid_barrier(GridBarrier *g, unsigned nblocks, unsigned cap, unsigned *status)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        volatile unsigned *vgen = &g->gen;
        const unsigned gen = *vgen;                    // read before arriving: only this barrier's last arrival changes it
        __threadfence();
        if (atomicAdd(&g->count, 1u) == nblocks - 1) {
            atomicExch(&g->count, 0u);
            atomicExch(&g->next, 0u);                  // every block is past its last take
            __threadfence();
            atomicAdd(&g->gen, 1u);
        } else {
            unsigned it = 0;
            while (*vgen == gen) {
                if (++it > cap) {
                    flag(status, LBMK_BIT_BARRIER);
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// Each warp takes chunks of `chunk` consecutive nodes (a multiple of 32)
// until the queue passes the last node.
template <int M, class Body>
__device__ __forceinline__ void tile_loop(const StepArgs &a, int chunk, unsigned *next, Body &&body)
{
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned c = 0;
        if (lane == 0) c = atomicAdd(next, 1u);
        c = __shfl_sync(0xffffffffu, c, 0);
        const long long base = (long long)c * chunk;
        if (base >= a.N) break;
        for (int k = lane; k < chunk; k += 32) {
            Node nd;
            nd.n = (int)(base + k);
            if (nd.n >= a.N) break;
            node_at(nd, a);
            body(nd);
        }
    }
}

// One time step of the persistent kernel over the buffers of b.
template <int M, bool FX>
__device__ __forceinline__ bool persist_step(const StepArgs &b, int tile, GridBarrier *bar, unsigned nb, unsigned cap)
{
    if (b.bc_x == 1) {
        const int nw = (ghost_count(b) + ghost_groups<M>() - 1) / ghost_groups<M>();
        const int per = blockDim.x / 32;
        for (int w = blockIdx.x + gridDim.x * (threadIdx.x / 32); w < nw; w += gridDim.x * per) ghost_warp<M>(b, w);
        if (!grid_barrier(bar, nb, cap, b.status)) return false;
    }
    tile_loop<M>(b, tile, &bar->next, [&](const Node &nd) {
        pre_node<M>(b, nd, sh_step + threadIdx.x, LBMK_BLOCK);
        diff_node<M, FX && kRefined<M, true>>(b, nd, sh_step + threadIdx.x, LBMK_BLOCK);
    });
    if (!grid_barrier(bar, nb, cap, b.status)) return false;
    tile_loop<M>(b, tile, &bar->next, [&](const Node &nd) { grad_node<M>(b, nd); });
    if (!grid_barrier(bar, nb, cap, b.status)) return false;
    // the two collisions read the same inputs and write disjoint sets; the
    // barrier between them only resets the queue, and separate loops keep
    // each one's arithmetic as in its own kernel (no values shared)
    tile_loop<M>(b, tile, &bar->next, [&](const Node &nd) { collide_energy<M>(b, nd); });
    if (!grid_barrier(bar, nb, cap, b.status)) return false;
    tile_loop<M>(b, tile, &bar->next, [&](const Node &nd) {
        chem_node<M>(b, nd.n, sh_step, LBMK_BLOCK);
        step_node<M, FX && kFixedStep<M>>(b, nd, sh_step, LBMK_BLOCK);
    });
    return grid_barrier(bar, nb, cap, b.status);
}

// a0 steps src -> dst, a1 the same with the buffers swapped: the steps
// alternate between the two parameter blocks, which the phases then read
// in place (no per-step copy of the arguments)
template <int M, bool FX>
__global__ void __launch_bounds__(LBMK_BLOCK, LBMK_PERSIST_MINB) k_persist(StepArgs a0, StepArgs a1, int nsteps, int tile,
                                                                      GridBarrier *bar, unsigned cap)
{
    const unsigned nb = gridDim.x;
    for (int t = 0; t < nsteps; t += 2) {
        if (!persist_step<M, FX>(a0, tile, bar, nb, cap)) return;
        if (t + 1 < nsteps && !persist_step<M, FX>(a1, tile, bar, nb, cap)) return;
    }
}

template <int M, bool FX>
int launch_persistent(const StepArgs &a, int nsteps, int tile_mult, GridBarrier *bar, unsigned cap)
{
    if (nsteps < 1 || tile_mult < 1) return (int)cudaErrorInvalidValue;
    int per_sm = 0, dev = 0, nsm = 0;
    static std::atomic<unsigned long long> opted{0};
    const int eo = opt_in_smem(k_persist<M, FX>, persist_smem<M>(LBMK_BLOCK), opted);
    if (eo) return eo;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persist<M, FX>, LBMK_BLOCK,
                                                                  persist_smem<M>(LBMK_BLOCK));
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return (int)e;
    const int tile = tile_mult * 32;                   // nodes per warp take
    const long long tiles = ((long long)a.N + LBMK_BLOCK - 1) / LBMK_BLOCK;
    const int blocks = (int)std::min<long long>((long long)per_sm * nsm, tiles);
    if (blocks < 1) return (int)cudaErrorInvalidConfiguration;
    StepArgs a0 = a, a1 = a;
    a1.src = a.dst;
    a1.dst = const_cast<void *>(a.src);
    int ns = nsteps, tl = tile;
    GridBarrier *bb = bar;
    unsigned cc = cap;
    void *args[] = {(void *)&a0, (void *)&a1, (void *)&ns, (void *)&tl, (void *)&bb, (void *)&cc};
    return (int)cudaLaunchCooperativeKernel((const void *)k_persist<M, FX>, dim3(blocks), dim3(LBMK_BLOCK), args,
                                            persist_smem<M>(LBMK_BLOCK), a.stream);
}
template <int M>
int run_persistent(const StepArgs &a, int nsteps, int tile_mult, GridBarrier *bar, unsigned cap)
{
    constexpr bool FX = kRefined<M, true> || kFixedStep<M>;
    if (FX && a.fixed) return launch_persistent<M, FX>(a, nsteps, tile_mult, bar, cap);
    return launch_persistent<M, false>(a, nsteps, tile_mult, bar, cap);
}
#endif  // LBMK_COHERENT_LOADS

template <int M>
int run_step(const StepArgs &a, cudaEvent_t *ev)
{
    for (int k = 0; k < LBMK_NKERNELS; ++k) {
        if (ev) cudaEventRecord(ev[k], a.stream);
        const int e = launch_one<M>(a, k);
        if (e) return e;
    }
    if (ev) cudaEventRecord(ev[LBMK_NKERNELS], a.stream);
    return (int)cudaGetLastError();
}

template <int M>
int run_moments(const StepArgs &a, unsigned mask, double *out)
{
    if (a.bc_x == 1) launch_ghost<M>(a);
    k_moments<M><<<grid_for(a.N), LBMK_BLOCK, 0, a.stream>>>(a, mask, out);
    return (int)cudaGetLastError();
}

template <int M>
int run_init(const StepArgs &a, const double *X, const double *T, const double *u, double P)
{
    k_init<M><<<grid_for(a.N), LBMK_BLOCK, 0, a.stream>>>(a, X, T, u, P);
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------
// Statistics of an initial state from which the mixed modes choose their
// rest references: per node rho = P m / (r_lat T) (m = sum_a X_a W_a) and
// rho_a = rho X_a W_a / m; over the lattice the minima of rho_a and rho and
// the sums of rho_a, rho and T.  Record of 2M+3 doubles: min rho_a (M),
// min rho, sum rho_a (M), sum rho, sum T.  Two passes with a fixed
// reduction order (LBMK_STAT_BLOCKS partial records, then one block), so
// that the result -- and every state that depends on it -- is the same
// from run to run.
// ---------------------------------------------------------------------
constexpr int LBMK_STAT_THREADS = 256;

__host__ __device__ constexpr int stat_len(int M) { return 2 * M + 3; }

template <int M>
__device__ __forceinline__ void stat_combine(double *acc, const double *o)
{
#pragma unroll
    for (int k = 0; k <= M; ++k) acc[k] = fmin(acc[k], o[k]);
#pragma unroll
    for (int k = M + 1; k < stat_len(M); ++k) acc[k] += o[k];
}

template <int M>
__device__ __forceinline__ void stat_identity(double *acc)
{
#pragma unroll
    for (int k = 0; k <= M; ++k) acc[k] = INFINITY;
#pragma unroll
    for (int k = M + 1; k < stat_len(M); ++k) acc[k] = 0.0;
}

// Tree reduction of the block's records in shared memory (fixed order);
// thread 0 leaves the block's record in sh[0 .. stat_len(M)).
template <int M>
__device__ __forceinline__ void stat_block_reduce(double *acc, double *sh)
{
    const int t = threadIdx.x;
#pragma unroll
    for (int k = 0; k < stat_len(M); ++k) sh[k * LBMK_STAT_THREADS + t] = acc[k];
    __syncthreads();
    for (int w = LBMK_STAT_THREADS / 2; w > 0; w >>= 1) {
        if (t < w) {
            double o[stat_len(M)];
#pragma unroll
            for (int k = 0; k < stat_len(M); ++k) o[k] = sh[k * LBMK_STAT_THREADS + t + w];
            stat_combine<M>(acc, o);
#pragma unroll
            for (int k = 0; k < stat_len(M); ++k) sh[k * LBMK_STAT_THREADS + t] = acc[k];
        }
        __syncthreads();
    }
}

template <int M>
__global__ void __launch_bounds__(LBMK_STAT_THREADS) k_stat_partial(StepArgs a, const double *X, const double *T,
                                                                     double P, double *partial)
{
    __shared__ double sh[stat_len(M) * LBMK_STAT_THREADS];
    const MechConst &mc = c_mech[a.slot];
    double acc[stat_len(M)];
    stat_identity<M>(acc);
    for (int n = blockIdx.x * LBMK_STAT_THREADS + threadIdx.x; n < a.N; n += gridDim.x * LBMK_STAT_THREADS) {
        double m = 0.0;
#pragma unroll
        for (int s = 0; s < M; ++s) m += X[(size_t)s * a.N + n] * mc.W[s];
        const double Tn = T[n];
        const double rho = P * m / (mc.r_lat * Tn);
        double o[stat_len(M)];
#pragma unroll
        for (int s = 0; s < M; ++s) {
            const double ra = rho * X[(size_t)s * a.N + n] * mc.W[s] / m;
            o[s] = ra;
            o[M + 1 + s] = ra;
        }
        o[M] = rho;
        o[2 * M + 1] = rho;
        o[2 * M + 2] = Tn;
        stat_combine<M>(acc, o);
    }
    stat_block_reduce<M>(acc, sh);
    if (threadIdx.x == 0)
        for (int k = 0; k < stat_len(M); ++k) partial[(size_t)k * gridDim.x + blockIdx.x] = sh[k * LBMK_STAT_THREADS];
}

template <int M>
__global__ void __launch_bounds__(LBMK_STAT_THREADS) k_stat_final(const double *partial, int nblocks, double *out)
{
    __shared__ double sh[stat_len(M) * LBMK_STAT_THREADS];
    double acc[stat_len(M)];
    stat_identity<M>(acc);
    for (int b = threadIdx.x; b < nblocks; b += LBMK_STAT_THREADS) {
        double o[stat_len(M)];
#pragma unroll
        for (int k = 0; k < stat_len(M); ++k) o[k] = partial[(size_t)k * nblocks + b];
        stat_combine<M>(acc, o);
    }
    stat_block_reduce<M>(acc, sh);
    if (threadIdx.x == 0)
        for (int k = 0; k < stat_len(M); ++k) out[k] = sh[k * LBMK_STAT_THREADS];
}

// scratch: device, at least LBMK_STAT_BLOCKS * (2M+3) doubles; out: device, 2M+3 doubles.
template <int M>
int run_ref_stats(const StepArgs &a, const double *X, const double *T, double P, double *scratch, double *out)
{
    const int nb = (int)std::min<long long>(LBMK_STAT_BLOCKS, ((long long)a.N + LBMK_STAT_THREADS - 1) /
                                                                  LBMK_STAT_THREADS);
    k_stat_partial<M><<<nb, LBMK_STAT_THREADS, 0, a.stream>>>(a, X, T, P, scratch);
    k_stat_final<M><<<1, LBMK_STAT_THREADS, 0, a.stream>>>(scratch, nb, out);
    return (int)cudaGetLastError();
}


// ---------------------------------------------------------------------
// Heat release rate hdot^c = -sum_a H_a rho_dot_a (Sec. 5b) of the state in
// src (the state lbm_moments reports) and its partial derivatives there.
// With the reaction enthalpy dH_k = sum_a W_a (nu''_ak - nu'_ak) H_a(T),
// hdot^c = -sum_k dH_k q_k, and q_k = F_k (k_f P_f - k_r P_r) with
//   k_f = A_k (T/T_ref)^b_k exp(-theta_k/T),  P_f, P_r the products of the
//   reactant and product concentrations c_a = rho_a / W_a,
//   k_r = k_f / K_c, ln K_c = -sum_a dnu_a g_a/(R_U T) + dn ln(P0/(r T)),
//   F = 1, [M] = sum_a eff_a c_a (third body) or Pr/(1+Pr) with
//   Pr = (k0/k_inf) [M] (Lindemann falloff; A_k is that of k_inf).
// The derivatives are taken at fixed densities (for d/dT) and at fixed
// temperature (for d/drho_a, every one of the M densities independent):
//   d ln k_f/dT = (b + theta/T)/T,
//   d ln K_c/dT = dH_k/(r T^2) - dn/T          (van 't Hoff; d(g_a/RT)/dT = -h_a/(R T^2)),
//   d ln q_k/d ln A_k = 1, or Pr/(1+Pr) for falloff (Pr scales as 1/k_inf),
//   d dH_k/dT = sum_a W_a dnu_a C_p,a.
// Each block sums hdot^c and d hdot^c/d ln A_k over its nodes (grid-stride,
// then a tree in shared memory, in a fixed order); k_hrr_final sums the
// blocks in a fixed order, so that the totals repeat from run to run.
// ---------------------------------------------------------------------


// hdot^c at one node state (T, rho_a) and its derivatives: d/dT into *dT,
// d/drho_a into drho[M], and d/d ln A_k added to dA[k * stride] (k < R).
template <int M, bool WITH_A = true>
__device__ __forceinline__ double hrr_node(const MechConst &mc, double T, const double *rho_a, double *dT_out,
                                           double *drho, double *dA, int stride)
{
    const double invT = 1.0 / T, lnTr = log(T) - mc.log_T_ref;
    const double lnc0 = log(mc.P0_over_r * invT);              // ln(P0/(r T))
    const double vhf = invT * invT / mc.r_lat;                 // 1/(r T^2), van 't Hoff factor
    double conc[M], WH[M], Wcp[M], g[M], dc[M];
#pragma unroll
    for (int s = 0; s < M; ++s) {
        conc[s] = rho_a[s] * mc.invW[s];
        WH[s] = mc.W[s] * H_spec(mc, s, T);
        Wcp[s] = mc.W[s] * cp_spec(mc, s, T);
        const double *gc = mc.gco[s];
        g[s] = fma(gc[0], 1.0 - log(T),
                   fma(fma(fma(fma(gc[4], T, gc[3]), T, gc[2]), T, gc[1]), T, fma(gc[5], invT, gc[6])));
        dc[s] = 0.0;
    }
    double hdot = 0.0, dT = 0.0;
    for (int k = 0; k < mc.R; ++k) {
        const int nr = mc.nreac[k], np = mc.nprod[k];
        double dH = 0.0, dHdT = 0.0, dG = 0.0, Pf = 1.0, Pp = 1.0;
        for (int j = 0; j < nr; ++j) {
            const int s = mc.reac[k][j];
            dH -= WH[s];
            dHdT -= Wcp[s];
            dG -= g[s];
            Pf *= conc[s];
        }
        for (int j = 0; j < np; ++j) {
            const int s = mc.prod[k][j];
            dH += WH[s];
            dHdT += Wcp[s];
            dG += g[s];
            Pp *= conc[s];
        }
        const double lnkf = fma(mc.b[k], lnTr, fma(-mc.theta[k], invT, mc.log_A[k]));
        const double kf = exp_table(lnkf);
        const double dlnkf = fma(mc.theta[k], invT, mc.b[k]) * invT;
        double kr = 0.0, dlnkr = 0.0;
        if (mc.rev[k]) {
            kr = exp_table(lnkf - fma((double)mc.dn[k], lnc0, -dG));       // k_f / K_c
            dlnkr = dlnkf - fma(dH, vhf, -mc.dn[k] * invT);
        }
        const double qf = kf * Pf, qr = kr * Pp, q0 = qf - qr;
        double F = 1.0, dFdT = 0.0, dFdcM = 0.0, sA = 1.0;
        const int type = mc.rtype[k];
        if (type != 0) {
            double cM = 0.0;
#pragma unroll
            for (int s = 0; s < M; ++s) cM = fma(mc.eff[k][s], conc[s], cM);
            if (type == 1) {
                F = cM;
                dFdcM = 1.0;
            } else {
                const double k0r = exp_table(fma(mc.dlow[k][1], lnTr, fma(-mc.dlow[k][2], invT, mc.dlow[k][0])));
                const double Pr = k0r * cM, i1 = 1.0 / (1.0 + Pr);
                F = Pr * i1;
                dFdcM = k0r * i1 * i1;
                dFdT = F * i1 * fma(mc.dlow[k][2], invT, mc.dlow[k][1]) * invT;
                sA = F;                                     // Pr/(1+Pr)
            }
        }
        const double q = F * q0;
        hdot -= dH * q;
        if constexpr (WITH_A) dA[k * stride] -= dH * q * sA;
        dT -= fma(dHdT, q, dH * fma(F, qf * dlnkf - qr * dlnkr, q0 * dFdT));
        // d q/d c_b: the reactant and product products with one factor left out
        const double wf = -dH * F * kf, wr = dH * F * kr;
        for (int j = 0; j < nr; ++j) {
            double pj = wf;
            for (int i = 0; i < nr; ++i)
                if (i != j) pj *= conc[mc.reac[k][i]];
            dc[mc.reac[k][j]] += pj;
        }
        if (mc.rev[k])
            for (int j = 0; j < np; ++j) {
                double pj = wr;
                for (int i = 0; i < np; ++i)
                    if (i != j) pj *= conc[mc.prod[k][i]];
                dc[mc.prod[k][j]] += pj;
            }
        if (type != 0) {
            const double wm = -dH * q0 * dFdcM;
#pragma unroll
            for (int s = 0; s < M; ++s) dc[s] = fma(wm, mc.eff[k][s], dc[s]);
        }
    }
    *dT_out = dT;
#pragma unroll
    for (int s = 0; s < M; ++s) drho[s] = dc[s] * mc.invW[s];      // c_a = rho_a / W_a
    return hdot;
}

template <int M>
__global__ void __launch_bounds__(LBMK_HRR_THREADS, 3) k_hrr(StepArgs a, double *dT_out, double *drho_out,
                                                          double *partial)
{
    __shared__ double sh_dA[LBMK_MAXR * LBMK_HRR_THREADS];
    __shared__ double sh_J[LBMK_HRR_THREADS];
    __shared__ double sh_ra[M * LBMK_HRR_THREADS];
    const MechConst &mc = c_mech[a.slot];
    const int t = threadIdx.x, R = mc.R;
    const size_t N = a.N;
    for (int k = 0; k < R; ++k) sh_dA[k * LBMK_HRR_THREADS + t] = 0.0;
    double Jt = 0.0;
    for (int n = blockIdx.x * LBMK_HRR_THREADS + t; n < a.N; n += gridDim.x * LBMK_HRR_THREADS) {
        Node nd;
        nd.n = n;
        node_at(nd, a);
        PullIdx p;
        make_pull(p, nd, a);
        Sums sm = {};
        const double T = node_temperature<M>(mc, a, p, n, sm, sh_ra + t, LBMK_HRR_THREADS);
        double rho_a[M];
#pragma unroll
        for (int s = 0; s < M; ++s) rho_a[s] = sh_ra[s * LBMK_HRR_THREADS + t];
        double dT, drho[M];
        Jt += hrr_node<M>(mc, T, rho_a, &dT, drho, sh_dA + t, LBMK_HRR_THREADS);
        if (dT_out) dT_out[n] = dT;
        if (drho_out)
#pragma unroll
            for (int s = 0; s < M; ++s) drho_out[(size_t)s * N + n] = drho[s];
    }
    sh_J[t] = Jt;
    __syncthreads();
    for (int w = LBMK_HRR_THREADS / 2; w > 0; w >>= 1) {
        if (t < w) {
            sh_J[t] += sh_J[t + w];
            for (int k = 0; k < R; ++k) sh_dA[k * LBMK_HRR_THREADS + t] += sh_dA[k * LBMK_HRR_THREADS + t + w];
        }
        __syncthreads();
    }
    if (t == 0) {
        double *o = partial + (size_t)blockIdx.x * (1 + R);
        o[0] = sh_J[0];
        for (int k = 0; k < R; ++k) o[1 + k] = sh_dA[k * LBMK_HRR_THREADS];
    }
}

// The chemistry of n given node states (rho_a [M][n], T [n]; device): the
// step's production rates (molar_production, as k_chem evaluates them) and
// hdot^c with its derivatives (hrr_node); each output may be null.
template <int M>
__global__ void __launch_bounds__(LBMK_BLOCK) k_chem_at(StepArgs a, int n, const double *rho_in, const double *T_in,
                                                        double *rho_dot, double *hdot, double *dT_out,
                                                        double *drho_out, double *dA_out)
{
    __shared__ double sh_act[M * LBMK_BLOCK];
    __shared__ double sh_g[M * LBMK_BLOCK];
    __shared__ WReal sh_w[M * LBMK_BLOCK];
    const MechConst &mc = c_mech[a.slot];
    const int t = threadIdx.x, i = blockIdx.x * LBMK_BLOCK + t;
    if (i >= n) return;
    double rho_a[M], conc[M];
#pragma unroll
    for (int s = 0; s < M; ++s) {
        rho_a[s] = rho_in[(size_t)s * n + i];
        conc[s] = rho_a[s] * mc.invW[s];
    }
    const double T = T_in[i];
    if (rho_dot) {
        production_rates<M>(mc, T, conc, sh_act, sh_g, sh_w, t, LBMK_BLOCK);
#pragma unroll
        for (int s = 0; s < M; ++s) rho_dot[(size_t)s * n + i] = mc.W[s] * (double)sh_w[s * LBMK_BLOCK + t];
    }
    if (hdot || dT_out || drho_out || dA_out) {
        double dT, drho[M], dA[LBMK_MAXR];
        for (int k = 0; k < mc.R; ++k) dA[k] = 0.0;
        const double h = hrr_node<M>(mc, T, rho_a, &dT, drho, dA, 1);
        if (hdot) hdot[i] = h;
        if (dT_out) dT_out[i] = dT;
        if (drho_out)
#pragma unroll
            for (int s = 0; s < M; ++s) drho_out[(size_t)s * n + i] = drho[s];
        if (dA_out)
            for (int k = 0; k < mc.R; ++k) dA_out[(size_t)k * n + i] = dA[k];
    }
}

// Temperatures of n given node states (Y [M][n], specific internal energy
// e [n], Newton starting points T0 [n]; device) by the step's Newton
// iteration (mixture_energy_poly, solve_T).
template <int M>
__global__ void __launch_bounds__(LBMK_BLOCK) k_temperature_at(StepArgs a, int n, const double *Y_in,
                                                               const double *e_in, const double *T0_in,
                                                               double *T_out)
{
    const MechConst &mc = c_mech[a.slot];
    const int i = blockIdx.x * LBMK_BLOCK + threadIdx.x;
    if (i >= n) return;
    double Y[M], eu[6];
#pragma unroll
    for (int s = 0; s < M; ++s) Y[s] = Y_in[(size_t)s * n + i];
    mixture_energy_poly<M>(mc, Y, eu);
    T_out[i] = solve_T(eu, e_in[i], T0_in[i], a.status);
}

// Column c of nb partial records of width w, summed in a fixed order.
__global__ void __launch_bounds__(LBMK_HRR_THREADS) k_hrr_final(const double *partial, int nb, int w, double *out)
{
    __shared__ double sh[LBMK_HRR_THREADS];
    const int t = threadIdx.x, c = blockIdx.x;
    double acc = 0.0;
    for (int b = t; b < nb; b += LBMK_HRR_THREADS) acc += partial[(size_t)b * w + c];
    sh[t] = acc;
    __syncthreads();
    for (int h = LBMK_HRR_THREADS / 2; h > 0; h >>= 1) {
        if (t < h) sh[t] += sh[t + h];
        __syncthreads();
    }
    if (t == 0) out[c] = sh[0];
}

// partial: hrr_blocks(N) (1 + R) doubles; out: 1 + R doubles
// {sum hdot^c, sum d hdot^c/d ln A_k}.
template <int M>
int run_hrr(const StepArgs &a, int R, double *dT, double *drho, double *partial, double *out)
{
    if (a.bc_x == 1) launch_ghost<M>(a);
    const int nb = lbmk::hrr_blocks(a.N);
    k_hrr<M><<<nb, LBMK_HRR_THREADS, 0, a.stream>>>(a, dT, drho, partial);
    k_hrr_final<<<1 + R, LBMK_HRR_THREADS, 0, a.stream>>>(partial, nb, 1 + R, out);
    return (int)cudaGetLastError();
}

template <int M>
int run_chem_at(const StepArgs &a, int n, const double *rho_a, const double *T, double *rho_dot, double *hdot,
                double *dT, double *drho, double *dA)
{
    if (n > 0)
        k_chem_at<M><<<grid_for(n), LBMK_BLOCK, 0, a.stream>>>(a, n, rho_a, T, rho_dot, hdot, dT, drho, dA);
    return (int)cudaGetLastError();
}

template <int M>
int run_temperature_at(const StepArgs &a, int n, const double *Y, const double *e, const double *T0, double *T)
{
    if (n > 0) k_temperature_at<M><<<grid_for(n), LBMK_BLOCK, 0, a.stream>>>(a, n, Y, e, T0, T);
    return (int)cudaGetLastError();
}


// ---------------------------------------------------------------------
// Gradient of J = sum_nodes hdot^c with respect to the stored populations
// F of the current state (periodic lattices), the source term of the
// objective in an adjoint of the step.  Node n pulls P_si(n) = F_si(n - c_i)
// and forms rho_a (a < M-1), rho, j and rho E from the pulled sets; the
// slaved density is rho - sum_a rho_a, Y_a = rho_a / rho, and T solves
// sum_a Y_a U_a(T) = e with e = rho E / rho - |j|^2 / (2 rho^2).  By the
// implicit function theorem dT = (de - sum_a U_a dY_a) / C_v.  With
// G_T = d hdot/dT and G_a = d hdot/d rho_a (hrr_node) and l = G_T / C_v:
//   d hdot/d rho_s = G_s - G_{M-1} - l (U_s - U_{M-1}) / rho   (s < M-1)
//   d hdot/d rho   = G_{M-1} + l (de/drho - (U_{M-1} - sum_a Y_a U_a) / rho),
//                    de/drho = -rho E / rho^2 + |j|^2 / rho^3
//   d hdot/d j_d   = -l u_d / rho,      d hdot/d (rho E) = l / rho,
// and dJ/dF_si(x) is the value of node x + c_i for its set (for f:
// d/drho + c_i . d/dj).
// ---------------------------------------------------------------------

// adj [M + 4][N]: d hdot/d rho_s (s < M-1), d/d rho, d/d j (3), d/d rho E.
template <int M>
__global__ void __launch_bounds__(LBMK_HRR_THREADS, 3) k_hrr_adj(StepArgs a, double *adj)
{
    const MechConst &mc = c_mech[a.slot];
    const int n = blockIdx.x * LBMK_HRR_THREADS + threadIdx.x;
    if (n >= a.N) return;
    const size_t N = a.N;
    Node nd;
    nd.n = n;
    node_at(nd, a);
    PullIdx p;
    make_pull(p, nd, a);
    __shared__ double sh_ra[M * LBMK_HRR_THREADS];
    Sums sm;
    double eu[6];
    const double T = node_temperature<M>(mc, a, p, n, sm, sh_ra + threadIdx.x, LBMK_HRR_THREADS, eu);
    const double rho = sm.rho;
    double rho_a[M], Y[M];
#pragma unroll
    for (int s = 0; s < M; ++s) {
        rho_a[s] = sh_ra[s * LBMK_HRR_THREADS + threadIdx.x];
        Y[s] = rho_a[s] / rho;
    }
    const double u[3] = {sm.j[0] / rho, sm.j[1] / rho, sm.j[2] / rho};
    double GT, G[M];
    hrr_node<M, false>(mc, T, rho_a, &GT, G, nullptr, 0);
    const double l = GT / dpoly5(eu, T), ir = 1.0 / rho;
    double U[M], Umix = 0.0;
#pragma unroll
    for (int s = 0; s < M; ++s) {
        U[s] = poly5(mc.uco[s], T);
        Umix = fma(Y[s], U[s], Umix);
    }
#pragma unroll
    for (int s = 0; s < M - 1; ++s) adj[(size_t)s * N + n] = G[s] - G[M - 1] - l * (U[s] - U[M - 1]) * ir;
    const double jsq = sm.j[0] * sm.j[0] + sm.j[1] * sm.j[1] + sm.j[2] * sm.j[2];
    const double dedrho = (jsq * ir - sm.rhoE) * ir * ir;
    adj[(size_t)(M - 1) * N + n] = G[M - 1] + l * (dedrho - (U[M - 1] - Umix) * ir);
#pragma unroll
    for (int d = 0; d < 3; ++d) adj[(size_t)(M + d) * N + n] = -l * u[d] * ir;
    adj[(size_t)(M + 3) * N + n] = l * ir;
}

// dJ/dF of set s (0..M), out [27][N]: each direction gathers from x + c_i.
template <int M>
__global__ void __launch_bounds__(LBMK_BLOCK) k_hrr_adj_gather(StepArgs a, const double *adj, int s, double *out)
{
    Node nd;
    if (!node_of(nd, a)) return;
    const size_t N = a.N;
    StencilIdx st;
    make_stencil(st, nd, a);
    for_dirs<0, LBMK_Q>([&](auto dd) {
        constexpr int I = decltype(dd)::value;
        const size_t nb = nb_of<I>(st, a);
        double v;
        if (s < M - 1) {
            v = adj[(size_t)s * N + nb];
        } else if (s == M - 1) {
            v = adj[(size_t)(M - 1) * N + nb];
            if (CX(I)) v += CX(I) * adj[(size_t)M * N + nb];
            if (CY(I)) v += CY(I) * adj[(size_t)(M + 1) * N + nb];
            if (CZ(I)) v += CZ(I) * adj[(size_t)(M + 2) * N + nb];
        } else {
            v = adj[(size_t)(M + 3) * N + nb];
        }
        out[(size_t)I * N + nd.n] = v;
    });
}

template <int M>
int run_hrr_adj(const StepArgs &a, double *adj)
{
    k_hrr_adj<M><<<grid_for(a.N, LBMK_HRR_THREADS), LBMK_HRR_THREADS, 0, a.stream>>>(a, adj);
    return (int)cudaGetLastError();
}

template <int M>
int run_hrr_adj_gather(const StepArgs &a, const double *adj, int s, double *out)
{
    k_hrr_adj_gather<M><<<grid_for(a.N), LBMK_BLOCK, 0, a.stream>>>(a, adj, s, out);
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------
// Flame diagnostics of the circular expanding flame (Sec. 5b), from the
// record k_pre forms for the current state:
//   S_d = [ hdot^c + div(lambda grad T) - rho (sum_a C_a,p Y_a du_a) . grad T ]
//         / (rho C_p |grad T|)                                   (Eq. (sd))
//   S_a = S_d + u . n,  n = -grad T / |grad T|,
// lambda = (1/omega_1 - 1/2) P C_p (Eq. (lambda)), C_p = sum_a Y_a C_a,p,
// the gradients by the isotropic stencil (the divergence as the sum of the
// component derivatives of lambda grad T).  Pass 1 forms grad T and
// lambda grad T (scratch [6][N]); pass 2 the rest.  S_d = S_a = 0 where
// grad T = 0.
// ---------------------------------------------------------------------
template <int M>
__global__ void __launch_bounds__(LBMK_BLOCK) k_flame1(StepArgs a, double *scr)
{
    const MechConst &mc = c_mech[a.slot];
    Node nd;
    if (!node_of(nd, a)) return;
    const size_t N = a.N;
    const int n = nd.n;
    const RecRows rr = rec_rows(M);
    const Real *R = rec(a);
    const double *Tr = a.macro + (size_t)DR_T * N;
    StencilIdx st;
    make_stencil(st, nd, a);
    double g[3] = {0.0, 0.0, 0.0};
    for_dirs<0, LBMK_Q>([&](auto dd) {
        constexpr int I = decltype(dd)::value;
        if constexpr (I != REST) {
            const double t = Tr[nb_of<I>(st, a)];
            if (CX(I)) g[0] = fma(WI(I) * CX(I), t, g[0]);
            if (CY(I)) g[1] = fma(WI(I) * CY(I), t, g[1]);
            if (CZ(I)) g[2] = fma(WI(I) * CZ(I), t, g[2]);
        }
    });
    const double T = Tr[n];
    double Cp = 0.0;
#pragma unroll
    for (int s = 0; s < M; ++s) Cp = fma((double)R[(size_t)(rr.y + s) * N + n], cp_spec(mc, s, T), Cp);
    const double lam = (1.0 / (double)R[(size_t)rr.om1 * N + n] - 0.5) * (double)R[(size_t)rr.p * N + n] * Cp;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        scr[(size_t)d * N + n] = 3.0 * g[d];
        scr[(size_t)(3 + d) * N + n] = lam * 3.0 * g[d];
    }
}

template <int M>
__global__ void __launch_bounds__(LBMK_HRR_THREADS) k_flame2(StepArgs a, const double *scr, double *Sd, double *Sa)
{
    const MechConst &mc = c_mech[a.slot];
    Node nd;
    if (!node_of(nd, a)) return;
    const size_t N = a.N;
    const int n = nd.n;
    const RecRows rr = rec_rows(M);
    const Real *R = rec(a);
    StencilIdx st;
    make_stencil(st, nd, a);
    double div = 0.0;
    for_dirs<0, LBMK_Q>([&](auto dd) {
        constexpr int I = decltype(dd)::value;
        if constexpr (I != REST) {
            const size_t nb = nb_of<I>(st, a);
            if (CX(I)) div = fma(WI(I) * CX(I), scr[(size_t)3 * N + nb], div);
            if (CY(I)) div = fma(WI(I) * CY(I), scr[(size_t)4 * N + nb], div);
            if (CZ(I)) div = fma(WI(I) * CZ(I), scr[(size_t)5 * N + nb], div);
        }
    });
    div *= 3.0;
    const double T = a.macro[(size_t)DR_T * N + n];
    const double rho = (double)R[(size_t)rr.rho * N + n];
    double rho_a[M], Y[M], fl[3] = {0.0, 0.0, 0.0}, Cp = 0.0;
#pragma unroll
    for (int s = 0; s < M; ++s) {
        Y[s] = (double)R[(size_t)(rr.y + s) * N + n];
        rho_a[s] = rho * Y[s];
        const double cpy = cp_spec(mc, s, T) * Y[s];
        Cp += cpy;
#pragma unroll
        for (int d = 0; d < 3; ++d) fl[d] = fma(cpy, (double)R[(size_t)(rr.du + 3 * s + d) * N + n], fl[d]);
    }
    double dT, drho[M];
    const double hdot = hrr_node<M, false>(mc, T, rho_a, &dT, drho, nullptr, 0);
    const double g[3] = {scr[n], scr[N + n], scr[2 * N + n]};
    const double gn = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    if (gn == 0.0) {
        Sd[n] = Sa[n] = 0.0;
        return;
    }
    const double num = hdot + div - rho * (fl[0] * g[0] + fl[1] * g[1] + fl[2] * g[2]);
    const double sd = num / (rho * Cp * gn);
    double un = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) un -= (double)R[(size_t)(rr.u + d) * N + n] * g[d];
    Sd[n] = sd;
    Sa[n] = sd + un / gn;
}

template <int M>
int run_flame_speeds(const StepArgs &a, double *scr, double *Sd, double *Sa)
{
    int e = 0;
    if (a.bc_x == 1) e = launch_one<M>(a, LBMK_K_GHOST);
    if (!e) e = launch_one<M>(a, LBMK_K_PRE);
    if (e) return e;
    k_flame1<M><<<grid_for(a.N), LBMK_BLOCK, 0, a.stream>>>(a, scr);
    k_flame2<M><<<grid_for(a.N, LBMK_HRR_THREADS), LBMK_HRR_THREADS, 0, a.stream>>>(a, scr, Sd, Sa);
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------
// Means along the isoline T = T_iso in the plane z = 0 (Eq. (rmean)):
// marching squares, one thread per cell (x, y)..(x+1, y+1) of the periodic
// x-y lattice: crossings where T - T_iso changes sign (T >= T_iso counts as
// above) at the linear interpolation point along the cell edge, with the K
// fields interpolated alike; two crossings make one straight segment, four
// are split by the mean of the corners; each segment adds its length and
// its length times the mean of its ends' distance from (cx, cy) and field
// values.  Per-block sums in a fixed order: partial [blocks][2 + K].
// ---------------------------------------------------------------------
#define LBMK_ISO_MAXK 8
__global__ void __launch_bounds__(LBMK_HRR_THREADS) k_isoline(int nx, int ny, int N, const double *T, double T_iso,
                                                               double cx, double cy, int K, const double *fields,
                                                               double *partial)
{
    __shared__ double sh[(2 + LBMK_ISO_MAXK) * LBMK_HRR_THREADS];
    const int t = threadIdx.x, W = 2 + K;
    double acc[2 + LBMK_ISO_MAXK];
    for (int k = 0; k < W; ++k) acc[k] = 0.0;
    const int cell = blockIdx.x * LBMK_HRR_THREADS + t;
    if (cell < nx * ny) {
        const int x = cell % nx, y = cell / nx;
        const int ox[4] = {0, 1, 1, 0}, oy[4] = {0, 0, 1, 1};
        int idx[4];
        double v[4];
        for (int c = 0; c < 4; ++c) {
            idx[c] = (x + ox[c]) % nx + nx * ((y + oy[c]) % ny);
            v[c] = T[idx[c]];
        }
        double px[4], py[4], pf[4][LBMK_ISO_MAXK];
        int ne = 0;
        for (int e = 0; e < 4; ++e) {
            const int aa = e, bb = (e + 1) % 4;
            if ((v[aa] >= T_iso) == (v[bb] >= T_iso)) continue;
            const double f = (T_iso - v[aa]) / (v[bb] - v[aa]);
            px[ne] = x + ox[aa] + f * (ox[bb] - ox[aa]);
            py[ne] = y + oy[aa] + f * (oy[bb] - oy[aa]);
            for (int k = 0; k < K; ++k) {
                const double fa = fields[(size_t)k * N + idx[aa]], fb = fields[(size_t)k * N + idx[bb]];
                pf[ne][k] = fa + f * (fb - fa);
            }
            ++ne;
        }
        int pr[2][2] = {{0, 1}, {2, 3}}, np = ne == 2 ? 1 : (ne == 4 ? 2 : 0);
        if (ne == 4) {
            const double vc = 0.25 * (v[0] + v[1] + v[2] + v[3]);
            if ((vc >= T_iso) != (v[0] >= T_iso)) {       // corners 0 and 2 cut off
                pr[0][0] = 3; pr[0][1] = 0; pr[1][0] = 1; pr[1][1] = 2;
            }
        }
        for (int q = 0; q < np; ++q) {
            const int i = pr[q][0], j = pr[q][1];
            const double L = sqrt((px[i] - px[j]) * (px[i] - px[j]) + (py[i] - py[j]) * (py[i] - py[j]));
            const double Ri = sqrt((px[i] - cx) * (px[i] - cx) + (py[i] - cy) * (py[i] - cy));
            const double Rj = sqrt((px[j] - cx) * (px[j] - cx) + (py[j] - cy) * (py[j] - cy));
            acc[0] += L;
            acc[1] += L * 0.5 * (Ri + Rj);
            for (int k = 0; k < K; ++k) acc[2 + k] += L * 0.5 * (pf[i][k] + pf[j][k]);
        }
    }
    for (int k = 0; k < W; ++k) sh[k * LBMK_HRR_THREADS + t] = acc[k];
    __syncthreads();
    for (int h = LBMK_HRR_THREADS / 2; h > 0; h >>= 1) {
        if (t < h)
            for (int k = 0; k < W; ++k) sh[k * LBMK_HRR_THREADS + t] += sh[k * LBMK_HRR_THREADS + t + h];
        __syncthreads();
    }
    if (t == 0)
        for (int k = 0; k < W; ++k) partial[(size_t)blockIdx.x * W + k] = sh[k * LBMK_HRR_THREADS];
}

}  // namespace

#define LBMK_DISPATCH(M_, CALL)                     \
    switch (M_) {                                   \
    case 2: return CALL(2);                         \
    case 3: return CALL(3);                         \
    case 9: return CALL(9);                         \
    default: return (int)cudaErrorInvalidValue;     \
    }
