// Per-face GP-WENO evaluation on the device (sm_103a).
//
// One call computes, for one face between stencil cells R and R+1 of a
// (2R+2)-cell stencil along the face normal:
//   - the Roe average of the two cells sharing the face and the left/right
//     eigenvectors of the primitive-variable system there (characteristic
//     variables of V = (rho, u, p), Section 6 of the paper);
//   - the projection of every stencil cell's primitive variables on each
//     characteristic field;
//   - per field, the GP-WENO left state (x* = x_i + dx/2 from the stencil of
//     cell i) and right state (x* = x_{i+1} - dx/2 from the stencil of cell
//     i+1): candidate predictions q^m = w_m . f_m (Eq. candidate_interp),
//     smoothness indicators beta = sum_h (P_h . f_m)^2 (Eq. beta-eigen, the
//     R+2 windows shared by both sides), nonlinear weights (Eq. weights) and
//     their combination (Eq. weight_sum);
//   - back-projection to the Riemann states U^L, U^R and the face flux of
//     Eq. riemann_prob: local Lax-Friedrichs, F = (F(U^L)+F(U^R))/2 -
//     alpha (U^R-U^L)/2 with alpha = max(|u_n|+c) over both states, or HLLC
//     (the paper's default solver, Section 7) with Einfeldt wave speeds.
// Stencil values arrive conserved and "normal-first": (rho, m_normal, m_tangential..., E).
//
// Nonlinear weights follow Eq. weights literally, omega_m ~ gamma_m / (eps + beta_m)^p,
// with one reciprocal per smoothness window shared by both sides of the face.
// In FP32 eps + beta is kept >= 1e-18 (eps rescaled out of the FP32 denormal
// range: (1e-36)^-2 would overflow); this changes omega only where every
// affected window holds data below ~1e-9, i.e. below FP32 resolution of the
// state.  FP64 uses eps = 1e-36 exactly.
#pragma once
#include <type_traits>
#include <cuda_runtime.h>

namespace gpweno {

template <typename T>
struct Num;

// FP32: single-instruction approximations (PTX rcp/rsqrt/sqrt .approx.ftz,
// about 1 ulp), enough for an FP32 path whose error budget is set by the
// stored FP32 state.
template <>
struct Num<float> {
    static __device__ __forceinline__ float rcp(float x)
    {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
    static __device__ __forceinline__ float rsqrt(float x)
    {
        float r;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
    static __device__ __forceinline__ float sqrt(float x)
    {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
    static __device__ __forceinline__ float fabs(float x) { return fabsf(x); }
    static __device__ __forceinline__ float fmax(float a, float b) { return fmaxf(a, b); }
    static __device__ __forceinline__ float fmin(float a, float b) { return fminf(a, b); }
    static __device__ __forceinline__ float rcp_ieee(float x) { return rcp(x); }
    static __device__ __forceinline__ float sqrt_ieee(float x) { return sqrt(x); }
    static __device__ __forceinline__ float pmax(float a, float b) { return fmaxf(a, b); }
    static __device__ __forceinline__ bool positive(float a) { return a > 0.0f; }
    // lower bound of eps + beta in FP32, so that (eps + beta)^-2 stays within range
    static constexpr float kEpsFloor = 1e-18f;
    static __device__ __forceinline__ float floored(float eps_beta) { return fmaxf(eps_beta, kEpsFloor); }
    // uncontracted multiply / add (never fused into an FMA, so every kernel rounds alike)
    static __device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
};

// FP64 runs on two lanes per SM (one sixty-fourth of the FP32 rate), so a kernel's time is its
// count of FP64 instructions.  Reciprocal and reciprocal square root start from the 20-bit
// hardware approximations on the high word (PTX rcp/rsqrt.approx.ftz.f64, special-function unit)
// and take one third-order step of the binomial series (Householder's method of order two):
//   1/a       = x / (1 - e) = x (1 + e + e^2 + ...),             e = 1 - a x,    |e| <= ~2^-19
//   a^(-1/2)  = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + ...),  e = 1 - a y^2
// with remainders below 2^-55: results within one unit in the last place, in 3 and 5 FP64
// instructions (the square root in 5) in place of an IEEE division or square root plus division.  Order tests and maxima
// run on the bit patterns in the integer units.  Measured per RK3 step: 512^2 R = 2 3629 -> 3086 us,
// 128^2 R = 3 3042 -> 2748 us; one 3D right-hand side of 70x61x45 2870 -> 2421 us.  Arguments are normal positive numbers
// (eps + beta, densities, sums of weights); zero, infinity or NaN give NaN, which the
// non-physical checks report.
template <>
struct Num<double> {
    static __device__ __forceinline__ double rcp(double a)
    {
        double x;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(a));
        const double e = fma(-a, x, 1.0);
        return fma(x, fma(e, e, e), x);
    }
    static __device__ __forceinline__ double rsqrt(double a)
    {
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
        const double e = fma(-(a * y), y, 1.0);
        return fma(y * e, fma(0.375, e, 0.5), y);
    }
    // Two Newton steps s + (a - s^2) y/2 from s = a y with exact residuals (relative error 2^-20 of s, 2^-39, then the last
    // rounding): 0.51 units in the last place in five instructions, where a times rsqrt(a) takes six, rounds twice more
    // and is up to 1.7 off.  y/2 is an integer subtraction in y's exponent.
    static __device__ __forceinline__ double sqrt(double a)
    {
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
        const double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));
        double s = __dmul_rn(a, y);
        s = fma(fma(-s, s, a), h, s);
        return fma(fma(-s, s, a), h, s);
    }
    // IEEE forms, zero and infinity included: once per cell, in the CFL rates
    static __device__ __forceinline__ double rcp_ieee(double x) { return 1.0 / x; }
    static __device__ __forceinline__ double sqrt_ieee(double x) { return ::sqrt(x); }
    static __device__ __forceinline__ double fabs(double x) { return ::fabs(x); }
    static __device__ __forceinline__ double fmax(double a, double b) { return ::fmax(a, b); }
    // maximum where at least one argument is >= 0, by the order of the bit patterns
    static __device__ __forceinline__ double pmax(double a, double b)
    {
        return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
    }
    // a > 0, by the bit pattern (false for NaN)
    static __device__ __forceinline__ bool positive(double a)
    {
        const long long i = __double_as_longlong(a);
        return i > 0 && i <= 0x7ff0000000000000LL;
    }
    static __device__ __forceinline__ double fmin(double a, double b) { return ::fmin(a, b); }
    // FP64 keeps eps as given (eps > 0)
    static constexpr double kEpsFloor = 0.0;
    static __device__ __forceinline__ double floored(double eps_beta) { return eps_beta; }
    static __device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
};

// Smallest of a and b, NaN if either is one.
__device__ __forceinline__ float min_nan(float a, float b)
{
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float min_nan(float a, float b, float c)
{
    float r;
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Whether all values that have to be positive were.  FP32 keeps the smallest of them (one three-input
// minimum for two values, NaN sticks) instead of a comparison each: six values per face cost three
// instructions, 4096^2 step 2460 -> 2400 us without the checks' share.  FP64 tests the bit patterns, in the
// integer units.
template <typename T>
struct Physical;
template <>
struct Physical<float> {
    float least = 1.0f;
    __device__ __forceinline__ void need(float a) { least = min_nan(least, a); }
    __device__ __forceinline__ void need(float a, float b) { least = min_nan(least, a, b); }
    __device__ __forceinline__ bool good() const { return least > 0.0f; }
};
template <>
struct Physical<double> {
    bool ok = true;
    __device__ __forceinline__ void need(double a) { ok = ok && Num<double>::positive(a); }
    __device__ __forceinline__ void need(double a, double b)
    {
        need(a);
        need(b);
    }
    __device__ __forceinline__ bool good() const { return ok; }
};

// Scheme variants chosen at compile time: bit 0 the non-zero-mean smoothness
// indicators, bit 1 the FD-Flux form, bit 2 GP-AO; bit 3 is not a scheme change
// but a grid with an external (halo) side, whose loaders read ghost layers from
// halo buffers -- a separate instantiation so that the loaders of the others stay
// as they are.
// Bit 4 (FP32): HLL and HLLC face fluxes; kernels without it are compiled for the local Lax-Friedrichs
// flux alone (2 % per step at 1024^2, 3 % in batches, 3-4 % in the GP-AO kernels).  FP64 kernels hold all three.
constexpr int kVarMean = 1, kVarFdFlux = 2, kVarAo = 4, kVarSlab = 8, kVarFlux = 16;
// Bit 5 (FP32): smoothness indicators in their own scale for plans whose weights leave the FP32 range in the one
// that the other kernels take (kUnitDifference, unit_scale_fits): sigma beyond about 5 (R = 2) and 6 dx (R = 3).
constexpr int kVarRange = 32;

// Whether the smoothness indicators are divided by the square of the last form's coefficient a (beta_weight), which
// saves an instruction per window: FP32 step of 4096^2 R = 2 2288 -> 2220 us, of 512^3 R = 3 50.7 -> 49.8 ms, HLLC R = 3
// 397 -> 387 us; none at R = 1 (777 x 613 25.3 us both ways).  The floor of eps + beta is divided alike (a = 1.6 at R = 2,
// 1.1 at R = 3 for sigma = 3 dx, growing with sigma), so (eps + beta)^-p grows by a^2p.  FP32 keeps the indicators'
// own scale where that leaves the range: in the kVarRange kernels; at R = 1 (a = 3 already); and
// with the centre's mean, whose weighted sums hold predictions of any size also where beta is at its floor.
template <typename T, int R, int VAR>
constexpr bool kUnitDifference = sizeof(T) == 8 || (R > 1 && (VAR & (kVarRange | kVarMean)) == 0);

// Weight tables of one plan in the arithmetic type.  Passed by value as a
// kernel parameter so every (warp-uniform) table read is a constant-bank
// operand.
//
// Window k (k = 0 .. R+1) is cells s-R+k .. s+k of the face's stencil.  The left state's sub-stencil
// k and the right state's sub-stencil k-1 are the same cells predicted at the same point, so one
// set of R+2 windows carries both sides' candidates as well as their smoothness indicators.
template <typename T, int R>
struct FaceTables {
    T w[R + 2][R + 1];    // candidate weights of window k at the face
    T s1[R + 2];          // sum_j w[k][j] - 1
    T gl[R + 1];          // linear weights of the left state (windows 0..R) over that of window kUnitL
    T gr[R + 1];          // linear weights of the right state (windows 1..R+1) over that of window kUnitR
    // smoothness factor of K_m(sigma), K_m^-1 = sum of squares of five forms of the window's sums
    // f_j + f_{R-j} and differences f_{R-j} - f_j (see window_factors): outer sum (A, B with the inner one or the
    // middle cell), inner (D), differences (kb the outer, kd the inner one), outer difference (a); divided by a where
    // the kernel takes it for 1, see kUnitDifference
    T A, B, D, a, kb, kd;
    T pA, pD;             // row sums of the two symmetric forms
    T eps;                // WENO epsilon in the same scale (FP32: at least the floor of Num<T>)
    T gamma;              // ratio of specific heats
    T gm1, igm1, hgm1;    // gamma - 1, its inverse and half of it
    int p;                // WENO power, 1 or 2
    int flux;             // face flux: 0 local Lax-Friedrichs, 1 HLLC, 2 HLL
};

// Window whose linear weight is the unit of each side's weights: the one that is never small
// against the others for any l/dx >= 1 (ratio at most 3.7, with FD-Flux 4.2), so the scaled sums stay in range.
template <int R>
constexpr int kUnitL = R == 2 ? 2 : 1;
template <int R>
constexpr int kUnitR = R + 1 - kUnitL<R>;

// Primitive reference state of the "cell-relative" evaluation (normal-first order).
template <typename T, int NC>
struct PrimRef {
    T rho;            // density of cell s
    T u[NC - 2];      // velocity of cell s
    T p;              // pressure of cell s
    T hp;             // E + p of cell s
    T mn;             // normal momentum rho u_n of cell s (the stored value)
};

// For a primitive perturbation w = V - V_s (V = (rho, u_n, u_t..., p)):
//   cw = U(V) - U(V_s)  (conservative perturbation)
//   G  = F(V) - F(V_s)  (normal-flux perturbation)
// written so that large reference quantities only multiply small ones:
//   g_a = rho u_a - rho_s u_s,a = rho w_a + u_s,a w_rho,  rho = rho_s + w_rho,  u = u_s + w_u
//   k   = rho|u|^2 - rho_s|u_s|^2 = sum_a (g_a u_a + rho_s u_s,a w_a)
//   E'  = w_p/(gamma-1) + k/2
//   G   = (g_n,  g_n u_n + m_s,n w_n + w_p,  g_n u_t + m_s,n w_t,  w_n (E+p)_s + u_n (E' + w_p)).
// Requires rho > 0 and p > 0 in `ph`; un and cs are the normal velocity and
// the sound speed of the full state.
template <typename T, int NC>
__device__ __forceinline__ void prim_pert(const PrimRef<T, NC> &r, const T (&w)[NC], T gam, T igm1, T (&G)[NC],
                                          T (&cw)[NC], T &un, T &cs, Physical<T> &ph)
{
    constexpr int NV = NC - 2, E = NC - 1;
    const T rho = r.rho + w[0];
    T u[NV], g[NV];
    T k = T(0);
#pragma unroll
    for (int a = 0; a < NV; ++a) {
        u[a] = r.u[a] + w[1 + a];
        g[a] = fma(rho, w[1 + a], r.u[a] * w[0]);
        k = fma(g[a], u[a], fma(r.rho * r.u[a], w[1 + a], k));
    }
    const T ep = fma(w[E], igm1, T(0.5) * k);
    cw[0] = w[0];
#pragma unroll
    for (int a = 0; a < NV; ++a) cw[1 + a] = g[a];
    cw[E] = ep;
    G[0] = g[0];
    G[1] = fma(g[0], u[0], fma(r.mn, w[1], w[E]));
#pragma unroll
    for (int a = 1; a < NV; ++a) G[1 + a] = fma(g[0], u[a], r.mn * w[1 + a]);
    G[E] = fma(w[1], r.hp, u[0] * (ep + w[E]));
    const T pr = r.p + w[E];
    un = u[0];
    cs = Num<T>::sqrt(Num<T>::pmax(gam * pr * Num<T>::rcp(rho), T(1e-30)));
    ph.need(rho, pr);
}

// Arithmetic of one characteristic field (T) or of two at once (float2: packed fma/add/mul .f32x2
// of sm_100 and later, each lane rounded as the scalar operation).
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vfma(float a, float2 b, float2 c) { return __ffma2_rn(f2(a), b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.0f), a); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float a, float2 b) { return __fmul2_rn(f2(a), b); }
// In FP64 the product is kept out of later sums (no FMA contraction), so that the 1D kernel that passes
// states between warps rounds as those that keep them in registers.
__device__ __forceinline__ float vmul_keep(float a, float b) { return a * b; }
__device__ __forceinline__ double vmul_keep(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float2 vmul_keep(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float vrcp(float a) { return Num<float>::rcp(a); }
__device__ __forceinline__ double vrcp(double a) { return Num<double>::rcp(a); }
__device__ __forceinline__ float2 vrcp(float2 a) { return make_float2(Num<float>::rcp(a.x), Num<float>::rcp(a.y)); }
template <typename V>
__device__ __forceinline__ V vset(double x) { return V(x); }
template <>
__device__ __forceinline__ float2 vset<float2>(double x) { return f2((float)x); }
__device__ __forceinline__ float vcast(float x, float) { return x; }
__device__ __forceinline__ double vcast(double x, double) { return x; }
__device__ __forceinline__ float2 vcast(float x, float2) { return f2(x); }

// Roe average of the two cells sharing a face (normal-first conserved uL =
// cell s, uR = cell s+1), the primitive eigen-system at it, and cell s as the
// primitive reference of the cell-relative evaluation:
//   L_V rows: (0, -an, 0, ap), (1, 0, 0, -ie), e_t, (0, an, 0, ap)
//   R_V cols: (1, -cr, 0, c^2), (1, 0, 0, 0),   e_t, (1, cr, 0, c^2)
// with an = rbar/(2c), ap = 1/(2c^2), ie = 1/c^2, cr = c/rbar, rbar = sqrt(rho_L rho_R).
// With the weight th = sqrt(rho_R) / (sqrt(rho_L) + sqrt(rho_R)) of cell s+1 the Roe velocity is
// u_s + th du and the Roe enthalpy's sound speed is
//   c^2 = c_L^2 + th (c_R^2 - c_L^2) + (gamma-1)/2 th (1-th) |du|^2,
// which needs no enthalpy and only the difference du.  A density <= 0 of either cell makes c^2 NaN or
// -infinity (its reciprocal square root is NaN or infinite), so c^2 > 0 checks the densities too.
template <typename T, int NC>
struct FaceRoe {
    static constexpr int NV = NC - 2, E = NC - 1;
    T gm1;
    T th;             // Roe weight of cell s+1
    T c2, c, ic;      // Roe sound speed squared, sound speed, 1/c
    T rbar, irb;      // sqrt(rho_L rho_R) and its inverse
    T an, ie, ap, cr;
    PrimRef<T, NC> ref;
    T Vs[NC];         // primitive state of cell s
    T dVn[NC];        // V_{s+1} - V_s

    // row kk of L_V applied to a primitive vector
    __device__ __forceinline__ T lrow(int kk, const T *v) const
    {
        if (kk == 0) return fma(ap, v[E], -an * v[1]);
        if (kk == E) return fma(ap, v[E], an * v[1]);
        if (kk == 1) return fma(-ie, v[E], v[0]);
        return v[kk];   // shear: tangential velocity
    }

    // Roe velocity
    __device__ __forceinline__ T vel(int a) const { return fma(th, dVn[1 + a], ref.u[a]); }

    // back-projection: the left and right primitive states relative to cell s
    __device__ __forceinline__ void left_state(const T (&dq)[NC], T (&w)[NC]) const
    {
        w[0] = dq[0] + dq[1] + dq[E];
        w[1] = vmul_keep(cr, dq[E] - dq[0]);
#pragma unroll
        for (int a = 2; a < E; ++a) w[a] = dq[a];
        w[E] = vmul_keep(c2, dq[0] + dq[E]);
    }
    __device__ __forceinline__ void right_state(const T (&dq)[NC], T (&w)[NC]) const
    {
        w[0] = dVn[0] + (dq[0] + dq[1] + dq[E]);
        w[1] = fma(cr, dq[E] - dq[0], dVn[1]);
#pragma unroll
        for (int a = 2; a < E; ++a) w[a] = dVn[a] + dq[a];
        w[E] = fma(c2, dq[0] + dq[E], dVn[E]);
    }

    // B = F(U_{s+1}) - F(U_s) from the exact conserved difference and the primitive one:
    // (dm_n, u'_n dm_n + m_n du_n + dp, u'_t dm_n + m_n du_t, hp du_n + u'_n (dE + dp)), u' = u_{s+1}
    __device__ __forceinline__ void flux_difference(const T (&us)[NC], const T (&ur)[NC], T (&B)[NC]) const
    {
        const T dm = ur[1] - us[1], un = ref.u[0] + dVn[1];
        B[0] = dm;
        B[1] = fma(dm, un, fma(ref.mn, dVn[1], dVn[E]));
#pragma unroll
        for (int a = 2; a < E; ++a) B[a] = fma(dm, ref.u[a - 1] + dVn[a], ref.mn * dVn[a]);
        B[E] = fma(dVn[1], ref.hp, un * ((ur[E] - us[E]) + dVn[E]));
    }

    // V_j - V_s from the exact conserved difference U_j - U_s by perturbation algebra (irj = 1/rho_j)
    __device__ __forceinline__ void prim_diff(const T (&uj)[NC], const T (&us)[NC], T irj, T (&dV)[NC]) const
    {
        T dU[NC];
#pragma unroll
        for (int a = 0; a < NC; ++a) dU[a] = uj[a] - us[a];
        T k = T(0);
        dV[0] = dU[0];
#pragma unroll
        for (int a = 0; a < NV; ++a) {
            const T du = fma(-ref.u[a], dU[0], dU[1 + a]) * irj;
            dV[1 + a] = du;
            k = fma(uj[1 + a], du, fma(ref.u[a], dU[1 + a], k));
        }
        dV[E] = gm1 * fma(T(-0.5), k, dU[E]);
    }
    __device__ __forceinline__ void prim_diff(const T (&uj)[NC], const T (&us)[NC], T (&dV)[NC]) const
    {
        prim_diff(uj, us, Num<T>::rcp(uj[0]), dV);
    }
};

// What the Roe average takes from each cell alone, for kernels that form it once per cell and not per face.
template <typename T, int NC>
struct CellPart {
    T rs, ir, s;                   // rho^-1/2, 1/rho, rho^1/2
    T u[NC - 2], p, hp, c2;        // used of cell s only
};

// PARTS: the cells' parts are given, otherwise formed here (in this order, which the compiler's register
// allocation in the 3D kernels answers to: 2 % at 512^3).
template <typename T, int NC, bool PARTS = false, typename Tables>
__device__ __forceinline__ FaceRoe<T, NC> face_roe(const T (&uL)[NC], const T (&uR)[NC], const Tables &tb,
                                                   const CellPart<T, NC> &L = {}, const CellPart<T, NC> &R = {})
{
    constexpr int NV = NC - 2, E = NC - 1;
    FaceRoe<T, NC> f;
    f.gm1 = tb.gm1;
    const T rL = uL[0], rR = uR[0];
    const T rsL = PARTS ? L.rs : Num<T>::rsqrt(rL), rsR = PARTS ? R.rs : Num<T>::rsqrt(rR);
    const T irL = PARTS ? L.ir : rsL * rsL, irR = PARTS ? R.ir : rsR * rsR;
    f.ref.rho = rL;
    T mu = T(0);
#pragma unroll
    for (int a = 0; a < NV; ++a) {
        f.ref.u[a] = PARTS ? L.u[a] : vmul_keep(uL[1 + a], irL);
        mu = fma(uL[1 + a], f.ref.u[a], mu);
    }
    f.ref.p = PARTS ? L.p : vmul_keep(f.gm1, fma(T(-0.5), mu, uL[E]));
    f.ref.hp = PARTS ? L.hp : uL[E] + f.ref.p;
    f.ref.mn = uL[1];
    f.Vs[0] = rL;
#pragma unroll
    for (int a = 0; a < NV; ++a) f.Vs[1 + a] = f.ref.u[a];
    f.Vs[E] = f.ref.p;
    f.prim_diff(uR, uL, irR, f.dVn);
    const T sL = PARTS ? L.s : vmul_keep(rL, rsL), sR = PARTS ? R.s : vmul_keep(rR, rsR);   // sqrt(rho)
    f.th = sR * Num<T>::rcp(sL + sR);
    T du2 = T(0);
#pragma unroll
    for (int a = 0; a < NV; ++a) du2 = fma(f.dVn[1 + a], f.dVn[1 + a], du2);
    const T cL2 = PARTS ? L.c2 : vmul_keep(tb.gamma * irL, f.ref.p), cR2 = tb.gamma * irR * (f.ref.p + f.dVn[E]);
    f.c2 = fma(tb.hgm1 * fma(-f.th, f.th, f.th), du2, fma(f.th, cR2 - cL2, cL2));
    f.ic = Num<T>::rsqrt(Num<T>::pmax(f.c2, T(1e-30)));
    f.c = f.c2 * f.ic;
    f.rbar = sL * sR;
    f.irb = rsL * rsR;
    f.an = T(0.5) * f.rbar * f.ic;
    f.ie = f.ic * f.ic;
    f.ap = T(0.5) * f.ie;
    f.cr = f.c * f.irb;
    return f;
}

// The part of cell U, with face_roe's roundings
template <typename T, int NC, typename Tables>
__device__ __forceinline__ CellPart<T, NC> cell_part(const T (&U)[NC], const Tables &tb)
{
    constexpr int NV = NC - 2, E = NC - 1;
    CellPart<T, NC> c;
    c.rs = Num<T>::rsqrt(U[0]);
    c.ir = c.rs * c.rs;
    c.s = vmul_keep(U[0], c.rs);
    T mu = T(0);
#pragma unroll
    for (int a = 0; a < NV; ++a) {
        c.u[a] = vmul_keep(U[1 + a], c.ir);
        mu = fma(U[1 + a], c.u[a], mu);
    }
    c.p = vmul_keep(tb.gm1, fma(T(-0.5), mu, U[E]));
    c.hp = U[E] + c.p;
    c.c2 = vmul_keep(tb.gamma * c.ir, c.p);
    return c;
}

// (eps + beta)^-p of one smoothness window: beta = f^T K_m(sigma)^-1 f (Eq. beta-eigen, in another
// orthogonal basis) over the window f[w..w+R] of data f_j - shift = d_j + (f_c - shift), with
// d_R = 0 (relative to the face's cell s).  pA, pD = (f_c - shift) times the row sums of the two
// symmetric forms, supplied by the caller (the differences' row sums vanish).  Triangular forms
// (window_factors) save 1 (R = 2) and 2 (R = 3) of 10 and 16 instructions per window against the eigenvector
// rows, and UNIT one more: the scale in which the coefficient a of the last form is 1 (kUnitDifference).
template <typename T, int R, bool UNIT, typename V, int NS>
__device__ __forceinline__ V beta_weight(const FaceTables<T, R> &tb, const V (&d)[NS], int w, V pA, V pD)
{
    // sum and difference of the window's cells j and R-j; `flip` picks the sign of all differences of a
    // window (their squares are used) so that a term with d_R = 0 is a plain copy
    const bool flip = w + R == R || (R == 3 && w + 2 == R);
    auto sum = [&](int j) {
        const int lo = w + j, hi = w + R - j;
        return lo == R ? d[hi] : (hi == R ? d[lo] : vadd(d[lo], d[hi]));
    };
    auto diff = [&](int j) {
        const int lo = flip ? w + R - j : w + j, hi = flip ? w + j : w + R - j;
        return lo == R ? d[hi] : vsub(d[hi], d[lo]);
    };
    V beta = vcast(tb.eps, V());   // (eps + beta), accumulated from eps
    V s = vfma(tb.A, sum(0), pA);
    const V t = diff(0), k = UNIT ? t : vmul(tb.a, t);
    if constexpr (R == 2) {
        V m = pD;
        if (w + 1 != R) {
            s = vfma(tb.B, d[w + 1], s);
            m = vfma(tb.D, d[w + 1], m);
        }
        beta = vfma(m, m, beta);
    }
    if constexpr (R == 3) {
        const V si = sum(1), ki = diff(1);
        s = vfma(tb.B, si, s);
        // t is a plain copy in the two windows that end at cell s, so its product starts n (512^3 50.0 -> 49.8 ms)
        const V m = vfma(tb.D, si, pD), n = vfma(tb.kd, ki, vmul(tb.kb, t));
        beta = vfma(m, m, beta);
        beta = vfma(n, n, beta);
    }
    beta = vfma(k, k, beta);
    beta = vfma(s, s, beta);
    const V x = vrcp(beta);
    return tb.p == 2 ? vmul(x, x) : x;
}

// Left and right GP-WENO states of a face in one characteristic field (or two, V = float2) from the
// data d_j relative to cell s (d_R = 0) and the value fc of cell s:
//   qL = q_L - f_s,  qR = q_R - f_{s+1}.
// Window k's candidate relative to cell s is q_k = sum_j w_kj d_{k+j} + fc (sum_j w_kj - 1), shared by
// both sides, and omega_m ~ gamma_m x_k with x_k = (eps + beta_k)^-p (Eq. weights); sum_m omega_m = 1
// is used exactly.  With the zero mean x_k and x_k q_k are shared too.  MEAN: the left side's windows
// shift by its centre, cell s (no shift), the right side's by cell s+1 (shift d_{R+1}).
template <typename T, int R, bool MEAN, bool UNIT, typename V, int NS>
__device__ __forceinline__ void weno_states(const FaceTables<T, R> &tb, const V (&d)[NS], V fc, V &qL, V &qR)
{
    constexpr int UL = kUnitL<R>, UR = kUnitR<R>;
    const V zero = vset<V>(0.0);
    const V lA = MEAN ? zero : vmul(tb.pA, fc), lD = MEAN ? zero : vmul(tb.pD, fc);
    const V rA = MEAN ? vmul(-tb.pA, d[R + 1]) : lA, rD = MEAN ? vmul(-tb.pD, d[R + 1]) : lD;
    V numL, denL, numR, denR;
    // the windows with a unit weight first, so that each side's sums start without a multiply
    auto window = [&](int k, V &xl, V &xr, V &tl, V &tr) {
        V q = vmul(tb.s1[k], fc);
#pragma unroll
        for (int j = 0; j <= R; ++j)
            if (k + j != R) q = vfma(tb.w[k][j], d[k + j], q);
        if (k <= R) {
            xl = beta_weight<T, R, UNIT>(tb, d, k, lA, lD);
            tl = vmul(xl, q);
        }
        if (k > 0) {
            if (MEAN || k > R) {
                xr = beta_weight<T, R, UNIT>(tb, d, k, rA, rD);
                tr = vmul(xr, q);
            } else {
                xr = xl;
                tr = tl;
            }
        }
    };
    V xl, xr, tl, tr;
    window(UL, xl, xr, tl, tr);
    numL = tl;
    denL = xl;
    if constexpr (UR == UL) {
        numR = tr;
        denR = xr;
    } else {
        V yl, yr, ul, ur;
        window(UR, yl, yr, ul, ur);
        numL = vfma(tb.gl[UR], ul, numL);
        denL = vfma(tb.gl[UR], yl, denL);
        numR = vfma(tb.gr[UL - 1], tr, ur);
        denR = vfma(tb.gr[UL - 1], xr, yr);
    }
#pragma unroll
    for (int k = 0; k <= R + 1; ++k) {
        if (k == UL || k == UR) continue;
        window(k, xl, xr, tl, tr);
        if (k <= R) {
            numL = vfma(tb.gl[k], tl, numL);
            denL = vfma(tb.gl[k], xl, denL);
        }
        if (k > 0) {
            numR = vfma(tb.gr[k - 1], tr, numR);
            denR = vfma(tb.gr[k - 1], xr, denR);
        }
    }
    qL = vmul_keep(numL, vrcp(denL));
    qR = vfma(numR, vrcp(denR), vneg(d[R + 1]));
}

// GP-AO tables (Appendix A) on top of the GP-WENO ones: R = 2 serves AO(2,3),
// R = 3 the recursive AO(3,2,3).  Weights of the full stencil S_R (hi), of
// S_{R-1} (lo, R = 3), of the three 3-point stencils of Eq. cweno_stencil, for
// the left (x* = +1/2) and right (x* = -1/2) states, with their sums minus
// one; half-form factors of K_N(sigma) for N = 2R+1, 2R-1, 3; the linear
// weights of Eq. CWENO-lin.
template <typename T, int R>
struct AoFaceTables : FaceTables<T, R> {
    static constexpr int NH = 2 * R + 1, NL = R > 2 ? 2 * R - 1 : 1;
    T whl[NH], whr[NH], shl, shr;
    T wll[NL], wlr[NL], sll, slr;
    T w3l[3][3], w3r[3][3], s3l[3], s3r[3];
    T Phi[NH][(NH + 1) / 2], Psum_hi[NH];
    T Plo[NL][(NL + 1) / 2], Psum_lo[NL];
    T P3[3][2], Psum3[3];
    T eps_ao;               // WENO epsilon (unscaled)
    T g_hi, g_hi1, ig_hi;   // gamma_HI, 1 - gamma_HI, 1 / gamma_HI
    T g3[3];                // gamma_m = ((1-gHI)(1-gLO)/2, (1-gHI) gLO, (1-gHI)(1-gLO)/2)
};

// (eps + beta)^-p with the FP32 floor on eps + beta (as for GP-WENO)
template <typename T>
__device__ __forceinline__ T inv_pow(T eps, T beta, int p)
{
    const T x = Num<T>::rcp(Num<T>::floored(Num<T>::add_rn(eps, beta)));
    return p == 2 ? Num<T>::mul_rn(x, x) : x;
}

// sum_h (P_h . (f - shift))^2 over the N-point window f[w..w+N-1] of data
// f_j = f_c + d_j (d_R = 0), P in half form (rows alternately symmetric and
// skew), pf_h = (f_c - shift) sum_j P_hj supplied by the caller.
template <typename T, int N, int R, int NS>
__device__ __forceinline__ T beta_window(const T (&Ph)[N][(N + 1) / 2], const T (&d)[NS], int w, const T (&pf)[N])
{
    constexpr int HALF = N / 2;
    T ps[HALF], ms[HALF];
#pragma unroll
    for (int j = 0; j < HALF; ++j) {
        const int lo = w + j, hi = w + N - 1 - j;
        ps[j] = lo == R ? d[hi] : (hi == R ? d[lo] : d[lo] + d[hi]);
        ms[j] = lo == R ? -d[hi] : (hi == R ? d[lo] : d[lo] - d[hi]);
    }
    T beta = T(0);
#pragma unroll
    for (int h = 0; h < N; ++h) {
        T dot;
        if (h % 2 == 0) {
            dot = pf[h];
            if (N % 2 == 1 && w + HALF != R) dot = fma(Ph[h][HALF], d[w + HALF], dot);
#pragma unroll
            for (int j = 0; j < HALF; ++j) dot = fma(Ph[h][j], ps[j], dot);
        } else {
            dot = Ph[h][0] * ms[0];
#pragma unroll
            for (int j = 1; j < HALF; ++j) dot = fma(Ph[h][j], ms[j], dot);
        }
        beta = fma(dot, dot, beta);
    }
    return beta;
}

// GP-AO(R,3) of Eq. GP-AO: the high-order prediction qh, with xh = (eps + beta^R)^-p,
// hybridised with the three 3-point predictions q3 (x3 likewise); weights of Eq.
// nonlin-AO with gamma_HI for the high-order stencil and gamma_m for the small ones.
// The combination's coefficients sum to one, so predictions relative to cell s
// combine to the hybrid relative to cell s.
template <typename T, int R>
__device__ __forceinline__ T ao_hybrid(const AoFaceTables<T, R> &ta, T qh, T xh, const T (&q3)[3], const T (&x3)[3])
{
    const T wh = ta.g_hi * xh;
    T w[3], sum = wh;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        w[m] = ta.g3[m] * x3[m];
        sum += w[m];
    }
    const T inv = Num<T>::rcp(sum);
    const T r = wh * inv * ta.ig_hi;   // omega^R / gamma_HI
    T q = r * qh;
#pragma unroll
    for (int m = 0; m < 3; ++m) q = fma(fma(w[m], inv, -r * ta.g3[m]), q3[m], q);
    return q;
}

// GP-AO prediction of one side of the face, relative to cell s, from the
// characteristic data d (relative to cell s, d_R = 0) and the centre value fc:
// left (RIGHT = false) from the stencil d[0..2R] of cell s at x* = +1/2, right
// from d[1..2R+1] of cell s+1 at x* = -1/2.  beta of each stencil is the
// data-fit term (1/2) f^T K_N(sigma)^-1 f of Eq. log-like, on f (zero mean) or
// on f minus the side's centre value (MEAN).  R = 3 adds the recursive
// hybridisation of AO(3,3) and AO(2,3) (Eqs. recursive-weights, AO-recursive).
template <typename T, int R, int NS, bool RIGHT, bool MEAN>
__device__ __forceinline__ T ao_side(const AoFaceTables<T, R> &ta, const T (&d)[NS], T fc)
{
    constexpr int NH = 2 * R + 1, NL = AoFaceTables<T, R>::NL;
    constexpr int o = RIGHT ? 1 : 0;
    const T shift = MEAN ? (RIGHT ? -d[R + 1] : T(0)) : fc;   // pf_h = Psum_h * shift
    T q3[3], x3[3];
    {
        T pf[3];
#pragma unroll
        for (int h = 0; h < 3; ++h) pf[h] = (h % 2 == 0) ? ta.Psum3[h] * shift : T(0);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int w0 = o + R - 2 + m;   // Eq. cweno_stencil: cells c-2..c, c-1..c+1, c..c+2
            T q = (RIGHT ? ta.s3r[m] : ta.s3l[m]) * fc;
#pragma unroll
            for (int j = 0; j < 3; ++j)
                if (w0 + j != R) q = fma(RIGHT ? ta.w3r[m][j] : ta.w3l[m][j], d[w0 + j], q);
            q3[m] = q;
            x3[m] = inv_pow<T>(ta.eps_ao, T(0.5) * beta_window<T, 3, R, NS>(ta.P3, d, w0, pf), ta.p);
        }
    }
    T pfh[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) pfh[h] = (h % 2 == 0) ? ta.Psum_hi[h] * shift : T(0);
    T qh = (RIGHT ? ta.shr : ta.shl) * fc;
#pragma unroll
    for (int j = 0; j < NH; ++j)
        if (o + j != R) qh = fma(RIGHT ? ta.whr[j] : ta.whl[j], d[o + j], qh);
    const T xh = inv_pow<T>(ta.eps_ao, T(0.5) * beta_window<T, NH, R, NS>(ta.Phi, d, o, pfh), ta.p);
    const T q_hi = ao_hybrid<T, R>(ta, qh, xh, q3, x3);
    if constexpr (R == 2) {
        return q_hi;
    } else {
        T pfl[NL];
#pragma unroll
        for (int h = 0; h < NL; ++h) pfl[h] = (h % 2 == 0) ? ta.Psum_lo[h] * shift : T(0);
        T ql = (RIGHT ? ta.slr : ta.sll) * fc;
#pragma unroll
        for (int j = 0; j < NL; ++j)
            if (o + 1 + j != R) ql = fma(RIGHT ? ta.wlr[j] : ta.wll[j], d[o + 1 + j], ql);
        const T xl = inv_pow<T>(ta.eps_ao, T(0.5) * beta_window<T, NL, R, NS>(ta.Plo, d, o + 1, pfl), ta.p);
        const T q_lo = ao_hybrid<T, R>(ta, ql, xl, q3, x3);
        const T vh = ta.g_hi * xh, vl = ta.g_hi1 * xl;
        const T inv = Num<T>::rcp(vh + vl);
        const T rh = vh * inv * ta.ig_hi;   // nu^R' / gamma_HI
        return fma(rh, q_hi, fma(-rh, ta.g_hi1, vl * inv) * q_lo);
    }
}

// Twice the face flux relative to F(U_s) of the two states: w primitive, G flux and c conserved relative to
// cell s, u and a their normal velocities and sound speeds.  LF: local Lax-Friedrichs only.
template <typename T, int NC, bool LF, typename Tables>
__device__ __forceinline__ void face_flux(const FaceRoe<T, NC> &f, const Tables &tb, const T (&wL)[NC],
                                          const T (&wR)[NC], const T (&GL)[NC], const T (&GR)[NC], const T (&cL)[NC],
                                          const T (&cR)[NC], T uL, T uR, T aL, T aR, T (&A)[NC])
{
    constexpr int E = NC - 1;
    const PrimRef<T, NC> &ref = f.ref;
    const T c = f.c;
    if (!LF && tb.flux == 1) {
        // HLLC with Einfeldt speeds from the Roe average.  The contact speed enters only
        // through S* - u_K = (dp - rho_K' (S_K' - u_K') du) / D (K' the other side), formed
        // from the small differences dp = p_R - p_L, du = u_R - u_L, so the star states
        // U*_K - U_K stay accurate increments.
        const T vel0 = f.vel(0);
        const T rhoL = ref.rho + wL[0], rhoR = ref.rho + wR[0];
        const T pLf = ref.p + wL[E], pRf = ref.p + wR[E];
        const T SL = Num<T>::fmin(uL - aL, vel0 - c), SR = Num<T>::fmax(uR + aR, vel0 + c);
        const T mL = rhoL * (SL - uL), mR = rhoR * (SR - uR);
        const T iD = Num<T>::rcp(mL - mR);
        const T dp = wR[E] - wL[E], du = wR[1] - wL[1];
        const T sL = (dp - mR * du) * iD;   // S* - u_L
        const T sR = (dp - mL * du) * iD;   // S* - u_R
        const T Ss = uL + sL;
        const T Es = ref.hp - ref.p;
        auto star = [&](const T (&w)[NC], const T (&cw)[NC], T rho, T pK, T mK, T SK, T sK, T (&dU)[NC]) {
            // U*_K - U_K with chi = rho_K (S_K - u_K) / (S_K - S*), chi - 1 = (S* - u_K) / (S_K - S*)
            const T q = Num<T>::rcp(mK * Num<T>::rcp(rho) - sK);   // 1 / (S_K - S*)
            const T chi1 = sK * q;
            dU[0] = rho * chi1;
            dU[1] = rho * fma(chi1, Ss, sK);
#pragma unroll
            for (int a = 2; a < E; ++a) dU[a] = rho * (ref.u[a - 1] + w[a]) * chi1;
            const T EK = Es + cw[E];
            // chi rho_K (S* - u_K)(S* + p_K / (rho_K (S_K - u_K))), with chi rho_K = m_K q
            dU[E] = fma(chi1, EK, mK * q * sK * (Ss + pK * Num<T>::rcp(mK)));
        };
        T dUL[NC], dUR[NC];
        star(wL, cL, rhoL, pLf, mL, SL, sL, dUL);
        star(wR, cR, rhoR, pRf, mR, SR, sR, dUR);
#pragma unroll
        for (int a = 0; a < NC; ++a) {
            T f;
            if (SL >= T(0)) f = GL[a];
            else if (SR <= T(0)) f = GR[a];
            else if (Ss >= T(0)) f = fma(SL, dUL[a], GL[a]);
            else f = fma(SR, dUR[a], GR[a]);
            A[a] = T(2) * f;
        }
    } else if (!LF && tb.flux == 2) {
        // HLL with the same Einfeldt speeds: F_L if S_L >= 0, F_R if S_R <= 0, else
        // (S_R F_L - S_L F_R + S_L S_R (U_R - U_L)) / (S_R - S_L); relative to F(U_s)
        // the flux terms keep that form with G_K = F_K - F(U_s) and c_K = U_K - U_s.
        const T vel0 = f.vel(0);
        const T SL = Num<T>::fmin(uL - aL, vel0 - c), SR = Num<T>::fmax(uR + aR, vel0 + c);
        const T iS = Num<T>::rcp(SR - SL);
#pragma unroll
        for (int a = 0; a < NC; ++a) {
            T f;
            if (SL >= T(0)) f = GL[a];
            else if (SR <= T(0)) f = GR[a];
            else f = (fma(SR, GL[a], -SL * GR[a]) + SL * SR * (cR[a] - cL[a])) * iS;
            A[a] = T(2) * f;
        }
    } else {
        const T alpha = Num<T>::pmax(Num<T>::fabs(uL) + aL, Num<T>::fabs(uR) + aR);
#pragma unroll
        for (int a = 0; a < NC; ++a) A[a] = fma(-alpha, cR[a] - cL[a], GL[a] + GR[a]);
    }
}

// One face, cell-relative form.  st[0..2R+1] is the normal-first conserved
// stencil; the face s+1/2 lies between st[R] (cell s) and st[R+1] (cell s+1).
// Outputs
//   A = 2 (F_{s+1/2} - F(U_s))      (numerical face flux relative to cell s)
//   M = 2 (F_{s+1/2} - F(U_{s+1}))  (relative to cell s+1)
// so that the flux jump across cell s, F_{s+1/2} - F_{s-1/2} = (A_s - M_{s-1}) / 2,
// is formed from small quantities only (the factor 2 spares the halving of the
// Lax-Friedrichs mean; the divergence's weights take it back).  In real arithmetic this is exactly
// the scheme: characteristic variables of the primitive variables
// V = (rho, u, p) with the eigenvectors of the primitive system at the Roe
// average of cells s, s+1 (Section 6; "FD-Primitive"), GP-WENO states by
// Eqs. candidate_interp, beta-eigen, weights, weight_sum, and the
// Lax-Friedrichs flux.  The rewriting only changes where FP rounding falls:
//   * primitive differences V_j - V_s come from the exact conserved
//     differences U_j - U_s by perturbation algebra, and are projected as
//     d_j = L (V_j - V_s) plus the centre value f_c = L V_s, so
//     q^m = w_m . d_m + f_c sum_j w_mj and P_h . f_m = P_h . d_m + f_c sum_j P_hj;
//   * the left state is V_s + R (q_L - L V_s) and the right state
//     V_{s+1} + R (q_R - L V_{s+1}), using R L = I and sum_m omega_m = 1;
//   * fluxes and conserved states are perturbations about V_s (prim_pert).
// Requires a physical Roe, left, right and neighbour state in `ph`.
// Bound: instruction issue and the FP32 pipe (FP32), the FP64 pipe (FP64), so the count of
// arithmetic instructions.  Sharing the candidates of a window between both sides, triangular
// smoothness forms, the Roe sound speed and the neighbour flux from differences, and doubled fluxes
// measured per step against the form without them: FP32 1024^2 R = 2 232 -> 205 us, 4096^2
// 2848 -> 2460 us, 3D 512^3 R = 3 63.1 -> 53.4 ms; FP64 512^2 R = 2 3086 -> 2702 us.
// LF: local Lax-Friedrichs only (tb.flux is not read).  P5: five fields packed in FP32.
template <typename T, int NC, int R, int VAR, bool LF, bool P5>
__device__ __forceinline__ void face_rel(const T (&st)[2 * R + 2][NC], const FaceTables<T, R> &tb, T (&A)[NC],
                                         T (&M)[NC], Physical<T> &ph)
{
    constexpr int NS = 2 * R + 2;
    constexpr int E = NC - 1;
    constexpr bool MEAN = (VAR & kVarMean) != 0, AO = (VAR & kVarAo) != 0;
    const FaceRoe<T, NC> f = face_roe<T, NC>(st[R], st[R + 1], tb);
    const T igm1 = tb.igm1;
    const PrimRef<T, NC> &ref = f.ref;
    const T(&dn)[NC] = f.dVn;

    // primitive differences V_j - V_s from the exact conserved differences
    T dV[NS][NC];
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        if (j == R || j == R + 1) {
#pragma unroll
            for (int a = 0; a < NC; ++a) dV[j][a] = j == R ? T(0) : dn[a];
            continue;
        }
        f.prim_diff(st[j], st[R], dV[j]);
    }

    T dqL[NC], dqR[NC];
    // FP32 GP-WENO in 1D and 2D: fields in pairs (0,1), (2,3) through packed
    // instructions, an odd last field (1D, 3D) through the scalar loop below.  3D takes the packed
    // form where its kernels have the registers for it (P5, see kPackPlane and kPackZ).
    constexpr bool kPacked = std::is_same<T, float>::value && !AO && (NC <= 4 || P5);
    constexpr int kScalarFrom = kPacked ? (NC / 2) * 2 : 0;
    if constexpr (kPacked) {
#pragma unroll
        for (int k0 = 0; k0 + 1 < NC; k0 += 2) {
            const int k1 = k0 + 1;
            const float2 fc = make_float2(f.lrow(k0, f.Vs), f.lrow(k1, f.Vs));
            float2 d[NS], qL, qR;
#pragma unroll
            for (int j = 0; j < NS; ++j)
                d[j] = (j == R) ? f2(0.0f) : make_float2(f.lrow(k0, dV[j]), f.lrow(k1, dV[j]));
            weno_states<T, R, MEAN, kUnitDifference<T, R, VAR>>(tb, d, fc, qL, qR);
            dqL[k0] = qL.x;
            dqR[k0] = qR.x;
            dqL[k1] = qL.y;
            dqR[k1] = qR.y;
        }
    }
#pragma unroll
    for (int kk = kScalarFrom; kk < NC; ++kk) {
        const T fc = f.lrow(kk, f.Vs);
        T d[NS];
#pragma unroll
        for (int j = 0; j < NS; ++j) d[j] = (j == R) ? T(0) : f.lrow(kk, dV[j]);
        if constexpr (AO) {
            // GP-AO predictions relative to cell s (the kernel parameter is AoFaceTables)
            const auto &ta = static_cast<const AoFaceTables<T, R> &>(tb);
            dqL[kk] = ao_side<T, R, NS, false, MEAN>(ta, d, fc);                 // q_L - L V_s
            dqR[kk] = ao_side<T, R, NS, true, MEAN>(ta, d, fc) - d[R + 1];      // q_R - L V_{s+1}
        } else {
            weno_states<T, R, MEAN, kUnitDifference<T, R, VAR>>(tb, d, fc, dqL[kk], dqR[kk]);
        }
    }

    T wL[NC], wR[NC];
    f.left_state(dqL, wL);
    f.right_state(dqR, wR);

    // --- face flux relative to F(U_s), and F(U_{s+1}) - F(U_s) ---------------
    T GL[NC], GR[NC], cL[NC], cR[NC], B[NC], uL, uR, aL, aR;
    prim_pert<T, NC>(ref, wL, tb.gamma, igm1, GL, cL, uL, aL, ph);
    prim_pert<T, NC>(ref, wR, tb.gamma, igm1, GR, cR, uR, aR, ph);
    f.flux_difference(st[R], st[R + 1], B);
    ph.need(f.c2, ref.p + dn[E]);
    face_flux<T, NC, LF>(f, tb, wL, wR, GL, GR, cL, cR, uL, uR, aL, aR, A);
#pragma unroll
    for (int a = 0; a < NC; ++a) M[a] = fma(T(-2), B[a], A[a]);
}

// Sum of the two reconstructed parts of one field (or two) of the FD-Flux form, relative to cell s:
// the left part from p (relative to its cell-s value fcp) on windows 0..R, the right part from m
// (fcm) on windows 1..R+1.  Zero mean: shifts fcp and fcm; MEAN: centres cell s and cell s+1.
template <typename T, int R, bool MEAN, bool UNIT, typename V, int NS>
__device__ __forceinline__ V fdf_state(const FaceTables<T, R> &tb, const V (&p)[NS], const V (&m)[NS], V fcp, V fcm)
{
    constexpr int UL = kUnitL<R>, UR = kUnitR<R>;
    const V zero = vset<V>(0.0);
    const V lA = MEAN ? zero : vmul(tb.pA, fcp), lD = MEAN ? zero : vmul(tb.pD, fcp);
    const V rA = MEAN ? vmul(-tb.pA, m[R + 1]) : vmul(tb.pA, fcm), rD = MEAN ? vmul(-tb.pD, m[R + 1]) : vmul(tb.pD, fcm);
    auto part = [&](const V(&d)[NS], V fc, int k, V sA, V sD, V &x) {
        V q = vmul(tb.s1[k], fc);
#pragma unroll
        for (int j = 0; j <= R; ++j)
            if (k + j != R) q = vfma(tb.w[k][j], d[k + j], q);
        x = beta_weight<T, R, UNIT>(tb, d, k, sA, sD);
        return vmul(x, q);
    };
    V denL, denR, x;
    V numL = part(p, fcp, UL, lA, lD, denL), numR = part(m, fcm, UR, rA, rD, denR);
#pragma unroll
    for (int k = 0; k <= R + 1; ++k) {
        if (k <= R && k != UL) {
            numL = vfma(tb.gl[k], part(p, fcp, k, lA, lD, x), numL);
            denL = vfma(tb.gl[k], x, denL);
        }
        if (k > 0 && k != UR) {
            numR = vfma(tb.gr[k - 1], part(m, fcm, k, rA, rD, x), numR);
            denR = vfma(tb.gr[k - 1], x, denR);
        }
    }
    return vfma(numL, vrcp(denL), vmul(numR, vrcp(denR)));
}

// One face of the FD-Flux form (Section 2), cell-relative; outputs as face_rel without the factor 2:
//   A = f^_{s+1/2} - F(U_s),  M = f^_{s+1/2} - F(U_{s+1}).
// The point fluxes are cell averages of the function whose face values are
// the numerical fluxes (Eqs. prim_F, design).  They are split by local
// Lax-Friedrichs, F+- = (F +- alpha U)/2 with alpha the largest |u_n| + c over
// the 2R+2 stencil cells, projected on the characteristic fields of the
// conservative Jacobian at the Roe average, l(X) = L_V (dV/dU) X with dV/dU
// taken at (rbar, vel, c) (the conservative Jacobian depends on the state only
// through vel and H, so these are its left eigenvectors up to row scaling),
// reconstructed by GP-WENO -- F+ on the stencil of cell s at x* = +1/2, F- on
// that of cell s+1 at x* = -1/2, the tables holding reconstruction weights --
// and projected back with (dU/dV) R_V.  Everything is relative to cell s:
// with d+-_j = (l(F_j - F_s) +- alpha l(U_j - U_s)) / 2 and g+-_s the cell-s
// values, each reconstructed part minus g+-_s is
// sum_m omega_m (w_m . d_m + (sum_j w_mj - 1) g+-_s), and g+_s + g-_s = l(F_s)
// projects back to F(U_s).  Requires physical states in `ph`.
template <typename T, int NC, int R, int VAR>
__device__ __forceinline__ void face_fdf(const T (&st)[2 * R + 2][NC], const FaceTables<T, R> &tb, T (&A)[NC],
                                         T (&M)[NC], Physical<T> &ph)
{
    constexpr int NS = 2 * R + 2, E = NC - 1, NV = NC - 2;
    constexpr bool MEAN = (VAR & kVarMean) != 0;
    const FaceRoe<T, NC> f = face_roe<T, NC>(st[R], st[R + 1], tb);
    T vel[NV], q2 = T(0), B[NC];
#pragma unroll
    for (int a = 0; a < NV; ++a) {
        vel[a] = f.vel(a);
        q2 = fma(vel[a], vel[a], q2);
    }
    ph.need(f.c2);

    // splitting speed: the largest |u_n| + c over the stencil
    T alpha = T(0);
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        const T ir = Num<T>::rcp(st[j][0]);
        T m2 = T(0);
#pragma unroll
        for (int a = 0; a < NV; ++a) m2 = fma(st[j][1 + a], st[j][1 + a], m2);
        const T pj = f.gm1 * fma(T(-0.5) * m2, ir, st[j][E]);
        ph.need(st[j][0], pj);
        alpha = Num<T>::pmax(alpha, Num<T>::fabs(st[j][1] * ir) +
                                        Num<T>::sqrt(Num<T>::pmax(tb.gamma * pj * ir, T(1e-30))));
    }
    // dV/dU at the Roe state applied to a conserved vector
    auto jac = [&](const T (&X)[NC], T (&Y)[NC]) {
        Y[0] = X[0];
        T k = T(0);
#pragma unroll
        for (int a = 0; a < NV; ++a) {
            Y[1 + a] = fma(-vel[a], X[0], X[1 + a]) * f.irb;
            k = fma(vel[a], X[1 + a], k);
        }
        Y[E] = f.gm1 * (fma(T(0.5) * q2, X[0], X[E]) - k);
    };
    // cell s: U_s and F(U_s)
    T Fs[NC];
    Fs[0] = st[R][1];
    Fs[1] = fma(st[R][1], f.ref.u[0], f.ref.p);
#pragma unroll
    for (int a = 1; a < NV; ++a) Fs[1 + a] = st[R][1] * f.ref.u[a];
    Fs[E] = f.ref.u[0] * f.ref.hp;
    T JUs[NC], JFs[NC];
    jac(st[R], JUs);
    jac(Fs, JFs);

    // characteristic increments of the split fluxes, relative to cell s
    T dp[NC][NS], dm[NC][NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        if (j == R) {
#pragma unroll
            for (int k = 0; k < NC; ++k) dp[k][j] = dm[k][j] = T(0);
            continue;
        }
        T dV[NC], G[NC], cw[NC], un, cs;
        f.prim_diff(st[j], st[R], dV);
        prim_pert<T, NC>(f.ref, dV, tb.gamma, tb.igm1, G, cw, un, cs, ph);
        if (j == R + 1) {
#pragma unroll
            for (int a = 0; a < NC; ++a) B[a] = G[a];
        }
        T dU[NC], JdU[NC], JG[NC];
#pragma unroll
        for (int a = 0; a < NC; ++a) dU[a] = st[j][a] - st[R][a];
        jac(dU, JdU);
        jac(G, JG);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const T lg = f.lrow(k, JG), lv = f.lrow(k, JdU);
            dp[k][j] = T(0.5) * fma(alpha, lv, lg);
            dm[k][j] = T(0.5) * fma(-alpha, lv, lg);
        }
    }

    T dq[NC];
    // FP32 in 1D and 2D: fields in pairs through packed instructions (as in face_rel);
    // 3D and an odd last field take the scalar loop.
    constexpr bool kPacked = std::is_same<T, float>::value && NC <= 4;
    constexpr int kScalarFrom = kPacked ? (NC / 2) * 2 : 0;
    if constexpr (kPacked) {
#pragma unroll
        for (int k0 = 0; k0 + 1 < NC; k0 += 2) {
            const int k1 = k0 + 1;
            const float2 lgs = make_float2(f.lrow(k0, JFs), f.lrow(k1, JFs));
            const float2 lvs = make_float2(f.lrow(k0, JUs), f.lrow(k1, JUs));
            float2 p2[NS], m2[NS];
#pragma unroll
            for (int j = 0; j < NS; ++j) {
                p2[j] = make_float2(dp[k0][j], dp[k1][j]);
                m2[j] = make_float2(dm[k0][j], dm[k1][j]);
            }
            const float2 q = fdf_state<T, R, MEAN, kUnitDifference<T, R, VAR>>(tb, p2, m2, vmul(0.5f, vfma(alpha, lvs, lgs)),
                                                   vmul(0.5f, vfma(-alpha, lvs, lgs)));
            dq[k0] = q.x;
            dq[k1] = q.y;
        }
    }
#pragma unroll
    for (int kk = kScalarFrom; kk < NC; ++kk) {
        const T lgs = f.lrow(kk, JFs), lvs = f.lrow(kk, JUs);
        dq[kk] = fdf_state<T, R, MEAN, kUnitDifference<T, R, VAR>>(tb, dp[kk], dm[kk], T(0.5) * fma(alpha, lvs, lgs),
                                       T(0.5) * fma(-alpha, lvs, lgs));
    }

    // back-projection A = (dU/dV) R_V dq at the Roe state
    T w[NC];
    w[0] = dq[0] + dq[1] + dq[E];
    w[1] = f.cr * (dq[E] - dq[0]);
#pragma unroll
    for (int a = 2; a < E; ++a) w[a] = dq[a];
    w[E] = f.c2 * (dq[0] + dq[E]);
    A[0] = w[0];
    T ke = T(0);
#pragma unroll
    for (int a = 0; a < NV; ++a) {
        A[1 + a] = fma(vel[a], w[0], f.rbar * w[1 + a]);
        ke = fma(vel[a], w[1 + a], ke);
    }
    A[E] = fma(T(0.5) * q2, w[0], fma(f.rbar, ke, w[E] * tb.igm1));
#pragma unroll
    for (int a = 0; a < NC; ++a) M[a] = A[a] - B[a];
}

// Kernel parameter type of a variant's tables.
template <typename T, int R, int VAR>
using TablesFor = typename std::conditional<(VAR & kVarAo) != 0, AoFaceTables<T, R>, FaceTables<T, R>>::type;

template <typename T, int NC, int R, int VAR, bool P5 = false>
__device__ __forceinline__ void face_eval(const T (&st)[2 * R + 2][NC], const FaceTables<T, R> &tb, T (&A)[NC],
                                          T (&M)[NC], Physical<T> &ph)
{
    constexpr bool kLf = std::is_same<T, float>::value && (VAR & kVarFlux) == 0;
    if constexpr ((VAR & kVarFdFlux) != 0) face_fdf<T, NC, R, VAR>(st, tb, A, M, ph);
    else face_rel<T, NC, R, VAR, kLf, P5>(st, tb, A, M, ph);
}

// Weights of the corrected-flux difference: with the face-flux correction
// f^_{s+1/2} = F + alpha D2F + beta D4F (Eqs. numFlux_cor, FD-ders; alpha = -1/24,
// beta = 3/640), f^_{i+1/2} - f^_{i-1/2} = sum_{k=-2..2} c_k dF_{i+k} where
// dF_s = F_{s+1/2} - F_{s-1/2} and c = (beta, alpha-4beta, 1-2alpha+6beta, alpha-4beta, beta).
// The jumps come doubled from face_rel (A - M), hence the halves; in the FD-Flux form the
// reconstructed flux is itself the numerical flux (Eq. design) and only the centre jump counts.
template <typename T, int VAR>
struct Divergence {
    static constexpr bool kPlain = (VAR & kVarFdFlux) != 0;
    static constexpr double al = -1.0 / 24.0, be = 3.0 / 640.0;
    static constexpr double c0 = kPlain ? 0.0 : 0.5 * be, c1 = kPlain ? 0.0 : 0.5 * (al - 4.0 * be),
                            c2 = kPlain ? 1.0 : 0.5 * (1.0 - 2.0 * al + 6.0 * be);
    // the flux difference across a cell from the five jumps around it
    static __device__ __forceinline__ T of(const T (&d)[5])
    {
        if constexpr (kPlain) return d[2];
        return fma(T(c0), d[4], fma(T(c1), d[3], fma(T(c2), d[2], fma(T(c1), d[1], T(c0) * d[0]))));
    }
    // the same along a march: `a` holds the partial sums of the next four cells (of the same
    // order of operations); takes the jump across cell s and returns the difference across s-2
    static __device__ __forceinline__ T march(T (&a)[4], T d)
    {
        if constexpr (kPlain) {
            const T out = a[0];
            a[0] = a[1];
            a[1] = d;
            return out;
        } else {
            const T out = fma(T(c0), d, a[0]);
            a[0] = fma(T(c1), d, a[1]);
            a[1] = fma(T(c2), d, a[2]);
            a[2] = fma(T(c1), d, a[3]);
            a[3] = T(c0) * d;
            return out;
        }
    }
};

// Index of cell i along a dimension of n cells after the boundary map:
// periodic wrap or zero-gradient clamp (outflow).  Periodic wrap is a full
// modulo, so grids narrower than the ghost width are handled.
__device__ __forceinline__ int bc_map(int i, int n, int periodic)
{
    if (i >= 0 && i < n) return i;
    if (periodic) {
        int r = i % n;
        return r < 0 ? r + n : r;
    }
    return i < 0 ? 0 : n - 1;
}

}  // namespace gpweno
