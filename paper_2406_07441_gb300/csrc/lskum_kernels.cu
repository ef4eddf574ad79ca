// sm_103a kernels of one implicit q-LSKUM pseudo-time iteration (Alg. 1):
//   k_grad      least-squares q-derivatives, first order + K inner iterations (Eq. 10, 16)
//   k_residual  defect-corrected kinetic split-flux residual (Eq. 11-15), local time
//               step and scalar LU-SGS diagonal (Eq. 26, 33-34), density-norm partials
//   k_norm_*    per-case residual norms, histories and stopping tests
//   k_sweeps    all levels of the forward and the backward LU-SGS sweep (Eq. 27) in
//               one cooperative launch, with exact (forward-mode AD) or increment
//               (Eq. 28) Jacobian-vector products, each point's axis products formed
//               once and gathered by its neighbours; k_sweep: one level with the
//               products formed per slot, where lists are too long for the packed form
//   k_update    U += dU, wall projection, q-variables and the per-point primal
//               quantities the next iteration's sweeps need
//
// GB300 has 62x more FP32 than FP64 throughput (1.2 FP64 TFLOP/s measured),
// and an SM's FP64 unit takes one warp instruction in 19 cycles, its integer
// pipes one in 1 or 2 (a 32-bit multiply-add into 64 bits in 4.5).  So the
// kernels that evaluate formulas per neighbour slot, the q-derivatives and the
// residual, run in 64-bit fixed point on the integer pipes (lskum_fixgrad.cuh,
// lskum_fixflux.cuh), with sums that are exact integers, and fall back to FP64
// where a state leaves the fixed-point ranges.  The sweeps, whose increments
// have no fixed range, stay in FP64 (or FP32) and issue few FP64
// instructions: every geometric quantity is precomputed per slot; the exact
// Jacobian products reuse erf and exp of each point's own state, computed once
// per iteration by k_update, so they have no transcendental call at all, and a
// neighbour's product along an axis is formed once and gathered.  Where FP64
// evaluates the split fluxes (the fallback, the update, the framed
// Jacobians, the increment products), exp and A = (1 + s erf S)/2 are the
// kernels' own (lskum_fastmath.cuh: fixed point, exp(-S^2) shared), as are
// signs and multiplications by 2 and 1/2 (integer steps) and, off the critical
// paths, multiplications (mul_i, lskum_intmul.cuh: correctly rounded, the same
// bits).
#include "lskum_internal.h"

#include <cstdint>

#include "lskum_fastmath.cuh"
#include "lskum_fixgrad.cuh"
#include "lskum_fluxtable.h"

namespace lskum {

namespace {

constexpr double kGm1 = 0.4;                              // gamma - 1 (gamma = 1.4)
constexpr double kInv2SqrtPi = 0.28209479177387814347;    // 1 / (2 sqrt(pi))
constexpr double kInvSqrtPi = 0.56418958354775628695;     // 1 / sqrt(pi)
constexpr unsigned kFull = 0xffffffffu;

constexpr int kErrTimeout = -6;  // LSKUM_ERR_TIMEOUT: the sweeps' wait at a level boundary

// Every kernel returns at once after a stop or a failure (the norm goes by
// what k_begin found: it records the iteration that fails).  When a case
// reaches its drop target, k_norm marks it kReachedTarget, so the sweeps and
// the update of that iteration still run; the next k_begin makes it
// kStopped, after which its points are left alone (a batch keeps iterating
// its other cases) and, once every case has stopped, sets stop.  In a batch
// a failure (non-finite norm, non-physical update) fails only its own case,
// which keeps its last good state; a single case fails the context.
__device__ __forceinline__ bool halted(const Ctrl *c)
{
    const volatile Ctrl *v = c;
    return (v->stop | v->error) != 0;
}

// Does this iteration's norm count?  (Not if the sweeps before it gave up
// waiting for one another: the iteration did not happen.)
__device__ __forceinline__ bool counted(const Ctrl *c)
{
    const volatile Ctrl *v = c;
    return v->live && v->error != kErrTimeout;
}

// Is point k's case stopped?  (Only batches have cases that stop while
// others run; a single case stops the whole context.)
__device__ __forceinline__ bool frozen_state(int32_t st)
{
    return st == kStopped || st == kFailed;
}

__device__ __forceinline__ bool frozen(const Dev &d, int k)
{
    return d.n_cases > 1 && frozen_state(((const volatile int32_t *)d.case_state)[d.case_of[k]]);
}

// The same for the sweeps, the explicit step and the update, which do not wait
// for the norm (it runs beside the update, and may be marking a case failed
// meanwhile): the residual has marked every case whose norm can become
// non-finite (d.suspect).
__device__ __forceinline__ bool halted_step(const Dev &d)
{
    return halted(d.ctrl) || (d.n_cases == 1 && d.suspect[0] != 0);
}
__device__ __forceinline__ bool frozen_step(const Dev &d, int k)
{
    return d.n_cases > 1 && (d.suspect[d.case_of[k]] != 0 || frozen(d, k));
}

// One copy of the function tables in global memory, for kernels that need
// them only at a few points (the sweeps: wall and outer points); kernels that
// evaluate them at every point stage them in shared memory instead.
__device__ MathTables g_math;

__global__ void k_init_math()
{
    load_math_tables(g_math);
}

// x with its sign flipped unless pos: an integer XOR of the sign bit, so a
// selected sign costs no FP64 (or FP32) instruction.
__device__ __forceinline__ double signed_by(double x, bool pos)
{
    return __hiloint2double(__double2hiint(x) ^ (pos ? 0 : (int)0x80000000), __double2loint(x));
}
__device__ __forceinline__ float signed_by(float x, bool pos)
{
    return __int_as_float(__float_as_int(x) ^ (pos ? 0 : (int)0x80000000));
}

// x / 2 and 2 x as a step of the exponent field on the integer pipe: the same
// bits as the FP64 multiplication whenever both x and the result are normal
// (a multiplication by a power of two is exact there).  Zeros and
// non-finite values come back unchanged, which is again the exact result;
// only magnitudes below 2^-1021 (halving: the result would be subnormal),
// subnormal inputs (doubling: returned as they are) and magnitudes above
// 2^1023 (doubling) differ, far outside what any quantity of the solver
// reaches.  FP32 keeps
// its multiplication (its pipe is not the bottleneck).
__device__ __forceinline__ double half_of(double x)
{
    const int hi = __double2hiint(x);
    const unsigned ex = ((unsigned)hi >> 20) & 0x7ffu;
    return __hiloint2double(ex - 2u < 0x7fdu ? hi - 0x00100000 : hi, __double2loint(x));
}
__device__ __forceinline__ double twice(double x)
{
    const int hi = __double2hiint(x);
    const unsigned ex = ((unsigned)hi >> 20) & 0x7ffu;
    return __hiloint2double(ex - 1u < 0x7fdu ? hi + 0x00100000 : hi, __double2loint(x));
}
__device__ __forceinline__ float half_of(float x) { return 0.5f * x; }
__device__ __forceinline__ float twice(float x) { return 2.0f * x; }

// Primitive state carried through the residual.
struct Prim {
    double rho, u, v, p, sb, isb, e1, e2;  // sb = sqrt(beta), isb = 1/sb,
                                           // e1 = 3.5 p + rho|u|^2/2, e2 = 3 p + rho|u|^2/2
    double bk;                             // 1 / (2 sqrt(pi beta)): B = exp(-S^2) bk
};

// Inverse of Eq. 14: beta = -q4/2, u = q2/(2 beta), v = q3/(2 beta),
// rho = exp(q1 + beta |u|^2) beta^(-1/(gamma-1)) with 1/(gamma-1) = 5/2,
// p = rho/(2 beta).  One reciprocal square root and one exp.  Its
// multiplications stay on the FP64 unit: every split flux of the slot waits
// for these primitives, and on that critical path the integer multiply's
// longer dependency chain costs more than the FP64 issue it would free
// (measured: the residual is 8% faster this way than with the integer
// multiply here, and 20% slower with every multiplication of the split flux
// on the FP64 unit too).
__device__ __forceinline__ Prim q_to_prim(const MathTables &T, const double q[4])
{
    Prim P;
    const double beta = signed_by(half_of(q[3]), false);  // -q4/2, the sign by XOR
    P.isb = rsqrt(beta);
    const double ib = P.isb * P.isb;   // 1/beta
    const double r = ib * ib * P.isb;  // beta^(-5/2)
    const double i2b = half_of(ib);    // 1/(2 beta)
    P.sb = beta * P.isb;
    P.u = q[1] * i2b;
    P.v = q[2] * i2b;
    const double q2 = fma(P.u, P.u, P.v * P.v);
    P.rho = exp_t(T, fma(beta, q2, q[0])) * r;
    P.p = P.rho * i2b;
    const double k = half_of(P.rho * q2);
    P.e1 = fma(3.5, P.p, k);
    P.e2 = fma(3.0, P.p, k);
    P.bk = kInv2SqrtPi * P.isb;
    return P;
}

// Kinetic split flux G_d^sg (half-range moments of the Maxwellian; sg = +1
// if pos, else -1, applied by negation) in unit direction d: (dx, dy) in a
// (t, n) frame (framed), else the x axis (xdir) or the y axis, where the
// axis components are selected on the integer pipe instead of multiplied by
// 0 and 1.  One body for every frame and axis keeps the residual's loop
// small enough for the instruction cache.
__device__ __forceinline__ void split_flux(const MathTables &T, const Prim &P, bool framed, bool xdir, double dx,
                                          double dy, bool pos, double G[4])
{
    const double ua = xdir ? P.u : P.v, uo = xdir ? P.v : P.u;  // along and across the axis
    const double ud = framed ? fma(P.u, dx, mul_i(P.v, dy)) : ua;
    const double S = ud * P.sb;  // FP64 unit: heads the exp/erfcx path (measured faster)
    double A, eS;
    split_A(T, S, pos, A, eS);
    const double B = mul_i(eS, P.bk);
    const double sB = signed_by(B, pos);
    const double M1 = fma(ud, A, sB);
    const double rm = mul_i(P.rho, M1);
    const double pA = mul_i(P.p, A);
    G[0] = rm;
    if (framed) {
        G[1] = fma(rm, P.u, mul_i(pA, dx));
        G[2] = fma(rm, P.v, mul_i(pA, dy));
    } else {
        const double ga = fma(rm, ua, pA), go = mul_i(rm, uo);
        G[1] = xdir ? ga : go;
        G[2] = xdir ? go : ga;
    }
    G[3] = fma(mul_i(ud, P.e1), A, mul_i(P.e2, sB));
}

// Primal quantities of a conserved state for the Jacobian products (FP64,
// or FP32 for the mixed-precision sweeps).
template <typename T>
struct PrimT {
    T rho, irho, u, v, p, beta, sb, isb, i2p, q2, e1, e2;
};
using PrimU = PrimT<double>;

__device__ __forceinline__ PrimU prim_from_cons(const double U[4])
{
    PrimU P;
    P.rho = U[0];
    P.irho = 1.0 / U[0];
    P.u = mul_i(U[1], P.irho);
    P.v = mul_i(U[2], P.irho);
    P.q2 = fma(P.u, P.u, mul_i(P.v, P.v));
    const double hr = half_of(P.rho);
    P.p = mul_i(kGm1, fma(-hr, P.q2, U[3]));
    const double k = mul_i(hr, P.q2);  // rho |u|^2 / 2
    P.i2p = 0.5 / P.p;
    P.beta = mul_i(P.rho, P.i2p);
    P.sb = sqrt(P.beta);
    P.isb = 1.0 / P.sb;
    P.e1 = fma(3.5, P.p, k);
    P.e2 = fma(3.0, P.p, k);
    return P;
}

// The same for the increment products, by the shortest chain: with Q = 2 rho p
// = 0.8 (rho E - |m|^2/2) everything needs one reciprocal square root, beside
// the one division, instead of three divisions and a square root in a row.
// (Only what flux_prim reads.)  Q is a product of two such values: where it
// leaves 2^-960 .. 2^1000 (or is not positive) the other form takes over.
__device__ __noinline__ void prim_by_division(const double U[4], PrimU &P)
{
    P = prim_from_cons(U);
}
__device__ __forceinline__ PrimU prim_short(const double U[4])
{
    PrimU P;
    const double hm = 0.5 * fma(U[1], U[1], __dmul_rn(U[2], U[2]));
    const double Q = 0.8 * fma(U[0], U[3], -hm);
    if ((unsigned)__double2hiint(Q) - (63u << 20) > (1960u << 20)) {
        prim_by_division(U, P);
        return P;
    }
    P.rho = U[0];
    P.irho = 1.0 / U[0];
    const double r = rsqrt(Q);
    P.sb = __dmul_rn(fabs(U[0]), r);
    P.u = __dmul_rn(U[1], P.irho);
    P.v = __dmul_rn(U[2], P.irho);
    P.p = __dmul_rn(0.5 * Q, P.irho);
    P.isb = __dmul_rn(__dmul_rn(Q, r), fabs(P.irho));
    const double k = __dmul_rn(hm, P.irho);
    P.e1 = fma(3.5, P.p, k);
    P.e2 = fma(3.0, P.p, k);
    return P;
}

template <typename T>
__device__ __forceinline__ PrimT<T> load_prim(const T *__restrict__ pr, int i)
{
    const T *r = pr + (size_t)i * kPrimStride;
    PrimT<T> P;
    P.rho = r[P_RHO];
    P.irho = r[P_IRHO];
    P.u = r[P_U];
    P.v = r[P_V];
    P.p = r[P_P];
    P.beta = r[P_BETA];
    P.sb = r[P_SB];
    P.isb = r[P_ISB];
    P.i2p = r[P_I2P];
    P.q2 = r[P_Q2];
    P.e1 = r[P_E1];
    P.e2 = r[P_E2];
    return P;
}

// Exact product A_d^sg(U) dl by forward-mode differentiation of
// U -> (rho, u, v, p) -> (beta, S, A, B) -> G_d^sg.  S, A = (1 + sg erf S)/2,
// exp(-S^2) and B of the state are inputs (precomputed per point for d = x, y).
// The direction-independent part of the tangent: derivatives of the
// primitive quantities along dl (shared by a neighbour's x and y split
// sub-stencils, computed once per neighbour).
template <typename T>
struct JvpBase {
    T drho, du, dv, dk, dp, dsb;
    T dsbi, de1, de2;  // dsb / sqrt(beta), d(3.5 p + k), d(3 p + k)
};

template <typename T>
__device__ __forceinline__ JvpBase<T> jvp_base(const PrimT<T> &P, const T dl[4])
{
    JvpBase<T> b;
    b.drho = dl[0];
    b.du = (dl[1] - P.u * b.drho) * P.irho;
    b.dv = (dl[2] - P.v * b.drho) * P.irho;
    const T dq2 = twice(P.u * b.du + P.v * b.dv);
    b.dk = half_of(b.drho * P.q2 + P.rho * dq2);  // d(rho |u|^2 / 2)
    b.dp = T(kGm1) * (dl[3] - b.dk);
    const T dbeta = (b.drho - twice(P.beta) * b.dp) * P.i2p;
    b.dsb = half_of(dbeta) * P.isb;
    b.dsbi = b.dsb * P.isb;
    b.de1 = T(3.5) * b.dp + b.dk;
    b.de2 = T(3.0) * b.dp + b.dk;
    return b;
}

// Tangent of the split flux in direction (dx, dy) with sign sg, given the
// primal S, A, exp(-S^2), B of that direction.
template <typename T>
__device__ __forceinline__ void jvp_dir(const PrimT<T> &P, const JvpBase<T> &b, T dx, T dy, T sg, T S, T A, T eS,
                                        T B, T out[4])
{
    const T ud = P.u * dx + P.v * dy;
    const T dud = b.du * dx + b.dv * dy;
    const T dS = dud * P.sb + ud * b.dsb;
    const T dA = sg * eS * dS * T(kInvSqrtPi);
    const T dB = -B * (T(2.0) * S * dS + b.dsbi);
    const T M1 = ud * A + sg * B;
    const T dM1 = dud * A + ud * dA + sg * dB;
    const T de1 = b.de1;
    const T de2 = b.de2;
    const T drm = b.drho * M1 + P.rho * dM1;  // d(rho M1)
    const T rm = P.rho * M1;
    out[0] = drm;
    out[1] = drm * P.u + rm * b.du + (b.dp * A + P.p * dA) * dx;
    out[2] = drm * P.v + rm * b.dv + (b.dp * A + P.p * dA) * dy;
    out[3] = (dud * P.e1 + ud * de1) * A + ud * P.e1 * dA + sg * (de2 * B + P.e2 * dB);
}

// The same product along an axis (DIR 0: d = (1,0), DIR 1: (0,1)) from the
// point's record: A, exp(-S^2)/sqrt(pi) (ek), B, 2 B S and u_d e1 precomputed
// per point, the direction-free tangents in the base, signs applied by
// negation (no multiplication by 0, 1 or +-1 is left to the FP64 pipe).
template <int DIR, typename T>
__device__ __forceinline__ void jvp_axis(const PrimT<T> &P, const JvpBase<T> &b, bool pos, T A, T ek, T B, T B2S,
                                         T ude1, T out[4])
{
    const T ud = DIR == 0 ? P.u : P.v;
    const T dud = DIR == 0 ? b.du : b.dv;
    const T dS = fma(dud, P.sb, ud * b.dsb);
    const T dA = signed_by(ek * dS, pos);
    const T sB = signed_by(B, pos);
    const T sdB = signed_by(fma(B2S, dS, B * b.dsbi), !pos);  // sg times the tangent of B
    const T M1 = fma(ud, A, sB);
    const T dM1 = fma(dud, A, fma(ud, dA, sdB));
    const T rm = P.rho * M1;
    const T drm = fma(b.drho, M1, P.rho * dM1);
    const T pA = fma(b.dp, A, P.p * dA);  // tangent of p A
    out[0] = drm;
    if (DIR == 0) {
        out[1] = fma(drm, P.u, fma(rm, b.du, pA));
        out[2] = fma(drm, P.v, rm * b.dv);
    } else {
        out[1] = fma(drm, P.u, rm * b.du);
        out[2] = fma(drm, P.v, fma(rm, b.dv, pA));
    }
    const T t1 = fma(dud, P.e1, ud * b.de1);
    const T t3 = fma(b.de2, sB, P.e2 * sdB);
    out[3] = fma(t1, A, fma(ude1, dA, t3));  // ude1 = u_d e1, from the record
}

// The same product with the axis chosen at run time (xdir: d = (1,0), else
// (0,1)) without a branch: the axis-dependent operands are selected on the
// integer pipe, so the lanes of a warp that form x- and y-products issue one
// FP64 sequence together.  Equal to jvp_axis<0 or 1> except that a pressure
// term of zero is added as +0 (an exactly zero product then has sign +).
template <typename T>
__device__ __forceinline__ void jvp_axis_sel(const PrimT<T> &P, const JvpBase<T> &b, bool xdir, bool pos, T A, T ek,
                                             T B, T B2S, T ude1, T out[4])
{
    const T ud = xdir ? P.u : P.v;
    const T dud = xdir ? b.du : b.dv;
    const T dS = fma(dud, P.sb, ud * b.dsb);
    const T dA = signed_by(ek * dS, pos);
    const T sB = signed_by(B, pos);
    const T sdB = signed_by(fma(B2S, dS, B * b.dsbi), !pos);
    const T M1 = fma(ud, A, sB);
    const T dM1 = fma(dud, A, fma(ud, dA, sdB));
    const T rm = P.rho * M1;
    const T drm = fma(b.drho, M1, P.rho * dM1);
    const T pA = fma(b.dp, A, P.p * dA);
    const T zero = T(0);
    out[0] = drm;
    out[1] = fma(drm, P.u, fma(rm, b.du, xdir ? pA : zero));
    out[2] = fma(drm, P.v, fma(rm, b.dv, xdir ? zero : pA));
    const T t1 = fma(dud, P.e1, ud * b.de1);
    const T t3 = fma(b.de2, sB, P.e2 * sdB);
    out[3] = fma(t1, A, fma(ude1, dA, t3));
}

// Both signs' products along an axis: bit for bit jvp_axis_sel's (the terms
// that change sign with it are formed once: rounding to nearest is symmetric),
// 34 FP64 instructions instead of 46.
template <typename T>
__device__ __forceinline__ void jvp_axis_pair(const PrimT<T> &P, const JvpBase<T> &b, bool xdir, T Ap, T Am, T ek, T B,
                                              T B2S, T ude1, T outp[4], T outm[4])
{
    const T ud = xdir ? P.u : P.v;
    const T dud = xdir ? b.du : b.dv;
    const T dS = fma(dud, P.sb, ud * b.dsb);
    const T dA = ek * dS;
    const T dB = fma(B2S, dS, B * b.dsbi);  // minus the tangent of B
    const T i1 = fma(ud, dA, -dB), pdA = P.p * dA;
    const T t1 = fma(dud, P.e1, ud * b.de1);
    const T t3 = fma(b.de2, B, P.e2 * -dB);
    const T i3 = fma(ude1, dA, t3);
    const T zero = T(0);
#pragma unroll
    for (int m = 0; m < 2; m++) {
        T *out = m ? outm : outp;
        const T A = m ? Am : Ap;
        const T M1 = fma(ud, A, m ? -B : B);
        const T dM1 = fma(dud, A, m ? -i1 : i1);
        const T rm = P.rho * M1;
        const T drm = fma(b.drho, M1, P.rho * dM1);
        const T pA = fma(b.dp, A, m ? -pdA : pdA);
        out[0] = drm;
        out[1] = fma(drm, P.u, fma(rm, b.du, xdir ? pA : zero));
        out[2] = fma(drm, P.v, fma(rm, b.dv, xdir ? zero : pA));
        out[3] = fma(t1, A, m ? -i3 : i3);
    }
}

// Unsplit Euler-flux Jacobian product A_d(U) dU in direction d = (dx, dy)
// (the tangent of G_d = (rho u_d, rho u u_d + p dx, rho v u_d + p dy,
// (E + p) u_d) along dU; the revised LU-SGS's S term).
__device__ __forceinline__ void euler_jvp(double rho, double u, double v, double p, const double dU[4], double dx,
                                          double dy, double out[4])
{
    const double irho = 1.0 / rho;
    const double ud = u * dx + v * dy;
    const double du = (dU[1] - u * dU[0]) * irho, dv = (dU[2] - v * dU[0]) * irho;
    const double dud = du * dx + dv * dy;
    const double dk = u * dU[1] + v * dU[2] - 0.5 * (u * u + v * v) * dU[0];  // d(rho |u|^2 / 2)
    const double dp = kGm1 * (dU[3] - dk);
    const double E = p / kGm1 + 0.5 * rho * (u * u + v * v);
    out[0] = dU[1] * dx + dU[2] * dy;
    out[1] = dU[1] * ud + rho * u * dud + dp * dx;
    out[2] = dU[2] * ud + rho * v * dud + dp * dy;
    out[3] = (dU[3] + dp) * ud + (E + p) * dud;
}

// (no contraction is left to the compiler: two evaluations of a state agree bit for bit)
__device__ __forceinline__ void flux_prim(const MathTables &T, const PrimU &P, double dx, double dy, bool pos,
                                          double G[4])
{
    const double ud = fma(P.u, dx, __dmul_rn(P.v, dy));
    const double S = __dmul_rn(ud, P.sb);
    double A, eS;
    split_A(T, S, pos, A, eS);
    const double B = __dmul_rn(__dmul_rn(eS, kInv2SqrtPi), P.isb);
    const double sB = signed_by(B, pos);
    const double M1 = fma(ud, A, sB);
    const double rm = __dmul_rn(P.rho, M1);
    const double pA = __dmul_rn(P.p, A);
    G[0] = rm;
    G[1] = fma(rm, P.u, __dmul_rn(pA, dx));
    G[2] = fma(rm, P.v, __dmul_rn(pA, dy));
    G[3] = fma(__dmul_rn(ud, P.e1), A, __dmul_rn(P.e2, sB));
}

__device__ __forceinline__ void flux_cons(const MathTables &T, const double U[4], double dx, double dy, bool pos,
                                          double G[4])
{
    flux_prim(T, prim_from_cons(U), dx, dy, pos, G);
}

template <int TPP, typename T>
__device__ __forceinline__ T group_sum(T v)
{
#pragma unroll
    for (int o = TPP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Four consecutive values from 16-byte-aligned storage (one point's product).
__device__ __forceinline__ void load4(const double *__restrict__ p, double v[4])
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}

// The same, and single values, of what other blocks write within the launch:
// ordinary coherent loads from L2, kept behind the level boundary whose
// acquire orders them (volatile, with a memory clobber: the compiler moves
// none of them across it, and takes none of them for read-only data).
__device__ __forceinline__ void load4_l2(const double *p, double v[4])
{
    asm volatile("ld.global.cg.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void load4_l2(const float *p, float v[4])
{
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ double load_l2(const double *p)
{
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float load_l2(const float *p)
{
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void store4(double *p, const double v[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void store4(float *p, const float v[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// ---------------------------------------------------------------------------
// q-derivatives: first order (Eq. 10), then Jacobi inner iterations of Eq. 16
// ---------------------------------------------------------------------------
// An inner iteration's right-hand side sum_i w_i (Delta q_i - Delta r_i .
// (grad q_i - grad q_0)/2) splits into the first-order term g1 = sum_i w_i
// Delta q_i, fixed across iterations, and -1/2 of
//   sum_i (w_i dx_i) px_i + (w_i dy_i) py_i - px_0 sum_i w_i dx_i - py_0 sum_i w_i dy_i
// with the coefficients (-1/2 w dx, ...) precomputed per slot, and the
// centre's as one more slot.
//
// Both passes run in 64-bit fixed point (lskum_fixgrad.cuh) on the integer
// pipes.  Two lanes per slot, each two of the four components: their sums (16
// 64-bit words) leave room for the loads in flight, and a pair reads one
// neighbour's record.  147,584 points, three passes: 0.293 ms in FP64 (its
// unit 92 % busy), 0.141 ms like this (0.033 first order, 0.047 per inner
// iteration, which reads 130 MB: 0.019 ms); 41,194 points 0.137 -> 0.054 ms.
// What is left is the gathers' latency with 20 warps per SM and the multiply
// pipe, half busy.  Rings of cp.async stages in shared memory (0.182 ms) and
// slots along a space-filling curve (the same) were no faster.

// 32 bytes with one load (a pair's 64-byte record is one L1 tag instead of two).
template <typename T>
__device__ __forceinline__ void load32(const T *p, uint4 &a, uint4 &b)
{
    asm("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
        : "l"(p));
}

// 2^e, |e| < 1023.
__device__ __forceinline__ double pow2(int e)
{
    return __hiloint2double((1023 + e) << 20, 0);
}

// The value of a stored G (or of a mark's FP64 derivative) in units of q.
__device__ __forceinline__ double g_value(int lo, int hi, const double *g, int ex, int unit)
{
    return fix_marked(hi) ? scalbn(*g, -ex) : scalbn((double)join_g(hi, lo), -unit);
}

// A point's word gb: the bits of its weights' remainders, and the powers of two
// of its case's units (fix_shift).
__device__ __forceinline__ int grad_bits(short2 gb, bool corr)
{
    return (corr ? gb.y : gb.x) & 255;
}
__device__ __forceinline__ int grad_shift(short2 gb)
{
    return gb.x >> 8 | (gb.y >> 8) << 8;
}

// What k_grad forms, in FP64, for a point that meets a marked value or has no
// fast scale: the lane's slots, its two components, v = x 0, x 1, y 0, y 1 in
// units of q without the first-order term (the lanes of a group add them).
template <int S, bool CORR>
__device__ __noinline__ void grad_fp64(const Dev &d, const double *__restrict__ q, int from, int k, int sub, int c2,
                                       double v[4])
{
    const int4 *__restrict__ gf = CORR ? d.gf[from] : nullptr;
    const double *__restrict__ g = CORR ? d.gq[from] : nullptr;
    const short4 ge = d.ge[k];
    const double lsb = pow2(-grad_bits(d.gb[k], CORR));
    const int shift = grad_shift(d.gb[k]);
    const int deg = d.deg[k];
    const int base = d.slice_off[k >> 5] + (k & 31);
    for (int c = 0; c < 4; c++) v[c] = 0.0;
    // (the centre after the last slot of the first lane)
    for (int j = sub, centre = 0; !centre && (j < deg || (CORR && sub == 0)); j += S) {
        centre = j >= deg;
        const int e = base + 32 * j;
        const int i = centre ? k : d.nbr[e];
        if (!CORR) {
            const uint4 w = d.wg[e];
            const double wx = fma((double)(int)w.y, lsb, (double)(int)w.x);
            const double wy = fma((double)(int)w.w, lsb, (double)(int)w.z);
            for (int c = 0; c < 2; c++) {
                const double dq = q[4 * (size_t)i + 2 * c2 + c] - q[4 * (size_t)k + 2 * c2 + c];
                v[c] = fma(wx, dq, v[c]);
                v[2 + c] = fma(wy, dq, v[2 + c]);
            }
        } else {
            const uint4 *w = centre ? d.wc + 2 * (size_t)k : d.wj + 2 * (size_t)e;
            const uint4 a = w[0], b = w[1];
            const double axx = fma((double)(int)a.y, lsb, (double)(int)a.x);
            const double axy = fma((double)(int)a.w, lsb, (double)(int)a.z);
            const double ayx = fma((double)(int)b.y, lsb, (double)(int)b.x);
            const double ayy = fma((double)(int)b.w, lsb, (double)(int)b.z);
            const short4 gi = d.ge[i];
            const int *f = reinterpret_cast<const int *>(gf + 4 * (size_t)i + 2 * c2);
            for (int c = 0; c < 2; c++) {
                const double *gx = g + 8 * (size_t)i + 2 * c2 + c;
                const int unit = fix_unit(2 * c2 + c, shift);
                const double x = g_value(f[4 * c], f[4 * c + 1], gx, gi.x, unit);
                const double y = g_value(f[4 * c + 2], f[4 * c + 3], gx + 4, gi.y, unit);
                v[c] = fma(axx, x, fma(axy, y, v[c]));
                v[2 + c] = fma(ayx, x, fma(ayy, y, v[2 + c]));
            }
        }
    }
    for (int c = 0; c < 4; c++) {
        const int p = c < 2 ? ge.z : ge.w;
        v[c] = p == kGradNoScale ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(v[c], (CORR ? p : 0) - 31);
    }
}

// Four slots' loads in flight per lane, the next four's neighbours with them:
// a gather takes about 1000 cycles, a slot's 32 multiply-adds 150.
// 128 threads and 96 registers, five blocks per SM.
constexpr int kGradBlock = 128, kGradUnroll = 4;

// Slot lanes per point of the q-derivatives for TPP lanes of the residual: a
// warp's slots are short here, so splitting a point's list pays only in the
// smallest clouds (40,621 points: one 0.054 ms, two 0.061; 10,240: equal).
template <int TPP>
constexpr int kGradLanes = TPP == 8 ? 2 : 1;

// Pass `to` buffer: first order (CORR false, buffer 2) or an inner iteration
// from buffer `from`; S slot lanes per point (2 S lanes in all).  The FP64
// derivatives are stored by the last pass and, with a mark, wherever the
// fixed-point form does not hold them.
template <int S, bool CORR>
__global__ void __launch_bounds__(kGradBlock, 5) k_grad(Dev d, StateSet st, int from, int to, bool last)
{
    if (halted(d.ctrl)) return;
    constexpr int L = 2 * S;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = gt / L, sub = (gt % L) >> 1, c2 = gt & 1;
    const bool active = k < d.n;
    const int kk = active ? k : d.n - 1;
    const short4 ge = d.ge[kk];
    bool bad = abs(ge.x) > kMaxGradExp || abs(ge.y) > kMaxGradExp || ge.z > kMaxGradShift || ge.w > kMaxGradShift;
    const int bits = grad_bits(d.gb[kk], CORR);
    bad |= bits < kMinGradBits;
    // every lane of a slice runs to the slice's width: a padding slot is the
    // point itself with weights 0
    const int beg = d.slice_off[kk >> 5], width = (d.slice_off[(kk >> 5) + 1] - beg) >> 5;
    int e = beg + (kk & 31) + 32 * sub;
    GradSum x[2] = {}, y[2] = {};
    auto slots = [&](auto &&load, auto &&use) {
        int i[kGradUnroll];
        int j = sub;
#pragma unroll
        for (int u = 0; u < kGradUnroll; u++) i[u] = j + u * S < width ? d.nbr[e + 32 * S * u] : kk;
        for (; j + (kGradUnroll - 1) * S < width; j += kGradUnroll * S) {
            decltype(load(0, 0)) v[kGradUnroll];
#pragma unroll
            for (int u = 0; u < kGradUnroll; u++, e += 32 * S) v[u] = load(e, i[u]);
#pragma unroll
            for (int u = 0; u < kGradUnroll; u++) i[u] = j + (u + kGradUnroll) * S < width ? d.nbr[e + 32 * S * u] : kk;
#pragma unroll
            for (int u = 0; u < kGradUnroll; u++) use(v[u]);
        }
#pragma unroll
        for (int u = 0; u < kGradUnroll - 1; u++, j += S, e += 32 * S)
            if (j < width) use(load(e, i[u]));
    };
    if (!CORR) {
        struct Slot {
            uint4 w;
            longlong2 q;
        };
        const longlong2 *__restrict__ qf = reinterpret_cast<const longlong2 *>(st.qf) + c2;
        const longlong2 q0 = qf[2 * (size_t)kk];
        bad |= fix_marked((int)(q0.x >> 32)) || fix_marked((int)(q0.y >> 32));
        const int64_t b0 = q0.x - 0x80000000ll, b1 = q0.y - 0x80000000ll;
        slots([&](int e, int i) { return Slot{d.wg[e], qf[2 * (size_t)i]}; },
              [&](const Slot &v) {
                  const uint4 &w = v.w;
                  bad |= fix_marked((int)(v.q.x >> 32)) || fix_marked((int)(v.q.y >> 32));
                  int dh, dl;
                  split_word(v.q.x - b0, dh, dl);
                  grad_add(x[0], w.x, w.y, dh, dl);
                  grad_add(y[0], w.z, w.w, dh, dl);
                  split_word(v.q.y - b1, dh, dl);
                  grad_add(x[1], w.x, w.y, dh, dl);
                  grad_add(y[1], w.z, w.w, dh, dl);
              });
    } else {
        struct Slot {
            uint4 a, b, g0, g1;
        };
        const int4 *__restrict__ gf = d.gf[from] + 2 * c2;
        auto load = [&](const uint4 *w, const int4 *g) {
            Slot v;
            load32(w, v.a, v.b);
            load32(g, v.g0, v.g1);
            return v;
        };
        auto use = [&](const Slot &v) {
            const uint4 &a = v.a, &b = v.b, &g0 = v.g0, &g1 = v.g1;
            bad |= fix_marked((int)g0.y);
            grad_add(x[0], a.x, a.y, g0.y, g0.x);
            grad_add(x[0], a.z, a.w, g0.w, g0.z);
            grad_add(x[1], a.x, a.y, g1.y, g1.x);
            grad_add(x[1], a.z, a.w, g1.w, g1.z);
            grad_add(y[0], b.x, b.y, g0.y, g0.x);
            grad_add(y[0], b.z, b.w, g0.w, g0.z);
            grad_add(y[1], b.x, b.y, g1.y, g1.x);
            grad_add(y[1], b.z, b.w, g1.w, g1.z);
        };
        if (sub == 0) use(load(d.wc + 2 * (size_t)kk, gf + 4 * (size_t)kk));
        slots([&](int e, int i) { return load(d.wj + 2 * (size_t)e, gf + 4 * (size_t)i); }, use);
    }
    // the group's sums: every second lane holds the same components
    int64_t hh[4], lo[4];
#pragma unroll
    for (int c = 0; c < 2; c++) {
        hh[c] = x[c].hh, lo[c] = grad_low(x[c], bits);
        hh[2 + c] = y[c].hh, lo[2 + c] = grad_low(y[c], bits);
    }
#pragma unroll
    for (int o = S; o > 1; o >>= 1) {
#pragma unroll
        for (int c = 0; c < 4; c++) {
            hh[c] += __shfl_xor_sync(kFull, hh[c], o);
            lo[c] += __shfl_xor_sync(kFull, lo[c], o);
        }
        bad |= __shfl_xor_sync(kFull, (int)bad, o) != 0;
    }
    int64_t v[4] = {0, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < 4; c++) {
        if (!bad) bad = !grad_value(hh[c], lo[c], bits, CORR ? (c < 2 ? ge.z : ge.w) : 0, v[c]);
    }
    double f[4] = {0.0, 0.0, 0.0, 0.0};  // a marked point's, in units of q
    if (CORR && !bad) {
        const int4 a = d.gf[2][4 * (size_t)kk + 2 * c2], b = d.gf[2][4 * (size_t)kk + 2 * c2 + 1];
        bad |= fix_marked(a.y);
        v[0] += join_g(a.y, a.x), v[2] += join_g(a.w, a.z);
        v[1] += join_g(b.y, b.x), v[3] += join_g(b.w, b.z);
    }
#pragma unroll
    for (int c = 0; c < 4; c++) bad |= !grad_in_range(v[c]);
    if (__any_sync(kFull, bad)) {
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        if (bad) grad_fp64<S, CORR>(d, st.q, from, kk, sub, c2, t);
#pragma unroll
        for (int c = 0; c < 4; c++) {
#pragma unroll
            for (int o = S; o > 1; o >>= 1) t[c] += __shfl_xor_sync(kFull, t[c], o);
        }
        if (bad) {
            bool fits = true;
            const int shift = grad_shift(d.gb[kk]);
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const int cc = 2 * c2 + (c & 1), unit = fix_unit(cc, shift);
                if (CORR) {
                    const int *a = reinterpret_cast<const int *>(d.gf[2] + 4 * (size_t)kk + cc) + 2 * (c >> 1);
                    t[c] += g_value(a[0], a[1], d.gq[2] + 8 * (size_t)kk + cc + 4 * (c >> 1), c < 2 ? ge.x : ge.y, unit);
                }
                fits = fits && fabs(t[c]) < scalbn(3.75, 60 - unit);
                f[c] = t[c];
                v[c] = fits ? __double2ll_rn(scalbn(t[c], unit)) : 0;
            }
            bad = !fits || abs(ge.x) > kMaxGradExp || abs(ge.y) > kMaxGradExp;
        }
    }
    if (!active || sub != 0) return;
    int4 a, b;
    split_g(v[0], a.y, a.x);
    split_g(v[2], a.w, a.z);
    split_g(v[1], b.y, b.x);
    split_g(v[3], b.w, b.z);
    if (bad) a = b = make_int4(0, INT32_MIN, 0, INT32_MIN);
    int4 *gf = d.gf[to] + 4 * (size_t)k + 2 * c2;
    gf[0] = a;
    gf[1] = b;
    if (last || bad) {
        double2 *g = reinterpret_cast<double2 *>(d.gq[to] + 8 * (size_t)k) + c2;
        if (bad) {
            g[0] = make_double2(scalbn(f[0], ge.x), scalbn(f[1], ge.x));
            g[2] = make_double2(scalbn(f[2], ge.y), scalbn(f[3], ge.y));
        } else {
            const int shift = grad_shift(d.gb[kk]), u0 = fix_unit(2 * c2, shift), u1 = fix_unit(2 * c2 + 1, shift);
            g[0] = make_double2((double)v[0] * pow2(ge.x - u0), (double)v[1] * pow2(ge.x - u1));
            g[2] = make_double2((double)v[2] * pow2(ge.y - u0), (double)v[3] * pow2(ge.y - u1));
        }
    }
}

// ---------------------------------------------------------------------------
// flux residual, time step, diagonal, norm partials
// ---------------------------------------------------------------------------
// The frame of point k: (1,0), (0,1), or (t, n) at wall and kinetic outer points.
__device__ __forceinline__ void point_frame(const Dev &d, int k, bool framed, double &e1x, double &e1y, double &e2x,
                                            double &e2y)
{
    e1x = 1.0, e1y = 0.0, e2x = 0.0, e2y = 1.0;
    if (framed) {
        const int ld = d.ld;
        e1x = d.geo[G_E1X * ld + k];
        e1y = d.geo[G_E1Y * ld + k];
        e2x = d.geo[G_E2X * ld + k];
        e2y = d.geo[G_E2Y * ld + k];
    }
}

// The sign of x with magnitude 0 (what 0 * x gives), on the integer pipe.
__device__ __forceinline__ double zero_like(double x)
{
    return __hiloint2double(__double2hiint(x) & (int)0x80000000, 0);
}

// The modified q-variables of a slot (Eq. 15): neighbour i's (q-variables q,
// q-derivatives x and y) and the point's own, over half the offset (hdx, hdy).
__device__ __forceinline__ void reconstruct(const double q[4], const double x[4], const double y[4],
                                            const double q0[4], const double gx0[4], const double gy0[4], double hdx,
                                            double hdy, double qi[4], double q0t[4])
{
#pragma unroll
    for (int c = 0; c < 4; c++) {
        qi[c] = fma(-hdx, x[c], fma(-hdy, y[c], q[c]));
        q0t[c] = fma(-hdx, gx0[c], fma(-hdy, gy0[c], q0[c]));
    }
}

// R += y with Kahan's compensated summation (W. Kahan, "Further remarks on
// reducing truncation errors", CACM 8(1), 1965): c carries the negated
// rounding error of the running sum into the next term.
__device__ __forceinline__ void comp_add(double &R, double &c, double y)
{
    const double t = R + y;
    c = (t - R) - y;  // what the addition lost (negated)
    R = t;
}

// The slots sub, sub + TPP, ... of point k in FP64, for states outside the
// fixed-point ranges (hypersonic, very hot or very dense, non-finite ones);
// the group's lanes add their sums.  In mixed precision the sums are
// compensated: the terms of a group of four slots, by FMAs, less the error
// carried so far, enter R by one compensated addition.
template <int TPP>
__device__ __forceinline__ void residual_slots(const Dev &d, const MathTables &T, const double *__restrict__ q,
                                               const double *__restrict__ g, int k, int sub, bool second, double R[4])
{
    const int ld = d.ld;
    const bool framed = d.flag[k] != kInterior;
    const double e1x = d.geo[G_E1X * ld + k], e1y = d.geo[G_E1Y * ld + k];
    const double e2x = d.geo[G_E2X * ld + k], e2y = d.geo[G_E2Y * ld + k];
    const double wsc = d.geo[G_WSC * ld + k];
    double q0[4], gx0[4], gy0[4];
    load4(q + 4 * (size_t)k, q0);
    load4(g + 8 * (size_t)k, gx0);
    load4(g + 8 * (size_t)k + 4, gy0);
    double y[4] = {0.0, 0.0, 0.0, 0.0}, carry[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 4; c++) R[c] = 0.0;
    const int deg = d.deg[k];
    const int base = d.slice_off[k >> 5] + (k & 31);
    int ng = 0;  // slots in the current group
    for (int j = sub; j < deg; j += TPP) {
        const int e = base + 32 * j;
        const int mb = d.memb[e];
        if (!mb) continue;
        const int i = d.nbr[e];
        const double hx = d.hxy[e].x, hy = d.hxy[e].y;
        double qn[4], xn[4], yn[4], qi[4], q0t[4];
        load4(q + 4 * (size_t)i, qn);
        load4(g + 8 * (size_t)i, xn);
        load4(g + 8 * (size_t)i + 4, yn);
        reconstruct(qn, xn, yn, q0, gx0, gy0, second ? hx : zero_like(hx), second ? hy : zero_like(hy), qi, q0t);
        const Prim Pi = q_to_prim(T, qi);
        const Prim P0 = q_to_prim(T, q0t);
#pragma unroll 1
        for (int sb = 0; sb < 2; sb++) {
            const int m = sb == 0 ? (mb & 3) : (mb >> 2);
            if (!m) continue;
            const bool pos = m & 1, xdir = sb == 0;
            const uint4 wq = d.wq[e];
            const double w = fma((double)(int)(xdir ? wq.y : wq.w), 0x1p-24, (double)(int)(xdir ? wq.x : wq.z)) * wsc;
            const double dx = xdir ? e1x : e2x, dy = xdir ? e1y : e2y;
            double Gi[4], G0[4];
            split_flux(T, Pi, framed, xdir, dx, dy, pos, Gi);
            split_flux(T, P0, framed, xdir, dx, dy, pos, G0);
#pragma unroll
            for (int c = 0; c < 4; c++) y[c] = fma(w, Gi[c] - G0[c], y[c]);
        }
        if (d.precision && ++ng == 4) {
#pragma unroll
            for (int c = 0; c < 4; c++) {
                comp_add(R[c], carry[c], y[c]);
                y[c] = -carry[c];
            }
            ng = 0;
        }
    }
#pragma unroll
    for (int c = 0; c < 4; c++) {
        if (d.precision && ng > 0) comp_add(R[c], carry[c], y[c]);
        R[c] = d.precision ? R[c] - carry[c] : y[c];
    }
}

// The same for a point among points inside the ranges.
template <int TPP>
__device__ __noinline__ void residual_fp64(const Dev &d, const double *__restrict__ q, const double *__restrict__ g,
                                           int k, int sub, bool second, double R[4])
{
    residual_slots<TPP>(d, g_math, q, g, k, sub, second, R);
}

// Is point k's residual formed in FP64 throughout (by k_residual_fp64)?
__device__ __forceinline__ bool hypersonic(const Dev &d, int k)
{
    return d.fp64_cases == 2 && d.case_fp64[d.case_of[k]] != 0;
}

// The ghost term of a kinetic outer point: the n- side is free-stream ghosts
// at the mirror images of the inside neighbours, LS_3(1) (G_n^-(U_inf) -
// G_n^-(U_0)) with LS_3(1) = -LS_2(1); first order (the point's own state).
__device__ __noinline__ void add_ghosts(const Dev &d, const double *__restrict__ U, int k, double e2x, double e2y,
                                        double R[4])
{
    const int ld = d.ld;
    const double *ui = d.case_uinf + 4 * d.case_of[k];
    double U0[4], Ui[4];
    bool same = true;
#pragma unroll
    for (int c = 0; c < 4; c++) {
        U0[c] = U[c * ld + k];
        Ui[c] = ui[c];
        same = same && U0[c] == Ui[c];
    }
    if (same) return;  // (equal states give exactly 0)
    double Gi[4], G0[4];
    flux_cons(g_math, Ui, e2x, e2y, false, Gi);
    flux_cons(g_math, U0, e2x, e2y, false, G0);
    const double l3 = d.geo[G_LS1_3 * ld + k];
#pragma unroll
    for (int c = 0; c < 4; c++) R[c] = fma(l3, Gi[c] - G0[c], R[c]);
}

// x, or 0 where x is negative, on the integer pipe.
__device__ __forceinline__ double positive_part(double x)
{
    const int m = ~(__double2hiint(x) >> 31);
    return __hiloint2double(__double2hiint(x) & m, __double2loint(x) & m);
}

// Local time step (reading: CFL min_i|dr| / (|u| + a)) and scalar diagonal of
// point k: Eq. 26 with the spectral radii of Eq. 34, kept at least sum_s
// rho_s sum_i |w_i| so that it bounds the off-diagonal blocks.  D and 1/D are
// stored (the sweeps multiply by 1/D).  One square root and one division: a
// from the record's 1/sqrt(beta) (a^2 = 0.7/beta), 1/min|dr| stored.
__device__ __forceinline__ void diag_point(const Dev &d, const StateSet &st, int k, double cfl, double e1x, double e1y,
                                           double e2x, double e2y)
{
    const int ld = d.ld;
    const double *pr = st.prim + (size_t)k * kPrimStride;
    const double u = pr[P_U], v = pr[P_V];
    const double a = 0.83666002653407554798 * pr[P_ISB];  // sqrt(0.7 / beta)
    const double idt = (sqrt(pr[P_Q2]) + a) * d.geo[G_IDMIN * ld + k] * (1.0 / cfl);
    if (d.scheme == 1) {  // explicit: D = 1/dt, the step is -dt R
        d.D[k] = idt;
        d.iD[k] = 1.0 / idt;
        return;
    }
    const double u1 = u * e1x + v * e1y, u2 = u * e2x + v * e2y;
    double D = idt;
    if (d.lusgs == 1) {  // revised LU-SGS: Jameson's splitting, rho(A_d) = |u_d| + a
        const double s1 = fabs(u1) + a, s2 = fabs(u2) + a;
        D += 0.5 * (s1 * (fabs(d.geo[G_LS1_0 * ld + k]) + fabs(d.geo[G_LS1_1 * ld + k])) +
                    s2 * (fabs(d.geo[G_LS1_2 * ld + k]) + fabs(d.geo[G_LS1_3 * ld + k])));
    } else {
        const double r0 = positive_part(u1 + a), r1 = positive_part(a - u1);
        const double r2 = positive_part(u2 + a), r3 = positive_part(a - u2);
        D -= r0 * d.geo[G_LS1_0 * ld + k];
        D += r1 * d.geo[G_LS1_1 * ld + k];
        D -= r2 * d.geo[G_LS1_2 * ld + k];
        D += r3 * d.geo[G_LS1_3 * ld + k];
        const double dom = r0 * d.geo[G_ABS_0 * ld + k] + r1 * d.geo[G_ABS_1 * ld + k] + r2 * d.geo[G_ABS_2 * ld + k] +
                           r3 * d.geo[G_ABS_3 * ld + k];
        D = D > dom ? D : dom;
    }
    d.D[k] = D;
    d.iD[k] = 1.0 / D;
}

// The CFL number of this iteration (counted by k_begin).
__device__ __forceinline__ double cfl_now(const Dev &d, int n1)
{
    return (d.ramp > 0.0 && (double)n1 < d.ramp) ? d.cfl * ((double)n1 / d.ramp) : d.cfl;
}

// Point k's residual from its sums: the ghost term, the store, and the diagonal
// (by k_diag with several lanes per point).
template <int TPP>
__device__ __forceinline__ void finish_residual(const Dev &d, const StateSet &st, int k, int fl, int n1, double e1x,
                                                double e1y, double e2x, double e2y, double R[4])
{
    if (fl == kOuter) add_ghosts(d, st.U, k, e2x, e2y, R);
#pragma unroll
    for (int c = 0; c < 4; c++) d.R[c * d.ld + k] = R[c];
    // (the sum of 2^28 squares of smaller values is finite)
    if (!(fabs(R[0]) < 8e149)) d.suspect[d.case_of[k]] = 1;
    if (TPP == 1) diag_point(d, st, k, cfl_now(d, n1), e1x, e1y, e2x, e2y);
}

// Diagonals of all swept points, a thread per point, for the launch shapes
// with several lanes per point in the residual: there a warp holds few
// points, and its FP64 sequence per point (about 45 instructions) would cost
// more than the fluxes it follows.  It needs only the state, so a captured
// iteration runs it beside the q-derivatives and the residual.
__global__ void __launch_bounds__(256) k_diag(Dev d, StateSet st)
{
    if (halted(d.ctrl)) return;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    const int fl = d.flag[k];
    if ((fl == kOuter && d.farfield != 1) || frozen(d, k)) return;
    double e1x, e1y, e2x, e2y;
    point_frame(d, k, fl != kInterior, e1x, e1y, e2x, e2y);
    diag_point(d, st, k, cfl_now(d, ((const volatile Ctrl *)d.ctrl)->it), e1x, e1y, e2x, e2y);
}

// Threads per block of the residual: 512 threads share an SM's registers and
// one copy of the tables (one lane per point: 0.229 ms on 147,584 points
// against 0.237 with two blocks of 256); with several lanes per point, the
// shapes of small clouds, two blocks of 256 spread the work over more SMs
// (10,240 points, two lanes: 0.032 ms against 0.038).
template <int TPP>
constexpr int kResBlock = TPP == 1 ? 512 : 256;
constexpr int kRes64Block = 128;

// Flux residual, local time step and scalar diagonal; TPP lanes per point
// over its slots, persistent blocks (a warp takes every W-th group of 32/TPP
// points, so a block loads the 46 KB of tables once).
// The reconstruction (16 FMAs per slot) runs on the FP64 unit; the inverse of
// Eq. 14, the four split fluxes of a slot and the weighted sums run in 64-bit
// fixed point on the integer pipes (lskum_fixflux.cuh), beside it.  The sums
// are exact integers, so R does not depend on the order of the slots or on
// TPP, and needs no compensation.  A framed point's velocities are rotated
// into its frame, where every split flux is along an axis, and the sum's
// momentum back out of it.  Measured on the 147,584-point cloud (1 lane per
// point): 0.649 ms with the fluxes in FP64 and integer-pipe multiplies, 0.693
// ms with compensated sums; 0.216 ms like this (41,194 points, four lanes:
// 0.235 -> 0.091 ms).  The FMA-heavy pipe, which runs the 32-bit multiplies,
// is about 70 % busy; four warps per scheduler (128 registers) do not hide
// the rest of the chains' latency.  Staging the next slot's records in shared
// memory, prefetching them, and a lane per state with more warps were slower.
template <int TPP>
__global__ void __launch_bounds__(kResBlock<TPP>, 512 / kResBlock<TPP>)
    k_residual(Dev d, StateSet st, const double *__restrict__ g)
{
    __shared__ __align__(16) uint64_t T[kFluxTableWords];
    if (halted(d.ctrl)) return;
    static_assert(kFluxTableR == kFluxRows && kFluxTableExp == kFluxExpRows && kFluxTableWords % 2 == 0, "tables");
    static_assert(kLn2Fx == kFluxLn2 && kInvLn2Fx == kFluxInvLn2, "the table's constants");
    for (int i = threadIdx.x; i < kFluxTableWords / 2; i += kResBlock<TPP>)
        reinterpret_cast<ulonglong2 *>(T)[i] = reinterpret_cast<const ulonglong2 *>(kFluxTable)[i];
    __syncthreads();
    const int n1 = ((const volatile Ctrl *)d.ctrl)->it;  // this iteration, counted by k_begin
    const bool second = n1 > d.first_order;  // first-order start: q~ = q
    const int ld = d.ld;
    const double *__restrict__ q = st.q;
    constexpr int kPts = 32 / TPP;
    const int lane = threadIdx.x & 31, sub = lane % TPP;
    const int tasks = (d.n + kPts - 1) / kPts;
    for (int task = (blockIdx.x * kResBlock<TPP> + threadIdx.x) / 32; task < tasks;
         task += gridDim.x * (kResBlock<TPP> / 32)) {
        const int k = task * kPts + lane / TPP;
        const bool active = k < d.n;
        const int kk = active ? k : d.n - 1;
        const int fl = d.flag[kk];
        const bool work = active && (fl != kOuter || d.farfield == 1) && !frozen(d, kk) && !hypersonic(d, kk);
        const bool framed = fl != kInterior;  // (t, n) frame: wall and kinetic outer points
        FxSum acc[4] = {};
        uint32_t bad = 0;
        const double *pr = st.prim + (size_t)kk * kPrimStride;
        const uint32_t sh = fx_shift((uint32_t)__double2hiint(pr[P_RHO]), (uint32_t)__double2hiint(pr[P_ISB]));
        if (work) {
            double q0[4], gx0[4], gy0[4];
            load4(q + 4 * (size_t)kk, q0);
            load4(g + 8 * (size_t)kk, gx0);
            load4(g + 8 * (size_t)kk + 4, gy0);
            const int deg = d.deg[kk];
            int e = d.slice_off[kk >> 5] + (kk & 31) + 32 * sub;
            int in = kk, mn = 0;
            if (sub < deg) {
                in = d.nbr[e];
                mn = d.memb[e];
            }
            for (int j = sub; j < deg; j += TPP, e += 32 * TPP) {
                const int i = in, m = mn;
                if (j + TPP < deg) {  // the next slot's index before this slot's work
                    in = d.nbr[e + 32 * TPP];
                    mn = d.memb[e + 32 * TPP];
                }
                if (!m) continue;
                double qn[4], xn[4], yn[4], qi[4], q0t[4];
                load4(q + 4 * (size_t)i, qn);
                load4(g + 8 * (size_t)i, xn);
                load4(g + 8 * (size_t)i + 4, yn);
                const double2 h = d.hxy[e];  // half offsets
                const uint4 wq = d.wq[e];
                reconstruct(qn, xn, yn, q0, gx0, gy0, second ? h.x : zero_like(h.x),
                            second ? h.y : zero_like(h.y), qi, q0t);
                // (a loop of at most one pass: as a predicated sequence this would
                // occupy the FP64 unit at every interior point too)
#pragma unroll 1
                for (int r = 0; r < (int)framed; r++) {
                    const double e1x = d.geo[G_E1X * ld + kk], e1y = d.geo[G_E1Y * ld + kk];
                    const double e2x = d.geo[G_E2X * ld + kk], e2y = d.geo[G_E2Y * ld + kk];
                    const double a = qi[1], b = q0t[1];
                    qi[1] = fma(a, e1x, qi[2] * e1y);
                    qi[2] = fma(a, e2x, qi[2] * e2y);
                    q0t[1] = fma(b, e1x, q0t[2] * e1y);
                    q0t[2] = fma(b, e2x, q0t[2] * e2y);
                }
                FxState si, s0;
                fx_state(T, qi[0], qi[1], qi[2], qi[3], si, bad, sh);
                fx_state(T, q0t[0], q0t[1], q0t[2], q0t[3], s0, bad, sh);
                if (m & 3) {
                    const bool pos = m & 1;
                    FxFlux Gi, G0;
                    fx_flux(T, si, si.u, si.su, si.v, si.sv, pos, Gi, bad);
                    fx_flux(T, s0, s0.u, s0.su, s0.v, s0.sv, pos, G0, bad);
                    const int wh = (int)wq.x, wl = (int)wq.y, sh = pos ? wh : -wh, sl = pos ? wl : -wl;
                    fx_add(acc[0], sh, sl, Gi.rm, G0.rm);
                    fx_add(acc[1], wh, wl, Gi.ga, G0.ga);
                    fx_add(acc[2], sh, sl, Gi.go, G0.go);
                    fx_add(acc[3], sh, sl, Gi.g3, G0.g3);
                }
                if (m & 12) {
                    const bool pos = m & 4;
                    FxFlux Gi, G0;
                    fx_flux(T, si, si.v, si.sv, si.u, si.su, pos, Gi, bad);
                    fx_flux(T, s0, s0.v, s0.sv, s0.u, s0.su, pos, G0, bad);
                    const int wh = (int)wq.z, wl = (int)wq.w, sh = pos ? wh : -wh, sl = pos ? wl : -wl;
                    fx_add(acc[0], sh, sl, Gi.rm, G0.rm);
                    fx_add(acc[2], wh, wl, Gi.ga, G0.ga);
                    fx_add(acc[1], sh, sl, Gi.go, G0.go);
                    fx_add(acc[3], sh, sl, Gi.g3, G0.g3);
                }
            }
        }
        double e1x, e1y, e2x, e2y;
        point_frame(d, kk, framed, e1x, e1y, e2x, e2y);
        double R[4];
#pragma unroll
        for (int c = 0; c < 4; c++) {
            acc[c].hh = group_sum<TPP>(acc[c].hh);
            acc[c].l = group_sum<TPP>(acc[c].l);
            acc[c].r = group_sum<TPP>(acc[c].r);
        }
        const double wsc = d.geo[G_WSC * ld + kk] * pow2(-(int)sh);
        R[0] = fx_total(acc[0]) * (wsc * 0x1p-27);
        R[3] = fx_total(acc[3]) * (wsc * 0x1p-23);
        const double Ra = fx_total(acc[1]) * (wsc * 0x1p-25), Ro = fx_total(acc[2]) * (wsc * 0x1p-25);
        R[1] = framed ? fma(Ra, e1x, Ro * e2x) : Ra;
        R[2] = framed ? fma(Ra, e1y, Ro * e2y) : Ro;
        // (work is the same for the lanes of a group; the whole warp takes part in the sums)
        bool slow = (bad >> 31) != 0;
#pragma unroll
        for (int o = TPP / 2; o > 0; o >>= 1) slow |= __shfl_xor_sync(kFull, (int)slow, o) != 0;
        if (__any_sync(kFull, slow)) {
            double Rs[4] = {0.0, 0.0, 0.0, 0.0};
            if (slow) residual_fp64<TPP>(d, q, g, kk, sub, second, Rs);
#pragma unroll
            for (int c = 0; c < 4; c++) {
                Rs[c] = group_sum<TPP>(Rs[c]);
                if (slow) R[c] = Rs[c];
            }
        }
        if (work && sub == 0) finish_residual<TPP>(d, st, k, fl, n1, e1x, e1y, e2x, e2y, R);
    }
}

// The residual of cases whose free stream is itself outside the fixed-point
// ranges (from M 2.86 on along an axis; decided per case at create): FP64
// throughout, the tables in shared memory.  Beside the fixed-point form every
// one of its points would be formed twice: 147,584 points at M 3.5 and 6
// 0.74 ms like this, 0.92 ms there (at M 2.5 the fixed-point form takes
// 0.22 ms).  128 threads, four blocks per SM (128 registers).
template <int TPP>
__global__ void __launch_bounds__(kRes64Block, 4) k_residual_fp64(Dev d, StateSet st, const double *__restrict__ g)
{
    __shared__ MathTables T;
    if (halted(d.ctrl)) return;
    load_math_tables(T);
    __syncthreads();
    const int n1 = ((const volatile Ctrl *)d.ctrl)->it;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = gt / TPP, sub = gt % TPP;
    const bool active = k < d.n;
    const int kk = active ? k : d.n - 1;
    const int fl = d.flag[kk];
    const bool work = active && (fl != kOuter || d.farfield == 1) && !frozen(d, kk) &&
                      (d.fp64_cases == 1 || hypersonic(d, kk));
    double R[4] = {0.0, 0.0, 0.0, 0.0};
    if (work) residual_slots<TPP>(d, T, st.q, g, kk, sub, n1 > d.first_order, R);
#pragma unroll
    for (int c = 0; c < 4; c++) R[c] = group_sum<TPP>(R[c]);
    if (work && sub == 0) {
        double e1x, e1y, e2x, e2y;
        point_frame(d, kk, fl != kInterior, e1x, e1y, e2x, e2y);
        finish_residual<TPP>(d, st, k, fl, n1, e1x, e1y, e2x, e2y, R);
    }
}

// ---------------------------------------------------------------------------
// per-case residual norms, histories and stopping tests (two stages)
// ---------------------------------------------------------------------------
// Stage 1: block j sums R_rho^2 over caller positions [blk_pos[j], blk_pos[j+1]),
// all of one case (frozen outer points hold R = 0).  Fixed order: warp butterfly,
// then warp 0.
__global__ void __launch_bounds__(256) k_norm_partials(Dev d)
{
    __shared__ double red[4][8];
    if (!counted(d.ctrl)) return;
    const int j = blockIdx.x;
    const int p = d.blk_pos[j] + threadIdx.x;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    if (p < d.blk_pos[j + 1]) {
        const int k = d.inv[p];
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const double r = d.R[c * d.ld + k];
            t[c] = r * r;
        }
    }
#pragma unroll
    for (int c = 0; c < 4; c++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t[c] += __shfl_xor_sync(kFull, t[c], o);
        if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = t[c];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int c = 0; c < 4; c++) {
            double s = threadIdx.x < 8 ? red[c][threadIdx.x] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
            if (threadIdx.x == 0) d.blk[4 * j + c] = s;
        }
    }
}

// Stage 2: one block per case adds the case's partials in a fixed order,
// records the norm and applies the stopping test.
__global__ void __launch_bounds__(256) k_norm_cases(Dev d)
{
    __shared__ double red[4][8];
    if (!counted(d.ctrl)) return;
    const int b = blockIdx.x;
    Ctrl *c = d.ctrl;
    if (frozen_state(((volatile int32_t *)c->case_state)[b])) return;  // block-uniform
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j = d.case_blk[b] + threadIdx.x; j < d.case_blk[b + 1]; j += blockDim.x)
#pragma unroll
        for (int q = 0; q < 4; q++) t[q] += d.blk[4 * j + q];
#pragma unroll
    for (int q = 0; q < 4; q++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t[q] += __shfl_xor_sync(kFull, t[q], o);
        if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = t[q];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double sq[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            sq[q] = threadIdx.x < 8 ? red[q][threadIdx.x] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sq[q] += __shfl_xor_sync(kFull, sq[q], o);
        }
        const double s = sq[0];
        if (threadIdx.x == 0) {
            const int n0 = c->case_it[b];
            if (n0 < c->hist_cap)
#pragma unroll
                for (int q = 0; q < 4; q++) c->hist4[((size_t)b * c->hist_cap + n0) * 4 + q] = sqrt(sq[q]);
            const double nrm = sqrt(s);
            const int n = c->case_it[b];
            if (n < c->hist_cap) c->hist[(size_t)b * c->hist_cap + n] = nrm;
            if (!(c->case_hist0[b] > 0.0)) c->case_hist0[b] = nrm;
            c->case_it[b] = n + 1;
            if (!isfinite(nrm) || d.suspect[b]) {
                if (c->n_cases > 1) {  // this case only: frozen from its sweeps on
                    c->case_state[b] = kFailed;
                    c->case_err[b] = -4;  // LSKUM_ERR_DIVERGED
                } else {
                    atomicExch(&c->error, -4);
                    atomicMin(&c->bad_point, -1 - b);
                }
            } else if (c->target > 0.0 && nrm / c->case_hist0[b] <= c->target) {
                atomicCAS(&c->case_state[b], (int32_t)kRunning, (int32_t)kReachedTarget);  // (not over a failed update)
            }
        }
    }
}

// ---------------------------------------------------------------------------
// LU-SGS sweep, one colour level; G lanes per point
// ---------------------------------------------------------------------------
// Positions [lb, le) of the level's point order (sw_fwd / sw_bwd).  The
// forward sweep sums over each point's lower list (neighbours earlier in the
// sweep order, whose dU* this sweep already produced), the backward sweep
// over its upper list (neighbours later in the order, dU already final).
// T is the sweep arithmetic: double, or float in the mixed-precision mode
// (increments, weights, primal records and Jacobian products in FP32; R and
// D are read in FP64 and rounded once per point).
template <typename T>
struct SweepBufs {
    T *dUs, *dU;
    const T *lo_w1, *lo_w2, *up_w1, *up_w2, *prim;
    T *jc;  // packed form's per-point axis products
};

template <typename T>
__device__ __forceinline__ SweepBufs<T> sweep_bufs(const Dev &d, const StateSet &st);

template <>
__device__ __forceinline__ SweepBufs<double> sweep_bufs<double>(const Dev &d, const StateSet &st)
{
    return {d.dUs, d.dU, d.lo_w1, d.lo_w2, d.up_w1, d.up_w2, st.prim, d.jc};
}

template <>
__device__ __forceinline__ SweepBufs<float> sweep_bufs<float>(const Dev &d, const StateSet &st)
{
    return {d.dUsf, d.dUf, d.lo_w1f, d.lo_w2f, d.up_w1f, d.up_w2f, st.primf, d.jcf};
}

// One slot of a point's lower / upper list: acc += w_s J_s(U_i) dW_i over the
// split sub-stencils s the slot joins (exact AD or increment products).
template <int JVP, typename T>
__device__ __forceinline__ void sweep_slot(const Dev &d, const StateSet &st, const MathTables &Tb,
                                           const T *dW, const T *__restrict__ pr, bool framed,
                                           double e1x, double e1y, double e2x, double e2y, int i, int mb, T w1,
                                           T w2, T acc[4])
{
    T dl[4];
    load4_l2(dW + 4 * (size_t)i, dl);
    if (JVP == 0 && !framed) {
        // interior frame: d = (1,0) or (0,1); A+-, exp(-S^2)/sqrt(pi), B,
        // 2 B S and u_d e1 precomputed per point
        const PrimT<T> P = load_prim(pr, i);
        const T *rec = pr + (size_t)i * kPrimStride;
        const JvpBase<T> jb = jvp_base(P, dl);
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const int m = s == 0 ? (mb & 3) : (mb >> 2);
            if (!m) continue;
            const bool pos = m & 1;
            T J[4];
            if (s == 0)
                jvp_axis<0, T>(P, jb, pos, rec[pos ? P_APX : P_AMX], rec[P_EKX], rec[P_BX], rec[P_BSX], rec[P_UE1],
                               J);
            else
                jvp_axis<1, T>(P, jb, pos, rec[pos ? P_APY : P_AMY], rec[P_EKY], rec[P_BY], rec[P_BSY], rec[P_VE1],
                               J);
            const T w = s == 0 ? w1 : w2;
#pragma unroll
            for (int c = 0; c < 4; c++) acc[c] = fma(w, J[c], acc[c]);
        }
    } else {
        // (t, n) frames and the increment form: evaluated in FP64
        double dld[4];
#pragma unroll
        for (int c = 0; c < 4; c++) dld[c] = (double)dl[c];
        const int ld = d.ld;
        double Ui[4], Up[4];
        PrimU P;
        JvpBase<double> jb{};
        if (JVP == 0) {
            P = load_prim(st.prim, i);
            jb = jvp_base(P, dld);
        } else {
#pragma unroll
            for (int c = 0; c < 4; c++) {
                Ui[c] = st.U[c * ld + i];
                Up[c] = Ui[c] + dld[c];
            }
        }
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const int m = s == 0 ? (mb & 3) : (mb >> 2);
            if (!m) continue;
            const bool pos = m & 1;
            const double sg = pos ? 1.0 : -1.0;
            const double ddx = s == 0 ? e1x : e2x, ddy = s == 0 ? e1y : e2y;
            double J[4];
            if (JVP == 0) {
                const double S = (P.u * ddx + P.v * ddy) * P.sb;
                double A, eS;
                split_A(Tb, S, pos, A, eS);
                jvp_dir(P, jb, ddx, ddy, sg, S, A, eS, eS * kInv2SqrtPi * P.isb, J);
            } else {
                double G1[4], G0[4];
                flux_cons(Tb, Up, ddx, ddy, pos, G1);
                flux_cons(Tb, Ui, ddx, ddy, pos, G0);
#pragma unroll
                for (int c = 0; c < 4; c++) J[c] = G1[c] - G0[c];
            }
            const T w = s == 0 ? w1 : w2;
#pragma unroll
            for (int c = 0; c < 4; c++) acc[c] = fma(w, (T)J[c], acc[c]);
        }
    }
}

// Point k's new increment from its list sum acc: forward dU*_k = -(R_k (+ S_k)
// + acc) / D_k, backward dU_k = dU*_k - acc / D_k; normal momentum removed at
// wall points.  Stored, and returned in w.
template <typename T>
__device__ __forceinline__ void sweep_point(bool FWD, const Dev &d, const StateSet &st, const SweepBufs<T> &sb, int k,
                                            bool wall, double e1x, double e1y, double e2x, double e2y,
                                            const T acc[4], T w[4])
{
    const int ld = d.ld;
    const T iD = (T)d.iD[k];
    if (FWD) {
        double rhs[4];
#pragma unroll
        for (int c = 0; c < 4; c++) rhs[c] = d.R[c * ld + k];
        if (d.lusgs == 1) {
            // revised LU-SGS: -R - S with S_0 = -1/2 sum_s LS_s(1) A_d(U_0) dU_0 of
            // the previous iteration's increment (still in dU: the backward
            // sweep of this iteration has not run)
            double dp[4];
#pragma unroll
            for (int c = 0; c < 4; c++) dp[c] = d.dUf ? (double)d.dUf[4 * k + c] : d.dU[4 * k + c];
            const double *pk = st.prim + (size_t)k * kPrimStride;
            double J1[4], J2[4];
            euler_jvp(pk[P_RHO], pk[P_U], pk[P_V], pk[P_P], dp, e1x, e1y, J1);
            euler_jvp(pk[P_RHO], pk[P_U], pk[P_V], pk[P_P], dp, e2x, e2y, J2);
            const double l1 = d.geo[G_LS1_0 * ld + k] + d.geo[G_LS1_1 * ld + k];
            const double l2 = d.geo[G_LS1_2 * ld + k] + d.geo[G_LS1_3 * ld + k];
#pragma unroll
            for (int c = 0; c < 4; c++) rhs[c] -= 0.5 * (l1 * J1[c] + l2 * J2[c]);  // R + S
        }
#pragma unroll
        for (int c = 0; c < 4; c++) w[c] = -((T)rhs[c] + acc[c]) * iD;
    } else {
#pragma unroll
        for (int c = 0; c < 4; c++) w[c] = fma(-acc[c], iD, load_l2(sb.dUs + 4 * (size_t)k + c));
    }
    if (wall) {
        const T nx = (T)d.wnx[k], ny = (T)d.wny[k];
        const T mn = w[1] * nx + w[2] * ny;
        w[1] -= mn * nx;
        w[2] -= mn * ny;
    }
    T *out = FWD ? sb.dUs : sb.dU;
#pragma unroll
    for (int c = 0; c < 4; c++) out[4 * k + c] = w[c];
}

// G lanes per point over the point's list, butterfly reduction.
template <int JVP, bool FWD, int G, typename T>
__global__ void __launch_bounds__(256) k_sweep(Dev d, StateSet st, int lb, int le)
{
    const MathTables &Tb = g_math;  // wall and outer points only: no per-block copy
    if (halted_step(d)) return;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    if (lb + (gt & ~31) / G >= le) return;  // the whole warp is past the level
    const int pos = lb + gt / G, sub = gt % G;
    const bool active = pos < le;
    const int k = (FWD ? d.sw_fwd : d.sw_bwd)[active ? pos : le - 1];
    const bool live = active && !frozen_step(d, k);
    const SweepBufs<T> sb = sweep_bufs<T>(d, st);
    const int32_t *__restrict__ off = FWD ? d.lo_off : d.up_off;
    const int32_t *__restrict__ nbr = FWD ? d.lo_nbr : d.up_nbr;
    const uint8_t *__restrict__ mbs = FWD ? d.lo_mb : d.up_mb;
    const T *__restrict__ w1s = FWD ? sb.lo_w1 : sb.up_w1;
    const T *__restrict__ w2s = FWD ? sb.lo_w2 : sb.up_w2;
    const T *__restrict__ dW = FWD ? sb.dUs : sb.dU;
    const int fk = d.flag[k];
    const bool wall = fk == kWall, framed = fk != kInterior;
    double e1x, e1y, e2x, e2y;
    point_frame(d, k, framed, e1x, e1y, e2x, e2y);
    T acc[4] = {T(0), T(0), T(0), T(0)};
    const int beg = off[k], end = live ? off[k + 1] : beg;
    for (int e = beg + sub; e < end; e += G)
        sweep_slot<JVP, T>(d, st, Tb, dW, sb.prim, framed, e1x, e1y, e2x, e2y, nbr[e], mbs[e], w1s[e], w2s[e], acc);
#pragma unroll
    for (int c = 0; c < 4; c++) acc[c] = group_sum<G>(acc[c]);
    T w[4];
    if (live && sub == 0) sweep_point<T>(FWD, d, st, sb, k, wall, e1x, e1y, e2x, e2y, acc, w);
}

// Axis product cb (0: x+, 1: x-, 2: y+, 3: y-) of point k's new increment w
// in the increment form, G_d(U_k + w) - G_d(U_k) in FP64 (the value an
// interior point whose list holds k would form for that sub-stencil),
// stored once for every later level to gather.  (The exact products are
// formed by jvp_axis_sel from the point's record, or from the framed
// points' precomputed Jacobians.)
template <typename T>
__device__ __forceinline__ void store_increment_product(const MathTables &Tb, const SweepBufs<T> &sb, const PrimU &P,
                                                        const double G0[4], int k, int cb)
{
    double G1[4];
    flux_prim(Tb, P, cb < 2 ? 1.0 : 0.0, cb < 2 ? 0.0 : 1.0, !(cb & 1), G1);
    T J[4];
#pragma unroll
    for (int c = 0; c < 4; c++) J[c] = (T)(G1[c] - G0[c]);
    store4(sb.jc + 16 * (size_t)k + 4 * cb, J);
}

// Split fluxes at the state of this iteration, which the increment products
// subtract: of every point along the axes (g0), and of every framed slot's
// neighbour in the point's frame (pk_g0).  They do not depend on the sweeps'
// increments, so they are formed beside the q-derivatives and the residual,
// whose integer work leaves the FP64 unit idle, instead of twice per point on
// the sweeps' critical path (41,194 points, an iteration: 0.804 ms with them
// there, 0.519 like this and with prim_short's chain).
__host__ __device__ inline int increment_base_items(const Dev &d)
{
    return 4 * d.n + 2 * (d.pk_lanes[0] + d.pk_lanes[1]);
}
__global__ void __launch_bounds__(256) k_increment_base(Dev d, StateSet st)
{
    __shared__ MathTables Tb;
    if (halted(d.ctrl)) return;
    load_math_tables(Tb);
    __syncthreads();
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= increment_base_items(d)) return;
    double dx, dy;
    bool pos;
    int i;
    double *out;
    if (t < 4 * d.n) {
        i = t >> 2;
        pos = !(t & 1);
        dx = t & 2 ? 0.0 : 1.0;
        dy = t & 2 ? 1.0 : 0.0;
        out = d.g0 + 4 * (size_t)t;
    } else {
        t -= 4 * d.n;
        const int dir = t >= 2 * d.pk_lanes[0];
        t -= dir ? 2 * d.pk_lanes[0] : 0;
        const int e = t >> 1, k = d.pk_k[dir][e], m = t & 1 ? d.pk_mb[dir][e] >> 2 : d.pk_mb[dir][e] & 3;
        if (k < 0 || !m) return;
        i = d.pk_nbr[dir][e];
        pos = m & 1;
        dx = d.geo[(t & 1 ? G_E2X : G_E1X) * d.ld + k];
        dy = d.geo[(t & 1 ? G_E2Y : G_E1Y) * d.ld + k];
        out = d.pk_g0[dir] + 4 * (size_t)t;
    }
    double U[4], G[4];
#pragma unroll
    for (int c = 0; c < 4; c++) U[c] = st.U[c * d.ld + i];
    flux_prim(Tb, prim_short(U), dx, dy, pos, G);
    store4(out, G);
}

// Jacobians of the framed points' products (exact products).  The split-flux
// Jacobian A_d^+-(U_i) is the derivative of G_d^+- at the state of this
// iteration and does not depend on the sweeps' increments, so every matrix
// that the two sweeps apply at the points in a (t, n) frame is formed all in
// parallel before the forward sweep; inside the levels the framed points'
// chains are then matrix-vector products.  Item t: one column of pk_jm of a
// slot lane -- M = w1 A_e1 + w2 A_e2 at the neighbour's state in the point's
// frame -- or of fj of a framed point and axis product -- A_x+-, A_y+- at the
// point's own state.  Column j is the forward-mode tangent along the unit
// vector e_j, evaluated in FP64 by the functions of the per-slot form (stored
// as T).
__host__ __device__ inline int framed_jac_items(const Dev &d)
{
    return 4 * (d.pk_lanes[0] + d.pk_lanes[1]) + 16 * d.nf;
}

template <typename T>
__device__ __forceinline__ void framed_jac_item(const Dev &d, const StateSet &st, const MathTables &Tb, int t)
{
    const int n0 = 4 * d.pk_lanes[0], n1 = 4 * d.pk_lanes[1];
    const int j = t & 3;  // n0 and n1 are multiples of 4
    double dl[4];
#pragma unroll
    for (int c = 0; c < 4; c++) dl[c] = c == j ? 1.0 : 0.0;  // the unit vector e_j
    if (t < n0 + n1) {
        const int dir = t < n0 ? 0 : 1;
        const int e = (t - (dir ? n0 : 0)) >> 2;
        T *M = (sizeof(T) == 4 ? (T *)d.pk_jmf[dir] : (T *)d.pk_jm[dir]) + 16 * (size_t)e;
        const int pos = d.pk_pt[dir][e];
        const int mb = d.pk_mb[dir][e];
        double col[4] = {0.0, 0.0, 0.0, 0.0};
        if (pos >= 0 && mb) {
            const int k = (dir == 0 ? d.sw_fwd : d.sw_bwd)[pos];
            double e1x, e1y, e2x, e2y;
            point_frame(d, k, true, e1x, e1y, e2x, e2y);
            const PrimU P = load_prim(st.prim, d.pk_nbr[dir][e]);
            const JvpBase<double> jb = jvp_base(P, dl);
#pragma unroll
            for (int s = 0; s < 2; s++) {
                const int m = s == 0 ? (mb & 3) : (mb >> 2);
                if (!m) continue;
                const bool pos_s = m & 1;
                const double sg = pos_s ? 1.0 : -1.0;
                const double ddx = s == 0 ? e1x : e2x, ddy = s == 0 ? e1y : e2y;
                const double S = (P.u * ddx + P.v * ddy) * P.sb;
                double A, eS, J[4];
                split_A(Tb, S, pos_s, A, eS);
                jvp_dir(P, jb, ddx, ddy, sg, S, A, eS, eS * kInv2SqrtPi * P.isb, J);
                const double w = s == 0 ? d.pk_w1[dir][e] : d.pk_w2[dir][e];
#pragma unroll
                for (int c = 0; c < 4; c++) col[c] = fma(w, J[c], col[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < 4; c++) M[4 * c + j] = (T)col[c];
        return;
    }
    const int u = t - n0 - n1;
    const int f = u >> 4, cb = (u >> 2) & 3;
    const int k = d.fpt[f];
    const PrimU P = load_prim(st.prim, k);
    const double *rec = st.prim + (size_t)k * kPrimStride;
    const JvpBase<double> jb = jvp_base(P, dl);
    const bool pos = !(cb & 1);
    double J[4];
    if (cb < 2)
        jvp_axis<0, double>(P, jb, pos, rec[pos ? P_APX : P_AMX], rec[P_EKX], rec[P_BX], rec[P_BSX], rec[P_UE1], J);
    else
        jvp_axis<1, double>(P, jb, pos, rec[pos ? P_APY : P_AMY], rec[P_EKY], rec[P_BY], rec[P_BSY], rec[P_VE1], J);
    T *F = (sizeof(T) == 4 ? (T *)d.fjf : (T *)d.fj) + 64 * (size_t)f + 16 * cb;
#pragma unroll
    for (int c = 0; c < 4; c++) F[4 * c + j] = (T)J[c];
}

template <typename T>
__global__ void __launch_bounds__(256) k_framed_jac(Dev d, StateSet st)
{
    __shared__ MathTables Tb;
    if (halted(d.ctrl)) return;
    load_math_tables(Tb);
    __syncthreads();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < framed_jac_items(d)) framed_jac_item<T>(d, st, Tb, t);
}

// Most threads per block of the sweeps' launch: two warps per scheduler keep
// the FP64 unit busy, and 255 registers hold what is loaded ahead.
constexpr int kSweepBlock = 256;

// A level boundary in two halves: every thread of a block arrives, then (after
// work that needs nothing of the other blocks) waits until all blocks of the
// launch have arrived with their stores visible (cooperative launch: all
// blocks are resident).  The arrivals are counted in ctrl->sweep_bar; the
// launch's last one (number `limit`) wraps it to 0 for the next launch.  The
// block's last warp arrives and polls for it.  The arrival releases the
// block's stores (the barrier before it orders them all before the one
// thread's release).  The poll is relaxed; the load that follows it acquires
// what the arrivals released, and the barrier behind it hands that on to the
// block's other threads.  The acquire empties L1; what was loaded ahead for a
// warp's first task of the level lies in registers and shared memory.
__device__ __forceinline__ void boundary_arrive(Ctrl *c, uint32_t limit, bool skip)
{
    __syncthreads();
    if (threadIdx.x == blockDim.x - 32 && !skip) {
        asm volatile("red.release.gpu.global.inc.u32 [%0], %1;" ::"l"(&c->sweep_bar), "r"(limit - 1) : "memory");
    }
}

// False past the time limit.
__device__ __forceinline__ bool boundary_wait(Ctrl *c, uint32_t target, uint32_t limit, uint64_t wait_ns)
{
    __shared__ int reached;
    if (threadIdx.x == blockDim.x - 32) {
        const volatile uint32_t *bar = &c->sweep_bar;
        uint64_t t0 = 0;
        int ok = 1;
        for (uint32_t tries = 1;; tries++) {
            uint32_t v = *bar;
            if (target == limit ? v == 0 : v >= target) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&c->sweep_bar) : "memory");
                break;
            }
            if ((tries & 1023) == 0) {
                uint64_t now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                if (now - t0 > wait_ns) {
                    atomicExch(&c->error, kErrTimeout);
                    ok = 0;
                    break;
                }
            }
        }
        reached = ok;
    }
    __syncthreads();
    return reached != 0;
}

// 16 bytes (8, for float2) of global memory into shared memory; .cg: from L2
// (values that other blocks write within the launch).
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <typename T>
struct Pair2;
template <>
struct Pair2<double> {
    using type = double2;
};
template <>
struct Pair2<float> {
    using type = float2;
};

// A warp's shared memory: the products of kDepth rows of slots in flight (two
// of kChunks 16-byte words per lane and row, a warp's lanes apart: conflict-
// free), and the weights of the first kRows rows.
constexpr int kDepth = 5, kRows = 10;
template <typename T>
constexpr int kChunks = 4 * (int)sizeof(T) / 16;
template <typename T>
struct WarpStage {
    uint4 J[kDepth][2 * kChunks<T>][32];
    typename Pair2<T>::type w[kRows][32];
};

// What a lane of an interior point's group reads that no block writes within
// the launch, loaded while the block waits at the level boundary: the point
// (-1: none, or frozen), the first kRows slots of its share of the list
// (their weights into shared memory), its entries of the point's primal
// record, its components of R and 1/D.
template <typename T>
struct LanePre {
    int k, rows;
    size_t base;
    uint32_t nm[kRows];
    PrimT<T> P;
    T Ap, Am, EK, B, BS, UE, iD;
    double R[2];
    double U[4], G0[8];  // increment products: the state, the fluxes of the lane's products there
};

template <int JVP, int L, typename T>
__device__ __forceinline__ void lane_load(const Dev &d, const StateSet &st, const SweepBufs<T> &sb, int dir, int g, int lane,
                                          WarpStage<T> &ws, LanePre<T> &a)
{
    const int p = lane / L, s = lane % L;
    a.k = d.lp_k[dir][kGroupPoints * g + p];
    const int len = a.k >= 0 ? d.lp_len[dir][kGroupPoints * g + p] : 0;
    const int off = d.lp_goff[dir][g];
    a.rows = (d.lp_goff[dir][g + 1] - off) / 32;  // the same for the warp
    a.base = (size_t)off + lane;
    if (a.k >= 0 && frozen_step(d, a.k)) a.k = -1;
    const int kk = a.k >= 0 ? a.k : 0;  // index for the loads of a slot without a point
#pragma unroll
    for (int r = 0; r < kRows; r++) {
        a.nm[r] = 0;
        if (a.k >= 0 && s + L * r < len) {
            const size_t e = a.base + 32 * r;
            a.nm[r] = d.lp_nm[dir][e];
            if (sizeof(T) == 4) cp_async8(&ws.w[r][lane], d.lp_wf[dir] + e);
            else cp_async16(&ws.w[r][lane], d.lp_w[dir] + e);
        }
    }
    cp_async_commit();
    if (JVP == 0) {
        const bool xdir = L == 2 ? s == 0 : s < 2, psg = !(s & 1);
        a.P = load_prim(sb.prim, kk);
        const T *rec = sb.prim + (size_t)kk * kPrimStride;
        if (L == 2) {
            a.Ap = rec[xdir ? P_APX : P_APY];
            a.Am = rec[xdir ? P_AMX : P_AMY];
        } else {
            a.Ap = rec[xdir ? (psg ? P_APX : P_AMX) : (psg ? P_APY : P_AMY)];
        }
        a.EK = rec[xdir ? P_EKX : P_EKY];
        a.B = rec[xdir ? P_BX : P_BY];
        a.BS = rec[xdir ? P_BSX : P_BSY];
        a.UE = rec[xdir ? P_UE1 : P_VE1];
    }
    if (JVP == 1) {
#pragma unroll
        for (int c = 0; c < 4; c++) a.U[c] = st.U[c * d.ld + kk];
#pragma unroll
        for (int c = 0; c < 4 / L; c++) load4(d.g0 + 16 * (size_t)kk + 4 * (4 / L * s + c), a.G0 + 4 * c);
    }
    a.iD = (T)d.iD[kk];
#pragma unroll
    for (int c = 0; c < 4 / L; c++) a.R[c] = dir == 0 ? d.R[(4 / L * s + c) * d.ld + kk] : 0.0;
}

// A slot's products of its neighbour (this sweep's earlier levels) into the stage.
template <typename T>
__device__ __forceinline__ void slot_fetch(const T *jc, uint32_t nm, uint4 (*to)[32], int lane)
{
    const size_t i = 16 * (size_t)(nm & 0x0fffffffu);
    const uint32_t mb = nm >> 28;
    if (mb & 3) {
        const T *J = jc + i + ((mb & 1) ? 0 : 4);
#pragma unroll
        for (int c = 0; c < kChunks<T>; c++) cp_async16(&to[c][lane], J + 16 / sizeof(T) * c);
    }
    if (mb & 12) {
        const T *J = jc + i + ((mb & 4) ? 8 : 12);
#pragma unroll
        for (int c = 0; c < kChunks<T>; c++) cp_async16(&to[kChunks<T> + c][lane], J + 16 / sizeof(T) * c);
    }
}
__device__ __forceinline__ void stage_read(const uint4 (*from)[32], int lane, double J[4])
{
    const double2 a = *reinterpret_cast<const double2 *>(&from[0][lane]);
    const double2 b = *reinterpret_cast<const double2 *>(&from[1][lane]);
    J[0] = a.x, J[1] = a.y, J[2] = b.x, J[3] = b.y;
}
__device__ __forceinline__ void stage_read(const uint4 (*from)[32], int lane, float J[4])
{
    const float4 a = *reinterpret_cast<const float4 *>(&from[0][lane]);
    J[0] = a.x, J[1] = a.y, J[2] = a.z, J[3] = a.w;
}

// A slot's products in the stage, weighted, into acc.
template <typename T>
__device__ __forceinline__ void slot_add(uint32_t nm, typename Pair2<T>::type w, const uint4 (*from)[32], int lane,
                                         T acc[4])
{
    T J[4];
    if ((nm >> 28) & 3) {
        stage_read(from, lane, J);
#pragma unroll
        for (int c = 0; c < 4; c++) acc[c] = fma(w.x, J[c], acc[c]);
    }
    if ((nm >> 28) & 12) {
        stage_read(from + kChunks<T>, lane, J);
#pragma unroll
        for (int c = 0; c < 4; c++) acc[c] = fma(w.y, J[c], acc[c]);
    }
}

// One group of 32 / L interior points, L lanes each (2 or 4).  Whatever L, a
// point's sum is (a0 + a1) + (a2 + a3), a_m the sum of its slots j = m (mod 4)
// in order: with two lanes, lane s keeps a_s and a_{s+2}.
template <int JVP, int L, typename T>
__device__ __forceinline__ void sweep_interior(const Dev &d, const StateSet &st, const SweepBufs<T> &sb, int dir,
                                               int lane, const LanePre<T> &a, WarpStage<T> &ws)
{
    constexpr int C = 4 / L;  // components that a lane finishes
    const int s = lane % L, k = a.k;
    const bool live = k >= 0;
    const bool fwd = dir == 0, plain = d.lusgs == 0;  // the revised LU-SGS adds its lagged term in sweep_point
    T acc[C][4], dus[C];
#pragma unroll
    for (int h = 0; h < C; h++) {
        dus[h] = T(0);
#pragma unroll
        for (int c = 0; c < 4; c++) acc[h][c] = T(0);
    }
#pragma unroll
    for (int r = 0; r < kDepth; r++) {
        slot_fetch(sb.jc, a.nm[r], ws.J[r], lane);
        cp_async_commit();
    }
    if (live && !fwd)
#pragma unroll
        for (int c = 0; c < C; c++) dus[c] = load_l2(sb.dUs + 4 * (size_t)k + C * s + c);
#pragma unroll
    for (int r = 0; r < kRows; r++) {
        if (r >= a.rows) break;
        cp_async_wait<kDepth - 1>();
        slot_add(a.nm[r], ws.w[r][lane], ws.J[r % kDepth], lane, acc[r % C]);
        if (r + kDepth < kRows) slot_fetch(sb.jc, a.nm[r + kDepth], ws.J[r % kDepth], lane);
        cp_async_commit();
    }
#pragma unroll 1
    for (int r = kRows; r < a.rows; r++) {  // lists longer than kRows L slots (padding has membership 0)
        const size_t e = a.base + 32 * (size_t)r;
        const uint32_t nm = live ? d.lp_nm[dir][e] : 0u;
        typename Pair2<T>::type w;
        if (sizeof(T) == 4) w.x = (T)d.lp_wf[dir][e].x, w.y = (T)d.lp_wf[dir][e].y;
        else w.x = (T)d.lp_w[dir][e].x, w.y = (T)d.lp_w[dir][e].y;
        slot_fetch(sb.jc, nm, ws.J[0], lane);
        cp_async_commit();
        cp_async_wait<0>();
        if (C == 2 && (r & 1)) slot_add(nm, w, ws.J[0], lane, acc[C - 1]);
        else slot_add(nm, w, ws.J[0], lane, acc[0]);
    }
    cp_async_wait<0>();
    // lane s gets components C s, ... of the lanes' sum
    T sum[C];
    if (L == 4) {
        const bool odd = s & 1, high = s & 2;
        const T p0 = (odd ? acc[0][1] : acc[0][0]) + __shfl_xor_sync(kFull, odd ? acc[0][0] : acc[0][1], 1);
        const T p1 = (odd ? acc[0][3] : acc[0][2]) + __shfl_xor_sync(kFull, odd ? acc[0][2] : acc[0][3], 1);
        sum[0] = (high ? p1 : p0) + __shfl_xor_sync(kFull, high ? p0 : p1, 2);
    } else {
#pragma unroll
        for (int c = 0; c < C; c++) {
            T pr[C];
#pragma unroll
            for (int h = 0; h < C; h++)
                pr[h] = (s ? acc[h][2 + c] : acc[h][c]) + __shfl_xor_sync(kFull, s ? acc[h][c] : acc[h][2 + c], 1);
            sum[c] = pr[0] + pr[C - 1];
        }
    }
    T w[4];
    if (plain) {
        // forward dU* = -(R + acc) / D, backward dU = dU* - acc / D
        T *out = (fwd ? sb.dUs : sb.dU) + 4 * (size_t)(live ? k : 0) + C * s;
        T wn[C];
#pragma unroll
        for (int c = 0; c < C; c++) wn[c] = fwd ? -((T)a.R[c] + sum[c]) * a.iD : fma(-sum[c], a.iD, dus[c]);
        if (live) {
#pragma unroll
            for (int c = 0; c < C; c++) out[c] = wn[c];
        }
#pragma unroll
        for (int c = 0; c < 4; c++) w[c] = __shfl_sync(kFull, wn[c % C], lane - s + c / C);
    } else {
        T tot[4];
#pragma unroll
        for (int c = 0; c < 4; c++) tot[c] = __shfl_sync(kFull, sum[c % C], lane - s + c / C), w[c] = T(0);
        if (live && s == 0) sweep_point<T>(fwd, d, st, sb, k, false, 1.0, 0.0, 0.0, 1.0, tot, w);
#pragma unroll
        for (int c = 0; c < 4; c++) w[c] = __shfl_sync(kFull, w[c], lane - s);
    }
    if (!live) return;
    if (JVP == 0) {
        const JvpBase<T> jb = jvp_base(a.P, w);
        T J[4];
        if (L == 4) {
            jvp_axis_sel<T>(a.P, jb, s < 2, !(s & 1), a.Ap, a.EK, a.B, a.BS, a.UE, J);
            store4(sb.jc + 16 * (size_t)k + 4 * s, J);
        } else {
            T Jm[4];
            jvp_axis_pair<T>(a.P, jb, s == 0, a.Ap, a.Am, a.EK, a.B, a.BS, a.UE, J, Jm);
            store4(sb.jc + 16 * (size_t)k + 8 * s, J);
            store4(sb.jc + 16 * (size_t)k + 8 * s + 4, Jm);
        }
    } else {
        double Up[4];
#pragma unroll
        for (int c = 0; c < 4; c++) Up[c] = a.U[c] + (double)w[c];
        const PrimU P = prim_short(Up);
#pragma unroll
        for (int c = 0; c < C; c++) store_increment_product<T>(g_math, sb, P, a.G0 + 4 * c, k, C * s + c);
    }
}

// A warp of packed slots of points in a (t, n) frame, exact products: what
// the level boundary does not change, loaded while the block waits there.
// The slot's point (-1: none, or frozen), its place among the point's lanes
// (r of seg, from lane head), the slot's neighbour and weighted Jacobian, the
// axis Jacobian that the lane applies, and in the point's first lane R, 1/D
// and the wall normal.
template <typename T>
struct FramedPre {
    int k, f, nb, steps, head, seg, r;
    bool slot, wall;
    T M[16], F[16], iD, nx, ny;
    double R[4];
};

template <typename T>
__device__ __forceinline__ const T *axis_jacobians(const Dev &d, int f)
{
    return (sizeof(T) == 4 ? (const T *)d.fjf : (const T *)d.fj) + 64 * (size_t)f;
}

template <typename T>
__device__ __forceinline__ void framed_load(const Dev &d, int dir, int fw, int lane, FramedPre<T> &a)
{
    const size_t e = (size_t)fw * 32 + lane;
    a.k = d.pk_k[dir][e];
    const int f2 = d.pk_f[dir][e];
    a.f = f2 >> 1;
    a.wall = f2 & 1;
    a.nb = d.pk_nbr[dir][e];
    a.slot = d.pk_mb[dir][e] != 0;
    a.steps = d.pk_steps[dir][fw];
    const T *M = (sizeof(T) == 4 ? (const T *)d.pk_jmf[dir] : (const T *)d.pk_jm[dir]) + 16 * e;
#pragma unroll
    for (int c = 0; c < 4; c++) load4_l2(M + 4 * c, a.M + 4 * c);
    const unsigned m = __match_any_sync(kFull, a.k);
    a.head = __ffs(m) - 1;
    a.seg = __popc(m);
    a.r = lane - a.head;
    const int k = a.k;
    if (k < 0) {
        a.slot = false;
        return;
    }
    if (a.r < 4) {
        const T *F = axis_jacobians<T>(d, a.f) + 16 * a.r;
#pragma unroll
        for (int c = 0; c < 4; c++) load4_l2(F + 4 * c, a.F + 4 * c);
    }
    if (a.r == 0) {
        a.iD = (T)d.iD[k];
        if (a.wall) {
            a.nx = (T)d.wnx[k];
            a.ny = (T)d.wny[k];
        }
#pragma unroll
        for (int c = 0; c < 4; c++) a.R[c] = dir == 0 ? d.R[c * d.ld + k] : 0.0;
    }
    if (frozen_step(d, k)) a.k = -1, a.slot = false;
}

template <typename T>
__device__ __forceinline__ void mat_vec(const T M[16], const T w[4], T J[4])
{
#pragma unroll
    for (int c = 0; c < 4; c++) {
        J[c] = M[4 * c] * w[0];
#pragma unroll
        for (int j = 1; j < 4; j++) J[c] = fma(M[4 * c + j], w[j], J[c]);
    }
}

template <typename T>
__device__ __forceinline__ void framed_run(const Dev &d, const SweepBufs<T> &sb, int dir, int lane,
                                           const FramedPre<T> &a)
{
    const bool fwd = dir == 0, live = a.k >= 0;
    const int k = a.k;
    T acc[4] = {T(0), T(0), T(0), T(0)}, dus[4] = {T(0), T(0), T(0), T(0)}, dl[4] = {T(0), T(0), T(0), T(0)};
    if (a.slot) load4_l2((fwd ? sb.dUs : sb.dU) + 4 * (size_t)a.nb, dl);  // earlier levels' increments
    if (live && a.r == 0 && !fwd) load4_l2(sb.dUs + 4 * (size_t)k, dus);
    if (a.slot) {
#pragma unroll
        for (int c = 0; c < 4; c++)
#pragma unroll
            for (int j = 0; j < 4; j++) acc[c] = fma(a.M[4 * c + j], dl[j], acc[c]);
    }
    // segmented suffix sum: lane l adds lane l + o of the same point; the
    // warp's longest list bounds the steps (warp-uniform)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        if (o >= (1 << a.steps)) break;
        T v[4];
#pragma unroll
        for (int c = 0; c < 4; c++) v[c] = __shfl_down_sync(kFull, acc[c], o);
        if (a.r + o < a.seg) {
#pragma unroll
            for (int c = 0; c < 4; c++) acc[c] += v[c];
        }
    }
    T w[4] = {T(0), T(0), T(0), T(0)};
    if (live && a.r == 0) {  // the point's first lane finishes it
#pragma unroll
        for (int c = 0; c < 4; c++) w[c] = fwd ? -((T)a.R[c] + acc[c]) * a.iD : fma(-acc[c], a.iD, dus[c]);
        if (a.wall) {
            const T mn = w[1] * a.nx + w[2] * a.ny;
            w[1] -= mn * a.nx;
            w[2] -= mn * a.ny;
        }
        store4((fwd ? sb.dUs : sb.dU) + 4 * (size_t)k, w);
    }
#pragma unroll
    for (int c = 0; c < 4; c++) w[c] = __shfl_sync(kFull, w[c], a.head);
    if (!live) return;
    // lane r of the point's seg lanes forms the axis products r, r + seg, ...
    T J[4];
    if (a.r < 4) {
        mat_vec(a.F, w, J);
        store4(sb.jc + 16 * (size_t)k + 4 * a.r, J);
    }
#pragma unroll 1
    for (int cb = a.r + a.seg; cb < 4; cb += a.seg) {
        const T *F = axis_jacobians<T>(d, a.f) + 16 * cb;
        T Fc[16];
#pragma unroll
        for (int c = 0; c < 4; c++) load4_l2(F + 4 * c, Fc + 4 * c);
        mat_vec(Fc, w, J);
        store4(sb.jc + 16 * (size_t)k + 4 * cb, J);
    }
}

// The same for the increment products and for the revised LU-SGS.
template <int JVP, typename T>
__device__ __noinline__ void sweep_framed(const Dev &d, const StateSet &st, const SweepBufs<T> &sb, int dir, int fw,
                                          int lane)
{
    const bool fwd = dir == 0;
    const T *dW = fwd ? sb.dUs : sb.dU;  // earlier levels' increments
    T acc[4] = {T(0), T(0), T(0), T(0)};
    T w[4] = {T(0), T(0), T(0), T(0)};
    const size_t e = (size_t)fw * 32 + lane;
    const int pos = d.pk_pt[dir][e];  // sweep position of the slot's point, -1: padding
    const int k = pos >= 0 ? (fwd ? d.sw_fwd : d.sw_bwd)[pos] : 0;
    const bool live = pos >= 0 && !frozen_step(d, k);
    const int fk = d.flag[k];
    const bool wall = fk == kWall, framed = fk != kInterior;
    double e1x, e1y, e2x, e2y;
    point_frame(d, k, framed, e1x, e1y, e2x, e2y);
    const int mb = d.pk_mb[dir][e];
    if (live && mb) {
        if (JVP == 0) {
            // the slot's weighted Jacobian, formed before the sweeps: acc += M dW_i
            const T *M = (sizeof(T) == 4 ? (const T *)d.pk_jmf[dir] : (const T *)d.pk_jm[dir]) + 16 * e;
            T dl[4];
            load4_l2(dW + 4 * (size_t)d.pk_nbr[dir][e], dl);
#pragma unroll
            for (int c = 0; c < 4; c++) {
                T Mc[4];
                load4_l2(M + 4 * c, Mc);
#pragma unroll
                for (int j = 0; j < 4; j++) acc[c] = fma(Mc[j], dl[j], acc[c]);
            }
        } else {
            const T w1 = sizeof(T) == 4 ? (T)d.pk_w1f[dir][e] : (T)d.pk_w1[dir][e];
            const T w2 = sizeof(T) == 4 ? (T)d.pk_w2f[dir][e] : (T)d.pk_w2[dir][e];
            const int i = d.pk_nbr[dir][e];
            T dl[4];
            load4_l2(dW + 4 * (size_t)i, dl);
            double Up[4];
#pragma unroll
            for (int c = 0; c < 4; c++) Up[c] = st.U[c * d.ld + i] + (double)dl[c];
            const PrimU P = prim_short(Up);
#pragma unroll
            for (int s = 0; s < 2; s++) {
                const int m = s == 0 ? (mb & 3) : (mb >> 2);
                if (!m) continue;
                double G1[4], G0[4];
                load4(d.pk_g0[dir] + 8 * e + 4 * s, G0);
                flux_prim(g_math, P, s == 0 ? e1x : e2x, s == 0 ? e1y : e2y, m & 1, G1);
#pragma unroll
                for (int c = 0; c < 4; c++) acc[c] = fma(s == 0 ? w1 : w2, (T)(G1[c] - G0[c]), acc[c]);
            }
        }
    }
    // segmented suffix sum: lane l adds lane l + o when both hold the same
    // point; the warp's longest list bounds the steps (warp-uniform)
    const int steps = d.pk_steps[dir][fw];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        if (o >= (1 << steps)) break;
        const int p2 = __shfl_down_sync(kFull, pos, o);
        T v[4];
#pragma unroll
        for (int c = 0; c < 4; c++) v[c] = __shfl_down_sync(kFull, acc[c], o);
        if (lane + o < 32 && p2 == pos) {
#pragma unroll
            for (int c = 0; c < 4; c++) acc[c] += v[c];
        }
    }
    // the point's lanes (consecutive; padding lanes form their own group):
    // the first finishes the point, then lane r of the point's seg lanes
    // forms the products r, r + seg, ... of the new increment
    const unsigned m = __match_any_sync(kFull, pos);
    const int head = __ffs(m) - 1, seg = __popc(m), r = lane - head;
    if (live && r == 0) sweep_point<T>(fwd, d, st, sb, k, wall, e1x, e1y, e2x, e2y, acc, w);
#pragma unroll
    for (int c = 0; c < 4; c++) w[c] = __shfl_sync(kFull, w[c], head);
    if (!live) return;
    if (JVP == 0) {
        // the point's axis Jacobians, formed before the sweeps
        const T *F = (sizeof(T) == 4 ? (const T *)d.fjf : (const T *)d.fj) + 64 * (size_t)d.fidx[k];
        for (int cb = r; cb < 4; cb += seg) {
            T J[4];
#pragma unroll
            for (int c = 0; c < 4; c++) {
                T Fc[4];
                load4_l2(F + 16 * cb + 4 * c, Fc);
                J[c] = Fc[0] * w[0];
#pragma unroll
                for (int j = 1; j < 4; j++) J[c] = fma(Fc[j], w[j], J[c]);
            }
            store4(sb.jc + 16 * (size_t)k + 4 * cb, J);
        }
    } else {
        double Up[4], G0[4];
#pragma unroll
        for (int c = 0; c < 4; c++) Up[c] = st.U[c * d.ld + k] + (double)w[c];
        const PrimU P = prim_short(Up);
        for (int cb = r; cb < 4; cb += seg) {
            load4(d.g0 + 16 * (size_t)k + 4 * cb, G0);
            store_increment_product<T>(g_math, sb, P, G0, k, cb);
        }
    }
}

// The sweeps' levels (dirs: 1 forward, 2 backward, 3 both), one cooperative
// launch.  A neighbour's Jacobian product along an axis depends only on the
// neighbour, the axis and the sub-stencil's sign, so a point forms the four
// axis products of its new increment once, and interior points gather them: 8
// FMAs per slot instead of ~70 FP64 instructions.  A point's sum depends only
// on its own list, in a fixed order, so a batch still equals its single
// solves bit for bit.  A level's tasks are one warp each: first its warps for
// the points in a (t, n) frame (their slots packed whole into warps at create,
// by best fit; a point with an empty list takes one idle slot), then its
// groups of interior points; task t goes to warp t / gridDim of block
// t % gridDim, so a level spreads over all SMs before it stacks up on one.
// Between levels all blocks meet; what the next level reads of the cloud and
// of the iteration's state is loaded while a block waits there, the values
// other blocks wrote (increments, axis products) after it, from L2.
// fuse: the framed points' Jacobians are formed here first (else by
// k_framed_jac beside the q-derivatives).
template <int JVP, typename T>
__global__ void __launch_bounds__(kSweepBlock, 1) k_sweeps(Dev d, StateSet st, int n_levels, int dirs, bool fuse)
{
    if (halted_step(d)) return;  // the same for every block: set by earlier launches only
    const int lane = threadIdx.x & 31, t0 = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int stride = (blockDim.x >> 5) * gridDim.x;
    const SweepBufs<T> sb = sweep_bufs<T>(d, st);
    const int steps = n_levels * (dirs == 3 ? 2 : 1);
    const uint32_t limit = (uint32_t)(steps - 1 + (fuse ? 1 : 0)) * gridDim.x;
    uint32_t target = 0;
    extern __shared__ __align__(16) unsigned char smem[];
    WarpStage<T> &ws = reinterpret_cast<WarpStage<T> *>(smem)[threadIdx.x >> 5];
    const bool exact = JVP == 0 && d.lusgs == 0;
    LanePre<T> pre;
    FramedPre<T> fpre;
    bool ready = false;  // pre or fpre holds the warp's first task of the level
    for (int step = fuse ? -1 : 0; step < steps; step++) {
        if (step < 0) {
            for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < framed_jac_items(d); t += gridDim.x * blockDim.x)
                framed_jac_item<T>(d, st, g_math, t);
        } else {
            const int dir = dirs == 3 ? (step < n_levels ? 0 : 1) : dirs - 1;
            const int l = dir == 0 ? step : steps - 1 - step;
            const int wb = d.lvl_fw[dir][l], wf = d.lvl_fw[dir][l + 1] - wb;
            const int g0 = d.lvl_in[dir][l], nt = wf + d.lvl_in[dir][l + 1] - g0;
            const bool two = d.lvl_lanes[l] == 2;
            for (int t = t0; t < nt; t += stride) {
                if (t < wf) {
                    if (exact) {
                        if (!ready) framed_load<T>(d, dir, wb + t, lane, fpre);
                        framed_run<T>(d, sb, dir, lane, fpre);
                    } else {
                        sweep_framed<JVP, T>(d, st, sb, dir, wb + t, lane);
                    }
                } else if (two) {
                    if (!ready) lane_load<JVP, 2, T>(d, st, sb, dir, g0 + t - wf, lane, ws, pre);
                    sweep_interior<JVP, 2, T>(d, st, sb, dir, lane, pre, ws);
                } else {
                    if (!ready) lane_load<JVP, 4, T>(d, st, sb, dir, g0 + t - wf, lane, ws, pre);
                    sweep_interior<JVP, 4, T>(d, st, sb, dir, lane, pre, ws);
                }
                ready = false;
            }
        }
        if (step + 1 < steps) {
            boundary_arrive(d.ctrl, limit, d.sweep_skip && blockIdx.x == 0);
            const int dir = dirs == 3 ? (step + 1 < n_levels ? 0 : 1) : dirs - 1;
            const int l = dir == 0 ? step + 1 : steps - 2 - step;
            const int wb = d.lvl_fw[dir][l], wf = d.lvl_fw[dir][l + 1] - wb;
            const int g0 = d.lvl_in[dir][l], nt = wf + d.lvl_in[dir][l + 1] - g0;
            if (t0 < wf) {
                // (before the first level the matrices may still be being formed)
                if (exact && step >= 0) {
                    framed_load<T>(d, dir, wb + t0, lane, fpre);
                    ready = true;
                }
            } else if (t0 < nt) {
                if (d.lvl_lanes[l] == 2) lane_load<JVP, 2, T>(d, st, sb, dir, g0 + t0 - wf, lane, ws, pre);
                else lane_load<JVP, 4, T>(d, st, sb, dir, g0 + t0 - wf, lane, ws, pre);
                ready = true;
            }
            target += gridDim.x;
            if (!boundary_wait(d.ctrl, target, limit, d.sweep_wait_ns)) {
                cp_async_wait<0>();  // what was loaded ahead
                return;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// state update (set cur -> set 1-cur) and per-point quantities of the new state
// ---------------------------------------------------------------------------
__global__ void k_begin(Ctrl *c, int32_t *suspect)
{
    c->live = 0;
    if (c->stop | c->error) return;
    int running = 0;
    for (int b = 0; b < c->n_cases; b++) {
        suspect[b] = 0;
        if (c->case_state[b] == kReachedTarget) c->case_state[b] = kStopped;
        if (c->case_state[b] == kFailedNow) c->case_state[b] = kFailed;
        running += !frozen_state(c->case_state[b]);
    }
    if (running == 0) {
        c->stop = 1;
    } else {
        c->it += 1;
        c->live = 1;
    }
}

// One kernel for both uses (inc: after an iteration, set cur -> 1 - cur; not
// inc: a new state in set cur), so that q and the per-point records of a
// given U come from the same instructions either way: a resumed checkpoint
// continues bit for bit.
// The function tables are read where they lie (two rows and two entries per
// point, from L1 and L2): staging 43 KB per block cost more than it saved, and
// blocks of 64 threads spread a small cloud over the SMs (147,584 points 0.045
// -> 0.038 ms, 41,194 0.026 -> 0.018, 10,240 0.018 -> 0.013).
constexpr int kUpdateBlock = 64;
__global__ void __launch_bounds__(kUpdateBlock) k_update(Dev d, int cur, bool inc, bool project)
{
    const MathTables &T = g_math;
    if (inc && halted_step(d)) return;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    const int ld = d.ld;
    const StateSet src = d.set[cur];
    const StateSet dst = d.set[inc ? 1 - cur : cur];
    const int fl = d.flag[k];
    double U[4];
#pragma unroll
    for (int c = 0; c < 4; c++) U[c] = src.U[c * ld + k];
    const bool moves = inc && (fl != kOuter || d.farfield == 1) && !frozen_step(d, k);
    if (moves) {
#pragma unroll
        for (int c = 0; c < 4; c++) U[c] += d.dUf ? (double)d.dUf[4 * k + c] : d.dU[4 * k + c];
    }
    // wall projection of a moved point, or of a new state built from
    // primitives or predicted (project): re-projecting a projected state
    // could change its last bits, and a stopped case must keep its state
    if (fl == kWall && (moves || (!inc && project))) {
        const double nx = d.wnx[k], ny = d.wny[k];
        const double mn = U[1] * nx + U[2] * ny;
        U[1] -= mn * nx;
        U[2] -= mn * ny;
    }
    const PrimU P = prim_from_cons(U);
    const bool ok = P.rho > 0.0 && P.p > 0.0 && isfinite(P.rho) && isfinite(P.p) && isfinite(P.u) &&
                    isfinite(P.v);
    if (!ok) {
        if (inc && d.n_cases > 1) {  // fail this case only; k_repair restores its state
            const int b = d.case_of[k];
            atomicExch(&d.ctrl->case_state[b], (int32_t)kFailedNow);
            atomicExch(&d.ctrl->case_err[b], -3);  // LSKUM_ERR_NONPOSITIVE
            atomicMin(&d.ctrl->case_bad[b], k);
        } else {
            atomicMin(&d.ctrl->bad_point, k);
            atomicExch(&d.ctrl->error, -3);
        }
        return;
    }
#pragma unroll
    for (int c = 0; c < 4; c++) dst.U[c * ld + k] = U[c];
    // q1 = ln rho + 2.5 ln beta - beta |u|^2 with one logarithm: ln(rho beta^2 sqrt(beta))
    double qn[4];
    qn[0] = fma(-P.beta, P.q2, log(mul_i(mul_i(P.rho, mul_i(P.beta, P.beta)), P.sb)));
    qn[1] = mul_i(twice(P.beta), P.u);
    qn[2] = mul_i(twice(P.beta), P.v);
    qn[3] = signed_by(twice(P.beta), false);
    store4(dst.q + 4 * (size_t)k, qn);
    longlong2 *qf = reinterpret_cast<longlong2 *>(dst.qf + 4 * (size_t)k);
    const int shift = d.n_cases > 1 ? d.case_shift[d.case_of[k]] : d.shift;
    qf[0] = make_longlong2(fix_q(qn[0], 0, shift), fix_q(qn[1], 1, shift));
    qf[1] = make_longlong2(fix_q(qn[2], 2, shift), fix_q(qn[3], 3, shift));
    // the per-point record, assembled in registers and stored as 16-byte
    // vectors (and, in mixed precision, its FP32 copy from the same registers)
    double rec[P_NFIELDS];
    rec[P_RHO] = P.rho;
    rec[P_IRHO] = P.irho;
    rec[P_U] = P.u;
    rec[P_V] = P.v;
    rec[P_P] = P.p;
    rec[P_BETA] = P.beta;
    rec[P_SB] = P.sb;
    rec[P_ISB] = P.isb;
    rec[P_I2P] = P.i2p;
    rec[P_Q2] = P.q2;
    rec[P_E1] = P.e1;
    rec[P_E2] = P.e2;
    const double sx = mul_i(P.u, P.sb), sy = mul_i(P.v, P.sb);
    double Ex, ex, Ey, ey;
    split_E(T, sx, Ex, ex);
    split_E(T, sy, Ey, ey);
    const double bk = mul_i(kInv2SqrtPi, P.isb);
    const double bx = mul_i(ex, bk), by = mul_i(ey, bk);
    rec[P_BSX] = mul_i(twice(bx), sx);
    rec[P_APX] = sx >= 0.0 ? 1.0 - Ex : Ex;
    rec[P_AMX] = sx >= 0.0 ? Ex : 1.0 - Ex;
    rec[P_EKX] = mul_i(ex, kInvSqrtPi);
    rec[P_BX] = bx;
    rec[P_BSY] = mul_i(twice(by), sy);
    rec[P_APY] = sy >= 0.0 ? 1.0 - Ey : Ey;
    rec[P_AMY] = sy >= 0.0 ? Ey : 1.0 - Ey;
    rec[P_EKY] = mul_i(ey, kInvSqrtPi);
    rec[P_BY] = by;
    rec[P_UE1] = mul_i(P.u, P.e1);
    rec[P_VE1] = mul_i(P.v, P.e1);
    static_assert(P_NFIELDS == kPrimStride && kPrimStride % 4 == 0, "record stored as whole vectors");
    double2 *pr2 = reinterpret_cast<double2 *>(dst.prim + (size_t)k * kPrimStride);
#pragma unroll
    for (int f = 0; f < P_NFIELDS / 2; f++) pr2[f] = make_double2(rec[2 * f], rec[2 * f + 1]);
    if (dst.primf) {  // mixed precision: the sweeps' FP32 copy of the record
        float4 *pf4 = reinterpret_cast<float4 *>(dst.primf + (size_t)k * kPrimStride);
#pragma unroll
        for (int f = 0; f < P_NFIELDS / 4; f++)
            pf4[f] = make_float4((float)rec[4 * f], (float)rec[4 * f + 1], (float)rec[4 * f + 2], (float)rec[4 * f + 3]);
    }
}

// Explicit scheme (the paper's solver (e)): dU = -dt R = -R / D at wall and
// interior points (and outer points under the kinetic far field), normal
// momentum removed at wall points; frozen outer points 0.
__global__ void __launch_bounds__(256) k_explicit(Dev d)
{
    if (halted_step(d)) return;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    const int ld = d.ld;
    double w[4] = {0.0, 0.0, 0.0, 0.0};
    const int fl = d.flag[k];
    if ((fl != kOuter || d.farfield == 1) && !frozen_step(d, k)) {
        const double dt = d.iD[k];
#pragma unroll
        for (int c = 0; c < 4; c++) w[c] = -dt * d.R[c * ld + k];
        if (fl == kWall) {
            const double nx = d.wnx[k], ny = d.wny[k];
            const double mn = w[1] * nx + w[2] * ny;
            w[1] -= mn * nx;
            w[2] -= mn * ny;
        }
    }
#pragma unroll
    for (int c = 0; c < 4; c++) d.dU[4 * k + c] = w[c];
}

// Batches: undo this iteration's update of the cases that failed in it (the
// new state set gets the old set's values), so a failed case keeps its last
// good state.
__global__ void __launch_bounds__(256) k_repair(Dev d, int cur)
{
    if (halted(d.ctrl)) return;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    if (((const volatile int32_t *)d.case_state)[d.case_of[k]] != kFailedNow) return;
    const int ld = d.ld;
    const StateSet src = d.set[cur], dst = d.set[1 - cur];
#pragma unroll
    for (int c = 0; c < 4; c++) {
        dst.U[c * ld + k] = src.U[c * ld + k];
        dst.q[4 * (size_t)k + c] = src.q[4 * (size_t)k + c];
        dst.qf[4 * (size_t)k + c] = src.qf[4 * (size_t)k + c];
    }
    for (int f = 0; f < kPrimStride; f++) dst.prim[(size_t)k * kPrimStride + f] = src.prim[(size_t)k * kPrimStride + f];
    if (src.primf)
        for (int f = 0; f < kPrimStride; f++)
            dst.primf[(size_t)k * kPrimStride + f] = src.primf[(size_t)k * kPrimStride + f];
}

__global__ void k_reset_ctrl(Ctrl *c)
{
    c->stop = 0;
    c->error = 0;
    c->bad_point = 0x7fffffff;
    c->sweep_bar = 0;
}

// After the update that checked a new state: if it is a state, every case runs
// again and failures are forgotten, with `history` as if newly created.
__global__ void k_accept_state(Ctrl *c, bool history)
{
    if (c->error) return;
    for (int b = threadIdx.x; b < c->n_cases; b += blockDim.x) {
        c->case_state[b] = kRunning;
        c->case_err[b] = 0;
        c->case_bad[b] = 0x7f7f7f7f;
        if (history) {
            c->case_it[b] = 0;
            c->case_hist0[b] = 0.0;
        }
    }
    if (history && threadIdx.x == 0) {
        c->it = 0;
        c->target = 0.0;
    }
}

__global__ void k_prep_run(Ctrl *c, double target)
{
    c->stop = 0;
    c->error = 0;
    c->bad_point = 0x7fffffff;
    c->sweep_bar = 0;
    c->target = target;
    c->it_start = c->it;
    for (int b = 0; b < c->n_cases; b++)
        c->case_state[b] = (c->case_state[b] == kFailed || c->case_state[b] == kFailedNow) ? kFailed : kRunning;
}

template <int TPP>
cudaError_t enqueue_grad(const Dev &d, int cur, cudaStream_t s, int *launches)
{
    constexpr int S = kGradLanes<TPP>;
    const int gb = (int)(((int64_t)d.n * 2 * S + kGradBlock - 1) / kGradBlock);
    const StateSet st = d.set[cur];
    k_grad<S, false><<<gb, kGradBlock, 0, s>>>(d, st, 0, 2, d.K == 0);
    (*launches)++;
    for (int it = 1; it <= d.K; it++) {
        k_grad<S, true><<<gb, kGradBlock, 0, s>>>(d, st, it == 1 ? 2 : it & 1, 1 - (it & 1), it == d.K);
        (*launches)++;
    }
    return cudaGetLastError();
}

template <int TPP>
cudaError_t enqueue_res(const Dev &d, const Launch &L, int cur, cudaStream_t s, int *launches)
{
    constexpr int block = kResBlock<TPP>;
    const int want = (d.n * TPP + block - 1) / block, most = L.sms * (512 / block);
    const double *g = d.gq[grad_buffer(d.K)];
    if (d.fp64_cases != 1) {
        k_residual<TPP><<<want < most ? want : most, block, 0, s>>>(d, d.set[cur], g);
        (*launches)++;
    }
    if (d.fp64_cases) {
        k_residual_fp64<TPP><<<(d.n * TPP + kRes64Block - 1) / kRes64Block, kRes64Block, 0, s>>>(d, d.set[cur], g);
        (*launches)++;
    }
    return cudaGetLastError();
}

cudaError_t enqueue_grad_res(const Dev &d, const Launch &L, int cur, cudaStream_t s, int *launches, bool grad,
                             bool res)
{
    cudaError_t e = cudaSuccess;
    switch (L.tpp) {
    case 1:
        if (grad) e = enqueue_grad<1>(d, cur, s, launches);
        if (res && e == cudaSuccess) e = enqueue_res<1>(d, L, cur, s, launches);
        break;
    case 2:
        if (grad) e = enqueue_grad<2>(d, cur, s, launches);
        if (res && e == cudaSuccess) e = enqueue_res<2>(d, L, cur, s, launches);
        break;
    case 4:
        if (grad) e = enqueue_grad<4>(d, cur, s, launches);
        if (res && e == cudaSuccess) e = enqueue_res<4>(d, L, cur, s, launches);
        break;
    case 8:
        if (grad) e = enqueue_grad<8>(d, cur, s, launches);
        if (res && e == cudaSuccess) e = enqueue_res<8>(d, L, cur, s, launches);
        break;
    default: return cudaErrorInvalidValue;
    }
    return e;
}

template <int JVP, int G>
void enqueue_sweeps_g(const Dev &d, int cur, int n_levels, const int32_t *lvl_beg, const int32_t *lvl_act_end,
                      cudaStream_t s, int *launches, bool fwd, bool bwd)
{
    const StateSet st = d.set[cur];
    for (int l = 0; fwd && l < n_levels; l++) {
        const int np = lvl_act_end[l] - lvl_beg[l];
        if (np <= 0) continue;
        const int blocks = (np * G + 255) / 256;
        if (d.precision) k_sweep<JVP, true, G, float><<<blocks, 256, 0, s>>>(d, st, lvl_beg[l], lvl_act_end[l]);
        else k_sweep<JVP, true, G, double><<<blocks, 256, 0, s>>>(d, st, lvl_beg[l], lvl_act_end[l]);
        (*launches)++;
    }
    for (int l = n_levels - 1; bwd && l >= 0; l--) {
        const int np = lvl_act_end[l] - lvl_beg[l];
        if (np <= 0) continue;
        const int blocks = (np * G + 255) / 256;
        if (d.precision) k_sweep<JVP, false, G, float><<<blocks, 256, 0, s>>>(d, st, lvl_beg[l], lvl_act_end[l]);
        else k_sweep<JVP, false, G, double><<<blocks, 256, 0, s>>>(d, st, lvl_beg[l], lvl_act_end[l]);
        (*launches)++;
    }
}

// The packed exact sweeps apply precomputed framed-point Jacobians.
bool needs_framed_jac(const Dev &d, const Launch &L)
{
    return d.scheme == 0 && d.jvp == 0 && L.sweep_lanes == 32 && (d.pk_jm[0] || d.pk_jmf[0]) && framed_jac_items(d) > 0;
}

void enqueue_framed_jac(const Dev &d, int cur, cudaStream_t s, int *launches)
{
    const int items = framed_jac_items(d);
    if (d.precision) k_framed_jac<float><<<(items + 255) / 256, 256, 0, s>>>(d, d.set[cur]);
    else k_framed_jac<double><<<(items + 255) / 256, 256, 0, s>>>(d, d.set[cur]);
    (*launches)++;
}

bool needs_increment_base(const Dev &d)
{
    return d.scheme == 0 && d.jvp == 1 && d.g0;
}

void enqueue_increment_base(const Dev &d, int cur, cudaStream_t s, int *launches)
{
    k_increment_base<<<(increment_base_items(d) + 255) / 256, 256, 0, s>>>(d, d.set[cur]);
    (*launches)++;
}

void enqueue_diag(const Dev &d, int cur, cudaStream_t s, int *launches)
{
    k_diag<<<(d.n + 255) / 256, 256, 0, s>>>(d, d.set[cur]);
    (*launches)++;
}

template <int JVP, typename T>
cudaError_t launch_sweeps(const Dev &d, const Launch &L, int cur, int n_levels, int dirs, bool fuse, cudaStream_t s)
{
    Dev dd = d;
    StateSet st = d.set[cur];
    void *args[] = {&dd, &st, &n_levels, &dirs, &fuse};
    const size_t smem = (size_t)(L.sw_threads / 32) * sizeof(WarpStage<T>);
    const void *kernel = (const void *)k_sweeps<JVP, T>;
    // (the kernel's limit is the process's: always the largest block's, so that
    // contexts of other sizes in other threads set the same)
    constexpr int most = kSweepBlock / 32 * (int)sizeof(WarpStage<T>);
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(kernel, dim3(L.sw_blocks), dim3(L.sw_threads), args, smem, s);
}

template <int JVP>
cudaError_t enqueue_sweeps_packed(const Dev &d, const Launch &L, int cur, int n_levels, cudaStream_t s, int *launches,
                                  bool fwd, bool bwd)
{
    // the framed points' Jacobians: by k_framed_jac in the packed shape
    // (beside the q-derivatives when captured), else by the sweeps' launch
    if (fwd && !L.side && needs_framed_jac(d, L)) enqueue_framed_jac(d, cur, s, launches);
    if (fwd && !L.side && needs_increment_base(d)) enqueue_increment_base(d, cur, s, launches);
    const bool fuse = fwd && JVP == 0 && L.sweep_lanes != 32 && framed_jac_items(d) > 0;
    const int dirs = (fwd ? 1 : 0) + (bwd ? 2 : 0);
    if (n_levels <= 0 || dirs == 0) return cudaSuccess;
    (*launches)++;
    return d.precision ? launch_sweeps<JVP, float>(d, L, cur, n_levels, dirs, fuse, s)
                       : launch_sweeps<JVP, double>(d, L, cur, n_levels, dirs, fuse, s);
}

// Clouds whose lists fit the packed layout use the gathered form in every
// shape (sweep_lanes 2, 4, 8 and 32 differ in who forms the framed points'
// Jacobians); a list of more than 32 lower or upper neighbours needs the
// per-slot form, one launch per level.
template <int JVP>
cudaError_t enqueue_sweeps(const Dev &d, const Launch &L, int cur, int n_levels, const int32_t *lvl_beg,
                           const int32_t *lvl_act_end, cudaStream_t s, int *launches, bool fwd, bool bwd)
{
    if (d.pk_pt[0]) return enqueue_sweeps_packed<JVP>(d, L, cur, n_levels, s, launches, fwd, bwd);
    switch (L.sweep_lanes) {
    case 2: enqueue_sweeps_g<JVP, 2>(d, cur, n_levels, lvl_beg, lvl_act_end, s, launches, fwd, bwd); break;
    case 4: enqueue_sweeps_g<JVP, 4>(d, cur, n_levels, lvl_beg, lvl_act_end, s, launches, fwd, bwd); break;
    case 8: enqueue_sweeps_g<JVP, 8>(d, cur, n_levels, lvl_beg, lvl_act_end, s, launches, fwd, bwd); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// The norm.  Nothing of an iteration waits for its result (see d.suspect), so
// a captured iteration runs it beside the update: 0.020 ms of the 0.36 ms of
// 41,194 points.  (Beside the sweeps it would delay their cooperative launch.)
cudaError_t enqueue_norm(const Dev &d, cudaStream_t s, int *launches)
{
    k_norm_partials<<<d.n_blk, 256, 0, s>>>(d);
    k_norm_cases<<<d.n_cases, 256, 0, s>>>(d);
    (*launches) += 2;
    return cudaGetLastError();
}

cudaError_t enqueue_phase(const Dev &d, const Launch &L, int cur, int ph, int n_levels, const int32_t *lvl_beg,
                          const int32_t *lvl_act_end, cudaStream_t s, int *launches)
{
    const bool side = L.side && (needs_framed_jac(d, L) || needs_increment_base(d) || L.tpp > 1);
    switch (ph) {
    case 0:
        k_begin<<<1, 1, 0, s>>>(d.ctrl, d.suspect);
        (*launches)++;
        if (side) {
            // what depends only on the state: a side branch beside the
            // q-derivatives and the residual
            cudaError_t e = cudaEventRecord(L.fork, s);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(L.side, L.fork, 0);
            if (e != cudaSuccess) return e;
            if (needs_framed_jac(d, L)) enqueue_framed_jac(d, cur, L.side, launches);
            if (L.tpp > 1) enqueue_diag(d, cur, L.side, launches);
            if (needs_increment_base(d)) enqueue_increment_base(d, cur, L.side, launches);
            e = cudaEventRecord(L.join, L.side);
            if (e != cudaSuccess) return e;
        }
        return enqueue_grad_res(d, L, cur, s, launches, true, false);
    case 1:
        if (!side && L.tpp > 1) enqueue_diag(d, cur, s, launches);
        return enqueue_grad_res(d, L, cur, s, launches, false, true);
    case 2: return L.side ? cudaSuccess : enqueue_norm(d, s, launches);  // (captured: beside the update)
    case 3:
    case 4:
        if (ph == 3 && side) {
            cudaError_t e = cudaStreamWaitEvent(s, L.join, 0);
            if (e != cudaSuccess) return e;
        }
        if (d.scheme == 1) {  // explicit: one step kernel instead of the two sweeps
            if (ph == 3) {
                k_explicit<<<(d.n + 255) / 256, 256, 0, s>>>(d);
                (*launches)++;
            }
            return cudaGetLastError();
        }
        {
            // a captured iteration enqueues both sweeps in phase 3
            const bool both = L.side != nullptr, fwd = ph == 3, bwd = both ? ph == 3 : ph == 4;
            if (d.jvp == 0) return enqueue_sweeps<0>(d, L, cur, n_levels, lvl_beg, lvl_act_end, s, launches, fwd, bwd);
            return enqueue_sweeps<1>(d, L, cur, n_levels, lvl_beg, lvl_act_end, s, launches, fwd, bwd);
        }
    case 5: {
        if (L.side) {
            cudaError_t e = cudaEventRecord(L.fork, s);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(L.side, L.fork, 0);
            if (e == cudaSuccess) e = enqueue_norm(d, L.side, launches);
            if (e == cudaSuccess) e = cudaEventRecord(L.join, L.side);
            if (e != cudaSuccess) return e;
        }
        k_update<<<(d.n + kUpdateBlock - 1) / kUpdateBlock, kUpdateBlock, 0, s>>>(d, cur, true, true);
        (*launches)++;
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess && L.side) e = cudaStreamWaitEvent(s, L.join, 0);
        if (e == cudaSuccess && d.n_cases > 1) {
            k_repair<<<(d.n + 255) / 256, 256, 0, s>>>(d, cur);
            (*launches)++;
            e = cudaGetLastError();
        }
        return e;
    }
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_iteration(const Dev &d, const Launch &L, int cur, int n_levels, const int32_t *lvl_beg,
                             const int32_t *lvl_act_end, cudaStream_t s, int *launches)
{
    for (int ph = 0; ph < 6; ph++) {
        cudaError_t e = enqueue_phase(d, L, cur, ph, n_levels, lvl_beg, lvl_act_end, s, launches);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_phase(const Dev &d, const Launch &L, int cur, int phase, int n_levels, const int32_t *lvl_beg,
                         const int32_t *lvl_act_end, cudaStream_t s)
{
    int launches = 0;
    Launch Li = L;  // one phase at a time: the framed Jacobians inline, in the forward sweep's phase
    Li.side = nullptr;
    return enqueue_phase(d, Li, cur, phase, n_levels, lvl_beg, lvl_act_end, s, &launches);
}

cudaError_t launch_init_state(const Dev &d, int cur, bool project, cudaStream_t s)
{
    k_update<<<(d.n + kUpdateBlock - 1) / kUpdateBlock, kUpdateBlock, 0, s>>>(d, cur, false, project);
    return cudaGetLastError();
}

namespace {

// Internal order (structure of arrays [c][ld] for stride 0, else point k's
// values at stride * k; FP64 or FP32) -> caller order [p][comps] on the device.
__global__ void k_to_caller(const double *src, const float *srcf, int comps, int stride, int ld, int n,
                            const int32_t *inv, double *out)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int k = inv[p];
    for (int c = 0; c < comps; c++) {
        const size_t i = stride ? (size_t)stride * k + c : (size_t)c * ld + k;
        out[(size_t)comps * p + c] = srcf ? (double)srcf[i] : src[i];
    }
}

// Caller order [p][4] -> internal structure of arrays [c][ld].
__global__ void k_from_caller(const double *in, int ld, int n, const int32_t *inv, double *U)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int k = inv[p];
#pragma unroll
    for (int c = 0; c < 4; c++) U[(size_t)c * ld + k] = in[(size_t)4 * p + c];
}

}  // namespace

cudaError_t launch_to_caller(const double *src, const float *srcf, int comps, int stride, int ld, int n,
                             const int32_t *inv, double *out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_to_caller<<<(n + 255) / 256, 256, 0, s>>>(src, srcf, comps, stride, ld, n, inv, out);
    return cudaGetLastError();
}

cudaError_t launch_from_caller(const double *in, int ld, int n, const int32_t *inv, double *U, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_from_caller<<<(n + 255) / 256, 256, 0, s>>>(in, ld, n, inv, U);
    return cudaGetLastError();
}

// The integer-pipe FP64 arithmetic on the device, for the self-test entry
// (op 0: a * b by mul_i; 1: exp(a) in fixed point; 2: erfcx(|a|)/2 in fixed
// point after the kernels' clamp of |a| to 9; 3: a * b on the FP64 unit).
__global__ void __launch_bounds__(256) k_selftest_fpint(int op, const double *a, const double *b, double *out, int n)
{
    __shared__ MathTables T;
    load_math_tables(T);
    __syncthreads();
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        double r;
        if (op == 0) {
            r = mul_i(a[k], b[k]);
        } else if (op == 1) {
            r = exp_t(T, a[k]);
        } else if (op == 2) {
            constexpr int kNineHi = 0x40220000;
            const int hs = __double2hiint(a[k]) & 0x7fffffff;
            const bool clamp = hs >= kNineHi;
            const int ha = clamp ? kNineHi : hs, la = clamp ? 0 : __double2loint(a[k]);
            const int iv = erfcx_interval(ha);
            r = erfcx_half_fx<kErfcxDeg>((uint32_t)ha, (uint32_t)la, iv, (const int64_t *)T.ecx[iv], T.esh[iv]);
        } else {
            r = a[k] * b[k];
        }
        out[k] = r;
    }
}

cudaError_t launch_selftest_fpint(int op, const double *a, const double *b, double *out, int n, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int blocks = (n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024;
    k_selftest_fpint<<<blocks, 256, 0, s>>>(op, a, b, out, n);
    return cudaGetLastError();
}

cudaError_t launch_init_math(cudaStream_t s)
{
    k_init_math<<<1, 256, 0, s>>>();
    return cudaGetLastError();
}

cudaError_t launch_prep_run(Ctrl *c, double target, cudaStream_t s)
{
    k_prep_run<<<1, 1, 0, s>>>(c, target);
    return cudaGetLastError();
}

cudaError_t launch_accept_state(Ctrl *ctrl, bool history, cudaStream_t s)
{
    k_accept_state<<<1, 64, 0, s>>>(ctrl, history);
    return cudaGetLastError();
}

cudaError_t launch_reset_ctrl(Ctrl *c, cudaStream_t s)
{
    k_reset_ctrl<<<1, 1, 0, s>>>(c);
    return cudaGetLastError();
}

}  // namespace lskum
