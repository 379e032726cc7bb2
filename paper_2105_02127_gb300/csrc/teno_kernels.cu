// teno_kernels.cu -- CUDA kernels of the TENO finite-volume residual for
// sm_103a (GB300).
//
// Per RK stage (Sec. 2.1, Eq. fv_governing_equation_semi_discrete):
//   recon_*_kernel    stencil differences, coefficient matvecs (Eqs.
//                     reconstruction_08/09 with |V'_s| folded into the
//                     matrices), smoothness indicators (Eq. WENO_smoothness in
//                     a beta-orthonormal basis, so beta = |a'|^2), TENO scale
//                     separation, cutoff and two-step selection (Eqs.
//                     new_scale_separation .. TENO_weight) and evaluation at
//                     the edge Gauss points;
//   face_flux_kernel  rotated HLL / HLLC (Sec. 4) or upwind flux at the Gauss
//                     points of each face, summed with weights and |A|;
//   gather_kernel     cell-centric, atomic-free sum of the three face fluxes
//                     (owner +, neighbour -), fused with the SSP-RK3 stage
//                     combination (Eq. fv_time_discretization_01);
//   max_lambda_kernel warp-shuffle / block reduction of the CFL signal speed.
// Adjoint (no counterpart in the paper): face_flux_vjp_kernel (dual-number
// flux Jacobians), recon_vjp_kernel (transposed matvecs with the selection
// frozen) and scatter_gather_kernel (reverse-stencil gather, no atomics).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "teno_fp64.cuh"
#include "teno_internal.h"

namespace teno {
namespace {

// Programmatic dependent launch.  The kernels are launched so that the next one
// starts when the last block of the one before it exits, and wait here for its
// completion (and its writes) before the first access to memory that a kernel
// writes: a launch's latency and prologue overlap the tail before it.  Ten
// launches of a small step took 80 us and take 61 (2,048 cells, scalar TENO3),
// a step of 32,768 cells TENO5 195 and 171.  No kernel triggers its successor
// earlier: blocks that wait on occupied SMs end up unevenly spread (14,792
// cells, scalar: 109 us a step, 177 with a trigger at the kernel's start).
// Constant data of the plan may be read before the wait.  What a kernel writes
// is read with plain loads only: the read-only path (ld.global.nc, const
// __restrict__) assumes data that no running kernel writes.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int kSmallEntries = kSmallK * kSmallN * kSmallM;  // 180
// stencil slots unrolled together in the reconstruction loops (loads of that
// many slots can be in flight per thread)
#ifndef TENO_RECON_UNROLL
#define TENO_RECON_UNROLL 2
#endif
constexpr int kSlotUnroll = TENO_RECON_UNROLL;
// the FP32-mixed kernels keep more slots in flight (4 measured best, 2 for
// the double-float and FP64 kernels)
#ifndef TENO_RECON_UNROLL_MIXED
#define TENO_RECON_UNROLL_MIXED 4
#endif
constexpr int kSlotUnrollMixed = TENO_RECON_UNROLL_MIXED;
constexpr int kSmallSlots = kSmallK * kSmallN;               // 36

template <typename T>
struct TypeTag {
  using type = T;
};

// ---------------------------------------------------------------- scalars
template <typename T>
__device__ __forceinline__ T tsqrt(T x);
template <>
__device__ __forceinline__ double tsqrt<double>(double x) { return sqrt(x); }
template <>
__device__ __forceinline__ float tsqrt<float>(float x) { return sqrtf(x); }

// scalar constants of every arithmetic type used by the flux templates
template <typename T>
struct Cst {
  __device__ __forceinline__ static T from(double x) { return T(x); }
};
template <typename T>
__device__ __forceinline__ T cst(double x) {
  return Cst<T>::from(x);
}

// forward-mode dual number with N directions over scalar type S (flux
// Jacobians of the adjoint)
template <int N, typename S = double>
struct Dual {
  S v;
  S d[N];
};
template <int N, typename S>
struct Cst<Dual<N, S>> {
  __device__ __forceinline__ static Dual<N, S> from(double x) {
    Dual<N, S> r;
    r.v = Cst<S>::from(x);
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = Cst<S>::from(0.0);
    return r;
  }
};
template <int N>
__device__ __forceinline__ Dual<N> mk(double v) {
  return Cst<Dual<N>>::from(v);
}
template <int N, typename S>
__device__ __forceinline__ Dual<N, S> operator+(const Dual<N, S>& a, const Dual<N, S>& b) {
  Dual<N, S> r;
  r.v = a.v + b.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] + b.d[i];
  return r;
}
template <int N, typename S>
__device__ __forceinline__ Dual<N, S> operator-(const Dual<N, S>& a, const Dual<N, S>& b) {
  Dual<N, S> r;
  r.v = a.v - b.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] - b.d[i];
  return r;
}
template <int N, typename S>
__device__ __forceinline__ Dual<N, S> operator-(const Dual<N, S>& a) {
  Dual<N, S> r;
  r.v = -a.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = -a.d[i];
  return r;
}
template <int N, typename S>
__device__ __forceinline__ Dual<N, S> operator*(const Dual<N, S>& a, const Dual<N, S>& b) {
  Dual<N, S> r;
  r.v = a.v * b.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * b.v + a.v * b.d[i];
  return r;
}
template <int N, typename S>
__device__ __forceinline__ Dual<N, S> operator*(double s, const Dual<N, S>& a) {
  const S ss = Cst<S>::from(s);
  Dual<N, S> r;
  r.v = ss * a.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = ss * a.d[i];
  return r;
}
template <int N, typename S>
__device__ __forceinline__ Dual<N, S> operator/(const Dual<N, S>& a, const Dual<N, S>& b) {
  Dual<N, S> r;
  r.v = a.v / b.v;
  const S ib = Cst<S>::from(1.0) / b.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = (a.d[i] - r.v * b.d[i]) * ib;
  return r;
}
__device__ __forceinline__ double val(double x);
__device__ __forceinline__ float val(float x);
template <int N, typename S>
__device__ __forceinline__ Dual<N, S> tsqrt(const Dual<N, S>& a) {
  Dual<N, S> r;
  r.v = tsqrt(a.v);
  // the root of a zero (a clamped pressure) carries no derivative
  const bool z = val(r.v) == decltype(val(r.v))(0);
  const S h = z ? r.v : Cst<S>::from(0.5) / r.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * h;
  return r;
}
__device__ __forceinline__ double val(double x) { return x; }
__device__ __forceinline__ float val(float x) { return x; }
template <int N, typename S>
__device__ __forceinline__ auto val(const Dual<N, S>& x) { return val(x.v); }
// min / max that ignore a NaN operand, like C's fmin / fmax (a wave speed
// from the sound speed of a state whose pressure rounds below zero is NaN;
// the other bound is then taken)
template <typename T>
__device__ __forceinline__ T vmin(const T& a, const T& b) {
  return (val(a) <= val(b) || val(b) != val(b)) ? a : b;
}
template <typename T>
__device__ __forceinline__ bool nonneg(const T& x) { return val(x) >= decltype(val(x))(0); }
template <typename T>
__device__ __forceinline__ T vmax(const T& a, const T& b) {
  return (val(a) >= val(b) || val(b) != val(b)) ? a : b;
}


// ------------------------------------------- double-float (FP32 pair) path
// Values are unevaluated sums hi + lo of two floats (|lo| <= ulp(hi)/2), about
// 48 significant bits: Dekker's double-length arithmetic ("A floating-point
// technique for extending the available precision", 1971) on FP32.  Sums use
// Knuth's two-sum (TAOCP vol. 2, 4.2.2), and Dekker's fast two-sum where the
// operands are ordered; products take the exact residual of a fused
// multiply-add in place of Dekker's splitting; the per-cell matrices are
// stored as (hi, lo) pairs.
// 8-byte aligned so that a pair moves through memory in one access
struct __align__(8) DF {
  float h, l;
};
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
// acc += a * b with a, b pairs; acc.l collects the rounding terms (the pair
// is renormalised by the caller)
__device__ __forceinline__ void df_mac(DF& acc, float2 a, DF b) {
  const float p = a.x * b.h;
  float e = fmaf(a.x, b.h, -p);
  e = fmaf(a.x, b.l, e);
  e = fmaf(a.y, b.h, e);
  const DF s = two_sum(acc.h, p);
  acc.h = s.h;
  acc.l += s.l + e;
}
__device__ __forceinline__ DF df_norm(DF a) { return two_sum(a.h, a.l); }
__device__ __forceinline__ DF d_to_df(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_to_double(DF a) { return (double)a.h + (double)a.l; }


// arithmetic on pairs (the Riemann flux of the FP64 path): sums renormalise
// once (Dekker's fast two-sum), products use the exact FMA residual, and
// quotients and square roots take Dekker's one correction step (div2, sqrt2
// of the 1971 paper: the exact remainder of the FP32 approximation, from an
// FMA, divided by the divisor or twice the root)
__device__ __forceinline__ DF fast_two_sum(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ DF operator+(DF a, DF b) {
  DF s = two_sum(a.h, b.h);
  s.l += a.l + b.l;
  return fast_two_sum(s.h, s.l);
}
__device__ __forceinline__ DF operator-(DF a) { return {-a.h, -a.l}; }
__device__ __forceinline__ DF operator-(DF a, DF b) { return a + (-b); }
__device__ __forceinline__ DF operator*(DF a, DF b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return fast_two_sum(p, e);
}
// Quotients: q1 from the correctly rounded reciprocal of b.h (1.5 ulp), the
// exact remainder a - b q1 in pairs, and its quotient by the same reciprocal
// (the correction carries a relative error of about one ulp); square roots:
// the correctly rounded FP32 root and a correction scaled by rsqrt/2.  Build
// with TENO_DF_IEEE_DIV=1 for IEEE FP32 divisions in both steps instead.
#ifndef TENO_DF_IEEE_DIV
#define TENO_DF_IEEE_DIV 0
#endif
// TENO_DF_APPROX=1 (default): start from the PTX approximate reciprocal and
// square root (relative error about 2^-22 each) instead of the correctly
// rounded ones; the one exact-remainder correction squares that error, so
// the pair results keep their ~2^-44 relative accuracy (face flux 3 %, flux
// VJP 5 % faster than with the correctly rounded starts).
#ifndef TENO_DF_APPROX
#define TENO_DF_APPROX 1
#endif
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ DF operator/(DF a, DF b) {
#if TENO_DF_IEEE_DIV
  const float q1 = a.h / b.h;
  const DF r = a - b * DF{q1, 0.f};
  return fast_two_sum(q1, r.h / b.h);
#else
#if TENO_DF_APPROX
  const float rb = rcp_approx(b.h);
#else
  const float rb = __frcp_rn(b.h);
#endif
  const float q1 = a.h * rb;
  const DF r = a - b * DF{q1, 0.f};
  return fast_two_sum(q1, r.h * rb);
#endif
}
__device__ __forceinline__ DF tsqrt(DF a) {
#if TENO_DF_APPROX && !TENO_DF_IEEE_DIV
  const float s = sqrt_approx(a.h);
#else
  const float s = sqrtf(a.h);
#endif
  if (!(a.h > 0.f)) return {s, 0.f};
  const DF r = a - DF{s, 0.f} * DF{s, 0.f};
#if TENO_DF_IEEE_DIV
  return fast_two_sum(s, r.h / (2.f * s));
#else
  return fast_two_sum(s, r.h * (0.5f * rsqrtf(a.h)));
#endif
}
__device__ __forceinline__ float val(DF x) { return x.h; }
template <>
struct Cst<DF> {
  __device__ __forceinline__ static DF from(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
  }
};
__device__ __forceinline__ DF vmin(const DF& a, const DF& b) {
  return (a.h < b.h || (a.h == b.h && a.l <= b.l) || b.h != b.h) ? a : b;
}
__device__ __forceinline__ DF vmax(const DF& a, const DF& b) {
  return (a.h > b.h || (a.h == b.h && a.l >= b.l) || b.h != b.h) ? a : b;
}
// c + a*b and conversion to FP64 for every scalar type of the flux kernels
// exact zero test (pairs: both parts; dual numbers: the value)
__device__ __forceinline__ bool is_zero(double x) { return x == 0.0; }
__device__ __forceinline__ bool is_zero(float x) { return x == 0.0f; }
__device__ __forceinline__ bool is_zero(DF x) { return x.h == 0.0f && x.l == 0.0f; }
template <int N, typename S>
__device__ __forceinline__ bool is_zero(const Dual<N, S>& x) { return is_zero(x.v); }

__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ DF madd(DF a, DF b, DF c) { return a * b + c; }
__device__ __forceinline__ double to_d(double x) { return x; }
__device__ __forceinline__ double to_d(float x) { return (double)x; }
__device__ __forceinline__ double to_d(DF x) { return (double)x.h + (double)x.l; }
// a stored Gauss-point value as the flux scalar type
template <typename S>
__device__ __forceinline__ S lift(double x) { return Cst<S>::from(x); }
template <typename S>
__device__ __forceinline__ S lift(float x) { return Cst<S>::from((double)x); }
template <typename S>
__device__ __forceinline__ S lift(DF x) {
  if constexpr (std::is_same<S, DF>::value)
    return x;
  else
    return S(to_d(x));
}
// branch decisions on dual numbers over pairs compare the (normalised) pairs
// lexicographically, which orders them as their exact sums; no conversion to
// FP64 on the device
__device__ __forceinline__ bool df_le(const DF& a, const DF& b) {
  return a.h < b.h || (a.h == b.h && a.l <= b.l);
}
template <int N>
__device__ __forceinline__ Dual<N, DF> vmin(const Dual<N, DF>& a, const Dual<N, DF>& b) {
  return (df_le(a.v, b.v) || b.v.h != b.v.h) ? a : b;
}
template <int N>
__device__ __forceinline__ Dual<N, DF> vmax(const Dual<N, DF>& a, const Dual<N, DF>& b) {
  return (df_le(b.v, a.v) || b.v.h != b.v.h) ? a : b;
}
template <int N>
__device__ __forceinline__ bool nonneg(const Dual<N, DF>& x) {
  return x.v.h > 0.f || (x.v.h == 0.f && x.v.l >= 0.f);
}
// a pressure in a side sound speed: negative values as zero, NaN kept.  A
// Gauss state at the positivity floor has a pressure about 1e-15 of its
// energy, below the resolution of the pair and FP32 evaluations; its sound
// speed is then zero, so the wave-speed bound is the particle speed and not
// the Roe bound alone.
template <typename T>
__device__ __forceinline__ T pos_part(const T& x) {
  return (nonneg(x) || val(x) != val(x)) ? x : x - x;
}

// reciprocal and square root of the Riemann solver
template <typename T>
__device__ __forceinline__ T flux_rcp(const T& one, const T& x) {
  return one / x;
}
template <>
__device__ __forceinline__ double flux_rcp<double>(const double&, const double& x) {
  return rcp_f64(x);
}
template <typename T>
__device__ __forceinline__ T flux_sqrt(const T& x) {
  return tsqrt(x);
}
template <>
__device__ __forceinline__ double flux_sqrt<double>(const double& x) {
  return sqrt_f64(x);
}

// ---------------------------------------------------------------- fluxes
// Euler flux through a face with unit normal n = (nx, ny): the state is
// expressed in the face frame (normal, tangential velocity), the 1D flux
// F^x is evaluated there and rotated back (Sec. 4.1, F^n = T^-1 F^x(T U)).
// constants of one face in the flux scalar type, converted once per face
template <typename T>
struct RiemannK {
  T one, half, gm1, gg, tnx, tny;
};
template <typename T>
__device__ __forceinline__ RiemannK<T> riemann_k(double nx, double ny, double g) {
  return {cst<T>(1.0), cst<T>(0.5), cst<T>(g - 1.0), cst<T>(g), cst<T>(nx), cst<T>(ny)};
}
// the same constants as dual numbers (zero derivatives; no conversion)
template <int N, typename S>
__device__ __forceinline__ RiemannK<Dual<N, S>> riemann_k_dual(const RiemannK<S>& k) {
  auto c = [](S x) {
    Dual<N, S> r = cst<Dual<N, S>>(0.0);
    r.v = x;
    return r;
  };
  return {c(k.one), c(k.half), c(k.gm1), c(k.gg), c(k.tnx), c(k.tny)};
}

template <typename T>
__device__ __forceinline__ void euler_riemann(const T* UL, const T* UR, const RiemannK<T>& K,
                                              int hllc, T* F) {
  const T one = K.one, half = K.half;
  const T gm1 = K.gm1, gg = K.gg;
  const T tnx = K.tnx, tny = K.tny;
  // left / right primitive variables in the face frame (one reciprocal per
  // density; every division below is by one of four reciprocals)
  T rL = UL[0], rR = UR[0];
  T irL = flux_rcp(one, rL), irR = flux_rcp(one, rR);
  T unL = (UL[1] * tnx + UL[2] * tny) * irL;
  T utL = (UL[2] * tnx - UL[1] * tny) * irL;
  T unR = (UR[1] * tnx + UR[2] * tny) * irR;
  T utR = (UR[2] * tnx - UR[1] * tny) * irR;
  T EL = UL[3], ER = UR[3];
  T pL = gm1 * (EL - half * rL * (unL * unL + utL * utL));
  T pR = gm1 * (ER - half * rR * (unR * unR + utR * utR));
  T cL = flux_sqrt(gg * pos_part(pL) * irL), cR = flux_sqrt(gg * pos_part(pR) * irR);
  T HL = (EL + pL) * irL, HR = (ER + pR) * irR;
  // Roe averages and Einfeldt wave speeds (Eq. wavespeed)
  T D = flux_sqrt(rR * irL);
  T iden = flux_rcp(one, one + D);
  T ua = (unL + unR * D) * iden;
  T va = (utL + utR * D) * iden;
  T Ha = (HL + HR * D) * iden;
  T ca = flux_sqrt(gm1 * (Ha - half * (ua * ua + va * va)));
  T SL = vmin(unL - cL, ua - ca);
  T SR = vmax(unR + cR, ua + ca);
  // 1D fluxes and conserved states in the face frame
  T mL = rL * unL, mR = rR * unR;
  T FL[4] = {mL, mL * unL + pL, mL * utL, unL * (EL + pL)};
  T FR[4] = {mR, mR * unR + pR, mR * utR, unR * (ER + pR)};
  T WL[4] = {rL, mL, rL * utL, EL};
  T WR[4] = {rR, mR, rR * utR, ER};
  T Fx[4];
  // HLLC's contact speed divides by aL - aR, zero only when both wave-speed
  // bounds equal the particle speeds (zero sound speed on both sides, e.g. a
  // wall Gauss state at zero pressure): the flux there is HLL's
  const T aL = rL * (SL - unL), aR = rR * (SR - unR);
  const T Dn = aL - aR;
  if (nonneg(SL)) {
#pragma unroll
    for (int k = 0; k < 4; ++k) Fx[k] = FL[k];
  } else if (nonneg(-SR)) {
#pragma unroll
    for (int k = 0; k < 4; ++k) Fx[k] = FR[k];
  } else if (!hllc || is_zero(Dn)) {
    T inv = flux_rcp(one, SR - SL);
    T sLR = SL * SR;
#pragma unroll
    for (int k = 0; k < 4; ++k) Fx[k] = (SR * FL[k] - SL * FR[k] + sLR * (WR[k] - WL[k])) * inv;
  } else {
    // HLLC: contact speed and star state of the side the face lies in; the
    // star energy f (E/r + (Ss - un)(Ss + p / (r (S - un)))) multiplied out,
    // so that nothing divides by S - un
    T Ss = (pR - pL + aL * unL - aR * unR) / Dn;
    bool left = nonneg(Ss);
    T r = left ? rL : rR, un = left ? unL : unR, ut = left ? utL : utR;
    T p = left ? pL : pR, S = left ? SL : SR, E = left ? EL : ER;
    T Smu = S - un, inv = flux_rcp(one, S - Ss);
    T gq = r * Smu;
    T f = gq * inv;
    T es = (Smu * E + (Ss - un) * (gq * Ss + p)) * inv;
    T Us[4] = {f, f * Ss, f * ut, es};
#pragma unroll
    for (int k = 0; k < 4; ++k) Fx[k] = (left ? FL[k] : FR[k]) + S * (Us[k] - (left ? WL[k] : WR[k]));
  }
  F[0] = Fx[0];
  F[1] = Fx[1] * tnx - Fx[2] * tny;
  F[2] = Fx[1] * tny + Fx[2] * tnx;
  F[3] = Fx[3];
}

// The FP64 solver, bound by the FP64 pipe: the same fluxes with the momenta in
// the face frame used as they are (rho u and rho v need no product), every
// multiply-add contracted, and comparisons on the bit patterns (integer
// instructions) where no operand is infinite or NaN.  131,072 cells, HLL: 139 us;
// the generic form above with these reciprocals and roots 166, with the IEEE
// ones 174.
__device__ __forceinline__ bool special(double x) {  // infinite or NaN
  return (~(unsigned)__double2hiint(x) & 0x7ff00000u) == 0u;
}
__device__ __forceinline__ int64_t order_key(double x) {  // both zeros map to 0
  const int64_t b = __double_as_longlong(x), m = b & 0x7fffffffffffffffLL;
  return b < 0 ? -m : m;
}
__device__ __forceinline__ bool le_bits(double a, double b) {  // a <= b
  return special(a) || special(b) ? a <= b : order_key(a) <= order_key(b);
}
template <>
__device__ __forceinline__ void euler_riemann<double>(const double* UL, const double* UR,
                                                      const RiemannK<double>& K, int hllc,
                                                      double* F) {
  const double nx = K.tnx, ny = K.tny, gm1 = K.gm1, gg = K.gg;
  struct Side {
    double r, ir, m, t, un, ut, E, p, e, c;
  };
  auto side = [&](const double* U) {
    Side s;
    s.r = U[0], s.E = U[3];
    s.ir = flux_rcp(1.0, s.r);
    s.m = fma(U[1], nx, U[2] * ny);
    s.t = fma(U[2], nx, -(U[1] * ny));
    s.un = s.m * s.ir;
    s.ut = s.t * s.ir;
    s.p = gm1 * fma(-0.5, fma(s.m, s.un, s.t * s.ut), s.E);
    s.e = s.E + s.p;
    const double pp = __double2hiint(s.p) >= 0 || special(s.p) ? s.p : 0.0;
    s.c = flux_sqrt(gg * pp * s.ir);
    return s;
  };
  const Side L = side(UL), R = side(UR);
  // Roe averages and Einfeldt wave speeds (Eq. wavespeed)
  const double D = flux_sqrt(R.r * L.ir);
  const double iden = flux_rcp(1.0, 1.0 + D);
  const double ua = fma(R.un, D, L.un) * iden, va = fma(R.ut, D, L.ut) * iden;
  const double Ha = fma(R.e * R.ir, D, L.e * L.ir) * iden;
  const double ca = flux_sqrt(gm1 * fma(-0.5, fma(ua, ua, va * va), Ha));
  const double l0 = L.un - L.c, l1 = ua - ca, r0 = R.un + R.c, r1 = ua + ca;
  const double SL = le_bits(l0, l1) || special(l1) && l1 != l1 ? l0 : l1;
  const double SR = le_bits(r1, r0) || special(r1) && r1 != r1 ? r0 : r1;
  auto flux = [&](const Side& s, double* f) {
    f[0] = s.m;
    f[1] = fma(s.m, s.un, s.p);
    f[2] = s.m * s.ut;
    f[3] = s.un * s.e;
  };
  double Fx[4];
  if (le_bits(0.0, SL)) {
    flux(L, Fx);
  } else if (le_bits(SR, 0.0)) {
    flux(R, Fx);
  } else {
    double FL[4], FR[4];
    flux(L, FL);
    flux(R, FR);
    const double WL[4] = {L.r, L.m, L.t, L.E}, WR[4] = {R.r, R.m, R.t, R.E};
    const double aL = L.r * (SL - L.un), aR = R.r * (SR - R.un), Dn = aL - aR;
    if (!hllc || __double_as_longlong(Dn) << 1 == 0) {
      const double inv = flux_rcp(1.0, SR - SL), a = SR * inv, b = SL * inv, s = a * SL;
#pragma unroll
      for (int k = 0; k < 4; ++k) Fx[k] = fma(a, FL[k], fma(-b, FR[k], s * (WR[k] - WL[k])));
    } else {
      const double Ss = (R.p - L.p + fma(aL, L.un, -(aR * R.un))) / Dn;
      const bool left = le_bits(0.0, Ss);
      const Side& s = left ? L : R;
      const double S = left ? SL : SR;
      const double Smu = S - s.un, inv = flux_rcp(1.0, S - Ss);
      const double gq = s.r * Smu, f = gq * inv;
      const double es = fma(Smu, s.E, (Ss - s.un) * fma(gq, Ss, s.p)) * inv;
      const double Us[4] = {f, f * Ss, f * s.ut, es};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        Fx[k] = fma(S, Us[k] - (left ? WL[k] : WR[k]), left ? FL[k] : FR[k]);
    }
  }
  F[0] = Fx[0];
  F[1] = fma(Fx[1], nx, -(Fx[2] * ny));
  F[2] = fma(Fx[1], ny, Fx[2] * nx);
  F[3] = Fx[3];
}

// normal advection speed of the scalar equation at face point (x, y): the
// constant velocity, or the rigid rotation omega phi(r) (-(y - y_c), x - x_c)
// of the solid-body case (Sec. 5) with the smoothstep taper phi from 1 at r1
// to 0 at r2 (none when r2 <= r1)
__device__ __forceinline__ double adv_normal(int field, double ax, double ay, double cx,
                                             double cy, double om, double r1, double r2,
                                             double x, double y, double nx, double ny) {
  if (field == 1) {
    const double dx = x - cx, dy = y - cy;
    double phi = 1.0;
    if (r2 > r1) {
      const double r = sqrt(dx * dx + dy * dy);
      if (r >= r2) {
        phi = 0.0;
      } else if (r > r1) {
        const double s = (r - r1) / (r2 - r1);
        phi = 1.0 - s * s * (3.0 - 2.0 * s);
      }
    }
    return om * phi * (-dy * nx + dx * ny);
  }
  return ax * nx + ay * ny;
}

// a <= b in the order the forward solver's min/max use (pairs: lexicographic)
template <typename T>
__device__ __forceinline__ bool le_ord(const T& a, const T& b) {
  if constexpr (std::is_same<T, DF>::value)
    return a.h < b.h || (a.h == b.h && a.l <= b.l);
  else
    return a <= b;
}

// Reverse mode of euler_riemann: given Fb = dJ/dF (face frame rotated back,
// the kernel's output frame), adds (dF/dU_L)^T Fb to ULb and (dF/dU_R)^T Fb
// to URb, with every branch (wave-speed min/max, HLL/HLLC region, HLLC side)
// frozen at the forward state.  The forward values are recomputed first;
// the adjoint statements then run in reverse order of the forward ones.
template <typename T>
__device__ __forceinline__ void euler_riemann_vjp(const T* UL, const T* UR, const RiemannK<T>& K,
                                                  int hllc, const T* Fb, T* ULb, T* URb) {
  const T one = K.one, half = K.half, two = K.one + K.one;
  const T gm1 = K.gm1, gg = K.gg, tnx = K.tnx, tny = K.tny;
  const T zero = one - one;
  // ---- forward
  const T rL = UL[0], rR = UR[0];
  const T irL = one / rL, irR = one / rR;
  const T mnL = UL[1] * tnx + UL[2] * tny, mtL = UL[2] * tnx - UL[1] * tny;
  const T mnR = UR[1] * tnx + UR[2] * tny, mtR = UR[2] * tnx - UR[1] * tny;
  const T unL = mnL * irL, utL = mtL * irL, unR = mnR * irR, utR = mtR * irR;
  const T EL = UL[3], ER = UR[3];
  const T qL = unL * unL + utL * utL, qR = unR * unR + utR * utR;
  const T pL = gm1 * (EL - half * rL * qL), pR = gm1 * (ER - half * rR * qR);
  const T cL = tsqrt(gg * pos_part(pL) * irL), cR = tsqrt(gg * pos_part(pR) * irR);
  const T HL = (EL + pL) * irL, HR = (ER + pR) * irR;
  const T D = tsqrt(rR * irL);
  const T iden = one / (one + D);
  const T ua = (unL + unR * D) * iden, va = (utL + utR * D) * iden;
  const T Ha = (HL + HR * D) * iden;
  const T ca = tsqrt(gm1 * (Ha - half * (ua * ua + va * va)));
  // the branches vmin / vmax take in the forward solver (NaN operands ignored)
  const T am = ua - ca, ap = ua + ca;
  const bool sl0 = le_ord(unL - cL, am) || val(am) != val(am);  // SL from the left state
  const bool sr0 = le_ord(ap, unR + cR) || val(ap) != val(ap);  // SR from the right state
  const T SL = sl0 ? unL - cL : ua - ca;
  const T SR = sr0 ? unR + cR : ua + ca;
  const T mL = rL * unL, mR = rR * unR;
  const T FL[4] = {mL, mL * unL + pL, mL * utL, unL * (EL + pL)};
  const T FR[4] = {mR, mR * unR + pR, mR * utR, unR * (ER + pR)};
  const T WL[4] = {rL, mL, rL * utL, EL};
  const T WR[4] = {rR, mR, rR * utR, ER};
  // ---- reverse
  T Fxb[4];
  Fxb[0] = Fb[0];
  Fxb[1] = Fb[1] * tnx + Fb[2] * tny;
  Fxb[2] = Fb[2] * tnx - Fb[1] * tny;
  Fxb[3] = Fb[3];
  T FLb[4], FRb[4], WLb[4], WRb[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) FLb[k] = FRb[k] = WLb[k] = WRb[k] = zero;
  T SLb = zero, SRb = zero;
  T rLb = zero, rRb = zero, unLb = zero, unRb = zero, utLb = zero, utRb = zero;
  T pLb = zero, pRb = zero, ELb = zero, ERb = zero;
  const bool hll = !hllc || is_zero(rL * (SL - unL) - rR * (SR - unR));
  if (nonneg(SL)) {
#pragma unroll
    for (int k = 0; k < 4; ++k) FLb[k] = Fxb[k];
  } else if (nonneg(-SR)) {
#pragma unroll
    for (int k = 0; k < 4; ++k) FRb[k] = Fxb[k];
  } else if (hll) {
    const T inv = one / (SR - SL), sLR = SL * SR;
    T invb = zero, sLRb = zero;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const T G = SR * FL[k] - SL * FR[k] + sLR * (WR[k] - WL[k]);
      invb = invb + Fxb[k] * G;
      const T Gb = Fxb[k] * inv;
      FLb[k] = Gb * SR;
      FRb[k] = zero - Gb * SL;
      WRb[k] = Gb * sLR;
      WLb[k] = zero - Gb * sLR;
      SRb = SRb + Gb * FL[k];
      SLb = SLb - Gb * FR[k];
      sLRb = sLRb + Gb * (WR[k] - WL[k]);
    }
    SRb = SRb + sLRb * SL;
    SLb = SLb + sLRb * SR;
    const T db = zero - invb * inv * inv;  // d(SR - SL)
    SRb = SRb + db;
    SLb = SLb - db;
  } else {
    const T aL = rL * (SL - unL), aR = rR * (SR - unR);
    const T Nn = pR - pL + aL * unL - aR * unR, Dn = aL - aR;
    const T Ss = Nn / Dn;
    const bool left = nonneg(Ss);
    const T r = left ? rL : rR, un = left ? unL : unR, ut = left ? utL : utR;
    const T p = left ? pL : pR, S = left ? SL : SR, E = left ? EL : ER;
    const T Smu = S - un, gq = r * Smu, den = S - Ss;
    const T f = gq / den;
    const T qs = gq * Ss + p;
    const T es = (Smu * E + (Ss - un) * qs) / den;
    const T Us[4] = {f, f * Ss, f * ut, es};
    const T* Wsd = left ? WL : WR;
    T Sb = zero, Ssb = zero, rb = zero, unb = zero, utb = zero, pb = zero, Eb = zero;
    T Usb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      Sb = Sb + Fxb[k] * (Us[k] - Wsd[k]);
      Usb[k] = S * Fxb[k];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (left) {
        FLb[k] = Fxb[k];
        WLb[k] = zero - S * Fxb[k];
      } else {
        FRb[k] = Fxb[k];
        WRb[k] = zero - S * Fxb[k];
      }
    }
    // Us = (f, f Ss, f ut, es)
    const T fb = Usb[0] + Usb[1] * Ss + Usb[2] * ut;
    Ssb = Ssb + Usb[1] * f;
    utb = utb + Usb[2] * f;
    const T esb = Usb[3];
    // es = (Smu E + (Ss - un) qs) / den, qs = gq Ss + p
    const T numb = esb / den;
    T denb = zero - esb * es / den;
    T Smub = numb * E;
    Eb = Eb + numb * Smu;
    Ssb = Ssb + numb * qs;
    unb = unb - numb * qs;
    const T qsb = numb * (Ss - un);
    T gqb = qsb * Ss;
    Ssb = Ssb + qsb * gq;
    pb = pb + qsb;
    // f = gq / den, den = S - Ss, gq = r Smu, Smu = S - un
    gqb = gqb + fb / den;
    denb = denb - fb * f / den;
    Sb = Sb + denb;
    Ssb = Ssb - denb;
    rb = rb + gqb * Smu;
    Smub = Smub + gqb * r;
    Sb = Sb + Smub;
    unb = unb - Smub;
    // Ss = Nn / Dn, Nn = pR - pL + aL unL - aR unR, Dn = aL - aR
    const T Nb = Ssb / Dn, Dnb = zero - Ssb * Ss / Dn;
    pRb = pRb + Nb;
    pLb = pLb - Nb;
    const T aLb = Nb * unL + Dnb, aRb = zero - Nb * unR - Dnb;
    unLb = unLb + Nb * aL;
    unRb = unRb - Nb * aR;
    // aL = rL (SL - unL), aR = rR (SR - unR)
    rLb = rLb + aLb * (SL - unL);
    SLb = SLb + aLb * rL;
    unLb = unLb - aLb * rL;
    rRb = rRb + aRb * (SR - unR);
    SRb = SRb + aRb * rR;
    unRb = unRb - aRb * rR;
    // the chosen side's variables
    if (left) {
      rLb = rLb + rb; unLb = unLb + unb; utLb = utLb + utb; pLb = pLb + pb; SLb = SLb + Sb;
      ELb = ELb + Eb;
    } else {
      rRb = rRb + rb; unRb = unRb + unb; utRb = utRb + utb; pRb = pRb + pb; SRb = SRb + Sb;
      ERb = ERb + Eb;
    }
  }
  // wave speeds (frozen min / max branches)
  T uab = zero, cab = zero, cLb = zero, cRb = zero;
  if (sl0) {
    unLb = unLb + SLb;
    cLb = cLb - SLb;
  } else {
    uab = uab + SLb;
    cab = cab - SLb;
  }
  if (sr0) {
    unRb = unRb + SRb;
    cRb = cRb + SRb;
  } else {
    uab = uab + SRb;
    cab = cab + SRb;
  }
  // F and W of both sides
  {
    const T mLb = FLb[0] + FLb[1] * unL + FLb[2] * utL + WLb[1];
    unLb = unLb + FLb[1] * mL + FLb[3] * (EL + pL) + mLb * rL;
    pLb = pLb + FLb[1] + FLb[3] * unL;
    utLb = utLb + FLb[2] * mL + WLb[2] * rL;
    ELb = ELb + FLb[3] * unL + WLb[3];
    rLb = rLb + WLb[0] + WLb[2] * utL + mLb * unL;
    const T mRb = FRb[0] + FRb[1] * unR + FRb[2] * utR + WRb[1];
    unRb = unRb + FRb[1] * mR + FRb[3] * (ER + pR) + mRb * rR;
    pRb = pRb + FRb[1] + FRb[3] * unR;
    utRb = utRb + FRb[2] * mR + WRb[2] * rR;
    ERb = ERb + FRb[3] * unR + WRb[3];
    rRb = rRb + WRb[0] + WRb[2] * utR + mRb * unR;
  }
  // Roe averages: ca = sqrt(gm1 (Ha - (ua^2 + va^2)/2)), ua, va, Ha, iden, D
  const T ca2b = cab / (two * ca);
  const T Hab = ca2b * gm1;
  uab = uab - ca2b * gm1 * ua;
  const T vab = zero - ca2b * gm1 * va;
  unLb = unLb + uab * iden;
  unRb = unRb + uab * D * iden;
  utLb = utLb + vab * iden;
  utRb = utRb + vab * D * iden;
  T HLb = Hab * iden, HRb = Hab * D * iden;
  const T idenb = uab * (unL + unR * D) + vab * (utL + utR * D) + Hab * (HL + HR * D);
  const T Db = uab * unR * iden + vab * utR * iden + Hab * HR * iden - idenb * iden * iden;
  const T rrb = Db / (two * D);  // d(rR irL)
  rRb = rRb + rrb * irL;
  T irLb = rrb * rR, irRb = zero;
  // H, c, p, q, u of both sides
  ELb = ELb + HLb * irL;
  pLb = pLb + HLb * irL;
  irLb = irLb + HLb * (EL + pL);
  ERb = ERb + HRb * irR;
  pRb = pRb + HRb * irR;
  irRb = irRb + HRb * (ER + pR);
  {
    // a zero sound speed (clamped or zero pressure) passes nothing back
    const T c2b = is_zero(cL) ? zero : cLb / (two * cL);
    pLb = pLb + c2b * gg * irL;
    irLb = irLb + c2b * gg * pL;
    const T c2bR = is_zero(cR) ? zero : cRb / (two * cR);
    pRb = pRb + c2bR * gg * irR;
    irRb = irRb + c2bR * gg * pR;
  }
  ELb = ELb + pLb * gm1;
  rLb = rLb - pLb * gm1 * half * qL;
  const T qLb = zero - pLb * gm1 * half * rL;
  ERb = ERb + pRb * gm1;
  rRb = rRb - pRb * gm1 * half * qR;
  const T qRb = zero - pRb * gm1 * half * rR;
  unLb = unLb + two * qLb * unL;
  utLb = utLb + two * qLb * utL;
  unRb = unRb + two * qRb * unR;
  utRb = utRb + two * qRb * utR;
  const T mnLb = unLb * irL, mtLb = utLb * irL, mnRb = unRb * irR, mtRb = utRb * irR;
  irLb = irLb + unLb * mnL + utLb * mtL;
  irRb = irRb + unRb * mnR + utRb * mtR;
  rLb = rLb - irLb * irL * irL;
  rRb = rRb - irRb * irR * irR;
  ULb[0] = ULb[0] + rLb;
  ULb[1] = ULb[1] + mnLb * tnx - mtLb * tny;
  ULb[2] = ULb[2] + mnLb * tny + mtLb * tnx;
  ULb[3] = ULb[3] + ELb;
  URb[0] = URb[0] + rRb;
  URb[1] = URb[1] + mnRb * tnx - mtRb * tny;
  URb[2] = URb[2] + mnRb * tny + mtRb * tnx;
  URb[3] = URb[3] + ERb;
}

// (dU_R/dU_L)^T URb added to ULb for the ghost state of a boundary point:
// mirror at a wall, identity at an outflow, constant at inflow and top
template <typename T>
__device__ __forceinline__ void ghost_vjp(int tag, const RiemannK<T>& K, const T* URb, T* ULb) {
  if (tag == TENO_BC_WALL) {
    const T two = K.one + K.one;
    const T mnb = (URb[1] * K.tnx + URb[2] * K.tny) * two;
    ULb[0] = ULb[0] + URb[0];
    ULb[1] = ULb[1] + URb[1] - mnb * K.tnx;
    ULb[2] = ULb[2] + URb[2] - mnb * K.tny;
    ULb[3] = ULb[3] + URb[3];
  } else if (tag == TENO_BC_OUTFLOW) {
#pragma unroll
    for (int k = 0; k < 4; ++k) ULb[k] = ULb[k] + URb[k];
  }
}

// ghost state of a boundary face point (tag: enum teno_bc)
template <typename T>
__device__ __forceinline__ void ghost_state(int tag, const T* UL, double nx, double ny, double x,
                                            double time, double g, T* UR) {
  if (tag == TENO_BC_WALL) {
    T mn = UL[1] * cst<T>(nx) + UL[2] * cst<T>(ny);
    UR[0] = UL[0];
    UR[1] = UL[1] - cst<T>(2.0 * nx) * mn;
    UR[2] = UL[2] - cst<T>(2.0 * ny) * mn;
    UR[3] = UL[3];
    return;
  }
  bool post = tag == TENO_BC_INFLOW;
  if (tag == TENO_BC_TOP) post = x < 0.1667 + (1.0 + 20.0 * time) / 1.732;
  if (tag == TENO_BC_INFLOW || tag == TENO_BC_TOP) {
    double r = post ? 8.0 : 1.4, u = post ? 7.145 : 0.0, v = post ? -4.125 : 0.0;
    double p = post ? 116.8333 : 1.0;
    UR[0] = cst<T>(r);
    UR[1] = cst<T>(r * u);
    UR[2] = cst<T>(r * v);
    UR[3] = cst<T>(p / (g - 1.0) + 0.5 * r * (u * u + v * v));
    return;
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) UR[k] = UL[k];
}

// Groups of NV = 4 values (the states at one Gauss point, the flux of one
// face) as 16-byte accesses; the arrays are cudaMalloc'd and indexed in whole
// groups, so every group starts on a 16-byte boundary.
template <int NV, typename T>
__device__ __forceinline__ void ld_group(const T* p, T (&x)[NV]) {
  if constexpr (NV == 4 && std::is_same<T, float>::value) {
    const float4 q = *(reinterpret_cast<const float4*>(p));
    x[0] = q.x, x[1] = q.y, x[2] = q.z, x[3] = q.w;
  } else if constexpr (NV == 4 && std::is_same<T, DF>::value) {
    const float4 q0 = *(reinterpret_cast<const float4*>(p));
    const float4 q1 = *(reinterpret_cast<const float4*>(p) + 1);
    x[0] = DF{q0.x, q0.y}, x[1] = DF{q0.z, q0.w}, x[2] = DF{q1.x, q1.y}, x[3] = DF{q1.z, q1.w};
  } else if constexpr (NV == 4 && std::is_same<T, double>::value) {
    const double2 q0 = *(reinterpret_cast<const double2*>(p));
    const double2 q1 = *(reinterpret_cast<const double2*>(p) + 1);
    x[0] = q0.x, x[1] = q0.y, x[2] = q1.x, x[3] = q1.y;
  } else {
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = p[v];
  }
}
template <int NV, typename T>
__device__ __forceinline__ void st_group(T* __restrict__ p, const T (&x)[NV]) {
  if constexpr (NV == 4 && std::is_same<T, float>::value) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  } else if constexpr (NV == 4 && std::is_same<T, DF>::value) {
    reinterpret_cast<float4*>(p)[0] = make_float4(x[0].h, x[0].l, x[1].h, x[1].l);
    reinterpret_cast<float4*>(p)[1] = make_float4(x[2].h, x[2].l, x[3].h, x[3].l);
  } else if constexpr (NV == 4 && std::is_same<T, double>::value) {
    reinterpret_cast<double2*>(p)[0] = make_double2(x[0], x[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(x[2], x[3]);
  } else {
#pragma unroll
    for (int v = 0; v < NV; ++v) p[v] = x[v];
  }
}

struct ReconArgs {
  const void* ahat;
  const int32_t* nbr;
  const uint8_t* smask;
  const double* U;
  const float2* Us;  // FP32 hi/lo split of U (mixed precision), [n_var][n_pad]
  void* Uq;
  uint8_t* sel_out;
  const uint8_t* sel_in;
  int64_t n_cell, n_pad;
  double ct, eps;
  int linear, e_entries;
  int scheme;   // 0 TENO, 1 CWENO
  double cw_dK; // CWENO d_K = 1 - 1/d'_K
  double* coef_out;  // characteristic mode: [n_pad][4][m + 15] coefficients out
  int force_near;       // W form: every cell decides through the pair / FP64 fallback
  uint32_t wait_polls;  // bulk-copy kernels: consumer mbarrier poll limit (0: give up at once)
};

// characteristic mode: store the cell's large and directional coefficients of
// variable v for the characteristic finish, in place of selection and
// evaluation: FP64 on the native path, (hi, lo) FP32 pairs on the pair and
// mixed paths (whose finish runs in pair arithmetic on the FP32 pipe)
template <int M, typename TC>
__device__ __forceinline__ void store_coefs(const ReconArgs& a, int64_t c, int v, const TC* acc,
                                            const TC (&as)[kSmallK][kSmallM]) {
  const int64_t base = ((int64_t)c * 4 + v) * (M + kSmallK * kSmallM);
  if constexpr (std::is_same<TC, double>::value) {
    double* o = a.coef_out + base;
#pragma unroll
    for (int l = 0; l < M; ++l) o[l] = acc[l];
#pragma unroll
    for (int k = 0; k < kSmallK; ++k)
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) o[M + k * kSmallM + l] = as[k][l];
  } else {
    float2* o = reinterpret_cast<float2*>(a.coef_out) + base;
    auto pr = [](const TC& x) {
      if constexpr (std::is_same<TC, DF>::value)
        return make_float2(x.h, x.l);
      else
        return make_float2(x, 0.f);
    };
#pragma unroll
    for (int l = 0; l < M; ++l) o[l] = pr(acc[l]);
#pragma unroll
    for (int k = 0; k < kSmallK; ++k)
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) o[M + k * kSmallM + l] = pr(as[k][l]);
  }
  if (a.sel_out) a.sel_out[(int64_t)v * a.n_pad + c] = 8;
}

// CWENO weights (Eqs. CWENOweight, CWENOOptimalLinearweight/02) from the
// smoothness indicators: alpha = d / (beta + eps)^4 with d_K = cw_dK and
// d_k = (1 - d_K)/K over the K present directional stencils; returns the
// factors of P = sK P_K + sum_k s[k] P_k, i.e. sK = w_K / d_K and
// s[k] = w_k - sK d_k (0 for absent stencils).
struct CwenoF {
  double sK, s[kSmallK];
};
// out of line: the CWENO option must not raise the register count of the
// TENO reconstruction kernels that share the finish code
__device__ __noinline__ CwenoF cweno_factors(double b0, double b1, double b2, double bK,
                                             int present, double dK_in, double eps) {
  const double beta[kSmallK + 1] = {b0, b1, b2, bK};
  CwenoF out;
  double& sK = out.sK;
  double* s = out.s;
  const int K = (present & 1) + ((present >> 1) & 1) + ((present >> 2) & 1);
  const double dK = K ? dK_in : 1.0, dk = K ? (1.0 - dK) / K : 0.0;
  double al[kSmallK + 1], sum = 0.0;
#pragma unroll
  for (int k = 0; k <= kSmallK; ++k) {
    const bool pr = k == kSmallK || ((present >> k) & 1);
    const double ib = 1.0 / (beta[k] + eps);
    const double i2 = ib * ib;
    al[k] = pr ? (k == kSmallK ? dK : dk) * (i2 * i2) : 0.0;
    sum += al[k];
  }
  sK = al[kSmallK] / sum / dK;
#pragma unroll
  for (int k = 0; k < kSmallK; ++k) s[k] = ((present >> k) & 1) ? al[k] / sum - sK * dk : 0.0;
  return out;
}

// TENO cutoff and two-step selection in FP64 (Eqs. new_scale_separation,
// normalize, cutoff, TENO_reconstruction111/222): chi_k >= C_T is evaluated as
// gamma_k >= C_T * sum_j gamma_j with gamma = (beta + eps)^-6.
__device__ __forceinline__ uint8_t select_fp64(const double* beta, int present, double ct,
                                               double eps) {
  double g[kSmallK + 1], S = 0.0;
#pragma unroll
  for (int k = 0; k <= kSmallK; ++k) {
    bool pr = k == kSmallK || ((present >> k) & 1);
    double ib = 1.0 / (beta[k] + eps);
    double i2 = ib * ib;
    g[k] = pr ? i2 * i2 * i2 : 0.0;
    S += g[k];
  }
  if (g[kSmallK] >= ct * S) return 8;
  double S2 = g[0] + g[1] + g[2];
  uint8_t sel = 0;
#pragma unroll
  for (int k = 0; k < kSmallK; ++k)
    if (((present >> k) & 1) && g[k] >= ct * S2) sel |= (uint8_t)(1u << k);
  return sel;
}

// FP32 evaluation of chi_k = 1 / sum_j ((beta_k+eps)/(beta_j+eps))^6 over the
// stencils in `mask`; *near is set when chi_k lies within the guard band
// 1e-3 C_T of C_T.  The FP32 betas are within 1.3e-6 (relative) of the FP64
// sums of the same squares, which moves chi by less than 3e-5 relative, so a
// decision outside the band equals the FP64 decision.
__device__ __forceinline__ bool chi_keep32(const float* t, int k, int mask, float ct, bool* near,
                                           float band = 1e-3f) {
  float s = 0.f;
#pragma unroll
  for (int j = 0; j <= kSmallK; ++j) {
    if (!((mask >> j) & 1)) continue;
    float r = t[k] / t[j];
    float r2 = r * r;
    s += r2 * r2 * r2;
  }
  float chi = 1.f / s;
  if (!(fabsf(chi - ct) > band * ct)) *near = true;
  return chi >= ct;
}

// As chi_keep32, for smoothness indicators known only to within a relative
// bound rho each (t_j = beta_j + eps in [t32_j / (1 + rho), t32_j / (1 - rho)]
// or tighter): every ratio t_k / t_j then lies within a factor
// (1 + rho) / (1 - rho) of its FP32 value, so chi lies within the factor
// f = ((1 + rho) / (1 - rho))^6 of the FP32 chi (times 1 + 1e-4 for the FP32
// evaluation itself); *near is set when that interval contains C_T.
__device__ __forceinline__ bool chi_keep32_bound(const float* t, int k, int mask, float ct,
                                                 float f, bool* near) {
  float s = 0.f;
#pragma unroll
  for (int j = 0; j <= kSmallK; ++j) {
    if (!((mask >> j) & 1)) continue;
    float r = t[k] / t[j];
    float r2 = r * r;
    s += r2 * r2 * r2;
  }
  const float chi = 1.f / s;
  if (!(chi > ct * f) && !(chi * f < ct)) *near = true;
  return chi >= ct;
}

// ------------------------------------------------------------ reconstruction
// thread (lane, v, z): cell tile*32 + lane, variable v.  A warp covers the 32
// cells of one tile for one variable, so every matrix entry is one coalesced
// 128/256-byte row; the other variables' warps hit it in L1.
// TA = double: the FP64 path.  TA = float: the mixed path -- stencil
// differences from the hi/lo FP32 split of U (as accurate as an FP64
// subtraction rounded to FP32), FP32 matvecs, FP32 beta and cutoff with an FP64
// fallback inside the guard band, FP32 Gauss-point values.
// selection, final coefficients and Gauss-point values of cell c, variable v
// (FP64-native and FP32-mixed paths)
// kExt: compile the CWENO and characteristic-mode branches (the TENO-only
// instantiations keep the register count of the default kernels down)
template <int M, int NQ, int NV, typename TA, typename TT, bool kExt = true>
__device__ __forceinline__ void plain_finish(const ReconArgs& a, const TT& ev, int64_t c, int v,
                                             double u0, float2 u0s, const TA (&acc)[M],
                                             const TA (&as)[kSmallK][kSmallM],
                                             TA* ostage = nullptr, int present_in = -1) {
  constexpr bool kMixed = std::is_same<TA, float>::value;
  if constexpr (kExt) {
    if (a.coef_out) {
      store_coefs<M, TA>(a, c, v, acc, as);
      return;
    }
  }
  const int present = present_in >= 0 ? present_in : a.smask[c];
  uint8_t sel;
  const bool cweno = kExt && a.scheme == 1 && !a.linear;
  TA cf[M];
  if (cweno) {
    // beta and weights in FP64 (from the FP32 coefficients on the mixed path)
    double beta[kSmallK + 1];
    double b = 0.0;
#pragma unroll
    for (int l = 0; l < M; ++l) b = fma((double)acc[l], (double)acc[l], b);
    beta[kSmallK] = b;
#pragma unroll
    for (int k = 0; k < kSmallK; ++k) {
      double q = 0.0;
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) q = fma((double)as[k][l], (double)as[k][l], q);
      beta[k] = q;
    }
    const CwenoF cw = cweno_factors(beta[0], beta[1], beta[2], beta[kSmallK], present, a.cw_dK,
                                    a.eps);
    const double sK = cw.sK;
    const double* sk = cw.s;
#pragma unroll
    for (int l = 0; l < M; ++l) cf[l] = TA(sK) * acc[l];
#pragma unroll
    for (int k = 0; k < kSmallK; ++k)
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) cf[l] = fma(TA(sk[k]), as[k][l], cf[l]);
    sel = 8;
  } else if (a.sel_in) {
    sel = a.sel_in[(int64_t)v * a.n_pad + c];
  } else if (a.linear) {
    sel = 8;
  } else {
    bool exact = !kMixed;
    if constexpr (kMixed) {
      // FP32 smoothness indicators (orthonormal basis: beta = |a'|^2) and cutoff
      float t[kSmallK + 1];
      {
        float b = 0.f;
#pragma unroll
        for (int l = 0; l < M; ++l) b = fmaf(acc[l], acc[l], b);
        t[kSmallK] = b + (float)a.eps;
#pragma unroll
        for (int k = 0; k < kSmallK; ++k) {
          float q = 0.f;
#pragma unroll
          for (int l = 0; l < kSmallM; ++l) q = fmaf(as[k][l], as[k][l], q);
          t[k] = q + (float)a.eps;
        }
      }
      const float ct = (float)a.ct;
      bool near = false;
      const int all = present | 8;
      if (chi_keep32(t, kSmallK, all, ct, &near)) {
        sel = 8;
      } else {
        sel = 0;
        const int smallm = present & 7;
#pragma unroll
        for (int k = 0; k < kSmallK; ++k)
          if (((present >> k) & 1) && chi_keep32(t, k, smallm, ct, &near))
            sel |= (uint8_t)(1u << k);
      }
      exact = near;
    }
    if (exact) {
      // FP64 smoothness indicators and decision
      double beta[kSmallK + 1];
      double b = 0.0;
#pragma unroll
      for (int l = 0; l < M; ++l) b = fma((double)acc[l], (double)acc[l], b);
      beta[kSmallK] = b;
#pragma unroll
      for (int k = 0; k < kSmallK; ++k) {
        double q = 0.0;
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) q = fma((double)as[k][l], (double)as[k][l], q);
        beta[k] = q;
      }
      sel = select_fp64(beta, present, a.ct, a.eps);
    }
  }
  if (a.sel_out) a.sel_out[(int64_t)v * a.n_pad + c] = sel;
  // final polynomial coefficients
  if (cweno) {
    // formed above
  } else if (sel & 8) {
#pragma unroll
    for (int l = 0; l < M; ++l) cf[l] = acc[l];
  } else {
    int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
    TA w = nd ? TA(1.0) / TA(nd) : TA(0);
#pragma unroll
    for (int l = 0; l < M; ++l) cf[l] = TA(0);
#pragma unroll
    for (int k = 0; k < kSmallK; ++k) {
      if (!((sel >> k) & 1)) continue;
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) cf[l] = fma(w, as[k][l], cf[l]);
    }
  }
  // values at the 3*NQ edge Gauss points: U_0 + Psi' c' (to Uq, or to the
  // caller's shared-memory stage with the same point stride NV)
  TA* __restrict__ out = ostage ? ostage : reinterpret_cast<TA*>(a.Uq) + c * (3 * NQ * NV) + v;
#pragma unroll
  for (int p = 0; p < 3 * NQ; ++p) {
    TA s = TA(0);
#pragma unroll
    for (int l = 0; l < M; ++l) {
      if constexpr (kMixed)
        s = fmaf(cf[l], ev.psi[p * kMaxM + l].x, s);  // FP32 table: hi parts
      else
        s = fma(cf[l], ev.psi[p * kMaxM + l], s);
    }
    if constexpr (kMixed)
      out[p * NV] = u0s.x + (s + u0s.y);
    else
      out[p * NV] = u0 + s;
  }
}


template <int M, int NS, int NQ, int NV, typename TA, typename TT>
__global__ void __launch_bounds__(128) recon_kernel(const ReconArgs a, const TT ev) {
  pdl_wait();
  constexpr bool kMixed = std::is_same<TA, float>::value;
  const int lane = threadIdx.x, v = threadIdx.y;
  const int64_t tile = (int64_t)blockIdx.x * blockDim.z + threadIdx.z;
  const int64_t c = tile * kTile + lane;
  if (c >= a.n_cell) return;
  constexpr int E = M * NS + kSmallEntries;
  constexpr int SL = NS + kSmallSlots;
  const double* Uv = a.U + (int64_t)v * a.n_pad;
  const float2* Usv = kMixed ? a.Us + (int64_t)v * a.n_pad : nullptr;
  double u0 = 0.0;
  float2 u0s = make_float2(0.f, 0.f);
  if constexpr (kMixed)
    u0s = Usv[c];
  else
    u0 = Uv[c];
  const TA* __restrict__ A = reinterpret_cast<const TA*>(a.ahat) + tile * (int64_t)E * kTile + lane;
  const int32_t* __restrict__ nb = a.nbr + tile * (int64_t)SL * kTile + lane;
  auto diff = [&](int j) -> TA {
    if constexpr (kMixed) {
      const float2 q = Usv[j];
      return (q.x - u0s.x) + (q.y - u0s.y);
    } else {
      return Uv[j] - u0;
    }
  };

  // large stencil: a' = A'' d  (d_s = U_s - U_0)
  TA acc[M];
#pragma unroll
  for (int l = 0; l < M; ++l) acc[l] = TA(0);
#pragma unroll (std::is_same<TA, float>::value ? kSlotUnrollMixed : kSlotUnroll)
  for (int s = 0; s < NS; ++s) {
    const TA d = diff(__ldg(nb + s * kTile));
    const TA* As = A + (int64_t)s * M * kTile;
#pragma unroll
    for (int l = 0; l < M; ++l) acc[l] = fma(__ldg(As + l * kTile), d, acc[l]);
  }
  // directional stencils
  TA as[kSmallK][kSmallM];
#pragma unroll
  for (int k = 0; k < kSmallK; ++k) {
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) as[k][l] = TA(0);
#pragma unroll (std::is_same<TA, float>::value ? kSlotUnrollMixed : kSlotUnroll)
    for (int s = 0; s < kSmallN; ++s) {
      const TA d = diff(__ldg(nb + (NS + k * kSmallN + s) * kTile));
      const TA* As = A + (int64_t)(M * NS + (k * kSmallN + s) * kSmallM) * kTile;
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) as[k][l] = fma(__ldg(As + l * kTile), d, as[k][l]);
    }
  }
  plain_finish<M, NQ, NV, TA, TT>(a, ev, c, v, u0, u0s, acc, as);
}

// FP64-accurate reconstruction with double-float arithmetic on the FP32 pipe:
// stencil differences from the (hi, lo) split of U, matvecs, beta and the
// Gauss-point evaluation in pairs (relative error ~2^-46 of the summed
// magnitudes); the cutoff is decided in FP32 with the guard band of the mixed
// path and in FP64 inside it; Gauss-point values are written in FP64.
// selection, final coefficients and Gauss-point values of cell c, variable v
// (double-float path), from the normalised stencil coefficients
template <int M, int NQ, int NV, bool kExt = true>
__device__ __forceinline__ void df_finish(const ReconArgs& a, const DFTable& ev, int64_t c, int v,
                                          const DF (&acc)[M],
                                          const DF (&as)[kSmallK][kSmallM],
                                          float2* ostage = nullptr, int present_in = -1) {
  if constexpr (kExt) {
    if (a.coef_out) {
      store_coefs<M, DF>(a, c, v, acc, as);
      return;
    }
  }
  const int present = present_in >= 0 ? present_in : a.smask[c];
  uint8_t sel;
  const bool cweno = kExt && a.scheme == 1 && !a.linear;
  DF cf[M];
  if (cweno) {
    // beta = |a'|^2 in pairs, weights in FP64, combination in pairs
    double beta[kSmallK + 1];
    {
      DF b = {0.f, 0.f};
#pragma unroll
      for (int l = 0; l < M; ++l) df_mac(b, make_float2(acc[l].h, acc[l].l), acc[l]);
      beta[kSmallK] = df_to_double(df_norm(b));
#pragma unroll
      for (int k = 0; k < kSmallK; ++k) {
        DF q = {0.f, 0.f};
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) df_mac(q, make_float2(as[k][l].h, as[k][l].l), as[k][l]);
        beta[k] = df_to_double(df_norm(q));
      }
    }
    const CwenoF cw = cweno_factors(beta[0], beta[1], beta[2], beta[kSmallK], present, a.cw_dK,
                                    a.eps);
    const double sK = cw.sK;
    const double* sk = cw.s;
    const DF fK = cst<DF>(sK);
#pragma unroll
    for (int l = 0; l < M; ++l) cf[l] = fK * acc[l];
#pragma unroll
    for (int k = 0; k < kSmallK; ++k) {
      const DF fk = cst<DF>(sk[k]);
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) cf[l] = cf[l] + fk * as[k][l];
    }
    sel = 8;
  } else if (a.sel_in) {
    sel = a.sel_in[(int64_t)v * a.n_pad + c];
  } else if (a.linear) {
    sel = 8;
  } else {
    // beta = |a'|^2 in pairs
    DF bt[kSmallK + 1];
    {
      DF b = {0.f, 0.f};
#pragma unroll
      for (int l = 0; l < M; ++l) df_mac(b, make_float2(acc[l].h, acc[l].l), acc[l]);
      bt[kSmallK] = df_norm(b);
#pragma unroll
      for (int k = 0; k < kSmallK; ++k) {
        DF q = {0.f, 0.f};
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) df_mac(q, make_float2(as[k][l].h, as[k][l].l), as[k][l]);
        bt[k] = df_norm(q);
      }
    }
    float t[kSmallK + 1];
#pragma unroll
    for (int k = 0; k <= kSmallK; ++k) t[k] = bt[k].h + (float)a.eps;
    const float ct = (float)a.ct;
    bool near = false;
    if (chi_keep32(t, kSmallK, present | 8, ct, &near)) {
      sel = 8;
    } else {
      sel = 0;
#pragma unroll
      for (int k = 0; k < kSmallK; ++k)
        if (((present >> k) & 1) && chi_keep32(t, k, present & 7, ct, &near))
          sel |= (uint8_t)(1u << k);
    }
    if (near) {
      double beta[kSmallK + 1];
#pragma unroll
      for (int k = 0; k <= kSmallK; ++k) beta[k] = df_to_double(bt[k]);
      sel = select_fp64(beta, present, a.ct, a.eps);
    }
  }
  if (a.sel_out) a.sel_out[(int64_t)v * a.n_pad + c] = sel;
  if (cweno) {
    // coefficients formed above
  } else if (sel & 8) {
#pragma unroll
    for (int l = 0; l < M; ++l) cf[l] = acc[l];
  } else {
    // equal weights: sum the kept polynomials, then divide by their number
    const int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
    const float fn = (float)(nd ? nd : 1);
#pragma unroll
    for (int l = 0; l < M; ++l) cf[l] = {0.f, 0.f};
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) {
      DF sum = {0.f, 0.f};
#pragma unroll
      for (int k = 0; k < kSmallK; ++k) {
        if (!((sel >> k) & 1)) continue;
        DF q = two_sum(sum.h, as[k][l].h);
        q.l += sum.l + as[k][l].l;
        sum = two_sum(q.h, q.l);
      }
      const float qh = sum.h / fn;
      const float r = fmaf(-qh, fn, sum.h);  // exact remainder
      cf[l] = two_sum(qh, (r + sum.l) / fn);
      if (!nd) cf[l] = {0.f, 0.f};
    }
  }
  // Gauss-point values as (hi, lo) pairs: split(U_0) + Psi' c'
  const float2 u0s = a.Us[(int64_t)v * a.n_pad + c];
  float2* __restrict__ out =
      ostage ? ostage : reinterpret_cast<float2*>(a.Uq) + c * (3 * NQ * NV) + v;
#pragma unroll
  for (int p = 0; p < 3 * NQ; ++p) {
    DF s = {0.f, 0.f};
#pragma unroll
    for (int l = 0; l < M; ++l) df_mac(s, ev.psi[p * kMaxM + l], cf[l]);
    const DF r = DF{u0s.x, u0s.y} + df_norm(s);
    out[p * NV] = make_float2(r.h, r.l);
  }
}


template <int M, int NS, int NQ, int NV>
__global__ void __launch_bounds__(128) recon_df_kernel(const ReconArgs a, const DFTable ev) {
  pdl_wait();
  const int lane = threadIdx.x, v = threadIdx.y;
  const int64_t tile = (int64_t)blockIdx.x * blockDim.z + threadIdx.z;
  const int64_t c = tile * kTile + lane;
  if (c >= a.n_cell) return;
  constexpr int E = M * NS + kSmallEntries;
  constexpr int SL = NS + kSmallSlots;
  const float2* Usv = a.Us + (int64_t)v * a.n_pad;
  const float2 u0s = Usv[c];
  const float2* __restrict__ A =
      reinterpret_cast<const float2*>(a.ahat) + tile * (int64_t)E * kTile + lane;
  const int32_t* __restrict__ nb = a.nbr + tile * (int64_t)SL * kTile + lane;
  auto diff = [&](int j) -> DF {
    const float2 q = Usv[j];
    DF s = two_sum(q.x, -u0s.x);
    s.l += q.y - u0s.y;
    return two_sum(s.h, s.l);
  };
  DF acc[M];
#pragma unroll
  for (int l = 0; l < M; ++l) acc[l] = {0.f, 0.f};
#pragma unroll (kSlotUnroll)
  for (int s = 0; s < NS; ++s) {
    const DF d = diff(__ldg(nb + s * kTile));
    const float2* As = A + (int64_t)s * M * kTile;
#pragma unroll
    for (int l = 0; l < M; ++l) df_mac(acc[l], __ldg(As + l * kTile), d);
  }
#pragma unroll
  for (int l = 0; l < M; ++l) acc[l] = df_norm(acc[l]);
  DF as[kSmallK][kSmallM];
#pragma unroll
  for (int k = 0; k < kSmallK; ++k) {
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) as[k][l] = {0.f, 0.f};
#pragma unroll (kSlotUnroll)
    for (int s = 0; s < kSmallN; ++s) {
      const DF d = diff(__ldg(nb + (NS + k * kSmallN + s) * kTile));
      const float2* As = A + (int64_t)(M * NS + (k * kSmallN + s) * kSmallM) * kTile;
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) df_mac(as[k][l], __ldg(As + l * kTile), d);
    }
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) as[k][l] = df_norm(as[k][l]);
  }
  df_finish<M, NQ, NV>(a, ev, c, v, acc, as);
}

// ------------------------------------------ halo-staged reconstruction
// The union of the stencils of a 32-cell tile (its "halo", <= kHaloMax cells,
// listed on the host) is gathered once into shared memory; every stencil
// difference then reads shared memory, and the only global stream of the
// main loop is the coalesced, independent stream of per-cell matrices.
// kMode 0: FP64 path (double-float), 1: FP32-mixed, 2: FP64 native.
template <int kMode>
struct HaloTraits;
template <>
struct HaloTraits<0> {
  using TE = float2;   // matrix entry
  using TS = float2;   // staged state (hi, lo split)
  using Acc = DF;
  using Tab = DFTable;
};
template <>
struct HaloTraits<1> {
  using TE = float;
  using TS = float2;
  using Acc = float;
  using Tab = DFTable;
};
template <>
struct HaloTraits<2> {
  using TE = double;
  using TS = double;
  using Acc = double;
  using Tab = EvalTable;
};

template <int M, int NS, int NQ, int NV, int kMode>
__global__ void __launch_bounds__(128) recon_halo_kernel(const ReconArgs a, const HaloArgs h,
                                                         const typename HaloTraits<kMode>::Tab ev) {
  pdl_wait();
  using TR = HaloTraits<kMode>;
  using TE = typename TR::TE;
  using TS = typename TR::TS;
  using Acc = typename TR::Acc;
  constexpr int TZ = 4 / NV;
  constexpr int E = M * NS + kSmallEntries;
  constexpr int SL = NS + kSmallSlots;
  __shared__ TS hs[TZ][NV][kHaloMax];
  const int lane = threadIdx.x, v = threadIdx.y, z = threadIdx.z;
  const int64_t n_tiles = (a.n_cell + kTile - 1) / kTile;
  const int64_t tile = (int64_t)blockIdx.x * TZ + z;
  const bool tvalid = tile < n_tiles;
  // cooperative gather of the tile's halo states (all vars) by its NV warps
  if (tvalid) {
    const int h0 = h.off[tile], H = h.off[tile + 1] - h0;
    for (int i = lane + kTile * v; i < H; i += kTile * NV) {
      const int id = __ldg(h.ids + h0 + i);
#pragma unroll
      for (int w = 0; w < NV; ++w) {
        if constexpr (kMode == 2)
          hs[z][w][i] = a.U[(int64_t)w * a.n_pad + id];
        else
          hs[z][w][i] = a.Us[(int64_t)w * a.n_pad + id];
      }
    }
  }
  __syncthreads();
  if (!tvalid) return;
  const int64_t c = tile * kTile + lane;  // pad lanes compute, but store nothing
  const int64_t cc = c < a.n_cell ? c : 0;
  double u0 = 0.0;
  float2 u0s = make_float2(0.f, 0.f);
  if constexpr (kMode == 2)
    u0 = a.U[(int64_t)v * a.n_pad + cc];
  else
    u0s = a.Us[(int64_t)v * a.n_pad + cc];
  const TS* __restrict__ st = hs[z][v];
  const TE* __restrict__ A = reinterpret_cast<const TE*>(a.ahat) + tile * (int64_t)E * kTile + lane;
  const uint16_t* __restrict__ nb = h.nbr_loc + tile * (int64_t)SL * kTile + lane;
  auto dif = [&](int s) -> Acc {
    const TS q = st[__ldg(nb + s * kTile) & kHaloPosMask];
    if constexpr (kMode == 0) {
      DF t = two_sum(q.x, -u0s.x);
      t.l += q.y - u0s.y;
      return two_sum(t.h, t.l);
    } else if constexpr (kMode == 1) {
      return (q.x - u0s.x) + (q.y - u0s.y);
    } else {
      return q - u0;
    }
  };
  auto mac = [](Acc& acc, TE m, Acc d) {
    if constexpr (kMode == 0)
      df_mac(acc, m, d);
    else
      acc = fma(m, d, acc);
  };
  Acc acc[M];
#pragma unroll
  for (int l = 0; l < M; ++l) acc[l] = Acc{};
#pragma unroll (kMode == 1 ? kSlotUnrollMixed : kSlotUnroll)
  for (int s = 0; s < NS; ++s) {
    const Acc d = dif(s);
    const TE* As = A + (int64_t)s * M * kTile;
#pragma unroll
    for (int l = 0; l < M; ++l) mac(acc[l], __ldg(As + l * kTile), d);
  }
  Acc as[kSmallK][kSmallM];
#pragma unroll
  for (int k = 0; k < kSmallK; ++k) {
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) as[k][l] = Acc{};
#pragma unroll (kMode == 1 ? kSlotUnrollMixed : kSlotUnroll)
    for (int s = 0; s < kSmallN; ++s) {
      const Acc d = dif(NS + k * kSmallN + s);
      const TE* As = A + (int64_t)(M * NS + (k * kSmallN + s) * kSmallM) * kTile;
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) mac(as[k][l], __ldg(As + l * kTile), d);
    }
  }
  if (c >= a.n_cell) return;
  if constexpr (kMode == 0) {
#pragma unroll
    for (int l = 0; l < M; ++l) acc[l] = df_norm(acc[l]);
#pragma unroll
    for (int k = 0; k < kSmallK; ++k)
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) as[k][l] = df_norm(as[k][l]);
    df_finish<M, NQ, NV, false>(a, ev, c, v, acc, as);
  } else if constexpr (kMode == 1) {
    plain_finish<M, NQ, NV, float, DFTable, false>(a, ev, c, v, 0.0, u0s, acc, as);
  } else {
    plain_finish<M, NQ, NV, double, EvalTable, false>(a, ev, c, v, u0, u0s, acc, as);
  }
}

// -------------------------------------------- TMA-staged reconstruction
// The per-cell matrices of a 32-cell tile are one contiguous block of global
// memory ([tile][entry][32]).  One producer lane streams that block into a
// ring of kRing shared-memory buffers with 1D bulk copies (cp.async.bulk,
// completion counted in bytes on the buffer's "full" mbarrier); the four
// consumer warps of the tile (one per conservative variable) wait on "full",
// accumulate from shared memory, and release the buffer on its "empty"
// mbarrier.  Every wait is bounded.  A wait that gives up sets bit 1 of the
// error flag and the block's abort flag in shared memory; from then on the
// consumers skip every wait and all work but still pass the consumer-only
// barriers of the remaining tiles (so no warp is left at a barrier), and the
// producer stops issuing, waits (bounded) for the copies it has in flight and
// returns.
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
constexpr uint32_t kWaitLimit = 1u << 22;
// wait for the completion of the phase with the given parity; false on give-up
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t i = 0; i < kWaitLimit; ++i)
    if (mbar_test(bar, parity)) return true;
  return false;
}
// as mbar_wait, also watching the block's abort flag: 1 phase complete, 0 gave
// up, 2 another thread of the block gave up first
__device__ __forceinline__ int mbar_wait_or_abort(uint64_t* bar, uint32_t parity,
                                                  const volatile int* abort,
                                                  uint32_t limit = kWaitLimit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_test(bar, parity)) return 1;
    if (*abort) return 2;
  }
  return 0;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

constexpr int kRing = 4;
constexpr int kConsumers = 4;  // one warp per conservative variable (Euler)

// cp.async (8-byte asynchronous global->shared copies) for the halo prefetch
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
// 16-byte asynchronous copy (both addresses 16-byte aligned), L2 only
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// barrier of the four consumer warps only (the producer warp does not take part)
__device__ __forceinline__ void consumer_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kConsumers * kTile) : "memory");
}

// Stage j of a tile's matrix block: kLPS large-stencil slots, or kSPS slots of
// one directional stencil.
template <int M, int NS, int kEsz, int kLPS, int kSPS, int kRingT = kRing>
struct StagePlan {
  static constexpr int kSlotL = M * kTile * kEsz;
  static constexpr int kSlotS = kSmallM * kTile * kEsz;
  static constexpr int kNL = (NS + kLPS - 1) / kLPS;
  static constexpr int kPerSmall = kSmallN / kSPS;
  static constexpr int kStages = kNL + kSmallK * kPerSmall;
  static constexpr int kMatL = kLPS * kSlotL, kMatS = kSPS * kSlotS;
  static constexpr int kMaxSlots = kLPS > kSPS ? kLPS : kSPS;
  static constexpr int kSlotN = kTile * 2;  // halo positions (uint16) of one slot
  // ring buffer: [matrix rows][halo positions]
  static constexpr int kNOff = kMatL > kMatS ? kMatL : kMatS;
  static constexpr int kMat = kNOff + kMaxSlots * kSlotN;
  static constexpr int kSL = NS + kSmallSlots;
  static constexpr int kE = M * NS + kSmallEntries;
  static constexpr int64_t kTileBytes = (int64_t)kE * kTile * kEsz;
  static constexpr size_t kHaloBytes = (size_t)2 * 4 * kHaloMax * sizeof(float2);
  static constexpr size_t kSmem =
      (size_t)kRingT * kMat + kHaloBytes + 2 * kRingT * sizeof(uint64_t) + 16;
  static_assert(kSmallN % kSPS == 0, "directional stencil split");
  static_assert(kMat % 16 == 0, "16-byte aligned buffers");
  __device__ static void stage(int j, int& slot0, int& nslot, int64_t& off, int& bytes, int& k) {
    if (j < kNL) {
      slot0 = j * kLPS;
      nslot = (NS - slot0) < kLPS ? (NS - slot0) : kLPS;
      off = (int64_t)slot0 * kSlotL;
      bytes = nslot * kSlotL;
      k = -1;
    } else {
      const int i = j - kNL;
      k = i / kPerSmall;
      const int s0 = (i % kPerSmall) * kSPS;
      slot0 = NS + k * kSmallN + s0;
      nslot = kSPS;
      off = (int64_t)(M * NS + (k * kSmallN + s0) * kSmallM) * kTile * kEsz;
      bytes = kSPS * kSlotS;
    }
  }
};

template <bool kDF, int M, int NS, int NQ>
struct TmaTraits {
  using TE = float2;  // matrix entry: (hi, lo)
  using Acc = DF;
  static constexpr int kLPS = 4, kSPS = 4, kRing = 4;
};
template <int M, int NS, int NQ>
struct TmaTraits<false, M, NS, NQ> {
  using TE = float;
  using Acc = float;
  static constexpr int kLPS = 4, kSPS = 4, kRing = 4;
};

// Halo prefetch pipeline of the bulk-copy reconstruction kernels (consumer
// threads).  The cp.async copies of a tile's halo need its halo ids, and the
// ids need the tile's halo offsets: the offsets are loaded two tiles ahead
// and the ids one tile ahead (two per thread: a halo has at most 256 cells
// and there are 128 consumer threads), so issuing the copies never waits on
// a global load.  Tiles advance by the grid size.
struct HaloPipe {
  static constexpr int kCT = kConsumers * kTile;
  static_assert(kHaloMax <= 2 * kCT, "two halo ids per consumer thread");
  const HaloArgs& h;
  const float2* Us;
  int64_t n_pad, n_tiles;
  int tid;
  int H1 = 0, id0 = 0, id1 = 0;  // ids of the next tile
  int h02 = 0, H2 = 0;           // offsets of the tile after it
  __device__ HaloPipe(const HaloArgs& h_, const float2* Us_, int64_t n_pad_, int64_t n_tiles_,
                      int tid_)
      : h(h_), Us(Us_), n_pad(n_pad_), n_tiles(n_tiles_), tid(tid_) {}
  __device__ void offsets(int64_t tile, int& h0, int& H) const {
    h0 = 0, H = 0;
    if (tile < n_tiles) {
      h0 = h.off[tile];
      H = h.off[tile + 1] - h0;
    }
  }
  __device__ void ids(int h0, int H) {
    H1 = H, id0 = 0, id1 = 0;
    if (tid < H) id0 = __ldg(h.ids + h0 + tid);
    if (tid + kCT < H) id1 = __ldg(h.ids + h0 + tid + kCT);
  }
  // copies of the halo whose ids are held into buffer hb, one commit group
  __device__ void issue(float2* halo, int hb) const {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      if (tid < H1) cp_async8(&halo[(hb * 4 + w) * kHaloMax + tid], Us + (int64_t)w * n_pad + id0);
      if (tid + kCT < H1)
        cp_async8(&halo[(hb * 4 + w) * kHaloMax + tid + kCT], Us + (int64_t)w * n_pad + id1);
    }
    cp_async_commit();
  }
  // prologue: the first tile's halo into buffer 0 (waits once), the ids of
  // the second tile and the offsets of the third
  __device__ void start(int64_t t0, int64_t G, float2* halo) {
    int h0, H;
    offsets(t0, h0, H);
    ids(h0, H);
    issue(halo, 0);
    offsets(t0 + G, h0, H);
    ids(h0, H);
    offsets(t0 + 2 * G, h02, H2);
  }
  // at tile t: the halo of t + G into buffer hb (an empty group past the
  // end), then the ids of t + 2G and the offsets of t + 3G
  __device__ void advance(int64_t t, int64_t G, float2* halo, int hb) {
    issue(halo, hb);
    ids(h02, H2);
    offsets(t + 3 * G, h02, H2);
  }
};

// Persistent kernel, Euler only.  Producer lane: the matrix block of every
// tile in kRing-deep bulk-copy stages.  Consumer warps (one per variable):
// the tile's stencil halo in a double-buffered shared-memory area, prefetched
// with cp.async one tile ahead; stencil differences from the halo, matrices
// from the ring.  kDF: FP64 path (double-float); !kDF: FP32-mixed path.
// CWENO and the characteristic mode only (the other modes of variant 2 have
// the W form and the tile kernel; with these modes' finish, which takes most of
// the registers and of a tile's time, the tile kernel's form measured slower at
// orders 5 and 6 on the pair path: 384 us against 490, 80,000 cells CWENO6).
// The pair kernel is held to two blocks per SM: uncapped it took 252 registers
// at TENO6, one block (five warps) per SM.
template <int M, int NS, int NQ, bool kDF>
__global__ void __launch_bounds__(kTile * (kConsumers + 1), kDF ? 2 : 0)
    recon_tma_kernel(const ReconArgs a, const HaloArgs h, const DFTable ev, int* err) {
  using TR = TmaTraits<kDF, M, NS, NQ>;
  using TE = typename TR::TE;
  constexpr int kRing = TR::kRing;
  using P = StagePlan<M, NS, (int)sizeof(TE), TR::kLPS, TR::kSPS, kRing>;
  constexpr int NV = 4;
  constexpr int SL = NS + kSmallSlots;
  extern __shared__ __align__(128) unsigned char smem[];
  float2* halo = reinterpret_cast<float2*>(smem + (size_t)kRing * P::kMat);  // [2][NV][kHaloMax]
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)kRing * P::kMat + P::kHaloBytes);
  uint64_t* empty = full + kRing;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + kRing);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_tiles = (a.n_cell + kTile - 1) / kTile;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int i = 0; i < kRing; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kConsumers);
    }
    mbar_fence_init();
  }
  __syncthreads();
  if (warp == kConsumers) {
    // ---- producer lane: matrix blocks, tile after tile
    if (lane == 0) {
      int64_t g = 0;
      for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const unsigned char* src =
            reinterpret_cast<const unsigned char*>(a.ahat) + tile * P::kTileBytes;
        const unsigned char* sn =
            reinterpret_cast<const unsigned char*>(h.nbr_loc) + tile * (int64_t)P::kSL * P::kSlotN;
        for (int j = 0; j < P::kStages; ++j, ++g) {
          const int b = (int)(g % kRing);
          if (g >= kRing) {
            const int w = mbar_wait_or_abort(&empty[b], (uint32_t)((g / kRing) - 1) & 1, abort_flag);
            if (w != 1) {
              if (w == 0) {
                atomicOr(err, 2);
                *abort_flag = 1;
              }
              for (int64_t i = g - kRing; i < g; ++i)
                mbar_wait(&full[i % kRing], (uint32_t)(i / kRing) & 1);
              return;
            }
          }
          int slot0, nslot, bytes, k;
          int64_t off;
          P::stage(j, slot0, nslot, off, bytes, k);
          const uint32_t bn = (uint32_t)(nslot * P::kSlotN);
          unsigned char* dst = smem + (size_t)b * P::kMat;
          mbar_expect_tx(&full[b], (uint32_t)bytes + bn);
          bulk_g2s(dst, src + off, (uint32_t)bytes, &full[b]);
          bulk_g2s(dst + P::kNOff, sn + slot0 * P::kSlotN, bn, &full[b]);
        }
      }
      // the block must not exit while a copy it issued is in flight (the
      // consumers skip their waits once a wait has given up)
      for (int64_t i = g > kRing ? g - kRing : 0; i < g; ++i)
        mbar_wait(&full[i % kRing], (uint32_t)(i / kRing) & 1);
    }
    return;
  }
  // ---- consumers
  pdl_wait();  // the states (the producer streams constant data before it)
  const int v = warp, tid = threadIdx.x;
  using Acc = typename TR::Acc;
  HaloPipe hp(h, a.Us, a.n_pad, n_tiles, tid);
  auto mac = [](Acc& acc, TE m, Acc d) {
    if constexpr (kDF)
      df_mac(acc, m, d);
    else
      acc = fmaf(m, d, acc);
  };
  int64_t g = 0;
  int hb = 0;
  bool dead = false;  // a bounded wait of this block gave up: skip all work
  hp.start(blockIdx.x, gridDim.x, halo);
  // the cell's own split state and stencil mask, loaded a tile ahead
  auto own = [&](int64_t tile, float2& u, int& pm) {
    const int64_t cc = tile * kTile + lane;
    const int64_t ci = (tile < n_tiles && cc < a.n_cell) ? cc : 0;
    u = a.Us[(int64_t)v * a.n_pad + ci];
    pm = a.smask[ci];
  };
  float2 u0n;
  int pmn;
  own(blockIdx.x, u0n, pmn);
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, hb ^= 1) {
    consumer_sync();  // every consumer is done with the other halo buffer
    hp.advance(tile, gridDim.x, halo, hb ^ 1);  // halo of the next tile, ids a tile ahead
    const float2 u0s = u0n;
    const int present = pmn;
    own(tile + gridDim.x, u0n, pmn);
    cp_async_wait<1>();  // this thread's copies of the current halo have landed
    consumer_sync();     // ... and everyone's
    const float2* st = halo + (hb * NV + v) * kHaloMax;
    const uint16_t* nb = h.nbr_loc + tile * (int64_t)SL * kTile + lane;
    const int64_t c = tile * kTile + lane;  // may be a pad lane of the last tile
    auto dif = [&](int idx) -> Acc {
      const float2 q = st[idx];
      if constexpr (kDF) {
        DF t = two_sum(q.x, -u0s.x);
        t.l += q.y - u0s.y;
        return two_sum(t.h, t.l);
      } else {
        return (q.x - u0s.x) + (q.y - u0s.y);
      }
    };
    Acc acc[M];
    Acc as[kSmallK][kSmallM];
#pragma unroll
    for (int l = 0; l < M; ++l) acc[l] = Acc{};
#pragma unroll
    for (int k = 0; k < kSmallK; ++k)
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) as[k][l] = Acc{};
    for (int j = 0; j < P::kStages; ++j, ++g) {
      const int b = (int)(g % kRing);
      int slot0, nslot, bytes, k;
      int64_t off;
      P::stage(j, slot0, nslot, off, bytes, k);
      if (!dead) {
        const int w =
            mbar_wait_or_abort(&full[b], (uint32_t)(g / kRing) & 1, abort_flag, a.wait_polls);
        if (w == 0) {
          atomicOr(err, 2);
          *abort_flag = 1;
        }
        dead = __any_sync(0xffffffffu, w != 1);
      }
      const TE* mat = reinterpret_cast<const TE*>(smem + (size_t)b * P::kMat) + lane;
      const uint16_t* nl = reinterpret_cast<const uint16_t*>(smem + (size_t)b * P::kMat + P::kNOff) + lane;
      if (dead) {
        // skip the stage
      } else if (k < 0) {
#pragma unroll
        for (int s = 0; s < TR::kLPS; ++s) {
          if (s < nslot) {
            const Acc d = dif(nl[s * kTile] & kHaloPosMask);
#pragma unroll
            for (int l = 0; l < M; ++l) mac(acc[l], mat[(s * M + l) * kTile], d);
          }
        }
      } else {
#pragma unroll
        for (int kk = 0; kk < kSmallK; ++kk) {
          if (kk != k) continue;
#pragma unroll
          for (int s = 0; s < TR::kSPS; ++s) {
            const Acc d = dif(nl[s * kTile] & kHaloPosMask);
#pragma unroll
            for (int l = 0; l < kSmallM; ++l) mac(as[kk][l], mat[(s * kSmallM + l) * kTile], d);
          }
        }
      }
      __syncwarp();
      if (lane == 0 && !dead) mbar_arrive(&empty[b]);
    }
    if (!dead && c < a.n_cell) {
      if constexpr (kDF) {
#pragma unroll
        for (int l = 0; l < M; ++l) acc[l] = df_norm(acc[l]);
#pragma unroll
        for (int k = 0; k < kSmallK; ++k)
#pragma unroll
          for (int l = 0; l < kSmallM; ++l) as[k][l] = df_norm(as[k][l]);
        df_finish<M, NQ, NV, true>(a, ev, c, v, acc, as, nullptr, present);
      } else {
        plain_finish<M, NQ, NV, float, DFTable, true>(a, ev, c, v, 0.0, u0s, acc, as, nullptr,
                                                      present);
      }
    }
  }
  cp_async_wait<0>();
}

// ------------------------------------------- FP64 paths, W form (variant 2)
// The reconstruction with the work split by what each quantity needs:
//  - the Gauss-point values of the large polynomial are U_0 + W d with
//    W = Psi' G precomputed per cell.  The sums W d run in fixed point: the
//    tile's halo states become integers Y of one power-of-two unit per tile
//    and variable, relative to the tile's first cell, so differences are exact
//    integer subtractions, and W is stored in fixed point with one unit per
//    cell (WDot).  A product costs an FP64 multiply-add 64 lane slots (GB300's
//    FP64 rate is 1/64 of its FP32 rate) and a pair multiply-add 12 FP32
//    instructions; here it costs three wide integer multiply-adds (FP64 path;
//    each holds its pipe for about 5 clocks a warp) or one and two FP32
//    multiply-adds (pairs).  The states' rounding to the tile's unit is one of
//    the largest difference in the tile, up to 2^-51 of it (pairs) or 2^-57; where
//    that is more than some cell's own rounding (the small side of a jump that
//    the tile holds, own_scale) the tile's integers take 62 bits and each lane the
//    bits of them that its cell needs, and cells for which these do not do either
//    are summed in floating point (w_direct);
//  - the smoothness indicators feed only the cutoff decision.  beta = |a|^2
//    for the coefficients a = G d; the part of a in the row space of Psi' is
//    a linear image T y of the values y = W d that are known anyway, so only
//    the rows Q2' G of its orthogonal complement (m - 3 N_q of m) are stored
//    and summed, in FP32, with a rigorous error bound: 5,770 bytes a cell at
//    TENO6, where W with all rows and their bounds took 8,046.  Where the
//    bound does not separate chi from C_T the coefficients and beta are
//    recomputed (pairs, or FP64) and the decision is taken in FP64;
//  - directional values (cells where the large stencil is cut) are evaluated
//    from the (hi, lo) or FP64 matrices.
// The last two are lists a warp works off apart from its tiles: one undecided
// cell at a time by all lanes, 32 directional cells one per lane, so that their
// chains of loads stall the warp once and not per cell and slot.
// Bound: HBM and issue at large meshes (1.56 GB a launch at 262,088 cells TENO6:
// 341 us, 318 without the look at the cells' own scales; with pair products, all
// rows and per-tile block barriers 470 us), the FP64 path by issue at four
// consumer warps a block and four blocks (131,072 cells: 235 us; FP64
// multiply-adds 608 us), small meshes by the time of one tile (2,046 cells TENO5:
// 39 us, 52 before).

// Variables a consumer warp takes: two on the pair path, where the sums of
// both share every shared-memory read of W and of the rows (262,088 cells,
// TENO6: 326 us, 364 with one, before later steps); one on the FP64 path, whose integer
// sums need the registers (131,072 cells: 234 us against 256 with two).
template <typename HT>
constexpr int w_vars() {
  return std::is_same<HT, double>::value ? 1 : 2;
}

template <int M, int NS, int NQ3, typename HT>
struct WPlan {
  static constexpr int kVW = w_vars<HT>(), kWWarps = 4 / kVW;
  static constexpr int kMC = wform_rows(M, NQ3);  // complement rows of a large slot
  static constexpr int kLPS = wform_lps(NS);      // large slots a stage
  static constexpr int kNG = kLPS * kMC, kNW = kLPS * NQ3;  // rows and W entries of a stage
  static constexpr int kGB = kNG * kTile * 4, kWB = kNW * kTile * 8;
  static constexpr int kSB = kSmallN * kSmallM * kTile * 4;  // rows of a directional stencil
  static constexpr int kSlotN = kTile * 2;  // halo offsets (uint16) of one slot
  static constexpr int kNL = NS / kLPS;
  static constexpr int kStages = kSmallK + kNL;  // the directional stencils first
  static constexpr int kStatBytes = kWStat * kTile * 4;
  // ring buffer of a large stage: [FP32 rows][W][halo offsets][cell words];
  // of a directional stage: [FP32 rows][halo offsets]
  static constexpr int kWOff = kGB, kNOff = kWOff + kWB;
  static constexpr int kXOff = kNOff + kLPS * kSlotN;
  static constexpr int kBufL = kXOff + kStatBytes, kBufS = kSB + kSmallN * kSlotN;
  static constexpr int kBuf = (kBufL > kBufS ? kBufL : kBufS);
  static constexpr int kE32 = NS * kMC + kSmallK * kSmallN * kSmallM;  // floats per lane
  static constexpr int kEW = NS * NQ3;                                 // W entries per lane
  static constexpr int kSL = NS + kSmallSlots;
  static constexpr int kTileBytes = kWTile * 4;
  static constexpr int kHaloRow = kHaloMax + kTile;     // halo states, then the tile's own
  static constexpr int kHalo = 2 * 4 * kHaloRow * 8;    // double-buffered, per variable
  static constexpr int kListN = (kVW + 1) * kTile;      // deferred cells of a warp
  // per warp: the differences of one cell, or the tile's directional indicators
  static constexpr int kScratch = kSL * 8 > kVW * kSmallK * 2 * kTile * 4
                                      ? kSL * 8
                                      : kVW * kSmallK * 2 * kTile * 4;
  // what own_scale needs of the tile's cells beyond a warp's own variables, two
  // buffers a warp: the other one of rho and E (pairs), or both and wstat's last word
  static constexpr int kOwn2 = (3 - kVW) * kTile * 8 + (kVW == 1 ? kTile * 4 : 0);
  static constexpr int kFixed = kHalo + 2 * kTileBytes + kWWarps * 2 * kOwn2 +
                                kWWarps * (kListN * 8 + kScratch) + 16 * 8 + 16;
  // four blocks per SM (96 threads of up to 168 registers, or 160 of 96); the
  // ring takes what is left of their quarter of the 227 KB of shared memory
  static constexpr int kRoom = (227 * 1024 / 4 - 1024 - kFixed) / kBuf;
  static constexpr int kRingW = kRoom < 2 ? 2 : (kRoom > 5 ? 5 : kRoom);
  static constexpr size_t kSmem = (size_t)kRingW * kBuf + kFixed;
  static_assert(NS % kLPS == 0, "whole stages");
  static_assert(kBuf % 16 == 0 && kWOff % 16 == 0 && kNOff % 16 == 0 && kXOff % 16 == 0 &&
                    kSB % 16 == 0 && kTileBytes % 16 == 0,
                "bulk-copy alignment");
};

// Upper bound of |beta32 - beta| relative to beta32 + eps, for beta32 the FP32
// sum of squares of m coefficients whose absolute errors sum to at most E:
// |sum a32^2 - sum a^2| <= sum e_l (2 |a32_l| + e_l) <= 2 E sqrt(beta32) + E^2,
// and the FP32 sum of squares adds (m + 2) u beta32 (u = 2^-24).  Returns a
// value >= 1 when the bound is not informative.
__device__ __forceinline__ float beta_rel_bound(float beta32, float E, int m, float eps) {
  const float u = 5.9604645e-8f;
  const float eb = (float)(m + 2) * u * beta32 + E * (2.0001f * sqrt_approx(beta32) + E);
  const float t = beta32 + eps;
  if (!(eb < 0.5f * t)) return 1.f;
  return 1.0002f * eb * rcp_approx(t - eb);
}
// The coefficients of n differences known to 2u relative plus one unit q each:
// coefficient l errs by at most (n + 7) u S_l + q sum_s |G_ls| with
// S_l = sum_s |G_ls| |d_s|, and sum_l S_l = sum_s colsum_s |d_s| <=
// |colsum|_2 |d|_2 (norm: |colsum|_2, rounded up; dd: sum of the squared FP32
// differences).
__device__ __forceinline__ float dot_bound(float norm, float dd, float q, int n) {
  const float u = 5.9604645e-8f;
  const float len = sqrt_approx(dd) * 1.0002f;
  return norm * ((float)(n + 7) * u * len + 7.f * q) * 1.0001f;  // sqrt(n) <= 7
}

// 2^e as FP32 (zero below the normal range, infinity above it)
__device__ __forceinline__ float exp2i(int e) {
  return e < -126 ? 0.f : (e > 127 ? __int_as_float(0x7f800000) : __int_as_float((e + 127) << 23));
}
// 2^e as FP64, |e| <= 1000
__device__ __forceinline__ double exp2d(int e) { return __hiloint2double((e + 1023) << 20, 0); }
// m 2^sh rounded to the nearest integer, m >= 0
__device__ __forceinline__ int64_t shift_round(int64_t m, int sh) {
  if (sh >= 0) return (int64_t)((uint64_t)m << sh);
  if (sh < -62) return 0;
  return (m + ((int64_t)1 << (-sh - 1))) >> -sh;
}
// x 2^k as an integer, rounded (|x| 2^k < 2^62)
__device__ __forceinline__ int64_t to_fix(float x, int k) {
  const int b = __float_as_int(x);
  const int ef = (b >> 23) & 0xff;
  const int64_t m = (b & 0x7fffff) | (ef ? 0x800000 : 0);
  const int64_t r = shift_round(m, (ef ? ef : 1) - 150 + k);
  return b < 0 ? -r : r;
}
__device__ __forceinline__ int64_t to_fix(double x, int k) {
  const int hi = __double2hiint(x);
  const int ef = (hi >> 20) & 0x7ff;
  const int64_t m = ((int64_t)((hi & 0xfffff) | (ef ? 0x100000 : 0)) << 32) |
                    (uint32_t)__double2loint(x);
  const int64_t r = shift_round(m, (ef ? ef : 1) - 1075 + k);
  return hi < 0 ? -r : r;
}
__device__ __forceinline__ int64_t to_fix(float2 x, int k) { return to_fix(x.x, k) + to_fix(x.y, k); }
// x 2^k as an integer modulo 2^64, rounded: differences below 2^63 come out of it
__device__ __forceinline__ int64_t to_fix_mod(double x, int k) {
  const int ef = max((__double2hiint(x) >> 20) & 0x7ff, 1);
  return ef - 1075 + k > 63 ? 0 : to_fix(x, k);
}
// magnitude bits of a state (ordered like |x|) and their unbiased exponent;
// kFixExpBad marks infinities and NaN
constexpr int kFixExpBad = 1 << 20;
__device__ __forceinline__ unsigned mag_bits(float2 x) {
  return (unsigned)__float_as_int(x.x) & 0x7fffffffu;
}
__device__ __forceinline__ unsigned mag_bits(double x) {
  return (unsigned)__double2hiint(x) & 0x7fffffffu;
}
template <typename HT>
__device__ __forceinline__ int mag_exp(unsigned m) {
  if constexpr (std::is_same<HT, double>::value) {
    const int f = (int)(m >> 20);
    return f == 0x7ff ? kFixExpBad : f - 1023;
  } else {
    const int f = (int)(m >> 23);
    return f == 0xff ? kFixExpBad : (f ? f : 1) - 127;
  }
}
// limbs x = h 2^30 + l with l in [0, 2^30)
constexpr int kFixB = 30;
// entry e of a stage's W (pairs of entries as 16 bytes a lane, a last odd one
// as 8) and of its FP32 rows (fours as 16 bytes, the rest one by one)
template <int N>
__device__ __forceinline__ int2 w_entry(const unsigned char* wb, int lane, int e) {
  if (e < N / 2 * 2) {
    const int4 q = reinterpret_cast<const int4*>(wb)[(e / 2) * kTile + lane];
    return e & 1 ? make_int2(q.z, q.w) : make_int2(q.x, q.y);
  }
  return reinterpret_cast<const int2*>(wb)[e * kTile + lane];
}
template <int N>
__device__ __forceinline__ float g_entry(const unsigned char* gb, int lane, int e) {
  if (e < N / 4 * 4) {
    const float4 q = reinterpret_cast<const float4*>(gb)[(e / 4) * kTile + lane];
    return (e & 3) == 0 ? q.x : ((e & 3) == 1 ? q.y : ((e & 3) == 2 ? q.z : q.w));
  }
  return reinterpret_cast<const float*>(gb)[e * kTile + lane];
}
__device__ __forceinline__ void mad_wide(int64_t& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// (hh, mid) += (w.x 2^30 + w.y) (dh 2^30 + dl), without the low product
__device__ __forceinline__ void fix_mac(int64_t& hh, int64_t& mid, int2 w, int dh, int dl) {
  mad_wide(hh, w.x, dh);
  mad_wide(mid, w.x, dl);
  mad_wide(mid, w.y, dh);
}
__device__ __forceinline__ int64_t fix_sum(int64_t hh, int64_t mid) {
  return hh + ((mid + ((int64_t)1 << (kFixB - 1))) >> kFixB);
}

// The sums W d of the two paths: difference parts D, accumulator A.
template <typename HT>
struct WDot;
// FP64 path (kN): integers throughout, as fix_mac.
template <>
struct WDot<double> {
  static constexpr int kBits = 57;      // |Y| < 2^57
  // bound of the sum's error: kErr units 2^exp, plus kErrD 2^-kc |d|_2
  static constexpr float kErr = 256.f, kErrD = 0.f;
  // own_scale's weight of s (an exponent): the values are rounded to 2^-53 of it, the sum to
  // |W|_1 < 2^(60 - kc) units
  __device__ __forceinline__ static int own_weight(int kc) { return kc - 58; }
  // an integer of |x| 2^sc < 2^57
  __device__ __forceinline__ static int64_t fix(double x, int sc, double) { return to_fix(x, sc); }
  struct D {
    int h, l;
  };
  struct A {
    int64_t hh = 0, mid = 0;
  };
  struct W {
    int2 m;
  };
  __device__ __forceinline__ static W entry(int2 m) { return {m}; }
  __device__ __forceinline__ static float c(int sc) { return exp2i(kFixB - sc); }
  // the parts and the FP32 value (c = 2^(30 - sc)) of a difference d 2^-sh
  __device__ __forceinline__ static float split(int64_t d, int sh, float c, D& o) {
    o.h = (int)(d >> (kFixB + sh));
    o.l = (int)(d >> sh) & ((1 << kFixB) - 1);
    return fmaf((float)o.h, c, (float)o.l * (c * (1.f / 1073741824.f)));
  }
  __device__ __forceinline__ static void mac(A& a, W w, D d) {
    fix_mac(a.hh, a.mid, w.m, d.h, d.l);
  }
  __device__ __forceinline__ static int64_t sum(const A& a) { return fix_sum(a.hh, a.mid); }
  __device__ __forceinline__ static int exp(int kc, int sc) { return 2 * kFixB - kc - sc; }
};
// Pairs: w = wh + wl with wh a 32-bit integer (sum_s |w_ps| < 2^31) and wl an
// FP32 fraction, d = (dh + dl) 2^B likewise (|dh| <= 2^30): sum wh dh is exact
// in 64 bits and wl dh + wh dl, 2^-31 of it, is an FP32 sum (two FP32
// multiply-adds in the place of two wide ones; a wide multiply-add holds its
// pipe for 5 clocks).  The states' rounding is half a unit each, so the sum errs
// by at most |W|_1 units, and by about a third of |W|_2 units as a rule; the FP32
// part adds about as much.
template <int kB>
struct WPairDot {
  static constexpr int kBits = kB + 29;
  // the FP32 sum's 2 n roundings, each 2^-25 of |x| <= sum (|wl| |dh| + |wh| |dl|) <=
  // (sqrt(n) |dh|_2 + 2^31) / 2
  static constexpr float kErr = 8192.f, kErrD = 2e-5f;
  // (the pairs that the states become in every other kernel of this path are
  // rounded to 2^-49 of them before the difference, so |W|_1 is on both sides)
  __device__ __forceinline__ static int own_weight(int) { return 0; }
  // an integer of |x| 2^sc < 2^51, from the low bits of 1.5 2^52 + x 2^sc (c = 2^sc)
  __device__ __forceinline__ static int64_t fix(double x, int, double c) {
    return __double_as_longlong(fma(x, c, 6755399441055744.0)) - 0x4338000000000000LL;
  }
  struct D {
    int h;
    float hf, lf;
  };
  struct A {
    int64_t hh = 0;
    float x = 0.f;
  };
  struct W {
    int h;
    float hf, lf;
  };
  __device__ __forceinline__ static W entry(int2 m) {
    return {m.x, (float)m.x, __int_as_float(m.y)};
  }
  __device__ __forceinline__ static float c(int sc) { return exp2i(kB - sc); }
  __device__ __forceinline__ static float split(int64_t d, int sh, float c, D& o) {
    const int z = (int)(d >> sh);
    o.h = (int)(d >> (kB + sh)) + ((z >> (kB - 1)) & 1);
    o.hf = (float)o.h;
    o.lf = (float)((z << (32 - kB)) >> (32 - kB)) * (1.f / (1 << kB));
    return (o.hf + o.lf) * c;
  }
  __device__ __forceinline__ static void mac(A& a, W w, D d) {
    mad_wide(a.hh, w.h, d.h);
    a.x = fmaf(w.hf, d.lf, a.x);
    a.x = fmaf(w.lf, d.hf, a.x);
  }
  // (sum wh dh + x) 2^exp
  __device__ __forceinline__ static DF value(const A& a, float s2, float s1, float s0) {
    const float h = (float)(int)(a.hh >> 42) * s2;
    const float m = (float)(int)((a.hh >> 21) & 0x1fffff) * s1;
    const float l = ((float)(int)(a.hh & 0x1fffff) + a.x) * s0;
    const DF r = fast_two_sum(h, m);
    return two_sum(r.h, r.l + l);
  }
  __device__ __forceinline__ static double value_d(const A& a) {
    return (double)a.hh + (double)a.x;
  }
  __device__ __forceinline__ static int exp(int kc, int sc) { return kB - kc - sc; }
};
// (the low bits of an FP64 sum give 51-bit differences)
template <>
struct WDot<float2> : WPairDot<22> {};
// Whether a cell keeps its own precision in units of 2^-sc: w s or max|d| is at
// least 2^(kBits - 2) units, for the differences d of its large stencil (es, ed:
// exponents of s and max|d|, w: own_weight).  That bounds the units' rounding by
// that of the sums in the path's own arithmetic: 2^-49 of s or |d| for pairs, 2^-53
// of s and 2^-55 of |d| in FP64.  s is |U_0|, and for a momentum at least 2^-6
// sqrt(rho E) (sqrt(rho E) >= |m| / 2^(1/2)): the flux rounds to 2^-49 or 2^-53 of
// sqrt(rho E) however small the momentum is, so a decaying tail of it (15 % of the
// shear layer's cells by |m| alone) has nothing to keep.
template <typename Dot>
__device__ __forceinline__ bool own_scale(int es, int ed, int kc, int sc) {
  return max(es + Dot::own_weight(kc), ed) >= Dot::kBits - 2 - sc;
}
// pair difference U_s - U_0 of a neighbour (FP32 hi/lo splits of the states)
__device__ __forceinline__ DF pair_dif(float2 q, float2 u0s) {
  DF t = two_sum(q.x, -u0s.x);
  t.l += q.y - u0s.y;
  return two_sum(t.h, t.l);
}

// Arithmetic of the deferred evaluations: pairs (float2 states) or FP64.
template <typename HT>
struct WArith;
template <>
struct WArith<float2> {
  using Acc = DF;
  __device__ __forceinline__ static DF zero() { return DF{0.f, 0.f}; }
  __device__ __forceinline__ static DF dif(float2 q, float2 u0) { return pair_dif(q, u0); }
  __device__ __forceinline__ static void mac(DF& acc, float2 m, DF d) { df_mac(acc, m, d); }
  __device__ __forceinline__ static DF norm(DF x) { return df_norm(x); }
  __device__ __forceinline__ static float2 entry(DF x) { return make_float2(x.h, x.l); }
  __device__ __forceinline__ static DF shfl(DF x, int l) {
    return DF{__shfl_sync(0xffffffffu, x.h, l), __shfl_sync(0xffffffffu, x.l, l)};
  }
  __device__ __forceinline__ static DF add(DF a, DF b) {
    DF q = two_sum(a.h, b.h);
    q.l += a.l + b.l;
    return two_sum(q.h, q.l);
  }
  __device__ __forceinline__ static DF div(DF a, int n) {  // exact remainder correction
    const float fn = (float)n, qh = a.h / fn, r = fmaf(-qh, fn, a.h);
    return two_sum(qh, (r + a.l) / fn);
  }
  __device__ __forceinline__ static float2 value(float2 u0, DF x) {
    const DF r = DF{u0.x, u0.y} + x;
    return make_float2(r.h, r.l);
  }
};
template <>
struct WArith<double> {
  using Acc = double;
  __device__ __forceinline__ static double zero() { return 0.0; }
  __device__ __forceinline__ static double dif(double q, double u0) { return q - u0; }
  __device__ __forceinline__ static void mac(double& acc, double m, double d) {
    acc = fma(m, d, acc);
  }
  __device__ __forceinline__ static double norm(double x) { return x; }
  __device__ __forceinline__ static double entry(double x) { return x; }
  __device__ __forceinline__ static double shfl(double x, int l) {
    return __shfl_sync(0xffffffffu, x, l);
  }
  __device__ __forceinline__ static double add(double a, double b) { return a + b; }
  __device__ __forceinline__ static double div(double a, int n) { return a / (double)n; }
  __device__ __forceinline__ static double value(double u0, double x) { return u0 + x; }
};

// Cutoff decision of one cell in FP64, by the whole warp (the cells it is
// needed for are few and far between, so one lane per cell would leave the
// warp waiting for a chain of loads).  A: the cell's matrices at its lane,
// nb: its stencil cells, st: the states of the variable, dsc: the warp's
// scratch.  The differences are gathered one slot per lane, then lane q forms
// coefficient q (of the large stencil's m and the directional 15), and beta
// and the decision follow in every lane.
template <int M, int NS, typename HT>
__device__ __noinline__ int w_select(const HT* A, const int32_t* nb, const HT* st, HT u0,
                                     int present, double ct, double eps, HT* dsc) {
  using Ar = WArith<HT>;
  using Acc = typename Ar::Acc;
  constexpr int SL = NS + kSmallSlots, NC = M + kSmallK * kSmallM;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < (SL + kTile - 1) / kTile; ++i) {
    const int s = lane + i * kTile;
    if (s < SL) dsc[s] = Ar::entry(Ar::dif(st[__ldg(nb + s * kTile)], u0));
  }
  __syncwarp();
  auto coef = [&](int q) {
    Acc acc = Ar::zero();
    const bool lg = q < M;
    const int k = lg ? 0 : (q - M) / kSmallM, l = lg ? q : (q - M) % kSmallM;
    const int n = q >= NC ? 0 : (lg ? NS : kSmallN);
    const int rows = lg ? M : kSmallM;
    const HT* Aq = A + (int64_t)(lg ? l : M * NS + k * kSmallN * kSmallM + l) * kTile;
    const HT* dq = dsc + (lg ? 0 : NS + k * kSmallN);
#pragma unroll 6
    for (int s = 0; s < n; ++s) {
      const HT d = dq[s];
      if constexpr (std::is_same<HT, double>::value)
        Ar::mac(acc, __ldg(Aq + (int64_t)s * rows * kTile), d);
      else
        Ar::mac(acc, __ldg(Aq + (int64_t)s * rows * kTile), DF{d.x, d.y});
    }
    return Ar::norm(acc);
  };
  const Acc c0 = coef(lane);
  Acc c1 = Ar::zero();
  if constexpr (NC > kTile) c1 = coef(lane + kTile);
  __syncwarp();
  auto sum_sq = [&](int q0, int n) {
    Acc b = Ar::zero();
#pragma unroll 1
    for (int q = q0; q < q0 + n; ++q) {
      const Acc x = Ar::shfl(q < kTile ? c0 : c1, q & 31);
      Ar::mac(b, Ar::entry(x), x);
    }
    return to_d(Ar::norm(b));
  };
  double beta[kSmallK + 1];
  beta[kSmallK] = sum_sq(0, M);
#pragma unroll
  for (int k = 0; k < kSmallK; ++k)
    beta[k] = (present >> k) & 1 ? sum_sq(M + k * kSmallM, kSmallM) : 0.0;
  return select_fp64(beta, present, ct, eps);
}

// Gauss-point values of the equally weighted kept directional polynomials
// (step ii of the selection), one cell and variable per lane; psi: the
// [point][kMaxM] table of Psi'.  A stencil's cells and states are requested
// together, its matrix entries four slots at a time.
template <int M, int NS, int NQ3, int NV, typename HT>
__device__ __noinline__ void w_small(const HT* A, const int32_t* nb, const HT* st, HT u0, int sel,
                                     const HT* psi, HT* out) {
  using Ar = WArith<HT>;
  using Acc = typename Ar::Acc;
  Acc sum[kSmallM];
#pragma unroll
  for (int l = 0; l < kSmallM; ++l) sum[l] = Ar::zero();
#pragma unroll 1
  for (int k = 0; k < kSmallK; ++k) {
    if (!((sel >> k) & 1)) continue;
    const int32_t* nk = nb + (NS + k * kSmallN) * kTile;
    const HT* Ak = A + (int64_t)(M * NS + k * kSmallN * kSmallM) * kTile;
    int id[kSmallN];
    HT q[kSmallN];
#pragma unroll
    for (int s = 0; s < kSmallN; ++s) id[s] = __ldg(nk + s * kTile);
#pragma unroll
    for (int s = 0; s < kSmallN; ++s) q[s] = st[id[s]];
    Acc as[kSmallM];
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) as[l] = Ar::zero();
#pragma unroll
    for (int s = 0; s < kSmallN; ++s) {
      const Acc d = Ar::dif(q[s], u0);
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) Ar::mac(as[l], __ldg(Ak + (s * kSmallM + l) * kTile), d);
    }
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) sum[l] = Ar::add(sum[l], Ar::norm(as[l]));
  }
  const int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
  Acc cf[kSmallM];
#pragma unroll
  for (int l = 0; l < kSmallM; ++l) cf[l] = nd ? Ar::div(sum[l], nd) : Ar::zero();
#pragma unroll 1
  for (int p = 0; p < NQ3; ++p) {
    Acc sp = Ar::zero();
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) Ar::mac(sp, __ldg(psi + p * kMaxM + l), cf[l]);
    out[p * NV] = Ar::value(u0, Ar::norm(sp));
  }
}

// Large-stencil values of a cell whose tile holds an infinity, a NaN or a
// magnitude outside the fixed-point range, or too large a difference for the
// cell's own scale (own_scale): U_0 + W d in floating point.
template <int NS, int NQ3, int NV>
__device__ __noinline__ void w_direct(const int2* W, int lane, int kc, const int32_t* nb,
                                      const float2* st, float2 u0s, float2* out) {
#pragma unroll 1
  for (int p = 0; p < NQ3; ++p) {
    DF acc = {0.f, 0.f};
#pragma unroll 1
    for (int s = 0; s < NS; ++s) {
      const int2 w = W[wform_w_index(NS, NQ3, s, p, lane)];
      const DF q = d_to_df(ldexp((double)w.x + (double)__int_as_float(w.y), -kc));
      df_mac(acc, make_float2(q.h, q.l), pair_dif(st[nb[s * kTile]], u0s));
    }
    const DF r = DF{u0s.x, u0s.y} + df_norm(acc);
    out[p * NV] = make_float2(r.h, r.l);
  }
}
template <int NS, int NQ3, int NV>
__device__ __noinline__ void w_direct(const int2* W, int lane, int kc, const int32_t* nb,
                                      const double* st, double u0, double* out) {
#pragma unroll 1
  for (int p = 0; p < NQ3; ++p) {
    double acc = 0.0;
#pragma unroll 1
    for (int s = 0; s < NS; ++s) {
      const int2 w = W[wform_w_index(NS, NQ3, s, p, lane)];
      const double x = ldexp((double)w.x * 1073741824.0 + (double)w.y, -kc);
      acc = fma(x, st[nb[s * kTile]] - u0, acc);
    }
    out[p * NV] = u0 + acc;
  }
}

// position in a ring of kN buffers: the buffer, and the parity of its phase
template <int kN>
struct RingPos {
  int b = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next() {
    if (++b == kN) b = 0, ph ^= 1;
  }
};

// The cutoff screen's decisions from the FP32 indicators t known within the
// factor f of chi: the selection, | 256 where C_T lies within that factor of
// some chi.  Out of line: few cells need it.
__device__ __noinline__ int w_screen(float t0, float t1, float t2, float tK, int present, float ct,
                                     float f) {
  const float t[kSmallK + 1] = {t0, t1, t2, tK};
  bool near = false;
  int sel = 8;
  if (!chi_keep32_bound(t, kSmallK, present | 8, ct, f, &near)) {
    sel = 0;
#pragma unroll
    for (int k = 0; k < kSmallK; ++k)
      if (((present >> k) & 1) && chi_keep32_bound(t, k, present & 7, ct, f, &near)) sel |= 1 << k;
  }
  return sel | (near ? 256 : 0);
}

// deferred cells: the cell in the low word; the high word's flags, and the
// selection where it is decided
// (bits 0-3 of it: a selection override passes a caller's bytes, whose other bits
// mean nothing and would reach the variable)
constexpr int kDefNear = 1, kDefDirect = 2, kDefSel = 8;  // selection from bit 3
constexpr int kDefVar = 256;                              // variable from bit 8

struct WArgs {
  const void* psi;    // Psi' as pairs or FP64
  const float* g32;   // FP32 rows of the complement and the directional stencils
  const int2* w;      // W in fixed point
  const uint16_t* pos;  // [tile][slot][32] byte offsets of the stencil cells in a halo row
  const int32_t* tile;  // [tile][kWTile] halo cells, lanes that hold a cell, halo ids
  const int32_t* st;  // [tile][kWStat][32]: column-sum norms of the four stencils (FP32), then
                      // the exponent of W's unit (low half) and the stencil mask (bit 16)
  WTable t;
};

// Works off n <= 32 deferred cells: the undecided ones one by one, then one
// per lane.
template <int M, int NS, int NQ, typename HT>
__device__ __noinline__ void w_deferred(const ReconArgs& a, const WArgs& wa, const int2* list,
                                        int n, HT* dsc) {
  constexpr int NQ3 = 3 * NQ, NV = 4, E = M * NS + kSmallEntries, SL = NS + kSmallSlots;
  const int lane = threadIdx.x & 31;
  const int2 mine = lane < n ? list[lane] : make_int2(0, 0);
  auto states = [&](int v) {
    if constexpr (std::is_same<HT, double>::value)
      return a.U + (int64_t)v * a.n_pad;
    else
      return a.Us + (int64_t)v * a.n_pad;
  };
  auto matrices = [&](int64_t c) {
    return reinterpret_cast<const HT*>(a.ahat) + c / kTile * (int64_t)E * kTile + c % kTile;
  };
  auto cells = [&](int64_t c) { return a.nbr + c / kTile * (int64_t)SL * kTile + c % kTile; };
  int sel = (mine.y >> 3) & 15;
  unsigned near = __ballot_sync(0xffffffffu, lane < n && (mine.y & kDefNear));
  for (; near; near &= near - 1) {
    const int src = __ffs(near) - 1;
    const int64_t c = __shfl_sync(0xffffffffu, mine.x, src);
    const HT* st = states(__shfl_sync(0xffffffffu, mine.y / kDefVar, src));
    const int r = w_select<M, NS, HT>(matrices(c), cells(c), st, st[c], a.smask[c], a.ct, a.eps, dsc);
    if (lane == src) sel = r;
  }
  if (lane >= n) return;
  const int64_t c = mine.x;
  const int v = mine.y / kDefVar;
  const HT* st = states(v);
  if ((mine.y & kDefNear) && a.sel_out) a.sel_out[(int64_t)v * a.n_pad + c] = (uint8_t)sel;
  HT* out = reinterpret_cast<HT*>(a.Uq) + c * (NQ3 * NV) + v;
  if (!(sel & 8)) {
    w_small<M, NS, NQ3, NV, HT>(matrices(c), cells(c), st, st[c], sel,
                                reinterpret_cast<const HT*>(wa.psi), out);
  } else if (mine.y & kDefDirect) {
    const int64_t tile = c / kTile;
    const int cl = (int)(c % kTile);
    const int kc = (int16_t)(wa.st[(tile * kWStat + kWStat - 1) * kTile + cl] & 0xffff);
    w_direct<NS, NQ3, NV>(wa.w + tile * (int64_t)(NS * NQ3) * kTile, cl, kc, cells(c), st, st[c],
                          out);
  }
}

// HT = float2: the FP64 path in pairs (Gauss values as (hi, lo) FP32 pairs);
// HT = double: the native FP64 path.  Persistent blocks of consumer warps
// (kVW variables each) and a producer lane that streams the tiles' matrices in
// ring stages, and their halo ids, with bulk copies; each consumer warp
// gathers its variables' halo states of the next tile with cp.async.  Every
// hand-over is an mbarrier with bounded waits and no warp reads what another
// consumer wrote, so the consumer warps run without block barriers.
template <int M, int NS, int NQ, typename HT>
__global__ void __launch_bounds__(kTile * (4 / w_vars<HT>() + 1), 4)
    recon_tma_w_kernel(const ReconArgs a, const WArgs wa, int* err) {
  constexpr bool kN = std::is_same<HT, double>::value;
  constexpr int NQ3 = 3 * NQ, NV = 4;
  using P = WPlan<M, NS, NQ3, HT>;
  using Dot = WDot<HT>;
  constexpr int kVW = P::kVW, kWWarps = P::kWWarps;
  constexpr int kR = P::kRingW, MC = P::kMC, R = M < NQ3 ? M : NQ3;
  constexpr int kPer = NQ3 * NV;  // Gauss-point values per cell
  extern __shared__ __align__(128) unsigned char smem[];
  double* halo = reinterpret_cast<double*>(smem + (size_t)kR * P::kBuf);  // [2][NV][kHaloRow]
  int32_t* tblk = reinterpret_cast<int32_t*>(halo + 2 * NV * P::kHaloRow);  // [2][kWTile]
  unsigned char* owns = reinterpret_cast<unsigned char*>(tblk + 2 * kWTile);  // [kWWarps][2][kOwn2]
  int2* list = reinterpret_cast<int2*>(owns + kWWarps * 2 * P::kOwn2);  // [kWWarps][kListN]
  HT* scratch = reinterpret_cast<HT*>(list + kWWarps * P::kListN);  // [kWWarps][kScratch]
  uint64_t* full = reinterpret_cast<uint64_t*>(scratch + kWWarps * (P::kScratch / 8));
  uint64_t* empty = full + kR;
  uint64_t* tfull = empty + kR;
  uint64_t* tempty = tfull + 2;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(full + 16);
  static_assert(2 * kR + 4 <= 16, "mbarriers");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_tiles = (a.n_cell + kTile - 1) / kTile;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int i = 0; i < kR; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kWWarps);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], kWWarps);
    }
    mbar_fence_init();
  }
  __syncthreads();
  if (warp == kWWarps) {
    // ---- producer lane: the halo ids two tiles ahead, the ring stages of
    // every tile
    if (lane == 0) {
      RingPos<kR> rp;
      bool lap = false;  // every buffer has been filled once
      int it = 0;
      // the block must not exit while a copy it issued is in flight: the last
      // kR stages (buffers before rp.b are one phase ahead) and id blocks
      auto drain = [&](int n_blk) {
        for (int b = 0; b < kR; ++b)
          if (b < rp.b || lap) mbar_wait(&full[b], b < rp.b ? rp.ph : rp.ph ^ 1);
        for (int i = n_blk > 2 ? n_blk - 2 : 0; i < n_blk; ++i)
          mbar_wait(&tfull[i & 1], (uint32_t)(i >> 1) & 1);
      };
      auto gave_up = [&](int w, int n_blk) {
        if (w == 0) {
          atomicOr(err, 2);
          *abort_flag = 1;
        }
        drain(n_blk);
      };
      auto block = [&](int64_t tile, int i) {
        if (tile >= n_tiles) return;
        mbar_expect_tx(&tfull[i & 1], P::kTileBytes);
        bulk_g2s(tblk + (i & 1) * kWTile, wa.tile + tile * kWTile, P::kTileBytes, &tfull[i & 1]);
      };
      int n_blk = 0;  // halo-id blocks issued
      for (; n_blk < 2 && blockIdx.x + (int64_t)n_blk * gridDim.x < n_tiles; ++n_blk)
        block(blockIdx.x + (int64_t)n_blk * gridDim.x, n_blk);
      for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
        const unsigned char* sg =
            reinterpret_cast<const unsigned char*>(wa.g32) + tile * (int64_t)P::kE32 * kTile * 4;
        const unsigned char* sw =
            reinterpret_cast<const unsigned char*>(wa.w) + tile * (int64_t)P::kEW * kTile * 8;
        const unsigned char* sn =
            reinterpret_cast<const unsigned char*>(wa.pos) + tile * (int64_t)P::kSL * P::kSlotN;
        for (int j = 0; j < P::kStages; ++j) {
          const int b = rp.b;
          if (lap) {
            const int w = mbar_wait_or_abort(&empty[b], rp.ph ^ 1, abort_flag);
            if (w != 1) return gave_up(w, n_blk);
          }
          unsigned char* dst = smem + b * P::kBuf;
          if (j < kSmallK) {
            mbar_expect_tx(&full[b], P::kSB + kSmallN * P::kSlotN);
            bulk_g2s(dst, sg + P::kNL * P::kGB + j * P::kSB, P::kSB, &full[b]);
            bulk_g2s(dst + P::kSB, sn + (NS + j * kSmallN) * P::kSlotN, kSmallN * P::kSlotN,
                     &full[b]);
          } else {
            const int i = j - kSmallK;
            const bool last = j == P::kStages - 1;
            mbar_expect_tx(&full[b], P::kGB + P::kWB + P::kLPS * P::kSlotN +
                                         (last ? P::kStatBytes : 0));
            if constexpr (MC > 0) bulk_g2s(dst, sg + i * P::kGB, P::kGB, &full[b]);
            bulk_g2s(dst + P::kWOff, sw + i * P::kWB, P::kWB, &full[b]);
            bulk_g2s(dst + P::kNOff, sn + i * P::kLPS * P::kSlotN, P::kLPS * P::kSlotN, &full[b]);
            if (last) bulk_g2s(dst + P::kXOff, wa.st + tile * kWStat * kTile, P::kStatBytes, &full[b]);
          }
          rp.next();
          lap |= rp.b == 0;
        }
        const int64_t nxt = tile + 2 * (int64_t)gridDim.x;
        if (nxt < n_tiles) {
          const int w =
              mbar_wait_or_abort(&tempty[it & 1], (uint32_t)(it >> 1) & 1, abort_flag);
          if (w != 1) return gave_up(w, n_blk);
          block(nxt, n_blk++);
        }
      }
      drain(n_blk);
    }
    return;
  }
  // ---- consumers (warp w: kVW variables from kVW w)
  pdl_wait();  // the states (the producer streams constant data before it)
  constexpr int kPerLane = kHaloMax / kTile;
  const int v0 = warp * kVW;
  int2* mylist = list + warp * P::kListN;
  HT* dsc = scratch + warp * (P::kScratch / 8);
  // beta and |d|^2 of the directional stencils, [kSmallK][kVW][2][32]: twelve
  // registers less in the large stencil's loop
  float* tsd = reinterpret_cast<float*>(dsc) + lane;
  unsigned char* own2 = owns + warp * 2 * P::kOwn2;
  int n_def = 0, it = 0;
  RingPos<kR> rp;
  // the wait of one consumer warp; false: some wait of the block gave up
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    const int w = mbar_wait_or_abort(bar, parity, abort_flag, a.wait_polls);
    if (w == 0) {
      atomicOr(err, 2);
      *abort_flag = 1;
    }
    return !__any_sync(0xffffffffu, w != 1);
  };
  // the halo and own states of this block's i-th tile, one commit group (an
  // empty one past the end); H and held: its halo cells, the lanes that hold
  // a cell (a partition's layout has gaps)
  auto gather = [&](int64_t tile, int i, int& H, unsigned& held) {
    bool ok = true;
    if (tile < n_tiles) {
      ok = wait(&tfull[i & 1], (uint32_t)(i >> 1) & 1);
      if (ok) {
        const int32_t* tb = tblk + (i & 1) * kWTile;
        const double* src = a.U + (int64_t)v0 * a.n_pad;
        double* dst = halo + ((i & 1) * NV + v0) * P::kHaloRow;
        H = tb[0];
        held = (unsigned)tb[1];
#pragma unroll
        for (int k = 0; k < kPerLane; ++k)
          if (lane + k * kTile < H) {
            const int id = tb[4 + lane + k * kTile];
#pragma unroll
            for (int w = 0; w < kVW; ++w)
              cp_async8(dst + w * P::kHaloRow + lane + k * kTile, src + w * a.n_pad + id);
          }
        const int64_t c = tile * kTile + lane;
#pragma unroll
        for (int w = 0; w < kVW; ++w)
          cp_async8(dst + w * P::kHaloRow + kHaloMax + lane,
                    src + w * a.n_pad + (c < a.n_cell ? c : 0));
        double* o2 = reinterpret_cast<double*>(own2 + (i & 1) * P::kOwn2) + lane;
        if constexpr (kN) {
          if (v0 == 1 || v0 == 2)
#pragma unroll
            for (int k = 0; k < 2; ++k)
              cp_async8(o2 + k * kTile, a.U + 3 * k * a.n_pad + (c < a.n_cell ? c : 0));
          cp_async4(reinterpret_cast<int32_t*>(own2 + (i & 1) * P::kOwn2 + 2 * kTile * 8) + lane,
                    wa.st + (tile * kWStat + kWStat - 1) * kTile + lane);
        } else {
          cp_async8(o2, a.U + (v0 == 0 ? 3 : 0) * a.n_pad + (c < a.n_cell ? c : 0));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[i & 1]);
      }
    }
    cp_async_commit();
    return ok;
  };
  int H, Hn = 0;
  unsigned held, heldn = 0u;
  if (!gather(blockIdx.x, 0, Hn, heldn)) {
    cp_async_wait<0>();
    return;
  }
  bool alive = true;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
    const int64_t c = tile * kTile + lane;  // may be a pad lane of the last tile
    H = Hn;
    held = heldn;
    __syncwarp();  // every lane is done with the other halo buffer
    if (!(alive = gather(tile + gridDim.x, it + 1, Hn, heldn))) break;
    cp_async_wait<1>();
    __syncwarp();
    double* hv = halo + ((it & 1) * NV + v0) * P::kHaloRow;
    const bool mine = (held >> lane) & 1;
    // ---- the halo states relative to the tile's first cell in fixed point,
    // in place (Dot::kBits of the largest difference).  The unit depends on
    // the set of the tile's cells and halo only, so a partition, which keeps
    // whole tiles, gets the same bits
    const unsigned char* st = reinterpret_cast<const unsigned char*>(hv);
    int64_t y0[kVW];
    int sc[kVW], sh[kVW];  // units: the cell's 2^-sc, the tile's 2^-(sc + sh)
    int float_w[kVW];      // 1: the tile's states have no unit, 2: too coarse a one for the cell
    {
      const int n_mine = (H - lane + kTile - 1) / kTile;  // this lane's halo cells
      unsigned mx[kVW];
      double ref[kVW], own[kVW];
#pragma unroll
      for (int w = 0; w < kVW; ++w) {
        const double u0 = hv[w * P::kHaloRow + kHaloMax + lane];
        ref[w] = __shfl_sync(0xffffffffu, u0, 0);
        own[w] = u0 - ref[w];
        mx[w] = mine ? mag_bits(own[w]) : 0u;
      }
#pragma unroll 2
      for (int i = 0; i < n_mine; ++i)
#pragma unroll
        for (int w = 0; w < kVW; ++w) {
          double* q = hv + w * P::kHaloRow + lane + i * kTile;
          const double d = *q - ref[w];
          *q = d;  // one FP64 operation per state (the FP64 pipe is the slow one)
          mx[w] = max(mx[w], mag_bits(d));
        }
      // a cell's scale (own_scale), first without its differences
      const unsigned char* o2 = own2 + (it & 1) * P::kOwn2;
      int kc = 0;
      if constexpr (kN)
        kc = (int)(int16_t)(reinterpret_cast<const int32_t*>(o2 + 2 * kTile * 8)[lane] & 0xffff);
      int es[kVW];
      bool coarse = false;
#pragma unroll
      for (int w = 0; w < kVW; ++w) {
        mx[w] = __reduce_max_sync(0xffffffffu, mx[w]);
        // |U - U_ref| < 2^(e + 1); a difference below 2^-900 counts as none
        const int e = max(mx[w] ? mag_exp<double>(mx[w]) : 0, -900);
        float_w[w] = e > 100;
        sc[w] = float_w[w] ? 0 : Dot::kBits - 1 - e;
        sh[w] = 0;
        es[w] = mag_exp<double>(mag_bits(hv[w * P::kHaloRow + kHaloMax + lane]));
        if (v0 + w == 1 || v0 + w == 2) {  // rho and E, in either order
          const double* x = reinterpret_cast<const double*>(o2) + lane;
          const double y = kN ? x[kTile] : hv[(kVW - 1 - w) * P::kHaloRow + kHaloMax + lane];
          const int e2 = mag_exp<double>(mag_bits(*x)) + mag_exp<double>(mag_bits(y));
          es[w] = max(es[w], (e2 >> 1) - 6);
        }
        coarse |= mine && mx[w] && !float_w[w] && !own_scale<Dot>(es[w], -5000, kc, sc[w]);
      }
      bool wide = __any_sync(0xffffffffu, coarse);
      int ed[kVW];
      if (wide) {  // then with them
        unsigned ml[kVW] = {};
        const uint16_t* gp = wa.pos + tile * (int64_t)(P::kSL * kTile) + lane;
        __syncwarp();
        constexpr int kN1 = NS > 30 ? NS / 3 : NS / 2;  // some slots usually show enough
#pragma unroll 1
        for (int i0 = 0; wide && i0 < NS; i0 += kN1) {
#pragma unroll
          for (int i = 0; i < kN1; ++i) {
            const int off = __ldg(gp + (i0 + i) * kTile);
#pragma unroll
            for (int w = 0; w < kVW; ++w)
              ml[w] = max(ml[w], mag_bits(*reinterpret_cast<const double*>(
                                              st + w * (P::kHaloRow * 8) + off) -
                                          own[w]));
          }
          coarse = false;
#pragma unroll
          for (int w = 0; w < kVW; ++w) {
            ed[w] = mag_exp<double>(ml[w]);
            coarse |= mine && mx[w] && !float_w[w] && !own_scale<Dot>(es[w], ed[w], kc, sc[w]);
          }
          wide = __any_sync(0xffffffffu, coarse);
        }
      }
      if (!wide) {
        double cf[kVW];
#pragma unroll
        for (int w = 0; w < kVW; ++w) {
          cf[w] = exp2d(sc[w]);
          y0[w] = mine && !float_w[w] ? Dot::fix(own[w], sc[w], cf[w]) : 0;
        }
#pragma unroll 2
        for (int i = 0; i < n_mine; ++i)
#pragma unroll
          for (int w = 0; w < kVW; ++w) {
            double* q = hv + w * P::kHaloRow + lane + i * kTile;
            *q = __longlong_as_double(float_w[w] ? 0 : Dot::fix(*q, sc[w], cf[w]));
          }
      } else {
        // 62 bits for the largest difference in the tile, from the states themselves
        // (U - U_ref is rounded to 2^-53 of it), and of these kBits for its own
        // largest for each cell: pairs reach cells 2^-12 of the tile's largest
        // difference, FP64 2^-5 or so (|W|_1).  (A second copy of the loops below
        // with lane units of any size cost the tiles that never enter it 8 to 16 %:
        // registers.)
        const int32_t* ids = wa.tile + tile * kWTile + 4 + lane;
        __syncwarp();
#pragma unroll 1
        for (int i = 0; i < n_mine; ++i) {
          const int id = __ldg(ids + i * kTile);
#pragma unroll
          for (int w = 0; w < kVW; ++w) {
            const double u = a.U[(int64_t)(v0 + w) * a.n_pad + id];
            hv[w * P::kHaloRow + lane + i * kTile] =
                __longlong_as_double(float_w[w] ? 0 : to_fix_mod(u, sc[w] + 61 - Dot::kBits));
          }
        }
#pragma unroll
        for (int w = 0; w < kVW; ++w) {
          y0[w] = 0;
          if (!mine || float_w[w]) continue;
          const int sT = sc[w] + 61 - Dot::kBits;  // |U - U_0| 2^sT < 2^62
          sh[w] = max(0, ed[w] + 1 + sT - Dot::kBits);
          sc[w] = sT - sh[w];
          // (with half a unit of the cell, so that the shift rounds)
          y0[w] = to_fix_mod(hv[w * P::kHaloRow + kHaloMax + lane], sT) -
                  (int64_t)((1ull << sh[w]) >> 1);
          if (!own_scale<Dot>(es[w], ed[w], kc, sc[w])) float_w[w] = 2;
        }
      }
      __syncwarp();
    }
    // the difference to the cell at a byte offset of the halo row, in units of
    // the tile; its FP32 values below err by 3u relative plus 2^7 of these (the
    // directional ones, which may exceed the large stencil's) or 2^6 of the
    // cell's.  The 64-bit conversion would take the FP64 pipe.
    auto dif = [&](int w, int off) {
      return *reinterpret_cast<const int64_t*>(st + w * (P::kHaloRow * 8) + off) - y0[w];
    };
    float cd[kVW];  // their FP32 scale
#pragma unroll
    for (int w = 0; w < kVW; ++w) cd[w] = exp2i(-sc[w] - sh[w]);
    // ---- directional stencils: FP32 smoothness indicators
#pragma unroll 1
    for (int k = 0; k < kSmallK; ++k, rp.next()) {
      if (!(alive = wait(&full[rp.b], rp.ph))) break;
      const unsigned char* buf = smem + rp.b * P::kBuf;
      const uint16_t* nl = reinterpret_cast<const uint16_t*>(buf + P::kSB) + lane;
      float s[kVW][kSmallM], dd[kVW];
#pragma unroll
      for (int w = 0; w < kVW; ++w) {
        dd[w] = 0.f;
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) s[w][l] = 0.f;
      }
      // four slots (five fours of rows) at a time
#pragma unroll 1
      for (int i = 0; i < kSmallN; i += 4) {
        float f[kVW][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int off = nl[(i + j) * kTile];
#pragma unroll
          for (int w = 0; w < kVW; ++w) {
            const int64_t x = dif(w, off);
            f[w][j] = fmaf((float)(int)((x + 0x80000000LL) >> 32), cd[w] * 4294967296.f,
                           (float)(int)x * cd[w]);
            dd[w] = fmaf(f[w][j], f[w][j], dd[w]);
          }
        }
#pragma unroll
        for (int e = 0; e < 4 * kSmallM; ++e) {
          const float m = g_entry<4 * kSmallM>(buf + i * kSmallM * kTile * 4, lane, e);
#pragma unroll
          for (int w = 0; w < kVW; ++w)
            s[w][e % kSmallM] = fmaf(m, f[w][e / kSmallM], s[w][e % kSmallM]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[rp.b]);
#pragma unroll
      for (int w = 0; w < kVW; ++w) {
        float q = 0.f;
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) q = fmaf(s[w][l], s[w][l], q);
        tsd[(k * kVW + w) * 2 * kTile] = q;
        tsd[(k * kVW + w) * 2 * kTile + kTile] = dd[w];
      }
    }
    if (!alive) break;
    // ---- large stencil: W d in fixed point, complement rows in FP32
#pragma unroll
    for (int w = 0; w < kVW; ++w) cd[w] = Dot::c(sc[w]);
    typename Dot::A acc[kVW][NQ3];
    float a32[kVW][MC > 0 ? MC : 1], dL[kVW], norm[kSmallK + 1];
    int stat = 0;
#pragma unroll
    for (int w = 0; w < kVW; ++w) {
      dL[w] = 0.f;
#pragma unroll
      for (int l = 0; l < MC; ++l) a32[w][l] = 0.f;
    }
#pragma unroll 1
    for (int j = 0; j < P::kNL; ++j, rp.next()) {
      if (!(alive = wait(&full[rp.b], rp.ph))) break;
      const unsigned char* buf = smem + rp.b * P::kBuf;
      const uint16_t* nl = reinterpret_cast<const uint16_t*>(buf + P::kNOff) + lane;
      typename Dot::D d[kVW][P::kLPS];
      float f[kVW][P::kLPS];
#pragma unroll
      for (int s = 0; s < P::kLPS; ++s) {
        const int off = nl[s * kTile];
#pragma unroll
        for (int w = 0; w < kVW; ++w) {
          f[w][s] = Dot::split(dif(w, off), sh[w], cd[w], d[w][s]);
          dL[w] = fmaf(f[w][s], f[w][s], dL[w]);
        }
      }
      if constexpr (MC > 0) {
#pragma unroll
        for (int e = 0; e < P::kNG; ++e) {
          const float m = g_entry<P::kNG>(buf, lane, e);
#pragma unroll
          for (int w = 0; w < kVW; ++w) a32[w][e % MC] = fmaf(m, f[w][e / MC], a32[w][e % MC]);
        }
      }
#pragma unroll
      for (int e = 0; e < P::kNW; ++e) {
        const typename Dot::W m = Dot::entry(w_entry<P::kNW>(buf + P::kWOff, lane, e));
#pragma unroll
        for (int w = 0; w < kVW; ++w) Dot::mac(acc[w][e % NQ3], m, d[w][e / NQ3]);
      }
      if (j == P::kNL - 1) {
        const int32_t* xs = reinterpret_cast<const int32_t*>(buf + P::kXOff) + lane;
#pragma unroll
        for (int k = 0; k <= kSmallK; ++k) norm[k] = __int_as_float(xs[k * kTile]);
        stat = xs[kSmallK * kTile + kTile];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[rp.b]);
    }
    if (!alive) break;
    // ---- selection
    const int present = (stat >> 16) & 7, kc = (int)(int16_t)(stat & 0xffff);
    int eT[kVW], sel[kVW];  // W d = (the sum) 2^eT
    bool near[kVW];
    HT val[kVW][NQ3];
#pragma unroll
    for (int w = 0; w < kVW; ++w) {
      const int v = v0 + w;
      // units of the differences' FP32 errors (the cell's own state is off by half a unit
      // of the cell)
      const float cu = 80.f * exp2i(-sc[w]), cs = 160.f * exp2i(-sc[w] - sh[w]) + exp2i(-sc[w]);
      eT[w] = Dot::exp(kc, sc[w]);
      const float s0 = exp2i(eT[w]);
      // Gauss-point values, and W d in FP32 (y)
      float y[NQ3];
      const double u0d = hv[w * P::kHaloRow + kHaloMax + lane];
      if constexpr (kN) {
        const double sT = __hiloint2double((eT[w] + 1023) << 20, 0);
#pragma unroll
        for (int p = 0; p < NQ3; ++p) {
          const int64_t T = Dot::sum(acc[w][p]);
          y[p] = fmaf((float)(int)(T >> 31), s0 * 2147483648.f, (float)(int)(T & 0x7fffffff) * s0);
          val[w][p] = fma((double)T, sT, u0d);
        }
      } else {
        const float s2 = exp2i(eT[w] + 42), s1 = exp2i(eT[w] + 21);
        // the split the state kernels write, and the bits of the state below it
        const DF u0 = d_to_df(u0d);
        const float u0r = (float)((u0d - (double)u0.h) - (double)u0.l);
#pragma unroll
        for (int p = 0; p < NQ3; ++p) {
          DF x = Dot::value(acc[w][p], s2, s1, s0);
          x.l += u0r;
          y[p] = x.h;
          const DF r = u0 + x;
          val[w][p] = make_float2(r.h, r.l);
        }
        if (eT[w] < -120) {  // units below the FP32 range (states near 1e-30): FP64
          const double sT = ldexp(1.0, eT[w]);
#pragma unroll
          for (int p = 0; p < NQ3; ++p) {
            const DF r = d_to_df(fma(Dot::value_d(acc[w][p]), sT, u0d));
            val[w][p] = make_float2(r.h, r.l);
          }
        }
      }
      sel[w] = 8;
      near[w] = false;
      if (!mine) {
        // no cell: large stencil, nothing to decide
      } else if (a.sel_in) {
        sel[w] = a.sel_in[(int64_t)v * a.n_pad + c];
      } else if (!a.linear) {
        const float eps = (float)a.eps;
        float t[kSmallK + 1], rho = 0.f;
        // the coefficients in the row space of Psi' are T y, y within 2u
        // relative plus Dot::kErr units of the fixed-point sum
        float bsum = 0.f, E = 0.f;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          float q = 0.f;
#pragma unroll
          for (int p = 0; p < (NQ3 <= M ? i + 1 : NQ3); ++p)
            q = fmaf(wa.t.t[i * NQ3 + p], y[p], q);
          bsum = fmaf(q, q, bsum);
        }
#pragma unroll
        for (int p = 0; p < NQ3; ++p) E = fmaf(wa.t.cs[p], fabsf(y[p]), E);
        const float l2 = sqrt_approx(dL[w]) * 1.0002f;
        E = (NQ3 + 5) * 5.9604645e-8f * 1.0001f * E +
            wa.t.cs_all * fmaf(Dot::kErr, s0, Dot::kErrD * l2 * exp2i(-kc));
#pragma unroll
        for (int l = 0; l < MC; ++l) bsum = fmaf(a32[w][l], a32[w][l], bsum);
        if constexpr (MC > 0) E += dot_bound(norm[kSmallK], dL[w], cu, NS);
        t[kSmallK] = bsum + eps;
        rho = beta_rel_bound(bsum, E * 1.0001f, M, eps);
#pragma unroll
        for (int k = 0; k < kSmallK; ++k) {
          const float* td = tsd + (k * kVW + w) * 2 * kTile;
          t[k] = td[0] + eps;
          if ((present >> k) & 1)
            rho = fmaxf(rho, beta_rel_bound(td[0], dot_bound(norm[k], td[kTile], cs, kSmallN),
                                            kSmallM, eps));
        }
        // chi lies within the factor f of its FP32 value under the beta bounds
        // (an eps below the squares of flushed differences decides nothing here)
        near[w] = a.force_near || float_w[w] == 1 || !(rho < 0.25f) ||
                  (sc[w] > 120 && eps < 1e-30f);
        const float q = (1.f + rho) * rcp_approx(1.f - fminf(rho, 0.5f));
        const float q2 = q * q;
        const float f = q2 * q2 * q2 * 1.0002f;
        const float ct = (float)a.ct;
        // most cells keep the large stencil by far: chi_K >= 1 / (1 + 3 r^6) with
        // r the ratio to the smallest directional indicator (2 % for rounding)
        float tm = t[kSmallK];
#pragma unroll
        for (int k = 0; k < kSmallK; ++k)
          if ((present >> k) & 1) tm = fminf(tm, t[k]);
        const float rr = t[kSmallK] * rcp_approx(tm), r2 = rr * rr;
        if (!(fmaf(3.06f * r2, r2 * r2, 1.02f) * (ct * f) < 1.f)) {
          const int x = w_screen(t[0], t[1], t[2], t[kSmallK], present, ct, f);
          near[w] |= (x & 256) != 0;
          sel[w] = x & 15;
        }
      }
    }
    // ---- Gauss-point values of the large polynomial, both variables of a
    // point in one store where both keep it (or may)
    bool put[kVW], both = c < a.n_cell;
#pragma unroll
    for (int w = 0; w < kVW; ++w) {
      if (c < a.n_cell && a.sel_out && !near[w])
        a.sel_out[(int64_t)(v0 + w) * a.n_pad + c] = (uint8_t)sel[w];
      put[w] = c < a.n_cell && !float_w[w] && (near[w] || (sel[w] & 8));
      both &= put[w];
    }
    {
      HT* __restrict__ out = reinterpret_cast<HT*>(a.Uq) + c * kPer + v0;
      bool each = true;
      if constexpr (kVW == 2)  // both variables of a point in 16 bytes
        if (both) {
          each = false;
#pragma unroll
          for (int p = 0; p < NQ3; ++p)
            *reinterpret_cast<float4*>(out + p * NV) =
                make_float4(val[0][p].x, val[0][p].y, val[1][p].x, val[1][p].y);
        }
      if (each) {
#pragma unroll
        for (int w = 0; w < kVW; ++w)
          if (put[w])
#pragma unroll
            for (int p = 0; p < NQ3; ++p) out[p * NV + w] = val[w][p];
      }
    }
    // ---- defer what the fixed-point values do not settle
#pragma unroll
    for (int w = 0; w < kVW; ++w) {
      const bool def = mine && (near[w] || float_w[w] || !(sel[w] & 8));
      const unsigned bal = __ballot_sync(0xffffffffu, def);
      if (def)
        mylist[n_def + __popc(bal & ((1u << lane) - 1u))] =
            make_int2((int)c, (near[w] ? kDefNear : 0) | (float_w[w] ? kDefDirect : 0) |
                                  (sel[w] & 15) * kDefSel | (v0 + w) * kDefVar);
      n_def += __popc(bal);
    }
    __syncwarp();
    while (n_def >= kTile) {
      n_def -= kTile;
      w_deferred<M, NS, NQ, HT>(a, wa, mylist + n_def, kTile, dsc);
      __syncwarp();
    }
  }
  cp_async_wait<0>();
  if (alive && n_def) w_deferred<M, NS, NQ, HT>(a, wa, mylist, n_def, dsc);
}

// ------------------------------------------- FP32-mixed TENO, tile kernel (variant 2)
// The reconstruction of the mixed path, Euler and scalar: FP32 differences and
// multiply-adds, slot by slot in stencil order.  The pipeline is the W form's: a
// producer lane streams a tile's matrices in ring stages and its halo ids with
// bulk copies; each consumer warp gathers its variables' halo states of the next
// tile with cp.async and runs through its tiles without block barriers; four
// matrix entries are read from shared memory at a time, and one read serves both
// of an Euler warp's variables.
// Bound: HBM at large meshes (0.71 GB a launch at 262,088 cells TENO5: 150 us,
// 166 with one variable a warp and two block barriers a tile), the time of a
// tile at small ones (1,152 cells: Euler TENO3 11.3 us, 12.8 before; scalar
// TENO3, which read its matrices straight from global memory, 8.9 and 13.4).
template <int M, int NS, int NQ, int NV>
struct TPlan {
  static constexpr int kVW = NV == 4 ? 2 : 1, kWarps = NV / kVW;  // variables a warp
  static constexpr int kBlocks = NV == 1 ? 6 : 4;
  static constexpr int kEsz = 4;
  static constexpr int kLPS = tile_lps(NS), kSPS = kSmallN;
  static constexpr int kNL = NS / kLPS;
  static constexpr int kStages = kSmallK + kNL;  // the directional stencils first
  static constexpr int kEL = kLPS * M, kES = kSPS * kSmallM;    // entries of a stage, per lane
  static constexpr int kLB = kEL * kTile * kEsz, kSB = kES * kTile * kEsz;
  static constexpr int kSlotN = kTile * 2;  // halo offsets (uint16) of one slot
  static constexpr int kNOff = kLB > kSB ? kLB : kSB;
  static constexpr int kMaxSlots = kLPS > kSPS ? kLPS : kSPS;
  static constexpr int kBuf = kNOff + kMaxSlots * kSlotN;
  static constexpr int64_t kTileMat = (int64_t)(M * NS + kSmallEntries) * kTile * kEsz;
  static constexpr int kSL = NS + kSmallSlots;
  static constexpr int kTileBytes = kWTile * 4;
  static constexpr int kHaloRow = kHaloMax + kTile;  // halo states, then the tile's own
  static constexpr int kHalo = 2 * NV * kHaloRow * 8;
  // Euler: a warp's Gauss values [cell][point][variable], odd row
  static constexpr int kOutRow = 3 * NQ * kVW + 1;
  static constexpr int kOut = NV == 4 ? kWarps * kTile * kOutRow * 4 : 0;
  static constexpr int kFixed = kHalo + 2 * kTileBytes + kOut + 16 * 8 + 16;
  static constexpr int kRoom = (227 * 1024 / kBlocks - 1024 - kFixed) / kBuf;
  static constexpr int kRing = kRoom < 2 ? 2 : (kRoom > 5 ? 5 : kRoom);
  static constexpr size_t kSmem = (size_t)kRing * kBuf + kFixed;
  static_assert(NS % kLPS == 0, "whole stages");
  static_assert(kBuf % 16 == 0 && kNOff % 16 == 0 && kLB % 16 == 0 && kSB % 16 == 0 &&
                    kOut % 16 == 0,
                "bulk-copy alignment");
};

template <int M, int NS, int NQ, int NV>
__global__ void __launch_bounds__(kTile*(TPlan<M, NS, NQ, NV>::kWarps + 1),
                                  (TPlan<M, NS, NQ, NV>::kBlocks))
    recon_tile_kernel(const ReconArgs a, const uint16_t* __restrict__ pos,
                      const int32_t* __restrict__ tiles, const DFTable ev, int* err) {
  using P = TPlan<M, NS, NQ, NV>;
  using St = float2;  // halo states: the (hi, lo) split
  constexpr int kR = P::kRing, kVW = P::kVW, kWarps = P::kWarps, NQ3 = 3 * NQ;
  extern __shared__ __align__(128) unsigned char smem[];
  St* halo = reinterpret_cast<St*>(smem + (size_t)kR * P::kBuf);            // [2][NV][kHaloRow]
  int32_t* tblk = reinterpret_cast<int32_t*>(halo + 2 * NV * P::kHaloRow);  // [2][kWTile]
  float* ostg = reinterpret_cast<float*>(tblk + 2 * kWTile);                // [kWarps][32][kOutRow]
  uint64_t* full = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(ostg) + P::kOut);
  uint64_t* empty = full + kR;
  uint64_t* tfull = empty + kR;
  uint64_t* tempty = tfull + 2;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(full + 16);
  static_assert(2 * kR + 4 <= 16, "mbarriers");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_tiles = (a.n_cell + kTile - 1) / kTile;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int i = 0; i < kR; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kWarps);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], kWarps);
    }
    mbar_fence_init();
  }
  __syncthreads();
  if (warp == kWarps) {
    // ---- producer lane
    if (lane == 0) {
      RingPos<kR> rp;
      bool lap = false;  // every buffer has been filled once
      int it = 0;
      // the block must not exit while a copy it issued is in flight: the last
      // kR stages (buffers before rp.b are one phase ahead) and id blocks
      auto drain = [&](int n_blk) {
        for (int b = 0; b < kR; ++b)
          if (b < rp.b || lap) mbar_wait(&full[b], b < rp.b ? rp.ph : rp.ph ^ 1);
        for (int i = n_blk > 2 ? n_blk - 2 : 0; i < n_blk; ++i)
          mbar_wait(&tfull[i & 1], (uint32_t)(i >> 1) & 1);
      };
      auto gave_up = [&](int w, int n_blk) {
        if (w == 0) {
          atomicOr(err, 2);
          *abort_flag = 1;
        }
        drain(n_blk);
      };
      auto block = [&](int64_t tile, int i) {
        mbar_expect_tx(&tfull[i & 1], P::kTileBytes);
        bulk_g2s(tblk + (i & 1) * kWTile, tiles + tile * kWTile, P::kTileBytes, &tfull[i & 1]);
      };
      int n_blk = 0;  // halo-id blocks issued
      for (; n_blk < 2 && blockIdx.x + (int64_t)n_blk * gridDim.x < n_tiles; ++n_blk)
        block(blockIdx.x + (int64_t)n_blk * gridDim.x, n_blk);
      for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
        const unsigned char* sa = reinterpret_cast<const unsigned char*>(a.ahat) + tile * P::kTileMat;
        const unsigned char* sn =
            reinterpret_cast<const unsigned char*>(pos) + tile * (int64_t)P::kSL * P::kSlotN;
        for (int j = 0; j < P::kStages; ++j) {
          const int b = rp.b;
          if (lap) {
            const int w = mbar_wait_or_abort(&empty[b], rp.ph ^ 1, abort_flag);
            if (w != 1) return gave_up(w, n_blk);
          }
          unsigned char* dst = smem + b * P::kBuf;
          const int js = j - kSmallK;  // large stage
          const unsigned char* src = js < 0 ? sa + P::kNL * P::kLB + j * P::kSB : sa + js * P::kLB;
          const int bytes = js < 0 ? P::kSB : P::kLB;
          const int slot = js < 0 ? NS + j * P::kSPS : js * P::kLPS;
          const int nslot = js < 0 ? P::kSPS : P::kLPS;
          mbar_expect_tx(&full[b], bytes + nslot * P::kSlotN);
          bulk_g2s(dst, src, bytes, &full[b]);
          bulk_g2s(dst + P::kNOff, sn + slot * P::kSlotN, nslot * P::kSlotN, &full[b]);
          rp.next();
          lap |= rp.b == 0;
        }
        const int64_t nxt = tile + 2 * (int64_t)gridDim.x;
        if (nxt < n_tiles) {
          const int w = mbar_wait_or_abort(&tempty[it & 1], (uint32_t)(it >> 1) & 1, abort_flag);
          if (w != 1) return gave_up(w, n_blk);
          block(nxt, n_blk++);
        }
      }
      drain(n_blk);
    }
    return;
  }
  // ---- consumers (warp w: kVW variables from kVW w)
  pdl_wait();  // the states (the producer streams constant data before it)
  constexpr int kPerLane = kHaloMax / kTile;
  const int v0 = warp * kVW;
  int it = 0;
  RingPos<kR> rp;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    const int w = mbar_wait_or_abort(bar, parity, abort_flag, a.wait_polls);
    if (w == 0) {
      atomicOr(err, 2);
      *abort_flag = 1;
    }
    return !__any_sync(0xffffffffu, w != 1);
  };
  auto gather = [&](int64_t tile, int i) {
    bool ok = true;
    if (tile < n_tiles) {
      ok = wait(&tfull[i & 1], (uint32_t)(i >> 1) & 1);
      if (ok) {
        const int32_t* tb = tblk + (i & 1) * kWTile;
        const St* src = a.Us + (int64_t)v0 * a.n_pad;
        St* dst = halo + ((i & 1) * NV + v0) * P::kHaloRow;
        const int H = tb[0];
#pragma unroll
        for (int k = 0; k < kPerLane; ++k)
          if (lane + k * kTile < H) {
            const int id = tb[4 + lane + k * kTile];
#pragma unroll
            for (int w = 0; w < kVW; ++w)
              cp_async8(dst + w * P::kHaloRow + lane + k * kTile, src + w * a.n_pad + id);
          }
        const int64_t c = tile * kTile + lane;
#pragma unroll
        for (int w = 0; w < kVW; ++w)
          cp_async8(dst + w * P::kHaloRow + kHaloMax + lane,
                    src + w * a.n_pad + (c < a.n_cell ? c : 0));
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[i & 1]);
      }
    }
    cp_async_commit();
    return ok;
  };
  if (!gather(blockIdx.x, 0)) {
    cp_async_wait<0>();
    return;
  }
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
    const int64_t c = tile * kTile + lane;  // may be a pad lane of the last tile
    __syncwarp();  // every lane is done with the other halo buffer
    if (!gather(tile + gridDim.x, it + 1)) break;
    const int present = a.smask[c < a.n_cell ? c : 0];
    cp_async_wait<1>();
    __syncwarp();
    St* hv = halo + ((it & 1) * NV + v0) * P::kHaloRow;
    float2 u0s[kVW];
#pragma unroll
    for (int w = 0; w < kVW; ++w) u0s[w] = hv[w * P::kHaloRow + kHaloMax + lane];
    const unsigned char* st = reinterpret_cast<const unsigned char*>(hv);
    auto dif = [&](int w, int off) {
      const float2 x = *reinterpret_cast<const float2*>(st + w * (P::kHaloRow * 8) + off);
      return (x.x - u0s[w].x) + (x.y - u0s[w].y);
    };
    // one stage's products: entries e = slot * kRows + l of the buffer
    auto stage = [&](auto nslots, auto rows, const unsigned char* buf, auto& acc) {
      constexpr int kS = decltype(nslots)::value, kRows = decltype(rows)::value, kN = kS * kRows;
      const uint16_t* nl = reinterpret_cast<const uint16_t*>(buf + P::kNOff) + lane;
      float d[kVW][kS];
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        const int off = nl[s * kTile];
#pragma unroll
        for (int w = 0; w < kVW; ++w) d[w][s] = dif(w, off);
      }
#pragma unroll
      for (int e = 0; e < kN; ++e) {
        const float m = g_entry<kN>(buf, lane, e);
#pragma unroll
        for (int w = 0; w < kVW; ++w) acc[w][e % kRows] = fmaf(m, d[w][e / kRows], acc[w][e % kRows]);
      }
    };
    float as[kSmallK][kVW][kSmallM] = {}, acc[kVW][M] = {};
    bool alive = true;
#pragma unroll
    for (int k = 0; alive && k < kSmallK; ++k) {
      if (!(alive = wait(&full[rp.b], rp.ph))) break;
      stage(std::integral_constant<int, P::kSPS>{}, std::integral_constant<int, kSmallM>{},
            smem + rp.b * P::kBuf, as[k]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[rp.b]);
      rp.next();
    }
#pragma unroll 1
    for (int j = 0; alive && j < P::kNL; ++j) {
      if (!(alive = wait(&full[rp.b], rp.ph))) break;
      stage(std::integral_constant<int, P::kLPS>{}, std::integral_constant<int, M>{},
            smem + rp.b * P::kBuf, acc);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[rp.b]);
      rp.next();
    }
    if (!alive) break;
    // ---- selection and Gauss-point values
    if (c < a.n_cell) {
#pragma unroll
      for (int w = 0; w < kVW; ++w) {
        float aw[kSmallK][kSmallM];
#pragma unroll
        for (int k = 0; k < kSmallK; ++k)
#pragma unroll
          for (int l = 0; l < kSmallM; ++l) aw[k][l] = as[k][w][l];
        plain_finish<M, NQ, kVW, float, DFTable, false>(
            a, ev, c, v0 + w, 0.0, u0s[w], acc[w], aw,
            NV == 4 ? ostg + (warp * kTile + lane) * P::kOutRow + w : nullptr, present);
      }
    }
    // Euler: the warp's values, staged, in rows of consecutive cells
    if constexpr (P::kOut > 0) {
      __syncwarp();
      const int n = (int)min((int64_t)kTile, a.n_cell - tile * kTile) * NQ3;
      const float* o = ostg + warp * kTile * P::kOutRow;
      float* dst = reinterpret_cast<float*>(a.Uq) + tile * kTile * (NQ3 * NV) + v0;
#pragma unroll 3
      for (int e = lane; e < n; e += kTile) {
        const float* q = o + e / NQ3 * P::kOutRow + e % NQ3 * kVW;
        *reinterpret_cast<float2*>(dst + e * NV) = make_float2(q[0], q[1]);
      }
      __syncwarp();
    }
  }
  cp_async_wait<0>();
}

// ------------------------------------ characteristic variables (charvar)
// Characteristic reconstruction (Sec. 2.3 prefers characteristic variables):
// thread (cell, local edge e).  The coefficients of the four conservative
// variables are projected on the characteristic fields of the edge's outward
// normal at the cell-average state, L = L' T and R = T^T R' with T the
// rotation to the edge frame and L', R' the textbook eigenvectors of the 1D
// Euler flux Jacobian in that frame (fields u-c, entropy, shear, u+c).  Each
// field takes its own TENO selection (select_fp64), and the edge's Gauss-point
// values are U_0 + R (Psi' c~).  FP64 throughout; the values are stored in the
// path's Gauss-point type.
template <typename TQ>
__device__ __forceinline__ TQ from_d(double x) {
  if constexpr (std::is_same<TQ, DF>::value) {
    const float h = (float)x;
    return DF{h, (float)(x - (double)h)};
  } else {
    return (TQ)x;
  }
}

template <int M, int NQ, typename TQ>
__global__ void __launch_bounds__(128) char_finish_kernel(
    const double* coef, const double* U,
    const uint8_t* __restrict__ smask, const int32_t* __restrict__ c_faces,
    const double* __restrict__ f_geom, const EvalTable ev, TQ* __restrict__ Uq, int64_t n_cell,
    int64_t n_pad, double g, double ct, double eps, int linear) {
  pdl_wait();
  constexpr int C = M + kSmallK * kSmallM;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_cell * 3) return;
  const int64_t c = idx / 3;
  const int e = (int)(idx % 3);
  const int cf = c_faces[3 * c + e];
  const int64_t f = cf >> 1;
  const double sg = (cf & 1) ? -1.0 : 1.0;  // the neighbour's normal is the opposite one
  const double nx = sg * f_geom[5 * f], ny = sg * f_geom[5 * f + 1];
  double W[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) W[v] = U[(int64_t)v * n_pad + c];
  // eigenvectors at the cell average
  const double r = W[0], un = (W[1] * nx + W[2] * ny) / r, ut = (W[2] * nx - W[1] * ny) / r;
  const double q2 = un * un + ut * ut, p = (g - 1.0) * (W[3] - 0.5 * r * q2);
  const double cs = sqrt(g * p / r), H = (W[3] + p) / r;
  const double b1 = (g - 1.0) / (cs * cs), b2 = 0.5 * b1 * q2;
  const double Lf[4][4] = {
      {0.5 * (b2 + un / cs), 0.5 * (-b1 * un - 1.0 / cs), -0.5 * b1 * ut, 0.5 * b1},
      {1.0 - b2, b1 * un, b1 * ut, -b1},
      {-ut, 0.0, 1.0, 0.0},
      {0.5 * (b2 - un / cs), 0.5 * (-b1 * un + 1.0 / cs), -0.5 * b1 * ut, 0.5 * b1}};
  const double Rf[4][4] = {{1.0, 1.0, 0.0, 1.0},
                           {un - cs, un, 0.0, un + cs},
                           {ut, ut, 1.0, ut},
                           {H - un * cs, 0.5 * q2, ut, H + un * cs}};
  // L = L' T, R = T^T R' with T = rotation (m_x, m_y) -> (m_n, m_t)
  double L[4][4], R[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    L[i][0] = Lf[i][0];
    L[i][1] = Lf[i][1] * nx - Lf[i][2] * ny;
    L[i][2] = Lf[i][1] * ny + Lf[i][2] * nx;
    L[i][3] = Lf[i][3];
    R[0][i] = Rf[0][i];
    R[1][i] = nx * Rf[1][i] - ny * Rf[2][i];
    R[2][i] = ny * Rf[1][i] + nx * Rf[2][i];
    R[3][i] = Rf[3][i];
  }
  const int present = smask[c];
  const double* cv = coef + c * 4 * C;
  // coefficient l of characteristic field i (recomputed where it is needed:
  // holding a field's C coefficients, and the full L and R, spilled)
  auto chc = [&](int i, int l) {
    return L[i][0] * cv[l] + L[i][1] * cv[C + l] + L[i][2] * cv[2 * C + l] + L[i][3] * cv[3 * C + l];
  };
  double corr[4][NQ];
#pragma unroll
  for (int v = 0; v < 4; ++v)
#pragma unroll
    for (int q = 0; q < NQ; ++q) corr[v][q] = 0.0;
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    uint8_t sel = 8;
    if (!linear) {
      double beta[kSmallK + 1];
      double b = 0.0;
#pragma unroll 4
      for (int l = 0; l < M; ++l) {
        const double x = chc(i, l);
        b = fma(x, x, b);
      }
      beta[kSmallK] = b;
#pragma unroll
      for (int k = 0; k < kSmallK; ++k) {
        double bq = 0.0;
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) {
          const double x = chc(i, M + k * kSmallM + l);
          bq = fma(x, x, bq);
        }
        beta[k] = bq;
      }
      sel = select_fp64(beta, present, ct, eps);
    }
    double gq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) gq[q] = 0.0;
    if (sel & 8) {
#pragma unroll 4
      for (int l = 0; l < M; ++l) {
        const double x = chc(i, l);
#pragma unroll
        for (int q = 0; q < NQ; ++q) gq[q] = fma(x, ev.psi[(e * NQ + q) * kMaxM + l], gq[q]);
      }
    } else {
      // equal weights over the kept directional quadratics (kSmallM terms)
      const int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
      const double w = nd ? 1.0 / nd : 0.0;
      double cfin[kSmallM];
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) cfin[l] = 0.0;
#pragma unroll
      for (int k = 0; k < kSmallK; ++k) {
        if (!((sel >> k) & 1)) continue;
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) cfin[l] = fma(w, chc(i, M + k * kSmallM + l), cfin[l]);
      }
#pragma unroll
      for (int l = 0; l < kSmallM; ++l)
#pragma unroll
        for (int q = 0; q < NQ; ++q) gq[q] = fma(cfin[l], ev.psi[(e * NQ + q) * kMaxM + l], gq[q]);
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int v = 0; v < 4; ++v) corr[v][q] = fma(R[v][i], gq[q], corr[v][q]);
  }
  TQ* out = Uq + ((int64_t)(c * 3 + e) * NQ) * 4;
#pragma unroll
  for (int q = 0; q < NQ; ++q)
#pragma unroll
    for (int v = 0; v < 4; ++v) out[q * 4 + v] = from_d<TQ>(W[v] + corr[v][q]);
}

// The characteristic finish of the pair and mixed paths in pair arithmetic
// on the FP32 pipe (the FP64 version above is FP64-pipe bound): the same
// steps, from the (hi, lo) coefficients the reconstruction wrote.  The
// selection is screened in FP32 with the guard band of the pair path and
// decided in FP64 inside it; the Gauss values are written as pairs (pair
// path) or FP32 (mixed path).
template <int M, int NQ, typename TQ>
__global__ void __launch_bounds__(128) char_finish_df_kernel(
    const float2* coef, const double* U,
    const uint8_t* __restrict__ smask, const int32_t* __restrict__ c_faces,
    const double* __restrict__ f_geom, const DFTable ev, TQ* __restrict__ Uq, int64_t n_cell,
    int64_t n_pad, double g, double ct, double eps, int linear) {
  pdl_wait();
  constexpr int C = M + kSmallK * kSmallM;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_cell * 3) return;
  const int64_t c = idx / 3;
  const int e = (int)(idx % 3);
  const int cf = c_faces[3 * c + e];
  const int64_t f = cf >> 1;
  const double sg = (cf & 1) ? -1.0 : 1.0;  // the neighbour's normal is the opposite one
  const DF nx = cst<DF>(sg * f_geom[5 * f]), ny = cst<DF>(sg * f_geom[5 * f + 1]);
  const DF one = {1.f, 0.f}, half = {0.5f, 0.f}, zero = {0.f, 0.f};
  const DF gm1 = cst<DF>(g - 1.0), gg = cst<DF>(g);
  DF W[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) W[v] = cst<DF>(U[(int64_t)v * n_pad + c]);
  // eigenvectors at the cell average, in the edge frame, then rotated
  const DF ir = one / W[0];
  const DF un = (W[1] * nx + W[2] * ny) * ir, ut = (W[2] * nx - W[1] * ny) * ir;
  const DF q2 = un * un + ut * ut;
  const DF p = gm1 * (W[3] - half * W[0] * q2);
  const DF cs = tsqrt(gg * p * ir), ics = one / cs, H = (W[3] + p) * ir;
  const DF b1 = gm1 * ics * ics, b2 = half * b1 * q2;
  const DF Lf[4][4] = {{half * (b2 + un * ics), half * (-(b1 * un) - ics), -(half * b1 * ut), half * b1},
                       {one - b2, b1 * un, b1 * ut, -b1},
                       {-ut, zero, one, zero},
                       {half * (b2 - un * ics), half * (-(b1 * un) + ics), -(half * b1 * ut), half * b1}};
  const DF Rf[4][4] = {{one, one, zero, one},
                       {un - cs, un, zero, un + cs},
                       {ut, ut, one, ut},
                       {H - un * cs, half * q2, ut, H + un * cs}};
  DF L[4][4], R[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    L[i][0] = Lf[i][0];
    L[i][1] = Lf[i][1] * nx - Lf[i][2] * ny;
    L[i][2] = Lf[i][1] * ny + Lf[i][2] * nx;
    L[i][3] = Lf[i][3];
    R[0][i] = Rf[0][i];
    R[1][i] = nx * Rf[1][i] - ny * Rf[2][i];
    R[2][i] = ny * Rf[1][i] + nx * Rf[2][i];
    R[3][i] = Rf[3][i];
  }
  const int present = smask[c];
  const float2* cv = coef + c * 4 * C;
  auto cp = [&](int j) { const float2 x = cv[j]; return DF{x.x, x.y}; };
  // coefficient l of characteristic field i (recomputed where it is needed)
  auto chc = [&](int i, int l) {
    return ((L[i][0] * cp(l) + L[i][1] * cp(C + l)) + L[i][2] * cp(2 * C + l)) +
           L[i][3] * cp(3 * C + l);
  };
  DF corr[4][NQ];
#pragma unroll
  for (int v = 0; v < 4; ++v)
#pragma unroll
    for (int q = 0; q < NQ; ++q) corr[v][q] = zero;
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    uint8_t sel = 8;
    if (!linear) {
      DF bt[kSmallK + 1];
      {
        DF b = zero;
#pragma unroll 4
        for (int l = 0; l < M; ++l) {
          const DF x = chc(i, l);
          df_mac(b, make_float2(x.h, x.l), x);
        }
        bt[kSmallK] = df_norm(b);
#pragma unroll
        for (int k = 0; k < kSmallK; ++k) {
          DF q = zero;
#pragma unroll
          for (int l = 0; l < kSmallM; ++l) {
            const DF x = chc(i, M + k * kSmallM + l);
            df_mac(q, make_float2(x.h, x.l), x);
          }
          bt[k] = df_norm(q);
        }
      }
      float t[kSmallK + 1];
#pragma unroll
      for (int k = 0; k <= kSmallK; ++k) t[k] = bt[k].h + (float)eps;
      bool near = false;
      if (chi_keep32(t, kSmallK, present | 8, (float)ct, &near)) {
        sel = 8;
      } else {
        sel = 0;
#pragma unroll
        for (int k = 0; k < kSmallK; ++k)
          if (((present >> k) & 1) && chi_keep32(t, k, present & 7, (float)ct, &near))
            sel |= (uint8_t)(1u << k);
      }
      if (near) {
        double beta[kSmallK + 1];
#pragma unroll
        for (int k = 0; k <= kSmallK; ++k) beta[k] = df_to_double(bt[k]);
        sel = select_fp64(beta, present, ct, eps);
      }
    }
    DF gq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) gq[q] = zero;
    if (sel & 8) {
#pragma unroll 4
      for (int l = 0; l < M; ++l) {
        const DF x = chc(i, l);
#pragma unroll
        for (int q = 0; q < NQ; ++q) df_mac(gq[q], ev.psi[(e * NQ + q) * kMaxM + l], x);
      }
    } else {
      // equal weights over the kept directional quadratics (kSmallM terms)
      const int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
      const DF fn = {(float)(nd ? nd : 1), 0.f};
#pragma unroll
      for (int l = 0; l < kSmallM; ++l) {
        DF sum = zero;
#pragma unroll
        for (int k = 0; k < kSmallK; ++k)
          if ((sel >> k) & 1) sum = sum + chc(i, M + k * kSmallM + l);
        const DF x = nd ? sum / fn : zero;
#pragma unroll
        for (int q = 0; q < NQ; ++q) df_mac(gq[q], ev.psi[(e * NQ + q) * kMaxM + l], x);
      }
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const DF gn = df_norm(gq[q]);
#pragma unroll
      for (int v = 0; v < 4; ++v) corr[v][q] = corr[v][q] + R[v][i] * gn;
    }
  }
  TQ* out = Uq + ((int64_t)(c * 3 + e) * NQ) * 4;
#pragma unroll
  for (int q = 0; q < NQ; ++q)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const DF r = W[v] + corr[v][q];
      if constexpr (std::is_same<TQ, DF>::value)
        out[q * 4 + v] = r;
      else
        out[q * 4 + v] = r.h;
    }
}

// FP32 hi/lo split of a state: hi = fl32(U), lo = fl32(U - hi)
// Positivity scaling of the reconstruction (Euler; an option, not in the
// paper, which reports its schemes robust on the Mach-10 shock case without
// stating a positivity treatment): Zhang and Shu's limiter.  Each cell's
// Gauss-point states U_q move towards the cell average, U_0 + theta (U_q -
// U_0), with the largest theta <= 1 that keeps the density, then the
// pressure, at least eps = min(1e-13, the average's value) at every face
// Gauss point of the cell.  The reconstruction is linear in its coefficients,
// so scaling the point values equals scaling the polynomial's deviation from
// its mean (the average is unchanged).  Density: theta = (rho_0 - eps) /
// (rho_0 - rho_q) where rho_q < eps; pressure (concave along the segment from
// the average): 60 bisection halvings of [0, 1].  FP64.
__device__ __forceinline__ double pp_pressure(double g, const double* W) {
  return (g - 1.0) * (W[3] - 0.5 * (W[1] * W[1] + W[2] * W[2]) / W[0]);
}

// Largest theta in [0, 1] (60 halvings) that keeps rho > 0 and p >= ep along
// U0 + theta (W - U0), where p < ep at theta = 1.
__device__ __forceinline__ double pp_theta(double g, const double* U0, const double* W, double ep) {
  double D[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) D[v] = W[v] - U0[v];
  auto holds = [&](double th) {
    double X[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) X[v] = U0[v] + th * D[v];
    return X[0] > 0.0 && pp_pressure(g, X) >= ep;
  };
  double lo = 0.0, hi = 1.0;
  int it = 0;
  // The bound is the root r of rho (E - ep / (g - 1)) - |m|^2 / 2, a quadratic
  // in theta.  The halvings that lead to the smallest dyadic interval around r
  // +- 2^-30 are skipped: p is concave in theta, so at their midpoints it
  // stands off ep by at least 2^-30 (p_0 - ep), above its rounding where p_0 is
  // 2^-16 of the energy or more; below that all 60 are made, and so they are
  // if the interval's ends do not confirm it.
  if (pp_pressure(g, U0) - ep > 1.6e-5 * U0[3]) {
    const double e0 = U0[3] - ep / (g - 1.0);
    const double A = D[0] * D[3] - 0.5 * (D[1] * D[1] + D[2] * D[2]);
    const double B = U0[0] * D[3] + D[0] * e0 - (U0[1] * D[1] + U0[2] * D[2]);
    const double C = U0[0] * e0 - 0.5 * (U0[1] * U0[1] + U0[2] * U0[2]);
    const double q = sqrt(B * B - 4.0 * A * C);
    const double r = B <= 0.0 ? 2.0 * C / (q - B) : (-B - q) / (2.0 * A);
    const double r0 = r - 0x1p-30, r1 = r + 0x1p-30;
    if (r0 > 0.0 && r1 < 1.0) {
      // common leading bits of the two ends, as 30-bit fractions
      const unsigned k0 = (unsigned)(r0 * 0x1p30), k1 = (unsigned)(r1 * 0x1p30);
      const int n = k0 == k1 ? 30 : __clz(k0 ^ k1) - 2;
      const double w = 1.0 / (double)(1u << n), l = (double)(k0 >> (30 - n)) * w;
      if ((l == 0.0 || holds(l)) && (l + w >= 1.0 || !holds(l + w))) {
        lo = l;
        hi = l + w;
        it = n;
      }
    }
  }
  for (; it < 60; ++it) {
    const double sm = 0.5 * (lo + hi);
    if (holds(sm))
      lo = sm;
    else
      hi = sm;
  }
  return lo;
}

// One thread per (cell, Gauss point), 32 cells a block: a cell's theta is the
// smallest of its points'.  Bound: the FP64 latency of the points that break
// the floor, 30 bisection steps of an FP64 division each; one thread per cell
// that took its points in turn, 60 steps each, left a few lanes of the warps at
// the shock working for 309 us (double Mach reflection, 32,768 cells; now 62).
template <int NQ, typename TQ>
__global__ void __launch_bounds__(32 * 3 * NQ) positivity_kernel(const double* U,
                                                                 TQ* __restrict__ Uq,
                                                                 int64_t n_cell, int64_t n_pad,
                                                                 double g) {
  pdl_wait();
  constexpr int NP = 3 * NQ;
  __shared__ double s_th[32 * NP];
  const int64_t i = (int64_t)blockIdx.x * (32 * NP) + threadIdx.x;
  const int64_t c = i / NP;
  const bool in = c < n_cell;
  const int base = (int)threadIdx.x / NP * NP;
  double U0[4], W[4], er = 0.0, ep = 0.0;
  if (in) {
    TQ x[4];
    ld_group<4>(Uq + i * 4, x);
#pragma unroll
    for (int v = 0; v < 4; ++v) U0[v] = U[v * n_pad + c], W[v] = to_d(x[v]);
    er = fmin(1e-13, U0[0]);
    ep = fmin(1e-13, pp_pressure(g, U0));
  }
  // the cell's smallest theta from its points'
  auto cell_min = [&](double th) {
    s_th[threadIdx.x] = th;
    __syncthreads();
    double m = 1.0;
#pragma unroll
    for (int q = 0; q < NP; ++q) m = fmin(m, s_th[base + q]);
    __syncthreads();
    return m;
  };
  auto scale = [&](double th) {
#pragma unroll
    for (int v = 0; v < 4; ++v) W[v] = U0[v] + th * (W[v] - U0[v]);
  };
  bool scaled = false;
  // density
  const bool low = in && W[0] < er;
  if (__syncthreads_or(low)) {
    const double th = cell_min(low ? fmin(1.0, (U0[0] - er) / (U0[0] - W[0])) : 1.0);
    if (in && th < 1.0) {
      scaled = true;
      scale(th);
    }
  }
  // pressure
  const bool under = in && !(pp_pressure(g, W) >= ep);
  if (__syncthreads_or(under)) {
    const double th = cell_min(under ? pp_theta(g, U0, W, ep) : 1.0);
    if (in && th < 1.0) {
      scaled = true;
      scale(th);
    }
  }
  if (!scaled) return;
  TQ x[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) x[v] = from_d<TQ>(W[v]);
  st_group<4>(Uq + i * 4, x);
}

// The outflow layer (cells with a face on an outflow boundary) enters every
// face flux with its cell average: after the reconstruction, each Gauss slot
// of such a cell takes U_0 (in the Gauss-value type of the path).  One thread
// per (layer cell, slot).
template <int NV, int NQ3, typename TQ>
__global__ void layer_fill_kernel(const double* U, TQ* __restrict__ Uq,
                                  const int32_t* __restrict__ list, int64_t n, int64_t n_pad) {
  pdl_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * NQ3) return;
  const int64_t c = list[i / NQ3];
  const int p = (int)(i % NQ3);
  TQ* o = Uq + (c * NQ3 + p) * NV;
#pragma unroll
  for (int v = 0; v < NV; ++v) o[v] = from_d<TQ>(U[v * n_pad + c]);
}

// Adjoint of layer_fill_kernel: a layer cell's Gauss-slot cotangents (pairs
// on the pair path, FP64 otherwise) go to its cell average, summed per edge
// into ubd[cell][edge][var] (added to the cell's adjoint by the reverse
// gather), and the slots are cleared so that the reconstruction's adjoint
// sends nothing through the cell's polynomial.  One thread per (cell, edge).
template <int NV, int NQ, bool kPairs>
__global__ void layer_vjp_kernel(double* __restrict__ Uq_bar, double* __restrict__ ubd,
                                 const int32_t* __restrict__ list, int64_t n) {
  pdl_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * 3) return;
  const int64_t c = list[i / 3];
  const int e = (int)(i % 3);
  double acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0;
  const int64_t b = ((c * 3 + e) * NQ) * NV;
  for (int q = 0; q < NQ; ++q)
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int64_t j = b + q * NV + v;
      if constexpr (kPairs) {
        float2* u = reinterpret_cast<float2*>(Uq_bar) + j;
        acc[v] += (double)u->x + (double)u->y;
        *u = make_float2(0.f, 0.f);
      } else {
        acc[v] += Uq_bar[j];
        Uq_bar[j] = 0.0;
      }
    }
#pragma unroll
  for (int v = 0; v < NV; ++v) ubd[(c * 3 + e) * NV + v] = acc[v];
}

// Halo exchange of partitioned meshes (copy-based; each kernel touches only
// its own context's arrays).  pack: buf[v][i] = U[v][idx[i]]; unpack: the
// reverse, with the FP32 hi/lo split of the written states when Us is given;
// add = 1 adds instead (the adjoint's contributions returned to their owner).
__global__ void halo_pack_kernel(const double* U, int64_t ld,
                                 const int32_t* __restrict__ idx, int64_t n, int n_var,
                                 double* __restrict__ buf) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t c = idx[i];
  for (int v = 0; v < n_var; ++v) buf[v * n + i] = U[v * ld + c];
}
__global__ void halo_unpack_kernel(double* __restrict__ U, int64_t ld,
                                   const int32_t* __restrict__ idx, int64_t n, int n_var,
                                   const double* __restrict__ buf, float2* __restrict__ Us,
                                   int add) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t c = idx[i];
  for (int v = 0; v < n_var; ++v) {
    const double x = add ? U[v * ld + c] + buf[v * n + i] : buf[v * n + i];
    U[v * ld + c] = x;
    if (Us) {
      const float hi = (float)x;
      Us[v * ld + c] = make_float2(hi, (float)(x - (double)hi));
    }
  }
}

__global__ void split_kernel(const double* U, float2* __restrict__ Us, int64_t n_cell,
                             int64_t n_pad, int n_var) {
  pdl_wait();
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_cell) return;
  for (int v = 0; v < n_var; ++v) {
    const double u = U[v * n_pad + c];
    const float hi = (float)u;
    Us[v * n_pad + c] = make_float2(hi, (float)(u - (double)hi));
  }
}

// ------------------------------------------------------------------ fluxes
struct FaceArgs {
  const int32_t* f_cells;
  const int8_t* f_edges;
  const double* f_geom;
  const float2* f_geom2;  // [n_face][3] nx, ny, |A| as (hi, lo) pairs
  int64_t n_pad;
  int64_t n_face;
  double gamma, adv_x, adv_y, time;
  int adv_field;
  double adv_cx, adv_cy, adv_omega, adv_r1, adv_r2;
  double gw[kMaxNq], gt[kMaxNq];
  float2 gw2[kMaxNq], g2, gm12;  // Gauss weights, gamma, gamma - 1 as pairs
};

// face constants in the flux scalar type: FP64 from the double geometry,
// pairs and floats from the copy split on the host (no FP64 conversions)
template <typename T>
__device__ __forceinline__ void face_k(const double* fg, const float2* fg2, int64_t f, double g,
                                       float2 g2, float2 gm12, RiemannK<T>& rk, T& tl) {
  if constexpr (std::is_same<T, double>::value) {
    rk = riemann_k<double>(fg[5 * f], fg[5 * f + 1], g);
    tl = fg[5 * f + 2];
  } else if constexpr (std::is_same<T, DF>::value) {
    const float2 nx = fg2[3 * f], ny = fg2[3 * f + 1], ln = fg2[3 * f + 2];
    rk = {DF{1.f, 0.f}, DF{0.5f, 0.f}, DF{gm12.x, gm12.y}, DF{g2.x, g2.y}, DF{nx.x, nx.y},
          DF{ny.x, ny.y}};
    tl = DF{ln.x, ln.y};
  } else {
    rk = {1.f, 0.5f, gm12.x, g2.x, fg2[3 * f].x, fg2[3 * f + 1].x};
    tl = fg2[3 * f + 2].x;
  }
}
template <typename T>
__device__ __forceinline__ T gauss_w(double w, float2 w2) {
  if constexpr (std::is_same<T, double>::value)
    return w;
  else if constexpr (std::is_same<T, DF>::value)
    return DF{w2.x, w2.y};
  else
    return w2.x;
}

// One thread per (face, Gauss point), 64 faces a block; the points' fluxes go
// through shared memory to the face's weighted sum, in the order of the points.
// Bound: the issue of the Riemann solver (pairs, FP32) or the FP64 pipe at
// large meshes, the latency of one solve at small ones, where a thread that
// took a face's points in turn ran three of them in a row (32,768 cells TENO5
// pairs: 18.6 us for three points a thread, 12.8 now; 262,088 cells TENO6:
// 63 to 53.6; FP64, 131,072 cells: 199 to 174, 139 with the FP64 solver's own form).
constexpr int kFluxFaces = 64;

template <int NV, int NQ, int FLUX, typename T>
__global__ void __launch_bounds__(kFluxFaces * NQ)
    face_flux_kernel(const FaceArgs a, const T* Uq, T* __restrict__ K) {
  pdl_wait();
  __shared__ __align__(16) T sF[kFluxFaces * NQ * NV];
  const int64_t f0 = (int64_t)blockIdx.x * kFluxFaces;
  const int k = threadIdx.x % NQ;
  const int64_t f = f0 + threadIdx.x / NQ;
  if (f < a.n_face) {
    const int o = a.f_cells[2 * f], n = a.f_cells[2 * f + 1];
    const int eo = a.f_edges[2 * f], en = a.f_edges[2 * f + 1];
    RiemannK<T> rk;
    T tl;
    face_k<T>(a.f_geom, a.f_geom2, f, a.gamma, a.g2, a.gm12, rk, tl);
    // (the Gauss values of an outflow-layer cell are its cell average, written
    // by layer_fill_kernel: at an outflow face both states are that average)
    T UL[NV], UR[NV], F[NV];
    ld_group<NV>(Uq + ((int64_t)(o * 3 + eo) * NQ + k) * NV, UL);
    if (n >= 0) {
      ld_group<NV>(Uq + ((int64_t)(n * 3 + en) * NQ + (NQ - 1 - k)) * NV, UR);
    } else if constexpr (NV == 4) {
      const double nx = a.f_geom[5 * f], ny = a.f_geom[5 * f + 1], len = a.f_geom[5 * f + 2];
      const double x = a.f_geom[5 * f + 3] - ny * len * a.gt[k];
      ghost_state<T>(en, UL, nx, ny, x, a.time, a.gamma, UR);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) UR[v] = UL[v];
    }
    if constexpr (NV == 1) {
      const double nx = a.f_geom[5 * f], ny = a.f_geom[5 * f + 1], len = a.f_geom[5 * f + 2];
      const double xq = a.f_geom[5 * f + 3] - ny * len * a.gt[k];
      const double yq = a.f_geom[5 * f + 4] + nx * len * a.gt[k];
      const double an = adv_normal(a.adv_field, a.adv_x, a.adv_y, a.adv_cx, a.adv_cy,
                                   a.adv_omega, a.adv_r1, a.adv_r2, xq, yq, nx, ny);
      F[0] = cst<T>(an) * (an >= 0.0 ? UL[0] : UR[0]);
    } else {
      euler_riemann<T>(UL, UR, rk, FLUX == TENO_FLUX_HLLC, F);
    }
    st_group<NV>(sF + threadIdx.x * NV, F);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kFluxFaces * NV; e += kFluxFaces * NQ) {
    const int lf = e / NV, v = e % NV;
    if (f0 + lf >= a.n_face) break;
    RiemannK<T> rk;
    T tl;
    face_k<T>(a.f_geom, a.f_geom2, f0 + lf, a.gamma, a.g2, a.gm12, rk, tl);
    T acc = cst<T>(0.0);
#pragma unroll
    for (int q = 0; q < NQ; ++q)
      acc = madd(gauss_w<T>(a.gw[q], a.gw2[q]), sF[(lf * NQ + q) * NV + v], acc);
    K[f0 * NV + e] = acc * tl;
  }
}

// ------------------------------------------------------------------ gather
struct GatherArgs {
  const int32_t* c_faces;
  const double* inv_area;
  int64_t n_cell, n_pad;
  double gamma;
};

// CFL speed lambda = (|u| + c) / L of a cell from its conservative state in
// FP64 (a non-physical cell, rho <= 0, p <= 0 or NaN, makes it infinite, which
// the host reports as TENO_ENONPHYS; fmax would drop a NaN speed), or from the
// (hi, lo) split of the state and the pair 1/L in pair arithmetic on the FP32
// pipe (relative error ~1e-14, far below what a CFL step needs; false for a NaN
// speed, which is skipped as fmax skips it)
__device__ __forceinline__ double cfl_speed(const double* W, double gamma) {
  const double rho = W[0], u = W[1] / rho, v = W[2] / rho;
  const double p = (gamma - 1.0) * (W[3] - 0.5 * rho * (u * u + v * v));
  const double s = sqrt(u * u + v * v) + sqrt(gamma * p / rho);
  return !(rho > 0.0) || !(p > 0.0) ? __longlong_as_double(0x7ff0000000000000LL) : s;
}
__device__ __forceinline__ bool cfl_speed_split(const float2* q, float2 il, float2 g2, float2 gm12,
                                                DF* lam) {
  const DF one = {1.f, 0.f}, half = {0.5f, 0.f}, gg = {g2.x, g2.y}, gm1 = {gm12.x, gm12.y};
  const DF rho = {q[0].x, q[0].y}, mx = {q[1].x, q[1].y}, my = {q[2].x, q[2].y},
           E = {q[3].x, q[3].y};
  const DF ir = one / rho;
  const DF u = mx * ir, v = my * ir;
  const DF k = u * u + v * v;
  const DF p = gm1 * (E - half * rho * k);
  const DF sp = tsqrt(k) + tsqrt(gg * p * ir);
  *lam = sp * DF{il.x, il.y};
  return lam->h == lam->h;
}
// block maximum of non-negative lam (which order like their bit patterns) into
// *out; every thread of a 256-thread block takes part
__device__ __forceinline__ void block_max(double lam, unsigned long long* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lam = fmax(lam, __shfl_xor_sync(0xffffffffu, lam, o));
  __shared__ double red[32];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red[w] = lam;
  __syncthreads();
  if (w == 0) {
    lam = l < (int)(blockDim.x >> 5) ? red[l] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lam = fmax(lam, __shfl_xor_sync(0xffffffffu, lam, o));
    if (l == 0) atomicMax(out, (unsigned long long)__double_as_longlong(lam));
  }
}

// The next step's CFL maximum, taken by the update that makes its state (the
// last stage of a step with another one after it): the same per-cell speeds as
// max_lambda_kernel and max_lambda_split_kernel without their launch and read.
// A step of a small mesh is bound by its chain of launches, ten of them with the
// separate reduction: 2,048 cells, scalar TENO3, 63.5 -> 58 us a step, 32,768
// cells, Euler TENO5, 170 -> 162.
struct NextLam {
  unsigned long long* out = nullptr;   // maximum of this update's states, or none
  unsigned long long* zero = nullptr;  // a word to clear (an earlier stage), or none
  const double* cfl_len = nullptr;
  const float2* ilen2 = nullptr;
  const double* cell_speed = nullptr;
  double adv_speed = 0.0;
  float2 g2, gm12;
};

// (kLam: with the next step's CFL maximum; its own instantiation, because the
// other updates ran 4 % slower with its registers)
template <int NV, typename TK, bool kLam>
__global__ void __launch_bounds__(256) gather_kernel(const GatherArgs a, const TK* K,
                                                     const double* Un, const double* Us,
                                                     double* __restrict__ out, int mode, double cn,
                                                     double cs, double dt_fixed, double cfl,
                                                     const double* max_lam, int* flag,
                                                     float2* __restrict__ split,
                                                     const NextLam nl) {
  pdl_wait();
  // the step size once per block (one FP64 division, while the others load)
  __shared__ double s_dt;
  if (mode != 0 && threadIdx.x == 0) s_dt = max_lam ? cfl / *max_lam : dt_fixed;
  if (nl.zero && blockIdx.x == 0 && threadIdx.x == 0) *nl.zero = 0ull;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = c < a.n_cell;
  double acc[NV], un[NV], us[NV], ia = 0.0;
  if (in) {
    if constexpr (std::is_same<TK, DF>::value || std::is_same<TK, float>::value) {
      // pair (or FP32) fluxes summed in pairs on the FP32 pipe, one conversion
      // per variable; three FP32 terms sum exactly in a pair
      DF sum[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) sum[v] = DF{0.f, 0.f};
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const int cf = a.c_faces[3 * c + e];
        const int64_t f = cf >> 1;
        TK kf[NV];
        ld_group<NV>(K + f * NV, kf);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          DF k;
          if constexpr (std::is_same<TK, DF>::value)
            k = kf[v];
          else
            k = DF{kf[v], 0.f};
          sum[v] = (cf & 1) ? sum[v] - k : sum[v] + k;
        }
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = to_d(sum[v]);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = 0.0;
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const int cf = a.c_faces[3 * c + e];
        const int64_t f = cf >> 1;
        const double s = (cf & 1) ? -1.0 : 1.0;
        TK kf[NV];
        ld_group<NV>(K + f * NV, kf);
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = fma(s, to_d(kf[v]), acc[v]);
      }
    }
    ia = a.inv_area[c];
    if (mode == 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) out[v * a.n_pad + c] = -acc[v] * ia;
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) un[v] = Un[v * a.n_pad + c], us[v] = Us[v * a.n_pad + c];
    }
  }
  if (mode == 0) return;
  __syncthreads();
  double lam = 0.0;
  if (in) {
    const double wr = cs * s_dt * ia;  // the stage's weight of the face-flux sum
    double u[NV];
    float2 sp[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int64_t i = v * a.n_pad + c;
      u[v] = fma(-wr, acc[v], fma(cn, un[v], cs * us[v]));
      out[i] = u[v];
      if (split) {
        const float hi = (float)u[v];
        sp[v] = make_float2(hi, (float)(u[v] - (double)hi));
        split[i] = sp[v];
      }
    }
    if constexpr (NV == 4) {
      // rho > 0 and p > 0, the latter as rho E - |m|^2 / 2 > 0 (no division)
      const double rho = u[0];
      const double pr = u[3] * rho - 0.5 * (u[1] * u[1] + u[2] * u[2]);
      if (!(rho > 0.0) || !(pr > 0.0)) atomicOr(flag, 1);
    } else {
      if (!(u[0] == u[0])) atomicOr(flag, 1);
    }
    if constexpr (kLam) {
      if constexpr (NV == 1) {
        lam = (nl.cell_speed ? nl.cell_speed[c] : nl.adv_speed) / nl.cfl_len[c];
      } else if (split) {
        DF l;
        if (cfl_speed_split(sp, nl.ilen2[c], nl.g2, nl.gm12, &l)) lam = fmax(0.0, to_d(l));
      } else {
        lam = cfl_speed(u, a.gamma) / nl.cfl_len[c];
      }
    }
  }
  if constexpr (kLam) block_max(lam, nl.out);
}

// --------------------------------------------------------------- CFL speed
template <int NV>
__global__ void __launch_bounds__(256) max_lambda_kernel(const double* U,
                                                         const double* __restrict__ cfl_len,
                                                         int64_t n_cell, int64_t n_pad,
                                                         double gamma, double adv_speed,
                                                         const double* __restrict__ cell_speed,
                                                         unsigned long long* out) {
  pdl_wait();
  double lam = 0.0;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_cell;
       c += (int64_t)gridDim.x * blockDim.x) {
    double s;
    if constexpr (NV == 1) {
      s = cell_speed ? cell_speed[c] : adv_speed;
    } else {
      double W[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) W[v] = U[v * n_pad + c];
      s = cfl_speed(W, gamma);
    }
    lam = fmax(lam, s / cfl_len[c]);
  }
  block_max(lam, out);
}

// The same maximum from the (hi, lo) split of the state that the FP64 and
// mixed paths keep for the reconstruction (Euler): lambda_c = (|u| + c) / L_c
// in pair arithmetic on the FP32 pipe (relative error ~1e-14, far below what
// a CFL step needs) with 1/L_c as host-split pairs; the maximum as FP64
// bits.  Non-physical cells (NaN speed) are skipped as fmax skips them.
__global__ void __launch_bounds__(256) max_lambda_split_kernel(const float2* Us,
                                                               const float2* __restrict__ ilen2,
                                                               int64_t n_cell, int64_t n_pad,
                                                               float2 g2, float2 gm12,
                                                               unsigned long long* out) {
  pdl_wait();
  DF lam = {0.f, 0.f};
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_cell;
       c += (int64_t)gridDim.x * blockDim.x) {
    float2 q[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) q[v] = Us[v * n_pad + c];
    DF l;
    if (cfl_speed_split(q, ilen2[c], g2, gm12, &l)) lam = vmax(lam, l);
  }
  block_max(to_d(lam), out);
}

// -------------------------------------------------------------- utilities
__global__ void permute_kernel(const double* src, double* __restrict__ dst,
                               const int32_t* __restrict__ perm, int64_t n, int64_t ld_src,
                               int64_t ld_dst, int to_user) {
  pdl_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int v = blockIdx.y;
  if (i >= n) return;
  const int64_t u = perm[i];
  if (to_user)
    dst[v * ld_dst + u] = src[v * ld_src + i];
  else
    dst[v * ld_dst + i] = src[v * ld_src + u];
}

__global__ void permute_u8_kernel(const uint8_t* src, uint8_t* __restrict__ dst,
                                  const int32_t* __restrict__ perm, int64_t n, int64_t ld_src,
                                  int64_t ld_dst, int to_user) {
  pdl_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int v = blockIdx.y;
  if (i >= n) return;
  const int64_t u = perm[i];
  if (to_user)
    dst[v * ld_dst + u] = src[v * ld_src + i];
  else
    dst[v * ld_dst + i] = src[v * ld_src + u];
}

__global__ void axpby_kernel(double* out, const double* a, double ca, const double* b, double cb,
                             int64_t n) {
  pdl_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = ca * a[i] + cb * b[i];
}

// ------------------------------------------------------------------ adjoint
struct VjpArgs {
  const int32_t* f_cells;
  const int8_t* f_edges;
  const double* f_geom;
  const float2* f_geom2;
  float2 g2, gm12;
  int adv_field;
  double adv_cx, adv_cy, adv_omega, adv_r1, adv_r2;
  const double* inv_area;
  int64_t n_face, n_pad;
  double gamma, adv_x, adv_y, time;
  double gw[kMaxNq], gt[kMaxNq];
  float2 gw2[kMaxNq];  // Gauss weights as (hi, lo) pairs
};

// Uq_bar[(c,edge,q)] = w_q |A| (dF/dU_side)^T Kbar with Kbar = dJ/dK_f
// (R_o has -K/|V_o|, R_n has +K/|V_n|); every Gauss slot of every cell is
// written by exactly one face.  Euler: the hand-written reverse sweep of the
// Riemann solver (euler_riemann_vjp, ghost_vjp).  Scalar advection, and Euler
// when built with TENO_VJP_REVERSE=0: Jacobian columns from forward-mode dual
// numbers over scalar S, ND seeded directions per pass (an interior face
// seeds the NV components of U_L, then those of U_R; a boundary face only U_L,
// the ghost state carrying dU_R/dU_L).
// Euler flux VJP by the hand-written reverse sweep (1) or by forward-mode
// dual numbers (0; kept as the cross-check of the reverse sweep)
#ifndef TENO_VJP_REVERSE
#define TENO_VJP_REVERSE 1
#endif
constexpr bool kVjpReverse = TENO_VJP_REVERSE != 0;

// Uq_bar entry i: (hi, lo) pairs on the pair path (S = DF; read as pairs by
// the reconstruction VJP, no FP64 conversion on either side), FP64 on the
// native path
template <typename S>
__device__ __forceinline__ void store_bar(double* base, int i, S x) {
  if constexpr (std::is_same<S, DF>::value)
    reinterpret_cast<float2*>(base)[i] = make_float2(x.h, x.l);
  else
    base[i] = to_d(x);
}

// One thread per (face, Gauss point), 64 faces a block; the faces' cotangents
// are formed once and shared.  Bound: FP32 issue (pairs) at 168 registers, the
// latency of one reverse sweep at small meshes, where a thread that took a
// face's points in turn ran three in a row
// (8,320 cells TENO6, HLLC: 136 us a residual's adjoint, 122 now).  The states
// load while the cotangents are formed (1,048,352 cells TENO6: 706 us, 746 with
// the loads after the barrier; 32 faces a block 722).
// kTurn: one thread per face, its points in turn, 128 faces a block (HLL in pairs).
// At meshes that fill the machine many times over the latency no longer counts
// and three times the faces in flight cover the scattered reads better: from
// 524,288 faces on (points side by side / in turn: 393k faces 184 / 185 us, 786k
// 358 / 344, 1.57M 704 / 667, 12.6M 5,542 / 5,288).  HLLC and FP64 hold a face's
// cotangents through the sweeps at the price of spills: 786k faces 413 / 435 and
// 1,618 / 1,660.
constexpr int64_t kTurnFaces = (int64_t)1 << 19;
constexpr int kTurnBlock = 128;
template <int NV, int NQ, int FLUX, typename TQ, typename S, int ND, bool kTurn>
__global__ void __launch_bounds__(kTurn ? kTurnBlock : kFluxFaces * NQ,
                                  kTurn ? 3 : 384 / (kFluxFaces * NQ))
    face_flux_vjp_kernel(const VjpArgs a, const TQ* Uq, const double* w,
                         double* __restrict__ Uq_bar) {
  pdl_wait();
  static_assert((2 * NV) % ND == 0, "directions per pass must divide 2 NV");
  using D = Dual<ND, S>;
  __shared__ S sK[kTurn ? 1 : kFluxFaces * NV];
  const int64_t f0 = (int64_t)blockIdx.x * (kTurn ? kTurnBlock : kFluxFaces);
  // Kbar in FP64 from the FP64 weights, once per face in the flux scalar type
  auto kbar = [&](int64_t f, int v) {
    const int o = a.f_cells[2 * f], n = a.f_cells[2 * f + 1];
    double kb = -w[v * a.n_pad + o] * a.inv_area[o];
    if (n >= 0) kb = fma(w[v * a.n_pad + n], a.inv_area[n], kb);
    return cst<S>(kb);
  };
  if constexpr (!kTurn)
    for (int e = threadIdx.x; e < kFluxFaces * NV; e += kFluxFaces * NQ) {
      const int64_t f = f0 + e % kFluxFaces;
      if (f < a.n_face) sK[e % kFluxFaces * NV + e / kFluxFaces] = kbar(f, e / kFluxFaces);
    }
  const int lf = kTurn ? threadIdx.x : threadIdx.x / NQ;
  const bool in = f0 + lf < a.n_face;  // (past the end: the last face's loads)
  if (kTurn && !in) return;
  const int64_t f = in ? f0 + lf : a.n_face - 1;
  const int o = a.f_cells[2 * f], n = a.f_cells[2 * f + 1];
  const int eo = a.f_edges[2 * f], en = a.f_edges[2 * f + 1];
  const double nx = a.f_geom[5 * f], ny = a.f_geom[5 * f + 1], len = a.f_geom[5 * f + 2];
  S kf[NV];
  if constexpr (kTurn) {
#pragma unroll
    for (int v = 0; v < NV; ++v) kf[v] = kbar(f, v);
  }
  const S* Kb = kTurn ? kf : sK + lf * NV;
  const int n_pass = ((n >= 0 ? 2 * NV : NV) + ND - 1) / ND;
  RiemannK<S> rks;
  S tl;  // |A| in the flux scalar type
  face_k<S>(a.f_geom, a.f_geom2, f, a.gamma, a.g2, a.gm12, rks, tl);
  const RiemannK<D> rk = riemann_k_dual<ND, S>(rks);
  for (int k = kTurn ? 0 : threadIdx.x % NQ; k < NQ; k += kTurn ? 1 : NQ) {
    TQ ul[NV], ur[NV];
    ld_group<NV>(Uq + ((int64_t)(o * 3 + eo) * NQ + k) * NV, ul);
    if (n >= 0) ld_group<NV>(Uq + ((int64_t)(n * 3 + en) * NQ + (NQ - 1 - k)) * NV, ur);
    if constexpr (!kTurn) {
      __syncthreads();  // the cotangents, while the states load
      if (!in) return;
    }
    // x of the Gauss point (ghost states and the scalar field only)
    auto xq = [&]() { return a.f_geom[5 * f + 3] - ny * len * a.gt[k]; };
    const S wl = gauss_w<S>(a.gw[k], a.gw2[k]) * tl;
    S Kw[NV];  // w_k |A| Kbar in the flux scalar type
#pragma unroll
    for (int v = 0; v < NV; ++v) Kw[v] = wl * Kb[v];
    double* outL = Uq_bar + ((int64_t)(o * 3 + eo) * NQ + k) * NV;
    double* outR = n >= 0 ? Uq_bar + ((int64_t)(n * 3 + en) * NQ + (NQ - 1 - k)) * NV : outL;
    if constexpr (NV == 4 && kVjpReverse) {
      // reverse mode: one forward recomputation and its adjoint sweep
      S uL[NV], uR[NV], ULb[NV], URb[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        uL[v] = lift<S>(ul[v]);
        ULb[v] = cst<S>(0.0);
        URb[v] = cst<S>(0.0);
      }
      if (n >= 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) uR[v] = lift<S>(ur[v]);
      } else {
        ghost_state<S>(en, uL, nx, ny, xq(), a.time, a.gamma, uR);
      }
      euler_riemann_vjp<S>(uL, uR, rks, FLUX == TENO_FLUX_HLLC, Kw, ULb, URb);
      if (n < 0) ghost_vjp<S>(en, rks, URb, ULb);
      if constexpr (std::is_same<S, DF>::value) {
        st_group<NV>(reinterpret_cast<DF*>(outL), ULb);
        if (n >= 0) st_group<NV>(reinterpret_cast<DF*>(outR), URb);
      } else {
        st_group<NV>(outL, ULb);
        if (n >= 0) st_group<NV>(outR, URb);
      }
    } else {
      for (int pass = 0; pass < n_pass; ++pass) {
        const int dir0 = pass * ND;  // directions dir0 .. dir0+ND-1 of [U_L, U_R]
        D UL[NV], UR[NV], F[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          UL[v] = cst<D>(0.0);
          UL[v].v = lift<S>(ul[v]);
          if (v >= dir0 && v < dir0 + ND) UL[v].d[v - dir0] = cst<S>(1.0);
        }
        if (n >= 0) {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            UR[v] = cst<D>(0.0);
            UR[v].v = lift<S>(ur[v]);
            if (NV + v >= dir0 && NV + v < dir0 + ND) UR[v].d[NV + v - dir0] = cst<S>(1.0);
          }
        } else if constexpr (NV == 4) {
          ghost_state<D>(en, UL, nx, ny, xq(), a.time, a.gamma, UR);  // carries dUR/dUL
        } else {
#pragma unroll
          for (int v = 0; v < NV; ++v) UR[v] = UL[v];
        }
        if constexpr (NV == 1) {
          const double yq = a.f_geom[5 * f + 4] + nx * len * a.gt[k];
          const double an = adv_normal(a.adv_field, a.adv_x, a.adv_y, a.adv_cx, a.adv_cy,
                                       a.adv_omega, a.adv_r1, a.adv_r2, xq(), yq, nx, ny);
          F[0] = an * (an >= 0.0 ? UL[0] : UR[0]);
        } else {
          euler_riemann<D>(UL, UR, rk, FLUX == TENO_FLUX_HLLC, F);
        }
#pragma unroll
        for (int j = 0; j < ND; ++j) {
          S sacc = cst<S>(0.0);
#pragma unroll
          for (int i = 0; i < NV; ++i) sacc = madd(F[i].d[j], Kw[i], sacc);
          const int g = dir0 + j;
          if (g < NV)
            store_bar<S>(outL, g, sacc);
          else if (n >= 0)
            store_bar<S>(outR, g - NV, sacc);
        }
      }
    }
  }
}

// stencil slots unrolled in the reconstruction VJP kernels (matrix loads in
// flight per thread)
#ifndef TENO_VJP_SLOT_UNROLL
#define TENO_VJP_SLOT_UNROLL 2
#endif
constexpr int kVjpSlotUnroll = TENO_VJP_SLOT_UNROLL;

// d_bar[tile][slot][v][32] = (A''^T abar)_slot with abar = w_k Psi'^T Uq_bar
// (selection frozen); u_self = sum_p Uq_bar - sum_slot d_bar (dU_0 terms).
template <int M, int NS, int NQ, int NV, typename TS>
__global__ void __launch_bounds__(128) recon_vjp_kernel(const TS* __restrict__ ahat,
                                                        const uint8_t* sel_in,
                                                        const double* Uq_bar,
                                                        double* __restrict__ d_bar,
                                                        double* __restrict__ u_self,
                                                        int64_t n_cell, int64_t n_pad,
                                                        const EvalTable ev) {
  pdl_wait();
  const int lane = threadIdx.x, v = threadIdx.y;
  const int64_t tile = (int64_t)blockIdx.x * blockDim.z + threadIdx.z;
  const int64_t c = tile * kTile + lane;
  if (c >= n_cell) return;
  constexpr int E = M * NS + kSmallEntries;
  constexpr int SL = NS + kSmallSlots;
  const TS* A = ahat + tile * (int64_t)E * kTile + lane;
  // matrix entry as FP64 (pairs of the double-float storage are summed)
  auto ent = [](TS x) -> double {
    if constexpr (std::is_same<TS, float2>::value)
      return (double)x.x + (double)x.y;
    else
      return x;
  };
  double* db = d_bar + tile * (int64_t)SL * NV * kTile + lane * NV + v;
  double cb[M];
#pragma unroll
  for (int l = 0; l < M; ++l) cb[l] = 0.0;
  double u0b = 0.0;
  const double* ub = Uq_bar + c * (3 * NQ * NV) + v;
#pragma unroll
  for (int p = 0; p < 3 * NQ; ++p) {
    const double b = ub[p * NV];
    u0b += b;
#pragma unroll
    for (int l = 0; l < M; ++l) cb[l] = fma(b, ev.psi[p * kMaxM + l], cb[l]);
  }
  const uint8_t sel = sel_in[(int64_t)v * n_pad + c];
  double tot = 0.0;
  const bool large = sel & 8;
#pragma unroll (kVjpSlotUnroll)
  for (int s = 0; s < NS; ++s) {
    double t = 0.0;
    if (large) {
#pragma unroll
      for (int l = 0; l < M; ++l) t = fma(ent(A[(int64_t)(s * M + l) * kTile]), cb[l], t);
    }
    db[(int64_t)s * NV * kTile] = t;
    tot += t;
  }
  const int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
  const double w = (!large && nd) ? 1.0 / nd : 0.0;
#pragma unroll
  for (int k = 0; k < kSmallK; ++k) {
    const double wk = ((sel >> k) & 1) ? w : 0.0;
    for (int s = 0; s < kSmallN; ++s) {
      double t = 0.0;
      if (wk != 0.0) {
        const TS* As = A + (int64_t)(M * NS + (k * kSmallN + s) * kSmallM) * kTile;
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) t = fma(ent(As[l * kTile]), cb[l], t);
        t *= wk;
      }
      db[(int64_t)(NS + k * kSmallN + s) * NV * kTile] = t;
      tot += t;
    }
  }
  u_self[(int64_t)v * n_pad + c] = u0b - tot;
}

// Double-float version for the FP64 path (matrices stored as (hi, lo)
// pairs): the transposed matvecs run on the FP32 pipe; d_bar is written as
// pairs, u_self in FP64.
__device__ __forceinline__ DF df_div_small(DF a, int n) {  // a / n for n in 1..3
  const float fn = (float)n;
  const float qh = a.h / fn;
  const float r = fmaf(-qh, fn, a.h);  // exact remainder
  return two_sum(qh, (r + a.l) / fn);
}

template <int M, int NS, int NQ, int NV>
__global__ void __launch_bounds__(128) recon_vjp_df_kernel(const float2* __restrict__ ahat,
                                                           const uint8_t* sel_in,
                                                           const double* Uq_bar,
                                                           DF* __restrict__ d_bar,
                                                           double* __restrict__ u_self,
                                                           int64_t n_cell, int64_t n_pad,
                                                           const DFTable ev) {
  pdl_wait();
  const int lane = threadIdx.x, v = threadIdx.y;
  const int64_t tile = (int64_t)blockIdx.x * blockDim.z + threadIdx.z;
  const int64_t c = tile * kTile + lane;
  if (c >= n_cell) return;
  constexpr int E = M * NS + kSmallEntries;
  constexpr int SL = NS + kSmallSlots;
  const float2* A = ahat + tile * (int64_t)E * kTile + lane;
  DF* db = d_bar + tile * (int64_t)SL * NV * kTile + lane * NV + v;
  DF cb[M];
#pragma unroll
  for (int l = 0; l < M; ++l) cb[l] = {0.f, 0.f};
  DF u0b = {0.f, 0.f};
  // Uq_bar as (hi, lo) pairs (written so by the pair-path flux VJP)
  const float2* ub = reinterpret_cast<const float2*>(Uq_bar) + c * (3 * NQ * NV) + v;
#pragma unroll
  for (int p = 0; p < 3 * NQ; ++p) {
    const DF b = {ub[p * NV].x, ub[p * NV].y};
    u0b = u0b + b;
#pragma unroll
    for (int l = 0; l < M; ++l) df_mac(cb[l], ev.psi[p * kMaxM + l], b);
  }
#pragma unroll
  for (int l = 0; l < M; ++l) cb[l] = df_norm(cb[l]);
  const uint8_t sel = sel_in[(int64_t)v * n_pad + c];
  DF tot = {0.f, 0.f};
  const bool large = sel & 8;
#pragma unroll (kVjpSlotUnroll)
  for (int s = 0; s < NS; ++s) {
    DF t = {0.f, 0.f};
    if (large) {
#pragma unroll
      for (int l = 0; l < M; ++l)
        df_mac(t, A[(int64_t)(s * M + l) * kTile], cb[l]);
      t = df_norm(t);
    }
    db[(int64_t)s * NV * kTile] = t;
    tot = tot + t;
  }
  const int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
#pragma unroll
  for (int k = 0; k < kSmallK; ++k) {
    const bool on = !large && ((sel >> k) & 1);
    for (int s = 0; s < kSmallN; ++s) {
      DF t = {0.f, 0.f};
      if (on) {
        const float2* As = A + (int64_t)(M * NS + (k * kSmallN + s) * kSmallM) * kTile;
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) df_mac(t, As[l * kTile], cb[l]);
        t = df_div_small(df_norm(t), nd);
      }
      db[(int64_t)(NS + k * kSmallN + s) * NV * kTile] = t;
      tot = tot + t;
    }
  }
  u_self[(int64_t)v * n_pad + c] = to_d(u0b - tot);
}

// Tiled reconstruction VJP (FP64 path, Euler, W form).  With the selection
// frozen, Uq_p = U_0 + sum_s W_ps d_s for the large polynomial (W = Psi' G in
// the forward W-form kernel's fixed point), so d_bar_s = sum_p W_ps Uq_bar_p:
// NQ3 products per slot and no coefficient adjoint.  Directional stencils
// (cells whose large stencil is cut) take d_bar_s = (G_k^T Psi_k^T Uq_bar)_s /
// n_kept from their (hi, lo) matrices; their stages are streamed only for tiles
// where some (cell, variable) keeps a directional stencil, a predicate the
// producer and the consumers evaluate from the same selection bytes.  The products
// W^T Uq_bar run in fixed point, Uq_bar in 53 bits of the cell's largest; the
// contributions are pairs, so that each keeps its own precision however much the
// cotangents of a tile's cells differ.  Each lane adds its d_bar_s to the tile's
// halo accumulator in shared memory at the slot's halo position (lanes with equal
// positions in lane order, by ranks the host stores next to the positions; slots
// in stencil order: deterministic sums).  The host assigns the large-stencil
// members to slots so that the lanes of a tile do not share a cell within a slot,
// and these slots take one round.  At the end of the tile the accumulator is
// written as one pair per (halo entry, variable), so the reverse gather reads the
// few halo entries that hold a cell instead of every stencil slot that holds it.
// The tile's Uq_bar block is prefetched with cp.async one tile ahead.  Bound:
// instruction issue (131,072 cells TENO5 158 us, 152 with integer accumulators of
// one unit a tile; 8,320 cells TENO6 42, 44 with these; 1,048,352 cells TENO6 1,485
// and 1,425; pair products took 158, 43 and 1,575).
constexpr int kRingV = 4;
constexpr int kUbStride = 38;  // doubles per cell in the Uq_bar stage (16-byte rows)
constexpr int kHaccStride = kHaloMax + 4;  // pairs per variable row (conflict-free transpose)

template <int M, int NS, int NQ3>
struct VjpPlan {
  static constexpr int kLPS = 4, kSPS = 4;
  static constexpr int kLay = wform_lps(NS);          // slots of a layout stage
  static_assert(kLPS % kLay == 0, "whole layout stages");
  static constexpr int kSlotW = NQ3 * kTile * 8;      // W of one large slot
  static constexpr int kSlotS = kSmallM * kTile * 8;  // matrix pairs of one directional slot
  static constexpr int kSlotN = kTile * 2;            // halo positions (uint16) of one slot
  static constexpr int kNL = (NS + kLPS - 1) / kLPS;
  static constexpr int kPerSmall = kSmallN / kSPS;
  static constexpr int kStages = kNL + kSmallK * kPerSmall;
  static constexpr int kNOff = kLPS * kSlotW > kSPS * kSlotS ? kLPS * kSlotW : kSPS * kSlotS;
  static constexpr int kMat = kNOff + (kLPS > kSPS ? kLPS : kSPS) * kSlotN;
  static constexpr int kSL = NS + kSmallSlots;
  static constexpr int64_t kTileW = (int64_t)NS * NQ3 * kTile * 8;
  static constexpr int64_t kTileA = (int64_t)(M * NS + kSmallEntries) * kTile * 8;
  static constexpr size_t kUbOff = (size_t)kRingV * kMat;
  static constexpr size_t kUbBytes = (size_t)2 * kTile * kUbStride * 8;
  static constexpr size_t kHaccOff = kUbOff + kUbBytes;
  static constexpr size_t kHaccBytes = (size_t)4 * kHaccStride * 8;
  static constexpr size_t kBarOff = kHaccOff + kHaccBytes;
  static constexpr size_t kSmem = kBarOff + 2 * kRingV * 8 + 16 + 16;
  static_assert(NQ3 * 4 <= kUbStride, "Uq_bar row");
  static_assert(kSmallN % kSPS == 0, "directional stencil split");
  static_assert(kMat % 16 == 0 && kUbOff % 16 == 0 && kHaccOff % 16 == 0 && kBarOff % 8 == 0,
                "alignment");
  // stage j: slots [slot0, slot0 + nslot) of stencil k (-1: large, from W;
  // else from the directional matrices), source byte offset in the tile's
  // W or matrix block
  __device__ static void stage(int j, int& slot0, int& nslot, int& k, int64_t& off, int& bytes) {
    if (j < kNL) {
      slot0 = j * kLPS;
      nslot = (NS - slot0) < kLPS ? (NS - slot0) : kLPS;
      k = -1;
      off = (int64_t)slot0 * kSlotW;
      bytes = nslot * kSlotW;
    } else {
      const int i = j - kNL;
      k = i / kPerSmall;
      const int s0 = (i % kPerSmall) * kSPS;
      slot0 = NS + k * kSmallN + s0;
      nslot = kSPS;
      off = (int64_t)(M * NS + (k * kSmallN + s0) * kSmallM) * kTile * 8;
      bytes = kSPS * kSlotS;
    }
  }
};

// the (cell, variable) of this selection byte keeps directional stencils:
// its large stencil is cut and at least one directional stencil is kept
__device__ __forceinline__ bool vjp_needs_small(uint8_t sel) {
  return !(sel & 8) && (sel & 7);
}

template <int M, int NS, int NQ>
__global__ void __launch_bounds__(kTile * (kConsumers + 1), 3)
    recon_vjp_tma_kernel(const float2* __restrict__ ahat, const int2* __restrict__ wq,
                         const int32_t* __restrict__ wstat, const HaloArgs h,
                         const uint8_t* sel_in,
                         const double* Uq_bar, float2* __restrict__ part,
                         double* __restrict__ u_self, int64_t n_cell, int64_t n_pad,
                         const DFTable ev, int* err) {
  pdl_wait();
  constexpr int NV = 4, NQ3 = 3 * NQ, kPer = NQ3 * NV;
  using VP = VjpPlan<M, NS, NQ3>;
  using Dot = WPairDot<26>;
  extern __shared__ __align__(128) unsigned char smem[];
  double* ubs = reinterpret_cast<double*>(smem + VP::kUbOff);     // [2][32][kUbStride]
  float2* hacc = reinterpret_cast<float2*>(smem + VP::kHaccOff);  // [NV][kHaccStride]
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + VP::kBarOff);
  uint64_t* empty = full + kRingV;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + kRingV);
  int* need = const_cast<int*>(abort_flag) + 4;  // [NV] per-variable small-stencil flags
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_tiles = (n_cell + kTile - 1) / kTile;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int i = 0; i < kRingV; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kConsumers);
    }
    mbar_fence_init();
  }
  __syncthreads();
  if (warp == kConsumers) {
    // ---- producer lane: W blocks (and directional matrices where needed)
    if (lane == 0) {
      int64_t g = 0;
      for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const unsigned char* sw = reinterpret_cast<const unsigned char*>(wq) + tile * VP::kTileW;
        const unsigned char* sa = reinterpret_cast<const unsigned char*>(ahat) + tile * VP::kTileA;
        const unsigned char* sn =
            reinterpret_cast<const unsigned char*>(h.nbr_loc) + tile * (int64_t)VP::kSL * VP::kSlotN;
        // the tile's selection bytes: 2 x 16 per variable (rows of n_pad, a
        // multiple of 32), pad lanes masked
        const int nval = (int)min((int64_t)kTile, n_cell - tile * kTile);
        uint4 sw4[2 * NV];
#pragma unroll
        for (int w = 0; w < NV; ++w)
#pragma unroll
          for (int q = 0; q < 2; ++q)
            sw4[2 * w + q] =
                *(reinterpret_cast<const uint4*>(sel_in + (int64_t)w * n_pad + tile * kTile) + q);
        bool small = false;
#pragma unroll
        for (int w = 0; w < NV; ++w)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const uint32_t words[4] = {sw4[2 * w + q].x, sw4[2 * w + q].y, sw4[2 * w + q].z,
                                       sw4[2 * w + q].w};
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const uint8_t b = (uint8_t)(words[i >> 2] >> (8 * (i & 3)));
              small |= (16 * q + i < nval) && vjp_needs_small(b);
            }
          }
        const int n_stages = small ? VP::kStages : VP::kNL;
        for (int j = 0; j < n_stages; ++j, ++g) {
          const int b = (int)(g % kRingV);
          if (g >= kRingV) {
            const int w =
                mbar_wait_or_abort(&empty[b], (uint32_t)((g / kRingV) - 1) & 1, abort_flag);
            if (w != 1) {
              if (w == 0) {
                atomicOr(err, 2);
                *abort_flag = 1;
              }
              for (int64_t i = g - kRingV; i < g; ++i)
                mbar_wait(&full[i % kRingV], (uint32_t)(i / kRingV) & 1);
              return;
            }
          }
          int slot0, nslot, k, bytes;
          int64_t off;
          VP::stage(j, slot0, nslot, k, off, bytes);
          const uint32_t bn = (uint32_t)(nslot * VP::kSlotN);
          unsigned char* dst = smem + (size_t)b * VP::kMat;
          mbar_expect_tx(&full[b], (uint32_t)bytes + bn);
          bulk_g2s(dst, (k < 0 ? sw : sa) + off, (uint32_t)bytes, &full[b]);
          bulk_g2s(dst + VP::kNOff, sn + slot0 * VP::kSlotN, bn, &full[b]);
        }
      }
      // the block must not exit while a copy it issued is in flight
      for (int64_t i = g > kRingV ? g - kRingV : 0; i < g; ++i)
        mbar_wait(&full[i % kRingV], (uint32_t)(i / kRingV) & 1);
    }
    return;
  }
  // ---- consumers (warp v: variable v)
  const int v = warp, tid = threadIdx.x;
  // Uq_bar block of a tile (contiguous [cell][point][variable]) into stage hb
  auto prefetch = [&](int64_t tile, int hb) {
    const int nval = (int)min((int64_t)kTile, n_cell - tile * kTile);
    const double* src = Uq_bar + tile * kTile * kPer;
    double* dst = ubs + (size_t)hb * kTile * kUbStride;
    for (int e = tid; e < nval * (kPer / 2); e += kConsumers * kTile) {
      const int cl = e / (kPer / 2), w = e - cl * (kPer / 2);
      cp_async16(dst + cl * kUbStride + 2 * w, src + (int64_t)cl * kPer + 2 * w);
    }
    cp_async_commit();
  };
  float2* hrow = hacc + v * kHaccStride;
  // add t at the halo position of code (bits 0-7); lanes with equal positions
  // in the order of their precomputed ranks (bits 8-12)
  auto accumulate = [&](bool act, int code, DF t) {
    const int hp = code & kHaloPosMask;
    const unsigned rank = (unsigned)code >> 8;
    const unsigned rmax = __reduce_max_sync(0xffffffffu, act ? rank : 0u);
    for (unsigned r = 0; r <= rmax; ++r) {
      if (act && rank == r) {
        const float2 q = hrow[hp];
        const DF x = DF{q.x, q.y} + t;
        hrow[hp] = make_float2(x.h, x.l);
      }
      __syncwarp();
    }
  };
  int64_t g = 0;
  int hb = 0;
  bool dead = false;
  if ((int64_t)blockIdx.x < n_tiles) prefetch(blockIdx.x, 0);
  // the halo offsets, the selection byte and the exponent of W's unit of a
  // tile, loaded a tile ahead
  auto pre = [&](int64_t tile, int& h0, int& H, uint8_t& sl, int& kc) {
    h0 = 0, H = 0, sl = 0, kc = 0;
    if (tile < n_tiles) {
      h0 = h.off[tile];
      H = h.off[tile + 1] - h0;
      const int64_t cc = tile * kTile + lane;
      if (cc < n_cell) sl = sel_in[(int64_t)v * n_pad + cc];
      kc = (int)(int16_t)(wstat[(tile * kWStat + kWStat - 1) * kTile + lane] & 0xffff);
    }
  };
  int h0n, Hn, kcn;
  uint8_t seln;
  pre(blockIdx.x, h0n, Hn, seln, kcn);
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, hb ^= 1) {
    consumer_sync();  // the previous tile's accumulator, flags and Uq_bar stage are released
    const int64_t nxt = tile + gridDim.x;
    if (nxt < n_tiles)
      prefetch(nxt, hb ^ 1);
    else
      cp_async_commit();
    const int h0 = h0n, H = Hn, kc = kcn;
    const uint8_t sel = seln;
    pre(nxt, h0n, Hn, seln, kcn);
    for (int i = lane; i < H; i += kTile) hrow[i] = make_float2(0.f, 0.f);
    const int64_t c = tile * kTile + lane;
    const bool valid = c < n_cell;
    const bool vs = __any_sync(0xffffffffu, valid && vjp_needs_small(sel));
    if (lane == 0) need[v] = vs;
    cp_async_wait<1>();
    consumer_sync();  // the tile's Uq_bar has landed; the flags are set
    const bool small = need[0] | need[1] | need[2] | need[3];
    const int n_stages = small ? VP::kStages : VP::kNL;
    const bool large = valid && (sel & 8);
    const int nd = (sel & 1) + ((sel >> 1) & 1) + ((sel >> 2) & 1);
    // Uq_bar of (c, v) at the Gauss points: in fixed point, 53 bits of the
    // largest, unit 2^-sb; and the coefficient adjoints of the directional
    // polynomials (first kSmallM basis functions) in pairs, where the block
    // needs them
    typename Dot::D bd[NQ3];
    float sT;  // scale of a contribution
    DF u0b = {0.f, 0.f};
    DF cbs[kSmallM];
#pragma unroll
    for (int l = 0; l < kSmallM; ++l) cbs[l] = {0.f, 0.f};
    {
      const float2* us = reinterpret_cast<const float2*>(ubs) +
                         (size_t)hb * kTile * kUbStride + lane * kUbStride + v;
      float2 q[NQ3];
      unsigned mx = 0u;
#pragma unroll
      for (int p = 0; p < NQ3; ++p) {
        q[p] = valid ? us[p * NV] : make_float2(0.f, 0.f);
        mx = max(mx, mag_bits(q[p]));
        u0b = u0b + DF{q[p].x, q[p].y};
      }
      if (small && valid && !large) {
#pragma unroll
        for (int p = 0; p < NQ3; ++p)
#pragma unroll
          for (int l = 0; l < kSmallM; ++l)
            df_mac(cbs[l], ev.psi[p * kMaxM + l], DF{q[p].x, q[p].y});
#pragma unroll
        for (int l = 0; l < kSmallM; ++l) cbs[l] = df_norm(cbs[l]);
      }
      const int e = mag_exp<float2>(mx);
      const bool bad = e == kFixExpBad;
      const int sb = bad ? 0 : 52 - e;
#pragma unroll
      for (int p = 0; p < NQ3; ++p) Dot::split(bad ? 0 : to_fix(q[p], sb), 0, 0.f, bd[p]);
      // (zero where the large stencil gives nothing; an infinity or a NaN goes to
      // every cell of the stencil; denormal for cotangents below 2^-114)
      const int uT = Dot::exp(kc, sb);
      sT = uT + 42 >= -126 ? exp2i(uT + 42) : __int_as_float(1 << max(uT + 42 + 149, 0));
      if (!large) sT = 0.f;
      if (large && bad) sT = __int_as_float(0x7fffffff);
    }
    DF tot = {0.f, 0.f};
    for (int j = 0; j < n_stages; ++j, ++g) {
      const int b = (int)(g % kRingV);
      int slot0, nslot, k, bytes;
      int64_t off;
      VP::stage(j, slot0, nslot, k, off, bytes);
      if (!dead) {
        const int w = mbar_wait_or_abort(&full[b], (uint32_t)(g / kRingV) & 1, abort_flag);
        if (w == 0) {
          atomicOr(err, 2);
          *abort_flag = 1;
        }
        dead = __any_sync(0xffffffffu, w != 1);
      }
      const unsigned char* buf = smem + (size_t)b * VP::kMat;
      const uint16_t* nl = reinterpret_cast<const uint16_t*>(buf + VP::kNOff) + lane;
      auto add = [&](bool on, int s, DF t) {
        accumulate(on, nl[s * kTile], t);
        const DF q = two_sum(tot.h, t.h);  // running sum, renormalised at the end
        tot.h = q.h;
        tot.l += q.l + t.l;
      };
      if (dead) {
        // skip the stage
      } else if (k < 0) {
        if (__any_sync(0xffffffffu, large)) {
          // the stage's slot values first (independent chains), then their
          // accumulation slot by slot
          DF ts[VP::kLPS];
#pragma unroll
          for (int s = 0; s < VP::kLPS; ++s) {
            typename Dot::A acc;
#pragma unroll
            for (int p = 0; p < NQ3; ++p)
              Dot::mac(
                  acc,
                  Dot::entry(w_entry<VP::kLay * NQ3>(
                      buf + s / VP::kLay * VP::kLay * VP::kSlotW, lane, s % VP::kLay * NQ3 + p)),
                  bd[p]);
            // |T| < 9 2^31 2^27 < 2^61.2 units of 2^(26 - kc - sb) (its FP32 part below
            // 2^35, rounded to 16 units) as a pair, of limbs of 21 bits that FP32 holds
            const int64_t T = acc.hh + (int64_t)__float2int_rn(acc.x * 0.0625f) * 16;
            const float h2 = (float)(int)(T >> 42);
            const float h1 = (float)((int)(T >> 21) & 0x1fffff) * 0x1p-21f;
            const float h0 = (float)((int)T & 0x1fffff) * 0x1p-42f;
            const DF x = fast_two_sum(h2, h1);
            ts[s] = DF{x.h * sT, (x.l + h0) * sT};
          }
#pragma unroll
          for (int s = 0; s < VP::kLPS; ++s)
            if (s < nslot) add(large, s, ts[s]);
        }
      } else {
        const bool on = valid && !large && ((sel >> k) & 1);
        if (__any_sync(0xffffffffu, on)) {
          const float2* mat = reinterpret_cast<const float2*>(buf) + lane;
#pragma unroll
          for (int s = 0; s < VP::kSPS; ++s) {
            DF t = {0.f, 0.f};
            if (on) {
#pragma unroll
              for (int l = 0; l < kSmallM; ++l) df_mac(t, mat[(s * kSmallM + l) * kTile], cbs[l]);
              t = df_div_small(df_norm(t), nd);
            }
            add(on, s, t);
          }
        }
      }
      __syncwarp();
      if (lane == 0 && !dead) mbar_arrive(&empty[b]);
    }
    if (valid && !dead) u_self[(int64_t)v * n_pad + c] = to_d(u0b - df_norm(tot));
    consumer_sync();  // every variable's accumulator is complete
    if (!dead) {
      float2* dst = part + (int64_t)h0 * NV;
      for (int e = tid; e < H * NV; e += kConsumers * kTile)
        dst[e] = hacc[(e & 3) * kHaccStride + (e >> 2)];
    }
  }
  cp_async_wait<0>();
}

#ifndef TENO_SCATTER_BATCH
#define TENO_SCATTER_BATCH 4
#endif
constexpr int kScatterBatch = TENO_SCATTER_BATCH;
// v[j] = u_self[j] + sum over the stencil slots that hold cell j.  d_bar is
// [tile][slot][lane][var]: the NV values of one slot entry are one 32-byte
// sector (NV = 4), read with vector loads; rev_idx holds entry numbers
// (tile * SL + slot) * 32 + lane.
template <int NV, typename TD>
__global__ void __launch_bounds__(256) scatter_gather_kernel(const int64_t* __restrict__ rev_off,
                                                             const int32_t* __restrict__ rev_idx,
                                                             const TD* d_bar,
                                                             const double* u_self0,
                                                             double* __restrict__ out,
                                                             int64_t n_cell, int64_t n_pad,
                                                             const double* ubd) {
  pdl_wait();
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_cell) return;
  const int64_t r0 = rev_off[j], r1 = rev_off[j + 1];
  // the cell's own term, plus what its Gauss slots owe its average (outflow
  // layer cells, written by layer_vjp_kernel; zero elsewhere)
  double u_self[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    u_self[v] = u_self0[v * n_pad + j];
    if (ubd) u_self[v] += (ubd[(j * 3 + 0) * NV + v] + ubd[(j * 3 + 1) * NV + v]) +
                          ubd[(j * 3 + 2) * NV + v];
  }
  if constexpr (std::is_same<TD, DF>::value) {
    DF acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = d_to_df(u_self[v]);
    int64_t r = r0;
    if constexpr (NV == 4) {
      // kScatterBatch entries per round: every index, then every sector, is
      // requested before any is used (independent loads in flight)
      for (; r + kScatterBatch <= r1; r += kScatterBatch) {
        int id[kScatterBatch];
#pragma unroll
        for (int i = 0; i < kScatterBatch; ++i) id[i] = __ldg(rev_idx + r + i);
        float4 a[kScatterBatch], b[kScatterBatch];
#pragma unroll
        for (int i = 0; i < kScatterBatch; ++i) {
          const float4* e = reinterpret_cast<const float4*>(d_bar + (int64_t)id[i] * NV);
          a[i] = e[0];
          b[i] = e[1];
        }
#pragma unroll
        for (int i = 0; i < kScatterBatch; ++i) {
          acc[0] = acc[0] + DF{a[i].x, a[i].y};
          acc[1] = acc[1] + DF{a[i].z, a[i].w};
          acc[2] = acc[2] + DF{b[i].x, b[i].y};
          acc[3] = acc[3] + DF{b[i].z, b[i].w};
        }
      }
    }
    for (; r < r1; ++r) {
      const TD* e = d_bar + (int64_t)rev_idx[r] * NV;
      if constexpr (NV == 4) {
        const float4 a = *reinterpret_cast<const float4*>(e);
        const float4 b = *(reinterpret_cast<const float4*>(e) + 1);
        acc[0] = acc[0] + DF{a.x, a.y};
        acc[1] = acc[1] + DF{a.z, a.w};
        acc[2] = acc[2] + DF{b.x, b.y};
        acc[3] = acc[3] + DF{b.z, b.w};
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = acc[v] + e[v];
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) out[v * n_pad + j] = to_d(acc[v]);
  } else {
    double acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = u_self[v];
    for (int64_t r = r0; r < r1; ++r) {
      const TD* e = d_bar + (int64_t)rev_idx[r] * NV;
      if constexpr (NV == 4) {
        const double2 a = *reinterpret_cast<const double2*>(e);
        const double2 b = *(reinterpret_cast<const double2*>(e) + 1);
        acc[0] += a.x;
        acc[1] += a.y;
        acc[2] += b.x;
        acc[3] += b.y;
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] += e[v];
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) out[v * n_pad + j] = acc[v];
  }
}

template <typename F>
cudaError_t dispatch_order(int order, F&& f) {
  switch (order) {
    case 3: return f(std::integral_constant<int, 5>{}, std::integral_constant<int, 12>{});
    case 4: return f(std::integral_constant<int, 9>{}, std::integral_constant<int, 20>{});
    case 5: return f(std::integral_constant<int, 14>{}, std::integral_constant<int, 30>{});
    case 6: return f(std::integral_constant<int, 20>{}, std::integral_constant<int, 42>{});
  }
  return cudaErrorInvalidValue;
}

// launch with the programmatic-serialization attribute (pdl_wait)
// (the callers return cudaGetLastError())
template <typename... KA, typename... A>
void launch(void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
            A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, KA(args)...);
}

}  // namespace

// ---------------------------------------------------------------- launchers
// blocks of a persistent kernel: what is resident, at most one per tile
template <typename K>
cudaError_t resident_grid(K kern, int threads, size_t smem, int64_t tiles, unsigned* grid) {
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem)) !=
      cudaSuccess)
    return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  *grid = (unsigned)std::min<int64_t>(tiles, (int64_t)per_sm * sms);
  return cudaSuccess;
}

template <int M, int NS, int NQ, int NV>
cudaError_t launch_recon_tile(const ReconArgs& a, const DeviceMesh& dm, cudaStream_t st) {
  using P = TPlan<M, NS, NQ, NV>;
  auto kern = recon_tile_kernel<M, NS, NQ, NV>;
  const int threads = kTile * (P::kWarps + 1);
  unsigned grid = 0;
  const cudaError_t e =
      resident_grid(kern, threads, P::kSmem, (a.n_cell + kTile - 1) / kTile, &grid);
  if (e != cudaSuccess) return e;
  ReconArgs b = a;
  b.ahat = dm.tmat;
  launch(kern, grid, threads, P::kSmem, st, b, dm.wpos, dm.wtile, dm.eval_df, dm.err_flag);
  return cudaGetLastError();
}

template <int M, int NS, int NQ, bool kDF>
cudaError_t launch_recon_tma(const ReconArgs& a, const DeviceMesh& dm, cudaStream_t st) {
  using TR = TmaTraits<kDF, M, NS, NQ>;
  using P = StagePlan<M, NS, (int)sizeof(typename TR::TE), TR::kLPS, TR::kSPS, TR::kRing>;
  auto kern = recon_tma_kernel<M, NS, NQ, kDF>;
  const int threads = kTile * (kConsumers + 1);
  unsigned grid = 0;
  const cudaError_t e =
      resident_grid(kern, threads, P::kSmem, (a.n_cell + kTile - 1) / kTile, &grid);
  if (e != cudaSuccess) return e;
  launch(kern, grid, threads, P::kSmem, st, a, dm.halo, dm.eval_df, dm.err_flag);
  return cudaGetLastError();
}

template <int M, int NS, int NQ, typename HT>
cudaError_t launch_recon_tma_w(const ReconArgs& a, const DeviceMesh& dm, int* err,
                               cudaStream_t st) {
  using P = WPlan<M, NS, 3 * NQ, HT>;
  auto kern = recon_tma_w_kernel<M, NS, NQ, HT>;
  const int threads = kTile * (P::kWWarps + 1);
  unsigned grid = 0;
  const cudaError_t e =
      resident_grid(kern, threads, P::kSmem, (a.n_cell + kTile - 1) / kTile, &grid);
  if (e != cudaSuccess) return e;
  WArgs wa;
  wa.psi = std::is_same<HT, double>::value ? (const void*)dm.psi_d : (const void*)dm.psi_df;
  wa.g32 = dm.g32;
  wa.w = dm.wq;
  wa.pos = dm.wpos;
  wa.tile = dm.wtile;
  wa.st = dm.wstat;
  wa.t = dm.wt;
  launch(kern, grid, threads, P::kSmem, st, a, wa, err);
  return cudaGetLastError();
}

cudaError_t launch_char_finish(const DeviceMesh& dm, const double* U, void* Uq, cudaStream_t st) {
  if (!dm.coef_out || dm.n_var != 4) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)((dm.n_recon * 3 + 127) / 128);
  return dispatch_order(dm.order, [&](auto Mc, auto NSc) -> cudaError_t {
    constexpr int M = decltype(Mc)::value;
    (void)NSc;
    constexpr int NQ = (M <= 9) ? 2 : 3;
    if (dm.nq != NQ) return cudaErrorInvalidValue;
    auto go = [&](auto tq) -> cudaError_t {
      using TQ = typename decltype(tq)::type;
      if constexpr (std::is_same<TQ, double>::value)
        launch(char_finish_kernel<M, NQ, TQ>, grid, 128, 0, st, dm.coef_out, U, dm.smask,
               dm.c_faces, dm.f_geom, dm.eval, (TQ*)Uq, dm.n_recon,
               dm.n_pad, dm.gamma, dm.ct, dm.eps, dm.linear);
      else
        launch(char_finish_df_kernel<M, NQ, TQ>, grid, 128, 0, st,
               reinterpret_cast<const float2*>(dm.coef_out), U, dm.smask, dm.c_faces, dm.f_geom,
               dm.eval_df, (TQ*)Uq, dm.n_recon, dm.n_pad, dm.gamma, dm.ct, dm.eps, dm.linear);
      return cudaGetLastError();
    };
    if (dm.precision == TENO_FP64) return go(TypeTag<DF>{});
    if (dm.precision == TENO_FP32_MIXED) return go(TypeTag<float>{});
    return go(TypeTag<double>{});
  });
}

cudaError_t launch_recon(const DeviceMesh& dm, const double* U, const float2* Us, void* Uq,
                         uint8_t* sel_out, const uint8_t* sel_in, cudaStream_t st) {
  if (dm.precision != TENO_FP64_NATIVE && !Us) return cudaErrorInvalidValue;
  ReconArgs a;
  a.ahat = dm.ahat;
  a.nbr = dm.nbr;
  a.smask = dm.smask;
  a.U = U;
  a.Us = Us;
  a.Uq = Uq;
  a.sel_out = sel_out;
  a.sel_in = sel_in;
  a.n_cell = dm.n_recon;  // the cells reconstructed (all cells, or a partition's compute set)
  a.n_pad = dm.n_pad;
  a.ct = dm.ct;
  a.eps = dm.eps;
  a.linear = dm.linear;
  a.e_entries = dm.e_entries;
  a.scheme = dm.scheme;
  a.cw_dK = 1.0 - 1.0 / dm.cweno_dk;
  a.coef_out = dm.charvar ? dm.coef_out : nullptr;
  a.force_near = dm.debug & 1;
  a.wait_polls = (dm.debug & 2) ? 0u : kWaitLimit;
  const int64_t tiles = (a.n_cell + kTile - 1) / kTile;
  return dispatch_order(dm.order, [&](auto Mc, auto NSc) -> cudaError_t {
    constexpr int M = decltype(Mc)::value, NS = decltype(NSc)::value;
    auto go = [&](auto nqc, auto nvc) -> cudaError_t {
      constexpr int NQ = decltype(nqc)::value, NV = decltype(nvc)::value;
      // variant 2 where every tile has its halo: the W form (Euler TENO in FP64
      // and pairs), the tile kernel (dm.tmat: TENO on the mixed path, scalar
      // too), and on Euler's mixed and pair paths the bulk-copy kernel of CWENO
      // and the characteristic mode.  What is left of variant 2 (scalar FP64
      // and pairs) takes the halo kernel, compiled for TENO in conservative
      // variables only, or the direct kernels.
      const bool ext = dm.scheme != 0 || dm.charvar != 0;
      if (dm.variant == 2 && dm.err_flag && dm.halo.off) {
        if (dm.tmat) return launch_recon_tile<M, NS, NQ, NV>(a, dm, st);
        if constexpr (NV == 4) {
          if (dm.wq && dm.psi_d)
            return launch_recon_tma_w<M, NS, NQ, double>(a, dm, dm.err_flag, st);
          if (dm.wq && dm.psi_df)
            return launch_recon_tma_w<M, NS, NQ, float2>(a, dm, dm.err_flag, st);
          if (ext && dm.precision == TENO_FP64) return launch_recon_tma<M, NS, NQ, true>(a, dm, st);
          if (ext && dm.precision == TENO_FP32_MIXED)
            return launch_recon_tma<M, NS, NQ, false>(a, dm, st);
        }
      }
      if (!ext && dm.variant != 1 && dm.halo.off) {
        constexpr int TZh = 4 / NV;
        dim3 block(kTile, NV, TZh);
        dim3 grid((unsigned)((tiles + TZh - 1) / TZh));
        if (dm.precision == TENO_FP64)
          launch(recon_halo_kernel<M, NS, NQ, NV, 0>, grid, block, 0, st, a, dm.halo, dm.eval_df);
        else if (dm.precision == TENO_FP32_MIXED)
          launch(recon_halo_kernel<M, NS, NQ, NV, 1>, grid, block, 0, st, a, dm.halo, dm.eval_df);
        else
          launch(recon_halo_kernel<M, NS, NQ, NV, 2>, grid, block, 0, st, a, dm.halo, dm.eval);
        return cudaGetLastError();
      }
      constexpr int TZ = 4 / NV;  // 128 threads per block
      dim3 block(kTile, NV, TZ);
      dim3 grid((unsigned)((tiles + TZ - 1) / TZ));
      if (dm.precision == TENO_FP64_NATIVE)
        launch(recon_kernel<M, NS, NQ, NV, double, EvalTable>, grid, block, 0, st, a, dm.eval);
      else if (dm.precision == TENO_FP64)
        launch(recon_df_kernel<M, NS, NQ, NV>, grid, block, 0, st, a, dm.eval_df);
      else
        launch(recon_kernel<M, NS, NQ, NV, float, DFTable>, grid, block, 0, st, a, dm.eval_df);
      return cudaGetLastError();
    };
    constexpr int NQd = (M <= 9) ? 2 : 3;
    if (dm.nq != NQd) return cudaErrorInvalidValue;
    if (dm.n_var == 1) return go(std::integral_constant<int, NQd>{}, std::integral_constant<int, 1>{});
    return go(std::integral_constant<int, NQd>{}, std::integral_constant<int, 4>{});
  });
}

// (hi, lo) float pair of a double, on the host
static float2 split2(double x) {
  const float h = (float)x;
  return make_float2(h, (float)(x - (double)h));
}

static FaceArgs face_args(const DeviceMesh& dm, double time) {
  FaceArgs a;
  a.f_cells = dm.f_cells;
  a.f_edges = dm.f_edges;
  a.f_geom = dm.f_geom;
  a.f_geom2 = dm.f_geom2;
  a.n_pad = dm.n_pad;
  a.n_face = dm.n_face;
  a.gamma = dm.gamma;
  a.adv_x = dm.adv_x;
  a.adv_y = dm.adv_y;
  a.adv_field = dm.adv_field;
  a.adv_cx = dm.adv_cx;
  a.adv_cy = dm.adv_cy;
  a.adv_omega = dm.adv_omega;
  a.adv_r1 = dm.adv_r1;
  a.adv_r2 = dm.adv_r2;
  a.time = time;
  for (int k = 0; k < kMaxNq; ++k) {
    a.gw[k] = dm.gw[k];
    a.gt[k] = dm.gt[k];
    a.gw2[k] = split2(dm.gw[k]);
  }
  a.g2 = split2(dm.gamma);
  a.gm12 = split2(dm.gamma - 1.0);
  return a;
}

cudaError_t launch_face_flux(const DeviceMesh& dm, const void* Uq, void* K, double time,
                             cudaStream_t st) {
  FaceArgs a = face_args(dm, time);
  const unsigned grid = (unsigned)((dm.n_face + kFluxFaces - 1) / kFluxFaces);
  auto go = [&](auto nvc, auto nqc, auto flc) -> cudaError_t {
    constexpr int NV = decltype(nvc)::value, NQ = decltype(nqc)::value,
                  FL = decltype(flc)::value;
    if (dm.precision == TENO_FP64_NATIVE)
      launch(face_flux_kernel<NV, NQ, FL, double>, grid, kFluxFaces * NQ, 0, st, a,
             (const double*)Uq, (double*)K);
    else if (dm.precision == TENO_FP64)
      launch(face_flux_kernel<NV, NQ, FL, DF>, grid, kFluxFaces * NQ, 0, st, a, (const DF*)Uq,
             (DF*)K);
    else
      launch(face_flux_kernel<NV, NQ, FL, float>, grid, kFluxFaces * NQ, 0, st, a, (const float*)Uq,
             (float*)K);
    return cudaGetLastError();
  };
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  using I3 = std::integral_constant<int, 3>;
  using I4 = std::integral_constant<int, 4>;
  using F0 = std::integral_constant<int, TENO_FLUX_UPWIND>;
  using F1 = std::integral_constant<int, TENO_FLUX_HLL>;
  using F2 = std::integral_constant<int, TENO_FLUX_HLLC>;
  if (dm.n_var == 1) return dm.nq == 2 ? go(I1{}, I2{}, F0{}) : go(I1{}, I3{}, F0{});
  if (dm.flux == TENO_FLUX_HLL) return dm.nq == 2 ? go(I4{}, I2{}, F1{}) : go(I4{}, I3{}, F1{});
  return dm.nq == 2 ? go(I4{}, I2{}, F2{}) : go(I4{}, I3{}, F2{});
}

cudaError_t launch_gather(const DeviceMesh& dm, const void* K, const double* Un, const double* Us,
                          double* out, int mode, double cn, double cs, double dt_fixed,
                          const double* max_lam, int* flag, float2* split, double* lam_next,
                          double* lam_zero, cudaStream_t st) {
  GatherArgs a{dm.c_faces, dm.inv_area, dm.n_update, dm.n_pad, dm.gamma};
  NextLam nl;
  nl.out = (unsigned long long*)lam_next;
  nl.zero = (unsigned long long*)lam_zero;
  nl.cfl_len = dm.cfl_len;
  nl.ilen2 = dm.cfl_ilen2;
  nl.cell_speed = dm.n_var == 1 ? dm.cell_speed : nullptr;
  nl.adv_speed = sqrt(dm.adv_x * dm.adv_x + dm.adv_y * dm.adv_y);
  nl.g2 = split2(dm.gamma);
  nl.gm12 = split2(dm.gamma - 1.0);
  const unsigned grid = (unsigned)((dm.n_update + 255) / 256);
  auto go = [&](auto nvc, auto tkc) {
    constexpr int NV = decltype(nvc)::value;
    using TK = typename decltype(tkc)::type;
    launch(lam_next ? gather_kernel<NV, TK, true> : gather_kernel<NV, TK, false>, grid, 256, 0, st,
           a, (const TK*)K, Un, Us, out, mode, cn, cs, dt_fixed, dm.cfl, max_lam, flag, split, nl);
  };
  using I1 = std::integral_constant<int, 1>;
  using I4 = std::integral_constant<int, 4>;
  const bool one = dm.n_var == 1;
  if (dm.precision == TENO_FP64_NATIVE) {
    if (one) go(I1{}, TypeTag<double>{}); else go(I4{}, TypeTag<double>{});
  } else if (dm.precision == TENO_FP64) {
    if (one) go(I1{}, TypeTag<DF>{}); else go(I4{}, TypeTag<DF>{});
  } else {
    if (one) go(I1{}, TypeTag<float>{}); else go(I4{}, TypeTag<float>{});
  }
  return cudaGetLastError();
}

cudaError_t launch_layer_fill(const DeviceMesh& dm, const double* U, void* Uq, cudaStream_t st) {
  if (!dm.fo_n) return cudaSuccess;
  const int64_t nt = dm.fo_n * 3 * dm.nq;
  const unsigned grid = (unsigned)((nt + 255) / 256);
  auto go = [&](auto nvc, auto nqc) {
    constexpr int NV = decltype(nvc)::value, NQ3 = 3 * decltype(nqc)::value;
    if (dm.precision == TENO_FP64)
      launch(layer_fill_kernel<NV, NQ3, DF>, grid, 256, 0, st, U, (DF*)Uq, dm.fo_list, dm.fo_n,
             dm.n_pad);
    else if (dm.precision == TENO_FP32_MIXED)
      launch(layer_fill_kernel<NV, NQ3, float>, grid, 256, 0, st, U, (float*)Uq, dm.fo_list,
             dm.fo_n, dm.n_pad);
    else
      launch(layer_fill_kernel<NV, NQ3, double>, grid, 256, 0, st, U, (double*)Uq, dm.fo_list,
             dm.fo_n, dm.n_pad);
  };
  using I1 = std::integral_constant<int, 1>;
  using I4 = std::integral_constant<int, 4>;
  using Q2 = std::integral_constant<int, 2>;
  using Q3 = std::integral_constant<int, 3>;
  if (dm.n_var == 1) {
    if (dm.nq == 2) go(I1{}, Q2{}); else go(I1{}, Q3{});
  } else {
    if (dm.nq == 2) go(I4{}, Q2{}); else go(I4{}, Q3{});
  }
  return cudaGetLastError();
}

cudaError_t launch_layer_vjp(const DeviceMesh& dm, double* Uq_bar, double* ubd, cudaStream_t st) {
  if (!dm.fo_n) return cudaSuccess;
  const unsigned grid = (unsigned)((dm.fo_n * 3 + 255) / 256);
  const bool pairs = dm.precision == TENO_FP64;
  auto go = [&](auto nvc, auto nqc) {
    constexpr int NV = decltype(nvc)::value, NQ = decltype(nqc)::value;
    if (pairs)
      launch(layer_vjp_kernel<NV, NQ, true>, grid, 256, 0, st, Uq_bar, ubd, dm.fo_list, dm.fo_n);
    else
      launch(layer_vjp_kernel<NV, NQ, false>, grid, 256, 0, st, Uq_bar, ubd, dm.fo_list, dm.fo_n);
  };
  using I1 = std::integral_constant<int, 1>;
  using I4 = std::integral_constant<int, 4>;
  using Q2 = std::integral_constant<int, 2>;
  using Q3 = std::integral_constant<int, 3>;
  if (dm.n_var == 1) {
    if (dm.nq == 2) go(I1{}, Q2{}); else go(I1{}, Q3{});
  } else {
    if (dm.nq == 2) go(I4{}, Q2{}); else go(I4{}, Q3{});
  }
  return cudaGetLastError();
}

cudaError_t launch_positivity(const DeviceMesh& dm, const double* U, void* Uq,
                              cudaStream_t st) {
  if (dm.n_var != 4) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)((dm.n_recon + 31) / 32);
  auto go = [&](auto nq, auto tq) -> cudaError_t {
    constexpr int NQ = decltype(nq)::value;
    using TQ = typename decltype(tq)::type;
    launch(positivity_kernel<NQ, TQ>, grid, 32 * 3 * NQ, 0, st, U, (TQ*)Uq, dm.n_recon, dm.n_pad,
           dm.gamma);
    return cudaGetLastError();
  };
  auto by_type = [&](auto nq) -> cudaError_t {
    if (dm.precision == TENO_FP64) return go(nq, TypeTag<DF>{});
    if (dm.precision == TENO_FP32_MIXED) return go(nq, TypeTag<float>{});
    return go(nq, TypeTag<double>{});
  };
  if (dm.nq == 2) return by_type(std::integral_constant<int, 2>{});
  if (dm.nq == 3) return by_type(std::integral_constant<int, 3>{});
  return cudaErrorInvalidValue;
}

cudaError_t launch_halo_pack(const double* U, int64_t ld, const int32_t* idx, int64_t n,
                             int n_var, double* buf, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  halo_pack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(U, ld, idx, n, n_var, buf);
  return cudaGetLastError();
}
cudaError_t launch_halo_unpack(double* U, int64_t ld, const int32_t* idx, int64_t n, int n_var,
                               const double* buf, float2* Us, int add, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  halo_unpack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(U, ld, idx, n, n_var, buf, Us,
                                                                 add);
  return cudaGetLastError();
}

cudaError_t launch_split(const DeviceMesh& dm, const double* U, float2* Us, cudaStream_t st) {
  launch(split_kernel, (unsigned)((dm.n_cell + 255) / 256), 256, 0, st, U, Us, dm.n_cell, dm.n_pad,
         dm.n_var);
  return cudaGetLastError();
}

cudaError_t launch_max_lambda(const DeviceMesh& dm, const double* U, double* max_lam,
                              cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(max_lam, 0, sizeof(double), st);
  if (e != cudaSuccess) return e;
  int64_t blocks = (dm.n_update + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  const double adv = sqrt(dm.adv_x * dm.adv_x + dm.adv_y * dm.adv_y);
  if (dm.n_var == 1)
    launch(max_lambda_kernel<1>, (unsigned)blocks, 256, 0, st, U, dm.cfl_len, dm.n_update, dm.n_pad,
           dm.gamma, adv, dm.cell_speed,
           (unsigned long long*)max_lam);
  else
    launch(max_lambda_kernel<4>, (unsigned)blocks, 256, 0, st, U, dm.cfl_len, dm.n_update, dm.n_pad,
           dm.gamma, adv, nullptr,
           (unsigned long long*)max_lam);
  return cudaGetLastError();
}

cudaError_t launch_max_lambda_split(const DeviceMesh& dm, const float2* Us, double* max_lam,
                                    cudaStream_t st) {
  if (dm.n_var != 4 || !dm.cfl_ilen2 || !Us) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(max_lam, 0, sizeof(double), st);
  if (e != cudaSuccess) return e;
  int64_t blocks = (dm.n_update + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  launch(max_lambda_split_kernel, (unsigned)blocks, 256, 0, st, Us, dm.cfl_ilen2, dm.n_update,
         dm.n_pad, split2(dm.gamma), split2(dm.gamma - 1.0),
         (unsigned long long*)max_lam);
  return cudaGetLastError();
}

cudaError_t launch_permute(const double* src, double* dst, const int32_t* perm, int64_t n,
                           int64_t ld_src, int64_t ld_dst, int n_var, int to_user,
                           cudaStream_t st) {
  dim3 grid((unsigned)((n + 255) / 256), n_var);
  launch(permute_kernel, grid, 256, 0, st, src, dst, perm, n, ld_src, ld_dst, to_user);
  return cudaGetLastError();
}

cudaError_t launch_permute_u8(const uint8_t* src, uint8_t* dst, const int32_t* perm, int64_t n,
                              int64_t ld_src, int64_t ld_dst, int n_var, int to_user,
                              cudaStream_t st) {
  dim3 grid((unsigned)((n + 255) / 256), n_var);
  launch(permute_u8_kernel, grid, 256, 0, st, src, dst, perm, n, ld_src, ld_dst, to_user);
  return cudaGetLastError();
}

cudaError_t launch_axpby(double* out, const double* a, double ca, const double* b, double cb,
                         int64_t n, cudaStream_t st) {
  launch(axpby_kernel, (unsigned)((n + 255) / 256), 256, 0, st, out, a, ca, b, cb, n);
  return cudaGetLastError();
}

#ifndef TENO_VJP_DIRS
#define TENO_VJP_DIRS 2
#endif
constexpr int kVjpDirs = TENO_VJP_DIRS;

cudaError_t launch_face_flux_vjp(const DeviceMesh& dm, const void* Uq, const double* w,
                                 double* Uq_bar, double time, cudaStream_t st) {
  VjpArgs a;
  a.f_cells = dm.f_cells;
  a.f_edges = dm.f_edges;
  a.f_geom = dm.f_geom;
  a.f_geom2 = dm.f_geom2;
  a.g2 = split2(dm.gamma);
  a.gm12 = split2(dm.gamma - 1.0);
  a.inv_area = dm.inv_area;
  a.n_face = dm.n_face;
  a.n_pad = dm.n_pad;
  a.gamma = dm.gamma;
  a.adv_x = dm.adv_x;
  a.adv_y = dm.adv_y;
  a.adv_field = dm.adv_field;
  a.adv_cx = dm.adv_cx;
  a.adv_cy = dm.adv_cy;
  a.adv_omega = dm.adv_omega;
  a.adv_r1 = dm.adv_r1;
  a.adv_r2 = dm.adv_r2;
  a.time = time;
  for (int k = 0; k < kMaxNq; ++k) {
    a.gw[k] = dm.gw[k];
    a.gt[k] = dm.gt[k];
    a.gw2[k] = split2(dm.gw[k]);
  }
  const unsigned grid = (unsigned)((dm.n_face + kFluxFaces - 1) / kFluxFaces);
  auto go = [&](auto nvc, auto nqc, auto flc, auto tqc) {
    constexpr int NV = decltype(nvc)::value, NQ = decltype(nqc)::value,
                  FL = decltype(flc)::value;
    using TQ = typename decltype(tqc)::type;
    // pairs: FP32-pipe dual numbers, kVjpDirs directions per pass; FP64:
    // all 2 NV directions of an interior face in one pass
    if constexpr (std::is_same<TQ, DF>::value) {
      constexpr int ND = NV < kVjpDirs ? NV : kVjpDirs;
      if constexpr (NV == 4 && FL == TENO_FLUX_HLL)
        if (dm.n_face >= kTurnFaces) {
          launch(face_flux_vjp_kernel<NV, NQ, FL, TQ, DF, ND, true>,
                 (unsigned)((dm.n_face + kTurnBlock - 1) / kTurnBlock), kTurnBlock, 0, st, a,
                 (const TQ*)Uq, w, Uq_bar);
          return;
        }
      launch(face_flux_vjp_kernel<NV, NQ, FL, TQ, DF, ND, false>, grid, kFluxFaces * NQ, 0, st, a,
             (const TQ*)Uq, w, Uq_bar);
    } else {
      launch(face_flux_vjp_kernel<NV, NQ, FL, TQ, double, 2 * NV, false>, grid, kFluxFaces * NQ, 0,
             st, a, (const TQ*)Uq, w, Uq_bar);
    }
  };
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  using I3 = std::integral_constant<int, 3>;
  using I4 = std::integral_constant<int, 4>;
  using F0 = std::integral_constant<int, TENO_FLUX_UPWIND>;
  using F1 = std::integral_constant<int, TENO_FLUX_HLL>;
  using F2 = std::integral_constant<int, TENO_FLUX_HLLC>;
  auto pick = [&](auto tqc) {
    if (dm.n_var == 1) {
      if (dm.nq == 2) go(I1{}, I2{}, F0{}, tqc); else go(I1{}, I3{}, F0{}, tqc);
    } else if (dm.flux == TENO_FLUX_HLL) {
      if (dm.nq == 2) go(I4{}, I2{}, F1{}, tqc); else go(I4{}, I3{}, F1{}, tqc);
    } else {
      if (dm.nq == 2) go(I4{}, I2{}, F2{}, tqc); else go(I4{}, I3{}, F2{}, tqc);
    }
  };
  if (dm.precision == TENO_FP64)
    pick(TypeTag<DF>{});
  else
    pick(TypeTag<double>{});
  return cudaGetLastError();
}

cudaError_t launch_recon_vjp(const DeviceMesh& dm, const uint8_t* sel, const double* Uq_bar,
                             double* d_bar, double* u_self, cudaStream_t st) {
  const int64_t tiles = (dm.n_recon + kTile - 1) / kTile;
  return dispatch_order(dm.order, [&](auto Mc, auto NSc) -> cudaError_t {
    constexpr int M = decltype(Mc)::value, NS = decltype(NSc)::value;
    constexpr int NQ = (M <= 9) ? 2 : 3;
    if (dm.nq != NQ) return cudaErrorInvalidValue;
    auto go = [&](auto nvc, auto tsc) {
      constexpr int NV = decltype(nvc)::value;
      using TS = typename decltype(tsc)::type;
      constexpr int TZ = 4 / NV;
      dim3 block(kTile, NV, TZ);
      const unsigned grid = (unsigned)((tiles + TZ - 1) / TZ);
      if constexpr (std::is_same<TS, float2>::value)
        launch(recon_vjp_df_kernel<M, NS, NQ, NV>, grid, block, 0, st, (const float2*)dm.ahat, sel,
               Uq_bar, (DF*)d_bar, u_self, dm.n_recon, dm.n_pad,
               dm.eval_df);
      else
        launch(recon_vjp_kernel<M, NS, NQ, NV, TS>, grid, block, 0, st, (const TS*)dm.ahat, sel,
               Uq_bar, d_bar, u_self, dm.n_recon, dm.n_pad, dm.eval);
    };
    using I1 = std::integral_constant<int, 1>;
    using I4 = std::integral_constant<int, 4>;
    if (dm.precision == TENO_FP64) {
      if (dm.n_var == 1) go(I1{}, TypeTag<float2>{});
      else go(I4{}, TypeTag<float2>{});
    } else {
      if (dm.n_var == 1) go(I1{}, TypeTag<double>{});
      else go(I4{}, TypeTag<double>{});
    }
    return cudaGetLastError();
  });
}

template <int M, int NS, int NQ>
cudaError_t launch_recon_vjp_tma_t(const DeviceMesh& dm, const uint8_t* sel, const double* Uq_bar,
                                   float2* part, double* u_self, cudaStream_t st) {
  using VP = VjpPlan<M, NS, 3 * NQ>;
  auto kern = recon_vjp_tma_kernel<M, NS, NQ>;
  const int threads = kTile * (kConsumers + 1);
  unsigned grid = 0;
  const cudaError_t e =
      resident_grid(kern, threads, VP::kSmem, (dm.n_recon + kTile - 1) / kTile, &grid);
  if (e != cudaSuccess) return e;
  launch(kern, grid, threads, VP::kSmem, st, (const float2*)dm.ahat, dm.wq, dm.wstat, dm.halo, sel,
         Uq_bar, part, u_self, dm.n_recon, dm.n_pad, dm.eval_df, dm.err_flag);
  return cudaGetLastError();
}

cudaError_t launch_recon_vjp_tma(const DeviceMesh& dm, const uint8_t* sel, const double* Uq_bar,
                                 double* part, double* u_self, cudaStream_t st) {
  if (dm.precision != TENO_FP64 || dm.n_var != 4 || !dm.halo.off || !dm.wq || !dm.err_flag)
    return cudaErrorInvalidValue;
  return dispatch_order(dm.order, [&](auto Mc, auto NSc) -> cudaError_t {
    constexpr int M = decltype(Mc)::value, NS = decltype(NSc)::value;
    constexpr int NQ = (M <= 9) ? 2 : 3;
    if (dm.nq != NQ) return cudaErrorInvalidValue;
    return launch_recon_vjp_tma_t<M, NS, NQ>(dm, sel, Uq_bar, reinterpret_cast<float2*>(part),
                                             u_self, st);
  });
}

cudaError_t launch_scatter_gather(const DeviceMesh& dm, const int64_t* rev_off,
                                  const int32_t* rev_idx, const double* d_bar,
                                  const double* u_self, double* v, const double* ubd,
                                  cudaStream_t st) {
  const unsigned grid = (unsigned)((dm.n_cell + 255) / 256);
  const bool pairs = dm.precision == TENO_FP64;  // d_bar holds (hi, lo) pairs
  if (dm.n_var == 1) {
    if (pairs)
      launch(scatter_gather_kernel<1, DF>, grid, 256, 0, st, rev_off, rev_idx, (const DF*)d_bar,
             u_self, v, dm.n_cell, dm.n_pad, ubd);
    else
      launch(scatter_gather_kernel<1, double>, grid, 256, 0, st, rev_off, rev_idx, d_bar, u_self, v,
             dm.n_cell, dm.n_pad, ubd);
  } else {
    if (pairs)
      launch(scatter_gather_kernel<4, DF>, grid, 256, 0, st, rev_off, rev_idx, (const DF*)d_bar,
             u_self, v, dm.n_cell, dm.n_pad, ubd);
    else
      launch(scatter_gather_kernel<4, double>, grid, 256, 0, st, rev_off, rev_idx, d_bar, u_self, v,
             dm.n_cell, dm.n_pad, ubd);
  }
  return cudaGetLastError();
}
}  // namespace teno
