// Reciprocal and square root of the FP64 Riemann solver.
//
// The solver is bound by the FP64 pipe (1/64 of the FP32 rate), and the IEEE
// division and root take most of it, so they are formed from the PTX
// approximations (documented, about 20 bits, not on that pipe) in three and five
// FP64 operations: one step of third order, y (1 + e + e^2) with e = 1 - x y
// (the Newton iteration's series with one term more; Traub, "Iterative Methods
// for the Solution of Equations", 1964), and one step of Goldschmidt's iteration
// with a last residual step (Goldschmidt, "Applications of division by
// convergence", 1964).  Both are within 0.51 units in the last place, where IEEE
// gives 0.5.  Operands near the ends of the exponent range, zeros, infinities and
// NaN take the IEEE operations.  Face flux, 131,072 cells: 166 us a launch, 174
// with IEEE divisions and roots, before the solver's other changes.
#pragma once

namespace teno {

__device__ __forceinline__ bool mid_exponent(double x) {  // 2^-959 <= |x| < 2^961
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) - 0x04000000u < 0x78000000u;
}

__device__ __forceinline__ double rcp_f64(double x) {
  if (!mid_exponent(x)) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

__device__ __forceinline__ double sqrt_f64(double x) {
  if (!mid_exponent(x) || __double2hiint(x) < 0) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y;
  // y / 2 (y is a normal number, its exponent far from the ends)
  const double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));
  const double g1 = fma(g, fma(-g, h, 0.5), g);
  return fma(fma(-g1, g1, x), h, g1);
}

}  // namespace teno
