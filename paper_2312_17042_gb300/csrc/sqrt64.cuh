// sqrt64.cuh -- the square root of the FP64 flux.
//
// sqrt(x) takes 9 slots of the FP64 pipe, which bounds the flux; a coupled iteration on g ~ sqrt(x) and
// h ~ 1 / (2 sqrt(x)) (Goldschmidt) from the hardware estimate and the residual correction g + (x - g^2) h take 6.
// With four roots a face point: 145.4 against 152.4 us for the flux at 131 072 triangles, 87.5 against 90.8 us at
// 24 576 tetrahedra. The estimate's error squares twice, so that the result is the correctly rounded root
// unless the exact one is within some 2^-27 of a unit of the midpoint between two numbers.
// The residual needs x far enough above the subnormal numbers to be exact: from 2^-959 on; below, and for zeros,
// negative, infinite and NaN arguments, sqrt itself, behind a branch inside the assembly: one that the compiler sees
// changes which products of the callers become fused multiply-adds, hence their last places (a 200-step shock tube
// then moved by 5e-12); the instruction under a predicate instead of the branch took 168.8 us.
#pragma once

namespace cteno {

__device__ __forceinline__ double sqrt64(const double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double g = x * y, h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));  // y / 2
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  g = fma(fma(-g, g, x), h, g);
  asm("{\n\t.reg .pred p;\n\t"
      "setp.lt.u32 p, %2, %3;\n\t"
      "@p bra done;\n\t"
      "sqrt.rn.f64 %0, %1;\n"
      "done:\n\t}"
      : "+d"(g)
      : "d"(x), "r"(__double2hiint(x) - (64 << 20)), "n"((0x7FF - 64) << 20));
  return g;
}

}  // namespace cteno
