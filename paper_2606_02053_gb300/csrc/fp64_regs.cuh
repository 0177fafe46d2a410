// FP64 arithmetic as three-register multiply-adds.
//
// GB300's FP64 pipe takes a multiply-add whose three operands are registers in
// 16 cycles per warp and SM, and a multiply, an add, or a multiply-add with a
// constant or immediate operand in 19 (measured: 2.00 against 1.68 results per
// clock and SM, with one warp per scheduler or many).  fma(a, b, -0) is a b and
// fma(a, 1, b) is a + b, both exactly and with the same rounding; the constants
// have to sit in registers, so they are loaded from memory, where the compiler
// cannot see their values and turn the multiply-adds back.
#pragma once

struct Fp64Regs {
  double nz, one, two, half;  // -0, 1, 2, 1/2
};

namespace cosmos {

static __device__ const double fp64_constants[4] = {-0.0, 1.0, 2.0, 0.5};

__device__ __forceinline__ Fp64Regs fp64_regs() {
  Fp64Regs k;
  asm volatile("ld.volatile.global.f64 %0, [%1];" : "=d"(k.nz) : "l"(fp64_constants));
  asm volatile("ld.volatile.global.f64 %0, [%1];" : "=d"(k.one) : "l"(fp64_constants + 1));
  asm volatile("ld.volatile.global.f64 %0, [%1];" : "=d"(k.two) : "l"(fp64_constants + 2));
  asm volatile("ld.volatile.global.f64 %0, [%1];" : "=d"(k.half) : "l"(fp64_constants + 3));
  return k;
}

__device__ __forceinline__ double mul3(double a, double b, const Fp64Regs& k) { return fma(a, b, k.nz); }
__device__ __forceinline__ double add3(double a, double b, const Fp64Regs& k) { return fma(a, k.one, b); }
__device__ __forceinline__ double sub3(double a, double b, const Fp64Regs& k) { return fma(-b, k.one, a); }

}  // namespace cosmos
