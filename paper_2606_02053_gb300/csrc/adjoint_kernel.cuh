// Reverse mode (vector-Jacobian product) of the right-hand side F(U):
//   v = (dF/dU)^T w
// F(U)(p) = A(inputs at p) + KO(U)(p) - sum_d (H_d(p) - H_d(p - e_d)) / h_d,
// the inputs being U(p) and finite differences of U around p.  On a periodic
// grid the centred stencils transpose to D_d^T = -D_d, D_dd^T = D_dd,
// (D_a D_b)^T = D_a D_b and KO^T = KO, so
//   v_f = abar_f - sum_d D_d(dbar_{f,d}) + sum_ab D_ab(ddbar_{f,ab}) + KO(w_f) + (fluid terms)
// with (abar, dbar, ddbar) the cotangents of the algebra inputs (pass 1, the
// generated reverse of the pointwise algebra) and the fluid terms from the
// reverse of the face fluxes and of the primitive recovery.
#pragma once

#include "stage_kernel.cuh"

namespace cosmos {

struct VjpArgs {
  DevGrid g;
  Coef c;
  AlgebraParams ap;
  FluidParams fp;
  const double* __restrict__ U;     // linearisation point
  const double* __restrict__ prim;  // primitives at U (fluid)
  const double* __restrict__ W;     // cotangent of F(U) (state layout)
  const double* __restrict__ D;     // derivative-pass output at U (KO slots unused)
  double* CB;                       // [NIN][pts] input cotangents (pass 1)
  double* FC;                       // [3][34][pts] face-input cotangents (fluid)
  double* VF;                       // [nf][pts] fluid contributions to v (fluid)
  // pass 2 outputs:  lam += v;  knext = a_lam * lam0 + a_v * v  (knext optional)
  const double* __restrict__ lam0;
  double* lam;
  double* knext;
  double a_lam, a_v;
};

// Inputs of the reverse algebra at one point: the forward inputs (state,
// derivative buffer, fluid density) followed by the cotangents W of the
// outputs, each read from global memory where the generated code uses it.
template <class T>
struct VjpIn {
  const VjpArgs& a;
  long fs, c;
  __device__ __forceinline__ double operator[](int k) const {
    constexpr int NDER0 = 3 * T::ND1 + 6 * T::ND2;
    if (k < T::NF) return ldg(a.U + (long)k * fs, c);
    if (k < T::NF + NDER0) return ldg(a.D + (long)(k - T::NF) * fs, c);
    if (k < T::NIN) return ldg(a.prim, c);
    return ldg(a.W + (long)(k - T::NIN) * fs, c);
  }
};

// Input cotangents, stored to CB as soon as the generated code has each one.
struct VjpOut {
  double* CB;
  long fs, c;
  struct Slot {
    double* p;
    __device__ __forceinline__ void operator=(double v) const { *p = v; }
  };
  __device__ __forceinline__ Slot operator[](int m) const { return Slot{CB + (long)m * fs + c}; }
};

// Threads per block of the kernels below: short blocks spread a small grid evenly over the SMs,
// 41580 points being 2.1 blocks of 128 per SM, where an SM with three takes half as long again.  VJP of 45 x 33 x
// 28: blocks of 128 471 us, of 64 429, of 32 410; reverse step of 96^3: 38.56, 38.44, 38.50 ms.
constexpr int VJP_THREADS = 32;

#ifndef COSMOS_VJP_MIN_BLOCKS
// reverse algebra: the registers are sized for 3 x 128 resident threads per SM (12 of its blocks of VJP_THREADS)
#define COSMOS_VJP_MIN_BLOCKS 3
#endif

template <class T>
__global__ void __launch_bounds__(BX* BY, COSMOS_VJP_MIN_BLOCKS) vjp_pass1_kernel(const VjpArgs a) {
  int i, j, k;
  if (!point_of<true>(a.g, i, j, k)) return;
  const long fs = a.g.fstride;
  const long c = ((long)k * a.g.ny + j) * a.g.pitch + i;
  const VjpIn<T> in{a, fs, c};
  VjpOut out{a.CB, fs, c};
  T::rhs_vjp(in, out, a.ap, fp64_regs());
}

// Face-flux reverse: H_d(p) enters F at p (-1/h) and at p + e_d (+1/h).
template <int D>
__device__ __forceinline__ void face_vjp(const VjpArgs& a, const Nbr& n, const Fp64Regs& kr) {
  const long fs = a.g.fstride;
  double in[34 + 4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const long off = disp<D>(n, o - 1);
#pragma unroll
    for (int m = 0; m < 4; ++m) in[4 * o + m] = ldg(a.prim + m * fs, off);
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const long off = disp<D>(n, s);
    double* q = in + 16 + 9 * s;
    q[0] = ldg(a.U, off);
    q[1] = ldg(a.U + 17 * fs, off);
    q[2] = ldg(a.U + (18 + D) * fs, off);
#pragma unroll
    for (int m = 0; m < 6; ++m) q[3 + m] = ldg(a.U + (1 + m) * fs, off);
  }
  const long up = disp<D>(n, 1);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const double* Wm = a.W + (long)(24 + m) * fs;
    in[34 + m] = (ldg(Wm, up) - ldg(Wm, n.c)) * a.c.ih[D];
  }
  double out[34];
  if (D == 0) fluid_face_flux_0_vjp(in, out, a.fp, kr);
  if (D == 1) fluid_face_flux_1_vjp(in, out, a.fp, kr);
  if (D == 2) fluid_face_flux_2_vjp(in, out, a.fp, kr);
#pragma unroll
  for (int m = 0; m < 34; ++m) a.FC[(long)(34 * D + m) * fs + n.c] = out[m];
}

static __global__ void __launch_bounds__(BX* BY) vjp_face_kernel(const VjpArgs a) {
  int i, j, k;
  if (!point_of<true>(a.g, i, j, k)) return;
  const Nbr n = make_nbr(a.g, i, j, k);
  const Fp64Regs kr = fp64_regs();
  face_vjp<0>(a, n, kr);
  face_vjp<1>(a, n, kr);
  face_vjp<2>(a, n, kr);
}

// Per cell: gather the face-input cotangents that refer to this cell, add the
// algebra's d/d rho, run the reverse of the primitive recovery, and store the
// fluid contributions to v (chi, gt, alpha, beta, tau, S) in VF.
template <int D>
__device__ __forceinline__ void gather_face_cot(const VjpArgs& a, const Nbr& n, double qb[4], double mb[9]) {
  const long fs = a.g.fstride;
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const long off = disp<D>(n, 1 - o);  // face p = c - (o - 1) e_d sees cell c as its input o
#pragma unroll
    for (int m = 0; m < 4; ++m) qb[m] += ldg(a.FC + (long)(34 * D + 4 * o + m) * fs, off);
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const long off = disp<D>(n, -s);  // face p = c - s e_d sees cell c as its metric side s
#pragma unroll
    for (int m = 0; m < 9; ++m) mb[m] += ldg(a.FC + (long)(34 * D + 16 + 9 * s + m) * fs, off);
  }
}

template <class T>
__global__ void __launch_bounds__(BX* BY) vjp_cell_kernel(const VjpArgs a) {
  int i, j, k;
  if (!point_of<true>(a.g, i, j, k)) return;
  const Nbr n = make_nbr(a.g, i, j, k);
  const long fs = a.g.fstride;
  double qb[4] = {ldg(a.CB + (long)(T::NIN - 1) * fs, n.c), 0.0, 0.0, 0.0};  // d/d rho from the algebra
  double mb[3][9];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int m = 0; m < 9; ++m) mb[d][m] = 0.0;
  gather_face_cot<0>(a, n, qb, mb[0]);
  gather_face_cot<1>(a, n, qb, mb[1]);
  gather_face_cot<2>(a, n, qb, mb[2]);
  double in[11 + 4];
  in[0] = ldg(a.U, n.c);
#pragma unroll
  for (int m = 0; m < 6; ++m) in[1 + m] = ldg(a.U + (1 + m) * fs, n.c);
#pragma unroll
  for (int m = 0; m < 4; ++m) in[7 + m] = ldg(a.U + (24 + m) * fs, n.c);
#pragma unroll
  for (int m = 0; m < 4; ++m) in[11 + m] = qb[m];
  double pb[11];
  fluid_prim_vjp(in, pb, a.fp, fp64_regs());
  double vf[T::NF];
#pragma unroll
  for (int f = 0; f < T::NF; ++f) vf[f] = 0.0;
  vf[0] = pb[0] + mb[0][0] + mb[1][0] + mb[2][0];
#pragma unroll
  for (int m = 0; m < 6; ++m) vf[1 + m] = pb[1 + m] + mb[0][3 + m] + mb[1][3 + m] + mb[2][3 + m];
  vf[17] = mb[0][1] + mb[1][1] + mb[2][1];
#pragma unroll
  for (int d = 0; d < 3; ++d) vf[18 + d] = mb[d][2];
#pragma unroll
  for (int m = 0; m < 4; ++m) vf[24 + m] = pb[7 + m];
#pragma unroll
  for (int f = 0; f < T::NF; ++f) a.VF[(long)f * fs + n.c] = vf[f];
}

// Stencils of the reverse sweep, in three-register multiply-adds (fp64_regs.cuh)
// with the coefficients in registers.
struct RevCoef {
  double d1a[3], d1b[3], d2a[3], d2b[3];
  Fp64Regs k;
};

// The coefficients through shared memory: read from there they are registers
// for the compiler, read from the kernel's arguments they become constant operands.
__device__ __forceinline__ RevCoef rev_coef(const Coef& c, double (&s)[12]) {
  const int t = threadIdx.y * blockDim.x + threadIdx.x;
  if (t == 0) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      s[d] = c.d1a[d];
      s[3 + d] = c.d1b[d];
      s[6 + d] = c.d2a[d];
      s[9 + d] = c.d2b[d];
    }
  }
  __syncthreads();
  RevCoef r;
  const volatile double* v = s;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    r.d1a[d] = v[d];
    r.d1b[d] = v[3 + d];
    r.d2a[d] = v[6 + d];
    r.d2b[d] = v[9 + d];
  }
  r.k = fp64_regs();
  return r;
}

// v - D_d F
template <int D>
__device__ __forceinline__ double sub_d1(double v, const double* __restrict__ F, const Nbr& n, const RevCoef& c) {
  const double a = sub3(ldg(F, disp<D>(n, 1)), ldg(F, disp<D>(n, -1)), c.k);
  const double b = sub3(ldg(F, disp<D>(n, 2)), ldg(F, disp<D>(n, -2)), c.k);
  return fma(-c.d1a[D], a, fma(c.d1b[D], b, v));
}

// v + D_dd F
template <int D>
__device__ __forceinline__ double add_d2(double v, const double* __restrict__ F, const Nbr& n, const RevCoef& c) {
  const double f0 = ldg(F, n.c);
  const double s1 = add3(sub3(ldg(F, disp<D>(n, 1)), f0, c.k), sub3(ldg(F, disp<D>(n, -1)), f0, c.k), c.k);
  const double s2 = add3(sub3(ldg(F, disp<D>(n, 2)), f0, c.k), sub3(ldg(F, disp<D>(n, -2)), f0, c.k), c.k);
  return fma(c.d2a[D], s1, fma(-c.d2b[D], s2, v));
}

// First half of the transposed mixed stencils.  With the second-derivative
// cotangents c_ab of a field and its first-derivative ones d_a,
//   -D_x d_x + D_x D_y c_xy + D_x D_z c_xz = -D_x (d_x - D_y c_xy - D_z c_xz),
//   -D_y d_y + D_y D_z c_yz = -D_y (d_y - D_z c_yz):
// the brackets replace d_x and d_y here, three first derivatives per field instead of
// three 16-point stencils in the second half (FP64-bound: 250 against 720 operations
// per point for the 11 fields).
template <class T>
__global__ void __launch_bounds__(BX* BY) vjp_fold_kernel(const VjpArgs a) {
  __shared__ double cf[12];
  const RevCoef c = rev_coef(a.c, cf);
  int i, j, k;
  if (!point_of<true>(a.g, i, j, k)) return;
  const Nbr n = make_nbr(a.g, i, j, k);
  const long fs = a.g.fstride;
#pragma unroll 1
  for (int m2 = 0; m2 < T::ND2; ++m2) {
    double* d = a.CB + (long)(T::NF + 3 * T::d1_slot(T::d2_field(m2))) * fs;
    const double* C = a.CB + (long)(T::NF + 3 * T::ND1 + 6 * m2) * fs;
    d[n.c] = sub_d1<1>(sub_d1<2>(d[n.c], C + 2 * fs, n, c), C + fs, n, c);
    d[fs + n.c] = sub_d1<2>(d[fs + n.c], C + 4 * fs, n, c);
  }
}

// Transposed stencils + RK4 reverse-sweep accumulation, one field at a time
// (each v_f depends on the cotangents of field f only), after vjp_fold_kernel.
template <class T>
__global__ void __launch_bounds__(BX* BY, 3) vjp_pass2_kernel(const VjpArgs a) {
  __shared__ double cf[12];
  const RevCoef c = rev_coef(a.c, cf);
  int i, j, k;
  if (!point_of<true>(a.g, i, j, k)) return;
  const Nbr n = make_nbr(a.g, i, j, k);
  const long fs = a.g.fstride;
  const bool ko_equal = a.c.ko[0] == a.c.ko[1] && a.c.ko[1] == a.c.ko[2];
#pragma unroll 1
  for (int f = 0; f < T::NF; ++f) {
    double v = ldg(a.CB + (long)f * fs, n.c);
    const int m = T::d1_slot(f);
    if (m >= 0) {
      const double* G = a.CB + (long)(T::NF + 3 * m) * fs;
      v = sub_d1<2>(sub_d1<1>(sub_d1<0>(v, G, n, c), G + fs, n, c), G + 2 * fs, n, c);
    }
    const int m2 = T::d2_slot(f);
    if (m2 >= 0) {
      const double* G = a.CB + (long)(T::NF + 3 * T::ND1 + 6 * m2) * fs;
      v = add_d2<2>(add_d2<1>(add_d2<0>(v, G, n, c), G + 3 * fs, n, c), G + 5 * fs, n, c);
    }
    if (!(T::FLUID && f >= 24 && f < 28)) {  // KO is symmetric: KO^T w = KO w
      const double* Wf = a.W + (long)f * fs;
      v = ko_equal ? ko_add_uniform(Wf, n, a.c, ldg(Wf, n.c), v, c.k) : ko_add(Wf, n, a.c, ldg(Wf, n.c), v);
    }
    if constexpr (T::FLUID) v = add3(v, ldg(a.VF + (long)f * fs, n.c), c.k);
    const long o = (long)f * fs + n.c;
    a.lam[o] += v;
    if (a.knext) a.knext[o] = a.a_lam * ldg(a.lam0, o) + a.a_v * v;
  }
}

// Gather traits for the vacuum layout (used by the initial-data reverse).
struct T_vac_adj {
  static constexpr int NF = alg_vac::NF, ND1 = alg_vac::ND1, ND2 = alg_vac::ND2, NIN = alg_vac::NIN;
  static constexpr bool FLUID = false, SCALAR = false;
  __device__ static constexpr int d1_field(int m) { return alg_vac::d1_field(m); }
  __device__ static constexpr int d2_field(int m) { return alg_vac::d2_field(m); }
};

#define COSMOS_DEFINE_ADJOINT(NAME, IS_FLUID)                                                                     \
  struct A_##NAME {                                                                                             \
    static constexpr int NF = alg_##NAME::NF, ND1 = alg_##NAME::ND1, ND2 = alg_##NAME::ND2,                     \
                         NIN = alg_##NAME::NIN;                                                                 \
    static constexpr bool FLUID = IS_FLUID, SCALAR = false;                                                     \
    __device__ static constexpr int d1_field(int m) { return alg_##NAME::d1_field(m); }                        \
    __device__ static constexpr int d2_field(int m) { return alg_##NAME::d2_field(m); }                        \
    __device__ static constexpr int d1_slot(int f) { return alg_##NAME::d1_slot(f); }                          \
    __device__ static constexpr int d2_slot(int f) { return alg_##NAME::d2_slot(f); }                          \
    template <class In, class Out>                                                                              \
    __device__ static __forceinline__ void rhs_vjp(const In& in, Out&& out, const AlgebraParams& p,             \
                                                   const Fp64Regs& k) {                                         \
      alg_##NAME::rhs_vjp(in, out, p, k);                                                                       \
    }                                                                                                           \
  };                                                                                                            \
  cudaError_t launch_vjp_##NAME(const VjpArgs& a, cudaStream_t s) {                                             \
    constexpr int block = VJP_THREADS;                                                                          \
    const unsigned grid = flat_grid(a.g, block);                                                                \
    vjp_pass1_kernel<A_##NAME><<<grid, block, 0, s>>>(a);                                                       \
    cudaError_t e = cudaGetLastError();                                                                         \
    if (e != cudaSuccess) return e;                                                                             \
    if (IS_FLUID) {                                                                                             \
      vjp_face_kernel<<<grid, block, 0, s>>>(a);                                                                \
      if ((e = cudaGetLastError()) != cudaSuccess) return e;                                                    \
      vjp_cell_kernel<A_##NAME><<<grid, block, 0, s>>>(a);                                                      \
      if ((e = cudaGetLastError()) != cudaSuccess) return e;                                                    \
    }                                                                                                           \
    vjp_fold_kernel<A_##NAME><<<grid, block, 0, s>>>(a);                                                        \
    if ((e = cudaGetLastError()) != cudaSuccess) return e;                                                      \
    vjp_pass2_kernel<A_##NAME><<<grid, block, 0, s>>>(a);                                                       \
    return cudaGetLastError();                                                                                  \
  }

}  // namespace cosmos
