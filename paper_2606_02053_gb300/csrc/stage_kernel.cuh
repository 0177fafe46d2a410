// Point-wise stencils in FP64 and the kernels that use them: the constraints
// (constraint_kernel), and the per-variant launchers (COSMOS_DEFINE_VARIANT).
// The right-hand side with its RK4 stage combine is stage_split.cuh, on the
// exact integer differences of stage_int.cuh.
//
// Every stencil is written so that its large cancellations happen in exact
// neighbour differences.
#pragma once

#include "common.cuh"

namespace cosmos {

template <int D>
__device__ __forceinline__ long disp(const Nbr& n, int o) {
  if (D == 0) return n.z[3] + n.y[3] + n.x[o + 3];
  if (D == 1) return n.z[3] + n.y[o + 3] + n.x[3];
  return n.z[o + 3] + n.y[3] + n.x[3];
}

template <int A, int B>
__device__ __forceinline__ long disp2(const Nbr& n, int oa, int ob) {
  int o[3] = {0, 0, 0};
  o[A] = oa;
  o[B] = ob;
  return n.z[o[2] + 3] + n.y[o[1] + 3] + n.x[o[0] + 3];
}

// D_d f = a (f+1 - f-1) - b (f+2 - f-2)
template <int D>
__device__ __forceinline__ double fd1(const double* __restrict__ F, const Nbr& n, const Coef& c) {
  const double a = ldg(F, disp<D>(n, 1)) - ldg(F, disp<D>(n, -1));
  const double b = ldg(F, disp<D>(n, 2)) - ldg(F, disp<D>(n, -2));
  return a * c.d1a[D] - b * c.d1b[D];
}

// D_dd f = a ((f+1 - f0) + (f-1 - f0)) - b ((f+2 - f0) + (f-2 - f0))
template <int D>
__device__ __forceinline__ double fd2(const double* __restrict__ F, const Nbr& n, const Coef& c, double f0) {
  const double s1 = (ldg(F, disp<D>(n, 1)) - f0) + (ldg(F, disp<D>(n, -1)) - f0);
  const double s2 = (ldg(F, disp<D>(n, 2)) - f0) + (ldg(F, disp<D>(n, -2)) - f0);
  return s1 * c.d2a[D] - s2 * c.d2b[D];
}

// D_A D_B f = [64 Q11 - 8 (Q12 + Q21) + Q22] / (144 h_A h_B),
// Q_pq = (f(p, q) - f(-p, q)) - (f(p, -q) - f(-p, -q))  (the 16-point product stencil)
template <int A, int B>
__device__ __forceinline__ double fdmix(const double* __restrict__ F, const Nbr& n, double cm) {
  double q[2][2];
#pragma unroll
  for (int p = 1; p <= 2; ++p)
#pragma unroll
    for (int r = 1; r <= 2; ++r) {
      const double u = ldg(F, disp2<A, B>(n, p, r)) - ldg(F, disp2<A, B>(n, -p, r));
      const double v = ldg(F, disp2<A, B>(n, p, -r)) - ldg(F, disp2<A, B>(n, -p, -r));
      q[p - 1][r - 1] = u - v;
    }
  const double cross = q[0][1] + q[1][0];
  return q[0][0] * (64.0 * cm) + (q[1][1] * cm - cross * (8.0 * cm));
}

// rhs + sigma/64 sum_d (1/h_d) [ (f+3 + f-3) - 6 (f+2 + f-2) + 15 (f+1 + f-1) - 20 f0 ]
// grouped as (s3 - s2) - 5 (s2 - s1) + 10 (s1 - 2 f0), s_k = f+k + f-k: the same
// coefficients, and every bracket is exactly zero when the neighbours equal f0.
template <int D>
__device__ __forceinline__ double ko_dir(const double* __restrict__ F, const Nbr& n, double f0) {
  const double s1 = ldg(F, disp<D>(n, 1)) + ldg(F, disp<D>(n, -1));
  const double s2 = ldg(F, disp<D>(n, 2)) + ldg(F, disp<D>(n, -2));
  const double s3 = ldg(F, disp<D>(n, 3)) + ldg(F, disp<D>(n, -3));
  const double t = fma(-2.0, f0, s1);
  return fma(10.0, t, fma(-5.0, s2 - s1, s3 - s2));
}

__device__ __forceinline__ double ko_add(const double* __restrict__ F, const Nbr& n, const Coef& c, double f0,
                                         double r) {
  r = fma(c.ko[0], ko_dir<0>(F, n, f0), r);
  r = fma(c.ko[1], ko_dir<1>(F, n, f0), r);
  r = fma(c.ko[2], ko_dir<2>(F, n, f0), r);
  return r;
}

// v + the Kreiss-Oliger term of a field on a grid with equal spacing along the
// three axes (one coefficient c.ko[0]): the bracket is linear in s_k, so the three
// axes are summed first, P_k = sum_d (f(+k e_d) + f(-k e_d)), and combined once:
// (P3 - P2) - 5 (P2 - P1) + 10 (P1 - 6 f0).  For a constant field every P_k and
// 6 f0 are the same single rounding of 6 f0, so each bracket is exactly zero.
__device__ __forceinline__ double ko_add_uniform(const double* __restrict__ F, const Nbr& n, const Coef& c, double f0,
                                                 double v, const Fp64Regs& k) {
  double P[3];
#pragma unroll
  for (int o = 1; o <= 3; ++o)
    P[o - 1] = add3(add3(add3(ldg(F, disp<0>(n, o)), ldg(F, disp<0>(n, -o)), k),
                         add3(ldg(F, disp<1>(n, o)), ldg(F, disp<1>(n, -o)), k), k),
                    add3(ldg(F, disp<2>(n, o)), ldg(F, disp<2>(n, -o)), k), k);
  const double t = sub3(P[0], __dmul_rn(6.0, f0), k);  // __dmul_rn: the product is rounded, never fused
  return fma(c.ko[0], fma(10.0, t, fma(-5.0, sub3(P[1], P[0], k), sub3(P[2], P[1], k))), v);
}

// Inputs of the generated algebra at one point (layout documented in codegen/bssn.py).
template <class T>
__device__ __forceinline__ void gather(const double* __restrict__ U, const double* __restrict__ prim, const Nbr& n,
                                       const Coef& c, long fs, double* in) {
#pragma unroll
  for (int f = 0; f < T::NF; ++f) in[f] = ldg(U + (long)f * fs, n.c);
#pragma unroll
  for (int m = 0; m < T::ND1; ++m) {
    const double* F = U + (long)T::d1_field(m) * fs;
    in[T::NF + 3 * m + 0] = fd1<0>(F, n, c);
    in[T::NF + 3 * m + 1] = fd1<1>(F, n, c);
    in[T::NF + 3 * m + 2] = fd1<2>(F, n, c);
  }
#pragma unroll
  for (int m = 0; m < T::ND2; ++m) {
    const int f = T::d2_field(m);
    const double* F = U + (long)f * fs;
    const double f0 = in[f];
    const int b = T::NF + 3 * T::ND1 + 6 * m;
    in[b + 0] = fd2<0>(F, n, c, f0);
    in[b + 1] = fdmix<0, 1>(F, n, c.mix[0]);
    in[b + 2] = fdmix<0, 2>(F, n, c.mix[1]);
    in[b + 3] = fd2<1>(F, n, c, f0);
    in[b + 4] = fdmix<1, 2>(F, n, c.mix[2]);
    in[b + 5] = fd2<2>(F, n, c, f0);
  }
  if constexpr (T::FLUID) in[T::NIN - 1] = ldg(prim, n.c);
}

template <class T>
__device__ __forceinline__ int ko_slot(int f) {
  return (T::FLUID && f >= 28) ? f - 4 : f;
}

}  // namespace cosmos

#include "stage_int.cuh"

namespace cosmos {

// Point (i, j, k) of work item `t` (thread `lane` of the block) of a batch:
// 2D tiles of blockDim.x x blockDim.y points in one z-plane, or runs of
// blockDim.x * blockDim.y consecutive points in memory order.  Returns false
// for a thread past the grid edge.
__device__ __forceinline__ bool batch_point(const BatchTile& t, const DevGrid& g, int mapping, int& i, int& j,
                                            int& k) {
  if (mapping == BATCH_MAP_TILE2D) {
    i = t.a * blockDim.x + threadIdx.x;
    j = t.b * blockDim.y + threadIdx.y;
    k = t.c;
    return i < g.nx && j < g.ny;
  }
  const long p = (long)t.a + threadIdx.y * blockDim.x + threadIdx.x;
  const long npts = (long)g.nx * g.ny * g.nz;
  if (p >= npts) return false;
  i = (int)(p % g.nx);
  j = (int)((p / g.nx) % g.ny);
  k = (int)(p / ((long)g.nx * g.ny));
  return true;
}

// Constraints H, M^i per point plus per-block partial norms.  The differences are FP64 differences of
// neighbouring values (770 of the kernel's 1335 FP64 instructions per point; 128^3 with the fluid 5.6 ms),
// so that small values of a field keep their relative accuracy and a NaN stays in its stencil neighbourhood:
// the integer differences of stage_int.cuh (3.6 ms, 24 doubles a point of workspace) are exact relative to a
// field's largest value over the grid only, and one NaN spoils them everywhere.
template <class T>
__global__ void __launch_bounds__(BX* BY, 2) constraint_kernel(const ConstraintArgs a) {
  const int i = blockIdx.x * BX + threadIdx.x;
  const int j = blockIdx.y * BY + threadIdx.y;
  const int k = blockIdx.z;
  const bool valid = (i < a.g.nx) && (j < a.g.ny);
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (valid) {
    const Nbr n = make_nbr(a.g, i, j, k);
    const long fs = a.g.fstride;
    double in[T::NIN];
    gather<T>(a.U, a.prim, n, a.c, fs, in);
    T::constraints(in, v, a.ap, fp64_regs());
    if (a.hm) {
#pragma unroll
      for (int m = 0; m < 4; ++m) a.hm[(long)m * fs + n.c] = v[m];
    }
  }
  double r[8];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    r[m] = v[m] * v[m];
    r[4 + m] = fabs(v[m]);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      r[m] += __shfl_down_sync(0xffffffffu, r[m], off);
      r[4 + m] = fmax(r[4 + m], __shfl_down_sync(0xffffffffu, r[4 + m], off));
    }
  }
  __shared__ double red[BY][8];
  if (threadIdx.x == 0) {
#pragma unroll
    for (int m = 0; m < 8; ++m) red[threadIdx.y][m] = r[m];
  }
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    double s[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) s[m] = red[0][m];
    for (int w = 1; w < BY; ++w) {
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        s[m] += red[w][m];
        s[4 + m] = fmax(s[4 + m], red[w][4 + m]);
      }
    }
    const long b = ((long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
#pragma unroll
    for (int m = 0; m < 8; ++m) a.partial[b * 8 + m] = s[m];
  }
}

#define COSMOS_DEFINE_VARIANT(NAME, IS_FLUID, IS_SCALAR)                                                          \
  struct T_##NAME {                                                                                             \
    static constexpr int NF = alg_##NAME::NF, ND1 = alg_##NAME::ND1, ND2 = alg_##NAME::ND2,                     \
                         NIN = alg_##NAME::NIN;                                                                 \
    static constexpr bool FLUID = IS_FLUID, SCALAR = IS_SCALAR;                                                 \
    __device__ static constexpr int d1_field(int m) { return alg_##NAME::d1_field(m); }                        \
    __device__ static constexpr int d2_field(int m) { return alg_##NAME::d2_field(m); }                        \
    __device__ static constexpr int d1_slot(int f) { return alg_##NAME::d1_slot(f); }                          \
    __device__ static constexpr int d2_slot(int f) { return alg_##NAME::d2_slot(f); }                          \
    static constexpr bool SPLIT_EARLY = alg_##NAME::SPLIT_EARLY;                                                    \
    static constexpr int SA = alg_##NAME::SA, SB = alg_##NAME::SB;                                                  \
    __device__ static constexpr int out_slot(int f) { return alg_##NAME::out_slot(f); }                             \
    template <class InA, class InB, class Out, class Next>                                                          \
    __device__ static __forceinline__ void rhs_split(const InA& ina, const InB& inb, Out&& out, Next&& next,        \
                                                     const AlgebraParams& p, const Fp64Regs& k) {                   \
      alg_##NAME::rhs_split(ina, inb, out, next, p, k);                                                           \
    }                                                                                                               \
    __device__ static __forceinline__ void constraints(const double* in, double* out, const AlgebraParams& p,       \
                                                       const Fp64Regs& k) {                                       \
      alg_##NAME::constraints(in, out, p, k);                                                                     \
    }                                                                                                           \
  };                                                                                                            \
  cudaError_t launch_stage_##NAME(const StageArgs& a, int mode, cudaStream_t s) {                                   \
    if (!a.L) return cudaErrorInvalidValue; /* the differences are those of the limb copy */                        \
    const long tiles = stage_tiles(a.g, a.k_hi - a.k_lo);                                                           \
    return launch_split<T_##NAME, false>(a, nullptr, nullptr, tiles, nullptr, mode, a.eq, thin_tiles(a.g), s);      \
  }                                                                                                                 \
  cudaError_t launch_deriv_##NAME(const StageArgs& a, cudaStream_t s) {                                             \
    if (!a.L) return cudaErrorInvalidValue;                                                                         \
    if (near_indices(a.g))                                                                                          \
      ideriv_kernel<T_##NAME, true><<<ideriv_grid(a.g), dim3(BX, DBY), 0, s>>>(a);                                  \
    else                                                                                                            \
      ideriv_kernel<T_##NAME, false><<<ideriv_grid(a.g), dim3(BX, DBY), 0, s>>>(a);                                 \
    return cudaGetLastError();                                                                                      \
  }                                                                                                                 \
  cudaError_t launch_batch_stage_##NAME(const StageArgs* args, const BatchTile* tiles, long ntiles,                 \
                                        const double* kref, int mode, bool eq, bool thin, cudaStream_t s) {         \
    StageArgs none;                                                                                                 \
    memset(&none, 0, sizeof(none));                                                                                 \
    return launch_split<T_##NAME, true>(none, args, tiles, ntiles, kref, mode, eq, thin, s);                        \
  }                                                                                                                 \
  cudaError_t launch_constraints_##NAME(const ConstraintArgs& a, cudaStream_t s) {                              \
    constraint_kernel<T_##NAME><<<point_grid(a.g), dim3(BX, BY), 0, s>>>(a);                                    \
    return cudaGetLastError();                                                                                  \
  }

}  // namespace cosmos
