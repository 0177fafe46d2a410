// Finite differences in exact integer arithmetic.
//
// GB300 runs FP64 at 2 operations per clock per SM and 32-bit integer adds and
// multiply-adds at about 60: the finite-difference and Kreiss-Oliger stencils,
// integer-coefficient sums of neighbouring values, are cheaper in integer
// arithmetic than in FP64, and can be made exact there.  The stage kernel
// (stage_split.cuh) forms them tile by tile; ideriv_kernel below writes them to
// memory for the reverse mode.
//
// Representation ("limbs"): every value f of one field is held as the signed
// 64-bit integer V = f 2^(1085 - e_ref), with e_ref the largest biased FP64
// exponent of the field over the grid: the field's largest value has
// 53 + 10 significant bits (|V| < 2^63), every value down to 2^-10 of it is
// exact, and smaller ones are truncated by at most 2^-62 of the largest (a
// relative 2e-15 even of a 256^3 second derivative of such a field, where the
// tolerance is 1e-12).  A stencil sum_o c_o f_o with integer c_o (sum |c_o| <= 324,
// the mixed derivative on staged first-derivative sums) needs up to 72 bits.
// It is carried as (w, h): w the sum of the V modulo 2^64, h the sum of their
// upper parts floor(V / 2^42), which stays below 2^30.  The lower parts add less
// than 324 x 2^42 < 2^51, so h tells whether the sum fits 64 bits (then it is w),
// and if not, w - h 2^42, taken modulo 2^64, is the exact difference: the sum is
// h 2^42 + that.  Two words and one, three instructions a sum, none to take a
// loaded value apart but one shift (three 21-bit digits took four, and ten to
// put a sum together again).  Each result is rounded once to FP64 (round to nearest even).
//
// The state is converted to limbs by a pre-pass (limbs.cu: the exponent of
// every field, then the conversion).
#pragma once

#include "common.cuh"

namespace cosmos {

constexpr int LIMB_EXTRA = 10;                    // significant bits below the largest value's last place

struct Limb {
  unsigned long long w;  // the sum modulo 2^64
  int h;                 // the sum of floor(V / 2^42)
};
__host__ __device__ __forceinline__ Limb l_add(Limb a, Limb b) { return {a.w + b.w, a.h + b.h}; }
__host__ __device__ __forceinline__ Limb l_sub(Limb a, Limb b) { return {a.w - b.w, a.h - b.h}; }
// k > 0
__host__ __device__ __forceinline__ Limb l_mul(Limb a, int k) { return {a.w * (unsigned)k, a.h * k}; }
// 8 a - b, the first-derivative sum of a = f(+1) - f(-1), b = f(+2) - f(-2)
__host__ __device__ __forceinline__ Limb l_d1(Limb a, Limb b) { return l_sub(l_mul(a, 8), b); }

// V of f for a field with reference exponent e_ref (>= the exponent of f).
__device__ __forceinline__ long long to_limbs(double f, int e_ref) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(f);
  const int e = (int)((b >> 52) & 0x7FF);
  unsigned long long M = b & 0xFFFFFFFFFFFFFull;
  if (e) M |= 1ull << 52;
  const int s = (e ? e : 1) - e_ref + LIMB_EXTRA;  // V = M 2^s, s <= 10
  const unsigned long long V = s >= 0 ? M << s : (s > -64 ? M >> (-s) : 0ull);
  return (b >> 63) ? -(long long)V : (long long)V;
}

__host__ __device__ __forceinline__ Limb limb_of(long long V) { return {(unsigned long long)V, (int)(V >> 42)}; }

// e_ref outside the range in which every sum's exponent is that of a normal
// number (uniform over a field).
__host__ __device__ __forceinline__ bool limb_odd(int e_ref) { return e_ref < 80 || e_ref > 1960; }

// limb_big: the sum may not fit a signed 64-bit word (|h| 2^42 near 2^63 or above).
constexpr int LIMB_FIT = (1 << 21) - (1 << 11);  // LIMB_FIT 2^42 + 2^51 < 2^63
__host__ __device__ __forceinline__ bool limb_big(Limb S) { return (unsigned)(S.h + LIMB_FIT) >= 2u * LIMB_FIT; }

// FP64 value (bits; round to nearest even) of the sum S times 2^(e_ref + twos - 1085), e_ref the
// field's exponent (2047: it holds Inf or NaN); ODD = limb_odd(e_ref); ANY: also for sums with limb_big.
//
// The sum is taken into one signed 64-bit word; where it does not fit, its low 8
// or 9 bits are dropped first, their "any set" kept in the lowest bit: at least
// two bits are dropped again below, so that bit never is the last kept one and
// the rounding is that of the whole sum.  The magnitude's leading one is moved
// to bit 63 of a pair of 32-bit words, the upper 53 bits are kept, and the
// dropped 11 (in the upper bits of r) round to nearest even through the carry
// of r + (2^31 - 1) + the last kept bit; the leading one, or a carry out of the
// significand, adds into the exponent field.  About 25 instructions, without a
// branch, so that the conversions of one thread overlap; a 128-bit path for the
// large sums, taken by half the warps on data that vary along every axis, cost
// as many again.
template <bool ODD, bool ANY>
__host__ __device__ __forceinline__ unsigned long long limb_bits(Limb S, int e_ref, int twos = 0) {
  long long v = (long long)S.w;
  int ex = e_ref + twos;
  if (ANY) {
    const long long t1 = (long long)(S.w - ((unsigned long long)(unsigned)S.h << 42));  // |t1| < 2^51
    const int ah = S.h < 0 ? -S.h : S.h;
    // big sums: below 2^70 (2^62 after 8) / below 2^72 (below 2^63 after 9)
    const int sh = limb_big(S) ? (ah < (1 << 28) ? 8 : 9) : 0;
    v = (t1 >> sh) + (long long)(((unsigned long long)(unsigned)S.h << (10 - sh)) << 32);
    v |= ((unsigned)t1 & ((1u << sh) - 1u)) ? 1 : 0;
    ex += sh;
  }
  const int sg = (int)(v >> 63);
  const unsigned long long u = (unsigned long long)((v ^ (long long)sg) - (long long)sg);
  const unsigned hi = (unsigned)(u >> 32), lo = (unsigned)u;
  const bool one = hi == 0;  // one word
  const unsigned h = one ? lo : hi, l = one ? 0u : lo;
  const int E = one ? ex - 32 : ex;
#ifdef __CUDA_ARCH__
  const int s = __clz((int)h);
  const unsigned h2 = __funnelshift_l(l, h, s), l2 = l << (s & 31);
#else
  const int s = h ? __builtin_clz(h) : 32;
  const unsigned h2 = s & 31 ? h << s | l >> (32 - s) : h, l2 = l << (s & 31);
#endif
  const unsigned mh = h2 >> 11, ml = (h2 << 21) | (l2 >> 11);
  const unsigned r = l2 << 21, up = 0x7FFFFFFFu + (ml & 1u);
  // biased exponent 63 - s + E - 1085 + 1023, of which the leading one is 1
  const unsigned eb = (unsigned)(E - s) << 20;
#ifdef __CUDA_ARCH__
  unsigned drop, bl, bh;
  asm("add.cc.u32 %0, %3, %4;\n\taddc.cc.u32 %1, %5, 0;\n\taddc.u32 %2, %6, %7;"
      : "=r"(drop), "=r"(bl), "=r"(bh)
      : "r"(r), "r"(up), "r"(ml), "r"(mh), "r"(eb));
#else
  const unsigned inc = (unsigned)(((unsigned long long)r + up) >> 32);
  const unsigned long long sum = (((unsigned long long)mh << 32) | ml) + inc;
  unsigned bl = (unsigned)sum, bh = (unsigned)(sum >> 32) + eb;
#endif
  if (ODD) {
    if (e_ref >= 2047) return 0x7FF8000000000000ull;  // the field holds Inf or NaN
    const int be = E - s + (int)((bh - eb) >> 20);    // biased exponent
    if (be <= 0) bh = bl = 0;                         // below the normal range: far below any stencil of this field
    if (be >= 2047) {
      bh = 0x7FFu << 20;
      bl = 0;
    }
  }
  if (h == 0) bh = 0;  // bl is zero already
  bh |= (unsigned)sg & 0x80000000u;
  return ((unsigned long long)bh << 32) | bl;
}

template <bool ODD>
__device__ __forceinline__ double limb_value(Limb S, int e_ref, int twos = 0) {
  return __longlong_as_double((long long)limb_bits<ODD, true>(S, e_ref, twos));
}

// N sums of one field in one warp (every lane takes part) at once, the q-th times 2^twos[q]: the form
// without the large sums' part when no lane has one.
template <bool ODD, int N>
__device__ __forceinline__ void limb_values(const Limb (&S)[N], int e, const int (&twos)[N], double (&v)[N]) {
  unsigned top = 0;
#pragma unroll
  for (int q = 0; q < N; ++q) top = max(top, (unsigned)(S[q].h + LIMB_FIT));
  if (__any_sync(0xffffffffu, top >= 2u * LIMB_FIT)) {
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = limb_value<ODD>(S[q], e, twos[q]);
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = __longlong_as_double((long long)limb_bits<ODD, false>(S[q], e, twos[q]));
  }
}

// ---------------------------------------------------------------------------
// Pre-pass.  Slot s of the limb copy holds field s, except that with the fluid
// on the fields after the fluid ones (the scalar) move down by 4 (the fluid
// fields have no derivatives in this pass).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int limb_field(int s, int fluid) { return (fluid && s >= 24) ? s + 4 : s; }

// ---------------------------------------------------------------------------
// Integer stencils (digit sums; the caller converts and scales)
// ---------------------------------------------------------------------------
__device__ __forceinline__ Limb ldl(const long long* __restrict__ L, int o) { return limb_of(__ldg(L + o)); }

// Sums staged in shared memory as int4 (the last word unused): one 128-bit access each.
__device__ __forceinline__ int4 p4(Limb v) { return make_int4((int)v.w, (int)(v.w >> 32), v.h, 0); }
__device__ __forceinline__ Limb q3(int4 v) {
  return {((unsigned long long)(unsigned)v.y << 32) | (unsigned)v.x, v.z};
}

// Periodic neighbour offsets of one point within one field, as 32-bit
// element offsets (a field of the grids this pass accepts has < 2^31 points).
struct NbrI {
  int x[7], y[7], z[7];
  int c;
};

// Periodic index of a in [-n, 2n): a compare and a select instead of the
// integer division of wrap_index.
__device__ __forceinline__ int wrap_near(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

template <bool NEAR>
__device__ __forceinline__ int wrap_i(int a, int n) { return NEAR ? wrap_near(a, n) : wrap_index(a, n); }

template <bool NEAR>
__device__ __forceinline__ NbrI make_nbri(const DevGrid& g, int i, int j, int k) {
  NbrI n;
  const int row = g.pitch, plane = g.pitch * g.ny;
#pragma unroll
  for (int o = -3; o <= 3; ++o) {
    n.x[o + 3] = wrap_i<NEAR>(i + o, g.nx);
    n.y[o + 3] = wrap_i<NEAR>(j + o, g.ny) * row;
    n.z[o + 3] = wrap_i<NEAR>(k + o, g.nz) * plane;
  }
  n.c = n.z[3] + n.y[3] + n.x[3];
  return n;
}


template <int D>
__device__ __forceinline__ int dispi(const NbrI& n, int o) {
  if (D == 0) return n.z[3] + n.y[3] + n.x[o + 3];
  if (D == 1) return n.z[3] + n.y[o + 3] + n.x[3];
  return n.z[o + 3] + n.y[3] + n.x[3];
}

template <bool NEAR>
__device__ __forceinline__ int limb_plane_off(const DevGrid& g, int x, int y, int k) {
  return (wrap_i<NEAR>(k, g.nz) * g.ny + wrap_i<NEAR>(y, g.ny)) * g.pitch + wrap_i<NEAR>(x, g.nx);
}

// Digit sums of D_y (rows j0 .. j0+DBY-1) and D_z (rows j0-2 .. j0+DBY+1) on
// the x-extended tile (halo 2), unscaled.
template <bool NEAR>
__device__ __forceinline__ void stage_dydz_int(const DevGrid& g, const long long* __restrict__ Lf, int i0, int j0,
                                                 int k, int tid, int4* __restrict__ sDy, int4* __restrict__ sDz) {
  constexpr int TXH = BX + 4;
  for (int q = tid; q < TXH * DBY; q += BX * DBY) {
    const int qx = q % TXH, qy = q / TXH;
    const int x = i0 - 2 + qx, y = j0 + qy;
    sDy[q] = p4(l_d1(l_sub(ldl(Lf, limb_plane_off<NEAR>(g, x, y + 1, k)),
                           ldl(Lf, limb_plane_off<NEAR>(g, x, y - 1, k))),
                     l_sub(ldl(Lf, limb_plane_off<NEAR>(g, x, y + 2, k)), ldl(Lf, limb_plane_off<NEAR>(g, x, y - 2, k)))));
  }
  for (int q = tid; q < TXH * (DBY + 4); q += BX * DBY) {
    const int qx = q % TXH, qy = q / TXH;
    const int x = i0 - 2 + qx, y = j0 - 2 + qy;
    sDz[q] = p4(l_d1(l_sub(ldl(Lf, limb_plane_off<NEAR>(g, x, y, k + 1)),
                           ldl(Lf, limb_plane_off<NEAR>(g, x, y, k - 1))),
                     l_sub(ldl(Lf, limb_plane_off<NEAR>(g, x, y, k + 2)), ldl(Lf, limb_plane_off<NEAR>(g, x, y, k - 2)))));
  }
}


// D1 sum 8 (f+1 - f-1) - (f+2 - f-2) of axis D at point n, and with it
// s_k = f(+k) + f(-k), k = 1, 2.
template <int D>
__device__ __forceinline__ void iaxis(const long long* __restrict__ L, const NbrI& n, Limb& d1, Limb& s1, Limb& s2) {
  const Limb p1 = ldl(L, dispi<D>(n, 1)), m1 = ldl(L, dispi<D>(n, -1));
  const Limb p2 = ldl(L, dispi<D>(n, 2)), m2 = ldl(L, dispi<D>(n, -2));
  d1 = l_d1(l_sub(p1, m1), l_sub(p2, m2));
  s1 = l_add(p1, m1);
  s2 = l_add(p2, m2);
}

template <int D>
__device__ __forceinline__ Limb id1(const long long* __restrict__ L, const NbrI& n) {
  Limb d1, s1, s2;
  iaxis<D>(L, n, d1, s1, s2);
  return d1;
}

// First derivatives of a field that has no second ones.
template <class T, bool ODD>
__device__ __forceinline__ void ideriv_d1_point(const StageArgs& a, int m, const NbrI& n, int e) {
  const long fs = a.dfs;
  const int s = ko_slot<T>(T::d1_field(m));
  const long long* Lf = a.L + (long)s * a.g.fstride;
  double* __restrict__ D = a.D + (long)(3 * m) * fs + n.c;
  D[0] = limb_value<ODD>(id1<0>(Lf, n), e) * a.c.d1b[0];
  D[fs] = limb_value<ODD>(id1<1>(Lf, n), e) * a.c.d1b[1];
  D[2 * fs] = limb_value<ODD>(id1<2>(Lf, n), e) * a.c.d1b[2];
}

// First and second derivatives of field m2 at point n, each written as soon as
// it is formed; D_y and D_z sums come from the staging area.
template <class T, bool ODD>
__device__ __forceinline__ void ideriv_d2_point(const StageArgs& a, int m2, const NbrI& n, int e, int tx, int ty,
                                                const int4* __restrict__ sDy, const int4* __restrict__ sDz) {
  constexpr int TXH = BX + 4;
  const long fs = a.dfs;
  const Coef& c = a.c;
  double* __restrict__ D = a.D;
  const int f = T::d2_field(m2);
  const int s = ko_slot<T>(f);
  const long long* Lf = a.L + (long)s * a.g.fstride;
  const int m1 = T::d1_slot(f);
  const long b = (long)(3 * T::ND1 + 6 * m2) * fs + n.c;
  const Limb f30 = l_mul(ldl(Lf, n.c), 30);
  Limb d1, s1, s2;
  // second derivative 16 (f+1 + f-1) - (f+2 + f-2) - 30 f0 of axis AX into slot SL
#define COSMOS_IAXIS2(AX, SL)          \
  iaxis<AX>(Lf, n, d1, s1, s2);        \
  D[b + SL * fs] = limb_value<ODD>(l_sub(l_sub(l_mul(s1, 16), s2), f30), e) * c.d2b[AX];
  COSMOS_IAXIS2(0, 0)
  D[(long)(3 * m1 + 0) * fs + n.c] = limb_value<ODD>(d1, e) * c.d1b[0];
  COSMOS_IAXIS2(1, 3)
  COSMOS_IAXIS2(2, 5)
#undef COSMOS_IAXIS2
  const int4* ry = sDy + ty * TXH + tx + 2;        // D_y sums at (i + o, j)
  const int4* rz = sDz + (ty + 2) * TXH + tx + 2;  // D_z sums at (i + o, j), row stride TXH along y
  D[(long)(3 * m1 + 1) * fs + n.c] = limb_value<ODD>(q3(ry[0]), e) * c.d1b[1];
  D[(long)(3 * m1 + 2) * fs + n.c] = limb_value<ODD>(q3(rz[0]), e) * c.d1b[2];
  D[b + 1 * fs] =
      limb_value<ODD>(l_d1(l_sub(q3(ry[1]), q3(ry[-1])), l_sub(q3(ry[2]), q3(ry[-2]))), e) * c.mix[0];
  D[b + 2 * fs] =
      limb_value<ODD>(l_d1(l_sub(q3(rz[1]), q3(rz[-1])), l_sub(q3(rz[2]), q3(rz[-2]))), e) * c.mix[1];
  D[b + 4 * fs] = limb_value<ODD>(l_d1(l_sub(q3(rz[TXH]), q3(rz[-TXH])),
                                        l_sub(q3(rz[2 * TXH]), q3(rz[-2 * TXH]))), e) * c.mix[2];
}

// One BX x DBY tile of one z-plane (block of BX x DBY threads); the D_y / D_z
// sums of one second-derivative field at a time are staged in shared memory.
template <class T, bool NEAR>
__device__ __forceinline__ void ideriv_tile(const StageArgs& a, int i0, int j0, int k, int4* __restrict__ sDy,
                                            int4* __restrict__ sDz) {
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * BX + tx;
  const int i = i0 + tx, j = j0 + ty;
  const bool valid = i < a.g.nx && j < a.g.ny;
  const NbrI n = make_nbri<NEAR>(a.g, i, j, k);
  const long fs = a.g.fstride;
#pragma unroll 1
  for (int m = 0; m < T::ND1; ++m) {
    if (T::d2_slot(T::d1_field(m)) >= 0) continue;
    const int e = max(a.E[ko_slot<T>(T::d1_field(m))], 1);
    if (!valid) continue;
    if (limb_odd(e))
      ideriv_d1_point<T, true>(a, m, n, e);
    else
      ideriv_d1_point<T, false>(a, m, n, e);
  }
#pragma unroll 1
  for (int m2 = 0; m2 < T::ND2; ++m2) {
    const int f = T::d2_field(m2);
    stage_dydz_int<NEAR>(a.g, a.L + (long)ko_slot<T>(f) * fs, i0, j0, k, tid, sDy, sDz);
    __syncthreads();
    if (valid) {
      const int e = max(a.E[ko_slot<T>(f)], 1);
      if (limb_odd(e))
        ideriv_d2_point<T, true>(a, m2, n, e, tx, ty, sDy, sDz);
      else
        ideriv_d2_point<T, false>(a, m2, n, e, tx, ty, sDy, sDz);
    }
    __syncthreads();
  }
}

// NEAR: near_indices holds for the grid (for every grid of a batch).
template <class T, bool NEAR>
__global__ void __launch_bounds__(BX* DBY, COSMOS_IDERIV_MIN_BLOCKS) ideriv_kernel(const StageArgs a) {
  __shared__ int4 sDy[(BX + 4) * DBY], sDz[(BX + 4) * (DBY + 4)];
  ideriv_tile<T, NEAR>(a, blockIdx.x * BX, blockIdx.y * DBY, blockIdx.z, sDy, sDz);
}

}  // namespace cosmos
