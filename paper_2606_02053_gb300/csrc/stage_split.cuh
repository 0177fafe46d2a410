// One RK4 stage as one persistent kernel: finite differences, pointwise
// algebra and stage combine of a tile side by side in one block.
//
// What bounds it: the algebra is FP64 work (718 instructions per point in
// vacuum, 190 more in the advection, dissipation and combine beside it) at 2 multiply-adds per clock per SM
// (lone multiplies and adds 1.7), and one warp per scheduler nearly keeps that
// pipe full (a dependent chain of one warp issues one multiply-add per 64
// cycles, its whole rate).  The finite differences are integer work
// (stage_int.cuh) on units that the algebra leaves idle.  As two kernels one
// after the other each left the other's units idle, and the 162 differences
// per point travelled through memory.  Here a block has one algebra warpgroup
// with 200 registers a thread and SPLIT_GROUPS difference warpgroups with 104,
// and the differences of a tile (SPLIT_TX x SPLIT_TY points of one z-plane, a
// point per algebra thread) go through shared memory.  256^3 vacuum stage: 10.0
// + 27.5 ms as two kernels, 30.3 ms as this one (its algebra warps wait for the
// others in under 3% of their time); 128^3 fluid 5.4 -> 4.6 ms.  The algebra with 240 or 224 registers, the difference warps with 88 or 96,
// and four groups of 64 were within 1 to 3% and slower.
//
// The algebra runs in two phases of about equal length (codegen/bssn.py,
// split_layout): the first reads region A (conformal metric and Gamma: the
// Ricci tensor), the second region B (everything else).  While the first
// phase works on a tile the difference warps fill its region B, while the second does
// they fill region A of the next tile, so neither region needs a second copy.
// The second phase leaves its outputs in region B, and the difference warps do
// the stage combine with them (their many threads hide the latency of the
// state and accumulator loads that one algebra warp per scheduler could not).
//
//   algebra warps:     | wait A(t) | phase 1 | free A | wait B(t) | phase 2, r -> B | done |
//   difference warps:  | fill B(t) | wait free A | fill A(t+1) | wait done | combine(t) |
//
// Units: with l = 12 h_x as the unit of length every difference of equal
// spacing is its exact integer sum, rounded once, without a factor: 12 h d_k f,
// (12 h)^2 d_k d_k f = 3 (16 s1 - s2 - 30 f0) 2^2 and (12 h)^2 d_a d_b f are the
// digit sums themselves.  Fields that carry inverse lengths (K, At, Gt, B, Pi:
// one; tau, S, rho: two) are scaled by l or l^2 where they enter, and the
// outputs by a power of 1/l in the stage combine, where a factor is there
// anyway.  K - K_ref is formed before the scaling (it cancels).
#pragma once

#include "stage_kernel.cuh"

namespace cosmos {

constexpr int SPLIT_PTS = SPLIT_TX * SPLIT_TY;
constexpr int SPLIT_GROUPS = 3;  // difference warpgroups
constexpr int SPLIT_THREADS = SPLIT_PTS * (1 + SPLIT_GROUPS);
static_assert(SPLIT_PTS == 128, "one point per thread of a warpgroup");
// Registers: the pool is the launch's SPLIT_THREADS x (65536 / SPLIT_THREADS,
// rounded down to 8); the two shares below add up to no more than it.
constexpr int SPLIT_POOL = (65536 / SPLIT_THREADS) & ~7;
#ifndef COSMOS_SPLIT_REG_DIFF
#define COSMOS_SPLIT_REG_DIFF 104
#define COSMOS_SPLIT_REG_ALG 200
#endif
constexpr int SPLIT_REG_DIFF = COSMOS_SPLIT_REG_DIFF;
constexpr int SPLIT_REG_ALG = COSMOS_SPLIT_REG_ALG;
static_assert(SPLIT_REG_ALG + SPLIT_GROUPS * SPLIT_REG_DIFF <= SPLIT_POOL * (1 + SPLIT_GROUPS), "register shares");
// Staged D_y (tile rows) and D_z (rows with a 2-point halo) sums, both with a
// 2-point halo along x.
constexpr int SPLIT_XH = SPLIT_TX + 4;
constexpr int SPLIT_NDY = SPLIT_XH * SPLIT_TY, SPLIT_NDZ = SPLIT_XH * (SPLIT_TY + 4);
// Periodic offsets of the rows, columns and planes a tile touches (3-point halo)
constexpr int SPLIT_NXW = SPLIT_TX + 6, SPLIT_NYW = SPLIT_TY + 6, SPLIT_NZW = 7;

// Named barriers (0 is left to __syncthreads)
constexpr int BAR_FULL_A = 1, BAR_FREE_A = 2, BAR_FULL_B = 3, BAR_DONE_B = 4, BAR_DIFF = 5, BAR_GROUP = 6;

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Region layouts (the order of codegen/bssn.py, split_layout).
template <class T>
struct Slots {
  static constexpr int A = T::SA, B = T::SB;
  // (d_k, dd_p, m of a second-derivative field; d_k, m of a first-derivative one)
  // region A: 6 x 10 (metric), 3 x 4 (Gamma), metric, shift, inverse metric, At (SPLIT_EARLY), fluid: chi,
  // tau, S_i, rho
  static constexpr int A_GT = 0, A_GAM = 60, A_STATE = 72;
  static constexpr int A_NSTATE = 15 + (T::SPLIT_EARLY ? 6 : 0) + (T::FLUID ? 6 : 0);
  // region B: ND2B x 10 (chi, alpha, beta^i, phi), K (4), merged advections, states, output slots
  static constexpr int ND2B = 5 + (T::SCALAR ? 1 : 0), NM = 9 + (T::SCALAR ? 1 : 0);
  static constexpr int B_K = 10 * ND2B, B_M = B_K + 4, B_STATE = B_M + NM;
  static constexpr int B_NSTATE = 20 + (T::FLUID ? 5 : 0) + (T::SCALAR ? 1 : 0);
  static constexpr int B_KDIFF = 18;  // K - K_ref
  static constexpr int PHI = T::FLUID ? 28 : 24;
  static_assert(A == A_STATE + A_NSTATE, "region A");
  static_assert(B == B_STATE + B_NSTATE + 9 + (T::FLUID ? 4 : 0), "region B");
  // field of the m-th second-derivative block of region B
  __device__ static __forceinline__ int b_d2(int m) { return m == 0 ? 0 : (m == 1 ? 17 : (m < 5 ? 16 + m : PHI)); }
  // field of the m-th merged advection
  __device__ static __forceinline__ int b_m(int m) { return m < 6 ? 8 + m : (m < 9 ? 15 + m : PHI + 1); }
  // field of the s-th state of each region, -1 for rho, -2 - m for field m of G
  __device__ static constexpr int a_state(int s) {
    constexpr int E = T::SPLIT_EARLY ? 21 : 15;
    return s < 6 ? 1 + s
                 : (s < 9 ? 12 + s : (s < 15 ? 7 - s : (s < E ? s - 7 : (s == E ? 0 : (s < E + 5 ? 23 + s - E : -1)))));
  }
  __device__ static constexpr int b_state(int s) {
    return s < 14 ? s
                  : (s == 14 ? 17
                             : (s < 18 ? s + 6
                                       : (s == B_KDIFF ? 7
                                                       : (s == 19 ? -8 : (T::FLUID ? (s < 24 ? s + 4 : (s == 24 ? -1 : 29))
                                                                                   : 25)))));
  }
  // powers of the unit of length on a state (B^i enters without its own)
  __device__ static constexpr int state_degree(int f) {
    return f == -1 ? 2 : (f < 0 || (f >= 21 && f < 24) ? 0 : degree(f));
  }
  // powers of the unit of length that field f (and its time derivative, one more) carries
  __device__ static constexpr int degree(int f) {
    if (f >= 24) return (T::FLUID && f < 28) ? 2 : (f == PHI ? 0 : 1);
    return ((f >= 7 && f <= 16) || f >= 21) ? 1 : 0;
  }
};

template <class T>
constexpr size_t split_smem_bytes() {
  return sizeof(double) * SPLIT_PTS * (T::SA + T::SB) + sizeof(int4) * SPLIT_GROUPS * (SPLIT_NDY + SPLIT_NDZ) +
         sizeof(int) * (SPLIT_GROUPS * (48 + 32) + 32);
}

// Tile w of the plane range of one grid, or of a batch's tile list: SPLIT_TX points along x from i0,
// SPLIT_TY rows along y from j0 at plane k of z, or (THIN, thin_tiles in common.cuh) along z from j0 at
// row k of y.
struct SplitTile {
  int i0, j0, k, inst;
};

struct SlotIn {
  const double* s;
  __device__ __forceinline__ double operator[](int k) const { return s[k * SPLIT_PTS]; }
};

template <class T>
struct SlotOut {
  double* s;
  struct Slot {
    double* p;
    __device__ __forceinline__ void operator=(double v) const { *p = v; }
  };
  __device__ __forceinline__ Slot operator[](int f) const { return Slot{s + T::out_slot(f) * SPLIT_PTS}; }
};

// What a difference thread needs of a tile and its instance.  Offsets are in
// bytes within one field, 32 bits (validate_stage refuses fields beyond 4 GiB,
// which with the other fields and buffers of a stage exceed the device's memory):
// added to a field's base, which is uniform, they need no 64-bit arithmetic.
struct DiffCtx {
  const char* L;
  const char* U;
  long fb;           // bytes of one field
  unsigned c;        // the point itself (clamped into the grid)
  unsigned o[3];     // that without its offset along each axis,
  int p[3];          // and its place along each axis in the offset tables
  unsigned b[4];     // staged sums q = t + 128 j of this thread: offset without the axis differenced
  double r[3];       // h_x / h_d (unequal spacing)
};

__device__ __forceinline__ long long ldv(const char* __restrict__ base, unsigned o) {
  return __ldg(reinterpret_cast<const long long*>(base + o));
}
__device__ __forceinline__ double ldd(const char* __restrict__ base, unsigned o) {
  return __ldg(reinterpret_cast<const double*>(base + o));
}

// Axes of a tile: 0 = x, 1 = that of its rows, 2 = the third.  Slots are by the grid's axes.
template <class T, bool EQ, bool THIN>
struct DiffGroup {
  static constexpr int ROW = THIN ? 2 : 1, OUT = THIN ? 1 : 2;  // grid axes of tile axes 1 and 2, and the reverse
  const int t;     // thread of the group = point of the tile
  const int g;     // group
  double* sA;      // region A + t
  double* sB;      // region B + t
  int4* sDy;       // staged D_y sums, the D_z sums after them
  unsigned* xw;    // periodic offsets: columns i0 - 3 .., then rows, then planes
  int* ex;         // reference exponents
  int* rec;        // largest exponents written so far (all groups)

  __device__ __forceinline__ void sync() const { bar_sync(BAR_GROUP + g, SPLIT_PTS); }

  // Offsets of the tile for this group; every thread of the group calls it.
  __device__ __forceinline__ void begin(const StageArgs& a, const SplitTile& w, DiffCtx& x) const {
    sync();  // the group is done with the tables of the tile before
    constexpr int NSLOT = 24 + (T::SCALAR ? 2 : 0);
    const unsigned row = 8u * (unsigned)a.g.pitch, plane = row * (unsigned)a.g.ny;
    if (t < SPLIT_NXW)
      xw[t] = 8u * (unsigned)wrap_index(w.i0 - 3 + t, a.g.nx);
    else if (t < SPLIT_NXW + SPLIT_NYW)
      xw[t] = (THIN ? plane : row) * (unsigned)wrap_index(w.j0 - 3 + t - SPLIT_NXW, THIN ? a.g.nz : a.g.ny);
    else if (t < SPLIT_NXW + SPLIT_NYW + SPLIT_NZW)
      xw[t] = (THIN ? row : plane) * (unsigned)wrap_index(w.k - 3 + t - SPLIT_NXW - SPLIT_NYW, THIN ? a.g.ny : a.g.nz);
    else if (t >= 64 && t < 64 + NSLOT)
      ex[t - 64] = max(a.E[t - 64], 1);
    sync();
    const unsigned *yw = xw + SPLIT_NXW, *zw = yw + SPLIT_NYW;
    // threads past the edge take the last column / row: their results are not stored
    const int tx = min(t % SPLIT_TX, a.g.nx - 1 - w.i0), ty = min(t / SPLIT_TX, (THIN ? a.g.nz : a.g.ny) - 1 - w.j0);
    const unsigned cx = xw[tx + 3], cy = yw[ty + 3], cz = zw[3];
    x.c = cx + cy + cz;
    x.o[0] = cy + cz;
    x.o[1] = cx + cz;
    x.o[2] = cx + cy;
    x.p[0] = tx + 3;
    x.p[1] = SPLIT_NXW + ty + 3;
    x.p[2] = SPLIT_NXW + SPLIT_NYW + 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int q = t + SPLIT_PTS * j, z = q - SPLIT_NDY;
      x.b[j] = q < SPLIT_NDY ? xw[q % SPLIT_XH + 1] + cz
                             : (q < SPLIT_NDY + SPLIT_NDZ ? xw[z % SPLIT_XH + 1] + yw[z / SPLIT_XH + 1] : 0u);
    }
    x.L = reinterpret_cast<const char*>(a.L);
    x.U = reinterpret_cast<const char*>(a.U);
    x.fb = 8 * a.g.fstride;
    if (!EQ) {
#pragma unroll
      for (int d = 0; d < 3; ++d) x.r[d] = a.ratio[d == 0 ? 0 : (d == 1 ? ROW : OUT)];
    }
  }

  // Place of the centre of staged sum q = t + 128 j along the differenced axis in the offset tables.
  __device__ __forceinline__ int centre(int j) const {
    const int q = t + SPLIT_PTS * j;
    return q < SPLIT_NDY ? SPLIT_NXW + 3 + q / SPLIT_XH : SPLIT_NXW + SPLIT_NYW + 3;
  }

  // The six neighbours -3, -2, -1, 1, 2, 3 along axis d.  Their offsets come from the tables each
  // time: held in registers they would spill others.
  __device__ __forceinline__ void load(const char* __restrict__ L, const DiffCtx& x, int d, long long (&n)[6]) const {
    const unsigned* const o = xw + x.p[d];
#pragma unroll
    for (int q = 0; q < 6; ++q) n[q] = ldv(L, x.o[d] + o[q < 3 ? q - 3 : q - 2]);
  }

  // D1 sum and s_k = f(+k) + f(-k) along one axis
  __device__ __forceinline__ static void axis(const long long (&n)[6], Limb& d1, Limb& s1, Limb& s2, Limb& s3) {
    const Limb p1 = limb_of(n[3]), m1 = limb_of(n[2]), p2 = limb_of(n[4]), m2 = limb_of(n[1]);
    d1 = l_d1(l_sub(p1, m1), l_sub(p2, m2));
    s1 = l_add(p1, m1);
    s2 = l_add(p2, m2);
    s3 = l_add(limb_of(n[5]), limb_of(n[0]));
  }
  // 3 (16 s1 - s2 - 30 f0), f30 = 30 f0: 2^2 of the factor 12 goes into the exponent
  __device__ __forceinline__ static Limb second(Limb s1, Limb s2, Limb f30) {
    return l_mul(l_sub(l_sub(l_mul(s1, 16), s2), f30), 3);
  }
  // s3 - 6 s2 + 15 s1 - f20, f20 = 20 f0 per axis in the sums
  __device__ __forceinline__ static Limb bracket(Limb s1, Limb s2, Limb s3, Limb f20) {
    return l_add(s3, l_sub(l_mul(l_sub(l_mul(s1, 5), l_mul(s2, 2)), 3), f20));
  }

  // Ten slots of a second-derivative field (all of degree 0): d_k, dd_p, and b^k d_k with the KO term.
  template <bool ODD>
  __device__ __forceinline__ void d2_slots(const DiffCtx& x, const char* __restrict__ L, int e, double kos,
                                           const double* b, double* dst) const {
    // sums along tile axes 1 and 2 with their halos; every load in flight before the first use
    long long r[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (t + SPLIT_PTS * j < SPLIT_NDY + SPLIT_NDZ) {
        const unsigned* const o = xw + centre(j);
        r[j][0] = ldv(L, x.b[j] + o[-2]);
        r[j][1] = ldv(L, x.b[j] + o[-1]);
        r[j][2] = ldv(L, x.b[j] + o[1]);
        r[j][3] = ldv(L, x.b[j] + o[2]);
      }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (t + SPLIT_PTS * j < SPLIT_NDY + SPLIT_NDZ)
        sDy[t + SPLIT_PTS * j] =
            p4(l_d1(l_sub(limb_of(r[j][2]), limb_of(r[j][1])), l_sub(limb_of(r[j][3]), limb_of(r[j][0]))));
    // two axes' loads in flight while the third's are issued behind the first axis
    long long n0[6], n1[6], n2[6];
    const long long nc = ldv(L, x.c);
    load(L, x, 0, n0);
    load(L, x, 1, n1);
    const Limb f0 = limb_of(nc), f30 = l_mul(f0, 30);
    Limb d1, s1, s2, s3;
    double dx, ko = 0.0;
    if (EQ) {
      Limb P1, P2, P3, yy;
      axis(n0, d1, P1, P2, P3);
      load(L, x, 2, n2);
      {
        const Limb S[2] = {d1, second(P1, P2, f30)};
        const int twos[2] = {0, 2};
        double v[2];
        limb_values<ODD>(S, e, twos, v);
        dx = v[0];
        dst[0] = v[0];
        dst[3 * SPLIT_PTS] = v[1];
      }
      axis(n1, d1, s1, s2, s3);
      yy = second(s1, s2, f30);
      P1 = l_add(P1, s1);
      P2 = l_add(P2, s2);
      P3 = l_add(P3, s3);
      axis(n2, d1, s1, s2, s3);
      P1 = l_add(P1, s1);
      P2 = l_add(P2, s2);
      P3 = l_add(P3, s3);
      const Limb S[3] = {yy, second(s1, s2, f30), bracket(P1, P2, P3, l_mul(f30, 2))};
      const int twos[3] = {2, 2, 0};
      double v[3];
      limb_values<ODD>(S, e, twos, v);
      dst[(THIN ? 8 : 6) * SPLIT_PTS] = v[0];
      dst[(THIN ? 6 : 8) * SPLIT_PTS] = v[1];
      ko = v[2];
    } else {
      const Limb f20 = l_mul(f0, 20);
      load(L, x, 2, n2);
#define COSMOS_SPLIT_AXIS(AX, SL)                                               \
  {                                                                             \
    axis(n##AX, d1, s1, s2, s3);                                                \
    const Limb S[3] = {d1, second(s1, s2, f30), bracket(s1, s2, s3, f20)};      \
    const int twos[3] = {0, 2, 0};                                              \
    double v[3];                                                                \
    limb_values<ODD>(S, e, twos, v);                                                 \
    if (AX == 0) dst[0] = dx = v[0];                                            \
    dst[SL * SPLIT_PTS] = v[1] * (x.r[AX] * x.r[AX]);                           \
    ko = fma(x.r[AX], v[2], ko);                                                \
  }
      // in the order of the grid's axes: ko is a rounded sum
      COSMOS_SPLIT_AXIS(0, 3)
      if constexpr (THIN) {
        COSMOS_SPLIT_AXIS(2, 6)
        COSMOS_SPLIT_AXIS(1, 8)
      } else {
        COSMOS_SPLIT_AXIS(1, 6)
        COSMOS_SPLIT_AXIS(2, 8)
      }
#undef COSMOS_SPLIT_AXIS
    }
    sync();
    const int4* ry = sDy + (t / SPLIT_TX) * SPLIT_XH + t % SPLIT_TX + 2;
    const int4* rz = sDy + SPLIT_NDY + (t / SPLIT_TX + 2) * SPLIT_XH + t % SPLIT_TX + 2;
    auto mixed = [](const int4* r, int st) {
      return l_d1(l_sub(q3(r[st]), q3(r[-st])), l_sub(q3(r[2 * st]), q3(r[-2 * st])));
    };
    const Limb S[5] = {q3(ry[0]), q3(rz[0]), mixed(ry, 1), mixed(rz, 1), mixed(rz, SPLIT_XH)};
    const int twos[5] = {};
    double v[5];
    limb_values<ODD>(S, e, twos, v);
    if (!EQ) {
      v[0] *= x.r[1];
      v[1] *= x.r[2];
      v[2] *= x.r[1];
      v[3] *= x.r[2];
      v[4] *= x.r[1] * x.r[2];
    }
    dst[ROW * SPLIT_PTS] = v[0];
    dst[OUT * SPLIT_PTS] = v[1];
    dst[(3 + ROW) * SPLIT_PTS] = v[2];
    dst[(3 + OUT) * SPLIT_PTS] = v[3];
    dst[7 * SPLIT_PTS] = v[4];
    double m = kos * ko;
    if (b) m = fma(b[0], dx, fma(b[SPLIT_PTS], v[ROW - 1], fma(b[2 * SPLIT_PTS], v[OUT - 1], m)));
    dst[9 * SPLIT_PTS] = m;
    sync();
  }

  __device__ __forceinline__ void d2_field(const DiffCtx& x, int f, double kos, const double* b, double* dst) const {
    const int s = ko_slot<T>(f), e = ex[s];
    const char* __restrict__ L = x.L + s * x.fb;
    if (limb_odd(e))
      d2_slots<true>(x, L, e, kos, b, dst);
    else
      d2_slots<false>(x, L, e, kos, b, dst);
  }

  // First derivatives (v[0 .. 2]) and KO bracket (v[3]) of field f.
  template <bool ODD>
  __device__ __forceinline__ void d1_values(const DiffCtx& x, const char* __restrict__ L, int e, double (&v)[4]) const {
    long long n[3][6];
    const Limb f0 = limb_of(ldv(L, x.c));
#pragma unroll
    for (int d = 0; d < 3; ++d) load(L, x, d, n[d]);
    Limb D[3], s1, s2, s3;
    if (EQ) {
      Limb P1, P2, P3;
      axis(n[0], D[0], P1, P2, P3);
      axis(n[1], D[1], s1, s2, s3);
      P1 = l_add(P1, s1);
      P2 = l_add(P2, s2);
      P3 = l_add(P3, s3);
      axis(n[2], D[2], s1, s2, s3);
      P1 = l_add(P1, s1);
      P2 = l_add(P2, s2);
      P3 = l_add(P3, s3);
      const Limb S[4] = {D[0], D[ROW], D[OUT], bracket(P1, P2, P3, l_mul(f0, 60))};
      const int twos[4] = {};
      limb_values<ODD>(S, e, twos, v);
    } else {
      const Limb f20 = l_mul(f0, 20);
      const int twos[2] = {};
      v[3] = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {  // grid axis, u that of the tile
        const int u = d == 0 ? 0 : (d == 1 ? ROW : OUT);
        axis(n[u], D[d], s1, s2, s3);
        const Limb S[2] = {D[d], bracket(s1, s2, s3, f20)};
        double w[2];
        limb_values<ODD>(S, e, twos, w);
        v[d] = w[0] * x.r[u];
        v[3] = fma(x.r[u], w[1], v[3]);
      }
    }
  }

  __device__ __forceinline__ void d1_sums(const DiffCtx& x, int f, double (&v)[4]) const {
    const int s = ko_slot<T>(f), e = ex[s];
    const char* __restrict__ L = x.L + s * x.fb;
    if (limb_odd(e))
      d1_values<true>(x, L, e, v);
    else
      d1_values<false>(x, L, e, v);
  }

  // l (b^k d_k f + KO term) of a field of degree 1 into m, its differences into dst (if given);
  // b: slots of the shift (null: not advected).
  __device__ __forceinline__ void d1_field(const DiffCtx& x, int f, const StageArgs& a, const double* b, double* dst,
                                           double* m) const {
    double v[4];
    d1_sums(x, f, v);
    if (dst) {
#pragma unroll
      for (int q = 0; q < 3; ++q) dst[q * SPLIT_PTS] = v[q];
    }
    double s = a.ap.ko * v[3];
    if (b) s = fma(b[0], v[0], fma(b[SPLIT_PTS], v[1], fma(b[2 * SPLIT_PTS], v[2], s)));
    *m = a.len * s;
  }

  // f: field of U, -1 for rho, -2 - m for field m of G
  __device__ __forceinline__ static double state(const StageArgs& a, const DiffCtx& x, int f) {
    if (f == -1) return ldd(reinterpret_cast<const char*>(a.prim), x.c);
    if (f < 0) return ldd(reinterpret_cast<const char*>(a.G) + (-2 - f) * x.fb, x.c);
    return ldd(x.U + f * x.fb, x.c);
  }

  // State values into their slots (G = the group, known at compile time, so that fields and factors are):
  // every SPLIT_GROUPS-th slot of the region, all loads in flight at once.
  template <int G>
  __device__ __forceinline__ void state_a(const StageArgs& a, const DiffCtx& x) const {
    using S = Slots<T>;
    constexpr int N = (S::A_NSTATE - G + SPLIT_GROUPS - 1) / SPLIT_GROUPS;
    double st[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      st[q] = state(a, x, S::a_state(G + q * SPLIT_GROUPS));
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int s = G + q * SPLIT_GROUPS, d = S::state_degree(S::a_state(s));
      sA[(S::A_STATE + s) * SPLIT_PTS] = d == 2 ? st[q] * a.len2 : (d == 1 ? st[q] * a.len : st[q]);
    }
  }

  template <int G>
  __device__ __forceinline__ void state_b(const StageArgs& a, double kref, const DiffCtx& x) const {
    using S = Slots<T>;
    constexpr int N = (S::B_NSTATE - G + SPLIT_GROUPS - 1) / SPLIT_GROUPS;
    double st[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      st[q] = state(a, x, S::b_state(G + q * SPLIT_GROUPS));
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int s = G + q * SPLIT_GROUPS, d = S::state_degree(S::b_state(s));
      // K - K_ref cancels: formed before any scaling
      sB[(S::B_STATE + s) * SPLIT_PTS] =
          s == S::B_KDIFF ? st[q] - kref : (d == 2 ? st[q] * a.len2 : (d == 1 ? st[q] * a.len : st[q]));
    }
  }

  __device__ __forceinline__ void fill_a(const StageArgs& a, const SplitTile& w) const {
    using S = Slots<T>;
    DiffCtx x;
    begin(a, w, x);
    if (g == 0)
      state_a<0>(a, x);
    else if (g == 1)
      state_a<1>(a, x);
    else
      state_a<2>(a, x);
    bar_sync(BAR_DIFF, SPLIT_THREADS - SPLIT_PTS);  // the shift's slots, which the groups share, are written
    const double* const b = sA + (S::A_STATE + 6) * SPLIT_PTS;
#pragma unroll 1
    for (int m = g; m < 6; m += SPLIT_GROUPS) d2_field(x, 1 + m, a.ap.ko, b, sA + (S::A_GT + 10 * m) * SPLIT_PTS);
    double* const gam = sA + (S::A_GAM + 4 * g) * SPLIT_PTS;
    d1_field(x, 14 + g, a, b, gam, gam + 3 * SPLIT_PTS);
  }

  __device__ __forceinline__ void fill_b(const StageArgs& a, double kref, const SplitTile& w) const {
    using S = Slots<T>;
    DiffCtx x;
    begin(a, w, x);
    if (g == 0)
      state_b<0>(a, kref, x);
    else if (g == 1)
      state_b<1>(a, kref, x);
    else
      state_b<2>(a, kref, x);
    // the shift's slots are those of region A, which is filled again only after every group is here
    // through; a frozen shift is not advected: beta^i (blocks 2 to 4) and B^i
    const double* const b = sA + (S::A_STATE + 6) * SPLIT_PTS;
    const double* const bs = a.ap.shift_on != 0.0 ? b : nullptr;
#pragma unroll 1
    for (int m = g; m < S::ND2B; m += SPLIT_GROUPS)
      d2_field(x, S::b_d2(m), a.ap.ko, m >= 2 && m < 5 ? bs : b, sB + 10 * m * SPLIT_PTS);
    // K and the merged advections, 1 + NM first-derivative fields: the group with fewer
    // second-derivative fields takes more of them
    constexpr int NG = T::SCALAR ? 4 : 3;
    const int lo = g * NG, hi = g == SPLIT_GROUPS - 1 ? 1 + S::NM : lo + NG;
#pragma unroll 1
    for (int m = lo; m < hi; ++m) {
      const int f = m == 0 ? 7 : S::b_m(m - 1);
      d1_field(x, f, a, f >= 21 && f < 24 ? bs : b, m == 0 ? sB + S::B_K * SPLIT_PTS : nullptr, sB + (m == 0 ? S::B_K + 3 : S::B_M + m - 1) * SPLIT_PTS);
    }
  }

  // Stage combine of the tile's outputs (in their region-B slots): fields G, G + SPLIT_GROUPS, ...
  template <int G>
  __device__ __forceinline__ void combine(const StageArgs& a, int mode, const SplitTile& w) const {
    using S = Slots<T>;
    const int i = w.i0 + t % SPLIT_TX, j = THIN ? w.k : w.j0 + t / SPLIT_TX, k = THIN ? w.j0 + t / SPLIT_TX : w.k;
    const bool valid = i < a.g.nx && (THIN ? k < a.k_hi : j < a.g.ny);
    const long fb = 8 * a.g.fstride;
    const unsigned row = 8u * (unsigned)a.g.pitch, plane = row * (unsigned)a.g.ny;
    const unsigned c = valid ? plane * (unsigned)k + row * (unsigned)j + 8u * (unsigned)i : 0u;
    const bool add = mode == MODE_S23 || mode == MODE_S4;
    const char* const u0 = mode == MODE_S4 ? reinterpret_cast<const char*>(a.U0w) : reinterpret_cast<const char*>(a.U0);
    char* const acc = reinterpret_cast<char*>(a.acc);
    char* const out = reinterpret_cast<char*>(mode == MODE_S4 ? a.U0w : a.out);
    constexpr int N = (T::NF - G + SPLIT_GROUPS - 1) / SPLIT_GROUPS;
    double u[N], ac[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {  // every load in flight before the first use
      const int f = G + q * SPLIT_GROUPS;
      u[q] = valid && mode != MODE_RHS ? *reinterpret_cast<const double*>(u0 + f * fb + c) : 0.0;
      ac[q] = valid && add ? *reinterpret_cast<const double*>(acc + f * fb + c) : 0.0;
    }
    // the fluid's fluxes: direction d of field 24 + m at 8 (4 d + m) fs
    constexpr int F = T::FLUID ? 24 + (G + SPLIT_GROUPS - 24 % SPLIT_GROUPS) % SPLIT_GROUPS : T::NF;
    constexpr int NFL = T::FLUID ? (27 - F) / SPLIT_GROUPS + 1 : 0;
    double H[NFL > 0 ? NFL : 1][6];
    if (T::FLUID) {
      const unsigned cx = c - 8u * (unsigned)i + 8u * (unsigned)wrap_index(i - 1, a.g.nx);
      const unsigned cy = c + row * (unsigned)(wrap_index(j - 1, a.g.ny) - j);
      const unsigned cz = c + plane * (unsigned)(wrap_index(k - 1, a.g.nz) - k);
#pragma unroll
      for (int q = 0; q < NFL; ++q)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const char* h = reinterpret_cast<const char*>(a.flux) + (F + q * SPLIT_GROUPS - 24 + 4 * d) * fb;
          H[q][2 * d] = valid ? ldd(h, c) : 0.0;
          H[q][2 * d + 1] = valid ? ldd(h, d == 0 ? cx : (d == 1 ? cy : cz)) : 0.0;
        }
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int f = G + q * SPLIT_GROUPS;
      // r in the units of the grid = factor inv_len of the slot's value; the factor is part
      // of the products below, except for the fluid (flux divergence), formed here
      double r = sB[T::out_slot(f) * SPLIT_PTS];
      int s = S::degree(f);
      if (T::FLUID && f >= 24 && f < 28) {
        const int m = (f - F) / SPLIT_GROUPS;
        r *= a.inv_len[s];
        s = 3;
        r -= (H[m][0] - H[m][1]) * a.c.ih[0];
        r -= (H[m][2] - H[m][3]) * a.c.ih[1];
        r -= (H[m][4] - H[m][5]) * a.c.ih[2];
      }
      double* const o = reinterpret_cast<double*>(out + f * fb + c);
      if (mode == MODE_RHS) {
        if (valid) *o = r * a.inv_len[s];
      } else if (mode == MODE_S4) {
        if (valid) *o = fma(a.cdt, fma(a.inv_len[s], r, ac[q]), u[q]);
      } else {
        const double v = fma(a.cdt_len[s], r, u[q]);
        if (valid) {
          *o = v;
          *reinterpret_cast<double*>(acc + f * fb + c) = mode == MODE_S1 ? r * a.inv_len[s] : fma(a.bk_len[s], r, ac[q]);
        }
        if (a.E_rec && !(T::FLUID && f >= 24 && f < 28)) {
          // largest biased exponent of the stored values (the next stage's reference)
          const unsigned e = valid ? (unsigned)(((unsigned long long)__double_as_longlong(v) >> 52) & 0x7FFu) : 0u;
          const unsigned m = __reduce_max_sync(0xffffffffu, e);
          if ((t & 31) == 0) atomicMax(rec + ko_slot<T>(f), (int)m);
        }
      }
    }
  }

  __device__ __forceinline__ void combine(const StageArgs& a, int mode, const SplitTile& w) const {
    if (g == 0)
      combine<0>(a, mode, w);
    else if (g == 1)
      combine<1>(a, mode, w);
    else
      combine<2>(a, mode, w);
  }
};

// The difference warps' part of the kernel below (its arguments; t: point of the tile).
template <class T, bool BATCH, bool EQ, bool THIN>
__device__ __forceinline__ void difference_warps(const StageArgs& one, const StageArgs* __restrict__ args,
                                                 const BatchTile* __restrict__ tiles, long ntiles,
                                                 const double* __restrict__ kref, int mode, int t, double* A, double* B,
                                                 int4* stage, int* tables, int* rec) {
  constexpr int NSLOT = 24 + (T::SCALAR ? 2 : 0);
  const int tx = (one.g.nx + SPLIT_TX - 1) / SPLIT_TX;
  const int ty = ((THIN ? one.k_hi - one.k_lo : one.g.ny) + SPLIT_TY - 1) / SPLIT_TY;
  auto tile_at = [&](long w) {
    if (BATCH) {
      const BatchTile b = tiles[w];
      return SplitTile{b.a * SPLIT_TX, b.b * SPLIT_TY, b.c, b.inst};
    }
    const int q = (int)w;  // tiles of one grid: less than 2^31
    const int j0 = q / tx % ty * SPLIT_TY, k = q / (tx * ty);
    return SplitTile{q % tx * SPLIT_TX, THIN ? j0 + one.k_lo : j0, THIN ? k : k + one.k_lo, 0};
  };
  const int g = __shfl_sync(0xffffffffu, (int)threadIdx.x / SPLIT_PTS - 1, 0);  // uniform, and known to be
  int* const tab = tables + g * 80;
  int4* const st = stage + g * (SPLIT_NDY + SPLIT_NDZ);
  const DiffGroup<T, EQ, THIN> d{t, g, A + t, B + t, st, reinterpret_cast<unsigned*>(tab), tab + 48, rec};
  auto flush = [&](const StageArgs& a) {  // the record of the instance that ends here
    bar_sync(BAR_DIFF, SPLIT_THREADS - SPLIT_PTS);
    if (g == 0 && t < NSLOT && a.E_rec && mode != MODE_RHS && mode != MODE_S4) {
      atomicMax(a.E_rec + 32 * t, (unsigned)rec[t]);
      rec[t] = 0;
    }
    if (!BATCH && g == 0 && a.E_rec && a.E_next) {
      // the last block to end (no block waits for another) leaves the record as the exponents of
      // the next stage, and clean; every block has read the exponents of this stage by then
      __threadfence();
      bar_sync(BAR_GROUP, SPLIT_PTS);
      if (t == 0) rec[31] = (int)atomicAdd(a.E_rec + 1, 1u);
      bar_sync(BAR_GROUP, SPLIT_PTS);
      if (rec[31] == (int)gridDim.x - 1) {
        __threadfence();
        if (t < NSLOT) a.E_next[t] = (int)atomicExch(a.E_rec + 32 * t, 0u);
        if (t == 0) a.E_rec[1] = 0u;
      }
    }
  };
  if (blockIdx.x >= ntiles) return;
  SplitTile cur = tile_at(blockIdx.x);
  d.fill_a(BATCH ? args[cur.inst] : one, cur);
  bar_arrive(BAR_FULL_A, SPLIT_THREADS);
  for (long w = blockIdx.x; w < ntiles; w += gridDim.x) {
    const StageArgs& a = BATCH ? args[cur.inst] : one;
    d.fill_b(a, BATCH ? kref[cur.inst] : one.ap.Kref, cur);
    bar_arrive(BAR_FULL_B, SPLIT_THREADS);
    const bool more = w + gridDim.x < ntiles;
    SplitTile nxt = cur;
    if (more) {
      nxt = tile_at(w + gridDim.x);
      bar_sync(BAR_FREE_A, SPLIT_THREADS);
      d.fill_a(BATCH ? args[nxt.inst] : one, nxt);
      bar_arrive(BAR_FULL_A, SPLIT_THREADS);
    }
    bar_sync(BAR_DONE_B, SPLIT_THREADS);
    d.combine(a, mode, cur);
    // no group refills region B (or its record) while another still reads it
    if (!more || nxt.inst != cur.inst) flush(a);
    bar_sync(BAR_DIFF, SPLIT_THREADS - SPLIT_PTS);
    cur = nxt;
  }
}

// BATCH: tiles from a list, arguments per instance with K_ref in kref; else
// the planes k_lo .. of the grid of `one`.  THIN: tiles along z, of every grid.
template <class T, bool BATCH, bool EQ, bool THIN>
__global__ void __launch_bounds__(SPLIT_THREADS, 1)
    split_stage_kernel(const __grid_constant__ StageArgs one, const StageArgs* __restrict__ args,
                       const BatchTile* __restrict__ tiles, long ntiles, const double* __restrict__ kref, int mode) {
  extern __shared__ double smem[];
  using S = Slots<T>;
  double* const A = smem;
  double* const B = smem + S::A * SPLIT_PTS;
  int4* const stage = reinterpret_cast<int4*>(B + S::B * SPLIT_PTS);
  int* const tables = reinterpret_cast<int*>(stage + SPLIT_GROUPS * (SPLIT_NDY + SPLIT_NDZ));
  int* const rec = tables + SPLIT_GROUPS * 80;
  if (threadIdx.x < 32) rec[threadIdx.x] = 0;
  grid_wait();
  __syncthreads();
  const int t = threadIdx.x % SPLIT_PTS;
  if (threadIdx.x < SPLIT_PTS) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(SPLIT_REG_ALG));
    const Fp64Regs k = fp64_regs();
    for (long w = blockIdx.x; w < ntiles; w += gridDim.x) {
      const bool more = w + gridDim.x < ntiles;
      AlgebraParams ap = one.ap;
      if (BATCH) ap = args[tiles[w].inst].ap;
      bar_sync(BAR_FULL_A, SPLIT_THREADS);
      T::rhs_split(SlotIn{A + t}, SlotIn{B + t}, SlotOut<T>{B + t},
                   [&] {
                     if (more) bar_arrive(BAR_FREE_A, SPLIT_THREADS);
                     bar_sync(BAR_FULL_B, SPLIT_THREADS);
                   },
                   ap, k);
      bar_arrive(BAR_DONE_B, SPLIT_THREADS);
    }
    return;
  }
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SPLIT_REG_DIFF));
  difference_warps<T, BATCH, EQ, THIN>(one, args, tiles, ntiles, kref, mode, t, A, B, stage, tables, rec);
}

// One block per SM, no more than there are tiles.
template <class T, bool BATCH, bool EQ, bool THIN>
cudaError_t launch_split_as(const StageArgs& one, const StageArgs* args, const BatchTile* tiles, long ntiles,
                            const double* kref, int mode, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  constexpr size_t bytes = split_smem_bytes<T>();
  static_assert(bytes <= 232448, "shared memory of one block");
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(split_stage_kernel<T, BATCH, EQ, THIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  const int blocks = (int)(ntiles < sms ? ntiles : sms);
  return launch_early(split_stage_kernel<T, BATCH, EQ, THIN>, dim3(blocks), SPLIT_THREADS, bytes, s, one, args, tiles, ntiles,
                      kref, mode);
}

// eq: equal spacing, thin: tiles along z (of every grid of a batch)
template <class T, bool BATCH>
cudaError_t launch_split(const StageArgs& one, const StageArgs* args, const BatchTile* tiles, long ntiles,
                         const double* kref, int mode, bool eq, bool thin, cudaStream_t s) {
  if (ntiles <= 0) return cudaSuccess;
  if (thin)
    return eq ? launch_split_as<T, BATCH, true, true>(one, args, tiles, ntiles, kref, mode, s)
              : launch_split_as<T, BATCH, false, true>(one, args, tiles, ntiles, kref, mode, s);
  return eq ? launch_split_as<T, BATCH, true, false>(one, args, tiles, ntiles, kref, mode, s)
            : launch_split_as<T, BATCH, false, false>(one, args, tiles, ntiles, kref, mode, s);
}

}  // namespace cosmos
