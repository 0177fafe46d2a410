// Internal definitions shared by the CUDA translation units of libcosmos_gb300.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "../../include/cosmos.h"
#include "fp64_regs.cuh"
#include "generated/bssn_algebra.cuh"
#include "generated/fluid_algebra.cuh"

namespace cosmos {

// A kernel launched with launch_early may be on the chip before its predecessor in the stream has ended: as
// soon as every block of that has passed grid_trigger, or ended.  So its first act is grid_wait, in every
// thread, which ends when the predecessor has, with all that it wrote to be seen.  That hides a launch behind
// the tail of the kernel before it: a 32^3 step 364 -> 353 us, 64^3 with the fluid 3.925 -> 3.898 ms.
// Only the exponent scan triggers by itself.  The limb copy at its start: a 32^3 step 352 us, but a 256^3 one
// 127.8 instead of 127.1 ms; the stage kernel from its last tile on: 368 us.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_early(void (*kernel)(P...), dim3 grid, int threads, size_t bytes, cudaStream_t s, A... args) {
  cudaLaunchAttribute early = {};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = bytes;
  c.stream = s;
  c.attrs = &early;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

constexpr double PI = 3.14159265358979323846;
constexpr int BX = 32;  // threads per block along x (one warp = one row)
constexpr int BY = 4;   // rows per block
#ifndef COSMOS_DERIV_ROWS
#define COSMOS_DERIV_ROWS 8
#endif
constexpr int DBY = COSMOS_DERIV_ROWS;  // rows per block of the reverse mode's derivative pass
// tile of one z-plane in the stage kernel (stage_split.cuh), one point per algebra thread
constexpr int SPLIT_TX = 16, SPLIT_TY = 8;

// Grid description as the kernels see it.
struct DevGrid {
  int nx, ny, nz, pitch;
  long fstride;  // doubles between fields
  double h[3];
};

// Periodic neighbour offsets of one point for offsets -3..3 per direction,
// already multiplied by the memory stride of that direction.
struct Nbr {
  long x[7], y[7], z[7];
  long c;  // offset of the point itself
};

__device__ __forceinline__ int wrap_index(int a, int n) {
  a %= n;
  return a < 0 ? a + n : a;
}

__device__ __forceinline__ Nbr make_nbr(const DevGrid& g, int i, int j, int k) {
  Nbr n;
  const long row = g.pitch, plane = (long)g.pitch * g.ny;
#pragma unroll
  for (int o = -3; o <= 3; ++o) {
    n.x[o + 3] = wrap_index(i + o, g.nx);
    n.y[o + 3] = wrap_index(j + o, g.ny) * row;
    n.z[o + 3] = wrap_index(k + o, g.nz) * plane;
  }
  n.c = n.z[3] + n.y[3] + n.x[3];
  return n;
}

// Offset of the point displaced by (dx, dy, dz), |d| <= 3.
__device__ __forceinline__ long at(const Nbr& n, int dx, int dy, int dz) {
  return n.z[dz + 3] + n.y[dy + 3] + n.x[dx + 3];
}

__device__ __forceinline__ double ldg(const double* __restrict__ p, long o) { return __ldg(p + o); }

// Stencil coefficients derived on the host from the grid spacing.
struct Coef {
  double d1a[3], d1b[3];  // D1 = a (f+1 - f-1) - b (f+2 - f-2):   a = 8/(12h), b = 1/(12h)
  double d2a[3], d2b[3];  // D2 = a s1 - b s2:                         a = 16/(12h^2), b = 1/(12h^2)
  double mix[3];          // mixed xy, xz, yz:  1/(144 h_a h_b)
  double ko[3];           // sigma/(64 h_d)
  double ih[3];           // 1/h_d (flux divergence)
};

// Tiles of a plane of few rows run along z instead of y: of SPLIT_TY = 8 rows a plane of 1 to 3 leaves more than
// half without a point, and a tile takes its time all the same.  A stage of 256 x 1 x 256: 907 -> 160 us, of
// 256 x 3 x 256: 938 -> 422.  From 4 rows on the tiles run along y, which is the form measured everywhere else.
inline bool thin_tiles(const DevGrid& g) { return g.ny < SPLIT_TY / 2 && g.nz > g.ny; }
// Tiles of k_cnt planes of a grid.
inline long stage_tiles(const DevGrid& g, int k_cnt) {
  const bool thin = thin_tiles(g);
  return (long)((g.nx + SPLIT_TX - 1) / SPLIT_TX) * (((thin ? k_cnt : g.ny) + SPLIT_TY - 1) / SPLIT_TY) * (thin ? g.ny : k_cnt);
}

Coef make_coef(const cosmos_grid* g, double sigma);
DevGrid make_devgrid(const cosmos_grid* g);
double K_ref(const cosmos_params* p, double t);                 // background trace at time t
AlgebraParams algebra_params(const cosmos_params* p, double t); // runtime parameters of the algebra
int validate(const cosmos_grid* g, const cosmos_params* p);     // COSMOS_OK or COSMOS_EINVAL
// The same for a call that launches the stage kernel: its offsets within a field are 32-bit counts of bytes
// (stage_split.cuh), so a field has at most 2^29 points.
int validate_stage(const cosmos_grid* g, const cosmos_params* p);

// RK4 stage modes
enum StageMode { MODE_RHS = 0, MODE_S1 = 1, MODE_S23 = 2, MODE_S4 = 3 };

struct StageArgs {
  DevGrid g;
  Coef c;
  AlgebraParams ap;                // eta and ko in the units of stage_split.cuh (l = 12 h_x), Kref as given
  const double* __restrict__ U;    // stencil input (stage state)
  const double* __restrict__ U0;   // U_n (pointwise) -- MODE_S1/S23
  double* U0w;                     // U_n written in MODE_S4
  double* out;                     // MODE_RHS: rhs;  MODE_S1/S23: U_next
  double* acc;                     // accumulator
  const double* __restrict__ prim; // fluid primitives [4][pts] (fluid only)
  const double* __restrict__ flux; // fluid face fluxes [3][4][pts] (fluid only)
  double* D;                       // finite differences of U for the reverse mode (ideriv_kernel only)
  long dfs;                        // their field stride: g.fstride, an argument of its own because ideriv_kernel is faster
                                   // so (45 x 33 x 28: 57.1 -> 53.9 us; of a 402 us VJP 398.7)
  double cdt;                      // dt * c_{s+1}, or dt/6 in MODE_S4
  double len, len2;                // l = 12 h_x, l^2
  double inv_len[4];               // 1/l, 1/l^2, 1/l^3 (per degree of the field, stage_split.cuh), 1
  double cdt_len[4], bk_len[4];    // cdt and the accumulator weight (2 for stages 2, 3) times those
  double ratio[3];                 // h_x / h_d
  int eq;                          // equal spacing
  int k_lo, k_hi;                  // planes k_lo .. k_hi - 1
  const long long* __restrict__ L; // limb copy of U (stage_int.cuh)
  const int* __restrict__ E;       // reference exponent of each limb slot
  const double* __restrict__ G;    // inverse conformal metric (6 fields) and 1/chi of U (launch_to_limbs)
  unsigned* E_rec;                 // stages 1-3: records the largest biased exponent of each limb
                                   // slot of U_next at E_rec[32 slot] (null: no record)
  int* E_next;                     // one grid: the block that ends last moves the record there and clears it
                                   // (E_rec[1] counts the blocks that have ended; null: it stays)
};
// Fills the units of `a` (its grid, ap, cdt given) for dissipation sigma.
void set_units(StageArgs* a, double sigma, double bk);

// Doubles per point of the finite differences that the reverse mode keeps:
// first and second derivatives.
inline int nder(int scalar) { return 3 * (24 + 2 * scalar) + 6 * (11 + scalar); }

// One work item of a batch: instance `inst`; for 2D tiles (a, b, c) = (block
// column, block row, z-plane), for linear runs a = first point index.
struct BatchTile {
  int inst, a, b, c;
};
enum BatchMapping { BATCH_MAP_TILE2D = 0, BATCH_MAP_LINEAR = 1 };

struct ConstraintArgs {
  DevGrid g;
  Coef c;
  AlgebraParams ap;
  const double* __restrict__ U;
  const double* __restrict__ prim;
  double* hm;        // [4][pts] or null
  double* partial;   // [nblocks][8]: sum of squares (4) and max abs (4)
};

#ifndef COSMOS_IDERIV_MIN_BLOCKS
#define COSMOS_IDERIV_MIN_BLOCKS 4  // integer derivative pass: resident blocks (of BX x DBY threads) per SM
#endif

// Launchers implemented per matter variant (stage_<variant>.cu).
cudaError_t launch_stage_vac(const StageArgs& a, int mode, cudaStream_t s);
cudaError_t launch_stage_fluid(const StageArgs& a, int mode, cudaStream_t s);
cudaError_t launch_stage_scalar(const StageArgs& a, int mode, cudaStream_t s);
cudaError_t launch_stage_fluid_scalar(const StageArgs& a, int mode, cudaStream_t s);
cudaError_t launch_deriv_vac(const StageArgs& a, cudaStream_t s);  // finite differences into a.D
cudaError_t launch_deriv_fluid(const StageArgs& a, cudaStream_t s);
cudaError_t launch_deriv_scalar(const StageArgs& a, cudaStream_t s);
cudaError_t launch_deriv_fluid_scalar(const StageArgs& a, cudaStream_t s);
// batched stage over the tile list (SPLIT_TX x SPLIT_TY of one plane), K_ref per instance;
// eq, thin: those of every grid of the list (a.eq, thin_tiles)
typedef cudaError_t (*BatchStageLauncher)(const StageArgs*, const BatchTile*, long, const double*, int, bool, bool, cudaStream_t);
cudaError_t launch_batch_stage_vac(const StageArgs*, const BatchTile*, long, const double*, int, bool, bool, cudaStream_t);
cudaError_t launch_batch_stage_fluid(const StageArgs*, const BatchTile*, long, const double*, int, bool, bool, cudaStream_t);
cudaError_t launch_batch_stage_scalar(const StageArgs*, const BatchTile*, long, const double*, int, bool, bool, cudaStream_t);
cudaError_t launch_batch_stage_fluid_scalar(const StageArgs*, const BatchTile*, long, const double*, int, bool,
                                            bool, cudaStream_t);
cudaError_t launch_batch_fluid(const StageArgs* args, const BatchTile* tiles, long ntiles, int mapping, double w,
                               dim3 grid, dim3 block, cudaStream_t s);
cudaError_t launch_constraints_vac(const ConstraintArgs& a, cudaStream_t s);
cudaError_t launch_constraints_fluid(const ConstraintArgs& a, cudaStream_t s);
cudaError_t launch_constraints_scalar(const ConstraintArgs& a, cudaStream_t s);
cudaError_t launch_constraints_fluid_scalar(const ConstraintArgs& a, cudaStream_t s);

// adjoint_<variant>.cu
struct VjpArgs;
cudaError_t launch_vjp_vac(const VjpArgs& a, cudaStream_t s);
cudaError_t launch_vjp_fluid(const VjpArgs& a, cudaStream_t s);
cudaError_t launch_vjp_scalar(const VjpArgs& a, cudaStream_t s);
cudaError_t launch_vjp_fluid_scalar(const VjpArgs& a, cudaStream_t s);
cudaError_t launch_init_zeta_vjp(const DevGrid& g, const Coef& c, const AlgebraParams& ap, const double* U,
                                 const double* lam, double* CB10, int fluid, double* zbar, cudaStream_t s);

// limbs.cu: exponents of limb slots s_lo .. s_hi - 1 of U and its limb copy
// (slot s = field s, or s + 4 past the fluid fields when the fluid is on), and, if
// G is given and slot 6 is among them (fields 0 .. 6 are there then), the inverse
// conformal metric and 1/chi into G (7 fields)
cudaError_t launch_limbs(const DevGrid& g, const double* U, int fluid, int s_lo, int s_hi, int* E, long long* L,
                         double* G, cudaStream_t s);
// the limb copy (and G) with given exponents E (no scan), left in keep too unless that is null; the exponent scan alone
cudaError_t launch_to_limbs(const DevGrid& g, const double* U, int fluid, int s_lo, int s_hi, const int* E, int* keep,
                            long long* L, double* G, cudaStream_t s);
cudaError_t launch_field_exponents(const DevGrid& g, const double* U, int fluid, int s_lo, int s_hi, int* E,
                                   cudaStream_t s);
// E[s] = rec[32 s] and rec[32 s] = 0 for s < nslot (the exponents a stage recorded)
cudaError_t launch_exponents_from_record(unsigned* rec, int* E, int nslot, cudaStream_t s);
// the batched limb copy with the exponents already in args[i].E; blocks: batch_limb_blocks of the instance with most points
unsigned batch_limb_blocks(const DevGrid& largest);
cudaError_t launch_batch_to_limbs(const StageArgs* args, int n, unsigned blocks, int nslot, int fluid, cudaStream_t s);
// the same for every instance of a batch (args[i] = instance i's stage arguments;
// E_all = the n x nslot exponents, contiguous, args[i].E = E_all + i nslot)
cudaError_t launch_batch_limbs(const StageArgs* args, int n, unsigned blocks, int nslot, int fluid, int* E_all,
                               cudaStream_t s);

// fluid.cu
cudaError_t launch_fluid_prim(const DevGrid& g, const double* U, double* prim, double w, cudaStream_t s);
cudaError_t launch_fluid_flux(const DevGrid& g, const double* U, const double* prim, double* flux, double w,
                              int nf_offset_fluid, cudaStream_t s);

inline dim3 point_grid(const DevGrid& g) { return dim3((g.nx + BX - 1) / BX, (g.ny + BY - 1) / BY, g.nz); }

// A point per thread of the reverse mode's and the fluid's FP64 kernels, in runs (one block each) of the whole
// grid, so that every lane has one: BX x BY tiles of a plane of 45 x 33 points leave 42% of the lanes without
// (a VJP of 45 x 33 x 28: 698 -> 473 us), of 97 x 80 points 24% (an RK4 step with fluid and scalar of
// 97 x 80 x 66: 10.47 -> 9.68 ms).  On a plane that the tiles cover exactly both are the same work; there the fluid
// kernels keep the tiles, which take no division (128^3: 0.3% of a step).
inline bool tiles_exact(const DevGrid& g) { return g.nx % BX == 0 && g.ny % BY == 0; }
inline unsigned flat_grid(const DevGrid& g, int threads) {
  return (unsigned)(((long)g.nx * g.ny * g.nz + threads - 1) / threads);
}
template <bool FLAT>
__device__ __forceinline__ bool point_of(const DevGrid& g, int& i, int& j, int& k) {
  if (FLAT) {
    const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;  // grids have less than 2^31 points
    const unsigned row = p / (unsigned)g.nx;
    i = (int)(p - row * (unsigned)g.nx);
    k = (int)(row / (unsigned)g.ny);
    j = (int)(row - (unsigned)k * (unsigned)g.ny);
    return k < g.nz;
  }
  i = blockIdx.x * BX + threadIdx.x;
  j = blockIdx.y * BY + threadIdx.y;
  k = blockIdx.z;
  return i < g.nx && j < g.ny;
}
// reverse mode's derivative pass: one BX x DBY tile of one z-plane per block
inline dim3 ideriv_grid(const DevGrid& g) { return dim3((g.nx + BX - 1) / BX, (g.ny + DBY - 1) / DBY, g.nz); }
// Every index the integer derivative pass forms for a tile lies in [-n, 2n)
// along each axis, so one compare and select wraps it (stage_int.cuh,
// wrap_near): x in [i0 - 3, i0 + BX + 2] with i0 <= nx - 1, y in
// [j0 - 3, j0 + DBY + 2] with j0 <= ny - 1, z in [k - 3, k + 3] with k <= nz - 1.
__host__ __device__ inline bool near_indices(const DevGrid& g) { return g.nx >= BX + 3 && g.ny >= DBY + 3 && g.nz >= 3; }

}  // namespace cosmos
