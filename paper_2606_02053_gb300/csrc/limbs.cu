// Pre-pass of the integer differences (stage_int.cuh): the reference
// exponent of every limb slot, then the limb copy of the stage state.
//
// Both are passes over memory.  A slot is taken as one flat run of its
// fstride values (without the padding columns), LIMB_RUN values per block and
// turn, LIMB_EACH of them in flight per thread.  By rows, a 32-point row kept half
// of a block idle: 24 fields of 32^3: copy 15.3 -> 4.7 us, scan 33 -> 5.3; 64^3: copy
// 50 -> 14 us; 256^3: 0.89 ms, 7.2 TB/s.  With the inverse metric and 1/chi beside it
// 256^3 takes 1.1 ms, and the step, whose algebra no longer forms them, 132.6 ->
// 127.1 ms (generic 250 x 198 x 203: 80.3 -> 78.2).
#include "stage_kernel.cuh"

namespace cosmos {

constexpr int LIMB_THREADS = 256, LIMB_EACH = 4, LIMB_RUN = LIMB_THREADS * LIMB_EACH;

// Offset p of a slot's flat run stands for a point of the grid (not for a padding column or beyond the end).
template <bool PADDED>
__device__ __forceinline__ bool on_grid(const DevGrid& g, long p) {
  return p < g.fstride && !(PADDED && (unsigned)p % (unsigned)g.pitch >= (unsigned)g.nx);  // fstride < 2^31
}

// Largest biased exponent over the points of one slot, into *E (one atomic per block).
__device__ __forceinline__ void scan_slot(const DevGrid& g, const double* __restrict__ F, unsigned* E) {
  __shared__ unsigned top[LIMB_THREADS / 32];
  unsigned m = 0;
  const bool padded = g.pitch != g.nx;
  for (long o = (long)blockIdx.x * LIMB_RUN + threadIdx.x; o - threadIdx.x < g.fstride; o += (long)gridDim.x * LIMB_RUN) {
    unsigned long long b[LIMB_EACH];
#pragma unroll
    for (int q = 0; q < LIMB_EACH; ++q) {
      const long p = o + q * LIMB_THREADS;
      const bool on = padded ? on_grid<true>(g, p) : on_grid<false>(g, p);
      b[q] = on ? (unsigned long long)__double_as_longlong(__ldg(F + p)) : 0ull;
    }
#pragma unroll
    for (int q = 0; q < LIMB_EACH; ++q) m = max(m, (unsigned)((b[q] >> 52) & 0x7FF));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) top[threadIdx.x / 32] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < LIMB_THREADS / 32; ++w) m = max(m, top[w]);
    atomicMax(E, m);
  }
}

// PADDED: pitch > nx
template <bool PADDED>
__device__ __forceinline__ void copy_slot(const DevGrid& g, const double* __restrict__ F, int e_ref,
                                          long long* __restrict__ L, long first, long stride) {
  const unsigned pitch = (unsigned)g.pitch, step = PADDED ? LIMB_THREADS % pitch : 0u;
  for (long o = first * LIMB_RUN + threadIdx.x; o < g.fstride; o += stride * LIMB_RUN) {
    double v[LIMB_EACH];
    bool on[LIMB_EACH];
    unsigned col = PADDED ? (unsigned)o % pitch : 0u;  // one division for the run's values, 15% of the copy with one each
#pragma unroll
    for (int q = 0; q < LIMB_EACH; ++q) {
      on[q] = o + q * LIMB_THREADS < g.fstride && !(PADDED && col >= (unsigned)g.nx);
      col += step;
      if (PADDED && col >= pitch) col -= pitch;
      v[q] = on[q] ? __ldg(F + o + q * LIMB_THREADS) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < LIMB_EACH; ++q)
      if (on[q]) L[o + q * LIMB_THREADS] = to_limbs(v[q], e_ref);
  }
}

// Limb copies of chi and the conformal metric (slots 0 .. 6) and, of the same loads, the inverse metric and
// 1/chi of each point into G: blocks first, first + stride, .. of LIMB_THREADS points.  The stage's algebra
// has one warp per scheduler, which the latency of the determinant and its reciprocal bounds; here many warps
// are in flight and the FP64 instructions run beside the copies of the other slots, whose bound is memory.
template <bool PADDED>
__device__ __forceinline__ void copy_metric(const DevGrid& g, const double* __restrict__ U, const int* __restrict__ E,
                                            long long* __restrict__ L, double* __restrict__ G, long first, long stride) {
  const Fp64Regs k = fp64_regs();
  const long fs = g.fstride;
  for (long o = first * LIMB_THREADS + threadIdx.x; o < fs; o += stride * LIMB_THREADS) {
    if (PADDED && !on_grid<true>(g, o)) continue;
    double v[7];
#pragma unroll
    for (int m = 0; m < 7; ++m) v[m] = __ldg(U + m * fs + o);
    if (L) {  // null: G alone
#pragma unroll
      for (int m = 0; m < 7; ++m) L[m * fs + o] = to_limbs(v[m], max(E[m], 1));
    }
    const double* q = v + 1;  // xx xy xz yy yz zz
    const double c[6] = {fma(-q[4], q[4], mul3(q[3], q[5], k)), fma(-q[1], q[5], mul3(q[2], q[4], k)),
                         fma(-q[2], q[3], mul3(q[1], q[4], k)), fma(-q[2], q[2], mul3(q[0], q[5], k)),
                         fma(-q[0], q[4], mul3(q[1], q[2], k)), fma(-q[1], q[1], mul3(q[0], q[3], k))};
    const double idet = 1.0 / fma(q[2], c[2], fma(q[1], c[1], mul3(q[0], c[0], k)));
#pragma unroll
    for (int m = 0; m < 6; ++m) G[m * fs + o] = mul3(c[m], idet, k);
    G[6 * fs + o] = 1.0 / v[0];
  }
}

// Work of one block in a pass over all slots below s_hi (> 6) with G: of every LIMB_EACH + s_hi - 7 blocks, the
// first LIMB_EACH take LIMB_RUN points of chi and the metric, the others LIMB_RUN points of one slot each, so
// that the two kinds are on an SM together.
template <bool PADDED>
__device__ __forceinline__ void copy_all(const DevGrid& g, const double* __restrict__ U, int s_hi, int fluid,
                                         const int* __restrict__ E, long long* __restrict__ L, double* __restrict__ G) {
  const int each = LIMB_EACH + s_hi - 7, q = blockIdx.x % each;
  const long c = blockIdx.x / each, nc = gridDim.x / each;
  if (q < LIMB_EACH) {
    copy_metric<PADDED>(g, U, E, L, G, c * LIMB_EACH + q, nc * LIMB_EACH);
  } else {
    const int s = 7 + q - LIMB_EACH;
    copy_slot<PADDED>(g, U + (long)limb_field(s, fluid) * g.fstride, max(E[s], 1), L + (long)s * g.fstride, c, nc);
  }
}

// blockIdx.y = slot (from s_lo)
__global__ void __launch_bounds__(LIMB_THREADS) field_exponent_kernel(const DevGrid g, const double* __restrict__ U,
                                                                      int s_lo, int fluid, int* __restrict__ E) {
  const int s = s_lo + blockIdx.y;
  grid_trigger();
  scan_slot(g, U + (long)limb_field(s, fluid) * g.fstride, (unsigned*)E + s);
}

template <bool PADDED>
__global__ void __launch_bounds__(LIMB_THREADS) to_limbs_kernel(const DevGrid g, const double* __restrict__ U, int s_lo,
                                                                int fluid, const int* __restrict__ E,
                                                                long long* __restrict__ L) {
  const int s = s_lo + blockIdx.y;
  copy_slot<PADDED>(g, U + (long)limb_field(s, fluid) * g.fstride, max(E[s], 1), L + (long)s * g.fstride, blockIdx.x,
                    gridDim.x);
}

// all slots below s_hi (> 6) with G; keep: E is left there too (null: not)
template <bool PADDED>
__global__ void __launch_bounds__(LIMB_THREADS) to_limbs_all_kernel(const DevGrid g, const double* __restrict__ U,
                                                                    int s_hi, int fluid, const int* __restrict__ E,
                                                                    int* __restrict__ keep, long long* __restrict__ L,
                                                                    double* __restrict__ G) {
  grid_wait();
  if (keep && blockIdx.x == 0 && threadIdx.x < s_hi) keep[threadIdx.x] = E[threadIdx.x];
  copy_all<PADDED>(g, U, s_hi, fluid, E, L, G);
}

// G alone
template <bool PADDED>
__global__ void __launch_bounds__(LIMB_THREADS) metric_kernel(const DevGrid g, const double* __restrict__ U,
                                                              double* __restrict__ G) {
  copy_metric<PADDED>(g, U, nullptr, nullptr, G, blockIdx.x, gridDim.x);
}

// The same for a batch: blockIdx.z = instance; the arguments of instance i are
// args[i] (its stage input U, grid, limb copy and exponents).
__global__ void __launch_bounds__(LIMB_THREADS) batch_field_exponent_kernel(const StageArgs* __restrict__ args, int fluid) {
  const StageArgs& a = args[blockIdx.z];
  const DevGrid g = a.g;
  scan_slot(g, a.U + (long)limb_field(blockIdx.y, fluid) * g.fstride, (unsigned*)a.E + blockIdx.y);
}

// blockIdx.y = instance
__global__ void __launch_bounds__(LIMB_THREADS) batch_to_limbs_kernel(const StageArgs* __restrict__ args, int nslot,
                                                                      int fluid) {
  grid_wait();
  const StageArgs& a = args[blockIdx.y];
  if (a.g.pitch == a.g.nx)
    copy_all<false>(a.g, a.U, nslot, fluid, a.E, const_cast<long long*>(a.L), const_cast<double*>(a.G));
  else
    copy_all<true>(a.g, a.U, nslot, fluid, a.E, const_cast<long long*>(a.L), const_cast<double*>(a.G));
}

// Blocks along a slot: the copy has no turn to repeat up to the largest grids;
// the scan repeats, so that a block's one atomic stands for many values.
static unsigned copy_blocks(const DevGrid& g) { return (unsigned)((g.fstride + LIMB_RUN - 1) / LIMB_RUN); }
static unsigned scan_blocks(const DevGrid& g) {
  const unsigned b = copy_blocks(g);
  return b < 128 ? b : 128;
}

// Blocks along a slot of every instance of a batch: what its largest needs, but no more than 128 (others repeat).
// 128 for grids of any size were 2688 blocks an instance in the copy, nearly all without a point on small ones:
// a step of 1024 grids of 4^3 22.3 ms, with one each 3.8; of 64 grids of 16^3 3.2 ms, with four 2.1.
unsigned batch_limb_blocks(const DevGrid& largest) {
  const unsigned b = copy_blocks(largest);
  return b < 128 ? b : 128;
}

cudaError_t launch_batch_limbs(const StageArgs* args, int n, unsigned blocks, int nslot, int fluid, int* E_all,
                               cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(E_all, 0, sizeof(int) * (size_t)n * nslot, s);
  if (e != cudaSuccess) return e;
  batch_field_exponent_kernel<<<dim3(blocks, (unsigned)nslot, (unsigned)n), LIMB_THREADS, 0, s>>>(args, fluid);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return launch_batch_to_limbs(args, n, blocks, nslot, fluid, s);
}

cudaError_t launch_limbs(const DevGrid& g, const double* U, int fluid, int s_lo, int s_hi, int* E, long long* L,
                         double* G, cudaStream_t s) {
  const cudaError_t e = launch_field_exponents(g, U, fluid, s_lo, s_hi, E, s);
  return e != cudaSuccess ? e : launch_to_limbs(g, U, fluid, s_lo, s_hi, E, nullptr, L, G, s);
}

// The limb copy of slots s_lo .. s_hi - 1 with the reference exponents given
// in E (no scan), which are left in keep too unless that is null.
cudaError_t launch_to_limbs(const DevGrid& g, const double* U, int fluid, int s_lo, int s_hi, const int* E, int* keep,
                            long long* L, double* G, cudaStream_t s) {
  if (s_hi <= s_lo) return cudaSuccess;
  const unsigned blocks = copy_blocks(g);
  const bool padded = g.pitch != g.nx;  // kernels of their own: with the test in one, the unpadded copy took 3% longer
  if (G && s_lo == 0 && s_hi > 6) {
    return launch_early(padded ? to_limbs_all_kernel<true> : to_limbs_all_kernel<false>,
                        dim3(blocks * (unsigned)(LIMB_EACH + s_hi - 7)), LIMB_THREADS, 0, s, g, U, s_hi, fluid, E, keep, L, G);
  }
  if (keep) {
    const cudaError_t e = cudaMemcpyAsync(keep + s_lo, E + s_lo, sizeof(int) * (s_hi - s_lo), cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
  }
  if (G && s_lo <= 6 && s_hi > 6) {
    (padded ? metric_kernel<true> : metric_kernel<false>)<<<blocks * LIMB_EACH, LIMB_THREADS, 0, s>>>(g, U, G);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  (padded ? to_limbs_kernel<true> : to_limbs_kernel<false>)<<<dim3(blocks, (unsigned)(s_hi - s_lo)), LIMB_THREADS, 0, s>>>(
      g, U, s_lo, fluid, E, L);
  return cudaGetLastError();
}

// Only the exponent scan of slots s_lo .. s_hi - 1 into E.
cudaError_t launch_field_exponents(const DevGrid& g, const double* U, int fluid, int s_lo, int s_hi, int* E,
                                   cudaStream_t s) {
  if (s_hi <= s_lo) return cudaSuccess;
  const cudaError_t e = cudaMemsetAsync(E + s_lo, 0, sizeof(int) * (s_hi - s_lo), s);
  if (e != cudaSuccess) return e;
  field_exponent_kernel<<<dim3(scan_blocks(g), (unsigned)(s_hi - s_lo)), LIMB_THREADS, 0, s>>>(g, U, s_lo, fluid, E);
  return cudaGetLastError();
}

__global__ void exponents_from_record_kernel(unsigned* __restrict__ rec, int* __restrict__ E, int nslot) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nslot; s += gridDim.x * blockDim.x) {
    E[s] = (int)rec[32 * s];
    rec[32 * s] = 0u;
  }
}

cudaError_t launch_exponents_from_record(unsigned* rec, int* E, int nslot, cudaStream_t s) {
  exponents_from_record_kernel<<<(nslot + 255) / 256, 256, 0, s>>>(rec, E, nslot);
  return cudaGetLastError();
}

// The batched limb copy with the exponents already in args[i].E (no scan).
cudaError_t launch_batch_to_limbs(const StageArgs* args, int n, unsigned blocks, int nslot, int fluid, cudaStream_t s) {
  return launch_early(batch_to_limbs_kernel, dim3(blocks * (unsigned)(LIMB_EACH + nslot - 7), (unsigned)n), LIMB_THREADS,
                      0, s, args, nslot, fluid);
}

}  // namespace cosmos
