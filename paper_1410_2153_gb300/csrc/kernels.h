// Device and launch helpers shared by the solve kernels (solve.cu) and the
// multiple right-hand-side solve kernels (solve_multi.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "internal.h"

namespace asmg {
namespace kern {

constexpr int TPB = 256;
constexpr int RED_BLOCKS = 152 * 4;  // persistent reduction grid: 4 CTAs per SM
constexpr int VEC_BLOCKS = 152 * 8;  // grid of the vector-only PCG kernels: 8 CTAs (full occupancy) per SM

inline int nblk(int64_t n, int t = TPB) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + t - 1) / t, 1 << 24)); }
// Grid of a reduction kernel: one block per TPB rows up to the persistent grid
// `cap`.  Every block leaves a partial that its last block (grid_reduce) or
// every block of the next kernel (up to DIRECT_BLOCKS) adds up, so blocks
// without rows only lengthen that tail: at 3,969 rows k_dots took 16 us on
// 1,216 blocks (cold), and the 65^2 FP64 solve ran 1,583 us with the full grids
// and a ticket, 1,471 us with these (12 batched grids x 4 columns: 10.9 ms,
// 8.3 ms).
inline int red_grid(int64_t rows, int cap) { return std::min(cap, nblk(rows)); }

// Block size of a row-parallel launch: 256 threads when that fills every SM
// twice, else 64 so that small colour classes still spread over all SMs.
constexpr int NSM = 152;
inline int rows_tpb(int64_t rows) { return rows >= (int64_t)NSM * 2 * 256 ? 256 : 64; }

// Kernel launch with dynamic shared memory, optionally with programmatic dependent launch.
template <typename... KArgs, typename... Args>
void launch_smem(bool pdl, void (*kern)(KArgs...), int64_t grid, int block, size_t smem, cudaStream_t s,
                 Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  ASMG_CUDA(cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...));
}

// Kernel launch, optionally with programmatic dependent launch (the kernel may
// start while its predecessor on the stream finishes; see pdl_wait below).
template <typename... KArgs, typename... Args>
void launch(bool pdl, void (*kern)(KArgs...), int64_t grid, int block, cudaStream_t s, Args... args) {
  if (!pdl) {
    kern<<<(unsigned)grid, (unsigned)block, 0, s>>>(static_cast<KArgs>(args)...);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  ASMG_CUDA(cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...));
}

// Programmatic dependent launch: every solve kernel first loads what was
// written at setup (matrix rows, index lists), then waits for the preceding
// kernel (griddepcontrol.wait) and at once lets the next kernel launch
// (griddepcontrol.launch_dependents): the next kernel's blocks start as soon
// as all of this one's run, and load their own rows while this one works.
// Their wait still covers this kernel's end, and with it every earlier one's:
// a kernel ends only after its own wait.  Triggering at the kernel's end
// instead leaves those loads exposed (kuhn129 mixed 40.8 ms, 39.4 ms with the
// trigger here; graded 513^2 FP64 42.2, 40.3; four columns on 513^2 3.95,
// 3.63).  Triggering before the wait lets kernels pile up several deep, their
// waiting blocks holding the slots of the one that runs (graded 2049^2 258.0
// -> 267.6 ms).  Launched without the attribute, both instructions are no-ops.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A SELL-32 row held in registers (up to N entries; longer rows read the rest later).
constexpr int MAXW = 10;
template <class T, int N = MAXW>
struct Row {
  int64_t b = 0, lane = 0;
  int w = 0;
  int32_t c[N];
  T v[N];
};

// f(N) with the entries a row kernel holds per row.  A launch of one wave of
// threads hides its latency by its loads in flight, one of several waves by its
// occupancy, which the registers of a long row cost it: with 16 entries
// throughout graded 2049^2 BF16 takes 256 ms, with 10 217.5, with 8 on launches
// of several waves 211.6 (6 or 4 there: 212.2, 216.8; kuhn129 36.6 -> 35.7 ms);
// with 6 throughout 331^2 mixed goes from 1.56 to 1.69 ms.
constexpr int WIDE_W = 8;
template <int SMALL = MAXW, class F>
void by_rows(int64_t rows, F f) {
  if (rows <= (int64_t)NSM * 2048)
    f(std::integral_constant<int, SMALL>{});
  else
    f(std::integral_constant<int, WIDE_W>{});
}
constexpr int TRANSFER_W = 16;  // P and P^T rows of a small launch (10 entries on average in 2D, 15 in 3D)

// Matrix values as stored (FP64, FP32 or BF16), widened to the arithmetic
// type exactly; the ldg forms read through the read-only path, the ldcs forms
// stream (evict first).
__device__ __forceinline__ double ldg_val(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldg_val(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ldg_val(const bf16v* p) {
  return __uint_as_float((uint32_t)__ldg(&p->bits) << 16);
}
__device__ __forceinline__ double ldcs_val(const double* p) { return __ldcs(p); }
__device__ __forceinline__ float ldcs_val(const float* p) { return __ldcs(p); }
__device__ __forceinline__ float ldcs_val(const bf16v* p) {
  return __uint_as_float((uint32_t)__ldcs(&p->bits) << 16);
}
__device__ __forceinline__ double val_of(double v) { return v; }
__device__ __forceinline__ float val_of(float v) { return v; }
__device__ __forceinline__ float val_of(bf16v v) { return __uint_as_float((uint32_t)v.bits << 16); }

template <class T, int N, class V>
__device__ __forceinline__ void row_load(Row<T, N>& R, int64_t row, const int64_t* __restrict__ off,
                                         const int32_t* __restrict__ col, const V* __restrict__ val) {
  const int64_t sl = row >> 5;
  R.lane = row & 31;
  R.b = __ldg(off + sl);
  R.w = (int)((__ldg(off + sl + 1) - R.b) >> 5);
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (k < R.w) {
      const int64_t e = R.b + ((int64_t)k << 5) + R.lane;
      R.c[k] = __ldcs(col + e);
      R.v[k] = (T)ldcs_val(val + e);
    }
}

template <class T, int N, class V, class X>
__device__ __forceinline__ T row_dot(const Row<T, N>& R, const int32_t* __restrict__ col, const V* __restrict__ val,
                                     const X* x) {
  T s = 0;
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (k < R.w) s += R.v[k] * (T)x[R.c[k]];
  for (int k = N; k < R.w; ++k) {
    const int64_t e = R.b + ((int64_t)k << 5) + R.lane;
    s += (T)ldg_val(val + e) * (T)x[__ldg(col + e)];
  }
  return s;
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  v = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
  if (w == 0)
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;  // valid in thread 0
}

// v[j] of a block's threads -> its partials (value j of block b at j * grid + b)
template <int NV>
__device__ __forceinline__ void block_partials(const double (&v)[NV], double* partial) {
  __shared__ double sh[32];
  for (int j = 0; j < NV; ++j) {
    const double t = block_sum(v[j], sh);
    if (threadIdx.x == 0) partial[j * gridDim.x + blockIdx.x] = t;
  }
}

// The sums of nb blocks' partials, in block order; valid in thread 0.
template <int NV>
__device__ __forceinline__ void sum_partials(double (&v)[NV], const double* partial, unsigned nb) {
  __shared__ double sh[32];
  for (int j = 0; j < NV; ++j) {
    // the partials of this thread (blocks t, t + blockDim, ...) summed in
    // ascending order, eight loads in flight
    const double* pj = partial + (int64_t)j * nb;
    double s = 0;
    for (unsigned b = threadIdx.x; b < nb; b += 8 * blockDim.x) {
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned bb = b + u * blockDim.x;
        x[u] = bb < nb ? __ldcg(pj + bb) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) s += x[u];
    }
    v[j] = block_sum(s, sh);
  }
}

// Deterministic grid reduction of NV values: partials per block, the last
// block to finish sums them in block order.  Returns true in that block.
template <int NV>
__device__ bool grid_reduce(double (&v)[NV], double* partial, unsigned int* ticket) {
  __shared__ bool last;
  block_partials(v, partial);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!last) return false;
  __threadfence();
  sum_partials(v, partial, gridDim.x);
  if (threadIdx.x == 0) *ticket = 0;
  return true;
}

// Up to this many blocks a reduction's result is summed by every block of the
// kernel that uses it, from the partials, instead of by the reduction's last
// block: the ticket, that block's second pass and the read of its result drop
// out of the chain of a small solve (65^2 FP64 725 -> 695 us).  With more
// blocks the repeated sums cost more than they save.
constexpr int DIRECT_BLOCKS = 2 * NSM;

}  // namespace kern
}  // namespace asmg
