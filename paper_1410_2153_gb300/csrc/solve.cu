// The solve phase on the device: PCG (Sec. 5.2) preconditioned by the
// multiplicative auxiliary-space preconditioner (Algorithm 1) whose
// auxiliary correction is the V-cycle of Algorithm 2 on the nested grids.
//
// Layout.  Fine vectors live in a permuted, padded order: free dofs grouped
// by colour, each colour block padded to a multiple of 32 rows, so a colour
// sweep is one contiguous range of SELL-32 slices.  Auxiliary vectors are
// indexed by the free nodes of the finest auxiliary level (lattice Morton
// order); every coarser level's nodes are a subset, so one rhs vector F and
// one correction vector U serve all levels and the V-cycle updates them in
// place:
//   down, level l:  save F on N~_l (first pre-sweep), nu_pre forward sweeps
//                   on N~_l, F -= A_l U on the rows E_l touched by N~_l,
//                   F[parent] += 1/2 F[new child] (I_l^T).  U is 0 on the
//                   whole down path: the level's correction lives in its
//                   saved array us (SM row order) and never enters U there;
//   coarsest:       U = A_c^{-1} F on its nodes (explicit FP64 inverse);
//   up, level l:    U[new] = (U[p0] + U[p1]) / 2 (I_l), U += saved values,
//                   nu_post backward sweeps with the saved F.
// New nodes are midpoints of coarse edges (Sec. 3.3), hence the 1/2 weights.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <type_traits>
#include <vector>

#include "handle.h"
#include "kernels.h"
#include "small_run.h"

namespace asmg {

namespace {

using namespace kern;

// ------------------------------------------------------------- fine grid
// one colour of a Gauss-Seidel sweep: u_i += (rhs_i - (A u)_i) / a_ii
template <class T, class R>
__global__ void k_gs_fine(int64_t r0, int64_t nrows, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                          const T* __restrict__ val, const T* __restrict__ dinv, const R* __restrict__ rhs, T* u) {
  const int64_t i = r0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < r0 + nrows;
  Row<T> row;
  T di = 0;
  if (act) {
    row_load(row, i, off, col, val);
    di = dinv[i];
  }
  pdl_wait();
  if (act) {
    const T s = (T)rhs[i] - row_dot(row, col, val, u);
    u[i] += s * di;
  }
}

// rho = r - A u
template <class T>
__global__ void k_resid_fine(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                             const T* __restrict__ val, const double* __restrict__ r, const T* __restrict__ u,
                             T* __restrict__ rho) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < n;
  Row<T> row;
  if (act) row_load(row, i, off, col, val);
  pdl_wait();
  if (act) rho[i] = (T)r[i] - row_dot(row, col, val, u);
}

// F = P^T rho on the auxiliary nodes, and U = 0 (start of the V-cycle)
template <class T>
__global__ void k_restrict_fine(int64_t nJ, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                                const T* __restrict__ val, const T* __restrict__ rho, T* __restrict__ F,
                                T* __restrict__ U) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = k < nJ;
  Row<T> row;
  if (act) row_load(row, k, off, col, val);
  pdl_wait();
  if (act) {
    F[k] = row_dot(row, col, val, rho);
    U[k] = 0;
  }
}

// u += P U
template <class T>
__global__ void k_prolong_fine(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                               const T* __restrict__ val, const T* __restrict__ U, T* __restrict__ u) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < n;
  Row<T> row;
  if (act) row_load(row, i, off, col, val);
  pdl_wait();
  if (act) u[i] += row_dot(row, col, val, U);
}

// Jacobi smoother (S = D^{-1}): first step from zero, u = D^{-1} r
template <class T>
__global__ void k_jac_first(int64_t n, const T* __restrict__ dinv, const double* __restrict__ r, T* __restrict__ u) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < n;
  const T di = act ? dinv[i] : (T)0;
  pdl_wait();
  if (act) u[i] = di * (T)r[i];
}

// a further Jacobi step, u += D^{-1} rho with rho = r - A u taken before
template <class T>
__global__ void k_jac_add(int64_t n, const T* __restrict__ dinv, const T* __restrict__ rho, T* __restrict__ u) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < n;
  const T di = act ? dinv[i] : (T)0;
  pdl_wait();
  if (act) u[i] += di * rho[i];
}

// additive form: the auxiliary correction acts on r itself (rho = r)
template <class T>
__global__ void k_cast_fine(int64_t n, const double* __restrict__ r, T* __restrict__ rho) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (i < n) rho[i] = (T)r[i];
}

// ------------------------------------------------------ auxiliary levels
// one colour of an up (post-smoothing) sweep on the smoothing rows of a
// level: U[i] += (fs_k - (A_l U)_i) / a_ii with the F saved on the way down
template <class T, class V>
__global__ void k_gs_aux(int64_t k0, int64_t nk, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                         const V* __restrict__ val, const T* __restrict__ dinv, const int32_t* __restrict__ rows,
                         const T* __restrict__ fs, T* U) {
  const int64_t k = k0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1;
  Row<T> row;
  T di = 0;
  if (k < k0 + nk) {
    i = rows[k];
    if (i >= 0) {
      row_load(row, k, off, col, val);
      di = dinv[k];
    }
  }
  pdl_wait();
  if (i >= 0) {
    const T s = fs[k] - row_dot(row, col, val, U);
    U[i] += s * di;
  }
}

// one colour of a down (pre-smoothing) sweep, on the level's own correction
// us in SM row order.  The V-cycle reaches level l with U = 0, and the down
// path changes U only on N~_l, so the sweeps run on us alone with the rows'
// columns in N~_l (SMd).  In the first sweep us is 0 on this class and the
// later ones: only columns of earlier classes (below k0) are read, and the
// class's rows are set rather than updated.  The first sweep takes F and
// saves it in fs.
template <class T, class V>
__global__ void k_gs_aux_down(int64_t k0, int64_t nk, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                              const V* __restrict__ val, const T* __restrict__ dinv, const int32_t* __restrict__ rows,
                              const T* __restrict__ F, int first, T* __restrict__ fs, T* us) {
  const int64_t k = k0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1;
  Row<T> row;
  T di = 0;
  if (k < k0 + nk) {
    i = rows[k];
    if (i >= 0) {
      row_load(row, k, off, col, val);
      di = dinv[k];
    }
  }
  pdl_wait();
  if (i >= 0) {
    T f, acc = 0;
    if (first) {
      f = F[i];
      fs[k] = f;
#pragma unroll
      for (int q = 0; q < MAXW; ++q)
        if (q < row.w && row.c[q] < k0) acc += row.v[q] * us[row.c[q]];
      for (int q = MAXW; q < row.w; ++q) {
        const int64_t e = row.b + ((int64_t)q << 5) + row.lane;
        const int32_t c = __ldg(col + e);
        if (c < k0) acc += (T)ldg_val(val + e) * us[c];
      }
      us[k] = (f - acc) * di;
    } else {
      f = fs[k];
      acc = row_dot(row, col, val, us);
      us[k] += (f - acc) * di;
    }
  }
}

// F_i -= sum_{j in N~_l} a_ij U_j on the rows E_l
template <class T, class V>
__global__ void k_resid_aux(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                            const V* __restrict__ val, const int32_t* __restrict__ rows, const T* __restrict__ U,
                            T* __restrict__ F) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1;
  Row<T> row;
  if (k < n) {
    i = rows[k];
    if (i >= 0) row_load(row, k, off, col, val);
  }
  pdl_wait();
  if (i >= 0) F[i] -= row_dot(row, col, val, U);
}

// I_l^T: F[parent] += 1/2 sum F[new children]
template <class T>
__global__ void k_restrict_aux(int64_t npar, const int32_t* __restrict__ pid, const int32_t* __restrict__ pptr,
                               const int32_t* __restrict__ child, T* __restrict__ F) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t par = -1, p0 = 0, p1 = 0;
  if (t < npar) {
    par = pid[t];
    p0 = pptr[t];
    p1 = pptr[t + 1];
  }
  pdl_wait();
  if (par >= 0) {
    T acc = 0;
    for (int32_t p = p0; p < p1; ++p) acc += F[child[p]];
    F[par] += (T)0.5 * acc;
  }
}

// I_l: U[new] = (U[p0] + U[p1]) / 2, Dirichlet parents contribute 0
template <class T>
__global__ void k_prolong_aux(int64_t nnew, const int32_t* __restrict__ id, const int32_t* __restrict__ p0,
                              const int32_t* __restrict__ p1, T* U) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t a = -1, b = -1, me = -1;
  if (t < nnew) {
    a = p0[t];
    b = p1[t];
    me = id[t];
  }
  pdl_wait();
  if (me >= 0) {
    T v = 0;
    if (a >= 0) v += U[a];
    if (b >= 0) v += U[b];
    U[me] = (T)0.5 * v;
  }
}

template <class T>
__global__ void k_addsaved_aux(int64_t nsm, const int32_t* __restrict__ rows, const T* __restrict__ us, T* U) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int32_t i = t < nsm ? rows[t] : -1;
  pdl_wait();
  if (i >= 0) U[i] += us[t];
}

// coarsest level: U[cid] = A_c^{-1} F[cid] in FP64, one warp per row
template <class T>
__global__ void k_coarse(int64_t nc, const int32_t* __restrict__ cid, const double* __restrict__ inv,
                         const T* __restrict__ F, T* __restrict__ U) {
  const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  pdl_wait();
  if (row < nc) {
    double s = 0;
    for (int64_t j = lane; j < nc; j += 32) s += inv[row * nc + j] * (double)F[cid[j]];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) U[cid[row]] = (T)s;
  }
}

// ------------------------------------------- tiled sweeps (one launch each)
// One thread block per tile (see TileSweeps), a persistent grid over the
// tiles: the tile's rows -- its own rows of N~_l plus the halo its sweeps read
// -- are held in registers for all nu sweeps, one row per slot and thread; the
// rows' values live in shared memory and the colour phases are separated by
// __syncthreads.  A tile's block of setup data arrives by one bulk copy
// (cp.async.bulk, completion on an mbarrier): the first before the wait on the
// previous kernel, each further one while the block sweeps the tile before.
// Each row is updated with the same arithmetic, over the same stored entries
// in the same order, as k_gs_aux_down / k_gs_aux do; the entries a tile leaves
// out are exactly those whose value cannot reach the tile's own rows' results,
// so those results equal the class-by-class launches bit for bit.  Halo
// results are discarded.
//
// What bounds them is instructions and waits per colour phase, not the bytes:
// with the rows read from shared memory entry by entry a level of 3.46 M rows
// in five classes (graded 2049^2, BF16) took 118 us a direction at 18% of the
// DRAM rate; with the rows in registers, no test per entry and four blocks per
// SM it takes 78 us (graded 2049^2 solve 254.7 -> 231.6 ms, graded 513^2 FP64
// 40.3 -> 38.2 ms, 331^2 mixed 2.04 -> 1.98 ms).

// bound on the wait for a bulk copy (SM clock cycles, about 1 s): when it
// expires the block records the timeout, waits once more (bounded) for its
// copy to land, and ends
constexpr long long TILE_WAIT_CYCLES = 2000000000LL;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait for the mbarrier's phase of the given parity
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > TILE_WAIT_CYCLES) return false;
  return true;
}

// one thread: arm the barrier and start the copy of a tile's block; the block's
// earlier reads of the same shared memory came before a __syncthreads
__device__ __forceinline__ void tile_fetch(void* dst, const unsigned char* blob, const TileHead& h, uint64_t* bar) {
  const uint32_t b = smem_addr(bar);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"((uint32_t)h.bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(blob + h.off), "r"((uint32_t)h.bytes), "r"(b)
               : "memory");
}

__device__ __forceinline__ void tile_bar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Every thread waits for the copy (bounded): false in every thread when any
// thread's wait expired.  inject != 0 (failure injection, asmg_params::
// inject_timeout) takes the expired path without polling.
__device__ __forceinline__ bool tile_arrived(uint64_t* bar, uint32_t parity, int inject) {
  return __syncthreads_and(!inject && mbar_wait_bounded(smem_addr(bar), parity));
}

// after an expired wait: record it and give the copy a second bounded wait
// before the block ends
__device__ __forceinline__ void tile_expired(uint64_t* bar, uint32_t parity, int* timeout) {
  if (threadIdx.x == 0) atomicExch(timeout, 1);
  mbar_wait_bounded(smem_addr(bar), parity);
  __syncthreads();
}

// The entries of one row (up to W) in registers, and its product with the
// values in shared memory at `u`, summed in stored order.  Entries beyond the
// slice's width are zeros at offset 0 (their products leave the sum as it is),
// so the common widths run without a test per entry: a test, its branch and
// their waits cost more than the multiply-add.
// A0: entries multiplied whatever the width; the rest in groups of two.
template <class T, class V, int W>
struct TileRow {
  uint32_t c[(W + 1) / 2];
  T v[W];
  __device__ __forceinline__ void load(const uint32_t* words, const T* val, const TileSlice& h, int lane) {
#pragma unroll
    for (int e = 0; e < (W + 1) / 2; ++e) c[e] = 2 * e < h.w ? words[(h.words + e) * 32 + lane] : 0u;
#pragma unroll
    for (int e = 0; e < W; ++e) v[e] = e < h.w ? val[(h.vals + e) * 32 + lane] : (T)0;
  }
  __device__ __forceinline__ T term(const char* u, int e, T acc) const {
    return acc + v[e] * *reinterpret_cast<const T*>(u + ((e & 1) ? c[e / 2] >> 16 : c[e / 2] & 0xffffu));
  }
};
template <class T, int W>
struct TileRow<T, bf16v, W> {
  uint32_t c[W];
  __device__ __forceinline__ void load(const uint32_t* words, const T*, const TileSlice& h, int lane) {
#pragma unroll
    for (int e = 0; e < W; ++e) c[e] = e < h.w ? words[(h.words + e) * 32 + lane] : 0u;
  }
  __device__ __forceinline__ T term(const char* u, int e, T acc) const {
    return acc + (T)__uint_as_float(c[e] & 0xffff0000u) * *reinterpret_cast<const T*>(u + (c[e] & 0xffffu));
  }
};
template <class T, class V, int W>
__device__ __forceinline__ T tile_dot(const TileRow<T, V, W>& row, const char* u, int w) {
  constexpr int A0 = W <= 8 ? 6 : 8;
  T acc = 0;
#pragma unroll
  for (int e = 0; e < A0; ++e) acc = row.term(u, e, acc);
#pragma unroll
  for (int e = A0; e < W; e += 2)
    if (w > e) {
      acc = row.term(u, e, acc);
      acc = row.term(u, e + 1, acc);
    }
  return acc;
}

// the thread's rows of a tile, from the staged block
template <class T, class V, int S, int W>
struct TileRows {
  int wc[S];        // slice: width | colour class << 8 (-1 << 8: empty)
  TileRow<T, V, W> row[S];
  T di[S];
  int32_t g[S], ax[S];  // SM row (own k, halo -2 - k, padding -1), aux ID
  __device__ __forceinline__ void load(const unsigned char* blob, const TileHead& h, const TileLayout& lay) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const TileSlice* hdr = reinterpret_cast<const TileSlice*>(blob);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      wc[s] = -256;
      g[s] = -1;
      if (s < h.slots) {
        const TileSlice sl = hdr[s * TILE_WARPS + warp];
        wc[s] = sl.w | (int)sl.colour << 8;
        row[s].load(reinterpret_cast<const uint32_t*>(blob + lay.words), reinterpret_cast<const T*>(blob + lay.val), sl,
                    lane);
        di[s] = reinterpret_cast<const T*>(blob + lay.dinv)[s * TILE_THREADS + tid];
        g[s] = reinterpret_cast<const int32_t*>(blob + lay.lsm)[s * TILE_THREADS + tid];
        ax[s] = reinterpret_cast<const int32_t*>(blob + lay.laux)[s * TILE_THREADS + tid];
      }
    }
  }
  // one colour phase: u += (f - A u) / a_ii on the thread's rows of class c
  __device__ __forceinline__ void phase(int c, T* Ul, const T (&f)[S], T (&u)[S]) const {
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (wc[s] >> 8 == c) {
        const T acc = tile_dot(row[s], reinterpret_cast<const char*>(Ul), wc[s] & 255);
        u[s] += (f[s] - acc) * di[s];
        Ul[s * TILE_THREADS + threadIdx.x] = u[s];
      }
  }
};

// blocks per SM the kernels are compiled for: the most whose registers hold the
// rows (a few spilled words cost less than a fourth block gives, BF16: level of
// 3.46 M rows 115 us with three blocks, 80 us with four)
template <class T, class V, int S, int W>
constexpr int tile_min_blocks() {
  if (sizeof(T) == 8) return W > 8 ? (S > 2 ? 1 : 2) : S > 2 ? 2 : 3;
  return W > 8 ? 2 : S == 4 && !std::is_same<V, bf16v>::value ? 3 : 4;
}

// pre-sweeps: us (the level's own correction, SM order) starts at 0; the
// first sweep saves F on the tile's own rows in fs
template <class T, class V, int S, int W>
__global__ void __launch_bounds__(TILE_THREADS, tile_min_blocks<T, V, S, W>())
    k_tile_down(TileView<T> t, int ncol, int64_t vals, const T* __restrict__ F, T* __restrict__ fs,
                T* __restrict__ us, int nu, int* timeout, int inject) {
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t bar;
  T* Ul = reinterpret_cast<T*>(smraw);
  unsigned char* blob = smraw + vals;
  const int tid = threadIdx.x;
  int64_t tile = blockIdx.x;
  TileHead h = t.head[tile];
  if (tid == 0) {
    tile_bar_init(&bar);
    tile_fetch(blob, t.blob, h, &bar);
  }
  __syncthreads();  // the barrier is initialised before any thread polls it
  // the first tile's rows are in registers before the wait on the previous kernel
  TileRows<T, V, S, W> R;
  uint32_t parity = 0;
  bool ok = tile_arrived(&bar, parity, inject);
  if (ok) R.load(blob, h, tile_layout(h.slots, h.nwords, h.nvals, h.nx, sizeof(T)));
  pdl_wait();
  while (ok) {
    T f[S], u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      f[s] = R.g[s] != -1 ? F[R.ax[s]] : (T)0;
      u[s] = 0;
      Ul[s * TILE_THREADS + tid] = 0;
    }
    const uint32_t mask = h.cmask;
    tile += gridDim.x;
    const bool more = tile < t.ntiles;
    if (more) h = t.head[tile];
    __syncthreads();  // values in place, the block read by all
    if (tid == 0 && more) tile_fetch(blob, t.blob, h, &bar);
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (R.g[s] >= 0) fs[R.g[s]] = f[s];
    for (int sw = 0; sw < nu; ++sw)
      for (int c = 0; c < ncol; ++c) {
        if (!((mask >> min(c, 31)) & 1u)) continue;  // no row of this class in the tile
        R.phase(c, Ul, f, u);
        __syncthreads();
      }
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (R.g[s] >= 0) us[R.g[s]] = u[s];
    if (!more) return;
    parity ^= 1;
    ok = tile_arrived(&bar, parity, inject);
    if (ok) R.load(blob, h, tile_layout(h.slots, h.nwords, h.nvals, h.nx, sizeof(T)));
  }
  tile_expired(&bar, parity, timeout);
}

// start of the up path of a tiled level: the prolongation of the coarse
// correction (I_l: new nodes take the mean of their parents) plus the level's
// saved correction, and the saved rhs, written for every SM row to each place
// the row holds in the post-sweep tiles (own and halo copies; TileSweeps::
// pos).  U itself is not written, so the tiles can read their start values
// while other tiles write their results to U.
template <class T>
__global__ void k_up_init(int64_t nsm, const int32_t* __restrict__ rows, const int32_t* __restrict__ par0,
                          const int32_t* __restrict__ par1, const int64_t* __restrict__ pos_ptr,
                          const int32_t* __restrict__ pos, const T* __restrict__ U, const T* __restrict__ us,
                          const T* __restrict__ fs, T* __restrict__ ust, T* __restrict__ fsl) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1, a = -3, b = -3;
  int64_t p0 = 0, p1 = 0;
  if (k < nsm) {
    i = rows[k];
    a = par0[k];
    b = par1[k];
    p0 = pos_ptr[k];
    p1 = pos_ptr[k + 1];
  }
  pdl_wait();
  if (i >= 0) {
    T v;
    if (a == -3) {
      v = U[i];
    } else {
      T p = 0;
      if (a >= 0) p += U[a];
      if (b >= 0) p += U[b];
      v = (T)0.5 * p;
    }
    v = v + us[k];
    const T f = fs[k];
    for (int64_t q = p0; q < p1; ++q) {
      const int32_t o = pos[q];
      ust[o] = v;
      fsl[o] = f;
    }
  }
}

// post-sweeps (backward colour order) from the start values and saved rhs
// that k_up_init wrote in tile order (`per` local rows a tile); the columns
// outside N~_l (the tile's outside values) are read from U once; the tile's
// own rows are written to U
template <class T, class V, int S, int W>
__global__ void __launch_bounds__(TILE_THREADS, tile_min_blocks<T, V, S, W>())
    k_tile_up(TileView<T> t, int ncol, int64_t vals, const T* __restrict__ ust, const T* __restrict__ fsl, T* U,
              int nu, int* timeout, int inject) {
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t bar;
  T* Ul = reinterpret_cast<T*>(smraw);
  unsigned char* blob = smraw + vals;
  const int tid = threadIdx.x;
  int64_t tile = blockIdx.x;
  TileHead h = t.head[tile];
  if (tid == 0) {
    tile_bar_init(&bar);
    tile_fetch(blob, t.blob, h, &bar);
  }
  __syncthreads();  // the barrier is initialised before any thread polls it
  // the first tile's rows are in registers before the wait on the previous kernel
  TileRows<T, V, S, W> R;
  TileLayout lay = tile_layout(h.slots, h.nwords, h.nvals, h.nx, sizeof(T));
  uint32_t parity = 0;
  bool ok = tile_arrived(&bar, parity, inject);
  if (ok) R.load(blob, h, lay);
  pdl_wait();
  while (ok) {
    const int64_t base = tile * (S * TILE_THREADS) + tid;
    T f[S], u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      u[s] = ust[base + s * TILE_THREADS];
      f[s] = fsl[base + s * TILE_THREADS];
    }
    const int32_t* ext = reinterpret_cast<const int32_t*>(blob + lay.ext);
    for (int e = tid; e < h.nx; e += TILE_THREADS) Ul[S * TILE_THREADS + e] = U[ext[e]];
#pragma unroll
    for (int s = 0; s < S; ++s) Ul[s * TILE_THREADS + tid] = u[s];
    const uint32_t mask = h.cmask;
    tile += gridDim.x;
    const bool more = tile < t.ntiles;
    if (more) h = t.head[tile];
    __syncthreads();  // values in place, the block read by all
    if (tid == 0 && more) tile_fetch(blob, t.blob, h, &bar);
    for (int sw = 0; sw < nu; ++sw)
      for (int c = ncol - 1; c >= 0; --c) {
        if (!((mask >> min(c, 31)) & 1u)) continue;
        R.phase(c, Ul, f, u);
        __syncthreads();
      }
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (R.g[s] >= 0) U[R.ax[s]] = u[s];
    if (!more) return;
    lay = tile_layout(h.slots, h.nwords, h.nvals, h.nx, sizeof(T));
    parity ^= 1;
    ok = tile_arrived(&bar, parity, inject);
    if (ok) R.load(blob, h, lay);
  }
  tile_expired(&bar, parity, timeout);
}

// ------------------------------------------- near-boundary solve (Alg. 3)
// After the coarse-grid correction of a level with mixed boundaries:
// r_J = f_J - (A_l U)_J on the near-boundary set J = J_{l,j}, then the exact
// solve A_JJ d = r_J by block cyclic reduction (NbDev), then U_J += d.

// r_J in the factor's order (the saved rhs of a whole-level smoothing set)
template <class T>
__global__ void k_nb_resid(int64_t m, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                           const T* __restrict__ val, const int32_t* __restrict__ sm, const T* __restrict__ fs,
                           const T* U, double* __restrict__ rhs) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = q < m;
  Row<T> row;
  int32_t k = 0;
  if (act) {
    row_load(row, q, off, col, val);
    k = sm[q];
  }
  pdl_wait();
  if (act) rhs[q] = (double)(fs[k] - row_dot(row, col, val, U));
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// x := F^{-T} F^{-1} x for the lower Cholesky factor F (s x s, row-major) of
// a block, one warp; x in global memory (lane 0 writes, __syncwarp orders)
__device__ void nb_chol_solve(const double* __restrict__ F, int s, double* x) {
  const int lane = threadIdx.x & 31;
  for (int i = 0; i < s; ++i) {
    double t = 0;
    for (int k = lane; k < i; k += 32) t += F[(int64_t)i * s + k] * x[k];
    t = warp_sum(t);
    if (lane == 0) x[i] = (x[i] - t) / F[(int64_t)i * s + i];
    __syncwarp();
  }
  for (int i = s - 1; i >= 0; --i) {
    double t = 0;
    for (int k = i + 1 + lane; k < s; k += 32) t += F[(int64_t)k * s + i] * x[k];
    t = warp_sum(t);
    if (lane == 0) x[i] = (x[i] - t) / F[(int64_t)i * s + i];
    __syncwarp();
  }
}

// y -= M z for M (r x c, row-major), one warp, lanes over the rows
__device__ void nb_gemv_sub(const double* __restrict__ M, int r, int c, const double* z, double* y) {
  for (int i = threadIdx.x & 31; i < r; i += 32) {
    double t = y[i];
    for (int j = 0; j < c; ++j) t -= M[(int64_t)i * c + j] * z[j];
    y[i] = t;
  }
  __syncwarp();
}

__device__ void nb_copy(const double* src, double* dst, int n) {
  for (int i = threadIdx.x & 31; i < n; i += 32) dst[i] = src[i];
  __syncwarp();
}

constexpr int NB_TPB = 1024;

// One thread block: the rounds of the reduction (odd blocks solved, even
// blocks' right-hand sides updated), the last block, then the rounds
// backwards (odd blocks from their even neighbours), then U_J += d.  The
// blocks of a step are independent: one warp each.
template <class T>
__global__ void __launch_bounds__(NB_TPB) k_nb_solve(int R, const int32_t* __restrict__ nblk,
                                                     const int32_t* __restrict__ boff, const int64_t* __restrict__ btab,
                                                     const int64_t* __restrict__ voff, const double* __restrict__ mats,
                                                     int last_size, int64_t last_off, int64_t m,
                                                     const int32_t* __restrict__ aux, double* rhs, double* sol, T* U) {
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  pdl_wait();
  for (int r = 0; r < R; ++r) {
    const int n = nblk[r];
    const int64_t* bt = btab + (int64_t)boff[r] * 5;
    double* V = rhs + voff[r];
    double* Y = sol + voff[r];
    double* Vn = rhs + voff[r + 1];
    const int64_t* btn = r + 1 < R ? btab + (int64_t)boff[r + 1] * 5 : nullptr;
    for (int k = 1 + 2 * warp; k < n; k += 2 * nw) {
      const int sk = (int)bt[5 * k];
      const int64_t o = bt[5 * k + 1];
      nb_copy(V + o, Y + o, sk);
      nb_chol_solve(mats + bt[5 * k + 2], sk, Y + o);
    }
    __syncthreads();
    for (int e = 2 * warp; e < n; e += 2 * nw) {
      const int se = (int)bt[5 * e];
      const int64_t o = bt[5 * e + 1], on = btn ? btn[5 * (e / 2) + 1] : 0;
      nb_copy(V + o, Vn + on, se);
      if (e > 0) nb_gemv_sub(mats + bt[5 * e + 3], se, (int)bt[5 * (e - 1)], Y + bt[5 * (e - 1) + 1], Vn + on);
      if (e + 1 < n) nb_gemv_sub(mats + bt[5 * e + 4], se, (int)bt[5 * (e + 1)], Y + bt[5 * (e + 1) + 1], Vn + on);
    }
    __syncthreads();
  }
  if (warp == 0) {
    nb_copy(rhs + voff[R], sol + voff[R], last_size);
    nb_chol_solve(mats + last_off, last_size, sol + voff[R]);
  }
  __syncthreads();
  for (int r = R - 1; r >= 0; --r) {
    const int n = nblk[r];
    const int64_t* bt = btab + (int64_t)boff[r] * 5;
    const double* V = rhs + voff[r];
    double* S = sol + voff[r];
    const double* Sn = sol + voff[r + 1];
    const int64_t* btn = r + 1 < R ? btab + (int64_t)boff[r + 1] * 5 : nullptr;
    for (int e = 2 * warp; e < n; e += 2 * nw) {
      const int64_t on = btn ? btn[5 * (e / 2) + 1] : 0;
      nb_copy(Sn + on, S + bt[5 * e + 1], (int)bt[5 * e]);
    }
    __syncthreads();
    for (int k = 1 + 2 * warp; k < n; k += 2 * nw) {
      const int sk = (int)bt[5 * k];
      const int64_t o = bt[5 * k + 1];
      nb_copy(V + o, S + o, sk);
      nb_gemv_sub(mats + bt[5 * k + 3], sk, (int)bt[5 * (k - 1)], S + bt[5 * (k - 1) + 1], S + o);
      if (k + 1 < n) nb_gemv_sub(mats + bt[5 * k + 4], sk, (int)bt[5 * (k + 1)], S + bt[5 * (k + 1) + 1], S + o);
      nb_chol_solve(mats + bt[5 * k + 2], sk, S + o);
    }
    __syncthreads();
  }
  for (int64_t q = threadIdx.x; q < m; q += blockDim.x) U[aux[q]] += (T)sol[q];
}

// ------------------------------------------------------------------ PCG
__device__ __forceinline__ void set_cond(PcgScalars* sc, int cond, cudaGraphConditionalHandle hnd, int use_hnd) {
  sc->cond = cond;
  if (use_hnd) cudaGraphSetConditional(hnd, cond ? 1u : 0u);
}

// r = b - A x;  ||b||, ||r||; PCG scalars initialised
__global__ void k_pcg_init(int64_t n, SellView<double> A, const double* __restrict__ b, const double* __restrict__ x,
                           double* __restrict__ r, double* partial, unsigned int* ticket, PcgScalars* sc, double rtol,
                           int maxit, double* hist, cudaGraphConditionalHandle hnd, int use_hnd) {
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  Row<double> row;
  if (i0 < n) row_load(row, i0, A.off, A.col, A.val);
  pdl_wait();
  double v[2] = {0, 0};
  for (int64_t i = i0; i < n; i += st) {
    if (i != i0) row_load(row, i, A.off, A.col, A.val);
    double ri = b[i] - row_dot(row, A.col, A.val, x);
    r[i] = ri;
    v[0] += b[i] * b[i];
    v[1] += ri * ri;
  }
  if (grid_reduce<2>(v, partial, ticket) && threadIdx.x == 0) {
    sc->bnorm = sqrt(v[0]);
    sc->tol = rtol * sc->bnorm;
    sc->rr = v[1];
    sc->k = 0;
    sc->maxit = maxit;
    sc->status = 1;
    sc->rz = 0;
    sc->alpha = 0;
    sc->beta = 0;
    sc->timeout = 0;
    hist[0] = sqrt(v[1]);
    const bool conv = sqrt(v[1]) <= sc->tol;
    if (conv) sc->status = 0;
    set_cond(sc, (!conv && maxit > 0) ? 1 : 0, hnd, use_hnd);
  }
}

// <z, r>, <z, q_prev>  ->  beta (flexible: -alpha <z_{k+1}, q_k> / <z_k, r_k>), rz
template <class T>
__global__ void k_dots(int64_t n, const T* __restrict__ z, const double* __restrict__ r, const double* __restrict__ q,
                       double* partial, unsigned int* ticket, PcgScalars* sc) {
  pdl_wait();
  double v[2] = {0, 0};
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double zi = (double)z[i];
    v[0] += zi * r[i];
    v[1] += zi * q[i];
  }
  if (grid_reduce<2>(v, partial, ticket) && threadIdx.x == 0) {
    if (sc->k == 0) {
      sc->beta = 0;
    } else {
      sc->beta = -sc->alpha * v[1] / sc->rz;
    }
    sc->rz = v[0];
    if (!(v[0] > 0)) sc->status = ASMG_ERR_BREAKDOWN;
  }
}

// p = z + beta p
template <class T>
__global__ void k_pupd(int64_t n, const T* __restrict__ z, double* __restrict__ p, const PcgScalars* __restrict__ sc) {
  pdl_wait();
  const double beta = sc->beta;
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = (double)z[i] + beta * p[i];
}

// q = A p, <p, q>  ->  alpha.  Each row's entries are loaded into registers
// at once (row_load), the thread's first row before the wait on the previous
// kernel (graded 2049^2: 3.1 -> 4.3 TB/s against a plain loop over the row).
__global__ void k_spmv_dot(int64_t n, SellView<double> A, const double* __restrict__ p, double* __restrict__ q,
                           double* partial, unsigned int* ticket, PcgScalars* sc) {
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  Row<double> row;
  if (i0 < n) row_load(row, i0, A.off, A.col, A.val);
  pdl_wait();
  double v[1] = {0};
  for (int64_t i = i0; i < n; i += st) {
    if (i != i0) row_load(row, i, A.off, A.col, A.val);
    const double qi = row_dot(row, A.col, A.val, p);
    q[i] = qi;
    v[0] += p[i] * qi;
  }
  if (grid_reduce<1>(v, partial, ticket) && threadIdx.x == 0) {
    sc->pq = v[0];
    if (!(v[0] > 0) || sc->status == ASMG_ERR_BREAKDOWN) {
      sc->status = ASMG_ERR_BREAKDOWN;
      sc->alpha = 0;
    } else {
      sc->alpha = sc->rz / v[0];
    }
  }
}

// x += alpha p, r -= alpha q, ||r||  ->  history, stopping test
__global__ void k_axpy_norm(int64_t n, const double* __restrict__ p, const double* __restrict__ q,
                            double* __restrict__ x, double* __restrict__ r, double* partial, unsigned int* ticket,
                            PcgScalars* sc, double* hist, cudaGraphConditionalHandle hnd, int use_hnd) {
  pdl_wait();
  const double a = sc->alpha;
  double v[1] = {0};
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] += a * p[i];
    double ri = r[i] - a * q[i];
    r[i] = ri;
    v[0] += ri * ri;
  }
  if (grid_reduce<1>(v, partial, ticket) && threadIdx.x == 0) {
    if (sc->status == ASMG_ERR_BREAKDOWN) {
      set_cond(sc, 0, hnd, use_hnd);
      return;
    }
    if (sc->timeout) {
      sc->status = ASMG_ERR_TIMEOUT;
      set_cond(sc, 0, hnd, use_hnd);
      return;
    }
    sc->k += 1;
    sc->rr = v[0];
    const double nr = sqrt(v[0]);
    hist[sc->k] = nr;
    bool conv = nr <= sc->tol;
    if (conv) sc->status = 0;
    bool more = !conv && sc->k < sc->maxit && isfinite(nr);
    if (!isfinite(nr)) sc->status = ASMG_ERR_BREAKDOWN;
    set_cond(sc, more ? 1 : 0, hnd, use_hnd);
  }
}

// ASMG iteration: x += z
template <class T>
__global__ void k_xpz(int64_t n, const T* __restrict__ z, double* __restrict__ x) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] += (double)z[i];
}

// ASMG iteration: r = b - A x, ||r||  ->  history, stopping test
__global__ void k_iter_resid(int64_t n, SellView<double> A, const double* __restrict__ b, const double* __restrict__ x,
                             double* __restrict__ r, double* partial, unsigned int* ticket, PcgScalars* sc, double* hist,
                             cudaGraphConditionalHandle hnd, int use_hnd) {
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  Row<double> row;
  if (i0 < n) row_load(row, i0, A.off, A.col, A.val);
  pdl_wait();
  double v[1] = {0};
  for (int64_t i = i0; i < n; i += st) {
    if (i != i0) row_load(row, i, A.off, A.col, A.val);
    const double ri = b[i] - row_dot(row, A.col, A.val, x);
    r[i] = ri;
    v[0] += ri * ri;
  }
  if (grid_reduce<1>(v, partial, ticket) && threadIdx.x == 0) {
    if (sc->timeout) {
      sc->status = ASMG_ERR_TIMEOUT;
      set_cond(sc, 0, hnd, use_hnd);
      return;
    }
    sc->k += 1;
    sc->rr = v[0];
    const double nr = sqrt(v[0]);
    hist[sc->k] = nr;
    const bool conv = nr <= sc->tol;
    if (conv) sc->status = 0;
    if (!isfinite(nr)) sc->status = ASMG_ERR_BREAKDOWN;
    set_cond(sc, (!conv && sc->k < sc->maxit && isfinite(nr)) ? 1 : 0, hnd, use_hnd);
  }
}

__global__ void k_gather(int64_t n, const int32_t* __restrict__ vrow, const double* __restrict__ src,
                         double* __restrict__ dst) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t v = vrow[i];
  dst[i] = v >= 0 ? src[v] : 0.0;
}

// the same with the vertex array's address in device memory (batched solves:
// the graph stays, the caller's arrays change)
__global__ void k_gather_tab1(int64_t n, const int32_t* __restrict__ vrow, double* const* __restrict__ tab,
                              double* __restrict__ dst) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t v = vrow[i];
  dst[i] = v >= 0 ? tab[0][v] : 0.0;
}

__global__ void k_scatter_tab1(int64_t nv, const int32_t* __restrict__ rowv, const double* __restrict__ src,
                               double* const* __restrict__ tab) {
  const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= nv) return;
  const int32_t r = rowv[v];
  tab[0][v] = r >= 0 ? src[r] : 0.0;
}

template <class S>
__global__ void k_scatter(int64_t nv, const int32_t* __restrict__ rowv, const S* __restrict__ src,
                          double* __restrict__ dst) {
  const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= nv) return;
  const int32_t r = rowv[v];
  dst[v] = r >= 0 ? (double)src[r] : 0.0;
}

// --------------------------------------------------------- profiling
// With a profiler installed, every launch of the solve is bracketed by CUDA
// events on its stream and tagged with its kernel class and algorithmic bytes.
struct Profiler {
  cudaStream_t s = nullptr;
  std::vector<cudaEvent_t> ev;
  struct Rec {
    int cls;
    int64_t bytes;
    int e0;
    int level;  // index into Prec::lev of an auxiliary-level launch (down: level, up: -2 - level), else -1
  };
  std::vector<Rec> recs;
  int mark() {
    cudaEvent_t e;
    ASMG_CUDA(cudaEventCreate(&e));
    ASMG_CUDA(cudaEventRecord(e, s));
    ev.push_back(e);
    return (int)ev.size() - 1;
  }
  ~Profiler() {
    for (auto e : ev) cudaEventDestroy(e);
  }
};
thread_local Profiler* g_prof = nullptr;
thread_local int g_prof_level = -1;

#define LAUNCH(cls, bytes, ...)                                                  \
  do {                                                                          \
    int e0_ = g_prof ? g_prof->mark() : -1;                                     \
    __VA_ARGS__;                                                                \
    if (g_prof) {                                                               \
      g_prof->mark();                                                           \
      g_prof->recs.push_back(Profiler::Rec{(int)(cls), (int64_t)(bytes), e0_, g_prof_level}); \
    }                                                                           \
  } while (0)

// --------------------------------------------------------- enqueueing
template <class T>
SellView<T> fine_smoother(asmg_s& h);
template <>
SellView<double> fine_smoother<double>(asmg_s& h) { return view(h.A64); }
template <>
SellView<float> fine_smoother<float>(asmg_s& h) { return view(h.p32.Af); }
template <class T>
const T* fine_dinv(asmg_s& h);
template <>
const double* fine_dinv<double>(asmg_s& h) { return h.dinv64.p; }
template <>
const float* fine_dinv<float>(asmg_s& h) { return h.p32.dinv_f.p; }

template <class T>
Prec<T>& prec(asmg_s& h);
template <>
Prec<double>& prec<double>(asmg_s& h) { return h.p64; }
template <>
Prec<float>& prec<float>(asmg_s& h) { return h.p32; }

template <class T>
SlotPrec<T>& slotprec(Slot& S);
template <>
SlotPrec<double>& slotprec<double>(Slot& S) { return S.s64; }
template <>
SlotPrec<float>& slotprec<float>(Slot& S) { return S.s32; }

// compulsory bytes of a fused run: its block, the union's values and the
// smoothing rows' saved values
template <class T>
int64_t small_bytes(const SmallRun<T>& R, bool down) {
  const int64_t sz = sizeof(T);
  return (down ? R.v.bytes : R.v.up_bytes) + 2 * sz * (R.v.nunion + R.v.nsm);
}

// f(slots, width) with the tile kernel's compile-time sizes for a level's tiles
template <class T, class V, class F>
void tile_dispatch(const TileSweeps<T>& Tl, F f) {
  auto by_width = [&](auto sl) {
    if (Tl.width <= 8)
      f(sl, std::integral_constant<int, 8>{});
    else
      f(sl, std::integral_constant<int, TILE_MAXW>{});
  };
  if (Tl.slots == 1) by_width(std::integral_constant<int, 1>{});
  if (Tl.slots == 2) by_width(std::integral_constant<int, 2>{});
  if (Tl.slots == 3) by_width(std::integral_constant<int, 3>{});
  if (Tl.slots == 4) by_width(std::integral_constant<int, 4>{});
}

// the slot's timeout flag (PcgScalars::timeout, device memory)
int* timeout_flag(Slot& S) {
  return reinterpret_cast<int*>(reinterpret_cast<char*>(S.scal.p) + offsetof(PcgScalars, timeout));
}

// V: how the auxiliary-level matrices are read (T, or bf16v with level_bf16)
template <class T, class V>
int enqueue_vcycle(asmg_s& h, Slot& S, cudaStream_t s) {
  Prec<T>& P = prec<T>(h);
  SlotPrec<T>& SP = slotprec<T>(S);
  int launches = 0;
  const int64_t sz = sizeof(T), sv = sizeof(V);
  const int npre = h.prm.nu_pre, npost = h.prm.nu_post;
  const int nlev = (int)P.lev.size();
  const int ndeep = P.deep.v.nlev, nbot = P.bot.v.nlev;  // fused runs at the top and at the bottom
  if (ndeep) {
    LAUNCH(ASMG_PROF_AUX_SMALL, small_bytes(P.deep, true),
           small::launch_down<T, V, 1>(h.prm.use_pdl, P.deep, SP.F.p, SP.deep_fs.p, SP.deep_us.p, npre, s));
    ++launches;
  }
  for (int li = nlev - 1 - ndeep; li >= nbot; --li) {
    AuxLevelDev<T>& L = P.lev[li];
    auto SMd = view(L.SMd);
    g_prof_level = li;
    if (L.tiled_down) {
      // all pre-sweeps of the level in one launch (compulsory bytes: the
      // tiles' blocks once, F gathered and saved, us written)
      const TileSweeps<T>& Tl = L.tdown;
      const int64_t by = Tl.nnz_real * (sv + 2) + (Tl.interior + Tl.halo) * (8 + 2 * sz) + Tl.interior * (4 + sz);
      LAUNCH(ASMG_PROF_AUX_GS, by,
             tile_dispatch<T, V>(Tl, [&](auto sl, auto w) {
               constexpr int SL = decltype(sl)::value, W = decltype(w)::value;
               launch_smem(h.prm.use_pdl, k_tile_down<T, V, SL, W>,
                           std::min<int64_t>(Tl.ntiles, NSM * tile_min_blocks<T, V, SL, W>()), TILE_THREADS, Tl.smem(), s,
                           Tl.view(), L.ncolours, Tl.smem_values(), (const T*)SP.F.p, SP.fs[li].p, SP.us[li].p, npre,
                           timeout_flag(S), h.prm.inject_timeout);
             }));
      ++launches;
    }
    // pre-sweeps on us (SM order); the first also saves F on N~_l for the
    // post-sweeps (nu_pre >= 1)
    for (int sweep = 0; sweep < (L.tiled_down ? 0 : npre); ++sweep) {
      for (int c = 0; c < L.ncolours; ++c) {
        int64_t k0 = L.cstart[c], nk = L.cstart[c + 1] - L.cstart[c];
        if (!nk) continue;
        const int64_t by = L.cnnz_d[c] * (sv + 4) + L.crows[c] * (4 + (sweep == 0 ? 4 + 4 * sz : 4 * sz));
        LAUNCH(ASMG_PROF_AUX_GS, by,
               launch(h.prm.use_pdl, k_gs_aux_down<T, V>, nblk(nk, rows_tpb(nk)), rows_tpb(nk), s, k0, nk, SMd.off,
                      SMd.col, sell_vals(L.SMd, (const V*)nullptr), L.sm_dinv.p, L.sm_rows.p, (const T*)SP.F.p, sweep == 0 ? 1 : 0, SP.fs[li].p,
                      SP.us[li].p));
        ++launches;
      }
    }
    auto RS = view(L.RS);
    LAUNCH(ASMG_PROF_AUX_RESID, L.RS.nnz_real * (sv + 4) + L.nrs_real * (4 + 2 * sz) + L.nsm_real * sz,
           launch(h.prm.use_pdl, k_resid_aux<T, V>, nblk(L.nrs, rows_tpb(L.nrs)), rows_tpb(L.nrs), s, L.nrs, RS.off, RS.col, sell_vals(L.RS, (const V*)nullptr), L.rs_rows.p,
                  (const T*)SP.us[li].p, SP.F.p));
    LAUNCH(ASMG_PROF_AUX_TRANSFER, L.nchild * (4 + sz) + L.npar * (8 + 2 * sz),
           launch(h.prm.use_pdl, k_restrict_aux<T>, nblk(L.npar, rows_tpb(L.npar)), rows_tpb(L.npar), s, L.npar, L.rp_id.p,
                  L.rp_ptr.p, L.rp_child.p, SP.F.p));
    launches += 2;
  }
  g_prof_level = -1;
  if (nbot) {
    LAUNCH(ASMG_PROF_AUX_SMALL, small_bytes(P.bot, true),
           small::launch_down<T, V, 1>(h.prm.use_pdl, P.bot, SP.F.p, SP.bot_fs.p, SP.bot_us.p, npre, s));
    ++launches;
  }
  if (h.nc > 0) {
    LAUNCH(ASMG_PROF_COARSE, h.nc * h.nc * 8 + h.nc * (4 + 2 * sz),
           launch(h.prm.use_pdl, k_coarse<T>, nblk(h.nc * 32), TPB, s, h.nc, h.d_cid.p, h.d_cinv.p, SP.F.p, SP.U.p));
    ++launches;
  }
  if (nbot) {
    LAUNCH(ASMG_PROF_AUX_SMALL, small_bytes(P.bot, false),
           small::launch_up<T, V, 1>(h.prm.use_pdl, P.bot, SP.U.p, SP.bot_fs.p, SP.bot_us.p, npost, s));
    ++launches;
  }
  for (int li = nbot; li <= nlev - 1 - ndeep; ++li) {
    AuxLevelDev<T>& L = P.lev[li];
    auto SM = view(L.SM);
    g_prof_level = -2 - li;
    if (L.tiled_up) {
      const TileSweeps<T>& Tl = L.tup;
      LAUNCH(ASMG_PROF_AUX_TRANSFER,
             L.nsm_real * (28 + 3 * sz) + L.nnew * 2 * sz + (L.nsm_real - L.nnew) * sz +
                 (Tl.interior + Tl.halo) * (4 + 2 * sz),
             launch(h.prm.use_pdl, k_up_init<T>, nblk(L.nsm, rows_tpb(L.nsm)), rows_tpb(L.nsm), s, L.nsm, L.sm_rows.p,
                    L.sm_par0.p, L.sm_par1.p, Tl.pos_ptr.p, Tl.pos.p, (const T*)SP.U.p, (const T*)SP.us[li].p,
                    (const T*)SP.fs[li].p, SP.ust[li].p, SP.fsl[li].p));
      const int64_t by = Tl.nnz_real * (sv + 2) + (Tl.interior + Tl.halo) * (8 + 3 * sz) + Tl.interior * (4 + sz);
      LAUNCH(ASMG_PROF_AUX_GS, by,
             tile_dispatch<T, V>(Tl, [&](auto sl, auto w) {
               constexpr int SL = decltype(sl)::value, W = decltype(w)::value;
               launch_smem(h.prm.use_pdl, k_tile_up<T, V, SL, W>,
                           std::min<int64_t>(Tl.ntiles, NSM * tile_min_blocks<T, V, SL, W>()), TILE_THREADS, Tl.smem(), s,
                           Tl.view(), L.ncolours, Tl.smem_values(), (const T*)SP.ust[li].p, (const T*)SP.fsl[li].p,
                           SP.U.p, npost, timeout_flag(S), h.prm.inject_timeout);
             }));
      launches += 2;
      continue;
    }
    if (L.nnew) {
      LAUNCH(ASMG_PROF_AUX_TRANSFER, L.nnew * (12 + 3 * sz),
             launch(h.prm.use_pdl, k_prolong_aux<T>, nblk(L.nnew, rows_tpb(L.nnew)), rows_tpb(L.nnew), s, L.nnew, L.nn_id.p, L.nn_p0.p, L.nn_p1.p,
                    SP.U.p));
      ++launches;
    }
    LAUNCH(ASMG_PROF_AUX_TRANSFER, L.nsm_real * (4 + 3 * sz),
           launch(h.prm.use_pdl, k_addsaved_aux<T>, nblk(L.nsm, rows_tpb(L.nsm)), rows_tpb(L.nsm), s, L.nsm, L.sm_rows.p, SP.us[li].p, SP.U.p));
    ++launches;
    if (L.nb.m > 0) {
      // Algorithm 3: exact solve on the near-boundary set after the coarse correction
      const NbDev& N = L.nb;
      LAUNCH(ASMG_PROF_AUX_NB, L.NB.nnz_real * (sz + 4) + N.m * (16 + 2 * sz),
             launch(h.prm.use_pdl, k_nb_resid<T>, nblk(N.m), TPB, s, N.m, L.NB.off.p, L.NB.col.p, L.NB.val.p, N.sm.p,
                    (const T*)SP.fs[li].p, (const T*)SP.U.p, SP.nbr[li].p));
      LAUNCH(ASMG_PROF_AUX_NB, (int64_t)N.mats.n * 8 + N.m * (8 + 2 * sz),
             launch(h.prm.use_pdl, k_nb_solve<T>, 1, NB_TPB, s, N.R, N.nblk.p, N.boff.p, N.btab.p, N.voff.p,
                    (const double*)N.mats.p, N.last_size, N.last_off, N.m, N.aux.p, SP.nbr[li].p, SP.nbs[li].p,
                    SP.U.p));
      launches += 2;
    }
    for (int sweep = 0; sweep < npost; ++sweep)
      for (int c = L.ncolours - 1; c >= 0; --c) {
        int64_t k0 = L.cstart[c], nk = L.cstart[c + 1] - L.cstart[c];
        if (!nk) continue;
        LAUNCH(ASMG_PROF_AUX_GS, L.cnnz[c] * (sv + 4) + L.crows[c] * (4 + 5 * sz),
               launch(h.prm.use_pdl, k_gs_aux<T, V>, nblk(nk, rows_tpb(nk)), rows_tpb(nk), s, k0, nk, SM.off, SM.col, sell_vals(L.SM, (const V*)nullptr), L.sm_dinv.p,
                      L.sm_rows.p, (const T*)SP.fs[li].p, SP.U.p));
        ++launches;
      }
  }
  g_prof_level = -1;
  if (ndeep) {
    LAUNCH(ASMG_PROF_AUX_SMALL, small_bytes(P.deep, false),
           small::launch_up<T, V, 1>(h.prm.use_pdl, P.deep, SP.U.p, SP.deep_fs.p, SP.deep_us.p, npost, s));
    ++launches;
  }
  return launches;
}

// the V-cycle with the level matrices read in BF16 (mixed form with
// level_bf16) or in the arithmetic type
template <class T>
int enqueue_vcycle_vals(asmg_s& h, Slot& S, cudaStream_t s) {
  if constexpr (std::is_same<T, float>::value)
    if (h.prm.level_bf16) return enqueue_vcycle<float, bf16v>(h, S, s);
  return enqueue_vcycle<T, T>(h, S, s);
}

template <class T>
int enqueue_precond(asmg_s& h, Slot& S, const double* r, cudaStream_t s) {
  Prec<T>& P = prec<T>(h);
  SlotPrec<T>& SP = slotprec<T>(S);
  const SellView<T> A = fine_smoother<T>(h);
  const T* dinv = fine_dinv<T>(h);
  const int64_t sz = sizeof(T), n = h.n, nJ = h.nJ;
  const bool jacobi = h.prm.smoother == 1, additive = h.prm.additive == 1;
  int launches = 0;
  ASMG_CUDA(cudaMemsetAsync(SP.uf.p, 0, sizeof(T) * h.npad, s));
  const int ncol = (int)h.fine_cstart.size() - 1;
  bool zero = true;  // uf is still 0
  // u <- u + S (r - A u) (forward) or u + S^t (r - A u) (backward), fine_sweeps times
  auto smooth = [&](bool forward) {
    for (int m = 0; m < h.prm.fine_sweeps; ++m) {
      if (!jacobi) {
        for (int q = 0; q < ncol; ++q) {
          const int c = forward ? q : ncol - 1 - q;
          int64_t r0 = h.fine_cstart[c], nr = h.fine_cstart[c + 1] - r0;
          if (!nr) continue;
          LAUNCH(ASMG_PROF_FINE_GS, h.fine_cnnz[c] * (sz + 4) + h.fine_crows[c] * (8 + 4 * sz),
                 launch(h.prm.use_pdl, k_gs_fine<T, double>, nblk(nr, rows_tpb(nr)), rows_tpb(nr), s, r0, nr, A.off,
                        A.col, A.val, dinv, r, SP.uf.p));
          ++launches;
        }
      } else if (zero) {
        LAUNCH(ASMG_PROF_FINE_GS, n * (8 + 2 * sz),
               launch(h.prm.use_pdl, k_jac_first<T>, nblk(h.npad), TPB, s, h.npad, dinv, r, SP.uf.p));
        ++launches;
      } else {
        LAUNCH(ASMG_PROF_FINE_GS, h.A64.nnz_real * (sz + 4) + n * (8 + 2 * sz),
               launch(h.prm.use_pdl, k_resid_fine<T>, nblk(h.npad), TPB, s, h.npad, A.off, A.col, A.val, r, SP.uf.p,
                      SP.rho.p));
        LAUNCH(ASMG_PROF_FINE_GS, n * 4 * sz,
               launch(h.prm.use_pdl, k_jac_add<T>, nblk(h.npad), TPB, s, h.npad, dinv, SP.rho.p, SP.uf.p));
        launches += 2;
      }
      zero = false;
    }
  };
  // (1) u1 = S r
  smooth(true);
  // (2) multiplicative: u2 = u1 + P Btilde P^T (r - A u1);  additive: u1 + P Btilde P^T r
  if (h.nJ > 0) {
    if (additive) {
      LAUNCH(ASMG_PROF_FINE_RESID, n * (8 + sz),
             launch(h.prm.use_pdl, k_cast_fine<T>, nblk(h.npad), TPB, s, h.npad, r, SP.rho.p));
    } else {
      LAUNCH(ASMG_PROF_FINE_RESID, h.A64.nnz_real * (sz + 4) + n * (8 + 2 * sz),
             launch(h.prm.use_pdl, k_resid_fine<T>, nblk(h.npad), TPB, s, h.npad, A.off, A.col, A.val, r, SP.uf.p,
                    SP.rho.p));
    }
    auto PT = view(P.PT);
    LAUNCH(ASMG_PROF_RESTRICT, P.PT.nnz_real * (sz + 4) + n * sz + 2 * nJ * sz,
           launch(h.prm.use_pdl, k_restrict_fine<T>, nblk(h.nJpad), TPB, s, h.nJpad, PT.off, PT.col, PT.val, SP.rho.p, SP.F.p, SP.U.p));
    launches += 2;
    launches += enqueue_vcycle_vals<T>(h, S, s);
    auto PP = view(P.P);
    LAUNCH(ASMG_PROF_PROLONG, P.P.nnz_real * (sz + 4) + nJ * sz + 2 * n * sz,
           launch(h.prm.use_pdl, k_prolong_fine<T>, nblk(h.npad), TPB, s, h.npad, PP.off, PP.col, PP.val, SP.U.p, SP.uf.p));
    ++launches;
  }
  // (3) multiplicative only: u3 = u2 + S^T (r - A u2)
  if (!additive) smooth(false);
  ASMG_CUDA(cudaGetLastError());
  return launches;
}

template <class T>
int enqueue_body(asmg_s& h, Slot& S, cudaStream_t s, cudaGraphConditionalHandle hnd, int use_hnd) {
  int launches = enqueue_precond<T>(h, S, S.r.p, s);
  const T* z = slotprec<T>(S).uf.p;
  const int G = red_grid(h.npad, RED_BLOCKS), GV = red_grid(h.npad, VEC_BLOCKS);
  const int64_t n = h.n, sz = sizeof(T);
  LAUNCH(ASMG_PROF_CG_VECTOR, n * (sz + 16),
         launch(h.prm.use_pdl, k_dots<T>, GV, TPB, s, h.npad, z, S.r.p, S.q.p, S.partial.p, S.ticket.p, S.scal.p));
  LAUNCH(ASMG_PROF_CG_VECTOR, n * (sz + 16), launch(h.prm.use_pdl, k_pupd<T>, GV, TPB, s, h.npad, z, S.p.p, S.scal.p));
  LAUNCH(ASMG_PROF_CG_SPMV, h.A64.nnz_real * 12 + n * 16,
         launch(h.prm.use_pdl, k_spmv_dot, G, TPB, s, h.npad, view(h.A64), S.p.p, S.q.p, S.partial.p, S.ticket.p, S.scal.p));
  LAUNCH(ASMG_PROF_CG_VECTOR, n * 48,
         launch(h.prm.use_pdl, k_axpy_norm, GV, TPB, s, h.npad, S.p.p, S.q.p, S.x.p, S.r.p, S.partial.p, S.ticket.p, S.scal.p,
                                       S.hist.p, hnd, use_hnd));
  ASMG_CUDA(cudaGetLastError());
  return launches + 4;
}

// the ASMG iteration: z = B r, x += z, r = b - A x, stopping test
template <class T>
int enqueue_iteration(asmg_s& h, Slot& S, cudaStream_t s, cudaGraphConditionalHandle hnd, int use_hnd) {
  int launches = enqueue_precond<T>(h, S, S.r.p, s);
  const T* z = slotprec<T>(S).uf.p;
  const int G = red_grid(h.npad, RED_BLOCKS);
  const int64_t n = h.n, sz = sizeof(T);
  LAUNCH(ASMG_PROF_CG_VECTOR, n * (sz + 16), launch(h.prm.use_pdl, k_xpz<T>, G, TPB, s, h.npad, z, S.x.p));
  LAUNCH(ASMG_PROF_CG_SPMV, h.A64.nnz_real * 12 + n * 24,
         launch(h.prm.use_pdl, k_iter_resid, G, TPB, s, h.npad, view(h.A64), S.b.p, S.x.p, S.r.p, S.partial.p,
                S.ticket.p, S.scal.p, S.hist.p, hnd, use_hnd));
  ASMG_CUDA(cudaGetLastError());
  return launches + 2;
}

int enqueue_body_any(asmg_s& h, Slot& S, cudaStream_t s, cudaGraphConditionalHandle hnd, int use_hnd) {
  if (h.prm.iteration == 1)
    return h.prm.precision == ASMG_MIXED ? enqueue_iteration<float>(h, S, s, hnd, use_hnd)
                                         : enqueue_iteration<double>(h, S, s, hnd, use_hnd);
  return h.prm.precision == ASMG_MIXED ? enqueue_body<float>(h, S, s, hnd, use_hnd)
                                       : enqueue_body<double>(h, S, s, hnd, use_hnd);
}

void enqueue_init(asmg_s& h, Slot& S, double rtol, cudaStream_t s, cudaGraphConditionalHandle hnd, int use_hnd) {
  LAUNCH(ASMG_PROF_CG_VECTOR, h.A64.nnz_real * 12 + h.n * 32,
         launch(h.prm.use_pdl, k_pcg_init, red_grid(h.npad, RED_BLOCKS), TPB, s, h.npad, view(h.A64), S.b.p, S.x.p, S.r.p, S.partial.p, S.ticket.p,
                                               S.scal.p, rtol, h.prm.max_iter, S.hist.p, hnd, use_hnd));
  ASMG_CUDA(cudaGetLastError());
}

}  // namespace

void gather_rows(asmg_s& h, const double* vsrc, double* dst, cudaStream_t s) {
  launch(false, k_gather, nblk(h.npad), TPB, s, h.npad, h.d_vertex_of_row.p, vsrc, dst);
  ASMG_CUDA(cudaGetLastError());
}

void gather_rows_tab(asmg_s& h, double* const* tab, double* dst, cudaStream_t s) {
  launch(false, k_gather_tab1, nblk(h.npad), TPB, s, h.npad, h.d_vertex_of_row.p, tab, dst);
  ASMG_CUDA(cudaGetLastError());
}

void scatter_rows_tab(asmg_s& h, const double* src, double* const* tab, cudaStream_t s) {
  launch(false, k_scatter_tab1, nblk(h.mesh.nv), TPB, s, h.mesh.nv, h.d_row_of_vertex.p, src, tab);
  ASMG_CUDA(cudaGetLastError());
}

void scatter_rows(asmg_s& h, const void* src, bool src_float, double* vdst, cudaStream_t s) {
  if (src_float)
    launch(false, k_scatter<float>, nblk(h.mesh.nv), TPB, s, h.mesh.nv, h.d_row_of_vertex.p, (const float*)src, vdst);
  else
    launch(false, k_scatter<double>, nblk(h.mesh.nv), TPB, s, h.mesh.nv, h.d_row_of_vertex.p, (const double*)src, vdst);
  ASMG_CUDA(cudaGetLastError());
}

// (u, lambda) of every vertex side by side, 0 at Dirichlet vertices
__global__ void k_mask_pair(int64_t nv, const int32_t* __restrict__ rowv, const double* __restrict__ u,
                            const double* __restrict__ lambda, double2* __restrict__ pair) {
  const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= nv) return;
  pair[v] = rowv[v] >= 0 ? make_double2(u[v], lambda[v]) : make_double2(0.0, 0.0);
}

void mask_pair(asmg_s& h, const double* u, const double* lambda, double* pair, cudaStream_t s) {
  launch(false, k_mask_pair, nblk(h.mesh.nv), TPB, s, h.mesh.nv, h.d_row_of_vertex.p, u, lambda,
         reinterpret_cast<double2*>(pair));
  ASMG_CUDA(cudaGetLastError());
}

void precond_apply(asmg_s& h, const double* r_perm, cudaStream_t s) {
  Slot& S = *h.slots[0];
  if (h.prm.precision == ASMG_MIXED)
    enqueue_precond<float>(h, S, r_perm, s);
  else
    enqueue_precond<double>(h, S, r_perm, s);
}

// y = A x, a row's entries loaded into registers at once
__global__ void k_spmv64(int64_t n, SellView<double> A, const double* __restrict__ x, double* __restrict__ y) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  Row<double> row;
  row_load(row, i, A.off, A.col, A.val);
  y[i] = row_dot(row, A.col, A.val, x);
}

void spmv64(asmg_s& h, const double* x, double* y, cudaStream_t s) {
  launch(false, k_spmv64, nblk(h.npad), TPB, s, h.npad, view(h.A64), x, y);
  ASMG_CUDA(cudaGetLastError());
}

// Capture the graph of one solve into `g` (independent of other nodes):
//   init (r = b - A x, norms, condition) -> WHILE(cond) { body }.
// Returns the WHILE node.
cudaGraphNode_t capture_solve(asmg_s& h, Slot& S, double rtol, cudaGraph_t g, const cudaGraphNode_t* deps,
                              size_t ndeps) {
  cudaGraphConditionalHandle hnd;
  ASMG_CUDA(cudaGraphConditionalHandleCreate(&hnd, g, 0, 0));
  cudaStream_t cs;
  ASMG_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  ASMG_CUDA(cudaStreamBeginCaptureToGraph(cs, g, deps, nullptr, ndeps, cudaStreamCaptureModeThreadLocal));
  enqueue_init(h, S, rtol, cs, hnd, 1);
  // the WHILE node depends on the captured init kernel (the leaf of this capture)
  cudaStreamCaptureStatus st;
  const cudaGraphNode_t* leaf = nullptr;
  size_t nleaf = 0;
  ASMG_CUDA(cudaStreamGetCaptureInfo(cs, &st, nullptr, nullptr, &leaf, nullptr, &nleaf));
  std::vector<cudaGraphNode_t> leaves(leaf, leaf + nleaf);
  cudaGraph_t gg;
  ASMG_CUDA(cudaStreamEndCapture(cs, &gg));
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = hnd;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t cnode;
  ASMG_CUDA(cudaGraphAddNode(&cnode, g, leaves.data(), nullptr, leaves.size(), &cp));
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  ASMG_CUDA(cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  h.gpu_launches_per_iter = enqueue_body_any(h, S, cs, hnd, 1);
  cudaGraph_t bb;
  ASMG_CUDA(cudaStreamEndCapture(cs, &bb));
  ASMG_CUDA(cudaStreamDestroy(cs));
  return cnode;
}

static void build_graph(asmg_s& h, Slot& S, double rtol) {
  if (S.gexec) {
    cudaGraphExecDestroy(S.gexec);
    S.gexec = nullptr;
  }
  if (S.graph) {
    cudaGraphDestroy(S.graph);
    S.graph = nullptr;
  }
  cudaGraph_t g;
  ASMG_CUDA(cudaGraphCreate(&g, 0));
  capture_solve(h, S, rtol, g, nullptr, 0);
  ASMG_CUDA(cudaGraphInstantiate(&S.gexec, g, 0));
  S.graph = g;
}

int run_solve(asmg_s& h, Slot& S, double rtol, cudaStream_t s) {
  if (h.prm.use_graph) {
    // the graph bakes rtol into the init kernel's arguments: rebuild when it changes
    if (!S.gexec || S.graph_rtol != rtol) {
      build_graph(h, S, rtol);
      S.graph_rtol = rtol;
    }
    ASMG_CUDA(cudaGraphLaunch(S.gexec, s));
  } else {
    enqueue_init(h, S, rtol, s, 0, 0);
    for (int it = 0; it < h.prm.max_iter; ++it) {
      PcgScalars sc;
      ASMG_CUDA(cudaMemcpyAsync(&sc, S.scal.p, sizeof sc, cudaMemcpyDeviceToHost, s));
      ASMG_CUDA(cudaStreamSynchronize(s));
      if (!sc.cond) break;
      h.gpu_launches_per_iter = enqueue_body_any(h, S, s, 0, 0);
    }
  }
  return 0;
}

// One solve without the graph, every launch timed: per class launches,
// milliseconds and algorithmic bytes; returns the iteration count.
int profile_solve(asmg_s& h, double rtol, cudaStream_t s, double* out, double* out_levels, int nlev_out) {
  Slot& S = *h.slots[0];
  Profiler prof;
  prof.s = s;
  g_prof = &prof;
  int its = 0;
  try {
    enqueue_init(h, S, rtol, s, 0, 0);
    for (int it = 0; it < h.prm.max_iter; ++it) {
      PcgScalars sc;
      ASMG_CUDA(cudaMemcpyAsync(&sc, S.scal.p, sizeof sc, cudaMemcpyDeviceToHost, s));
      ASMG_CUDA(cudaStreamSynchronize(s));
      if (!sc.cond) break;
      enqueue_body_any(h, S, s, 0, 0);
      ++its;
    }
    ASMG_CUDA(cudaStreamSynchronize(s));
  } catch (...) {
    g_prof = nullptr;
    throw;
  }
  g_prof = nullptr;
  for (int k = 0; k < 3 * ASMG_PROF_NCLASS; ++k) out[k] = 0;
  if (out_levels)
    for (int k = 0; k < nlev_out * 2 * 3 * 3; ++k) out_levels[k] = 0;
  for (auto& r : prof.recs) {
    float ms = 0;
    ASMG_CUDA(cudaEventElapsedTime(&ms, prof.ev[r.e0], prof.ev[r.e0 + 1]));
    out[3 * r.cls] += 1;
    out[3 * r.cls + 1] += ms;
    out[3 * r.cls + 2] += (double)r.bytes;
    if (out_levels && r.level != -1) {
      // [level][down, up][sweeps, residual, transfer][launches, ms, bytes]
      const int li = r.level >= 0 ? r.level : -2 - r.level, dir = r.level >= 0 ? 0 : 1;
      const int kind = r.cls == ASMG_PROF_AUX_GS ? 0 : r.cls == ASMG_PROF_AUX_RESID ? 1 : 2;
      if (li < nlev_out) {
        double* o = out_levels + ((li * 2 + dir) * 3 + kind) * 3;
        o[0] += 1;
        o[1] += ms;
        o[2] += (double)r.bytes;
      }
    }
  }
  return its;
}

// The fused small-level runs, for one and for KRHS right-hand sides, and the
// kernels' shared-memory limits.
template <class T>
void setup_small(Prec<T>& P, bool bf16, cudaStream_t s) {
  small::build_runs(P, bf16, 1, P.deep, P.bot, s);
  small::build_runs(P, bf16, KRHS, P.deep_k, P.bot_k, s);
  // the attribute belongs to the kernel, not to this handle: every handle sets
  // the same bound
  auto attrs = [&](auto vtag) {
    using V = decltype(vtag);
    small::set_smem_limits<T, V, 1>();
    for (int slots = 1; slots <= TILE_SLOTS_MAX; ++slots)
      for (int width : {8, TILE_MAXW}) {
        TileSweeps<T> Tl;
        Tl.slots = slots;
        Tl.width = width;
        tile_dispatch<T, V>(Tl, [&](auto sl, auto w) {
          ASMG_CUDA(cudaFuncSetAttribute(k_tile_down<T, V, decltype(sl)::value, decltype(w)::value>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM_MAX));
          ASMG_CUDA(cudaFuncSetAttribute(k_tile_up<T, V, decltype(sl)::value, decltype(w)::value>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM_MAX));
        });
      }
  };
  attrs(T{});
  if constexpr (std::is_same<T, float>::value) attrs(bf16v{});
}

// Work state of one solve in precision T: vectors and per-level saved values.
template <class T>
void alloc_slot_prec(asmg_s& h, Prec<T>& P, SlotPrec<T>& SP, cudaStream_t s) {
  SP.uf.alloc(h.npad);
  SP.rho.alloc(h.npad);
  SP.F.alloc(std::max<int64_t>(h.nJpad, 1));
  SP.U.alloc(std::max<int64_t>(h.nJpad, 1));
  SP.uf.zero(s);
  SP.rho.zero(s);
  SP.F.zero(s);
  SP.U.zero(s);
  const int nlev = (int)P.lev.size();
  SP.fs.clear();
  SP.us.clear();
  SP.fs.resize(nlev);
  SP.us.resize(nlev);
  SP.nbr.clear();
  SP.nbs.clear();
  SP.nbr.resize(nlev);
  SP.nbs.resize(nlev);
  SP.ust.clear();
  SP.fsl.clear();
  SP.ust.resize(nlev);
  SP.fsl.resize(nlev);
  for (int li = 0; li < nlev; ++li) {
    SP.fs[li].alloc(std::max<int64_t>(P.lev[li].nsm, 1));
    SP.us[li].alloc(std::max<int64_t>(P.lev[li].nsm, 1));
    SP.fs[li].zero(s);
    SP.us[li].zero(s);
    if (P.lev[li].tiled_up) {
      // post-sweep start values and saved rhs in tile order (padding rows stay 0)
      SP.ust[li].alloc(std::max<int64_t>(P.lev[li].tup.nloc, 1));
      SP.fsl[li].alloc(std::max<int64_t>(P.lev[li].tup.nloc, 1));
      SP.ust[li].zero(s);
      SP.fsl[li].zero(s);
    }
    const NbDev& N = P.lev[li].nb;
    if (N.m > 0) {
      // the pools: every round's vector and the last block's (voff[R + 1] doubles)
      int64_t pool = 0;
      {
        std::vector<int64_t> vo = N.voff.download(s);
        pool = vo.back();
      }
      SP.nbr[li].alloc(pool);
      SP.nbs[li].alloc(pool);
      SP.nbr[li].zero(s);
      SP.nbs[li].zero(s);
    }
  }
  for (DBuf<T>* v : {&SP.deep_fs, &SP.deep_us}) v->alloc(std::max(P.deep.v.nsm, 1));
  for (DBuf<T>* v : {&SP.bot_fs, &SP.bot_us}) v->alloc(std::max(P.bot.v.nsm, 1));
}

// Schedule of the auxiliary levels (the autotuner, tile_rows = 0): each
// direction of a level that has tiles runs either its temporally blocked
// sweeps or its launches per colour class and sweep, with the same results.
// The choice is made on the device: one preconditioner application is
// captured as a CUDA graph and timed (median of 3 runs of 5 launches) with
// every level tiled both ways, then for each level in turn the post-sweeps
// and then the pre-sweeps are switched to class launches, each switch kept
// when it is faster by more than 0.5% (and 2 us).  Tiles of a direction left
// untiled are freed.
template <class T>
void autotune_levels(asmg_s& h, cudaStream_t s) {
  Prec<T>& P = prec<T>(h);
  Slot& S = *h.slots[0];
  const int nlev = (int)P.lev.size();
  std::vector<int> cand;
  for (int li = P.bot.v.nlev; li <= nlev - 1 - P.deep.v.nlev; ++li)
    if (P.lev[li].tiled) cand.push_back(li);
  if (cand.empty()) return;
  cudaStream_t cs;
  ASMG_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  cudaEvent_t e0, e1;
  ASMG_CUDA(cudaEventCreate(&e0));
  ASMG_CUDA(cudaEventCreate(&e1));
  auto time_once = [&]() -> float {
    cudaGraph_t g;
    cudaGraphExec_t ge;
    ASMG_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    enqueue_precond<T>(h, S, S.r.p, cs);
    ASMG_CUDA(cudaStreamEndCapture(cs, &g));
    ASMG_CUDA(cudaGraphInstantiate(&ge, g, 0));
    float best[3];
    for (int rep = 0; rep < 3; ++rep) {
      ASMG_CUDA(cudaGraphLaunch(ge, cs));
      ASMG_CUDA(cudaEventRecord(e0, cs));
      for (int k = 0; k < 5; ++k) ASMG_CUDA(cudaGraphLaunch(ge, cs));
      ASMG_CUDA(cudaEventRecord(e1, cs));
      ASMG_CUDA(cudaEventSynchronize(e1));
      ASMG_CUDA(cudaEventElapsedTime(&best[rep], e0, e1));
    }
    ASMG_CUDA(cudaGraphExecDestroy(ge));
    ASMG_CUDA(cudaGraphDestroy(g));
    std::sort(best, best + 3);
    return best[1] / 5;
  };
  try {
    float cur = time_once();
    for (int li : cand)
      for (bool* flag : {&P.lev[li].tiled_up, &P.lev[li].tiled_down}) {
        *flag = false;
        const float t = time_once();
        if (t < cur * 0.995f && cur - t > 0.002f) {
          cur = t;
        } else {
          *flag = true;
        }
      }
  } catch (...) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamDestroy(cs);
    throw;
  }
  ASMG_CUDA(cudaEventDestroy(e0));
  ASMG_CUDA(cudaEventDestroy(e1));
  ASMG_CUDA(cudaStreamDestroy(cs));
  for (int li : cand) {
    AuxLevelDev<T>& L = P.lev[li];
    if (!L.tiled_down) L.tdown = TileSweeps<T>();
    if (!L.tiled_up) {
      L.tup = TileSweeps<T>();
      slotprec<T>(S).ust[li] = DBuf<T>();
      slotprec<T>(S).fsl[li] = DBuf<T>();
    }
    L.tiled = L.tiled_down || L.tiled_up;
  }
}

Slot& add_slot(asmg_s& h, cudaStream_t s) {
  h.slots.emplace_back(new Slot());
  Slot& S = *h.slots.back();
  S.b.alloc(h.npad);
  S.x.alloc(h.npad);
  S.r.alloc(h.npad);
  S.p.alloc(h.npad);
  S.q.alloc(h.npad);
  S.b.zero(s);
  S.x.zero(s);
  S.r.zero(s);
  S.p.zero(s);
  S.q.zero(s);
  S.vb.alloc(h.mesh.nv);
  S.vu.alloc(h.mesh.nv);
  S.partial.alloc(std::max(4 * RED_BLOCKS, 2 * VEC_BLOCKS));
  S.ticket.alloc(1);
  S.ticket.zero(s);
  S.scal.alloc(1);
  S.scal.zero(s);
  S.hist.alloc(h.prm.max_iter + 1);
  if (h.prm.precision == ASMG_MIXED)
    alloc_slot_prec(h, h.p32, S.s32, s);
  else
    alloc_slot_prec(h, h.p64, S.s64, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
  return S;
}

// Levels inside the fused small-level runs never use their tiles: drop them.
template <class T>
void drop_unused_tiles(Prec<T>& P) {
  const int nlev = (int)P.lev.size();
  for (int li = 0; li < nlev; ++li)
    if (li < P.bot.v.nlev || li > nlev - 1 - P.deep.v.nlev) {
      P.lev[li].tiled = P.lev[li].tiled_down = P.lev[li].tiled_up = false;
      P.lev[li].tdown = TileSweeps<T>();
      P.lev[li].tup = TileSweeps<T>();
    }
}

void setup_solve(asmg_s& h, cudaStream_t s) {
  if (h.prm.precision == ASMG_MIXED) {
    setup_small(h.p32, h.prm.level_bf16 == 1, s);
    drop_unused_tiles(h.p32);
  } else {
    setup_small(h.p64, false, s);
    drop_unused_tiles(h.p64);
  }
  h.slots.clear();
  add_slot(h, s);
  if (h.prm.tile_rows == 0 && !h.prm.inject_timeout) {
    if (h.prm.precision == ASMG_MIXED)
      autotune_levels<float>(h, s);
    else
      autotune_levels<double>(h, s);
  }
}

}  // namespace asmg
