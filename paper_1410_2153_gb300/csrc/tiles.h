// Temporally blocked sweeps of an auxiliary level (TileSweeps, built by
// build_tiles), for one right-hand side (KC = 1) or KRHS interleaved ones.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "handle.h"
#include "kernels.h"
#include "small_run.h"

namespace asmg {
namespace tiles {

using kern::pdl_wait;
using small::VecK;

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
  __device__ __forceinline__ T value(int e) const { return v[e]; }
  __device__ __forceinline__ uint32_t at(int e) const { return (e & 1) ? c[e / 2] >> 16 : c[e / 2] & 0xffffu; }
};
template <class T, int W>
struct TileRow<T, bf16v, W> {
  uint32_t c[W];
  __device__ __forceinline__ void load(const uint32_t* words, const T*, const TileSlice& h, int lane) {
#pragma unroll
    for (int e = 0; e < W; ++e) c[e] = e < h.w ? words[(h.words + e) * 32 + lane] : 0u;
  }
  __device__ __forceinline__ T value(int e) const { return (T)__uint_as_float(c[e] & 0xffff0000u); }
  __device__ __forceinline__ uint32_t at(int e) const { return c[e] & 0xffffu; }
};
template <class T, class V, int W, int KC>
__device__ __forceinline__ void tile_term(const TileRow<T, V, W>& row, const char* u, int e, VecK<T, KC>& acc) {
  const VecK<T, KC> x = *reinterpret_cast<const VecK<T, KC>*>(u + row.at(e) * KC);
  const T a = row.value(e);
#pragma unroll
  for (int j = 0; j < KC; ++j) acc.v[j] += a * x.v[j];
}
template <class T, class V, int W, int KC>
__device__ __forceinline__ VecK<T, KC> tile_dot(const TileRow<T, V, W>& row, const char* u, int w) {
  constexpr int A0 = W <= 8 ? 6 : 8;
  VecK<T, KC> acc;
#pragma unroll
  for (int j = 0; j < KC; ++j) acc.v[j] = 0;
#pragma unroll
  for (int e = 0; e < A0; ++e) tile_term(row, u, e, acc);
#pragma unroll
  for (int e = A0; e < W; e += 2)
    if (w > e) {
      tile_term(row, u, e, acc);
      tile_term(row, u, e + 1, acc);
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
  // one colour phase: u += (f - A u) / a_ii on the thread's rows of class c.
  // One column keeps its rows' f and u in registers; KC columns read them from
  // shared memory (f at Fl).
  template <int KC>
  __device__ __forceinline__ void phase(int c, VecK<T, KC>* Ul, const VecK<T, KC>* Fl, const VecK<T, KC> (&f)[S],
                                        VecK<T, KC> (&u)[S]) const {
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (wc[s] >> 8 == c) {
        const int q = s * TILE_THREADS + threadIdx.x;
        const VecK<T, KC> acc = tile_dot<T, V, W, KC>(row[s], reinterpret_cast<const char*>(Ul), wc[s] & 255);
        const VecK<T, KC> fq = KC == 1 ? f[s] : Fl[q];
        VecK<T, KC> uq = KC == 1 ? u[s] : Ul[q];
#pragma unroll
        for (int j = 0; j < KC; ++j) uq.v[j] += (fq.v[j] - acc.v[j]) * di[s];
        if (KC == 1) u[s] = uq;
        Ul[q] = uq;
      }
  }
};

// blocks per SM the kernels are compiled for: the most whose registers hold the
// rows (a few spilled words cost less than a fourth block gives, BF16: level of
// 3.46 M rows 115 us with three blocks, 80 us with four)
template <class T, class V, int S, int W, int KC>
constexpr int tile_min_blocks() {
  if (sizeof(T) == 8) return KC > 1 ? (W > 8 || S > 2 ? 1 : 2) : W > 8 ? (S > 2 ? 1 : 2) : S > 2 ? 2 : 3;
  if (KC > 1) return W > 8 ? 2 : 3;
  return W > 8 ? 2 : S == 4 && !std::is_same<V, bf16v>::value ? 3 : 4;
}

// pre-sweeps: us (the level's own correction, SM order) starts at 0; the
// first sweep saves F on the tile's own rows in fs.  Their residual F - A us
// goes to fr: the rows are still in registers, where a launch of its own reads
// the level's matrix once more (331^2 mixed 1,536 -> 1,486 us, holed 257^2 mixed
// 1,917 -> 1,795 us, graded 2049^2 BF16 210.2 -> 205.1 ms).
template <class T, class V, int S, int W, int KC>
__global__ void __launch_bounds__(TILE_THREADS, tile_min_blocks<T, V, S, W, KC>())
    k_tile_down(TileView<T> t, int ncol, int fofs, int bofs, const T* __restrict__ Fg, T* __restrict__ fsg,
                T* __restrict__ usg, T* __restrict__ frg, int nu, int* timeout, int inject) {
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t bar;
  using X = VecK<T, KC>;
  X* Ul = reinterpret_cast<X*>(smraw);
  X* Fl = reinterpret_cast<X*>(smraw + fofs);  // KC > 1 only
  unsigned char* blob = smraw + bofs;
  const int tid = threadIdx.x;
  const X* F = reinterpret_cast<const X*>(Fg);
  X* fs = reinterpret_cast<X*>(fsg);
  X* us = reinterpret_cast<X*>(usg);
  X* fr = reinterpret_cast<X*>(frg);
  X zero;
#pragma unroll
  for (int j = 0; j < KC; ++j) zero.v[j] = 0;
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
    X f[S], u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      f[s] = R.g[s] != -1 ? F[R.ax[s]] : zero;
      u[s] = zero;
      Ul[s * TILE_THREADS + tid] = zero;
      if (KC > 1) Fl[s * TILE_THREADS + tid] = f[s];
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
        R.phase(c, Ul, Fl, f, u);
        __syncthreads();
      }
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (R.g[s] >= 0) {
        const int q = s * TILE_THREADS + tid;
        us[R.g[s]] = KC == 1 ? u[s] : Ul[q];
        const X acc = tile_dot<T, V, W, KC>(R.row[s], reinterpret_cast<const char*>(Ul), R.wc[s] & 255);
        X fq = KC == 1 ? f[s] : Fl[q];
#pragma unroll
        for (int j = 0; j < KC; ++j) fq.v[j] -= acc.v[j];
        fr[R.g[s]] = fq;
      }
    if (!more) return;
    parity ^= 1;
    ok = tile_arrived(&bar, parity, inject);
    if (ok) R.load(blob, h, tile_layout(h.slots, h.nwords, h.nvals, h.nx, sizeof(T)));
  }
  tile_expired(&bar, parity, timeout);
}

// index lists of a row (children, places in the tiles) read before the wait on
// the previous kernel; longer ones read the rest after it (331^2 mixed 1,487 ->
// 1,465 us, graded 513^2 FP64 28.6 -> 28.1 ms, graded 2049^2 BF16 205.2 -> 202.7 ms)
constexpr int AHEAD = 4;

// after tiled pre-sweeps: the residual and the restricted part of every node
// the coarser levels read (see TileRestrict)
template <class T, class V, int KC>
__global__ void k_restrict_tile(int64_t n1, int64_t n, const int32_t* __restrict__ id, const int32_t* __restrict__ src,
                                const int32_t* __restrict__ ptr, const int32_t* __restrict__ child,
                                const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                                const V* __restrict__ val, const T* __restrict__ frg, const T* __restrict__ usg,
                                T* __restrict__ Fg) {
  using X = VecK<T, KC>;
  const X* fr = reinterpret_cast<const X*>(frg);
  const X* us = reinterpret_cast<const X*>(usg);
  X* F = reinterpret_cast<X*>(Fg);
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1, k = 0, p0 = 0, p1 = 0;
  int32_t ch[AHEAD];
  kern::Row<T> row;
  if (t < n) {
    i = id[t];
    p0 = ptr[t];
    p1 = ptr[t + 1];
#pragma unroll
    for (int q = 0; q < AHEAD; ++q)
      if (p0 + q < p1) ch[q] = child[p0 + q];
    if (t < n1)
      k = src[t];
    else if (i >= 0)
      kern::row_load(row, t - n1, off, col, val);
  }
  pdl_wait();
  if (i >= 0) {
    X f;
    if (t < n1) {
      f = fr[k];
    } else {
      X acc;
#pragma unroll
      for (int j = 0; j < KC; ++j) acc.v[j] = 0;
#pragma unroll
      for (int q = 0; q < kern::MAXW; ++q)
        if (q < row.w) {
          const X x = us[row.c[q]];
#pragma unroll
          for (int j = 0; j < KC; ++j) acc.v[j] += row.v[q] * x.v[j];
        }
      for (int q = kern::MAXW; q < row.w; ++q) {
        const int64_t e = row.b + ((int64_t)q << 5) + row.lane;
        const T a = (T)kern::ldg_val(val + e);
        const X x = us[__ldg(col + e)];
#pragma unroll
        for (int j = 0; j < KC; ++j) acc.v[j] += a * x.v[j];
      }
      f = F[i];
#pragma unroll
      for (int j = 0; j < KC; ++j) f.v[j] -= acc.v[j];
    }
    if (p1 > p0) {
      X acc;
#pragma unroll
      for (int j = 0; j < KC; ++j) acc.v[j] = 0;
      auto add = [&](int32_t c) {
        const X x = fr[c];
#pragma unroll
        for (int j = 0; j < KC; ++j) acc.v[j] += x.v[j];
      };
#pragma unroll
      for (int q = 0; q < AHEAD; ++q)
        if (p0 + q < p1) add(ch[q]);
      for (int32_t p = p0 + AHEAD; p < p1; ++p) add(child[p]);
#pragma unroll
      for (int j = 0; j < KC; ++j) f.v[j] += (T)0.5 * acc.v[j];
    }
    F[i] = f;
  }
}

// start of the up path of a tiled level: the prolongation of the coarse
// correction (I_l: new nodes take the mean of their parents) plus the level's
// saved correction, and the saved rhs, written for every SM row to each place
// the row holds in the post-sweep tiles (own and halo copies; TileSweeps::
// pos).  U itself is not written, so the tiles can read their start values
// while other tiles write their results to U.
template <class T, int KC>
__global__ void k_up_init(int64_t nsm, const int32_t* __restrict__ rows, const int32_t* __restrict__ par0,
                          const int32_t* __restrict__ par1, const int64_t* __restrict__ pos_ptr,
                          const int32_t* __restrict__ pos, const T* __restrict__ Ug, const T* __restrict__ usg,
                          const T* __restrict__ fsg, T* __restrict__ ustg, T* __restrict__ fslg) {
  using X = VecK<T, KC>;
  const X* U = reinterpret_cast<const X*>(Ug);
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1, a = -3, b = -3;
  int64_t p0 = 0, p1 = 0;
  int32_t at[AHEAD];
  if (k < nsm) {
    i = rows[k];
    a = par0[k];
    b = par1[k];
    p0 = pos_ptr[k];
    p1 = pos_ptr[k + 1];
#pragma unroll
    for (int q = 0; q < AHEAD; ++q)
      if (p0 + q < p1) at[q] = pos[p0 + q];
  }
  pdl_wait();
  if (i >= 0) {
    X v;
    if (a == -3) {
      v = U[i];
    } else {
#pragma unroll
      for (int j = 0; j < KC; ++j) v.v[j] = 0;
      if (a >= 0) {
        const X p = U[a];
#pragma unroll
        for (int j = 0; j < KC; ++j) v.v[j] += p.v[j];
      }
      if (b >= 0) {
        const X p = U[b];
#pragma unroll
        for (int j = 0; j < KC; ++j) v.v[j] += p.v[j];
      }
#pragma unroll
      for (int j = 0; j < KC; ++j) v.v[j] = (T)0.5 * v.v[j];
    }
    const X s = reinterpret_cast<const X*>(usg)[k], f = reinterpret_cast<const X*>(fsg)[k];
#pragma unroll
    for (int j = 0; j < KC; ++j) v.v[j] = v.v[j] + s.v[j];
    auto put = [&](int32_t o) {
      reinterpret_cast<X*>(ustg)[o] = v;
      reinterpret_cast<X*>(fslg)[o] = f;
    };
#pragma unroll
    for (int q = 0; q < AHEAD; ++q)
      if (p0 + q < p1) put(at[q]);
    for (int64_t q = p0 + AHEAD; q < p1; ++q) put(pos[q]);
  }
}

// post-sweeps (backward colour order) from the start values and saved rhs
// that k_up_init wrote in tile order (`per` local rows a tile); the columns
// outside N~_l (the tile's outside values) are read from U once; the tile's
// own rows are written to U
template <class T, class V, int S, int W, int KC>
__global__ void __launch_bounds__(TILE_THREADS, tile_min_blocks<T, V, S, W, KC>())
    k_tile_up(TileView<T> t, int ncol, int fofs, int bofs, const T* __restrict__ ustg, const T* __restrict__ fslg,
              T* Ug, int nu, int* timeout, int inject) {
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t bar;
  using X = VecK<T, KC>;
  X* Ul = reinterpret_cast<X*>(smraw);
  X* Fl = reinterpret_cast<X*>(smraw + fofs);  // KC > 1 only
  unsigned char* blob = smraw + bofs;
  const int tid = threadIdx.x;
  const X* ust = reinterpret_cast<const X*>(ustg);
  const X* fsl = reinterpret_cast<const X*>(fslg);
  X* U = reinterpret_cast<X*>(Ug);
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
    X f[S], u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      u[s] = ust[base + s * TILE_THREADS];
      f[s] = fsl[base + s * TILE_THREADS];
    }
    const int32_t* ext = reinterpret_cast<const int32_t*>(blob + lay.ext);
    for (int e = tid; e < h.nx; e += TILE_THREADS) Ul[S * TILE_THREADS + e] = U[ext[e]];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      Ul[s * TILE_THREADS + tid] = u[s];
      if (KC > 1) Fl[s * TILE_THREADS + tid] = f[s];
    }
    const uint32_t mask = h.cmask;
    tile += gridDim.x;
    const bool more = tile < t.ntiles;
    if (more) h = t.head[tile];
    __syncthreads();  // values in place, the block read by all
    if (tid == 0 && more) tile_fetch(blob, t.blob, h, &bar);
    for (int sw = 0; sw < nu; ++sw)
      for (int c = ncol - 1; c >= 0; --c) {
        if (!((mask >> min(c, 31)) & 1u)) continue;
        R.phase(c, Ul, Fl, f, u);
        __syncthreads();
      }
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (R.g[s] >= 0) U[R.ax[s]] = KC == 1 ? u[s] : Ul[s * TILE_THREADS + tid];
    if (!more) return;
    lay = tile_layout(h.slots, h.nwords, h.nvals, h.nx, sizeof(T));
    parity ^= 1;
    ok = tile_arrived(&bar, parity, inject);
    if (ok) R.load(blob, h, lay);
  }
  tile_expired(&bar, parity, timeout);
}

// f(slots, width) with the tile kernels' compile-time sizes for a level's tiles
template <class T, class F>
void dispatch(const TileSweeps<T>& Tl, F f) {
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

// shared memory of a launch: the values, with KC > 1 the rows' rhs, the block
template <class T>
struct Smem {
  int fofs, bofs;
  int64_t total;
  Smem(const TileSweeps<T>& Tl, int kc) {
    auto pad = [](int64_t b) { return (b + 127) / 128 * 128; };
    const int64_t rows = (int64_t)Tl.slots * TILE_THREADS;
    fofs = (int)pad((rows + Tl.maxext) * kc * (int64_t)sizeof(T));
    bofs = fofs + (int)(kc > 1 ? pad(rows * kc * (int64_t)sizeof(T)) : 0);
    total = bofs + Tl.maxblob;
  }
};
constexpr int64_t SMEM_MAX_K = 200 * 1024;  // KC > 1

template <class T, class V, int KC>
void set_smem_limits() {
  for (int slots = 1; slots <= TILE_SLOTS_MAX; ++slots)
    for (int width : {8, TILE_MAXW}) {
      TileSweeps<T> Tl;
      Tl.slots = slots;
      Tl.width = width;
      dispatch(Tl, [&](auto sl, auto w) {
        const int limit = (int)(KC > 1 ? SMEM_MAX_K : TILE_SMEM_MAX);
        ASMG_CUDA(cudaFuncSetAttribute(k_tile_down<T, V, decltype(sl)::value, decltype(w)::value, KC>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
        ASMG_CUDA(cudaFuncSetAttribute(k_tile_up<T, V, decltype(sl)::value, decltype(w)::value, KC>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
      });
    }
}

template <class T, class V, int KC>
void launch_down(bool pdl, const TileSweeps<T>& Tl, int ncol, const T* F, T* fs, T* us, T* fr, int nu, int* timeout,
                 int inject, cudaStream_t s) {
  const Smem<T> sm(Tl, KC);
  dispatch(Tl, [&](auto sl, auto w) {
    constexpr int S = decltype(sl)::value, W = decltype(w)::value;
    kern::launch_smem(pdl, k_tile_down<T, V, S, W, KC>,
                      std::min<int64_t>(Tl.ntiles, kern::NSM * tile_min_blocks<T, V, S, W, KC>()), TILE_THREADS,
                      (size_t)sm.total, s, Tl.view(), ncol, sm.fofs, sm.bofs, F, fs, us, fr, nu, timeout, inject);
  });
}
template <class T, class V, int KC>
void launch_restrict(bool pdl, const TileRestrict<T>& R, const T* fr, const T* us, T* F, cudaStream_t s) {
  const int64_t n = R.n1 + R.n2;
  if (n == 0) return;
  kern::launch(pdl, k_restrict_tile<T, V, KC>, kern::nblk(n, kern::rows_tpb(n)), kern::rows_tpb(n), s, R.n1, n, R.id.p,
               R.src.p, R.ptr.p, R.child.p, R.X.off.p, R.X.col.p, sell_vals(R.X, (const V*)nullptr), fr, us, F);
}
template <class T, class V, int KC>
void launch_up(bool pdl, const TileSweeps<T>& Tl, int ncol, const T* ust, const T* fsl, T* U, int nu, int* timeout,
               int inject, cudaStream_t s) {
  const Smem<T> sm(Tl, KC);
  dispatch(Tl, [&](auto sl, auto w) {
    constexpr int S = decltype(sl)::value, W = decltype(w)::value;
    kern::launch_smem(pdl, k_tile_up<T, V, S, W, KC>,
                      std::min<int64_t>(Tl.ntiles, kern::NSM * tile_min_blocks<T, V, S, W, KC>()), TILE_THREADS,
                      (size_t)sm.total, s, Tl.view(), ncol, sm.fofs, sm.bofs, ust, fsl, U, nu, timeout, inject);
  });
}

}  // namespace tiles
}  // namespace asmg
