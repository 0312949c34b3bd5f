// Runs of small auxiliary levels in one thread block, for one right-hand side
// (KC = 1) or KRHS interleaved ones.
//
// A run's levels share one numbering of their nodes (the union of their rows
// E_l), so the rhs F and the correction U of the whole run live in shared
// memory from its first level to its last: they are read from global memory
// once at the start and written once at the end.  The run's setup data --
// rows in ELL form with 16-bit union columns, diagonal inverses, parents --
// is one block of bytes, copied into shared memory before the wait on the
// previous kernel.  Colour phases are separated by __syncthreads; the steps
// are those of k_gs_aux_down / k_resid_aux / k_restrict_aux (down) and
// k_prolong_aux / k_addsaved_aux / k_gs_aux (up), with a row's product
// subtracted from its rhs entry by entry.
//
// What bounds a run is the chain of phases on one SM, so only levels of at
// most small_lmax rows join one; larger levels are quicker spread over the SMs
// by the tiled sweeps.  Kernels that took levels of 8,192 rows and read each
// level's rows from global memory in every phase: 65^2 FP64 1,435 us per solve,
// graded 513^2 FP64 38.4 ms, 331^2 mixed 2,008 us; the same with levels above
// 1,024 rows tiled 917 us, 32.4 ms, 1,727 us; these kernels 776 us, 29.7 ms,
// 1,626 us.
//
// Rows of more than SMALL_MAXW entries (locally refined 3D grids: 19 to 27 on
// levels whose mean is 8) keep their first entries in ELL form and the rest in
// CSR, in kernels of their own; the ELL width is the one that takes the fewest
// entries.  Such levels, which no tile takes, join a run up to twice the rows:
// a launch per colour class and sweep is 24 to 32 launches for 88 or 1,024 rows.
// 25^3 vertices mapped by x -> x^3, no level fused -> the two finest: mixed
// 27.6 -> 26.6 ms, BF16 27.5 -> 26.5 ms; 41^3 mixed 68.9 -> 66.0 ms.  With a
// fixed ELL width of 16 the level of 1,024 rows does not fit in FP32 (27.4 ms),
// with the limit at 1,024 rows it stays out in BF16 too (27.3 ms).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <unordered_map>
#include <vector>

#include "handle.h"
#include "kernels.h"

namespace asmg {
namespace small {

using kern::pdl_wait;
using kern::val_of;

// the KC columns of one row of an interleaved vector
template <class T, int KC>
struct alignas(KC * sizeof(T) >= 16 ? 16 : KC * sizeof(T)) VecK {
  T v[KC];
};

// acc - sum_e val[e] x[col[e]] over row k of an ELL block of width w (stored order)
template <class T, class V, int W, int KC>
__device__ __forceinline__ void ell_sub(VecK<T, KC>& acc, const uint16_t* col, const V* val, int mp, int k, int w,
                                        const VecK<T, KC>* x) {
  int c[W];
  T v[W];
#pragma unroll
  for (int e = 0; e < W; ++e)
    if (e < w) {
      c[e] = col[e * mp + k];
      v[e] = (T)val_of(val[e * mp + k]);
    }
#pragma unroll
  for (int e = 0; e < W; ++e)
    if (e < w) {
      const VecK<T, KC> xe = x[c[e]];
#pragma unroll
      for (int j = 0; j < KC; ++j) acc.v[j] -= v[e] * xe.v[j];
    }
}

// W of the kernels for runs with rows of more than SMALL_MAXW entries
constexpr int SMALL_LONG = SMALL_MAXW + 1;

// acc less row k's product (stored order): ELL entries, and with W = SMALL_LONG
// what follows them in CSR
template <class T, class V, int W, int KC>
__device__ __forceinline__ void row_sub(VecK<T, KC>& acc, const uint16_t* col, const V* val, int mp, int k, int w,
                                        const unsigned char* B, const SmallRest& R, const VecK<T, KC>* x) {
  ell_sub<T, V, (W < SMALL_MAXW ? W : SMALL_MAXW), KC>(acc, col, val, mp, k, w, x);
  if constexpr (W == SMALL_LONG)
    if (R.ptr) {
      const uint16_t* ptr = reinterpret_cast<const uint16_t*>(B + R.ptr);
      const uint16_t* c = reinterpret_cast<const uint16_t*>(B + R.col);
      const V* v = reinterpret_cast<const V*>(B + R.val);
      for (int p = ptr[k]; p < ptr[k + 1]; ++p) {
        const VecK<T, KC> xe = x[c[p]];
        const T a = (T)val_of(v[p]);
#pragma unroll
        for (int j = 0; j < KC; ++j) acc.v[j] -= a * xe.v[j];
      }
    }
}

__device__ __forceinline__ void stage(unsigned char* dst, const unsigned char* src, int bytes) {
  for (int o = threadIdx.x * 16; o < bytes; o += blockDim.x * 16)
    *reinterpret_cast<uint4*>(dst + o) = __ldg(reinterpret_cast<const uint4*>(src + o));
}

// pre-smoothing, residual and restriction of the run's levels, finest first;
// fs and us: saved rhs and corrections of the levels' smoothing rows
template <class T, class V, int W, int KC>
__global__ void __launch_bounds__(1024, 1)
    k_small_down(SmallRunView R, T* Fg, T* fsg, T* usg, int nu) {
  extern __shared__ __align__(16) unsigned char smraw[];
  using X = VecK<T, KC>;
  X* F = reinterpret_cast<X*>(smraw);
  X* U = reinterpret_cast<X*>(smraw + small_pad16((int64_t)R.nunion * sizeof(X)));
  unsigned char* B = smraw + 2 * small_pad16((int64_t)R.nunion * sizeof(X));
  const int tid = threadIdx.x, nt = blockDim.x;
  stage(B, R.blob, R.bytes);
  X zero;
#pragma unroll
  for (int j = 0; j < KC; ++j) zero.v[j] = 0;
  for (int i = tid; i < R.nunion; i += nt) U[i] = zero;
  __syncthreads();
  const int32_t* gid = reinterpret_cast<const int32_t*>(B + R.o_gid);
  X* Fx = reinterpret_cast<X*>(Fg);
  X* fsx = reinterpret_cast<X*>(fsg);
  X* usx = reinterpret_cast<X*>(usg);
  pdl_wait();
  for (int i = tid; i < R.nunion; i += nt) F[i] = Fx[gid[i]];
  __syncthreads();
  for (int d = 0; d < R.nlev; ++d) {
    const SmallHead& L = reinterpret_cast<const SmallHead*>(B)[d];
    const uint16_t* row = reinterpret_cast<const uint16_t*>(B + L.o_row);
    const T* dinv = reinterpret_cast<const T*>(B + L.o_dinv);
    const uint16_t* smc = reinterpret_cast<const uint16_t*>(B + L.o_smc);
    const V* smv = reinterpret_cast<const V*>(B + L.o_smv);
    for (int k = tid; k < L.mS; k += nt) fsx[L.sm0 + k] = F[row[k]];
    for (int sw = 0; sw < nu; ++sw)
      for (int c = 0; c < L.ncol; ++c) {
        for (int k = L.cs[c] + tid; k < L.cs[c + 1]; k += nt) {
          const int r = row[k];
          X acc = F[r], u = U[r];
          row_sub<T, V, W, KC>(acc, smc, smv, L.mSp, k, L.wsm, B, L.sm_rest, U);
          const T di = dinv[k];
#pragma unroll
          for (int j = 0; j < KC; ++j) u.v[j] += acc.v[j] * di;
          U[r] = u;
        }
        __syncthreads();
      }
    const uint16_t* rsc = reinterpret_cast<const uint16_t*>(B + L.o_rsc);
    const V* rsv = reinterpret_cast<const V*>(B + L.o_rsv);
    for (int k = tid; k < L.mE; k += nt) {
      const int r = row[k];
      X acc = F[r];
      row_sub<T, V, W, KC>(acc, rsc, rsv, L.mEp, k, L.wrs, B, L.rs_rest, U);
      F[r] = acc;
    }
    __syncthreads();
    const uint16_t* rid = reinterpret_cast<const uint16_t*>(B + L.o_rid);
    const uint16_t* rptr = reinterpret_cast<const uint16_t*>(B + L.o_rptr);
    const uint16_t* rch = reinterpret_cast<const uint16_t*>(B + L.o_rch);
    for (int t = tid; t < L.npar; t += nt) {
      X acc = zero;
      for (int p = rptr[t]; p < rptr[t + 1]; ++p) {
        const X f = F[rch[p]];
#pragma unroll
        for (int j = 0; j < KC; ++j) acc.v[j] += f.v[j];
      }
      X f = F[rid[t]];
#pragma unroll
      for (int j = 0; j < KC; ++j) f.v[j] += (T)0.5 * acc.v[j];
      F[rid[t]] = f;
    }
    // the next level's correction starts from 0
    for (int k = tid; k < L.mS; k += nt) {
      usx[L.sm0 + k] = U[row[k]];
      U[row[k]] = zero;
    }
    __syncthreads();
  }
  for (int i = tid; i < R.nunion; i += nt) Fx[gid[i]] = F[i];
}

// prolongation, saved corrections and post-smoothing, coarsest level first
template <class T, class V, int W, int KC>
__global__ void __launch_bounds__(1024, 1)
    k_small_up(SmallRunView R, T* Ug, const T* fsg, const T* usg, int nu) {
  extern __shared__ __align__(16) unsigned char smraw[];
  using X = VecK<T, KC>;
  const int64_t usz = small_pad16((int64_t)R.nunion * sizeof(X)), ssz = small_pad16((int64_t)R.nsm * sizeof(X));
  X* U = reinterpret_cast<X*>(smraw);
  X* fs = reinterpret_cast<X*>(smraw + usz);
  X* us = reinterpret_cast<X*>(smraw + usz + ssz);
  unsigned char* B = smraw + usz + 2 * ssz;
  const int tid = threadIdx.x, nt = blockDim.x;
  stage(B, R.blob, R.up_bytes);
  __syncthreads();
  const int32_t* gid = reinterpret_cast<const int32_t*>(B + R.o_gid);
  X* Ux = reinterpret_cast<X*>(Ug);
  const X* fsx = reinterpret_cast<const X*>(fsg);
  const X* usx = reinterpret_cast<const X*>(usg);
  pdl_wait();
  for (int i = tid; i < R.nunion; i += nt) U[i] = Ux[gid[i]];
  for (int i = tid; i < R.nsm; i += nt) {
    fs[i] = fsx[i];
    us[i] = usx[i];
  }
  __syncthreads();
  for (int d = R.nlev - 1; d >= 0; --d) {
    const SmallHead& L = reinterpret_cast<const SmallHead*>(B)[d];
    const uint16_t* row = reinterpret_cast<const uint16_t*>(B + L.o_row);
    const T* dinv = reinterpret_cast<const T*>(B + L.o_dinv);
    const uint16_t* smc = reinterpret_cast<const uint16_t*>(B + L.o_smc);
    const V* smv = reinterpret_cast<const V*>(B + L.o_smv);
    const uint16_t* nn = reinterpret_cast<const uint16_t*>(B + L.o_nn);  // id, parent 0, parent 1 [nnew] each
    for (int t = tid; t < L.nnew; t += nt) {
      const int a = nn[L.nnew + t], b = nn[2 * L.nnew + t];
      X v;
#pragma unroll
      for (int j = 0; j < KC; ++j) {
        v.v[j] = 0;
        if (a != SMALL_NONE) v.v[j] += U[a].v[j];
        if (b != SMALL_NONE) v.v[j] += U[b].v[j];
        v.v[j] = (T)0.5 * v.v[j];
      }
      U[nn[t]] = v;
    }
    __syncthreads();
    for (int k = tid; k < L.mS; k += nt) {
      X u = U[row[k]];
      const X s = us[L.sm0 + k];
#pragma unroll
      for (int j = 0; j < KC; ++j) u.v[j] += s.v[j];
      U[row[k]] = u;
    }
    __syncthreads();
    for (int sw = 0; sw < nu; ++sw)
      for (int c = L.ncol - 1; c >= 0; --c) {
        for (int k = L.cs[c] + tid; k < L.cs[c + 1]; k += nt) {
          const int r = row[k];
          X acc = fs[L.sm0 + k], u = U[r];
          row_sub<T, V, W, KC>(acc, smc, smv, L.mSp, k, L.wsm, B, L.sm_rest, U);
          const T di = dinv[k];
#pragma unroll
          for (int j = 0; j < KC; ++j) u.v[j] += acc.v[j] * di;
          U[r] = u;
        }
        __syncthreads();
      }
  }
  for (int i = tid; i < R.nunion; i += nt) Ux[gid[i]] = U[i];
}

template <class T>
int64_t smem_down(const SmallRun<T>& R, int kc) {
  return 2 * small_pad16((int64_t)R.v.nunion * kc * sizeof(T)) + R.v.bytes;
}
template <class T>
int64_t smem_up(const SmallRun<T>& R, int kc) {
  return small_pad16((int64_t)R.v.nunion * kc * sizeof(T)) + 2 * small_pad16((int64_t)R.v.nsm * kc * sizeof(T)) +
         R.v.up_bytes;
}

// The run over the levels li (finest first): its block of setup data, in B.
// Returns false when the run does not fit one block's shared memory with kc
// columns.
template <class T>
bool build_run(const Prec<T>& P, const std::vector<int>& li, bool bf16, int kc, SmallRun<T>& R,
               std::vector<unsigned char>& B) {
  R = SmallRun<T>();
  R.v.nlev = (int)li.size();
  B.clear();
  auto put = [&](const void* p, size_t bytes) {
    const int32_t at = (int32_t)B.size();
    B.resize((size_t)small_pad16((int64_t)(at + bytes)), 0);
    if (bytes) std::memcpy(B.data() + at, p, bytes);
    return at;
  };
  std::vector<SmallHead> head(li.size());
  put(head.data(), head.size() * sizeof(SmallHead));
  std::unordered_map<int32_t, int32_t> at;
  std::vector<int32_t> gid;
  std::vector<std::vector<uint16_t>> rows;
  int max_rows = 0, width = 0;
  for (size_t d = 0; d < li.size(); ++d) {
    const SmallLevel<T>& M = P.lev[li[d]].small;
    std::vector<uint16_t> row(M.mE);
    for (int k = 0; k < M.mE; ++k) {
      const auto it = at.emplace(M.gid[k], (int32_t)gid.size());
      if (it.second) gid.push_back(M.gid[k]);
      row[k] = (uint16_t)it.first->second;
    }
    rows.push_back(std::move(row));
    max_rows = std::max(max_rows, M.mE);
  }
  if (gid.size() >= SMALL_NONE) return false;
  R.v.nunion = (int)gid.size();
  R.v.o_gid = put(gid.data(), gid.size() * sizeof(int32_t));
  auto values = [&](const std::vector<T>& v) {
    if (!bf16) return put(v.data(), v.size() * sizeof(T));
    std::vector<bf16v> b(v.size());
    for (size_t q = 0; q < v.size(); ++q) b[q].bits = bf16_bits((float)v[q]);
    return put(b.data(), b.size() * sizeof(bf16v));
  };
  // ELL form of rows given as CSR over local columns, and the entries past SMALL_MAXW
  bool fits = true;
  auto ell = [&](const std::vector<uint16_t>& row, const std::vector<int32_t>& ptr, const std::vector<uint16_t>& col,
                 const std::vector<T>& val, int& mp, int& w, int32_t& oc, int32_t& ov, SmallRest& rest) {
    const int m = (int)ptr.size() - 1;
    mp = (m + 31) / 32 * 32;
    int longest = 0;
    for (int k = 0; k < m; ++k) longest = std::max(longest, ptr[k + 1] - ptr[k]);
    width = std::max(width, longest);
    w = longest;
    if (longest > SMALL_MAXW) {
      // the ELL width that takes the fewest entries, padding included
      int64_t least = INT64_MAX;
      for (int x = 1; x <= SMALL_MAXW; ++x) {
        int64_t n = (int64_t)x * mp;
        for (int k = 0; k < m; ++k) n += std::max(0, ptr[k + 1] - ptr[k] - x);
        if (n <= least) {
          least = n;
          w = x;
        }
      }
    }
    std::vector<uint16_t> c((size_t)w * mp, 0), xp(1, 0), xc;
    std::vector<T> v((size_t)w * mp, (T)0), xv;
    for (int k = 0; k < m; ++k) {
      for (int p = ptr[k], e = 0; p < ptr[k + 1]; ++p, ++e) {
        if (e < w) {
          c[(size_t)e * mp + k] = row[col[p]];
          v[(size_t)e * mp + k] = val[p];
        } else {
          xc.push_back(row[col[p]]);
          xv.push_back(val[p]);
        }
      }
      xp.push_back((uint16_t)xc.size());
    }
    oc = put(c.data(), c.size() * sizeof(uint16_t));
    ov = values(v);
    rest = SmallRest{0, 0, 0};
    if (xc.empty()) return;
    if (xc.size() > UINT16_MAX) fits = false;
    rest.ptr = put(xp.data(), xp.size() * sizeof(uint16_t));
    rest.col = put(xc.data(), xc.size() * sizeof(uint16_t));
    rest.val = values(xv);
  };
  for (size_t d = 0; d < li.size(); ++d) {  // what both directions read
    const SmallLevel<T>& M = P.lev[li[d]].small;
    SmallHead& H = head[d];
    H.mS = M.mS;
    H.mE = M.mE;
    H.ncol = M.ncol;
    H.nnew = (int)M.nn_id.size();
    H.npar = (int)M.rp_id.size();
    H.sm0 = R.v.nsm;
    R.v.nsm += M.mS;
    for (int c = 0; c <= SMALL_MAXC; ++c) H.cs[c] = c <= M.ncol ? M.cs[c] : M.mS;
    H.o_row = put(rows[d].data(), rows[d].size() * sizeof(uint16_t));
    H.o_dinv = put(M.dinv.data(), M.dinv.size() * sizeof(T));
    ell(rows[d], M.sm_ptr, M.sm_col, M.sm_val, H.mSp, H.wsm, H.o_smc, H.o_smv, H.sm_rest);
    std::vector<uint16_t> nn;
    for (uint16_t k : M.nn_id) nn.push_back(rows[d][k]);
    for (const auto* p : {&M.nn_p0, &M.nn_p1})
      for (int32_t k : *p) nn.push_back(k < 0 ? (uint16_t)SMALL_NONE : rows[d][k]);
    H.o_nn = put(nn.data(), nn.size() * sizeof(uint16_t));
  }
  R.v.up_bytes = (int32_t)B.size();
  for (size_t d = 0; d < li.size(); ++d) {
    const SmallLevel<T>& M = P.lev[li[d]].small;
    SmallHead& H = head[d];
    ell(rows[d], M.rs_ptr, M.rs_col, M.rs_val, H.mEp, H.wrs, H.o_rsc, H.o_rsv, H.rs_rest);
    std::vector<uint16_t> id, ptr, ch;
    for (uint16_t k : M.rp_id) id.push_back(rows[d][k]);
    for (int32_t p : M.rp_ptr) ptr.push_back((uint16_t)p);
    for (uint16_t k : M.rp_child) ch.push_back(rows[d][k]);
    H.o_rid = put(id.data(), id.size() * sizeof(uint16_t));
    H.o_rptr = put(ptr.data(), ptr.size() * sizeof(uint16_t));
    H.o_rch = put(ch.data(), ch.size() * sizeof(uint16_t));
  }
  R.v.bytes = (int32_t)B.size();
  std::memcpy(B.data(), head.data(), head.size() * sizeof(SmallHead));
  R.width = width;
  R.threads = std::min(1024, std::max(128, (max_rows + 31) / 32 * 32));
  if (!fits || smem_down(R, kc) > SMALL_SMEM_MAX || smem_up(R, kc) > SMALL_SMEM_MAX) return false;
  return true;
}

// The fused runs of a hierarchy for kc columns: the longest run of small levels
// from the finest level down and from the coarsest V-cycle level up.
template <class T>
void build_runs(const Prec<T>& P, bool bf16, int kc, SmallRun<T>& deep, SmallRun<T>& bot, cudaStream_t s) {
  const int nlev = (int)P.lev.size();
  // the longest prefix of the given order of levels that fits (a run's size
  // grows with every level it takes)
  auto longest = [&](std::vector<int> order, bool finest_first, SmallRun<T>& out) {
    out = SmallRun<T>();
    std::vector<unsigned char> B;
    for (size_t n = order.size(); n > 0; --n) {
      std::vector<int> li(order.begin(), order.begin() + n);
      if (!finest_first) std::reverse(li.begin(), li.end());
      if (!build_run(P, li, bf16, kc, out, B)) {
        out = SmallRun<T>();
        continue;
      }
      out.blob.upload(B, s);
      out.v.blob = out.blob.p;
      ASMG_CUDA(cudaStreamSynchronize(s));
      return;
    }
  };
  std::vector<int> order;
  for (int k = nlev - 1; k >= 0 && P.lev[k].small.ok; --k) order.push_back(k);
  longest(order, true, deep);
  order.clear();
  for (int k = 0; k < nlev - deep.v.nlev && P.lev[k].small.ok; ++k) order.push_back(k);
  longest(order, false, bot);
}

// f(width) with the kernels' compile-time row width
template <class F>
void run_width(int width, F f) {
  if (width <= 8)
    f(std::integral_constant<int, 8>{});
  else if (width <= SMALL_MAXW)
    f(std::integral_constant<int, SMALL_MAXW>{});
  else
    f(std::integral_constant<int, SMALL_LONG>{});
}

template <class T, class V, int KC>
void set_smem_limits() {
  for (int w : {8, SMALL_MAXW, SMALL_LONG})
    run_width(w, [&](auto W) {
      ASMG_CUDA(cudaFuncSetAttribute(k_small_down<T, V, decltype(W)::value, KC>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM_MAX));
      ASMG_CUDA(cudaFuncSetAttribute(k_small_up<T, V, decltype(W)::value, KC>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM_MAX));
    });
}

template <class T, class V, int KC>
void launch_down(bool pdl, const SmallRun<T>& R, T* F, T* fs, T* us, int nu, cudaStream_t s) {
  run_width(R.width, [&](auto W) {
    kern::launch_smem(pdl, k_small_down<T, V, decltype(W)::value, KC>, 1, R.threads, (size_t)smem_down(R, KC), s, R.v,
                      F, fs, us, nu);
  });
}
template <class T, class V, int KC>
void launch_up(bool pdl, const SmallRun<T>& R, T* U, T* fs, T* us, int nu, cudaStream_t s) {
  run_width(R.width, [&](auto W) {
    kern::launch_smem(pdl, k_small_up<T, V, decltype(W)::value, KC>, 1, R.threads, (size_t)smem_up(R, KC), s, R.v, U,
                      (const T*)fs, (const T*)us, nu);
  });
}

}  // namespace small
}  // namespace asmg
