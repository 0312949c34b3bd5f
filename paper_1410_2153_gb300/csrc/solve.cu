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
#include "tiles.h"

namespace asmg {

namespace {

using namespace kern;

// ------------------------------------------------------------- fine grid
// one colour of a Gauss-Seidel sweep: u_i += (rhs_i - (A u)_i) / a_ii
template <class T, class R, int N>
__global__ void k_gs_fine(int64_t r0, int64_t nrows, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                          const T* __restrict__ val, const T* __restrict__ dinv, const R* __restrict__ rhs, T* u) {
  const int64_t i = r0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < r0 + nrows;
  Row<T, N> row;
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

// The forward sweep of S from u = 0 and the residual after it, on the halves of
// A they can read.  A row of class c reads only the values of earlier classes
// (Lo: columns before its class); afterwards its own equation holds for the
// values it saw, so the residual is minus the product with the later classes
// (Up): r_i - (A u)_i = -sum_{j later} a_ij u_j.  Together they read A once
// where a full sweep and a full residual read it twice, and the sweep needs no
// cleared u.  With the first and last class's steps taken by the CG kernels:
// 65^2 FP64 758 -> 718 us per solve, kuhn129 mixed 39.3 -> 36.6 ms.
template <class T, int N>
__global__ void k_gs_first(int64_t r0, int64_t nrows, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                           const T* __restrict__ val, const T* __restrict__ dinv, const double* __restrict__ rhs,
                           T* u) {
  const int64_t i = r0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < r0 + nrows;
  Row<T, N> row;
  T di = 0;
  if (act) {
    row_load(row, i, off, col, val);
    di = dinv[i];
  }
  pdl_wait();
  if (act) {
    const T s = (T)rhs[i] - row_dot(row, col, val, u);
    u[i] = s * di;
  }
}

template <class T, int N>
__global__ void k_resid_upper(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                              const T* __restrict__ val, const T* __restrict__ u, T* __restrict__ rho) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < n;
  Row<T, N> row;
  if (act) row_load(row, i, off, col, val);
  pdl_wait();
  if (act) rho[i] = -row_dot(row, col, val, u);
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
template <class T, int N>
__global__ void k_restrict_fine(int64_t nJ, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                                const T* __restrict__ val, const T* __restrict__ rho, T* __restrict__ F,
                                T* __restrict__ U) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = k < nJ;
  Row<T, N> row;
  if (act) row_load(row, k, off, col, val);
  pdl_wait();
  if (act) {
    F[k] = row_dot(row, col, val, rho);
    U[k] = 0;
  }
}

// u += P U
template <class T, int N>
__global__ void k_prolong_fine(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                               const T* __restrict__ val, const T* __restrict__ U, T* __restrict__ u) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool act = i < n;
  Row<T, N> row;
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
template <class T, class V, int N>
__global__ void k_gs_aux(int64_t k0, int64_t nk, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                         const V* __restrict__ val, const T* __restrict__ dinv, const int32_t* __restrict__ rows,
                         const T* __restrict__ fs, T* U) {
  const int64_t k = k0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1;
  Row<T, N> row;
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
template <class T, class V, int N>
__global__ void k_gs_aux_down(int64_t k0, int64_t nk, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                              const V* __restrict__ val, const T* __restrict__ dinv, const int32_t* __restrict__ rows,
                              const T* __restrict__ F, int first, T* __restrict__ fs, T* us) {
  const int64_t k = k0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1;
  Row<T, N> row;
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
      for (int q = 0; q < N; ++q)
        if (q < row.w && row.c[q] < k0) acc += row.v[q] * us[row.c[q]];
      for (int q = N; q < row.w; ++q) {
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
template <class T, class V, int N>
__global__ void k_resid_aux(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                            const V* __restrict__ val, const int32_t* __restrict__ rows, const T* __restrict__ U,
                            T* __restrict__ F) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int32_t i = -1;
  Row<T, N> row;
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

// coarsest level: U[cid] = A_c^{-1} F[cid] in FP64, one warp per row.  A lane's
// part of the row and its node IDs (setup data; the default cap of 512 nodes
// is 16 entries) are in registers before the wait on the previous kernel.
constexpr int COARSE_W = 16;
template <class T>
__global__ void k_coarse(int64_t nc, const int32_t* __restrict__ cid, const double* __restrict__ inv,
                         const T* __restrict__ F, T* __restrict__ U) {
  const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  double a[COARSE_W];
  int32_t id[COARSE_W];
  int32_t out = 0;
  if (row < nc) {
#pragma unroll
    for (int q = 0; q < COARSE_W; ++q) {
      const int64_t j = lane + 32 * q;
      if (j < nc) {
        a[q] = inv[row * nc + j];
        id[q] = cid[j];
      }
    }
    out = cid[row];
  }
  pdl_wait();
  if (row < nc) {
    double s = 0;
#pragma unroll
    for (int q = 0; q < COARSE_W; ++q)
      if (lane + 32 * q < nc) s += a[q] * (double)F[id[q]];
    for (int64_t j = lane + 32 * COARSE_W; j < nc; j += 32) s += inv[row * nc + j] * (double)F[cid[j]];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) U[out] = (T)s;
  }
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

// r = b - A x;  ||b||, ||r||; PCG scalars initialised.  The first n0 rows (the
// first colour class, which reads no other) also take the forward sweep's step
// u = r / a_ii, saving that launch; so does k_axpy_norm for the next iteration.
template <class T>
__global__ void k_pcg_init(int64_t n, SellView<double> A, const double* __restrict__ b, const double* __restrict__ x,
                           double* __restrict__ r, int64_t n0, const T* __restrict__ dinv, T* __restrict__ u,
                           double* partial, unsigned int* ticket, PcgScalars* sc, double rtol,
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
    if (i < n0) u[i] = (T)ri * dinv[i];
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
    sc->rz_next = 0;
    sc->alpha = 0;
    sc->beta = 0;
    sc->timeout = 0;
    hist[0] = sqrt(v[1]);
    const bool conv = sqrt(v[1]) <= sc->tol;
    if (conv) sc->status = 0;
    set_cond(sc, (!conv && maxit > 0) ? 1 : 0, hnd, use_hnd);
  }
}

// beta of this step from <z, q_prev> and the scalars of the step before
__device__ __forceinline__ double step_beta(const PcgScalars& sc, double zq) {
  return sc.k == 0 ? 0.0 : -sc.alpha * zq / sc.rz;
}
// alpha of this step from <p, q>; 0 on breakdown
__device__ __forceinline__ double step_alpha(const PcgScalars& sc, double pq) {
  return !(pq > 0) || sc.status == ASMG_ERR_BREAKDOWN ? 0.0 : sc.rz_next / pq;
}

// <z, r>, <z, q_prev>  ->  beta (flexible: -alpha <z_{k+1}, q_k> / <z_k, r_k>), rz.
// The first n0 rows (colour class 0, the last of the backward sweep) take their
// Gauss-Seidel step here: every other class is done, and no row reads theirs
// after it.
template <class T>
__global__ void k_dots(int64_t n, int64_t n0, SellView<T> A, const T* __restrict__ dinv, T* z,
                       const double* __restrict__ r, const double* __restrict__ q, double* partial,
                       unsigned int* ticket, PcgScalars* sc, int direct) {
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  Row<T> row;
  if (i0 < n0) row_load(row, i0, A.off, A.col, A.val);
  pdl_wait();
  double v[2] = {0, 0};
  int64_t i = i0;
  for (; i < n0; i += st) {
    if (i != i0) row_load(row, i, A.off, A.col, A.val);
    const double ri = r[i];
    const T s = (T)ri - row_dot(row, A.col, A.val, z);
    const T zi = z[i] + s * dinv[i];
    z[i] = zi;
    v[0] += (double)zi * ri;
    v[1] += (double)zi * q[i];
  }
#pragma unroll 4
  for (; i < n; i += st) {
    double zi = (double)z[i];
    v[0] += zi * r[i];
    v[1] += zi * q[i];
  }
  if (direct) {
    block_partials(v, partial);  // k_pupd sums them
  } else if (grid_reduce<2>(v, partial, ticket) && threadIdx.x == 0) {
    sc->beta = step_beta(*sc, v[1]);
    sc->rz_next = v[0];
    if (!(v[0] > 0)) sc->status = ASMG_ERR_BREAKDOWN;
  }
}

// p = z + beta p; nb > 0: beta from the nb partials of k_dots
template <class T>
__global__ void k_pupd(int64_t n, const T* __restrict__ z, double* __restrict__ p, const double* partial, int nb,
                       PcgScalars* sc) {
  __shared__ double sh_beta;
  pdl_wait();
  double beta;
  if (nb) {
    double v[2];
    sum_partials(v, partial, (unsigned)nb);
    if (threadIdx.x == 0) {
      sh_beta = step_beta(*sc, v[1]);  // reads k, alpha and rz, which this kernel does not write
      if (blockIdx.x == 0) {
        sc->beta = sh_beta;
        sc->rz_next = v[0];
        if (!(v[0] > 0)) sc->status = ASMG_ERR_BREAKDOWN;
      }
    }
    __syncthreads();
    beta = sh_beta;
  } else {
    beta = sc->beta;
  }
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = (double)z[i] + beta * p[i];
}

// q = A p, <p, q>  ->  alpha.  Each row's entries are loaded into registers
// at once (row_load), the thread's first row before the wait on the previous
// kernel (graded 2049^2: 3.1 -> 4.3 TB/s against a plain loop over the row).
template <int N>
__global__ void k_spmv_dot(int64_t n, SellView<double> A, const double* __restrict__ p, double* __restrict__ q,
                           double* partial, unsigned int* ticket, PcgScalars* sc, int direct) {
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  Row<double, N> row;
  if (i0 < n) row_load(row, i0, A.off, A.col, A.val);
  pdl_wait();
  double v[1] = {0};
  for (int64_t i = i0; i < n; i += st) {
    if (i != i0) row_load(row, i, A.off, A.col, A.val);
    const double qi = row_dot(row, A.col, A.val, p);
    q[i] = qi;
    v[0] += p[i] * qi;
  }
  if (direct) {
    block_partials(v, partial);  // k_axpy_norm sums them
  } else if (grid_reduce<1>(v, partial, ticket) && threadIdx.x == 0) {
    sc->pq = v[0];
    sc->alpha = step_alpha(*sc, v[0]);
    if (!(v[0] > 0)) sc->status = ASMG_ERR_BREAKDOWN;
  }
}

// x += alpha p, r -= alpha q, ||r||  ->  history, stopping test; on the first
// n0 rows the next forward sweep's first step (see k_pcg_init)
template <class T>
__global__ void k_axpy_norm(int64_t n, const double* __restrict__ p, const double* __restrict__ q,
                            double* __restrict__ x, double* __restrict__ r, int64_t n0, const T* __restrict__ dinv,
                            T* __restrict__ u, const double* pq_partial, int nb, double* partial,
                            unsigned int* ticket, PcgScalars* sc, double* hist, cudaGraphConditionalHandle hnd,
                            int use_hnd) {
  __shared__ double sh_alpha;
  pdl_wait();
  double a;
  if (nb) {  // alpha from the nb partials of k_spmv_dot
    double pq[1];
    sum_partials(pq, pq_partial, (unsigned)nb);
    if (threadIdx.x == 0) {
      sh_alpha = step_alpha(*sc, pq[0]);  // a breakdown written below leaves this 0 in every block
      if (blockIdx.x == 0) {
        sc->pq = pq[0];
        sc->alpha = sh_alpha;
        if (!(pq[0] > 0)) sc->status = ASMG_ERR_BREAKDOWN;
      }
    }
    __syncthreads();
    a = sh_alpha;
  } else {
    a = sc->alpha;
  }
  double v[1] = {0};
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] += a * p[i];
    double ri = r[i] - a * q[i];
    r[i] = ri;
    if (i < n0) u[i] = (T)ri * dinv[i];
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
    sc->rz = sc->rz_next;
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
thread_local int64_t* g_count_bytes = nullptr;  // set: launches only add up their bytes

#define LAUNCH(cls, bytes, ...)                                                  \
  do {                                                                          \
    if (g_count_bytes) {                                                        \
      *g_count_bytes += (int64_t)(bytes);                                       \
      break;                                                                    \
    }                                                                           \
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
      const int64_t by = Tl.nnz_real * (sv + 2) + (Tl.interior + Tl.halo) * (8 + 2 * sz) + Tl.interior * (4 + 2 * sz);
      LAUNCH(ASMG_PROF_AUX_GS, by,
             (tiles::launch_down<T, V, 1>(h.prm.use_pdl, Tl, L.ncolours, SP.F.p, SP.fs[li].p, SP.us[li].p, SP.fr[li].p, npre,
                                          timeout_flag(S), h.prm.inject_timeout, s)));
      const TileRestrict<T>& R = L.trest;
      LAUNCH(ASMG_PROF_AUX_TRANSFER, R.X.nnz_real * (sv + 4) + R.n1 * (12 + 2 * sz) + R.n2 * (8 + 2 * sz) + R.nchild * (4 + sz),
             (tiles::launch_restrict<T, V, 1>(h.prm.use_pdl, R, SP.fr[li].p, SP.us[li].p, SP.F.p, s)));
      launches += 2;
      continue;
    }
    // pre-sweeps on us (SM order); the first also saves F on N~_l for the
    // post-sweeps (nu_pre >= 1)
    for (int sweep = 0; sweep < npre; ++sweep) {
      for (int c = 0; c < L.ncolours; ++c) {
        int64_t k0 = L.cstart[c], nk = L.cstart[c + 1] - L.cstart[c];
        if (!nk) continue;
        const int64_t by = L.cnnz_d[c] * (sv + 4) + L.crows[c] * (4 + (sweep == 0 ? 4 + 4 * sz : 4 * sz));
        LAUNCH(ASMG_PROF_AUX_GS, by,
               (by_rows(nk, [&](auto w) {
               launch(h.prm.use_pdl, k_gs_aux_down<T, V, decltype(w)::value>, nblk(nk, rows_tpb(nk)), rows_tpb(nk), s, k0, nk, SMd.off,
                      SMd.col, sell_vals(L.SMd, (const V*)nullptr), L.sm_dinv.p, L.sm_rows.p, (const T*)SP.F.p, sweep == 0 ? 1 : 0, SP.fs[li].p,
                      SP.us[li].p);
             })));
        ++launches;
      }
    }
    auto RS = view(L.RS);
    LAUNCH(ASMG_PROF_AUX_RESID, L.RS.nnz_real * (sv + 4) + L.nrs_real * (4 + 2 * sz) + L.nsm_real * sz,
           (by_rows(L.nrs, [&](auto w) {
               launch(h.prm.use_pdl, k_resid_aux<T, V, decltype(w)::value>, nblk(L.nrs, rows_tpb(L.nrs)), rows_tpb(L.nrs), s, L.nrs, RS.off, RS.col, sell_vals(L.RS, (const V*)nullptr), L.rs_rows.p,
                  (const T*)SP.us[li].p, SP.F.p);
             })));
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
             launch(h.prm.use_pdl, tiles::k_up_init<T, 1>, nblk(L.nsm, rows_tpb(L.nsm)), rows_tpb(L.nsm), s, L.nsm, L.sm_rows.p,
                    L.sm_par0.p, L.sm_par1.p, Tl.pos_ptr.p, Tl.pos.p, (const T*)SP.U.p, (const T*)SP.us[li].p,
                    (const T*)SP.fs[li].p, SP.ust[li].p, SP.fsl[li].p));
      const int64_t by = Tl.nnz_real * (sv + 2) + (Tl.interior + Tl.halo) * (8 + 3 * sz) + Tl.interior * (4 + sz);
      LAUNCH(ASMG_PROF_AUX_GS, by,
             (tiles::launch_up<T, V, 1>(h.prm.use_pdl, Tl, L.ncolours, SP.ust[li].p, SP.fsl[li].p, SP.U.p, npost,
                                        timeout_flag(S), h.prm.inject_timeout, s)));
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
               (by_rows(nk, [&](auto w) {
               launch(h.prm.use_pdl, k_gs_aux<T, V, decltype(w)::value>, nblk(nk, rows_tpb(nk)), rows_tpb(nk), s, k0, nk, SM.off, SM.col, sell_vals(L.SM, (const V*)nullptr), L.sm_dinv.p,
                      L.sm_rows.p, (const T*)SP.fs[li].p, SP.U.p);
             })));
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

// The Gauss-Seidel sweep from u = 0 runs on the halves of A (see k_gs_first).
bool split_sweep(const asmg_s& h) { return h.prm.smoother == 0 && h.prm.fine_sweeps == 1; }
// PCG steps end and begin inside the neighbouring CG kernels (k_dots, k_axpy_norm)
int64_t fused_rows(const asmg_s& h) {
  return split_sweep(h) && !h.prm.additive && h.prm.iteration == 0 && h.fine_cstart.size() > 1 ? h.fine_cstart[1] : 0;
}

// first_done, last_later: the first class's forward step was taken by the
// kernel before, the last backward one is left to the kernel after
template <class T>
int enqueue_precond(asmg_s& h, Slot& S, const double* r, cudaStream_t s, bool first_done = false,
                    bool last_later = false) {
  Prec<T>& P = prec<T>(h);
  SlotPrec<T>& SP = slotprec<T>(S);
  const SellView<T> A = fine_smoother<T>(h);
  const T* dinv = fine_dinv<T>(h);
  const int64_t sz = sizeof(T), n = h.n, nJ = h.nJ;
  const bool jacobi = h.prm.smoother == 1, additive = h.prm.additive == 1, split = split_sweep(h);
  int launches = 0;
  const int ncol = (int)h.fine_cstart.size() - 1;
  bool zero = true;  // uf is still 0
  // u <- u + S (r - A u) (forward) or u + S^t (r - A u) (backward), fine_sweeps times
  auto smooth = [&](bool forward) {
    for (int m = 0; m < h.prm.fine_sweeps; ++m) {
      if (!jacobi) {
        for (int q = 0; q < ncol; ++q) {
          const int c = forward ? q : ncol - 1 - q;
          int64_t r0 = h.fine_cstart[c], nr = h.fine_cstart[c + 1] - r0;
          if (!nr || (!forward && last_later && c == 0 && m == h.prm.fine_sweeps - 1)) continue;
          LAUNCH(ASMG_PROF_FINE_GS, h.fine_cnnz[c] * (sz + 4) + h.fine_crows[c] * (8 + 4 * sz),
                 (by_rows(nr, [&](auto w) {
               launch(h.prm.use_pdl, k_gs_fine<T, double, decltype(w)::value>, nblk(nr, rows_tpb(nr)), rows_tpb(nr), s, r0, nr, A.off,
                        A.col, A.val, dinv, r, SP.uf.p);
             })));
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
  if (split) {
    auto Lo = view(P.Lo);
    for (int c = first_done ? 1 : 0; c < ncol; ++c) {
      const int64_t r0 = h.fine_cstart[c], nr = h.fine_cstart[c + 1] - r0;
      if (!nr) continue;
      LAUNCH(ASMG_PROF_FINE_GS, h.fine_lnnz[c] * (sz + 4) + h.fine_crows[c] * (8 + 3 * sz),
             (by_rows(nr, [&](auto w) {
               launch(h.prm.use_pdl, k_gs_first<T, decltype(w)::value>, nblk(nr, rows_tpb(nr)), rows_tpb(nr), s, r0, nr, Lo.off, Lo.col,
                    Lo.val, dinv, r, SP.uf.p);
             })));
      ++launches;
    }
  } else {
    if (!g_count_bytes) ASMG_CUDA(cudaMemsetAsync(SP.uf.p, 0, sizeof(T) * h.npad, s));
    smooth(true);
  }
  // (2) multiplicative: u2 = u1 + P Btilde P^T (r - A u1);  additive: u1 + P Btilde P^T r
  if (h.nJ > 0) {
    if (additive) {
      LAUNCH(ASMG_PROF_FINE_RESID, n * (8 + sz),
             launch(h.prm.use_pdl, k_cast_fine<T>, nblk(h.npad), TPB, s, h.npad, r, SP.rho.p));
    } else if (split) {
      auto Up = view(P.Up);
      LAUNCH(ASMG_PROF_FINE_RESID, P.Up.nnz_real * (sz + 4) + n * 2 * sz,
             (by_rows(h.npad, [&](auto w) {
               launch(h.prm.use_pdl, k_resid_upper<T, decltype(w)::value>, nblk(h.npad), TPB, s, h.npad, Up.off, Up.col, Up.val,
                    (const T*)SP.uf.p, SP.rho.p);
             })));
    } else {
      LAUNCH(ASMG_PROF_FINE_RESID, h.A64.nnz_real * (sz + 4) + n * (8 + 2 * sz),
             launch(h.prm.use_pdl, k_resid_fine<T>, nblk(h.npad), TPB, s, h.npad, A.off, A.col, A.val, r, SP.uf.p,
                    SP.rho.p));
    }
    auto PT = view(P.PT);
    LAUNCH(ASMG_PROF_RESTRICT, P.PT.nnz_real * (sz + 4) + n * sz + 2 * nJ * sz,
           (by_rows<TRANSFER_W>(h.nJpad, [&](auto w) {
               launch(h.prm.use_pdl, k_restrict_fine<T, decltype(w)::value>, nblk(h.nJpad), TPB, s, h.nJpad, PT.off, PT.col, PT.val, SP.rho.p, SP.F.p, SP.U.p);
             })));
    launches += 2;
    launches += enqueue_vcycle_vals<T>(h, S, s);
    auto PP = view(P.P);
    LAUNCH(ASMG_PROF_PROLONG, P.P.nnz_real * (sz + 4) + nJ * sz + 2 * n * sz,
           (by_rows<TRANSFER_W>(h.npad, [&](auto w) {
               launch(h.prm.use_pdl, k_prolong_fine<T, decltype(w)::value>, nblk(h.npad), TPB, s, h.npad, PP.off, PP.col, PP.val, SP.U.p, SP.uf.p);
             })));
    ++launches;
  }
  // (3) multiplicative only: u3 = u2 + S^T (r - A u2)
  if (!additive) smooth(false);
  ASMG_CUDA(cudaGetLastError());
  return launches;
}

template <class T>
int enqueue_body(asmg_s& h, Slot& S, cudaStream_t s, cudaGraphConditionalHandle hnd, int use_hnd) {
  const int64_t n0 = fused_rows(h);
  int launches = enqueue_precond<T>(h, S, S.r.p, s, n0 > 0, n0 > 0);
  T* z = slotprec<T>(S).uf.p;
  const T* dinv = fine_dinv<T>(h);
  const int G = red_grid(h.npad, RED_BLOCKS), GV = red_grid(h.npad, VEC_BLOCKS);
  const int nb = GV <= DIRECT_BLOCKS ? GV : 0;  // then G == GV
  double* pq = S.partial.p + 2 * VEC_BLOCKS;     // partials of <p, q>, which k_axpy_norm reads beside its own
  const int64_t n = h.n, sz = sizeof(T);
  LAUNCH(ASMG_PROF_CG_VECTOR, n * (sz + 16) + (n0 ? h.fine_cnnz[0] * (sz + 4) + h.fine_crows[0] * (8 + 2 * sz) : 0),
         launch(h.prm.use_pdl, k_dots<T>, GV, TPB, s, h.npad, n0, fine_smoother<T>(h), dinv, z, S.r.p, S.q.p,
                S.partial.p, S.ticket.p, S.scal.p, nb));
  LAUNCH(ASMG_PROF_CG_VECTOR, n * (sz + 16),
         launch(h.prm.use_pdl, k_pupd<T>, GV, TPB, s, h.npad, (const T*)z, S.p.p, (const double*)S.partial.p, nb,
                S.scal.p));
  LAUNCH(ASMG_PROF_CG_SPMV, h.A64.nnz_real * 12 + n * 16,
         (by_rows(h.npad, [&](auto w) {
               launch(h.prm.use_pdl, k_spmv_dot<decltype(w)::value>, G, TPB, s, h.npad, view(h.A64), S.p.p, S.q.p, pq, S.ticket.p, S.scal.p, nb);
             })));
  LAUNCH(ASMG_PROF_CG_VECTOR, n * 48 + n0 * 2 * sz,
         launch(h.prm.use_pdl, k_axpy_norm<T>, GV, TPB, s, h.npad, S.p.p, S.q.p, S.x.p, S.r.p, n0, dinv, z, (const double*)pq, nb,
                S.partial.p, S.ticket.p, S.scal.p, S.hist.p, hnd, use_hnd));
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

template <class T>
void enqueue_init_prec(asmg_s& h, Slot& S, double rtol, cudaStream_t s, cudaGraphConditionalHandle hnd, int use_hnd) {
  LAUNCH(ASMG_PROF_CG_VECTOR, h.A64.nnz_real * 12 + h.n * 32,
         launch(h.prm.use_pdl, k_pcg_init<T>, red_grid(h.npad, RED_BLOCKS), TPB, s, h.npad, view(h.A64), S.b.p, S.x.p,
                S.r.p, fused_rows(h), fine_dinv<T>(h), slotprec<T>(S).uf.p, S.partial.p, S.ticket.p, S.scal.p, rtol,
                h.prm.max_iter, S.hist.p, hnd, use_hnd));
  ASMG_CUDA(cudaGetLastError());
}

void enqueue_init(asmg_s& h, Slot& S, double rtol, cudaStream_t s, cudaGraphConditionalHandle hnd, int use_hnd) {
  if (h.prm.precision == ASMG_MIXED)
    enqueue_init_prec<float>(h, S, rtol, s, hnd, use_hnd);
  else
    enqueue_init_prec<double>(h, S, rtol, s, hnd, use_hnd);
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

static void enqueue_precond_any(asmg_s& h, Slot& S, cudaStream_t s) {
  if (h.prm.precision == ASMG_MIXED)
    enqueue_precond<float>(h, S, S.r.p, s);
  else
    enqueue_precond<double>(h, S, S.r.p, s);
}

// One application as a graph (use_graph): some 50 launches, which the host
// issues more slowly than the device runs them (kuhn65 FP64 306 -> 285 us).
void precond_apply(asmg_s& h, cudaStream_t s) {
  Slot& S = *h.slots[0];
  if (!h.prm.use_graph) {
    enqueue_precond_any(h, S, s);
    return;
  }
  if (!S.pexec) {
    cudaStream_t cs;
    cudaGraph_t g;
    ASMG_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    ASMG_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    enqueue_precond_any(h, S, cs);
    ASMG_CUDA(cudaStreamEndCapture(cs, &g));
    ASMG_CUDA(cudaStreamDestroy(cs));
    ASMG_CUDA(cudaGraphInstantiate(&S.pexec, g, 0));
    ASMG_CUDA(cudaGraphDestroy(g));
  }
  ASMG_CUDA(cudaGraphLaunch(S.pexec, s));
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

int64_t iteration_bytes(asmg_s& h) {
  int64_t bytes = 0;
  struct Counting {
    explicit Counting(int64_t* n) { g_count_bytes = n; }
    ~Counting() { g_count_bytes = nullptr; }
  } counting(&bytes);
  enqueue_body_any(h, *h.slots[0], nullptr, 0, 0);
  return bytes;
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
    tiles::set_smem_limits<T, V, 1>();
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
  SP.fr.clear();
  SP.fr.resize(nlev);
  for (int li = 0; li < nlev; ++li) {
    SP.fs[li].alloc(std::max<int64_t>(P.lev[li].nsm, 1));
    SP.us[li].alloc(std::max<int64_t>(P.lev[li].nsm, 1));
    SP.fs[li].zero(s);
    SP.us[li].zero(s);
    if (P.lev[li].tiled_down) {
      SP.fr[li].alloc(std::max<int64_t>(P.lev[li].nsm, 1));
      SP.fr[li].zero(s);
    }
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

// A level of at most this many tiles always runs them: they are one wave of
// blocks, about the time of one or two of the class launches they replace
// (level of 16,129 rows on graded 2049^2: 8 us against 4 launches a direction).
constexpr int64_t TILE_ALWAYS = 2 * NSM;

// Schedule of the auxiliary levels (the autotuner, tile_rows = 0): each
// direction of a level that has tiles runs either its temporally blocked
// sweeps or its launches per colour class and sweep, with the same results.
// The choice is made on the device: one preconditioner application is
// captured as a CUDA graph and timed (median of 3 runs of 5 launches) with
// every level tiled both ways, then for each level in turn the post-sweeps
// and then the pre-sweeps are switched to class launches, each switch kept
// when it is faster by more than 0.5% (and 2 us).
template <class T>
void autotune_levels(asmg_s& h, cudaStream_t s) {
  Prec<T>& P = prec<T>(h);
  Slot& S = *h.slots[0];
  const int nlev = (int)P.lev.size();
  std::vector<int> cand;
  for (int li = P.bot.v.nlev; li <= nlev - 1 - P.deep.v.nlev; ++li)
    if (P.lev[li].tiled && std::max(P.lev[li].tdown.ntiles, P.lev[li].tup.ntiles) > TILE_ALWAYS) cand.push_back(li);
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
}

// Free the tiles of directions that run class launches.
template <class T>
void drop_untiled(asmg_s& h) {
  Prec<T>& P = prec<T>(h);
  SlotPrec<T>& SP = slotprec<T>(*h.slots[0]);
  for (size_t li = 0; li < P.lev.size(); ++li) {
    AuxLevelDev<T>& L = P.lev[li];
    if (!L.tiled) continue;
    if (!L.tiled_down) {
      L.tdown = TileSweeps<T>();
      L.trest = TileRestrict<T>();
      SP.fr[li] = DBuf<T>();
    }
    if (!L.tiled_up) {
      L.tup = TileSweeps<T>();
      SP.ust[li] = DBuf<T>();
      SP.fsl[li] = DBuf<T>();
    }
    L.tiled = L.tiled_down || L.tiled_up;
  }
}

// The handle's schedule: measured when the handle is set up, kept when its
// coefficients change (they change neither the grids nor the work of a launch).
template <class T>
void schedule_levels(asmg_s& h, cudaStream_t s) {
  Prec<T>& P = prec<T>(h);
  const size_t nlev = P.lev.size();
  if (h.sched.size() != nlev) {
    autotune_levels<T>(h, s);
    h.sched.assign(nlev, 0);
    for (size_t li = 0; li < nlev; ++li)
      h.sched[li] = (uint8_t)((P.lev[li].tiled_down ? 1 : 0) | (P.lev[li].tiled_up ? 2 : 0));
  } else {
    for (size_t li = 0; li < nlev; ++li) {
      AuxLevelDev<T>& L = P.lev[li];
      L.tiled_down = L.tiled_down && (h.sched[li] & 1);
      L.tiled_up = L.tiled_up && (h.sched[li] & 2);
    }
  }
  drop_untiled<T>(h);
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
  S.partial.alloc(std::max(4 * RED_BLOCKS, 2 * VEC_BLOCKS + RED_BLOCKS));
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
      P.lev[li].trest = TileRestrict<T>();
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
  add_slot(h, s);
  if (h.prm.tile_rows == 0 && !h.prm.inject_timeout) {
    if (h.prm.precision == ASMG_MIXED)
      schedule_levels<float>(h, s);
    else
      schedule_levels<double>(h, s);
  }
}

}  // namespace asmg
