// C ABI entry points (include/asmg.h) and the setup pipeline.
#include <algorithm>
#include <array>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstddef>
#include <cstring>
#include <exception>
#include <numeric>
#include <thread>
#include <unordered_map>

#include "handle.h"

using namespace asmg;

namespace {

thread_local std::string g_err;

double now() {
  return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

bool is_device(const void* p) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

template <class T>
std::vector<T> to_host(const T* p, int64_t n, cudaStream_t s) {
  std::vector<T> h((size_t)n);
  if (n == 0) return h;
  if (is_device(p)) {
    ASMG_CUDA(cudaMemcpyAsync(h.data(), p, sizeof(T) * n, cudaMemcpyDeviceToHost, s));
    ASMG_CUDA(cudaStreamSynchronize(s));
  } else {
    std::memcpy(h.data(), p, sizeof(T) * n);
  }
  return h;
}

void copy_in(double* dst, const double* src, int64_t n, cudaStream_t s) {
  ASMG_CUDA(cudaMemcpyAsync(dst, src, 8 * n, is_device(src) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
}

void copy_out(double* dst, const double* src, int64_t n, cudaStream_t s) {
  ASMG_CUDA(cudaMemcpyAsync(dst, src, 8 * n, is_device(dst) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
}

// A device array the kernels read or write in place: memory of the current
// device, aligned for its type.  Anything else (host, managed or another
// device's memory) goes through the handle's staging arrays.
bool in_place(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int dev = -1;
  ASMG_CUDA(cudaGetDevice(&dev));
  return a.type == cudaMemoryTypeDevice && a.device == dev && (uintptr_t)p % sizeof(double) == 0;
}

// The caller's input array where kernels can read it: itself, or a staged copy.
// Staged copies in and out cost a call on device arrays more than its kernels:
// one operator product and one load vector on graded 1025^2 took 474 us with
// them and the kernels of that time, 178 us in place with kernels that read each
// row and element once.
const double* input(const double* user, double* stage, int64_t n, cudaStream_t s) {
  if (in_place(user)) return user;
  copy_in(stage, user, n, s);
  return stage;
}

int64_t pad32(int64_t n) { return (n + 31) / 32 * 32; }

// Temporally blocked sweeps (asmg_params::tile_rows = 0): own rows per tile on
// levels of two colour classes, and on levels of more (whose longer dependency
// chains make deeper halos, which larger tiles amortise) as a share of the rows
// a block holds (1,024).  A larger share overflows and its tiles are halved, a
// smaller one carries more halo: pre-sweeps at a share of 0.5 / 0.44 / 0.375
// take graded 2049^2 BF16 209.4 / 205.2 / 205.1 ms, graded 513^2 FP64 29.6 /
// 28.8 / 28.6 ms.  TILE_MAX_HALO: the largest halo accepted, as a multiple of
// the own rows.
constexpr int TILE_ROWS_2COL = 256;
constexpr double TILE_OWN = 0.375;
constexpr double TILE_MAX_HALO = 1.5;
constexpr int64_t TILE_MIN_ROWS = 64;  // smoothing rows of a tiled level (below, the fused runs hold every level)

// f(begin, end) over contiguous ranges of [0, n) on host threads
template <class F>
void host_for(int64_t n, F f) {
  unsigned nt = std::max(1u, std::min(32u, std::thread::hardware_concurrency()));
  if (n < (1 << 15)) nt = 1;
  std::vector<std::thread> th;
  for (unsigned t = 0; t < nt; ++t) th.emplace_back([&, t] { f(n * t / nt, n * (t + 1) / nt); });
  for (auto& x : th) x.join();
}

// rows of a host CSR selected and renumbered: out row k = A row sel[k] (or
// empty when sel[k] < 0), columns mapped by cmap (dropped when < 0); rows
// counted, then filled, in parallel
HostCSR select_rows(const HostCSR& A, const std::vector<int64_t>& sel, const std::vector<int32_t>* cmap,
                    const std::vector<uint8_t>* colkeep) {
  HostCSR B;
  B.nr = (int64_t)sel.size();
  B.nc = A.nc;
  B.ptr.assign(B.nr + 1, 0);
  auto keep = [&](int64_t p) {
    // couplings that vanish by symmetry are not stored
    return !(colkeep && !(*colkeep)[A.col[p]]) && A.val[p] != 0.0;
  };
  host_for(B.nr, [&](int64_t k0, int64_t k1) {
    for (int64_t k = k0; k < k1; ++k) {
      int64_t c = 0;
      if (sel[k] >= 0)
        for (int64_t p = A.ptr[sel[k]]; p < A.ptr[sel[k] + 1]; ++p) c += keep(p);
      B.ptr[k + 1] = c;
    }
  });
  for (int64_t k = 0; k < B.nr; ++k) B.ptr[k + 1] += B.ptr[k];
  B.col.resize(B.ptr[B.nr]);
  B.val.resize(B.ptr[B.nr]);
  host_for(B.nr, [&](int64_t k0, int64_t k1) {
    for (int64_t k = k0; k < k1; ++k) {
      if (sel[k] < 0) continue;
      int64_t q = B.ptr[k];
      for (int64_t p = A.ptr[sel[k]]; p < A.ptr[sel[k] + 1]; ++p)
        if (keep(p)) {
          B.col[q] = cmap ? (*cmap)[A.col[p]] : A.col[p];
          B.val[q] = A.val[p];
          ++q;
        }
    }
  });
  return B;
}

// The form of a small level that the fused runs take (small_run.h): local
// numbering (smoothing nodes in colour order first, then the other rows of
// E_l), 16-bit local columns.
template <class T>
void build_small(const AuxLevelHost& L, const HostCSR& Arows, const std::vector<uint8_t>& inset,
                 const std::vector<int64_t>& sel, const std::vector<int64_t>& rsel, const std::vector<T>& dinv_pad,
                 const std::vector<int32_t>& pid, const std::vector<int32_t>& pptr, const std::vector<int32_t>& child,
                 AuxLevelDev<T>& D) {
  SmallLevel<T>& S = D.small;
  S.ok = false;
  std::vector<int32_t> gid;
  std::vector<T> dinv;
  std::vector<int> cs(1, 0);
  for (int c = 0; c < D.ncolours; ++c) {
    for (int64_t k = D.cstart[c]; k < D.cstart[c + 1]; ++k)
      if (sel[k] >= 0) {
        gid.push_back((int32_t)sel[k]);
        dinv.push_back(dinv_pad[k]);
      }
    cs.push_back((int)gid.size());
  }
  const int mS = (int)gid.size();
  for (int64_t r : rsel)
    if (r >= 0 && !inset[r]) gid.push_back((int32_t)r);
  const int mE = (int)gid.size();
  if (mE > small_lmax_long<T>() || D.ncolours > SMALL_MAXC) return;
  if (mE > small_lmax<T>()) {
    int64_t longest = 0;
    for (int k = 0; k < mS; ++k) {
      int64_t n = 0;
      for (int64_t p = Arows.ptr[gid[k]]; p < Arows.ptr[gid[k] + 1]; ++p) n += Arows.val[p] != 0.0;
      longest = std::max(longest, n);
    }
    if (longest <= TILE_MAXW) return;
  }
  std::unordered_map<int32_t, int32_t> loc;
  loc.reserve(mE * 2);
  for (int k = 0; k < mE; ++k) loc[gid[k]] = k;
  auto L_ = [&](int32_t g) -> int32_t {
    auto it = loc.find(g);
    return it == loc.end() ? -1 : it->second;
  };
  std::vector<int32_t> sm_ptr(1, 0), rs_ptr(1, 0);
  std::vector<uint16_t> sm_col, rs_col;
  std::vector<T> sm_val, rs_val;
  for (int k = 0; k < mE; ++k) {
    const int32_t r = gid[k];
    for (int64_t p = Arows.ptr[r]; p < Arows.ptr[r + 1]; ++p) {
      if (Arows.val[p] == 0.0) continue;
      const int32_t c = Arows.col[p];
      if (k < mS) {
        const int32_t lc = L_(c);
        if (lc < 0) return;  // a neighbour outside E_l: keep the level on the general path
        sm_col.push_back((uint16_t)lc);
        sm_val.push_back((T)Arows.val[p]);
      }
      if (inset[c]) {
        const int32_t lc = L_(c);
        if (lc < 0) return;
        rs_col.push_back((uint16_t)lc);
        rs_val.push_back((T)Arows.val[p]);
      }
    }
    if (k < mS) sm_ptr.push_back((int32_t)sm_col.size());
    rs_ptr.push_back((int32_t)rs_col.size());
  }
  std::vector<uint16_t> nn_id, rp_id, rp_child;
  std::vector<int32_t> nn_p0, nn_p1, rp_ptr(1, 0);
  for (size_t t = 0; t < L.new_id.size(); ++t) {
    const int32_t a = L_(L.new_id[t]);
    const int32_t b0 = L.new_p0[t] >= 0 ? L_(L.new_p0[t]) : -1;
    const int32_t b1 = L.new_p1[t] >= 0 ? L_(L.new_p1[t]) : -1;
    if (a < 0 || (L.new_p0[t] >= 0 && b0 < 0) || (L.new_p1[t] >= 0 && b1 < 0)) return;
    nn_id.push_back((uint16_t)a);
    nn_p0.push_back(b0);
    nn_p1.push_back(b1);
  }
  for (size_t t = 0; t < pid.size(); ++t) {
    const int32_t a = L_(pid[t]);
    if (a < 0) return;
    rp_id.push_back((uint16_t)a);
    for (int32_t p = pptr[t]; p < pptr[t + 1]; ++p) {
      const int32_t b = L_(child[p]);
      if (b < 0) return;
      rp_child.push_back((uint16_t)b);
    }
    rp_ptr.push_back((int32_t)rp_child.size());
  }
  S.mS = mS;
  S.mE = mE;
  S.ncol = D.ncolours;
  S.cs = std::move(cs);
  S.gid = std::move(gid);
  S.sm_ptr = std::move(sm_ptr);
  S.sm_col = std::move(sm_col);
  S.sm_val = std::move(sm_val);
  S.dinv = std::move(dinv);
  S.rs_ptr = std::move(rs_ptr);
  S.rs_col = std::move(rs_col);
  S.rs_val = std::move(rs_val);
  S.nn_id = std::move(nn_id);
  S.nn_p0 = std::move(nn_p0);
  S.nn_p1 = std::move(nn_p1);
  S.rp_id = std::move(rp_id);
  S.rp_ptr = std::move(rp_ptr);
  S.rp_child = std::move(rp_child);
  S.ok = true;
}

// Tiles of one sweep direction of a level (TileSweeps).  The own rows of a
// tile are at most tile_rows consecutive smoothing rows in aux-ID order (a
// tile whose rows do not fit the kernel's registers is cut in half).  Its rows
// are the closure of the pairs (row, sweep) that the own rows' final values
// depend on: a row's value after sweep s reads its own value after sweep
// s - 1 and each coupled row j of N~_l either after sweep s (j's class is
// swept before the row's in this direction) or after sweep s - 1 (j's class
// comes later).  Before the first sweep the values are the start values:
// zero on the way down (such reads need no row), read from us on the way up
// (the row is kept, with its start value).  Every entry of a kept row that
// points to a row of N~_l outside the tile is left out: no pair of the
// closure reads it.  On the way down the own rows' residual reads the last
// value of every coupled row.  Entries of the post-sweeps' rows whose column lies
// outside N~_l become the tile's outside values.  SMd: SM-order rows with
// their N~_l columns as SM rows; SM: the same rows with all columns as aux
// IDs; pos: aux ID -> SM row.  Returns false (and builds nothing) when a row
// is longer than TILE_MAXW, when the closure of a single row does not fit, or
// when the halo exceeds max_halo times the own rows.
template <class T>
bool build_tiles(bool up, int nu, int tile_rows, const std::vector<int64_t>& sel, const std::vector<int64_t>& cstart,
                 const std::vector<T>& dinv, const HostCSR& SMd, const HostCSR& SM, const std::vector<int32_t>& pos,
                 double max_halo, unsigned max_threads, bool bf16, TileSweeps<T>& TS, cudaStream_t s) {
  const int64_t nsm = (int64_t)sel.size();
  const int ncol = (int)cstart.size() - 1;
  const int max_slots = TILE_SLOTS_MAX;
  std::vector<int32_t> colr(nsm);
  for (int c = 0; c < ncol; ++c)
    for (int64_t k = cstart[c]; k < cstart[c + 1]; ++k) colr[k] = c;
  std::vector<int32_t> own;
  for (int64_t k = 0; k < nsm; ++k)
    if (sel[k] >= 0) own.push_back((int32_t)k);
  std::sort(own.begin(), own.end(), [&](int32_t a, int32_t b) { return sel[a] < sel[b]; });
  const int64_t nbase = ((int64_t)own.size() + tile_rows - 1) / tile_rows;
  // a tile before its place in the level's arrays is known
  struct Out {
    int slots = 0;
    std::vector<int32_t> lrow;         // [slots * TILE_THREADS] SM row, -2 - SM row (halo) or -1
    std::vector<TileSlice> hdr;        // [slots * TILE_WARPS]
    std::vector<int32_t> rptr;         // entries of each local row
    std::vector<int32_t> rcol;         // local row, or -1 - e for the e-th outside value
    std::vector<double> rval;
    std::vector<int32_t> ext;
    uint32_t cmask = 0;
    int64_t words = 0, vals = 0;       // rows of 32 in its words and values
    TileLayout lay{};
    int64_t interior = 0, halo = 0, nnz = 0;
    int width = 0;
  };
  std::vector<std::vector<Out>> out(nbase);
  std::atomic<bool> fits(true);
  const unsigned nt = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)max_threads, nbase));
  std::vector<std::thread> th;
  for (unsigned wk = 0; wk < nt; ++wk)
    th.emplace_back([&, wk] {
      // stamps: mark[sw * nsm + k] == tag: pair (k, sw) needed; inx[k] == tag: k kept
      std::vector<int32_t> mark((size_t)nu * nsm, -1), inx(nsm, -1), loc(nsm, 0), ownm(nsm, -1);
      std::vector<std::pair<int32_t, int32_t>> stack;
      std::vector<int32_t> X;
      std::unordered_map<int32_t, int32_t> extpos;
      std::vector<std::pair<int64_t, int32_t>> rlen;
      std::vector<std::pair<int64_t, int64_t>> todo;
      int32_t tag = -1;
      for (int64_t t = nbase * wk / nt; t < nbase * (wk + 1) / nt && fits.load(std::memory_order_relaxed); ++t) {
        todo.assign(1, {t * tile_rows, std::min<int64_t>((int64_t)own.size(), (t + 1) * tile_rows)});
        while (!todo.empty()) {
          const auto [o0, o1] = todo.back();
          todo.pop_back();
          ++tag;
          stack.clear();
          X.clear();
          auto keep = [&](int32_t k) {
            if (inx[k] != tag) {
              inx[k] = tag;
              X.push_back(k);
            }
          };
          auto need = [&](int32_t k, int sw) {
            int32_t& m = mark[(size_t)sw * nsm + k];
            if (m != tag) {
              m = tag;
              stack.push_back({k, sw});
            }
          };
          for (int64_t q = o0; q < o1; ++q) {
            ownm[own[q]] = tag;
            need(own[q], nu - 1);
            // the residual of the own rows reads every coupled row's last value
            if (!up)
              for (int64_t p = SMd.ptr[own[q]]; p < SMd.ptr[own[q] + 1]; ++p) need(SMd.col[p], nu - 1);
          }
          while (!stack.empty()) {
            const auto [k, sw] = stack.back();
            stack.pop_back();
            keep(k);
            if (sw >= 1) need(k, sw - 1);
            for (int64_t p = SMd.ptr[k]; p < SMd.ptr[k + 1]; ++p) {
              const int32_t j = SMd.col[p];
              if (j == k) continue;
              const int cj = colr[j], ck = colr[k];
              const bool before = up ? cj > ck : cj < ck;
              if (before || cj == ck) need(j, sw);
              if (!before) {
                if (sw >= 1) need(j, sw - 1);
                else if (up) keep(j);
              }
            }
          }
          // rows by colour class; within a class, where order does not
          // matter, longest first so that the slices carry little padding
          auto row_len = [&](int32_t k) {
            int64_t n = 0;
            if (!up) {
              for (int64_t p = SMd.ptr[k]; p < SMd.ptr[k + 1]; ++p) n += inx[SMd.col[p]] == tag;
            } else {
              for (int64_t p = SM.ptr[k]; p < SM.ptr[k + 1]; ++p) {
                const int32_t j = pos[SM.col[p]];
                n += j < 0 || inx[j] == tag;
              }
            }
            return n;
          };
          std::sort(X.begin(), X.end());
          rlen.resize(X.size());
          for (size_t q = 0; q < X.size(); ++q) rlen[q] = {-row_len(X[q]), X[q]};
          Out O;
          std::vector<std::array<int64_t, 3>> slices;  // first and last + 1 in rlen, colour
          for (size_t x = 0, c = 0; c < (size_t)ncol; ++c) {
            const size_t x0 = x;
            while (x < X.size() && X[x] < cstart[c + 1]) ++x;
            std::sort(rlen.begin() + x0, rlen.begin() + x);
            for (size_t q = x0; q < x; q += 32)
              slices.push_back({(int64_t)q, (int64_t)std::min(x, q + 32), (int64_t)c});
          }
          // the slices of a class spread over the warps, each warp's slots filled evenly
          bool ok = (int)slices.size() <= max_slots * TILE_WARPS;
          if (ok) {
            O.slots = std::max(1, ((int)slices.size() + TILE_WARPS - 1) / TILE_WARPS);
            O.lrow.assign((size_t)O.slots * TILE_THREADS, -1);
            O.hdr.assign((size_t)O.slots * TILE_WARPS, TileSlice{0, 0, 0, -1});
            int total[TILE_WARPS] = {}, inclass[TILE_WARPS] = {};
            int64_t cls = -1;
            for (const auto& sl : slices) {
              if (sl[2] != cls) std::fill(inclass, inclass + TILE_WARPS, 0);
              cls = sl[2];
              int w = -1;
              for (int v = 0; v < TILE_WARPS; ++v)
                if (total[v] < O.slots &&
                    (w < 0 || inclass[v] < inclass[w] || (inclass[v] == inclass[w] && total[v] < total[w])))
                  w = v;
              const int slot = total[w]++;
              ++inclass[w];
              TileSlice& H = O.hdr[(size_t)slot * TILE_WARPS + w];
              H.colour = (int16_t)cls;
              H.w = (int16_t)std::min<int64_t>(-rlen[sl[0]].first, INT16_MAX);
              O.width = std::max<int>(O.width, H.w);
              for (int64_t q = sl[0]; q < sl[1]; ++q) {
                const int32_t k = rlen[q].second, r = slot * TILE_THREADS + w * 32 + (int32_t)(q - sl[0]);
                loc[k] = r;
                const bool mine = ownm[k] == tag;
                O.lrow[r] = mine ? k : -2 - k;
                ++(mine ? O.interior : O.halo);
              }
              O.cmask |= 1u << std::min<int64_t>(cls, 31);
            }
            extpos.clear();
            O.rptr.assign(1, 0);
            for (int32_t g : O.lrow) {
              if (g != -1) {
                const int32_t k = g >= 0 ? g : -2 - g;
                const HostCSR& M = up ? SM : SMd;
                for (int64_t p = M.ptr[k]; p < M.ptr[k + 1]; ++p) {
                  const int32_t a = M.col[p], j = up ? pos[a] : a;
                  if (j >= 0) {
                    if (inx[j] != tag) continue;
                    O.rcol.push_back(loc[j]);
                  } else {
                    const auto it = extpos.emplace(a, (int32_t)O.ext.size());
                    if (it.second) O.ext.push_back(a);
                    O.rcol.push_back(-1 - it.first->second);
                  }
                  O.rval.push_back(M.val[p]);
                }
              }
              O.rptr.push_back((int32_t)O.rcol.size());
            }
            // a row of 32 words per entry (BF16) or per two entries, a row of
            // 32 values per entry (FP32, FP64)
            for (TileSlice& H : O.hdr) {
              H.words = (uint16_t)O.words;
              H.vals = (uint16_t)O.vals;
              O.words += bf16 ? H.w : (H.w + 1) / 2;
              O.vals += bf16 ? 0 : H.w;
              O.nnz += 32 * (int64_t)H.w;
            }
          }
          if (ok && O.width > TILE_MAXW) {
            fits = false;
            break;
          }
          if (ok) {
            const int64_t values = max_slots * TILE_THREADS + (int64_t)O.ext.size();
            O.lay = tile_layout(O.slots, (int)O.words, (int)O.vals, (int)O.ext.size(), sizeof(T));
            ok = values <= TILE_VALUES_MAX && values * (int64_t)sizeof(T) + O.lay.end + 1024 <= TILE_SMEM_MAX;
          }
          if (!ok) {
            if (o1 - o0 <= 1) {
              fits = false;
              break;
            }
            const int64_t mid = (o0 + o1) / 2;
            todo.push_back({mid, o1});
            todo.push_back({o0, mid});
            continue;
          }
          out[t].push_back(std::move(O));
        }
      }
    });
  for (auto& x : th) x.join();
  if (!fits.load()) return false;
  std::vector<const Out*> tiles;
  for (auto& v : out)
    for (auto& O : v) tiles.push_back(&O);
  const int64_t ntiles = (int64_t)tiles.size();
  std::vector<TileHead> head(ntiles);
  int64_t bytes = 0;
  for (int64_t t = 0; t < ntiles; ++t) {
    const Out& O = *tiles[t];
    TS.slots = std::max(TS.slots, O.slots);
    TS.width = std::max(TS.width, O.width);
    TS.maxext = std::max(TS.maxext, (int)O.ext.size());
    TS.maxblob = std::max(TS.maxblob, O.lay.end);
    TS.interior += O.interior;
    TS.halo += O.halo;
    TS.nnz += O.nnz;
    TS.nnz_real += (int64_t)O.rcol.size();
    head[t] = TileHead{bytes, (int32_t)O.lay.end, (int32_t)O.words, (int32_t)O.vals, (int32_t)O.ext.size(), O.slots,
                       O.cmask};
    bytes += O.lay.end;
  }
  const int64_t per = (int64_t)TS.slots * TILE_THREADS;  // local rows of a tile
  if ((double)TS.halo > max_halo * (double)TS.interior || ntiles * per > INT32_MAX ||
      (int64_t)TS.smem() > TILE_SMEM_MAX) {
    TS = TileSweeps<T>();
    return false;
  }
  TS.ntiles = ntiles;
  TS.nloc = ntiles * per;
  std::vector<unsigned char> blob((size_t)bytes, 0);
  std::vector<int32_t> lsm((size_t)(up ? TS.nloc : 0), -1);
  auto pack = [&](int64_t t0, int64_t t1) {
    for (int64_t t = t0; t < t1; ++t) {
      const Out& O = *tiles[t];
      unsigned char* B = blob.data() + head[t].off;
      TileSlice* hdr = reinterpret_cast<TileSlice*>(B);
      uint32_t* words = reinterpret_cast<uint32_t*>(B + O.lay.words);
      T* val = reinterpret_cast<T*>(B + O.lay.val);
      T* dd = reinterpret_cast<T*>(B + O.lay.dinv);
      int32_t* sm = reinterpret_cast<int32_t*>(B + O.lay.lsm);
      int32_t* ax = reinterpret_cast<int32_t*>(B + O.lay.laux);
      std::copy(O.hdr.begin(), O.hdr.end(), hdr);
      std::copy(O.ext.begin(), O.ext.end(), reinterpret_cast<int32_t*>(B + O.lay.ext));
      if (up) std::copy(O.lrow.begin(), O.lrow.end(), lsm.begin() + t * per);
      for (int r = 0; r < O.slots * TILE_THREADS; ++r) {
        const TileSlice& H = hdr[r / 32];
        const int lane = r % 32;
        const int32_t g = O.lrow[r];
        sm[r] = g;
        if (g == -1) continue;
        const int32_t k = g >= 0 ? g : -2 - g;
        ax[r] = (int32_t)sel[k];
        dd[r] = dinv[k];
        for (int32_t p = O.rptr[r], e = 0; p < O.rptr[r + 1]; ++p, ++e) {
          const int32_t c = O.rcol[p];
          const uint32_t off = (uint32_t)((c >= 0 ? c : per + (-1 - c)) * (int64_t)sizeof(T));
          if (bf16) {
            words[(H.words + e) * 32 + lane] = ((uint32_t)bf16_bits((float)O.rval[p]) << 16) | off;
          } else {
            words[(H.words + e / 2) * 32 + lane] |= off << (16 * (e & 1));
            val[(H.vals + e) * 32 + lane] = (T)O.rval[p];
          }
        }
      }
    }
  };
  th.clear();
  for (unsigned wk = 0; wk < nt; ++wk) th.emplace_back([&, wk] { pack(ntiles * wk / nt, ntiles * (wk + 1) / nt); });
  for (auto& x : th) x.join();
  if (up) {
    // where each SM row sits in tile order (own and halo copies)
    std::vector<int64_t> pptr(nsm + 1, 0);
    for (int32_t g : lsm)
      if (g != -1) ++pptr[(g >= 0 ? g : -2 - g) + 1];
    for (int64_t k = 0; k < nsm; ++k) pptr[k + 1] += pptr[k];
    std::vector<int32_t> place(pptr[nsm]);
    std::vector<int64_t> fill(pptr.begin(), pptr.end() - 1);
    for (int64_t q = 0; q < TS.nloc; ++q)
      if (lsm[q] != -1) place[fill[lsm[q] >= 0 ? lsm[q] : -2 - lsm[q]]++] = (int32_t)q;
    TS.pos_ptr.upload(pptr, s);
    TS.pos.upload(place, s);
  }
  TS.head.upload(head, s);
  TS.blob.upload(blob, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
  return true;
}

// The near-boundary solve of a level (mixed boundaries, Algorithm 3) for the
// device: the rows of A_l on J_{l,j} in the factor's order (all columns) and
// the block cyclic reduction flattened into NbDev.
template <class T>
void build_nb_dev(const AuxLevelHost& L, const HostCSR& Arows, const std::vector<int32_t>& pos, AuxLevelDev<T>& D,
                  cudaStream_t s) {
  const nb::Factor& Fz = L.nb_fac;
  NbDev& N = D.nb;
  N.m = (int64_t)L.nb_id.size();
  if (N.m == 0) return;
  if (!Fz.ok || Fz.m != N.m) ASMG_FAIL(ASMG_ERR_BAD_MESH, "auxiliary level %d: no near-boundary factor", L.level);
  std::vector<int32_t> aux(N.m), sm(N.m);
  std::vector<int64_t> sel(N.m);
  for (int64_t q = 0; q < N.m; ++q) {
    const int32_t a = L.nb_id[Fz.order[q]];
    aux[q] = a;
    sm[q] = pos[a];
    sel[q] = a;
    if (sm[q] < 0) ASMG_FAIL(ASMG_ERR_BAD_MESH, "auxiliary level %d: near-boundary node outside the level", L.level);
  }
  HostCSR rows = select_rows(Arows, sel, nullptr, nullptr);
  sell_build<T>(D.NB, rows, 0, s);
  // block sizes of round 0, then the even blocks of each round form the next
  std::vector<int> sz0;
  for (size_t b = 0; b + 1 < Fz.bstart.size(); ++b) sz0.push_back((int)(Fz.bstart[b + 1] - Fz.bstart[b]));
  N.R = (int)Fz.rounds.size();
  std::vector<int32_t> nblk, boff;
  std::vector<int64_t> btab, voff(1, 0);
  std::vector<double> mats;
  auto put = [&](const nb::Blk& B) -> int64_t {
    if (B.empty()) return -1;
    const int64_t o = (int64_t)mats.size();
    mats.insert(mats.end(), B.a.begin(), B.a.end());
    return o;
  };
  std::vector<int> sz = sz0;
  for (int r = 0; r < N.R; ++r) {
    const nb::Round& Rd = Fz.rounds[r];
    if (Rd.n != (int)sz.size()) ASMG_FAIL(ASMG_ERR_CUDA, "near-boundary factor: inconsistent rounds");
    nblk.push_back(Rd.n);
    boff.push_back((int32_t)(btab.size() / 5));
    int64_t off = 0;
    for (int k = 0; k < Rd.n; ++k) {
      btab.push_back(sz[k]);
      btab.push_back(off);
      btab.push_back((k & 1) ? put(Rd.F[k]) : -1);
      btab.push_back(k > 0 ? put(Rd.Lo[k]) : -1);
      btab.push_back(k + 1 < Rd.n ? put(Rd.Up[k]) : -1);
      off += sz[k];
    }
    voff.push_back(voff.back() + off);
    std::vector<int> nx;
    for (int k = 0; k < Rd.n; k += 2) nx.push_back(sz[k]);
    sz.swap(nx);
  }
  if (sz.size() != 1 || Fz.last.r != sz[0]) ASMG_FAIL(ASMG_ERR_CUDA, "near-boundary factor: inconsistent last block");
  N.last_size = sz[0];
  N.last_off = put(Fz.last);
  voff.push_back(voff.back() + sz[0]);  // the last block's vector, then the pool size
  N.nblk_h = nblk;
  N.nblk.upload(nblk, s);
  N.boff.upload(boff, s);
  N.btab.upload(btab, s);
  N.voff.upload(voff, s);
  N.mats.upload(mats, s);
  N.aux.upload(aux, s);
  N.sm.upload(sm, s);
}

template <class T>
void build_level_dev(const AuxLevelHost& L, const HostCSR& Arows, const std::vector<int32_t>& colour,
                     const std::vector<uint8_t>& inset, const asmg_params& prm, AuxLevelDev<T>& D, cudaStream_t s) {
  D.level = L.level;
  // the mixed form may read the level matrices in BF16 (asmg_params::level_bf16)
  const bool bf16 = std::is_same<T, float>::value && prm.level_bf16 == 1;
  // smoothing rows ordered by (colour, id), colour blocks padded to 32
  int ncol = 0;
  for (int32_t id : L.smooth) ncol = std::max(ncol, colour[id] + 1);
  D.ncolours = ncol;
  std::vector<std::vector<int32_t>> byc(ncol);
  for (int32_t id : L.smooth) byc[colour[id]].push_back(id);
  std::vector<int64_t> sel;
  D.cstart.assign(1, 0);
  for (int c = 0; c < ncol; ++c) {
    for (int32_t id : byc[c]) sel.push_back(id);
    while (sel.size() % 32) sel.push_back(-1);
    D.cstart.push_back((int64_t)sel.size());
  }
  D.nsm = (int64_t)sel.size();
  D.nsm_real = (int64_t)L.smooth.size();
  std::vector<int32_t> rows(sel.size());
  std::vector<T> dinv(sel.size(), (T)0);
  for (size_t k = 0; k < sel.size(); ++k) {
    rows[k] = (int32_t)sel[k];
    if (sel[k] >= 0) {
      double dg = 0;
      for (int64_t p = Arows.ptr[sel[k]]; p < Arows.ptr[sel[k] + 1]; ++p)
        if (Arows.col[p] == sel[k]) dg = Arows.val[p];
      if (!(dg > 0)) ASMG_FAIL(ASMG_ERR_CUDA, "auxiliary level %d: non-positive diagonal", L.level);
      dinv[k] = (T)(1.0 / dg);
    }
  }
  HostCSR SM = select_rows(Arows, sel, nullptr, nullptr);
  // SM row index of every node of N~_l: the down sweeps and the residual work
  // on the level's own correction us (SM order), where every other node is 0
  std::vector<int32_t> pos(Arows.nr, -1);
  for (size_t k = 0; k < sel.size(); ++k)
    if (sel[k] >= 0) pos[sel[k]] = (int32_t)k;
  HostCSR SMd = select_rows(Arows, sel, &pos, &inset);
  D.cnnz.assign(ncol, 0);
  D.cnnz_d.assign(ncol, 0);
  D.crows.assign(ncol, 0);
  for (int c = 0; c < ncol; ++c)
    for (int64_t k = D.cstart[c]; k < D.cstart[c + 1]; ++k)
      if (sel[k] >= 0) {
        D.crows[c] += 1;
        D.cnnz[c] += SM.ptr[k + 1] - SM.ptr[k];
        D.cnnz_d[c] += SMd.ptr[k + 1] - SMd.ptr[k];
      }
  sell_build<T>(D.SM, SM, 0, s);
  sell_build<T>(D.SMd, SMd, 0, s);
  if constexpr (std::is_same<T, float>::value)
    if (bf16) {
      sell_bf16(D.SM, s);
      sell_bf16(D.SMd, s);
    }
  D.sm_rows.upload(rows, s);
  D.sm_dinv.upload(dinv, s);
  // temporal blocking of the level's sweeps (TileSweeps), with the default own
  // rows per tile and a halo of at most TILE_MAX_HALO times the own rows, or the
  // requested rows and any halo; every new node must be a smoothing row
  // (k_up_init prolongs through the smoothing rows)
  D.tiled = false;
  if (prm.tile_rows >= 0 && prm.nu_post >= 1) {
    bool ok = true;
    for (int32_t id : L.new_id)
      if (pos[id] < 0) ok = false;
    const double max_halo = prm.tile_rows > 0 ? 1e30 : TILE_MAX_HALO;
    const int cap = TILE_SLOTS_MAX * TILE_THREADS;
    const int trows = prm.tile_rows > 0 ? prm.tile_rows : ncol <= 2 ? TILE_ROWS_2COL : (int)(cap * TILE_OWN);
    if (ok && D.nsm_real >= TILE_MIN_ROWS) {
      // the two directions are built at the same time, each on half the host threads
      TileSweeps<T> td, tu;
      const unsigned half = std::max(1u, std::thread::hardware_concurrency() / 2);
      bool okd = false, oku = false;
      std::exception_ptr eu, ed;
      std::thread up_th([&] {
        try {
          oku = build_tiles<T>(true, prm.nu_post, trows, sel, D.cstart, dinv, SMd, SM, pos, max_halo, half, bf16, tu, s);
        } catch (...) {
          eu = std::current_exception();
        }
      });
      try {
        okd = build_tiles<T>(false, prm.nu_pre, trows, sel, D.cstart, dinv, SMd, SM, pos, max_halo, half, bf16, td, s);
      } catch (...) {
        ed = std::current_exception();
      }
      up_th.join();
      if (ed) std::rethrow_exception(ed);
      if (eu) std::rethrow_exception(eu);
      if (okd && oku) {
        std::vector<int32_t> p0(sel.size(), -3), p1(sel.size(), -3);
        for (size_t t = 0; t < L.new_id.size(); ++t) {
          p0[pos[L.new_id[t]]] = L.new_p0[t];
          p1[pos[L.new_id[t]]] = L.new_p1[t];
        }
        D.sm_par0.upload(p0, s);
        D.sm_par1.upload(p1, s);
        D.tdown = std::move(td);
        D.tup = std::move(tu);
        D.tiled = D.tiled_down = D.tiled_up = true;
        D.tile_rows = trows;
      }
    }
  }
  // residual rows: every row with an entry in a smoothing column
  std::vector<uint8_t> touched(Arows.nr, 0);
  host_for(Arows.nr, [&](int64_t i0, int64_t i1) {
    for (int64_t i = i0; i < i1; ++i)
      for (int64_t p = Arows.ptr[i]; p < Arows.ptr[i + 1]; ++p)
        if (inset[Arows.col[p]]) {
          touched[i] = 1;
          break;
        }
  });
  std::vector<int64_t> rsel;
  for (int64_t i = 0; i < Arows.nr; ++i)
    if (touched[i]) rsel.push_back(i);
  D.nrs_real = (int64_t)rsel.size();
  while (rsel.size() % 32) rsel.push_back(-1);
  D.nrs = (int64_t)rsel.size();
  HostCSR RS = select_rows(Arows, rsel, &pos, &inset);
  sell_build<T>(D.RS, RS, 0, s);
  if constexpr (std::is_same<T, float>::value)
    if (bf16) sell_bf16(D.RS, s);
  std::vector<int32_t> rsrows(rsel.begin(), rsel.end());
  D.rs_rows.upload(rsrows, s);
  // prolongation and restriction of the new nodes
  D.nnew = (int64_t)L.new_id.size();
  D.nn_id.upload(L.new_id, s);
  D.nn_p0.upload(L.new_p0, s);
  D.nn_p1.upload(L.new_p1, s);
  std::vector<std::pair<int32_t, int32_t>> pc;  // (parent, child)
  for (size_t k = 0; k < L.new_id.size(); ++k) {
    if (L.new_p0[k] >= 0) pc.push_back({L.new_p0[k], L.new_id[k]});
    if (L.new_p1[k] >= 0) pc.push_back({L.new_p1[k], L.new_id[k]});
  }
  std::sort(pc.begin(), pc.end());
  std::vector<int32_t> pid, pptr(1, 0), child;
  for (size_t k = 0; k < pc.size(); ++k) {
    if (k == 0 || pc[k].first != pc[k - 1].first) {
      if (k) pptr.push_back((int32_t)child.size());
      pid.push_back(pc[k].first);
    }
    child.push_back(pc[k].second);
  }
  if (!pid.empty()) pptr.push_back((int32_t)child.size());
  D.npar = (int64_t)pid.size();
  D.nchild = (int64_t)child.size();
  D.rp_id.upload(pid, s);
  D.rp_ptr.upload(pptr, s);
  D.rp_child.upload(child, s);
  if (D.tiled) {
    // residual and restriction after tiled pre-sweeps
    std::vector<uint8_t> isnew(Arows.nr, 0);
    for (int32_t id : L.new_id) isnew[id] = 1;
    std::vector<int32_t> par(Arows.nr, -1);
    for (size_t t = 0; t < pid.size(); ++t) par[pid[t]] = (int32_t)t;
    std::vector<int64_t> other;
    std::vector<int32_t> id, src, cptr(1, 0), cch;
    auto add = [&](int32_t v) {
      id.push_back(v);
      if (v >= 0 && par[v] >= 0)
        for (int32_t p = pptr[par[v]]; p < pptr[par[v] + 1]; ++p) cch.push_back(pos[child[p]]);
      cptr.push_back((int32_t)cch.size());
    };
    for (int64_t v = 0; v < Arows.nr; ++v) {
      if (isnew[v]) continue;
      if (pos[v] >= 0) {
        add((int32_t)v);
        src.push_back(pos[v]);
      } else if (touched[v] || par[v] >= 0) {
        other.push_back(v);
      }
    }
    while (id.size() % 32) add(-1);
    src.resize(id.size(), 0);
    D.trest.n1 = (int64_t)id.size();
    for (int64_t v : other) add((int32_t)v);
    while (id.size() % 32) add(-1);
    while (other.size() % 32) other.push_back(-1);
    D.trest.n2 = (int64_t)id.size() - D.trest.n1;
    D.trest.nchild = (int64_t)cch.size();
    sell_build<T>(D.trest.X, select_rows(Arows, other, &pos, &inset), 0, s);
    if constexpr (std::is_same<T, float>::value)
      if (bf16) sell_bf16(D.trest.X, s);
    D.trest.id.upload(id, s);
    D.trest.src.upload(src, s);
    D.trest.ptr.upload(cptr, s);
    D.trest.child.upload(cch, s);
    ASMG_CUDA(cudaStreamSynchronize(s));
  }
  build_nb_dev<T>(L, Arows, pos, D, s);
  // a level with a near-boundary solve keeps its own launches (the solve sits
  // between the coarse correction and the post-smoothing)
  if (D.nb.m == 0) build_small<T>(L, Arows, inset, sel, rsel, dinv, pid, pptr, child, D);
  else D.small.ok = false;
}

// triangles given by lattice keys -> device coordinates, ids, coefficients
struct TriDev {
  DBuf<double> xy, coef;
  DBuf<int32_t> id;
};

void upload_tris(const asmg_s& h, const std::vector<uint64_t>& keys, const std::vector<int32_t>& ids,
                 const std::vector<double>& coef, TriDev& T, cudaStream_t s) {
  const int dim = h.mesh.dim;
  std::vector<double> xy(keys.size() * dim);
  for (size_t k = 0; k < keys.size(); ++k) {
    if (dim == 2)
      lattice_point(h.tree, keys[k], &xy[2 * k]);
    else
      lattice_point3(h.tree, h.aux.LB, keys[k], &xy[3 * k]);
  }
  T.xy.upload(xy, s);
  T.id.upload(ids, s);
  T.coef.upload(coef, s);
}

template <class T>
void build_prec(asmg_s& h, Prec<T>& P, const HostCSR& Aperm, const std::vector<double>& dinv_perm, bool keep_transfer,
                cudaStream_t s) {
  if (std::is_same<T, float>::value) {
    sell_build<T>(P.Af, Aperm, 0, s);
    std::vector<T> d(dinv_perm.begin(), dinv_perm.end());
    P.dinv_f.upload(d, s);
  }
  if (h.prm.smoother == 0 && h.prm.fine_sweeps == 1) {
    // the halves of A the forward sweep from 0 and the residual after it read
    const int ncol = (int)h.fine_cstart.size() - 1;
    h.fine_lnnz.assign(ncol, 0);
    auto half = [&](bool lower) {
      HostCSR B;
      B.nr = Aperm.nr;
      B.nc = Aperm.nc;
      B.ptr.assign(B.nr + 1, 0);
      auto rows = [&](auto body) {
        for (int c = 0; c < ncol; ++c) {
          const int64_t r0 = h.fine_cstart[c], r1 = h.fine_cstart[c + 1];
          host_for(r1 - r0, [&](int64_t a, int64_t b) {
            for (int64_t i = r0 + a; i < r0 + b; ++i)
              body(i, [&](int64_t p) { return lower ? Aperm.col[p] < r0 : Aperm.col[p] >= r1; });
          });
        }
      };
      rows([&](int64_t i, auto in) {
        int64_t k = 0;
        for (int64_t p = Aperm.ptr[i]; p < Aperm.ptr[i + 1]; ++p) k += in(p);
        B.ptr[i + 1] = k;
      });
      for (int64_t i = 0; i < B.nr; ++i) B.ptr[i + 1] += B.ptr[i];
      B.col.resize(B.ptr[B.nr]);
      B.val.resize(B.ptr[B.nr]);
      rows([&](int64_t i, auto in) {
        int64_t q = B.ptr[i];
        for (int64_t p = Aperm.ptr[i]; p < Aperm.ptr[i + 1]; ++p)
          if (in(p)) {
            B.col[q] = Aperm.col[p];
            B.val[q++] = Aperm.val[p];
          }
      });
      if (lower)
        for (int c = 0; c < ncol; ++c) h.fine_lnnz[c] = B.ptr[h.fine_cstart[c + 1]] - B.ptr[h.fine_cstart[c]];
      return B;
    };
    sell_build<T>(P.Lo, half(true), 0, s);
    sell_build<T>(P.Up, half(false), 0, s);
  }
  if (keep_transfer) return;
  h.transfer_rows.clear();
  // transfer P (rows: permuted fine rows) and P^T (rows: aux nodes), built
  // by counting sort into flat CSR arrays; each row sorted by column
  const Triplets& Tp = h.aux.P;
  const int64_t m = (int64_t)Tp.r.size();
  auto to_csr = [&](int64_t nr, int64_t nc, bool transpose) {
    HostCSR A;
    A.nr = nr;
    A.nc = nc;
    A.ptr.assign(nr + 1, 0);
    for (int64_t k = 0; k < m; ++k) ++A.ptr[1 + (transpose ? Tp.c[k] : h.row_of_free[Tp.r[k]])];
    for (int64_t i = 0; i < nr; ++i) A.ptr[i + 1] += A.ptr[i];
    A.col.resize(m);
    A.val.resize(m);
    std::vector<int64_t> fill(A.ptr.begin(), A.ptr.end() - 1);
    for (int64_t k = 0; k < m; ++k) {
      const int32_t pr = h.row_of_free[Tp.r[k]];
      const int64_t row = transpose ? Tp.c[k] : pr;
      const int64_t q = fill[row]++;
      A.col[q] = transpose ? pr : Tp.c[k];
      A.val[q] = Tp.v[k];
    }
    std::vector<std::pair<int32_t, double>> tmp;
    for (int64_t i = 0; i < nr; ++i) {
      const int64_t b = A.ptr[i], e = A.ptr[i + 1];
      bool sorted = true;
      for (int64_t q = b + 1; q < e && sorted; ++q) sorted = A.col[q - 1] < A.col[q];
      if (sorted) continue;
      tmp.clear();
      for (int64_t q = b; q < e; ++q) tmp.push_back({A.col[q], A.val[q]});
      std::sort(tmp.begin(), tmp.end());
      for (int64_t q = b; q < e; ++q) {
        A.col[q] = tmp[q - b].first;
        A.val[q] = tmp[q - b].second;
      }
    }
    return A;
  };
  HostCSR Pc = to_csr(h.npad, h.nJpad, false), Ptc = to_csr(h.nJpad, h.npad, true);
  sell_build<T>(P.P, Pc, 0, s);
  sell_build<T>(P.PT, Ptc, 0, s);
  h.transfer_rows = h.row_of_free;
}

// Colouring option 2 on an auxiliary level: the lattice parity of each node
// of the smoothing set, (X + Y [+ Z]) / h_l mod 2 with h_l the lattice
// spacing of level l (2^(bits - l) on the lattice of the node keys), used when
// no two coupled nodes of the set share it (couplings as for the Jones-
// Plassmann colouring: |a_vw| > 1e-12 sqrt(a_vv a_ww), w != v).  Uniform
// levels are bipartite this way (couplings across hypotenuses vanish), so
// they take two colour classes.  Returns false, leaving `colour` as it is,
// when some coupled pair shares a parity.
bool parity_colour(const asmg_s& h, int l, const HostCSR& A, const std::vector<int32_t>& smooth,
                   const std::vector<uint8_t>& inset, std::vector<int32_t>& colour) {
  const int dim = h.mesh.dim;
  const int bits = dim == 2 ? h.tree.D : h.aux.LB;
  const uint64_t step = 1ULL << (bits - l);
  std::vector<int8_t> par(A.nr, -1);
  for (int32_t v : smooth) {
    const uint64_t k = h.aux.aux_key[v];
    uint64_t q[3] = {0, 0, 0};
    for (int j = 0; j < 64 / dim; ++j)
      for (int c = 0; c < dim; ++c)
        if ((k >> (dim * j + c)) & 1ULL) q[c] |= 1ULL << j;
    par[v] = (int8_t)(((q[0] + q[1] + q[2]) / step) & 1);
  }
  std::vector<double> diag(A.nr, 0.0);
  host_for(A.nr, [&](int64_t i0, int64_t i1) {
    for (int64_t i = i0; i < i1; ++i)
      for (int64_t p = A.ptr[i]; p < A.ptr[i + 1]; ++p)
        if (A.col[p] == i) diag[i] = A.val[p];
  });
  std::atomic<bool> ok(true);
  host_for((int64_t)smooth.size(), [&](int64_t k0, int64_t k1) {
    for (int64_t k = k0; k < k1 && ok.load(std::memory_order_relaxed); ++k) {
      const int32_t v = smooth[k];
      for (int64_t p = A.ptr[v]; p < A.ptr[v + 1]; ++p) {
        const int32_t w = A.col[p];
        if (w == v || !inset[w] || par[w] != par[v]) continue;
        if (std::fabs(A.val[p]) > 1e-12 * std::sqrt(diag[v] * diag[w])) {
          ok.store(false, std::memory_order_relaxed);
          break;
        }
      }
    }
  });
  if (!ok.load()) return false;
  for (int32_t v : smooth) colour[v] = par[v];
  return true;
}

void build_all(asmg_s& h, cudaStream_t s) {
  double t0 = now();
  MeshHost& m = h.mesh;
  const int64_t nv = m.nv, ne = m.ne;
  // ---- fine problem: free dofs, assembly, colouring, permutation
  h.free_of_vertex.assign(nv, -1);
  h.vertex_of_free.clear();
  for (int64_t v = 0; v < nv; ++v)
    if (m.bflag[v] != 1) {  // free and Neumann vertices are unknowns
      h.free_of_vertex[v] = (int32_t)h.vertex_of_free.size();
      h.vertex_of_free.push_back((int32_t)v);
    }
  h.n = (int64_t)h.vertex_of_free.size();
  if (h.n == 0) ASMG_FAIL(ASMG_ERR_BAD_MESH, "no free vertices");
  h.d_free_of_vertex.upload(h.free_of_vertex, s);
  h.A_host = assemble_mesh(m.dim, ne, h.dX.p, h.dE.p, h.d_free_of_vertex.p, h.dCoeff.p, h.n, s);
  {
    std::vector<uint8_t> all(h.n, 1);
    std::vector<uint64_t> pk(h.vertex_of_free.begin(), h.vertex_of_free.end());
    h.fine_colour = jp_colour_gpu(h.A_host, all, pk, s);
  }
  int ncol = 0;
  for (auto c : h.fine_colour) ncol = std::max(ncol, c + 1);
  std::vector<int64_t> sel;
  h.fine_cstart.assign(1, 0);
  {
    std::vector<std::vector<int32_t>> byc(ncol);
    for (int64_t i = 0; i < h.n; ++i) byc[h.fine_colour[i]].push_back((int32_t)i);
    for (int c = 0; c < ncol; ++c) {
      for (auto i : byc[c]) sel.push_back(i);
      while (sel.size() % 32) sel.push_back(-1);
      h.fine_cstart.push_back((int64_t)sel.size());
    }
  }
  h.npad = (int64_t)sel.size();
  h.row_of_free.assign(h.n, -1);
  std::vector<int32_t> vrow(h.npad, -1), rowv(nv, -1);
  for (int64_t k = 0; k < h.npad; ++k)
    if (sel[k] >= 0) {
      h.row_of_free[sel[k]] = (int32_t)k;
      vrow[k] = h.vertex_of_free[sel[k]];
      rowv[vrow[k]] = (int32_t)k;
    }
  h.d_vertex_of_row.upload(vrow, s);
  h.d_row_of_vertex.upload(rowv, s);
  HostCSR Aperm = select_rows(h.A_host, sel, &h.row_of_free, nullptr);
  std::vector<double> dinv(h.npad, 0.0);
  for (int64_t k = 0; k < h.npad; ++k)
    for (int64_t p = Aperm.ptr[k]; p < Aperm.ptr[k + 1]; ++p)
      if (Aperm.col[p] == k) dinv[k] = 1.0 / Aperm.val[p];
  sell_build<double>(h.A64, Aperm, 0, s);
  h.dinv64.upload(dinv, s);
  h.fine_cnnz.assign(ncol, 0);
  h.fine_crows.assign(ncol, 0);
  for (int c = 0; c < ncol; ++c)
    for (int64_t k = h.fine_cstart[c]; k < h.fine_cstart[c + 1]; ++k)
      if (sel[k] >= 0) {
        h.fine_crows[c] += 1;
        h.fine_cnnz[c] += Aperm.ptr[k + 1] - Aperm.ptr[k];
      }
  h.stats.t_fine = now() - t0;

  // ---- auxiliary hierarchy (host), transfer
  double t1 = now();
  // the transfer depends on the geometry only: a coefficient update keeps it,
  // and its device form too while the fine rows keep their order
  Triplets kept = std::move(h.aux.P);
  const bool same_rows = !kept.r.empty() && h.row_of_free == h.transfer_rows;
  h.aux = AuxHost();
  if (m.dim == 2)
    build_aux_host(m, h.tree, h.prm, h.aux);
  else
    build_aux_host3(m, h.tree, h.prm, h.aux);
  h.stats.t_aux = now() - t1;
  t1 = now();
  if (kept.r.empty())
    build_transfer(m, h.dX.p, h.dE.p, h.vertex_of_free, h.aux.sz, h.aux.P, s);
  else
    h.aux.P = std::move(kept);
  h.aux.sz = SZTable();
  h.stats.t_sz = now() - t1;
  double t2 = now();
  h.nJ = (int64_t)h.aux.aux_key.size();
  h.nJpad = pad32(h.nJ);

  // ---- auxiliary levels: device assembly, colouring, SELL
  h.level_smooth_keys.clear();
  h.level_smooth_colour.clear();
  h.level_rows.clear();
  h.p64.lev.clear();
  h.p32.lev.clear();
  h.stats.t_lv_assemble = h.stats.t_lv_colour = h.stats.t_lv_pack = h.stats.t_lv_export = 0;
  for (const AuxLevelHost& L : h.aux.levels) {
    double ta = now();
    std::vector<uint8_t> inset(h.nJ, 0);
    for (int32_t id : L.smooth) inset[id] = 1;
    TriDev T;
    upload_tris(h, L.tri_key, L.tri_id, L.tri_coef, T, s);
    DBuf<uint8_t> dkeep;
    dkeep.upload(inset, s);
    HostCSR Arows = assemble_simplices(m.dim, (int64_t)L.tri_coef.size(), T.xy.p, T.id.p, T.coef.p, dkeep.p, h.nJ, s);
    double tb = now();
    h.stats.t_lv_assemble += tb - ta;
    std::vector<int32_t> colour = jp_colour_gpu(Arows, inset, h.aux.aux_key, s);
    if (h.prm.colouring == 2) parity_colour(h, L.level, Arows, L.smooth, inset, colour);
    double tc = now();
    h.stats.t_lv_colour += tc - tb;
    // export copies
    std::vector<uint64_t> sk;
    std::vector<int32_t> sc;
    for (int32_t id : L.smooth) {
      sk.push_back(h.aux.aux_key[id]);
      sc.push_back(colour[id]);
    }
    h.level_smooth_keys.push_back(sk);
    h.level_smooth_colour.push_back(sc);
    Triplets tr;
    const int64_t nz = Arows.ptr[Arows.nr];
    tr.r.resize(nz);
    tr.c.assign(Arows.col.begin(), Arows.col.begin() + nz);
    tr.v.assign(Arows.val.begin(), Arows.val.begin() + nz);
    host_for(Arows.nr, [&](int64_t i0, int64_t i1) {
      for (int64_t i = i0; i < i1; ++i)
        for (int64_t p = Arows.ptr[i]; p < Arows.ptr[i + 1]; ++p) tr.r[p] = (int32_t)i;
    });
    h.level_rows.push_back(std::move(tr));
    double td = now();
    h.stats.t_lv_export += td - tc;
    if (h.prm.precision == ASMG_MIXED) {
      h.p32.lev.emplace_back();
      build_level_dev<float>(L, Arows, colour, inset, h.prm, h.p32.lev.back(), s);
    } else {
      h.p64.lev.emplace_back();
      build_level_dev<double>(L, Arows, colour, inset, h.prm, h.p64.lev.back(), s);
    }
    h.stats.t_lv_pack += now() - td;
  }
  double te = now();
  // ---- coarsest level: explicit inverse of A_c (B_0 = A_0^{-1})
  h.nc = (int64_t)h.aux.coarse_id.size();
  if (h.nc > 0) {
    std::vector<int32_t> loc(h.aux.coarse_tri_id.size());
    for (size_t k = 0; k < loc.size(); ++k) {
      int32_t id = h.aux.coarse_tri_id[k];
      loc[k] = id < 0 ? -1
                      : (int32_t)(std::lower_bound(h.aux.coarse_id.begin(), h.aux.coarse_id.end(), id) -
                                  h.aux.coarse_id.begin());
    }
    TriDev T;
    upload_tris(h, h.aux.coarse_tri_key, loc, h.aux.coarse_tri_coef, T, s);
    HostCSR Ac = assemble_simplices(m.dim, (int64_t)h.aux.coarse_tri_coef.size(), T.xy.p, T.id.p, T.coef.p, nullptr,
                                    h.nc, s);
    const int64_t n = h.nc;
    std::vector<double> M(n * n, 0.0);
    for (int64_t i = 0; i < n; ++i)
      for (int64_t p = Ac.ptr[i]; p < Ac.ptr[i + 1]; ++p) M[i * n + Ac.col[p]] = Ac.val[p];
    // Cholesky M = L L^T (lower, in place)
    for (int64_t j = 0; j < n; ++j) {
      double d = M[j * n + j];
      for (int64_t k = 0; k < j; ++k) d -= M[j * n + k] * M[j * n + k];
      if (!(d > 0)) ASMG_FAIL(ASMG_ERR_CUDA, "coarsest auxiliary matrix is not positive definite");
      d = std::sqrt(d);
      M[j * n + j] = d;
      for (int64_t i = j + 1; i < n; ++i) {
        double t = M[i * n + j];
        for (int64_t k = 0; k < j; ++k) t -= M[i * n + k] * M[j * n + k];
        M[i * n + j] = t / d;
      }
    }
    // inverse column by column: solve L L^T x = e_c
    // (columns are independent, on host threads: the whole coarse step 7.8 -> 2.4 ms at 225 nodes)
    std::vector<double> inv(n * n);
    const unsigned nt = (unsigned)std::max<int64_t>(1, std::min<int64_t>(std::thread::hardware_concurrency(), n / 16));
    std::vector<std::thread> th;
    for (unsigned w = 0; w < nt; ++w)
      th.emplace_back([&, w] {
        std::vector<double> y(n), x(n);
        for (int64_t c = n * w / nt; c < n * (w + 1) / nt; ++c) {
          for (int64_t i = 0; i < n; ++i) {
            double t = (i == c) ? 1.0 : 0.0;
            for (int64_t k = 0; k < i; ++k) t -= M[i * n + k] * y[k];
            y[i] = t / M[i * n + i];
          }
          for (int64_t i = n - 1; i >= 0; --i) {
            double t = y[i];
            for (int64_t k = i + 1; k < n; ++k) t -= M[k * n + i] * x[k];
            x[i] = t / M[i * n + i];
          }
          for (int64_t i = 0; i < n; ++i) inv[i * n + c] = x[i];
        }
      });
    for (auto& t : th) t.join();
    h.d_cinv.upload(inv, s);
    h.d_cid.upload(h.aux.coarse_id, s);
  }
  double tf = now();
  h.stats.t_coarse = tf - te;
  // ---- transfer and fine smoother copy
  if (h.prm.precision == ASMG_MIXED)
    build_prec<float>(h, h.p32, Aperm, dinv, same_rows, s);
  else
    build_prec<double>(h, h.p64, Aperm, dinv, same_rows, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
  double tg = now();
  h.stats.t_transfer = tg - tf;
  setup_solve(h, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
  h.stats.t_slots = now() - tg;
  h.stats.t_levels = now() - t2;
  h.bytes_iter = iteration_bytes(h);
  h.ready = true;
}

// f() with the device memory it needs: when that runs out, again without the
// handle's element stiffness, which the gradients can do without.
template <class F>
void with_room(asmg_s& h, F f) {
  try {
    f();
  } catch (const Error& e) {
    if (e.code != ASMG_ERR_OOM || !h.d_elem_stiff.p) throw;
    h.d_elem_stiff.release();
    f();
  }
}

// Adds a work state to a handle's; one that ran out of device memory half-way goes again.
template <class V, class F>
void grow(V& states, F add) {
  const size_t n = states.size();
  try {
    add();
  } catch (...) {
    states.resize(n);
    throw;
  }
}

int finish(int rc) { return rc; }

}  // namespace

namespace asmg {
void set_error(const char* fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_err = buf;
}
}  // namespace asmg

#define API_BEGIN \
  g_err.clear();  \
  try {
#define API_END                                   \
  }                                               \
  catch (const asmg::Error& e) {                  \
    g_err = e.msg;                                \
    return e.code;                                \
  }                                               \
  catch (const std::exception& e) {               \
    g_err = std::string("internal error: ") + e.what(); \
    return ASMG_ERR_CUDA;                         \
  }

extern "C" {

const char* amg_last_error(void) { return g_err.c_str(); }

int asmg_default_params(asmg_params* p) {
  if (!p) return ASMG_ERR_INVALID_ARG;
  p->n_min = 3;
  p->nu_pre = 2;
  p->nu_post = 2;
  p->coarse_max_dofs = 512;
  p->precision = ASMG_FP64;
  p->max_iter = 500;
  p->smoothing = 0;
  p->use_graph = 1;
  p->use_pdl = 1;
  p->smoother = 0;
  p->additive = 0;
  p->fine_sweeps = 1;
  p->iteration = 0;
  p->tile_rows = 0;
  p->inject_timeout = 0;
  p->nb_layers = 2;
  p->colouring = 2;
  p->level_bf16 = 0;
  return ASMG_OK;
}

int amg_setup(int dim, int64_t nv, const double* vertices, int64_t ne, const int32_t* elements, const uint8_t* boundary,
              const double* coeff, const asmg_params* params, void* stream, asmg_handle* out) {
  API_BEGIN
  if (!out) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!vertices || !elements || !boundary) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null input array");
  if (nv <= 0 || ne <= 0) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "nv and ne must be positive");
  if (dim != 2 && dim != 3) ASMG_FAIL(ASMG_ERR_UNSUPPORTED, "dim %d not supported (2 or 3)", dim);
  if (ne > (1LL << 31) / ((dim + 1) * (dim + 1)) || nv > (1LL << 31) - 1)
    ASMG_FAIL(ASMG_ERR_INVALID_ARG, "mesh too large");
  asmg_params prm;
  asmg_default_params(&prm);
  if (params) prm = *params;
  if (prm.n_min < 1 || prm.nu_pre < 1 || prm.nu_post < 0 || prm.coarse_max_dofs < 1 || prm.max_iter < 1 ||
      (prm.precision != ASMG_FP64 && prm.precision != ASMG_MIXED) || (prm.smoothing != 0 && prm.smoothing != 1) ||
      prm.coarse_max_dofs > 8192 || (prm.use_pdl != 0 && prm.use_pdl != 1) || (prm.use_graph != 0 && prm.use_graph != 1) ||
      (prm.smoother != 0 && prm.smoother != 1) || (prm.additive != 0 && prm.additive != 1) || prm.fine_sweeps < 1 ||
      prm.fine_sweeps > 8 || (prm.iteration != 0 && prm.iteration != 1) ||
      (prm.tile_rows != -1 && prm.tile_rows != 0 && (prm.tile_rows < 32 || prm.tile_rows > 65536)) ||
      (prm.inject_timeout != 0 && prm.inject_timeout != 1) || prm.nb_layers < -1 || prm.nb_layers > 16 ||
      (prm.colouring != 0 && prm.colouring != 2) || (prm.level_bf16 != 0 && prm.level_bf16 != 1) ||
      (prm.level_bf16 == 1 && prm.precision != ASMG_MIXED))
    ASMG_FAIL(ASMG_ERR_INVALID_ARG, "invalid parameter");
  cudaStream_t s = (cudaStream_t)stream;
  double t0 = now();
  std::unique_ptr<asmg_s> h(new asmg_s());
  h->prm = prm;
  MeshHost& m = h->mesh;
  m.dim = dim;
  m.nv = nv;
  m.ne = ne;
  m.X = to_host(vertices, nv * dim, s);
  m.E = to_host(elements, ne * (dim + 1), s);
  m.bflag = to_host(boundary, nv, s);
  if (coeff) m.coeff = to_host(coeff, ne, s);
  for (int64_t v = 0; v < nv; ++v) {
    if (m.bflag[v] > 2) ASMG_FAIL(ASMG_ERR_BAD_MESH, "boundary flag %d at vertex %lld", (int)m.bflag[v], (long long)v);
    if (m.bflag[v] == 2) m.mixed = true;
  }
  m.nb_layers = prm.nb_layers;
  if (m.mixed) {
    // the mixed grids are not nested and every level is smoothed as a whole;
    // the near-boundary solve runs between the coarse correction and the
    // post-smoothing, so those levels take the per-class launches
    h->prm.tile_rows = -1;
  }
  for (int64_t e = 0; e < (int64_t)m.coeff.size(); ++e)
    if (!(m.coeff[e] > 0) || !std::isfinite(m.coeff[e]))
      ASMG_FAIL(ASMG_ERR_BAD_MESH, "coefficient of element %lld is not positive and finite", (long long)e);
  h->dX.upload(m.X, s);
  h->dE.upload(m.E, s);
  if (!m.coeff.empty()) h->dCoeff.upload(m.coeff, s);
  // cluster tree (also checks index range and orientation)
  double tt = now();
  build_tree_gpu(dim, nv, h->dX.p, ne, h->dE.p, prm.n_min, s, h->tree);
  h->stats.t_tree = now() - tt;
  // does the domain fill the root box (the element measures add up to
  // L^dim)?  A domain that does not uses the Dirichlet auxiliary grids
  // (Sec. 3.4)
  {
    double meas = 0;
    for (int64_t e = 0; e < ne; ++e) {
      const int32_t* v = &m.E[(dim + 1) * e];
      if (dim == 2) {
        meas += 0.5 * ((m.X[2 * v[1]] - m.X[2 * v[0]]) * (m.X[2 * v[2] + 1] - m.X[2 * v[0] + 1]) -
                       (m.X[2 * v[2]] - m.X[2 * v[0]]) * (m.X[2 * v[1] + 1] - m.X[2 * v[0] + 1]));
      } else {
        double e3[3][3];
        for (int k = 0; k < 3; ++k)
          for (int r = 0; r < 3; ++r) e3[k][r] = m.X[3 * (int64_t)v[k + 1] + r] - m.X[3 * (int64_t)v[0] + r];
        meas += (e3[0][0] * (e3[1][1] * e3[2][2] - e3[1][2] * e3[2][1]) -
                 e3[0][1] * (e3[1][0] * e3[2][2] - e3[1][2] * e3[2][0]) +
                 e3[0][2] * (e3[1][0] * e3[2][1] - e3[1][1] * e3[2][0])) /
                6.0;
      }
    }
    const double box = std::pow(h->tree.L, dim);
    m.boxdomain = std::fabs(meas - box) <= 1e-12 * box;
  }
  build_all(*h, s);
  // load the allocation-free entry point's module (and so its fixed scratch
  // array) on this device now, so that its calls never create memory
  noalloc_scratch_for_current_device();
  h->pinned.alloc(READBACK_SCALARS + 8 * (size_t)READBACK_HIST);
  h->stats.t_total = now() - t0;
  *out = h.release();
  return ASMG_OK;
  API_END
}

void amg_destroy(asmg_handle h) { delete h; }

int amg_cluster_tree(int dim, int64_t nv, const double* vertices, int64_t ne, const int32_t* elements, uint64_t* keys,
                     int32_t* perm, void* stream) {
  API_BEGIN
  if (!vertices || !elements || !keys || !perm) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  if (dim != 2 && dim != 3) ASMG_FAIL(ASMG_ERR_UNSUPPORTED, "dim %d not supported", dim);
  if (nv <= 0 || ne <= 0) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "nv and ne must be positive");
  cudaStream_t s = (cudaStream_t)stream;
  DBuf<double> dX;
  DBuf<int32_t> dE;
  dX.upload(to_host(vertices, nv * dim, s), s);
  dE.upload(to_host(elements, ne * (dim + 1), s), s);
  TreeResult t;
  build_tree_gpu(dim, nv, dX.p, ne, dE.p, 3, s, t);
  ASMG_CUDA(cudaMemcpyAsync(keys, t.keys.p, 8 * ne, cudaMemcpyDefault, s));
  ASMG_CUDA(cudaMemcpyAsync(perm, t.perm.p, 4 * ne, cudaMemcpyDefault, s));
  ASMG_CUDA(cudaStreamSynchronize(s));
  return ASMG_OK;
  API_END
}

}  // extern "C"

struct asmg_batch_s {
  std::vector<asmg_handle> H;
  int nrhs = 0;
  double rtol = 0;
  bool multi = false;  // right-hand sides in groups of KRHS columns (SpMM form), one graph branch per group
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  // per branch its vertex arrays of this call: `per` right-hand sides, then
  // `per` solutions (NULL: an unused column, right-hand side 0); and the
  // branches' scalars read back
  int per = 1;
  std::vector<int64_t> generation;  // of each handle when the graph was captured
  DBuf<double*> tab;
  PinnedBuf tab_host, back;
  ~asmg_batch_s() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
  }
  Slot& slot(int p, int j) { return *H[p]->slots.at(1 + j); }
  MultiSlot& mslot(int p, int g) { return *H[p]->mslots.at(1 + g); }
};

namespace {
// Whether the branches of a batch, which run in any order, may read and write
// the caller's arrays where they lie: no solution meets another solution, nor a
// right-hand side of another branch (of its own branch it may: a branch gathers
// all its inputs before its solve).  One pass over the arrays by address, with
// the furthest end so far of the solutions and of the right-hand sides; for the
// latter, and for solutions met by a right-hand side, of two different branches.
struct ArrayRange {
  uintptr_t begin, end;
  int branch;
  bool out;
};
bool branches_apart(std::vector<ArrayRange>& R) {
  std::sort(R.begin(), R.end(), [](const ArrayRange& a, const ArrayRange& b) { return a.begin < b.begin; });
  struct Furthest {
    uintptr_t end[2] = {0, 0};  // of `branch`, and of any other branch
    int branch = -1;
    void add(const ArrayRange& r) {
      if (r.branch == branch) {
        end[0] = std::max(end[0], r.end);
      } else if (r.end > end[0]) {
        end[1] = end[0];
        end[0] = r.end;
        branch = r.branch;
      } else {
        end[1] = std::max(end[1], r.end);
      }
    }
    uintptr_t other(int b) const { return b == branch ? end[1] : end[0]; }
  } in, out;
  for (const ArrayRange& r : R) {
    if (r.begin < (r.out ? std::max(out.end[0], in.other(r.branch)) : out.other(r.branch))) return false;
    (r.out ? out : in).add(r);
  }
  return true;
}
}  // namespace

extern "C" {

int amg_batch_create(int nprob, const asmg_handle* handles, int nrhs, double rtol, void* stream, asmg_batch* out) {
  API_BEGIN
  if (!handles || !out || nprob <= 0 || nrhs <= 0) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "invalid batch arguments");
  if (!(rtol >= 0) || !std::isfinite(rtol)) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "rtol must be finite and >= 0");
  *out = nullptr;
  cudaStream_t s = (cudaStream_t)stream;
  std::unique_ptr<asmg_batch_s> B(new asmg_batch_s());
  B->H.assign(handles, handles + nprob);
  B->nrhs = nrhs;
  B->rtol = rtol;
  B->multi = nrhs > 1;
  for (auto h : B->H) {
    if (!h) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null handle in batch");
    h->check_ready();
    if (!multi_supported(*h)) B->multi = false;
  }
  const int ngroups = (nrhs + KRHS - 1) / KRHS;
  for (auto h : B->H) {
    if (B->multi) {
      while ((int)h->mslots.size() < 1 + ngroups) with_room(*h, [&] { grow(h->mslots, [&] { add_multi_slot(*h, s); }); });
    } else {
      while ((int)h->slots.size() < 1 + nrhs) with_room(*h, [&] { grow(h->slots, [&] { add_slot(*h, s); }); });
    }
  }
  B->per = B->multi ? KRHS : 1;
  for (auto h : B->H) B->generation.push_back(h->generation);
  const int nbranch = nprob * (B->multi ? ngroups : nrhs);
  B->tab.alloc(2 * (int64_t)B->per * nbranch);
  B->tab_host.alloc(sizeof(double*) * (size_t)B->tab.n);
  B->back.alloc(READBACK_SCALARS * (size_t)nbranch);
  ASMG_CUDA(cudaGraphCreate(&B->graph, 0));
  cudaStream_t cs;
  ASMG_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  if (B->multi) {
    // one branch per (problem, group of KRHS right-hand sides): gather, the
    // multiple solve's graph, scatter
    for (int p = 0; p < nprob; ++p)
      for (int g = 0; g < ngroups; ++g) {
        asmg_s& h = *B->H[p];
        MultiSlot& S = B->mslot(p, g);
        ASMG_CUDA(cudaStreamBeginCaptureToGraph(cs, B->graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
        double* const* tab = B->tab.p + 2 * KRHS * (int64_t)(p * ngroups + g);
        gather_multi_tab(h, tab, S.b.p, cs);
        gather_multi_tab(h, tab + KRHS, S.x.p, cs);
        cudaStreamCaptureStatus st;
        const cudaGraphNode_t* leaf = nullptr;
        size_t nleaf = 0;
        ASMG_CUDA(cudaStreamGetCaptureInfo(cs, &st, nullptr, nullptr, &leaf, nullptr, &nleaf));
        std::vector<cudaGraphNode_t> leaves(leaf, leaf + nleaf);
        cudaGraph_t gg;
        ASMG_CUDA(cudaStreamEndCapture(cs, &gg));
        cudaGraphNode_t wnode = capture_solve_multi(h, S, rtol, B->graph, leaves.data(), leaves.size());
        ASMG_CUDA(cudaStreamBeginCaptureToGraph(cs, B->graph, &wnode, nullptr, 1, cudaStreamCaptureModeThreadLocal));
        scatter_multi_tab(h, S.x.p, tab + KRHS, cs);
        ASMG_CUDA(cudaStreamEndCapture(cs, &gg));
      }
  }
  for (int p = 0; p < (B->multi ? 0 : nprob); ++p)
    for (int j = 0; j < nrhs; ++j) {
      asmg_s& h = *B->H[p];
      Slot& S = B->slot(p, j);
      // gather the rhs / initial guess (a root of its own branch)
      ASMG_CUDA(cudaStreamBeginCaptureToGraph(cs, B->graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
      double* const* tab = B->tab.p + 2 * (int64_t)(p * nrhs + j);
      gather_rows_tab(h, tab, S.b.p, cs);
      gather_rows_tab(h, tab + 1, S.x.p, cs);
      cudaStreamCaptureStatus st;
      const cudaGraphNode_t* leaf = nullptr;
      size_t nleaf = 0;
      ASMG_CUDA(cudaStreamGetCaptureInfo(cs, &st, nullptr, nullptr, &leaf, nullptr, &nleaf));
      std::vector<cudaGraphNode_t> leaves(leaf, leaf + nleaf);
      cudaGraph_t gg;
      ASMG_CUDA(cudaStreamEndCapture(cs, &gg));
      cudaGraphNode_t wnode = capture_solve(h, S, rtol, B->graph, leaves.data(), leaves.size());
      ASMG_CUDA(cudaStreamBeginCaptureToGraph(cs, B->graph, &wnode, nullptr, 1, cudaStreamCaptureModeThreadLocal));
      scatter_rows_tab(h, S.x.p, tab + 1, cs);
      ASMG_CUDA(cudaStreamEndCapture(cs, &gg));
    }
  ASMG_CUDA(cudaStreamDestroy(cs));
  ASMG_CUDA(cudaGraphInstantiate(&B->exec, B->graph, 0));
  *out = B.release();
  return ASMG_OK;
  API_END
}

int amg_batch_solve(asmg_batch B, const double* const* bs, double* const* us, int* iterations, int* status,
                    void* stream) {
  API_BEGIN
  if (!B || !bs || !us || !iterations) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  const int np = (int)B->H.size(), nr = B->nrhs;
  for (int k = 0; k < np * nr; ++k)
    if (!bs[k] || !us[k]) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null array in batch");
  for (int p = 0; p < np; ++p)
    if (B->H[p]->generation != B->generation[p])
      ASMG_FAIL(ASMG_ERR_INVALID_ARG, "problem %d's coefficients changed after the batch was created", p);
  // the branches read and write the caller's device arrays through the table;
  // other arrays are staged, and every array of a call whose arrays overlap
  // across branches: all inputs are then copied before the branches start, and
  // the solutions after they end, in order
  const int ngroups = B->multi ? (nr + KRHS - 1) / KRHS : nr;
  std::vector<ArrayRange> ranges;
  ranges.reserve(2 * (size_t)np * nr);
  for (int k = 0; k < np * nr; ++k)
    for (bool out : {false, true}) {
      const uintptr_t a = out ? (uintptr_t)us[k] : (uintptr_t)bs[k];
      ranges.push_back({a, a + 8 * (uintptr_t)B->H[k / nr]->mesh.nv, k / nr * ngroups + k % nr / B->per, out});
    }
  const bool apart = branches_apart(ranges);
  auto array = [&](const double* user, double* stage, int64_t n) {
    if (apart) return const_cast<double*>(input(user, stage, n, s));
    copy_in(stage, user, n, s);
    return stage;
  };
  double** tab = static_cast<double**>(B->tab_host.p);
  struct Out {
    double *user, *stage;
    int64_t n;
  };
  std::vector<Out> staged;
  for (int p = 0; p < np; ++p)
    for (int g = 0; g < ngroups; ++g) {
      const int64_t nv = B->H[p]->mesh.nv;
      double* vb = B->multi ? B->mslot(p, g).vb.p : B->slot(p, g).vb.p;
      double* vu = B->multi ? B->mslot(p, g).vu.p : B->slot(p, g).vu.p;
      double** t = tab + 2 * (int64_t)B->per * (p * ngroups + g);
      for (int c = 0; c < B->per; ++c) {
        const int j = g * B->per + c;
        t[c] = t[B->per + c] = nullptr;
        if (j >= nr) continue;
        const double* b = bs[p * nr + j];
        double* u = us[p * nr + j];
        t[c] = array(b, vb + c * nv, nv);
        t[B->per + c] = array(u, vu + c * nv, nv);
        if (t[B->per + c] != u) staged.push_back({u, vu + c * nv, nv});
      }
    }
  ASMG_CUDA(cudaMemcpyAsync(B->tab.p, tab, sizeof(double*) * (size_t)B->tab.n, cudaMemcpyHostToDevice, s));
  ASMG_CUDA(cudaGraphLaunch(B->exec, s));
  char* back = static_cast<char*>(B->back.p);
  for (int p = 0; p < np; ++p)
    for (int g = 0; g < ngroups; ++g) {
      char* dst = back + READBACK_SCALARS * (size_t)(p * ngroups + g);
      if (B->multi)
        ASMG_CUDA(cudaMemcpyAsync(dst, B->mslot(p, g).scal.p, sizeof(MultiScalars), cudaMemcpyDeviceToHost, s));
      else
        ASMG_CUDA(cudaMemcpyAsync(dst, B->slot(p, g).scal.p, sizeof(PcgScalars), cudaMemcpyDeviceToHost, s));
    }
  for (const Out& o : staged) copy_out(o.user, o.stage, o.n, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
  int worst = ASMG_OK;
  for (int p = 0; p < np; ++p)
    for (int j = 0; j < nr; ++j) {
      const char* src = back + READBACK_SCALARS * (size_t)(p * ngroups + j / B->per);
      int k, code;
      if (B->multi) {
        const MultiScalars& m = *reinterpret_cast<const MultiScalars*>(src);
        k = m.k[j % KRHS];
        code = m.status[j % KRHS];
      } else {
        const PcgScalars& m = *reinterpret_cast<const PcgScalars*>(src);
        k = m.k;
        code = m.status;
      }
      iterations[p * nr + j] = k;
      const int st = code == 0                    ? ASMG_OK
                     : code == ASMG_ERR_BREAKDOWN ? ASMG_ERR_BREAKDOWN
                     : code == ASMG_ERR_TIMEOUT   ? ASMG_ERR_TIMEOUT
                                                  : ASMG_NOT_CONVERGED;
      if (status) status[p * nr + j] = st;
      if (st < 0 || (worst == ASMG_OK && st != ASMG_OK)) worst = st;
    }
  if (worst == ASMG_ERR_BREAKDOWN) g_err = "PCG breakdown in a batched solve";
  if (worst == ASMG_ERR_TIMEOUT) g_err = "a bounded device wait expired in a batched solve";
  return worst;
  API_END
}

void amg_batch_destroy(asmg_batch B) { delete B; }

int amg_residual_norm_noalloc(asmg_handle h, const double* b, const double* u, double* out, void* stream) {
  API_BEGIN
  if (!h || !b || !u || !out) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  h->check_ready();
  residual_norm_noalloc(*h, b, u, out, (cudaStream_t)stream);
  return ASMG_OK;
  API_END
}

int amg_profile(asmg_handle h, const double* b, double rtol, double* out, int* iterations, void* stream) {
  API_BEGIN
  if (!h || !b || !out || !iterations) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  Slot& S0 = h->slot0();
  const int64_t nv = h->mesh.nv;
  gather_rows(*h, input(b, S0.vb.p, nv, s), S0.b.p, s);
  S0.x.zero(s);
  *iterations = profile_solve(*h, rtol, s, out);
  return ASMG_OK;
  API_END
}

int amg_profile_levels(asmg_handle h, const double* b, double rtol, double* out, double* out_levels, int nlev,
                       int* iterations, void* stream) {
  API_BEGIN
  if (!h || !b || !out || !out_levels || !iterations || nlev < 0)
    ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  Slot& S0 = h->slot0();
  const int64_t nv = h->mesh.nv;
  gather_rows(*h, input(b, S0.vb.p, nv, s), S0.b.p, s);
  S0.x.zero(s);
  *iterations = profile_solve(*h, rtol, s, out, out_levels, nlev);
  return ASMG_OK;
  API_END
}

int amg_solve(asmg_handle h, const double* b, double* u, double rtol, int* iterations, double* res_history,
              void* stream) {
  API_BEGIN
  if (!h || !b || !u || !iterations) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  if (!(rtol >= 0) || !std::isfinite(rtol)) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "rtol must be finite and >= 0");
  cudaStream_t s = (cudaStream_t)stream;
  Slot& S0 = h->slot0();
  const int64_t nv = h->mesh.nv;
  const bool direct = in_place(u);
  gather_rows(*h, input(b, S0.vb.p, nv, s), S0.b.p, s);
  gather_rows(*h, input(u, S0.vu.p, nv, s), S0.x.p, s);
  run_solve(*h, S0, rtol, s);
  scatter_rows(*h, S0.x.p, false, direct ? u : S0.vu.p, s);
  if (!direct) copy_out(u, S0.vu.p, nv, s);
  // the scalars and the start of the history come back together, in pinned memory
  PcgScalars& sc = *static_cast<PcgScalars*>(h->pinned.p);
  double* hist = reinterpret_cast<double*>(static_cast<char*>(h->pinned.p) + READBACK_SCALARS);
  const int nh = std::min(h->prm.max_iter + 1, READBACK_HIST);
  ASMG_CUDA(cudaMemcpyAsync(&sc, S0.scal.p, sizeof sc, cudaMemcpyDeviceToHost, s));
  if (res_history) ASMG_CUDA(cudaMemcpyAsync(hist, S0.hist.p, 8 * (size_t)nh, cudaMemcpyDeviceToHost, s));
  ASMG_CUDA(cudaStreamSynchronize(s));
  *iterations = sc.k;
  if (res_history) {
    std::memcpy(res_history, hist, 8 * (size_t)std::min(sc.k + 1, nh));
    if (sc.k + 1 > nh) {
      ASMG_CUDA(cudaMemcpyAsync(res_history + nh, S0.hist.p + nh, 8 * (size_t)(sc.k + 1 - nh), cudaMemcpyDeviceToHost, s));
      ASMG_CUDA(cudaStreamSynchronize(s));
    }
  }
  if (sc.status == ASMG_ERR_BREAKDOWN) {
    g_err = "PCG breakdown: <p, A p> or <r, z> not positive";
    return ASMG_ERR_BREAKDOWN;
  }
  if (sc.status == ASMG_ERR_TIMEOUT) {
    g_err = "a bounded device wait expired (a tile's shared-memory copy did not complete); u holds the last iterate";
    return ASMG_ERR_TIMEOUT;
  }
  return sc.status == 0 ? ASMG_OK : ASMG_NOT_CONVERGED;
  API_END
}

int amg_solve_multi(asmg_handle h, int k, const double* b, double* u, double rtol, int* iterations, int* status,
                    double* res_history, void* stream) {
  API_BEGIN
  if (!h || !b || !u || !iterations) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  h->check_ready();
  if (k < 1 || k > KRHS) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "k = %d right-hand sides (1..%d)", k, KRHS);
  if (!(rtol >= 0) || !std::isfinite(rtol)) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "rtol must be finite and >= 0");
  if (!multi_supported(*h))
    ASMG_FAIL(ASMG_ERR_UNSUPPORTED, "multiple right-hand sides need the multiplicative Gauss-Seidel PCG without "
                                    "Neumann vertices");
  cudaStream_t s = (cudaStream_t)stream;
  if (h->mslots.empty()) with_room(*h, [&] { grow(h->mslots, [&] { add_multi_slot(*h, s); }); });
  MultiSlot& S = *h->mslots[0];
  const int64_t nv = h->mesh.nv;
  const bool direct = in_place(u);
  gather_multi(*h, input(b, S.vb.p, k * nv, s), k, S.b.p, s);
  gather_multi(*h, input(u, S.vu.p, k * nv, s), k, S.x.p, s);
  run_solve_multi(*h, S, rtol, s);
  scatter_multi(*h, S.x.p, k, direct ? u : S.vu.p, s);
  if (!direct) copy_out(u, S.vu.p, k * nv, s);
  MultiScalars& sc = *static_cast<MultiScalars*>(h->pinned.p);
  ASMG_CUDA(cudaMemcpyAsync(&sc, S.scal.p, sizeof sc, cudaMemcpyDeviceToHost, s));
  ASMG_CUDA(cudaStreamSynchronize(s));
  const int64_t hl = h->prm.max_iter + 1;
  int worst = ASMG_OK;
  for (int c = 0; c < k; ++c) {
    iterations[c] = sc.k[c];
    const int st = sc.status[c] == 0                    ? ASMG_OK
                   : sc.status[c] == ASMG_ERR_BREAKDOWN ? ASMG_ERR_BREAKDOWN
                   : sc.status[c] == ASMG_ERR_TIMEOUT   ? ASMG_ERR_TIMEOUT
                                                        : ASMG_NOT_CONVERGED;
    if (status) status[c] = st;
    if (st < 0 || (worst == ASMG_OK && st != ASMG_OK)) worst = st;
    if (res_history)
      ASMG_CUDA(cudaMemcpyAsync(res_history + c * hl, S.hist.p + c * hl, 8 * (size_t)(sc.k[c] + 1),
                                cudaMemcpyDeviceToHost, s));
  }
  if (res_history) ASMG_CUDA(cudaStreamSynchronize(s));
  if (worst == ASMG_ERR_BREAKDOWN) g_err = "PCG breakdown in a column of a multiple solve";
  if (worst == ASMG_ERR_TIMEOUT) g_err = "a bounded device wait expired in a multiple solve";
  return worst;
  API_END
}

int amg_mass_apply(asmg_handle h, const double* f, double* bout, void* stream) {
  API_BEGIN
  if (!h || !f || !bout) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  Slot& S0 = h->slot0();
  const int64_t nv = h->mesh.nv;
  if (!h->d_v2e_ptr.p) {
    // elements around each vertex, ascending element index (counting sort)
    const MeshHost& m = h->mesh;
    const int nvert = m.dim + 1;
    std::vector<int64_t> ptr(nv + 1, 0);
    for (int64_t k = 0; k < m.ne * nvert; ++k) ++ptr[m.E[k] + 1];
    for (int64_t v = 0; v < nv; ++v) ptr[v + 1] += ptr[v];
    std::vector<int32_t> el(m.ne * nvert);
    std::vector<int64_t> fill(ptr.begin(), ptr.end() - 1);
    for (int64_t e = 0; e < m.ne; ++e)
      for (int k = 0; k < nvert; ++k) el[fill[m.E[e * nvert + k]]++] = (int32_t)e;
    // the handle takes the three arrays together: without all of them the next call builds them
    DBuf<int64_t> dptr;
    DBuf<int32_t> del;
    DBuf<double> dw;
    with_room(*h, [&] {
      dptr.upload(ptr, s);
      del.upload(el, s);
      dw.alloc(m.ne);
    });
    element_mass_gpu(m.dim, m.ne, h->dX.p, h->dE.p, dw.p, s);
    h->d_v2e_ptr = std::move(dptr);
    h->d_v2e = std::move(del);
    h->d_elem_mass = std::move(dw);
  }
  // the result goes straight to the caller's array unless it overlaps the input
  const bool overlap = (uintptr_t)f < (uintptr_t)(bout + nv) && (uintptr_t)bout < (uintptr_t)(f + nv);
  double* out = in_place(bout) && !overlap ? bout : S0.vu.p;
  mass_apply_gpu(h->mesh.dim, nv, h->d_v2e_ptr.p, h->d_v2e.p, h->d_elem_mass.p, h->dE.p, h->d_row_of_vertex.p,
                 input(f, S0.vb.p, nv, s), out, s);
  if (out != bout) copy_out(bout, out, nv, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
  return ASMG_OK;
  API_END
}

int amg_precond_apply(asmg_handle h, const double* r, double* z, void* stream) {
  API_BEGIN
  if (!h || !r || !z) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  Slot& S0 = h->slot0();
  const int64_t nv = h->mesh.nv;
  gather_rows(*h, input(r, S0.vb.p, nv, s), S0.r.p, s);
  int* tflag = reinterpret_cast<int*>(reinterpret_cast<char*>(S0.scal.p) + offsetof(PcgScalars, timeout));
  ASMG_CUDA(cudaMemsetAsync(tflag, 0, sizeof(int), s));
  precond_apply(*h, s);
  const bool direct = in_place(z);
  double* out = direct ? z : S0.vu.p;
  if (h->prm.precision == ASMG_MIXED)
    scatter_rows(*h, S0.s32.uf.p, true, out, s);
  else
    scatter_rows(*h, S0.s64.uf.p, false, out, s);
  if (!direct) copy_out(z, out, nv, s);
  int& tout = *static_cast<int*>(h->pinned.p);
  ASMG_CUDA(cudaMemcpyAsync(&tout, tflag, sizeof(int), cudaMemcpyDeviceToHost, s));
  ASMG_CUDA(cudaStreamSynchronize(s));
  if (tout) ASMG_FAIL(ASMG_ERR_TIMEOUT, "a bounded device wait expired (a tile's shared-memory copy did not complete)");
  return ASMG_OK;
  API_END
}

int amg_spmv(asmg_handle h, const double* x, double* y, void* stream) {
  API_BEGIN
  if (!h || !x || !y) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  Slot& S0 = h->slot0();
  const int64_t nv = h->mesh.nv;
  const bool direct = in_place(y);
  gather_rows(*h, input(x, S0.vb.p, nv, s), S0.p.p, s);
  spmv64(*h, S0.p.p, S0.q.p, s);
  scatter_rows(*h, S0.q.p, false, direct ? y : S0.vu.p, s);
  if (!direct) copy_out(y, S0.vu.p, nv, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
  return ASMG_OK;
  API_END
}

}  // extern "C"

namespace {
// dL/da (scale = NULL) or dL/dg = a dL/da for a = exp(g) (scale = the coefficients)
void element_grad_common(asmg_handle h, const double* u, const double* lambda, double* g, bool log_coeff,
                         cudaStream_t s) {
  Slot& S0 = h->slot0();
  const int64_t nv = h->mesh.nv, ne = h->mesh.ne;
  DBuf<double> dg;
  const bool dev = in_place(g);
  with_room(*h, [&] {
    if (!h->d_pair.p) h->d_pair.alloc(2 * nv);
    if (!dev) dg.alloc(ne);
  });
  double* out = dev ? g : dg.p;
  if (!h->d_elem_stiff.p && !h->elem_stiff_tried) {
    // element stiffness (a = 1), kept while nothing else needs its memory:
    // recomputing it bounds the gradient by the FP64 units
    h->elem_stiff_tried = true;
    try {
      h->d_elem_stiff.alloc(ne * (h->mesh.dim == 2 ? 3 : 6));
      element_stiffness_gpu(h->mesh.dim, ne, h->dX.p, h->dE.p, h->d_elem_stiff.p, s);
    } catch (const Error& e) {
      h->d_elem_stiff.release();
      if (e.code != ASMG_ERR_OOM) throw;
    }
  }
  // (u, lambda) per vertex, Dirichlet entries 0
  mask_pair(*h, input(u, S0.vb.p, nv, s), input(lambda, S0.vu.p, nv, s), h->d_pair.p, s);
  element_grad_gpu(h->mesh.dim, ne, h->dX.p, h->dE.p, h->d_elem_stiff.p, h->d_pair.p,
                   log_coeff ? h->dCoeff.p : nullptr, out, s);
  if (!dev) copy_out(g, dg.p, ne, s);
  ASMG_CUDA(cudaStreamSynchronize(s));
}

void set_coefficients(asmg_handle h, std::vector<double> c, cudaStream_t s) {
  for (int64_t e = 0; e < h->mesh.ne; ++e)
    if (!(c[e] > 0) || !std::isfinite(c[e]))
      ASMG_FAIL(ASMG_ERR_BAD_MESH, "coefficient of element %lld is not positive and finite", (long long)e);
  // from here on the old operators go: with them the work state and graphs that
  // point at them, and the handle's use until the new ones are complete
  h->ready = false;
  ++h->generation;
  h->slots.clear();
  h->mslots.clear();
  h->mesh.coeff = std::move(c);
  with_room(*h, [&] {
    h->dCoeff.upload(h->mesh.coeff, s);
    build_all(*h, s);
  });
}
}  // namespace

extern "C" {

int amg_element_grad(asmg_handle h, const double* u, const double* lambda, double* g, void* stream) {
  API_BEGIN
  if (!h || !u || !lambda || !g) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  element_grad_common(h, u, lambda, g, false, (cudaStream_t)stream);
  return ASMG_OK;
  API_END
}

int amg_element_grad_log(asmg_handle h, const double* u, const double* lambda, double* g, void* stream) {
  API_BEGIN
  if (!h || !u || !lambda || !g) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  element_grad_common(h, u, lambda, g, !h->mesh.coeff.empty(), (cudaStream_t)stream);
  return ASMG_OK;
  API_END
}

int amg_set_log_coefficients(asmg_handle h, const double* gl, void* stream) {
  API_BEGIN
  if (!h || !gl) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<double> c = to_host(gl, h->mesh.ne, s);
  for (auto& x : c) {
    if (!std::isfinite(x)) ASMG_FAIL(ASMG_ERR_BAD_MESH, "log-coefficient is not finite");
    x = std::exp(x);
  }
  set_coefficients(h, std::move(c), s);
  return ASMG_OK;
  API_END
}

int amg_update_coefficients(asmg_handle h, const double* coeff, void* stream) {
  API_BEGIN
  if (!h || !coeff) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  set_coefficients(h, to_host(coeff, h->mesh.ne, s), s);
  return ASMG_OK;
  API_END
}

int amg_info(asmg_handle h, int what, int level, int64_t* value) {
  API_BEGIN
  if (!h || !value) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  h->check_ready();
  auto lev_index = [&](int l) -> int {
    int k = l - (h->aux.c + 1);
    if (k < 0 || k >= (int)h->aux.levels.size()) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "level %d has no smoothing data", l);
    return k;
  };
  auto nsm = [&](int k) -> int64_t {
    return h->prm.precision == ASMG_MIXED ? h->p32.lev[k].nsm_real : h->p64.lev[k].nsm_real;
  };
  switch (what) {
    case ASMG_INFO_NFREE: *value = h->n; break;
    case ASMG_INFO_J: *value = h->aux.J; break;
    case ASMG_INFO_COARSE: *value = h->aux.c; break;
    case ASMG_INFO_NAUX:
      if (level < 0 || level > h->aux.J) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "bad level");
      if (!h->aux.phi.empty()) {
        // mixed grids: the nodes free on this level (phi <= l < psi)
        int64_t c = 0;
        for (size_t q = 0; q < h->aux.phi.size(); ++q) c += h->aux.phi[q] <= level && level < h->aux.psi[q];
        *value = c;
      } else {
        *value = h->aux.nlevel[level];
      }
      break;
    case ASMG_INFO_NSMOOTH: *value = level < 0 ? h->n : nsm(lev_index(level)); break;
    case ASMG_INFO_NCOLOURS:
      if (level < 0) {
        *value = (int64_t)h->fine_cstart.size() - 1;
      } else {
        int k = lev_index(level);
        *value = h->prm.precision == ASMG_MIXED ? h->p32.lev[k].ncolours : h->p64.lev[k].ncolours;
      }
      break;
    case ASMG_INFO_NTREE_LEVELS: *value = (int64_t)h->tree.seg.size(); break;
    case ASMG_INFO_NSEG:
      if (level < 0 || level >= (int)h->tree.seg.size()) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "bad level");
      *value = (int64_t)h->tree.seg[level].size() / 4;
      break;
    case ASMG_INFO_NSPLIT:
      if (level < 0 || level >= (int)h->aux.split.size()) *value = 0;
      else *value = (int64_t)h->aux.split[level].size();
      break;
    case ASMG_INFO_NNZ_A: *value = h->A64.nnz_real; break;
    case ASMG_INFO_NNZ_P: *value = (int64_t)h->aux.P.r.size(); break;
    case ASMG_INFO_NROWS_E: {
      int k = lev_index(level);
      *value = h->prm.precision == ASMG_MIXED ? h->p32.lev[k].nrs : h->p64.lev[k].nrs;
      break;
    }
    case ASMG_INFO_BYTES_ITER: *value = h->bytes_iter; break;
    case ASMG_INFO_NNZ_LEVEL: {
      int k = lev_index(level);
      *value = h->prm.precision == ASMG_MIXED ? h->p32.lev[k].SM.nnz_real + h->p32.lev[k].RS.nnz_real
                                              : h->p64.lev[k].SM.nnz_real + h->p64.lev[k].RS.nnz_real;
      break;
    }
    case ASMG_INFO_NTILES: {
      int k = lev_index(level);
      *value = h->prm.precision == ASMG_MIXED ? (h->p32.lev[k].tiled_down ? h->p32.lev[k].tdown.ntiles : 0)
                                              : (h->p64.lev[k].tiled_down ? h->p64.lev[k].tdown.ntiles : 0);
      break;
    }
    case ASMG_INFO_NTILES_UP: {
      int k = lev_index(level);
      *value = h->prm.precision == ASMG_MIXED ? (h->p32.lev[k].tiled_up ? h->p32.lev[k].tup.ntiles : 0)
                                              : (h->p64.lev[k].tiled_up ? h->p64.lev[k].tup.ntiles : 0);
      break;
    }
    case ASMG_INFO_HALO_ROWS: {
      int k = lev_index(level);
      *value = h->prm.precision == ASMG_MIXED ? h->p32.lev[k].tdown.halo : h->p64.lev[k].tdown.halo;
      break;
    }
    case ASMG_INFO_TILE_SLOTS:
    case ASMG_INFO_TILE_WIDTH: {
      const int k = lev_index(level);
      auto read = [&](const auto& L) -> int64_t {
        if (what == ASMG_INFO_TILE_SLOTS) return (L.tiled_down ? L.tdown.slots : 0) + 16 * (L.tiled_up ? L.tup.slots : 0);
        return (L.tiled_down ? L.tdown.width : 0) + 256 * (L.tiled_up ? L.tup.width : 0);
      };
      *value = h->prm.precision == ASMG_MIXED ? read(h->p32.lev[k]) : read(h->p64.lev[k]);
      break;
    }
    case 100: *value = h->gpu_launches_per_iter; break;
    case 101: *value = (int64_t)(h->stats.t_total * 1e6); break;
    case 102: *value = (int64_t)(h->stats.t_tree * 1e6); break;
    case 103: *value = (int64_t)(h->stats.t_aux * 1e6); break;
    case 104: *value = (int64_t)(h->stats.t_fine * 1e6); break;
    case 105: *value = (int64_t)(h->stats.t_levels * 1e6); break;
    case 108: *value = (int64_t)(h->stats.t_lv_assemble * 1e6); break;
    case 109: *value = (int64_t)(h->stats.t_lv_colour * 1e6); break;
    case 110: *value = (int64_t)(h->stats.t_lv_pack * 1e6); break;
    case 111: *value = (int64_t)(h->stats.t_lv_export * 1e6); break;
    case 112: *value = (int64_t)(h->stats.t_coarse * 1e6); break;
    case 113: *value = (int64_t)(h->stats.t_transfer * 1e6); break;
    case 114: *value = (int64_t)(h->stats.t_slots * 1e6); break;
    case 115: *value = (int64_t)(h->stats.t_sz * 1e6); break;
    default: ASMG_FAIL(ASMG_ERR_INVALID_ARG, "unknown info %d", what);
  }
  return ASMG_OK;
  API_END
}

int amg_export(asmg_handle h, int what, int level, void* buf, int64_t* count) {
  API_BEGIN
  if (!h || !count) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "null argument");
  h->check_ready();
  cudaStream_t s = 0;
  auto put = [&](const void* src, int64_t n, size_t elem) {
    *count = n;
    if (buf && n) std::memcpy(buf, src, elem * n);
  };
  auto trip = [&](const std::vector<uint64_t>& a, const std::vector<uint64_t>& b2, const std::vector<double>& v) {
    *count = (int64_t)v.size();
    if (!buf) return;
    char* o = (char*)buf;
    for (size_t k = 0; k < v.size(); ++k) {
      std::memcpy(o + 24 * k, &a[k], 8);
      std::memcpy(o + 24 * k + 8, &b2[k], 8);
      std::memcpy(o + 24 * k + 16, &v[k], 8);
    }
  };
  switch (what) {
    case ASMG_EXPORT_KEYS: {
      auto k = h->tree.keys.download(s);
      put(k.data(), (int64_t)k.size(), 8);
      break;
    }
    case ASMG_EXPORT_PERM: {
      auto k = h->tree.perm.download(s);
      put(k.data(), (int64_t)k.size(), 4);
      break;
    }
    case ASMG_EXPORT_SEG:
      if (level < 0 || level >= (int)h->tree.seg.size()) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "bad level");
      put(h->tree.seg[level].data(), (int64_t)h->tree.seg[level].size(), 8);
      break;
    case ASMG_EXPORT_SPLIT:
      if (level < 0 || level >= (int)h->aux.split.size()) {
        *count = 0;
      } else {
        put(h->aux.split[level].data(), (int64_t)h->aux.split[level].size(), 8);
      }
      break;
    case ASMG_EXPORT_AUX_KEYS: put(h->aux.aux_key.data(), (int64_t)h->aux.aux_key.size(), 8); break;
    case ASMG_EXPORT_FINE_COLOUR: put(h->fine_colour.data(), (int64_t)h->fine_colour.size(), 4); break;
    case ASMG_EXPORT_SMOOTH: {
      int k = level - (h->aux.c + 1);
      if (k < 0 || k >= (int)h->level_smooth_keys.size()) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "bad level");
      std::vector<uint64_t> v;
      for (size_t i = 0; i < h->level_smooth_keys[k].size(); ++i) {
        v.push_back(h->level_smooth_keys[k][i]);
        v.push_back((uint64_t)h->level_smooth_colour[k][i]);
      }
      put(v.data(), (int64_t)v.size(), 8);
      break;
    }
    case ASMG_EXPORT_LEVEL_ROWS: {
      int k = level - (h->aux.c + 1);
      std::vector<uint64_t> a, b2;
      std::vector<double> v;
      if (level == h->aux.c) {
        // coarsest level: full matrix from its triangles is not stored; export the inverse's source is not kept
        ASMG_FAIL(ASMG_ERR_INVALID_ARG, "the coarsest level keeps only its inverse");
      }
      if (k < 0 || k >= (int)h->level_rows.size()) ASMG_FAIL(ASMG_ERR_INVALID_ARG, "bad level");
      const Triplets& t = h->level_rows[k];
      for (size_t q = 0; q < t.v.size(); ++q) {
        a.push_back(h->aux.aux_key[t.r[q]]);
        b2.push_back(h->aux.aux_key[t.c[q]]);
        v.push_back(t.v[q]);
      }
      trip(a, b2, v);
      break;
    }
    case ASMG_EXPORT_P: {
      std::vector<uint64_t> a, b2;
      std::vector<double> v;
      const Triplets& t = h->aux.P;
      for (size_t q = 0; q < t.v.size(); ++q) {
        a.push_back((uint64_t)h->vertex_of_free[t.r[q]]);
        b2.push_back(h->aux.aux_key[t.c[q]]);
        v.push_back(t.v[q]);
      }
      trip(a, b2, v);
      break;
    }
    case ASMG_EXPORT_FINE_A: {
      std::vector<uint64_t> a, b2;
      std::vector<double> v;
      const HostCSR& A = h->A_host;
      for (int64_t i = 0; i < A.nr; ++i)
        for (int64_t p = A.ptr[i]; p < A.ptr[i + 1]; ++p) {
          a.push_back((uint64_t)h->vertex_of_free[i]);
          b2.push_back((uint64_t)h->vertex_of_free[A.col[p]]);
          v.push_back(A.val[p]);
        }
      trip(a, b2, v);
      break;
    }
    default: ASMG_FAIL(ASMG_ERR_INVALID_ARG, "unknown export %d", what);
  }
  return ASMG_OK;
  API_END
}

}  // extern "C"
