// The entry points of capi.cpp on the CPU, for test_host_entry.py.
//
// A CUDA runtime whose device memory is host memory (with a byte capacity, so
// that allocations can be made to fail) and whose graphs are lists of calls, run
// branch after branch in the order of their capture; and stand-ins for the parts
// of the library that launch kernels: a fine matrix without couplings, an empty
// hierarchy over one coarsest node, a solve that copies b to x.  Everything else
// is the library's own code.  A stand-in that would read an array the library
// does not hold counts it (shim_faults) and reads nothing.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <functional>
#include <map>
#include <set>

#include "../paper_1410_2153_gb300/csrc/handle.h"

using namespace asmg;

namespace {
std::map<char*, size_t> g_live;
std::set<char*> g_host;  // page-locked
size_t g_used = 0, g_peak = 0, g_capacity = SIZE_MAX;
cudaError_t g_last = cudaSuccess;
int g_faults = 0, g_solves = 0;
double g_coef0 = 1;  // the coefficient of element 0 at the last assembly
using Calls = std::vector<std::function<void()>>;
Calls* g_capture = nullptr;
std::map<const void*, HostCSR> g_sell;

void call(std::function<void()> f) {
  if (g_capture) g_capture->push_back(std::move(f));
  else f();
}
char* block_of(const void* p) {
  auto it = g_live.upper_bound((char*)p);
  if (it == g_live.begin()) return nullptr;
  --it;
  return (char*)p < it->first + std::max<size_t>(it->second, 1) ? it->first : nullptr;
}
bool readable(const void* p) {
  if (p && block_of(p)) return true;
  ++g_faults;
  return false;
}
HostCSR diagonal(int64_t n, double v) {
  HostCSR A;
  A.nr = A.nc = n;
  A.ptr.resize(n + 1);
  for (int64_t i = 0; i <= n; ++i) A.ptr[i] = i;
  for (int64_t i = 0; i < n; ++i) {
    A.col.push_back((int32_t)i);
    A.val.push_back(v);
  }
  return A;
}
}  // namespace

// ------------------------------------------------------------ CUDA runtime
extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
  if (n > g_capacity || g_used > g_capacity - n) return g_last = cudaErrorMemoryAllocation;
  *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
  g_live[(char*)*p] = n;
  g_used += n;
  g_peak = std::max(g_peak, g_used);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (p) {
    g_used -= g_live.at((char*)p);
    g_live.erase((char*)p);
    std::free(p);
  }
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return (*p = std::malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (!d || !s) return ++g_faults, cudaErrorInvalidValue;
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "stand-in error"; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  a->type = block_of(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  a->device = 0;
  return cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) {
  *g = reinterpret_cast<cudaGraph_t>(new Calls());
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  delete reinterpret_cast<Calls*>(g);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(new Calls(*reinterpret_cast<Calls*>(g)));
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  delete reinterpret_cast<Calls*>(e);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  for (auto& f : *reinterpret_cast<Calls*>(e)) f();
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = nullptr;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t g, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
  g_capture = reinterpret_cast<Calls*>(g);
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) {
  g_capture = nullptr;
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus*, unsigned long long*, cudaGraph_t*,
                                     const cudaGraphNode_t** deps, const cudaGraphEdgeData**, size_t* n) {
  if (deps) *deps = nullptr;
  if (n) *n = 0;
  return cudaSuccess;
}
}

// ------------------------------------------------- parts that launch kernels
namespace asmg {
template <class T>
void sell_build(Sell<T>& S, const HostCSR& rows, int32_t, cudaStream_t) {
  S.nrows = rows.nr;
  S.nnz_real = (int64_t)rows.col.size();
  g_sell[&S] = rows;
}
template void sell_build<double>(Sell<double>&, const HostCSR&, int32_t, cudaStream_t);
template void sell_build<float>(Sell<float>&, const HostCSR&, int32_t, cudaStream_t);
void sell_bf16(Sell<float>&, cudaStream_t) {}

void build_tree_gpu(int, int64_t, const double*, int64_t, const int32_t*, int, cudaStream_t, TreeResult& t) { t.L = 1; }
HostCSR assemble_mesh(int, int64_t, const double*, const int32_t*, const int32_t*, const double* coef, int64_t n,
                      cudaStream_t) {
  g_coef0 = coef ? coef[0] : 1;
  return diagonal(n, g_coef0);
}
// coarsest matrix: not positive definite for a coefficient above 1e100
HostCSR assemble_simplices(int, int64_t, const double*, const int32_t*, const double* coef, const uint8_t*, int64_t n,
                           cudaStream_t) {
  return diagonal(n, coef[0] > 1e100 ? -1 : 1);
}
// two colour classes for a coefficient of 2 and more, else one
std::vector<int32_t> jp_colour_gpu(const HostCSR& A, const std::vector<uint8_t>&, const std::vector<uint64_t>&,
                                   cudaStream_t) {
  std::vector<int32_t> c(A.nr, 0);
  for (int64_t i = 0; g_coef0 >= 2 && i < A.nr; ++i) c[i] = (int32_t)(i % 2);
  return c;
}
void build_aux_host(const MeshHost& m, const TreeResult&, const asmg_params&, AuxHost& a) {
  a.aux_key = {0};
  a.nlevel = {1, 1};
  a.J = 1;
  a.coarse_id = {0};
  a.coarse_tri_id = {0, -1, -1};
  a.coarse_tri_key = {0, 0, 0};
  a.coarse_tri_coef = {m.coeff.empty() ? 1 : m.coeff[0]};
}
void build_aux_host3(const MeshHost& m, const TreeResult& t, const asmg_params& p, AuxHost& a) { build_aux_host(m, t, p, a); }
void build_transfer(const MeshHost&, const double*, const int32_t*, const std::vector<int32_t>& vof, const SZTable&,
                    Triplets& P, cudaStream_t) {
  for (size_t i = 0; i < vof.size(); ++i) {
    P.r.push_back((int32_t)i);
    P.c.push_back(0);
    P.v.push_back((double)i + 1);
  }
}
void lattice_point(const TreeResult&, uint64_t, double* p) { p[0] = p[1] = 0; }
void lattice_point3(const TreeResult&, int, uint64_t, double* p) { p[0] = p[1] = p[2] = 0; }

bool multi_supported(const asmg_s&) { return true; }
Slot& add_slot(asmg_s& h, cudaStream_t) {
  h.slots.emplace_back(new Slot());
  Slot& S = *h.slots.back();
  for (DBuf<double>* v : {&S.b, &S.x, &S.r, &S.p, &S.q}) v->alloc(h.npad);
  S.vb.alloc(h.mesh.nv);
  S.vu.alloc(h.mesh.nv);
  S.hist.alloc(h.prm.max_iter + 1);
  S.scal.alloc(1);
  S.scal.zero(nullptr);
  (h.prm.precision == ASMG_MIXED ? (void)S.s32.uf.alloc(h.npad) : (void)S.s64.uf.alloc(h.npad));
  return S;
}
MultiSlot& add_multi_slot(asmg_s& h, cudaStream_t) {
  h.mslots.emplace_back(new MultiSlot());
  MultiSlot& S = *h.mslots.back();
  for (DBuf<double>* v : {&S.b, &S.x}) v->alloc(h.npad * KRHS);
  S.vb.alloc(h.mesh.nv * KRHS);
  S.vu.alloc(h.mesh.nv * KRHS);
  S.scal.alloc(1);
  S.scal.zero(nullptr);
  return S;
}
void setup_solve(asmg_s& h, cudaStream_t s) {
  h.slots.clear();
  h.mslots.clear();
  add_slot(h, s);
}
int run_solve(asmg_s&, Slot& S, double, cudaStream_t) {
  ++g_solves;
  if (readable(S.x.p)) std::copy(S.b.p, S.b.p + S.b.n, S.x.p);
  return 0;
}
void run_solve_multi(asmg_s&, MultiSlot& S, double, cudaStream_t) {
  ++g_solves;
  if (readable(S.x.p)) std::copy(S.b.p, S.b.p + S.b.n, S.x.p);
}
cudaGraphNode_t capture_solve(asmg_s& h, Slot& S, double, cudaGraph_t g, const cudaGraphNode_t*, size_t) {
  reinterpret_cast<Calls*>(g)->push_back([&] { run_solve(h, S, 0, nullptr); });
  return nullptr;
}
cudaGraphNode_t capture_solve_multi(asmg_s& h, MultiSlot& S, double, cudaGraph_t g, const cudaGraphNode_t*, size_t) {
  reinterpret_cast<Calls*>(g)->push_back([&] { run_solve_multi(h, S, 0, nullptr); });
  return nullptr;
}
int64_t iteration_bytes(asmg_s&) { return 0; }
int profile_solve(asmg_s&, double, cudaStream_t, double*, double*, int) {
  ++g_solves;
  return 0;
}
void precond_apply(asmg_s&, cudaStream_t) { ++g_solves; }
void spmv64(asmg_s&, const double*, double*, cudaStream_t) { ++g_solves; }
double* noalloc_scratch_for_current_device() { return nullptr; }
void residual_norm_noalloc(asmg_s&, const double*, const double*, double*, cudaStream_t) { ++g_solves; }

// column j of k interleaved ones
static void gather_col(asmg_s& h, const double* src, double* dst, int j, int k) {
  if (!readable(dst)) return;
  for (int64_t i = 0; i < h.npad; ++i) dst[i * k + j] = 0;
  for (int64_t v = 0; src && v < h.mesh.nv; ++v)
    if (h.d_row_of_vertex.p[v] >= 0) dst[(int64_t)h.d_row_of_vertex.p[v] * k + j] = src[v];
}
static void scatter_col(asmg_s& h, const double* src, double* dst, int j, int k) {
  if (!readable(src)) return;
  for (int64_t v = 0; dst && v < h.mesh.nv; ++v)
    dst[v] = h.d_row_of_vertex.p[v] >= 0 ? src[(int64_t)h.d_row_of_vertex.p[v] * k + j] : 0;
}
void gather_rows(asmg_s& h, const double* v, double* d, cudaStream_t) { gather_col(h, v, d, 0, 1); }
void scatter_rows(asmg_s& h, const void* s, bool f32, double* d, cudaStream_t) {
  if (!f32) scatter_col(h, (const double*)s, d, 0, 1);
}
void gather_rows_tab(asmg_s& h, double* const* tab, double* d, cudaStream_t) {
  call([&h, tab, d] { gather_col(h, tab[0], d, 0, 1); });
}
void scatter_rows_tab(asmg_s& h, const double* s, double* const* tab, cudaStream_t) {
  call([&h, tab, s] { scatter_col(h, s, tab[0], 0, 1); });
}
void gather_multi(asmg_s& h, const double* v, int k, double* d, cudaStream_t) {
  for (int j = 0; j < KRHS; ++j) gather_col(h, j < k ? v + j * h.mesh.nv : nullptr, d, j, KRHS);
}
void scatter_multi(asmg_s& h, const double* s, int k, double* d, cudaStream_t) {
  for (int j = 0; j < k; ++j) scatter_col(h, s, d + j * h.mesh.nv, j, KRHS);
}
void gather_multi_tab(asmg_s& h, double* const* tab, double* d, cudaStream_t) {
  call([&h, tab, d] {
    for (int j = 0; j < KRHS; ++j) gather_col(h, tab[j], d, j, KRHS);
  });
}
void scatter_multi_tab(asmg_s& h, const double* s, double* const* tab, cudaStream_t) {
  call([&h, tab, s] {
    for (int j = 0; j < KRHS; ++j) scatter_col(h, s, tab[j], j, KRHS);
  });
}

void element_mass_gpu(int, int64_t ne, const double*, const int32_t*, double* w, cudaStream_t) {
  ASMG_CUDA(cudaGetLastError());
  if (readable(w)) std::fill(w, w + ne, 1.0);
}
void mass_apply_gpu(int, int64_t nv, const int64_t* ptr, const int32_t* el, const double* w, const int32_t*,
                    const int32_t* row, const double* f, double* b, cudaStream_t) {
  ASMG_CUDA(cudaGetLastError());
  if (!readable(ptr) || !readable(el) || !readable(w)) return;
  for (int64_t v = 0; v < nv; ++v) {
    b[v] = 0;
    for (int64_t p = ptr[v]; row[v] >= 0 && p < ptr[v + 1]; ++p) b[v] += w[el[p]] * f[v];
  }
}
void element_stiffness_gpu(int, int64_t ne, const double*, const int32_t*, double* K, cudaStream_t) {
  ASMG_CUDA(cudaGetLastError());
  if (readable(K)) K[ne - 1] = 1;
}
void mask_pair(asmg_s& h, const double* u, const double* l, double* pair, cudaStream_t) {
  ASMG_CUDA(cudaGetLastError());
  if (!readable(pair)) return;
  for (int64_t v = 0; v < h.mesh.nv; ++v) {
    pair[2 * v] = u[v];
    pair[2 * v + 1] = l[v];
  }
}
void element_grad_gpu(int dim, int64_t ne, const double*, const int32_t* E, const double*, const double* pair,
                      const double* scale, double* g, cudaStream_t) {
  ASMG_CUDA(cudaGetLastError());
  if (!readable(pair)) return;
  for (int64_t e = 0; e < ne; ++e) {
    const int64_t v = E[e * (dim + 1)];
    g[e] = pair[2 * v] * pair[2 * v + 1] * (scale ? scale[e] : 1);
  }
}
}  // namespace asmg

// ----------------------------------------------------------------- the test's
extern "C" {
double* shim_device(int64_t n) {
  void* p = nullptr;
  return cudaMalloc(&p, 8 * (size_t)n) == cudaSuccess ? (double*)p : nullptr;
}
void shim_device_free(double* p) { cudaFree(p); }
int64_t shim_used() { return (int64_t)g_used; }
// the most bytes held since the last call; starts anew from what is held now
int64_t shim_peak() {
  const size_t p = g_peak;
  g_peak = g_used;
  return (int64_t)p;
}
void shim_capacity(int64_t bytes) { g_capacity = bytes < 0 ? SIZE_MAX : (size_t)bytes; }
int shim_faults() { return g_faults; }
int shim_solves() { return g_solves; }
// column counts of the transfer's rows in the order they were last laid out (row of the first column's entry values)
int64_t shim_transfer(asmg_handle h, double* val) {
  const HostCSR& P = g_sell[h->prm.precision == ASMG_MIXED ? (const void*)&h->p32.P : (const void*)&h->p64.P];
  for (int64_t i = 0; val && i < P.nr; ++i) val[i] = P.ptr[i + 1] > P.ptr[i] ? P.val[P.ptr[i]] : 0;
  return P.nr;
}
}
