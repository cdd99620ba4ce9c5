// gqt_host.cuh -- what the library's host translation units share: graph replay of
// launch loops, kernel dispatch over a handle's storage, and small launches.
#pragma once

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <map>
#include <string>
#include <type_traits>
#include <vector>

#include "gqt_df.cuh"
#include "gqt_internal.h"
#include "gqt_kernels.cuh"

namespace gqt {

extern std::atomic<uint64_t> g_launches;
bool prof_on();

// (2 - delta_m0) (-sign i)^m J_m(x), m < Np (Eq. 17).
std::vector<double2> evolve_coefs(double x, int sign, int Np);

// 2H~, 2U/dE (and 2[X,H~]) of an FP64 handle as pairs of FP32 numbers, split on first
// use and after an update, on the call's stream and before any capture.
void ensure_df(gqt_ham* h, cudaStream_t st);
void ensure_df_x(gqt_ham* h, cudaStream_t st);

// In-place evolution of NSET vector sets (each [n][R]) by the coefficients c of Eq. 17.
template <int NSET>
void launch_evolve_sets(gqt_ham* h, void* const* psi, int R, const std::vector<double2>& c, cudaStream_t st,
                        double* d_norms /* [nseg][R][2*NSET] or null */);
extern template void launch_evolve_sets<1>(gqt_ham*, void* const*, int, const std::vector<double2>&, cudaStream_t,
                                           double*);
extern template void launch_evolve_sets<2>(gqt_ham*, void* const*, int, const std::vector<double2>&, cudaStream_t,
                                           double*);
// One MSD time step (p, px) -> (U p, [X,U] p + U px).
void launch_msd_step(gqt_ham* h, void* p, void* px, int R, const std::vector<double2>& c, cudaStream_t st);

// ---------------------------------------------------------------- graphs

// Replays a loop of launches as a CUDA graph keyed by everything the launches
// depend on (kind, sizes, pointers, coefficients).  Capture and replay run on
// the handle's own non-blocking stream, ordered after and before the caller's
// stream by events, so the caller may pass the legacy default stream.
// 64-bit digest of a coefficient array (SplitMix64 finaliser folded over the
// words, so sign patterns cannot cancel); the array itself is stored with the
// graph and compared exactly on reuse.
inline uint64_t digest(const std::vector<double>& v) {
  uint64_t x = 0x243F6A8885A308D3ull ^ (uint64_t)v.size();
  for (double d : v) {
    uint64_t u;
    memcpy(&u, &d, 8);
    x = splitmix_mix(x ^ u) + 0x9E3779B97F4A7C15ull;
  }
  return x;
}

template <class F>
inline void run_graph(gqt_ham* h, std::string key, cudaStream_t st, F&& launches,
                      const std::vector<double>* data = nullptr) {
  if (!h->use_graphs || prof_on()) {
    launches(st);
    return;
  }
  if (data) {
    char buf[40];
    snprintf(buf, sizeof buf, "|d%016llx", (unsigned long long)digest(*data));
    key += buf;
    auto d = h->graph_data.find(key);
    if (d != h->graph_data.end() && d->second != *data) {  // digest collision: no graph
      launches(st);
      return;
    }
  }
  if (!h->gstream) {
    check_cuda(cudaStreamCreateWithFlags(&h->gstream, cudaStreamNonBlocking), "cudaStreamCreate");
    check_cuda(cudaEventCreateWithFlags(&h->gev[0], cudaEventDisableTiming), "cudaEventCreate");
    check_cuda(cudaEventCreateWithFlags(&h->gev[1], cudaEventDisableTiming), "cudaEventCreate");
  }
  auto it = h->graphs.find(key);
  if (it == h->graphs.end()) {
    if (h->graphs.size() >= 512) h->drop_graphs();
    cudaGraph_t graph = nullptr;
    check_cuda(cudaStreamBeginCapture(h->gstream, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture");
    try {
      launches(h->gstream);
    } catch (...) {
      cudaStreamEndCapture(h->gstream, &graph);
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      throw;
    }
    check_cuda(cudaStreamEndCapture(h->gstream, &graph), "cudaStreamEndCapture");
    cudaGraphExec_t exec = nullptr;
    cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    check_cuda(e, "cudaGraphInstantiate");
    it = h->graphs.emplace(key, exec).first;
    if (data) h->graph_data[key] = *data;
  }
  check_cuda(cudaEventRecord(h->gev[0], st), "cudaEventRecord");
  check_cuda(cudaStreamWaitEvent(h->gstream, h->gev[0], 0), "cudaStreamWaitEvent");
  check_cuda(cudaGraphLaunch(it->second, h->gstream), "cudaGraphLaunch");
  g_launches.fetch_add(1, std::memory_order_relaxed);
  check_cuda(cudaEventRecord(h->gev[1], h->gstream), "cudaEventRecord");
  check_cuda(cudaStreamWaitEvent(st, h->gev[1], 0), "cudaStreamWaitEvent");
}

inline std::string key_of(const char* op, std::initializer_list<const void*> ptrs, std::initializer_list<double> nums) {
  std::string k(op);
  char buf[64];
  for (auto p : ptrs) {
    snprintf(buf, sizeof buf, "|%p", p);
    k += buf;
  }
  for (auto x : nums) {
    snprintf(buf, sizeof buf, "|%.17g", x);
    k += buf;
  }
  return k;
}

// The exact bits of every expansion coefficient, as part of a graph key (a
// lossy hash can map U(+dt) and U(-dt), whose coefficients differ only in
// signs, to the same key).
inline std::string coef_bits(const std::vector<double2>& c) {
  std::string k("|c");
  char buf[40];
  for (const double2& q : c) {
    uint64_t u[2];
    memcpy(u, &q, 16);
    snprintf(buf, sizeof buf, "%016llx%016llx", (unsigned long long)u[0], (unsigned long long)u[1]);
    k += buf;
  }
  return k;
}

// dynamic shared memory of the CTA reductions (NV values per vector per warp)
inline size_t smem_bytes(const gqt_ham* h, int R, int nv) { return (size_t)nv * (h->threads / 32) * R * sizeof(double2); }

inline int rshift_of(int R) {
  int s = 0;
  while ((1 << s) < R) ++s;
  return s;
}

// ---------------------------------------------------------------- dispatch

template <bool FP64, bool CH>
inline Ell<FP64, CH> ell_of(const gqt_ham* h) {
  Ell<FP64, CH> e;
  e.n = (int)h->n;
  e.K = h->K;
  e.idx = (const int*)h->d_idx.p;
  e.hop2 = (const typename Ell<FP64, CH>::HT*)h->d_hop.p;
  e.diag2 = (const typename Ell<FP64, CH>::S*)h->d_diag.p;
  e.dx = (const typename Ell<FP64, CH>::S*)h->d_dx.p;
  e.cls = h->has_cls ? (const uint16_t*)h->d_cls.p : nullptr;
  e.cls_off = (const int*)h->d_cls_off.p;
  e.uni = !FP64 && h->hop_uniform32;
  e.h0 = (typename Ell<FP64, CH>::S)h->hop0f;
  e.row_shift = (h->use_sweep_order && h->row_shift > 0) ? h->row_shift : 0;
  return e;
}

template <class F>
inline void dispatch(const gqt_ham* h, F&& f) {
  if (h->prec == GQT_FP64) {
    if (h->hop_real)
      f(ell_of<true, false>(h));
    else
      f(ell_of<true, true>(h));
  } else {
    if (h->hop_real)
      f(ell_of<false, false>(h));
    else
      f(ell_of<false, true>(h));
  }
}

template <class E>
struct EllTraits;
template <bool FP64, bool CH>
struct EllTraits<Ell<FP64, CH>> {
  static constexpr bool fp64 = FP64;
  static constexpr bool ch = CH;
  using V = typename Prec<FP64>::V;
};

// Segment sums of the partial slots slot0 .. slot0 + nslots - 1 (and slot extra, if
// >= 0), in place, before k_reduce, k_reduce_dbl or a norm check reads them.
inline void launch_slot_sums(double2* partial, int nblocks, int R, const int* seg_blk, int nseg, int slot0, int nslots,
                             int extra, cudaStream_t st) {
  const long long items = (long long)(nslots + (extra >= 0 ? 1 : 0)) * nseg;
  k_slot_sums<<<(unsigned)std::min<long long>(items, 1 << 20), 256, 0, st>>>(partial, nblocks, R, seg_blk, nseg, slot0, nslots, extra);
  check_launch("k_slot_sums");
}

template <bool CH>
inline DfEll<CH> df_ell_of(const gqt_ham* h) {
  DfEll<CH> e;
  e.n = (int)h->n;
  e.K = h->K;
  e.idx = (const int*)h->d_idx.p;
  e.hop = (const typename DfHop<CH>::T*)h->d_hop_df.p;
  e.diag = (const float2*)h->d_diag_df.p;
  e.cls = h->has_cls ? (const uint16_t*)h->d_cls.p : nullptr;
  e.cls_off = (const int*)h->d_cls_off.p;
  e.xhop = (const typename DfHop<CH>::T*)h->d_xhop_df.p;
  if (h->hop_uniform) {
    const float a = (float)h->hop0;
    e.h0 = make_float2(a, (float)(h->hop0 - (double)a));
  }
  return e;
}


// FP64 vectors as pairs (T_0 of a row's or an evolution's chains).
template <int NV>
inline void launch_split(void* const* in, float4* const* out, size_t n, cudaStream_t st) {
  DfSplit<NV> A;
  for (int q = 0; q < NV; ++q) {
    A.in[q] = (const double2*)in[q];
    A.out[q] = out[q];
  }
  k_split_vec<NV><<<(int)std::min<size_t>((n + 255) / 256, (size_t)sm_count() * 8), 256, 0, st>>>(A, n);
  check_launch("k_split_vec");
}

inline bool is_pow2_r(int R) { return R == 1 || R == 2 || R == 4 || R == 8 || R == 16 || R == 32; }

// ---------------------------------------------------------------- status

inline gqt_status finish_call(gqt_ham* h, cudaStream_t st, const char* what) {
  int flag = 0;
  check_cuda(cudaMemcpyAsync(h->h_flag, h->d_flag.p, sizeof(int), cudaMemcpyDeviceToHost, st), "flag readback");
  check_cuda(cudaStreamSynchronize(st), what);
  flag = *h->h_flag;
  check_waits(flag, what);  // first: what the other checks saw may be its consequence
  if (flag & 4) throw Error(GQT_ENAN, std::string(what) + ": NaN or Inf in a result");
  if (flag & 2)
    throw Error(GQT_ERANGE, std::string(what) +
                                ": a Chebyshev moment exceeds |l||r|: the spectrum of H/dE is not inside [-1,1] "
                                "(energy scale too small)");
  if (flag & 8) throw Error(GQT_ENORM, std::string(what) + ": |U psi| differs from |psi| beyond tolerance");
  return GQT_OK;
}

inline void reset_flag(gqt_ham* h, cudaStream_t st) {
  check_cuda(cudaMemsetAsync(h->d_flag.p, 0, sizeof(int), st), "flag reset");
}

// ---------------------------------------------------------------- API helpers

#define API_BEGIN \
  gqt::NvtxRange nvtx_call_(__func__); \
  try {
#define API_END                                        \
  }                                                    \
  catch (const Error& e) {                             \
    set_error(e.what());                               \
    return e.code;                                     \
  }                                                    \
  catch (const std::bad_alloc&) {                      \
    set_error("host allocation failed");               \
    return GQT_ENOMEM;                                 \
  }                                                    \
  catch (const std::exception& e) {                    \
    set_error(std::string("internal error: ") + e.what()); \
    return GQT_EINVAL;                                 \
  }                                                    \
  return GQT_OK;

inline void require(bool c, const std::string& msg) {
  if (!c) throw Error(GQT_EINVAL, msg);
}

inline bool is_host_ptr(const void* p) {
  cudaPointerAttributes a;
  cudaError_t e = cudaPointerGetAttributes(&a, p);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return true;
  }
  return a.type == cudaMemoryTypeUnregistered || a.type == cudaMemoryTypeHost;
}

inline void check_common(gqt_ham* h, int R) {
  require(h != nullptr, "null handle");
  require(is_pow2_r(R), "R must be 1, 2, 4, 8, 16 or 32");
  int dev = -1;
  check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
  require(dev == h->device, "the current CUDA device is not the handle's device");
}

inline int resolve_np(gqt_ham* h, double dt, int Np) {
  require(std::isfinite(dt) && dt >= 0.0, "time step must be finite and >= 0");
  if (Np > 0) return Np;
  return np_rule_lib(h->dE * dt, 4096);
}

}  // namespace gqt
