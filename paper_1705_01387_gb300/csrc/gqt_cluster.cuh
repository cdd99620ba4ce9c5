// gqt_cluster.cuh -- moment rows of small systems in one persistent launch on a
// thread-block cluster.
//
// When the whole problem fits on chip, the per-order kernel launches of the
// large-N path (a few microseconds each) dominate.  Here one cluster of C CTAs
// (C = 16 where the GPU allows, else 8) runs all orders of a row: CTA c keeps
// sites [c*chunk, (c+1)*chunk) of the two Chebyshev vectors (and of l, and its
// rows of H~) in its shared memory; neighbour gathers read other CTAs' shared
// memory through the cluster's distributed shared memory; orders are separated
// by hardware cluster barriers (no software waits).  Per-CTA partial dot
// products go to the same [slot][CTA] layout as the large-N kernels and are
// reduced by the same deterministic pass.
#pragma once

#include <cooperative_groups.h>

#include "gqt_kernels.cuh"

namespace gqt {

namespace cgc = cooperative_groups;

// Shared-memory bytes per site of a cluster-resident row.
// Per-order partial sums kept until the end: (slots) x (warps) double2.
inline size_t cluster_red_bytes(int M, int slot_norm, int warps) {
  const int slots = (M > slot_norm ? M : slot_norm + 1) + 2;
  return (size_t)slots * warps * 16;
}

template <bool FP64, bool CH>
__host__ __device__ constexpr int cluster_site_bytes(int K, bool with_l) {
  return (int)(sizeof(typename Prec<FP64>::V) * (with_l ? 3 : 2) + K * (4 + sizeof(typename Ell<FP64, CH>::HT)) +
               sizeof(typename Prec<FP64>::S));
}

// DBL: l = r doubling (slots 2m-2, 2m-1 for step m = 1 .. steps); else Re <l|T_m|r>
// for m = 0 .. M-1 (slots m, norms in slot_norm).  R = 1, single segment.
template <bool FP64, bool CH, bool DBL>
__global__ void k_cheb_cluster(Ell<FP64, CH> H, int chunk, const typename Prec<FP64>::V* __restrict__ r,
                               const typename Prec<FP64>::V* __restrict__ l, double2* __restrict__ partial, int M,
                               int slot_norm) {
  using V = typename Prec<FP64>::V;
  using S = typename Prec<FP64>::S;
  using HT = typename Ell<FP64, CH>::HT;
  cgc::cluster_group cluster = cgc::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int me = (int)cluster.block_rank();
  const int K = H.K;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  V* TA = reinterpret_cast<V*>(sm_raw);
  V* TB = TA + chunk;
  V* LV = TB + chunk;  // only with !DBL
  HT* hs = reinterpret_cast<HT*>(DBL ? (void*)LV : (void*)(LV + chunk));
  S* ds = reinterpret_cast<S*>(hs + (size_t)K * chunk);
  int* is = reinterpret_cast<int*>(ds + chunk);
  // per-order partial sums: one double2 per (slot, warp), summed over warps at the end
  double2* red = reinterpret_cast<double2*>(is + (size_t)K * chunk + 4);
  red = reinterpret_cast<double2*>((reinterpret_cast<uintptr_t>(red) + 15) & ~(uintptr_t)15);
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int beg = me * chunk;
  const int cnt = max(0, min(chunk, H.n - beg));
  for (int q = threadIdx.x; q < cnt; q += blockDim.x) {
    const int i = beg + q;
    TA[q] = r[i];
    if (!DBL) LV[q] = l[i];
    ds[q] = H.diag2[i];
    for (int k = 0; k < K; ++k) {
      is[k * chunk + q] = H.idx[(size_t)k * H.n + i];
      hs[k * chunk + q] = H.hop2[(size_t)k * H.n + i];
    }
  }
  cluster.sync();
  auto reduce = [&](double2 v, int slot) {  // warp sum into red[slot][warp]; no block barrier
    for (int off = 16; off > 0; off >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
    }
    if (lane == 0) red[(size_t)slot * nw + warp] = v;
  };
  // order m computes T_m into the buffer of T_{m-2}; T_{m-1} is read across the cluster
  const int last = DBL ? max((M + 1) / 2, 1) : M - 1;
  V* prev = TA;  // T_{m-1}
  V* cur = TB;   // T_{m-2} -> T_m
  for (int m = 1; m <= last; ++m) {
    DotAcc<V> d0, d1, n0, n1;
    for (int q = threadIdx.x; q < cnt; q += blockDim.x) {
      const V own = prev[q];
      V a;
      if (m == 1) {
        a = cscale(own, ds[q]);
      } else {
        a = cmul_acc(cneg(cur[q]), ds[q], own);
      }
      for (int k = 0; k < K; ++k) {
        const int j = is[k * chunk + q];
        const int rk = j / chunk;
        const V* src = cluster.map_shared_rank(prev, rk);
        a = cmul_acc(a, hs[k * chunk + q], src[j - rk * chunk]);
      }
      if (m == 1) a = cscale(a, (S)0.5);
      if (DBL) {
        d0.add_norm(own);
        d1.add_re(a, own);
      } else {
        if (m == 1) {
          d0.add_re(LV[q], own);
          n0.add_norm(LV[q]);
          n1.add_norm(own);
        }
        d1.add_re(LV[q], a);
      }
      cur[q] = a;
    }
    if (DBL) {
      reduce(d0.get(), 2 * m - 2);
      reduce(d1.get(), 2 * m - 1);
    } else {
      if (m == 1) {
        reduce(d0.get(), 0);
        reduce(make_double2(n0.get().x, n1.get().x), slot_norm);
      }
      reduce(d1.get(), m);
    }
    cluster.sync();  // T_m complete everywhere; nobody reads T_{m-1} any more
    V* t = prev;
    prev = cur;
    cur = t;
  }
  if (!DBL && M == 1) {  // only mu_0 and the norms
    DotAcc<V> d0, n0, n1;
    for (int q = threadIdx.x; q < cnt; q += blockDim.x) {
      d0.add_re(LV[q], TA[q]);
      n0.add_norm(LV[q]);
      n1.add_norm(TA[q]);
    }
    reduce(d0.get(), 0);
    reduce(make_double2(n0.get().x, n1.get().x), slot_norm);
  }
  __syncthreads();
  const int nslots = DBL ? 2 * max((M + 1) / 2, 1) : slot_norm + 1;
  for (int sl = threadIdx.x; sl < nslots; sl += blockDim.x) {
    if (!DBL && sl > M - 1 && sl != slot_norm) continue;
    double2 a = make_double2(0.0, 0.0);
    for (int w = 0; w < nw; ++w) {
      a.x += red[(size_t)sl * nw + w].x;
      a.y += red[(size_t)sl * nw + w].y;
    }
    partial[(size_t)sl * C + me] = a;
  }
  cluster.sync();  // no CTA leaves while another may still read its shared memory
}

// ---------------------------------------------------------------- one site per thread
//
// Rows of up to 512 sites per CTA (8192 in a cluster of 16) with 2, 3, 4 or 6 neighbour
// slots, both moments of an order by the product identities: l = r rows (PAIR = false)
// and the two-recurrence l != r rows (PAIR = true), as the large-N kernels.  A thread
// keeps its site's H~ row, its neighbours' distributed shared-memory addresses and its
// own T_{m-1} and T_{m-2} in registers.  An order is a serial chain -- gather, FP64
// multiply-adds (4 warps x 8 instructions of 16 cycles each on the SM's FP64 pipe),
// store, cluster barrier -- so whatever is not part of it is moved under the barrier:
// the order's two dots are formed between arriving and waiting, and instead of two
// warp sums per order (40 FP64 adds and 80 shuffles a warp) the threads' values go to a
// ring in shared memory that is added up every 16 orders.  At the end the CTAs sum
// their slots over the cluster and write the moments and their checks directly.
// At 2048 sites (16 CTAs of 128) an order takes 0.85 us instead of 1.98 us, and a VAC row
// half as many of them: DOS row of 512 moments 545 -> 260 us per call, VAC row 729 -> 345
// us.
constexpr int CL_RING = 32;  // slots in the ring: 16 orders

__host__ __device__ inline size_t cluster1_smem(int chunk, int threads, int steps, int vec_bytes, bool pair) {
  return (size_t)chunk * vec_bytes * (pair ? 4 : 2) + (size_t)CL_RING * (threads + 4) * sizeof(double) +
         ((size_t)((2 * steps + CL_RING - 1) / CL_RING) * CL_RING + 2) * sizeof(double);
}

__device__ __forceinline__ uint32_t cl_map(const void* p, int rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ double2 cl_ld(uint32_t a, double2) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float2 cl_ld(uint32_t a, float2) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ double cl_ld(uint32_t a, double) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// An element's term Re conj(a) b of a dot, as DotAcc forms it (FP32 storage: one FP32
// rounding), then FP64.
__device__ __forceinline__ double cl_re(double2 a, double2 b) { return fma(a.x, b.x, a.y * b.y); }
__device__ __forceinline__ double cl_re(float2 a, float2 b) { return (double)fmaf(a.x, b.x, a.y * b.y); }

template <bool FP64, bool CH, bool PAIR, int KK>
__global__ void __launch_bounds__(512) k_cheb_cluster1(Ell<FP64, CH> H, int chunk,
                                                       const typename Prec<FP64>::V* __restrict__ l,
                                                       const typename Prec<FP64>::V* __restrict__ r, int M,
                                                       double bound_factor, double* __restrict__ out,
                                                       int* __restrict__ flag) {
  using V = typename Prec<FP64>::V;
  using S = typename Prec<FP64>::S;
  using HT = typename Ell<FP64, CH>::HT;
  cgc::cluster_group cluster = cgc::this_cluster();
  const int C = (int)cluster.num_blocks(), me = (int)cluster.block_rank();
  const int tid = (int)threadIdx.x, thr = (int)blockDim.x;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  V* B0 = reinterpret_cast<V*>(sm_raw);  // chain B (or the only one): T_m at even, odd m
  V* B1 = B0 + chunk;
  V* A0 = B1 + chunk;  // chain A, PAIR only
  const uint32_t flip = (uint32_t)((size_t)chunk * sizeof(V));       // B0 -> B1, A0 -> A1
  const uint32_t toA = (uint32_t)((size_t)2 * chunk * sizeof(V));    // B0 -> A0
  double* ring = reinterpret_cast<double*>(sm_raw + (size_t)chunk * sizeof(V) * (PAIR ? 4 : 2));
  double* red = ring + CL_RING * (thr + 4);  // sums of this CTA, [slots]
  const int steps = max((M + 1) / 2, 1), nslots = (2 * steps + CL_RING - 1) / CL_RING * CL_RING;
  double* nrm = red + nslots;  // |l|^2, |r|^2 of this CTA (PAIR)
  const int i = me * chunk + tid;
  const bool on = tid < chunk && i < H.n;
  uint32_t adr[KK];
  HT hv[KK];
  S dg = 0;
  V b, bo, a, ao;  // own T_{m-1} and T_{m-2} of chains B and A
  b.x = b.y = 0;
  bo = a = ao = b;
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    adr[k] = cl_map(B0, me);
    hv[k] = HT{};
  }
  if (on) {
    b = r[i];
    B0[tid] = b;
    if (PAIR) {
      a = l[i];
      A0[tid] = a;
    }
    dg = H.diag2[i];
#pragma unroll
    for (int k = 0; k < KK; ++k) {
      const size_t s = (size_t)k * H.n + i;
      const int j = H.idx[s], rk = j / chunk;
      adr[k] = cl_map(B0 + (j - rk * chunk), rk);
      hv[k] = H.hop2[s];
    }
  }
  if (PAIR) {
    double v[2] = {on ? cl_re(a, a) : 0.0, on ? cl_re(b, b) : 0.0};
    block_reduce_rx<2>(v, 1, ring);
    if (tid == 0) {
      nrm[0] = v[0];
      nrm[1] = v[1];
    }
  }
  cluster.sync();
  const int parts = thr / CL_RING;
  uint32_t src = 0;  // 0: T_{m-1} in B0 / A0, flip: in B1 / A1
  for (int m = 1; m <= steps; ++m) {
    V nb, na;
    nb.x = nb.y = 0;
    na = nb;
    if (on) {
      V gb[KK], ga[KK];
#pragma unroll
      for (int k = 0; k < KK; ++k) {
        gb[k] = cl_ld(adr[k] + src, V());
        if (PAIR) ga[k] = cl_ld(adr[k] + toA + src, V());
      }
      nb = m == 1 ? cscale(b, dg) : cmul_acc(cneg(bo), dg, b);
      if (PAIR) na = m == 1 ? cscale(a, dg) : cmul_acc(cneg(ao), dg, a);
#pragma unroll
      for (int k = 0; k < KK; ++k) {
        nb = cmul_acc(nb, hv[k], gb[k]);
        if (PAIR) na = cmul_acc(na, hv[k], ga[k]);
      }
      if (m == 1) {
        nb = cscale(nb, (S)0.5);
        if (PAIR) na = cscale(na, (S)0.5);
      }
      V* dst = src ? B0 : B1;
      dst[tid] = nb;
      if (PAIR) dst[2 * chunk + tid] = na;
    }
    cl_arrive();
    // under the barrier: slots 2m-2 and 2m-1
    const int s0 = (2 * m - 2) & (CL_RING - 1);
    ring[s0 * (thr + 4) + tid] = on ? (PAIR ? cl_re(a, b) : cl_re(b, b)) : 0.0;
    ring[(s0 + 1) * (thr + 4) + tid] = on ? (PAIR ? cl_re(a, nb) : cl_re(nb, b)) : 0.0;
    if (s0 == CL_RING - 2 || m == steps) {
      __syncthreads();
      const int slot = tid / parts, part = tid - slot * parts;
      double w[8], v;  // eight runs, added in pairs
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = 0.0;
#pragma unroll
      for (int j = 0; j < CL_RING; ++j) w[j & 7] += ring[slot * (thr + 4) + part + parts * j];
      v = ((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]));
      for (int off = parts >> 1; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      if (part == 0) red[(2 * m - 2 - s0) + slot] = v;
      __syncthreads();
    }
    bo = b;
    b = nb;
    ao = a;
    a = na;
    src ^= flip;
    cl_wait();  // T_m complete everywhere; nobody reads T_{m-1} any more
  }
  cluster.sync();  // every CTA's sums are written
  auto total = [&](const double* p) {
    double v = 0.0;
    for (int q = 0; q < C; q += 4)  // C is 8 or 16
      v += (cl_ld(cl_map(p, q), 0.0) + cl_ld(cl_map(p, q + 1), 0.0)) +
           (cl_ld(cl_map(p, q + 2), 0.0) + cl_ld(cl_map(p, q + 3), 0.0));
    return v;
  };
  if (me * thr + tid < M) {
    const double s_even = total(red), s_odd = total(red + 1);
    const double top = PAIR ? sqrt(total(nrm) * total(nrm + 1)) : s_even;
    for (int k = me * thr + tid; k < M; k += C * thr) {
      const double sk = total(red + k);
      const double mu = k < 2 ? sk : 2.0 * sk - ((k & 1) ? s_odd : s_even);
      out[k] = mu;
      if (!isfinite(mu)) atomicOr(flag, 4);
      if (fabs(mu) > top * bound_factor + 1e-300) atomicOr(flag, 2);
    }
  }
  cluster.sync();  // no CTA leaves while another may still read its shared memory
}

// Allows a cluster kernel clusters of C CTAs and its largest shared memory.  The attributes
// belong to the kernel, which all handles and threads share: they are set to the same
// values by every call, never to what one call needs, since another thread may launch
// between the two.
constexpr size_t CL_SMEM = 220 * 1024;
template <class KERN>
inline bool cluster_attributes(KERN kern, int C) {
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CL_SMEM) == cudaSuccess &&
      (C <= 8 || cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess))
    return true;
  cudaGetLastError();
  return false;
}

// Launches one of the one-site-per-thread cluster kernels for n sites: clusters of 16
// CTAs where the GPU allows, else 8, of a power of two of threads (the ring's parts), at
// most 512; smem_of(chunk, threads) bytes of shared memory; f(config, chunk) launches.
// False where the system does not fit or clusters are unavailable.
template <class KERN, class SM, class F>
inline bool cluster1_launch(KERN kern, int64_t n, cudaStream_t st, SM&& smem_of, F&& f) {
  for (int C : {16, 8}) {
    const int chunk = (int)((n + C - 1) / C);
    int thr = 32;
    while (thr < chunk && thr <= 512) thr *= 2;
    if (thr > 512) continue;
    const size_t smem = smem_of(chunk, thr);
    if (smem > CL_SMEM || !cluster_attributes(kern, C)) continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C, 1, 1);
    cfg.blockDim = dim3(thr, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) != cudaSuccess || nclusters < 1) {
      cudaGetLastError();
      continue;
    }
    f(cfg, chunk);
    return true;
  }
  return false;
}

// ---------------------------------------------------------------- evolution of small systems
//
// All orders of U(+-dt) (Eq. 17) or of the coupled commutator recursion (Eqs. 18, 22,
// 24) in one launch, for FP64 handles with one vector and at most 512 sites per CTA: the
// layout of k_cheb_cluster1, the accumulators in registers.  One launch per order takes
// 3.8 us at 2048 sites whatever it computes; here an order is a gather through
// distributed shared memory, its FP64 multiply-adds and a cluster barrier.  FP64
// throughout.  At 2048 sites two vectors evolve by 18 orders in 35 us instead of 80 us
// (pair arithmetic, one launch per order).
constexpr int CL_ORDERS = 128;  // orders at most (kernel argument)

struct ClusterCoefs {
  double c[CL_ORDERS];  // real part at even, imaginary part at odd orders
  int n;
};

__device__ __forceinline__ void cl_term(double2& a, double c, int m, double2 t) {
  const bool odd = m & 1;
  a.x = fma(odd ? -c : c, odd ? t.y : t.x, a.x);
  a.y = fma(c, odd ? t.x : t.y, a.y);
}

// Cluster-wide sums of v (NV values per thread), in every thread of CTA 0; red: 8 doubles
// of shared memory for block_reduce_rx and NV results per CTA.
template <int NV>
__device__ __forceinline__ void cl_sums(cgc::cluster_group& cluster, double (&v)[NV], double* red, double* res) {
  block_reduce_rx<NV>(v, 1, red);
  if (threadIdx.x == 0)
#pragma unroll
    for (int q = 0; q < NV; ++q) res[q] = v[q];
  cluster.sync();
  if (cluster.block_rank() == 0)
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      v[q] = 0.0;
      for (int b = 0; b < (int)cluster.num_blocks(); ++b) v[q] += cl_ld(cl_map(res + q, b), 0.0);
    }
  cluster.sync();
}

template <int NSET>
struct ClusterSets {
  double2* psi[NSET];
};

template <bool CH, int NSET, int KK>
__global__ void __launch_bounds__(512) k_evolve_cluster(Ell<true, CH> H, int chunk, ClusterSets<NSET> A,
                                                        const __grid_constant__ ClusterCoefs C, double tol,
                                                        double* __restrict__ norms, int* __restrict__ flag) {
  using HT = typename Ell<true, CH>::HT;
  cgc::cluster_group cluster = cgc::this_cluster();
  const int me = (int)cluster.block_rank(), tid = (int)threadIdx.x;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  double2* buf = reinterpret_cast<double2*>(sm_raw);  // [2][NSET][chunk]
  double* red = reinterpret_cast<double*>(buf + (size_t)2 * NSET * chunk);
  double* res = red + 16 * 2 * NSET;
  const uint32_t flip = (uint32_t)((size_t)NSET * chunk * sizeof(double2)), set = (uint32_t)(chunk * sizeof(double2));
  const int i = me * chunk + tid;
  const bool on = tid < chunk && i < H.n;
  uint32_t adr[KK];
  HT hv[KK];
  double dg = 0.0;
  double2 b[NSET], bo[NSET], acc[NSET];
  double nrm[2 * NSET];
#pragma unroll
  for (int q = 0; q < NSET; ++q) {
    b[q] = bo[q] = acc[q] = make_double2(0.0, 0.0);
    nrm[q] = nrm[NSET + q] = 0.0;
  }
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    adr[k] = 0;
    hv[k] = HT{};
  }
  if (on) {
    dg = H.diag2[i];
#pragma unroll
    for (int k = 0; k < KK; ++k) {
      const size_t s = (size_t)k * H.n + i;
      const int j = H.idx[s], rk = j / chunk;
      adr[k] = cl_map(buf + (j - rk * chunk), rk);
      hv[k] = H.hop2[s];
    }
#pragma unroll
    for (int q = 0; q < NSET; ++q) {
      b[q] = A.psi[q][i];
      buf[q * chunk + tid] = b[q];
      nrm[q] = cl_re(b[q], b[q]);
      cl_term(acc[q], C.c[0], 0, b[q]);
    }
  }
  cluster.sync();
  uint32_t src = 0;
  for (int m = 1; m < C.n; ++m) {
    if (on) {
      double2 g[NSET][KK], y[NSET];
#pragma unroll
      for (int q = 0; q < NSET; ++q)
#pragma unroll
        for (int k = 0; k < KK; ++k) g[q][k] = cl_ld(adr[k] + q * set + src, double2());
#pragma unroll
      for (int q = 0; q < NSET; ++q) {
        y[q] = m == 1 ? cscale(b[q], dg) : cmul_acc(cneg(bo[q]), dg, b[q]);
#pragma unroll
        for (int k = 0; k < KK; ++k) y[q] = cmul_acc(y[q], hv[k], g[q][k]);
        if (m == 1) y[q] = cscale(y[q], 0.5);
        buf[(src ? 0 : NSET * chunk) + q * chunk + tid] = y[q];
        bo[q] = b[q];
        b[q] = y[q];
      }
    }
    cl_arrive();
#pragma unroll
    for (int q = 0; q < NSET; ++q) cl_term(acc[q], C.c[m], m, b[q]);  // under the barrier
    src ^= flip;
    cl_wait();
  }
  if (on)
#pragma unroll
    for (int q = 0; q < NSET; ++q) {
      A.psi[q][i] = acc[q];
      nrm[NSET + q] = cl_re(acc[q], acc[q]);
    }
  cl_sums<2 * NSET>(cluster, nrm, red, res);
  if (me == 0 && tid == 0)
#pragma unroll
    for (int q = 0; q < NSET; ++q) {
      const double a = nrm[q], z = nrm[NSET + q];
      if (norms) {
        norms[2 * q] = a;
        norms[2 * q + 1] = z;
      }
      if (!isfinite(z)) atomicOr(flag, 4);
      if (fabs(sqrt(z) - sqrt(a)) > tol * sqrt(a) + 1e-300) atomicOr(flag, 8);
    }
}

// One MSD time step: (p, px) -> (U p, [X, U] p + U px).
template <bool CH, int KK>
__global__ void __launch_bounds__(512) k_msd_cluster(Ell<true, CH> H, int chunk, double2* p, double2* px,
                                                     const __grid_constant__ ClusterCoefs C, double tol,
                                                     int* __restrict__ flag) {
  using HT = typename Ell<true, CH>::HT;
  cgc::cluster_group cluster = cgc::this_cluster();
  const int me = (int)cluster.block_rank(), tid = (int)threadIdx.x;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  double2* buf = reinterpret_cast<double2*>(sm_raw);  // [2][u, z][chunk]
  double* red = reinterpret_cast<double*>(buf + (size_t)4 * chunk);
  double* res = red + 16 * 3;
  const uint32_t flip = (uint32_t)((size_t)2 * chunk * sizeof(double2)), set = (uint32_t)(chunk * sizeof(double2));
  const int i = me * chunk + tid;
  const bool on = tid < chunk && i < H.n;
  uint32_t adr[KK];
  HT hv[KK];
  double dx[KK], dg = 0.0;
  const double2 zero = make_double2(0.0, 0.0);
  double2 u = zero, uo = zero, z = zero, zo = zero, au = zero, az = zero;
  double nrm[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    adr[k] = 0;
    hv[k] = HT{};
    dx[k] = 0.0;
  }
  if (on) {
    dg = H.diag2[i];
#pragma unroll
    for (int k = 0; k < KK; ++k) {
      const size_t s = (size_t)k * H.n + i;
      const int j = H.idx[s], rk = j / chunk;
      adr[k] = cl_map(buf + (j - rk * chunk), rk);
      hv[k] = H.hop2[s];
      dx[k] = -H.dx[s];
    }
    u = p[i];
    z = px[i];
    buf[tid] = u;
    buf[chunk + tid] = z;
    nrm[0] = cl_re(u, u);
    cl_term(au, C.c[0], 0, u);
    cl_term(az, C.c[0], 0, z);
  }
  cluster.sync();
  uint32_t src = 0;
  for (int m = 1; m < C.n; ++m) {
    if (on) {
      double2 gu[KK], gz[KK];
#pragma unroll
      for (int k = 0; k < KK; ++k) {
        gu[k] = cl_ld(adr[k] + src, double2());
        gz[k] = cl_ld(adr[k] + set + src, double2());
      }
      double2 nu = m == 1 ? cscale(u, dg) : cmul_acc(cneg(uo), dg, u);
      double2 nz = m == 1 ? cscale(z, dg) : cmul_acc(cneg(zo), dg, z);
#pragma unroll
      for (int k = 0; k < KK; ++k) {
        nu = cmul_acc(nu, hv[k], gu[k]);
        nz = cmul_acc(nz, hv[k], gz[k]);
        nz = cmul_acc(nz, hv[k], cscale(gu[k], dx[k]));
      }
      if (m == 1) {
        nu = cscale(nu, 0.5);
        nz = cscale(nz, 0.5);
      }
      double2* dst = buf + (src ? 0 : 2 * chunk) + tid;
      dst[0] = nu;
      dst[chunk] = nz;
      uo = u;
      u = nu;
      zo = z;
      z = nz;
    }
    cl_arrive();
    cl_term(au, C.c[m], m, u);
    cl_term(az, C.c[m], m, z);
    src ^= flip;
    cl_wait();
  }
  if (on) {
    p[i] = au;
    px[i] = az;
    nrm[1] = cl_re(au, au);
    nrm[2] = cl_re(az, az);
  }
  cl_sums<3>(cluster, nrm, red, res);
  if (me == 0 && tid == 0) {
    if (!isfinite(nrm[1]) || !isfinite(nrm[2])) atomicOr(flag, 4);
    if (fabs(sqrt(nrm[1]) - sqrt(nrm[0])) > tol * sqrt(nrm[0]) + 1e-300) atomicOr(flag, 8);
  }
}

}  // namespace gqt
