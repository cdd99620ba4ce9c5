// gqt_evolve.cu -- time evolution U(+-dt) (Eq. 17) and the coupled commutator
// recursion of the MSD (Eqs. 18, 22, 24): kernels of the wavefront order and the
// loops over expansion orders.
//
// The sum of c_m T_m psi is kept in an accumulator (FP64, or pairs of FP32 numbers for
// FP64 handles with one vector).  Reading and writing it at every order costs as much
// traffic as the recursion itself (FP64 handles: 32 of 80 bytes per element and order;
// FP32 storage: 32 of 56), so it is touched every third order only: at order m a thread
// holds T_{m-2}, T_{m-1} and T_m of its element anyway and adds the three terms at once
// (pairs, two sets of 16.8M elements: 455 us per order before, 275 us without and 445 us
// with the accumulator now, both at the HBM rate; coupled orders of 4.2M: 131 -> 111 us).
// The coefficients (2 - d_m0) (-+i)^m J_m are purely real at even and purely imaginary
// at odd m, so a term costs one real multiplication per component instead of a complex
// one.

#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "gqt_cluster.cuh"
#include "gqt_host.cuh"

using namespace gqt;

namespace gqt {

// The accumulator's terms of one order m: c[j] multiplies T_{m-2+j} (real where m - 2 +
// j is even, times i where it is odd); on: this order adds its terms; acc_in: the
// accumulator holds earlier terms (else it is written without being read).
template <class C>
struct EvoTerms {
  C c[3];
  int odd;
  int on;
  int acc_in;
};

// ---------------------------------------------------------------- pairs of FP32 numbers (R = 1)

// U(dt) psi for NSET vector sets sharing H~ on pairs.  Orders by phase:
//   PH 0 (m = 1): out = T_1 = H~ T_0 from the pairs t1 = T_0; acc = c[1] T_0 + c[2] T_1
//                 where on (c[2] may be zero); |psi|^2 partials (slot);
//   PH 1 (2 <= m < Np - 1): out = 2H~ t1 - t2 (over t2, same element and thread);
//   PH 2 (m = Np - 1): psi = the sum in FP64 (hi + lo of two FP32 numbers is exact in
//                 FP64), |psi|^2 partials;
//   PH 3 (Np <= 2): psi = acc in FP64, |psi|^2 partials.
template <int NSET>
struct DfEvo {
  double2* psi[NSET];
  const float4* t1[NSET];
  const float4* t2[NSET];
  float4* out[NSET];
  float4* acc[NSET];
};

__device__ __forceinline__ double2 df_to_d2(float4 f) { return make_double2(df_value(f.x, f.z), df_value(f.y, f.w)); }

// CLS: neighbours by the row's class.  The commutator orders, which stream six vectors a
// site, lose more by its second dependent load (31 -> 34 us at N = 1M, K = 4) than the
// index array costs them.
template <bool CH, int KK, bool UH, bool CLS>
__device__ __forceinline__ void df_row_ops(const DfEll<CH>& H, int i, int (&idx)[KK],
                                           typename DfHop<CH>::T (&hv)[KK], float2& dg) {
  if (CLS) {
    row_neighbours<KK>(H.idx, H.cls, H.cls_off, H.n, i, row_class(H.cls, i), idx);
  } else {
#pragma unroll
    for (int k = 0; k < KK; ++k) idx[k] = __ldg(H.idx + (size_t)k * H.n + i);
  }
  if (!UH)
#pragma unroll
    for (int k = 0; k < KK; ++k) hv[k] = __ldg(H.hop + (size_t)k * H.n + i);
  dg = __ldg(H.diag + i);
}

// a += the order's three terms
__device__ __forceinline__ void df_terms(DfC& a, const EvoTerms<float2>& t, float4 tm2, float4 tm1, float4 tm) {
  if (t.odd) {
    dfc_mac_i(a, t.c[0], tm2);
    dfc_mac(a, t.c[1], tm1);
    dfc_mac_i(a, t.c[2], tm);
  } else {
    dfc_mac(a, t.c[0], tm2);
    dfc_mac_i(a, t.c[1], tm1);
    dfc_mac(a, t.c[2], tm);
  }
}

// acc + the terms, normalised; `first`: acc holds nothing yet
__device__ __forceinline__ float4 df_accumulate(const float4* acc, size_t e, const EvoTerms<float2>& t, float4 tm2,
                                                float4 tm1, float4 tm) {
  DfC a = t.acc_in ? dfc_of(acc[e]) : dfc_zero();
  df_terms(a, t, tm2, tm1, tm);
  return dfc_out(a, false);
}

template <bool CH, int KK, int NSET, int PH, bool UH = false>
__global__ void __launch_bounds__(256) k_evolve_df(DfEll<CH> H, const int4* __restrict__ tab, DfEvo<NSET> A,
                                                   EvoTerms<float2> t, double2* __restrict__ partial, int nblocks,
                                                   int slot) {
  using HT = typename DfHop<CH>::T;
  const int4 tb = tab[blockIdx.x];
  const size_t sege = (size_t)tb.y, step = (size_t)tb.w * blockDim.x;
  chain_wait();
  DfDot nrm[NSET];
  for (size_t e = (size_t)tb.x + (size_t)tb.z * blockDim.x + threadIdx.x; e < sege; e += step) {
    const int i = (int)e;
    if (PH == 3) {
#pragma unroll
      for (int q = 0; q < NSET; ++q) {
        const float4 f = A.acc[q][e];
        A.psi[q][e] = df_to_d2(f);
        nrm[q].add_norm(f);
      }
      continue;
    }
    int idx[KK];
    HT hv[KK];
    float2 dg;
    df_row_ops<CH, KK, UH, true>(H, i, idx, hv, dg);
#pragma unroll
    for (int q = 0; q < NSET; ++q) {
      const float4 own = A.t1[q][e];
      float4 nb[KK];
#pragma unroll
      for (int k = 0; k < KK; ++k) nb[k] = A.t1[q][idx[k]];
      const float4 t2 = PH == 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : A.t2[q][e];
      const float4 y = df_step_any<CH, KK, PH == 0, UH>(H, hv, dg, own, nb, t2);
      if (PH != 2) A.out[q][e] = y;
      if (PH == 0) nrm[q].add_norm(own);
      if (PH == 2 || t.on) {
        const float4 f = df_accumulate(A.acc[q], e, t, t2, own, y);
        if (PH == 2) {
          A.psi[q][e] = df_to_d2(f);
          nrm[q].add_norm(f);
        } else {
          A.acc[q][e] = f;
        }
      }
    }
  }
  if (PH != 1) {
    double v[NSET];
#pragma unroll
    for (int q = 0; q < NSET; ++q) v[q] = nrm[q].get();
    block_reduce_rx<NSET>(v, 1, reinterpret_cast<double*>(dyn_smem()));
    if (threadIdx.x == 0) {
#pragma unroll
      for (int q = 0; q < NSET; ++q) partial[(size_t)(slot + q) * nblocks + blockIdx.x] = make_double2(v[q], 0.0);
    }
  }
}

// One MSD time step's coupled orders (Eqs. 17, 18, 22, 24) on pairs, R = 1:
//   u_m = T_m(H~) p,  z_m = [X, T_m] p + T_m px,
//   z_m = 2[X,H~] u_{m-1} + 2H~ z_{m-1} - z_{m-2}  (z_1 = [X,H~] p + H~ px),
//   accp += c_m u_m (-> U(dt) p), accx += c_m z_m (-> [X,U(dt)]p + U(dt)px).
// Phases as k_evolve_df; the partial slots are those of k_msd_evolve
// (k_norm_check_msd reads them).
struct DfMsd {
  double2* p;
  double2* px;
  const float4* u1;
  const float4* u2;
  const float4* z1;
  const float4* z2;
  float4* uo;
  float4* zo;
  float4* accp;
  float4* accx;
};

template <bool CH, int KK, int PH, bool UH = false>
__global__ void __launch_bounds__(256) k_msd_evolve_df(DfEll<CH> H, const int4* __restrict__ tab, DfMsd B,
                                                       EvoTerms<float2> t, double2* __restrict__ partial, int nblocks,
                                                       int slot) {
  using HT = typename DfHop<CH>::T;
  const int4 tb = tab[blockIdx.x];
  const size_t sege = (size_t)tb.y, step = (size_t)tb.w * blockDim.x;
  chain_wait();
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  DfDot n0, n1;
  for (size_t e = (size_t)tb.x + (size_t)tb.z * blockDim.x + threadIdx.x; e < sege; e += step) {
    const int i = (int)e;
    if (PH == 3) {
      const float4 fp = B.accp[e], fx = B.accx[e];
      B.p[e] = df_to_d2(fp);
      B.px[e] = df_to_d2(fx);
      n0.add_norm(fp);
      n1.add_norm(fx);
      continue;
    }
    int idx[KK];
    HT hv[KK];
    float2 dg;
    df_row_ops<CH, KK, UH, false>(H, i, idx, hv, dg);
    const float4 u_own = B.u1[e], z_own = B.z1[e];
    float4 un[KK];
#pragma unroll
    for (int k = 0; k < KK; ++k) un[k] = B.u1[idx[k]];
    const float4 u2 = PH == 0 ? zero : B.u2[e], z2 = PH == 0 ? zero : B.z2[e];
    const float4 uo = df_step_any<CH, KK, PH == 0, UH>(H, hv, dg, u_own, un, u2);
    DfC a = df_start<PH == 0>(dg, z_own, z2);
    float4 zn[KK];
#pragma unroll
    for (int k = 0; k < KK; ++k) zn[k] = B.z1[idx[k]];
    if constexpr (UH) {
      dfc_mac_sum<KK>(a, H.h0, zn);
    } else {
#pragma unroll
      for (int k = 0; k < KK; ++k) dfc_mac(a, hv[k], zn[k]);
    }
#pragma unroll
    for (int k = 0; k < KK; ++k) dfc_mac(a, __ldg(H.xhop + (size_t)k * H.n + i), un[k]);
    const float4 zo = dfc_out(a, PH == 0);
    if (PH != 2) {
      B.uo[e] = uo;
      B.zo[e] = zo;
    }
    if (PH == 0) n0.add_norm(u_own);
    if (PH == 2 || t.on) {
      const float4 fp = df_accumulate(B.accp, e, t, u2, u_own, uo);
      const float4 fx = df_accumulate(B.accx, e, t, z2, z_own, zo);
      if (PH == 2) {
        B.p[e] = df_to_d2(fp);
        B.px[e] = df_to_d2(fx);
        n0.add_norm(fp);
        n1.add_norm(fx);
      } else {
        B.accp[e] = fp;
        B.accx[e] = fx;
      }
    }
  }
  if (PH != 1) {
    double v[2] = {n0.get(), n1.get()};
    block_reduce_rx<2>(v, 1, reinterpret_cast<double*>(dyn_smem()));
    if (threadIdx.x == 0) {
      partial[(size_t)slot * nblocks + blockIdx.x] = make_double2(v[0], 0.0);
      partial[(size_t)(slot + 1) * nblocks + blockIdx.x] = make_double2(v[1], 0.0);
    }
  }
}

// ---------------------------------------------------------------- storage precision, R vectors
//
// Wavefront form of k_evolve and k_msd_evolve for the neighbour counts 2, 3, 4 and 6:
// G = R / VW lanes serve one site, a lane holding VW vectors (two FP32 ones in one
// 16-byte load, one otherwise); the recursion's multiply-adds are in the order of
// k_evolve and k_msd_evolve, so the vectors equal theirs bit for bit.  k_evolve itself
// was bound by the FP64 pipe (four multiply-adds and two conversions per element where
// two of the products are by zero) and by its accumulator traffic: 669 us per order of 2 x
// 16.8M elements (R = 8), here 185 us for an order without and 521 us for one with
// the accumulator, 268 us on average.

__device__ __forceinline__ double2 widen(float2 a) { return make_double2(f2d(a.x), f2d(a.y)); }
__device__ __forceinline__ double2 widen(double2 a) { return a; }

template <int VW>
__device__ __forceinline__ void evo_ld(float2 (&d)[VW], const float2* p) {
  if (VW == 2) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    d[0] = make_float2(t.x, t.y);
    d[VW - 1] = make_float2(t.z, t.w);
  } else {
    d[0] = *p;
  }
}
template <int VW>
__device__ __forceinline__ void evo_ldg(float2 (&d)[VW], const float2* __restrict__ p) {
  if (VW == 2) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    d[0] = make_float2(t.x, t.y);
    d[VW - 1] = make_float2(t.z, t.w);
  } else {
    d[0] = __ldg(p);
  }
}
template <int VW>
__device__ __forceinline__ void evo_st(float2* p, const float2 (&d)[VW]) {
  if (VW == 2)
    *reinterpret_cast<float4*>(p) = make_float4(d[0].x, d[0].y, d[VW - 1].x, d[VW - 1].y);
  else
    *p = d[0];
}
template <int VW>
__device__ __forceinline__ void evo_ld(double2 (&d)[VW], const double2* p) {
#pragma unroll
  for (int w = 0; w < VW; ++w) d[w] = p[w];
}
template <int VW>
__device__ __forceinline__ void evo_ldg(double2 (&d)[VW], const double2* __restrict__ p) {
#pragma unroll
  for (int w = 0; w < VW; ++w) d[w] = __ldg(p + w);
}
template <int VW>
__device__ __forceinline__ void evo_st(double2* p, const double2 (&d)[VW]) {
#pragma unroll
  for (int w = 0; w < VW; ++w) p[w] = d[w];
}

// acc += c T (odd = 0) or i c T (odd = 1).  The operands are chosen, not the operations:
// two predicated variants of the multiply-adds would both take the FP64 pipe's time
// (an order with three terms of 2 x 16.8M FP32 elements: 941 us so, 521 us
// with the choice).
template <class V>
__device__ __forceinline__ void evo_term(double2& acc, double c, int odd, V tv) {
  V u;
  u.x = odd ? tv.y : tv.x;
  u.y = odd ? tv.x : tv.y;
  const double2 t = widen(u);
  acc.x = fma(odd ? -c : c, t.x, acc.x);
  acc.y = fma(c, t.y, acc.y);
}

template <class V, int VW>
__device__ __forceinline__ void evo_accumulate(double2 (&a)[VW], const EvoTerms<double>& t, const V (&tm2)[VW],
                                               const V (&tm1)[VW], const V (&tm)[VW], bool two) {
  if (!t.acc_in)
#pragma unroll
    for (int w = 0; w < VW; ++w) a[w] = make_double2(0.0, 0.0);
#pragma unroll
  for (int w = 0; w < VW; ++w) {
    if (!two) evo_term(a[w], t.c[0], t.odd, tm2[w]);
    evo_term(a[w], t.c[1], t.odd ^ 1, tm1[w]);
    evo_term(a[w], t.c[2], t.odd, tm[w]);
  }
}

// The H~ row of site i.
template <class E, int KK>
struct EvoRow {
  int idx[KK];
  typename E::HT hv[KK];
  typename E::S dg;
  __device__ __forceinline__ EvoRow(const E& H, int i) {
    row_neighbours<KK>(H.idx, H.cls, H.cls_off, H.n, i, row_class(H.cls, i), idx);
#pragma unroll
    for (int k = 0; k < KK; ++k) hv[k] = hop_of(H, k, i);
    dg = __ldg(H.diag2 + i);
  }
};

// Per-vector norms of a CTA into slot (vector r of lane lg: r = VW lg + w).
template <int NV, int VW>
__device__ __forceinline__ void evo_norms(double2 (&v)[NV * VW], int R, int G, double2* __restrict__ partial,
                                          int nblocks, int slot) {
  block_reduce_r<NV * VW>(v, G, dyn_smem());
  if ((int)threadIdx.x < G) {
#pragma unroll
    for (int q = 0; q < NV; ++q)
#pragma unroll
      for (int w = 0; w < VW; ++w)
        partial[((size_t)(slot + q) * nblocks + blockIdx.x) * R + VW * threadIdx.x + w] = v[q * VW + w];
  }
}

// Phases as k_evolve: 0 (m = 1): out = H~ t1, t1 = psi; 1: out = 2H~ t1 - t2; 2 (last):
// fin = the sum; 3 (Np <= 2): fin = acc.
template <int NSET, bool FP64, bool CH, int VW, int KK>
__global__ void __launch_bounds__(256) k_evolve_w(Ell<FP64, CH> H, const int4* __restrict__ tab, int R, int gs,
                                                  EvoSets<NSET, FP64> A, EvoTerms<double> t, int phase,
                                                  double2* __restrict__ partial, int nblocks, int slot) {
  using V = typename Prec<FP64>::V;
  using S = typename Prec<FP64>::S;
  const int4 tb = tab[blockIdx.x];
  const size_t ge = (size_t)tb.y << gs, step = (size_t)tb.w * blockDim.x;
  const int G = 1 << gs, off = VW * ((int)threadIdx.x & (G - 1));
  DotAcc<V> nrm[NSET * VW];
  for (size_t gi = ((size_t)tb.x << gs) + (size_t)tb.z * blockDim.x + threadIdx.x; gi < ge; gi += step) {
    const int i = site_of(H, (int)(gi >> gs));
    const size_t e = (size_t)i * R + off;
    if (phase == 3) {
#pragma unroll
      for (int q = 0; q < NSET; ++q) {
        double2 a[VW];
        V f[VW];
        evo_ld<VW>(a, A.acc[q] + e);
#pragma unroll
        for (int w = 0; w < VW; ++w) {
          f[w] = from_d2<V>(a[w]);
          nrm[q * VW + w].add_norm(f[w]);
        }
        evo_st<VW>(A.fin[q] + e, f);
      }
      continue;
    }
    // every load of both sets before the first store (which might alias them)
    const EvoRow<Ell<FP64, CH>, KK> row(H, i);
    V own[NSET][VW], t2[NSET][VW], nb[NSET][KK][VW], y[NSET][VW];
    double2 a[NSET][VW];
#pragma unroll
    for (int q = 0; q < NSET; ++q) {
      evo_ldg<VW>(own[q], A.t1[q] + e);
      if (phase != 0) evo_ld<VW>(t2[q], A.t2[q] + e);
#pragma unroll
      for (int k = 0; k < KK; ++k) evo_ldg<VW>(nb[q][k], A.t1[q] + (size_t)row.idx[k] * R + off);
      if (t.on && t.acc_in) evo_ld<VW>(a[q], A.acc[q] + e);
    }
#pragma unroll
    for (int q = 0; q < NSET; ++q)
#pragma unroll
      for (int w = 0; w < VW; ++w) {
        if (phase == 0) {
          t2[q][w].x = 0;
          t2[q][w].y = 0;
          y[q][w] = t2[q][w];
        } else {
          y[q][w] = cneg(t2[q][w]);
        }
        y[q][w] = cmul_acc(y[q][w], row.dg, own[q][w]);
#pragma unroll
        for (int k = 0; k < KK; ++k) y[q][w] = cmul_acc(y[q][w], row.hv[k], nb[q][k][w]);
        if (phase == 0) {
          y[q][w] = cscale(y[q][w], (S)0.5);
          nrm[q * VW + w].add_norm(own[q][w]);
        }
      }
    if (phase != 2)
#pragma unroll
      for (int q = 0; q < NSET; ++q) evo_st<VW>(A.out[q] + e, y[q]);
    if (t.on) {
#pragma unroll
      for (int q = 0; q < NSET; ++q) {
        evo_accumulate<V, VW>(a[q], t, t2[q], own[q], y[q], phase == 0);
        if (phase == 2) {
          V f[VW];
#pragma unroll
          for (int w = 0; w < VW; ++w) {
            f[w] = from_d2<V>(a[q][w]);
            nrm[q * VW + w].add_norm(f[w]);
          }
          evo_st<VW>(A.fin[q] + e, f);
        } else {
          evo_st<VW>(A.acc[q] + e, a[q]);
        }
      }
    }
  }
  if (phase != 1) {
    double2 v[NSET * VW];
#pragma unroll
    for (int q = 0; q < NSET * VW; ++q) v[q] = nrm[q].get();
    evo_norms<NSET, VW>(v, R, G, partial, nblocks, slot);
  }
}

template <bool FP64, bool CH, int VW, int KK>
__global__ void __launch_bounds__(256) k_msd_evolve_w(Ell<FP64, CH> H, const int4* __restrict__ tab, int R, int gs,
                                                      MsdBufs<FP64> B, EvoTerms<double> t, int phase,
                                                      double2* __restrict__ partial, int nblocks, int slot) {
  using V = typename Prec<FP64>::V;
  using S = typename Prec<FP64>::S;
  const int4 tb = tab[blockIdx.x];
  const size_t ge = (size_t)tb.y << gs, step = (size_t)tb.w * blockDim.x;
  const int G = 1 << gs, off = VW * ((int)threadIdx.x & (G - 1));
  DotAcc<V> nrm[2 * VW];
  for (size_t gi = ((size_t)tb.x << gs) + (size_t)tb.z * blockDim.x + threadIdx.x; gi < ge; gi += step) {
    const int i = site_of(H, (int)(gi >> gs));
    const size_t e = (size_t)i * R + off;
    if (phase == 3) {
      double2 a[VW], b[VW];
      V f[VW], x[VW];
      evo_ld<VW>(a, B.accp + e);
      evo_ld<VW>(b, B.accx + e);
#pragma unroll
      for (int w = 0; w < VW; ++w) {
        f[w] = from_d2<V>(a[w]);
        x[w] = from_d2<V>(b[w]);
        nrm[w].add_norm(f[w]);
        nrm[VW + w].add_norm(x[w]);
      }
      evo_st<VW>(B.p + e, f);
      evo_st<VW>(B.px + e, x);
      continue;
    }
    const EvoRow<Ell<FP64, CH>, KK> row(H, i);
    S dx[KK];
#pragma unroll
    for (int k = 0; k < KK; ++k) dx[k] = -__ldg(H.dx + (size_t)k * H.n + i);
    V uown[VW], zown[VW], u2[VW], z2[VW], u[VW], z[VW], un[KK][VW], zn[KK][VW];
    evo_ldg<VW>(uown, B.u1 + e);
    evo_ldg<VW>(zown, B.z1 + e);
    if (phase != 0) {
      evo_ld<VW>(u2, B.u2 + e);
      evo_ld<VW>(z2, B.z2 + e);
    }
    double2 a[VW], b[VW];
    if (t.on && t.acc_in) {
      evo_ld<VW>(a, B.accp + e);
      evo_ld<VW>(b, B.accx + e);
    }
#pragma unroll
    for (int k = 0; k < KK; ++k) {
      const size_t j = (size_t)row.idx[k] * R + off;
      evo_ldg<VW>(un[k], B.u1 + j);
      evo_ldg<VW>(zn[k], B.z1 + j);
    }
#pragma unroll
    for (int w = 0; w < VW; ++w) {
      if (phase == 0) {
        u2[w].x = u2[w].y = 0;
        z2[w] = u2[w];
        u[w] = z[w] = u2[w];
      } else {
        u[w] = cneg(u2[w]);
        z[w] = cneg(z2[w]);
      }
      u[w] = cmul_acc(u[w], row.dg, uown[w]);
#pragma unroll
      for (int k = 0; k < KK; ++k) {
        u[w] = cmul_acc(u[w], row.hv[k], un[k][w]);
        z[w] = cmul_acc(z[w], row.hv[k], cscale(un[k][w], dx[k]));
      }
      z[w] = cmul_acc(z[w], row.dg, zown[w]);
#pragma unroll
      for (int k = 0; k < KK; ++k) z[w] = cmul_acc(z[w], row.hv[k], zn[k][w]);
      if (phase == 0) {
        u[w] = cscale(u[w], (S)0.5);
        z[w] = cscale(z[w], (S)0.5);
        nrm[w].add_norm(uown[w]);
      }
    }
    if (phase != 2) {
      evo_st<VW>(B.uo + e, u);
      evo_st<VW>(B.zo + e, z);
    }
    if (t.on) {
      evo_accumulate<V, VW>(a, t, u2, uown, u, phase == 0);
      evo_accumulate<V, VW>(b, t, z2, zown, z, phase == 0);
      if (phase == 2) {
        V f[VW], x[VW];
#pragma unroll
        for (int w = 0; w < VW; ++w) {
          f[w] = from_d2<V>(a[w]);
          x[w] = from_d2<V>(b[w]);
          nrm[w].add_norm(f[w]);
          nrm[VW + w].add_norm(x[w]);
        }
        evo_st<VW>(B.p + e, f);
        evo_st<VW>(B.px + e, x);
      } else {
        evo_st<VW>(B.accp + e, a);
        evo_st<VW>(B.accx + e, b);
      }
    }
  }
  if (phase != 1) {
    double2 v[2 * VW];
#pragma unroll
    for (int q = 0; q < 2 * VW; ++q) v[q] = nrm[q].get();
    evo_norms<2, VW>(v, R, G, partial, nblocks, slot);
  }
}

}  // namespace gqt

// ====================================================================== loops over orders

namespace {

// Evolution orders of FP64 handles with one vector run on the FP32 pipes (pairs of
// FP32 numbers, gqt_df.cuh) when their moment rows do (FP64 arithmetic mode 1): the
// wavefront table and neighbour counts of the pair rows.
bool df_evo_applies(const gqt_ham* h, int R) {
  return h->prec == GQT_FP64 && h->fp64_arith == 1 && R == 1 && h->variant != 0 && h->threads <= 256 &&
         (h->K == 2 || h->K == 3 || h->K == 4 || h->K == 6) && h->d_dx.p != nullptr;
}

// The wavefront kernels in storage precision: the same neighbour counts and table, and
// at most 256 threads (the register bound they are compiled for).
bool wave_evo_applies(const gqt_ham* h) {
  return h->variant != 0 && h->threads <= 256 && (h->K == 2 || h->K == 3 || h->K == 4 || h->K == 6);
}

template <class F>
void with_K(int K, F&& f) {
  switch (K) {
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    default: f(std::integral_constant<int, 6>()); break;
  }
}

template <class F>
void df_dispatch(const gqt_ham* h, F&& f) {
  with_K(h->K, [&](auto kk) {
    if (h->hop_real)
      f(std::integral_constant<bool, false>(), kk);
    else
      f(std::integral_constant<bool, true>(), kk);
  });
}

int occupancy_of(const void* f, int threads, size_t smem) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 4;
  }
  return std::max(1, n);
}

// The non-zero part of coefficient m (real at even m, imaginary at odd m).
double coef_part(const std::vector<double2>& c, int m) { return (m & 1) ? c[m].y : c[m].x; }
void put_coef(float2& d, double v) {
  d.x = (float)v;
  d.y = (float)(v - (double)d.x);
}
void put_coef(double& d, double v) { d = v; }

// Terms of order m >= 1 of an expansion of Np orders.  The last order adds its terms,
// and so does every third one before it, down to the first of these, m0 = 2, 3 or 4; the
// terms below T_{m0-2} are added at order 1 (T_0 for m0 = 3, T_0 and T_1 for m0 = 4, and
// for expansions that end there).
template <class C>
EvoTerms<C> terms_of(const std::vector<double2>& c, int m) {
  const int Np = (int)c.size(), last = Np - 1;
  EvoTerms<C> t = {};
  t.odd = m & 1;
  auto put = [&](int j, int q) { put_coef(t.c[j], q < Np ? coef_part(c, q) : 0.0); };
  const int m0 = last >= 2 ? 2 + (last - 2) % 3 : 0;
  if (m == 1) {
    t.on = last < 2 || m0 > 2;
    put(1, 0);
    if (last < 2 || m0 == 4) put(2, 1);
  } else if ((last - m) % 3 == 0) {
    t.on = 1;
    t.acc_in = m > m0 || m0 > 2;
    for (int j = 0; j < 3; ++j) put(j, m - 2 + j);
  }
  return t;
}

template <int NSET>
void launch_evolve_df(gqt_ham* h, void* const* psi, const std::vector<double2>& c, cudaStream_t st, double* d_norms) {
  ensure_df(h, st);
  const int Np = (int)c.size();
  const size_t smem = (size_t)NSET * (h->threads / 32) * sizeof(double) + 16;
  int occ = h->blocks_per_sm;
  if (occ <= 0)
    df_dispatch(h, [&](auto ch, auto kk) {
      occ = occupancy_of((const void*)k_evolve_df<decltype(ch)::value, decltype(kk)::value, NSET, 1>, h->threads,
                         smem);
    });
  const BlockTable& T = h->table(1, occ);
  const int nb = T.nblocks;
  const size_t vb = h->vec_bytes(1);
  float4* W1[NSET];
  float4* W2[NSET];
  float4* ACC[NSET];
  for (int q = 0; q < NSET; ++q) {
    W1[q] = (float4*)h->ws(WS_E1 + 2 * q, vb).p;
    W2[q] = (float4*)h->ws(WS_E1 + 2 * q + 1, vb).p;
    ACC[q] = (float4*)h->ws(WS_ACC0 + q, vb).p;
  }
  double2* partial = (double2*)h->ws(WS_PARTIAL_EVO, (size_t)(2 * NSET) * nb * sizeof(double2)).p;
  const std::string key = key_of("evodf", {psi[0], psi[NSET - 1], W1[0], W2[0], ACC[0], partial, d_norms, T.d_blk.p},
                                 {(double)NSET, (double)Np, (double)h->threads, (double)nb}) + coef_bits(c);
  run_graph(h, key, st, [&](cudaStream_t s2) {
    launch_split<NSET>(psi, W2, (size_t)h->n, s2);
    df_dispatch(h, [&](auto ch, auto kk) {
      constexpr bool CH = decltype(ch)::value;
      constexpr int KK = decltype(kk)::value;
      const DfEll<CH> H = df_ell_of<CH>(h);
      const int4* tab = (const int4*)T.d_tab4.p;
      DfEvo<NSET> A;
      for (int q = 0; q < NSET; ++q) {
        A.psi[q] = (double2*)psi[q];
        A.t1[q] = W2[q];
        A.t2[q] = nullptr;
        A.out[q] = W1[q];
        A.acc[q] = ACC[q];
      }
      auto orders = [&](auto uh) {
        constexpr bool UH = decltype(uh)::value && !CH;  // one common hopping: no hop array read
        k_evolve_df<CH, KK, NSET, 0, UH><<<nb, h->threads, smem, s2>>>(H, tab, A, terms_of<float2>(c, 1), partial, nb,
                                                                       0);
        check_launch("k_evolve_df(0)");
        if (Np <= 2) {
          k_evolve_df<CH, KK, NSET, 3, UH><<<nb, h->threads, smem, s2>>>(H, tab, A, EvoTerms<float2>{}, partial, nb,
                                                                         NSET);
          check_launch("k_evolve_df(3)");
          return;
        }
        for (int m = 2; m < Np; ++m) {
          for (int q = 0; q < NSET; ++q) {
            A.t1[q] = (m - 1) % 2 == 1 ? W1[q] : W2[q];
            A.out[q] = (m % 2 == 1) ? W1[q] : W2[q];
            A.t2[q] = A.out[q];
          }
          size_t pe = prof_begin(s2);
          if (m == Np - 1)
            launch_chain(true, k_evolve_df<CH, KK, NSET, 2, UH>, nb, h->threads, smem, s2, H, tab, A, terms_of<float2>(c, m), partial,
                                                                           nb, NSET);
          else
            launch_chain(true, k_evolve_df<CH, KK, NSET, 1, UH>, nb, h->threads, smem, s2, H, tab, A, terms_of<float2>(c, m), partial,
                                                                           nb, NSET);
          check_launch("k_evolve_df");
          prof_end(pe, 1 + NSET, s2);
        }
      };
      if (h->hop_uniform)
        orders(std::true_type());
      else
        orders(std::false_type());
    });
    launch_slot_sums(partial, nb, 1, (const int*)T.d_seg_blk.p, h->nseg, 0, 2 * NSET, -1, s2);
    k_norm_check<<<1, 256, 0, s2>>>(partial, NSET, nb, 1, (const int*)T.d_seg_blk.p, h->nseg, 1e-10, d_norms,
                                    (int*)h->d_flag.p);
    check_launch("k_norm_check");
  });
}

void launch_msd_df(gqt_ham* h, void* p, void* px, const std::vector<double2>& c, cudaStream_t st) {
  ensure_df(h, st);
  ensure_df_x(h, st);
  const int Np = (int)c.size();
  const size_t smem = (size_t)2 * (h->threads / 32) * sizeof(double) + 16;
  int occ = h->blocks_per_sm;
  if (occ <= 0)
    df_dispatch(h, [&](auto ch, auto kk) {
      occ = occupancy_of((const void*)k_msd_evolve_df<decltype(ch)::value, decltype(kk)::value, 1>, h->threads, smem);
    });
  const BlockTable& T = h->table(1, occ);
  const int nb = T.nblocks;
  const size_t vb = h->vec_bytes(1);
  float4* U1 = (float4*)h->ws(WS_E1, vb).p;
  float4* U2 = (float4*)h->ws(WS_E1 + 1, vb).p;
  float4* Z1 = (float4*)h->ws(WS_E1 + 2, vb).p;
  float4* Z2 = (float4*)h->ws(WS_E1 + 3, vb).p;
  float4* AP = (float4*)h->ws(WS_ACC0, vb).p;
  float4* AX = (float4*)h->ws(WS_ACC0 + 1, vb).p;
  double2* partial = (double2*)h->ws(WS_PARTIAL_EVO, (size_t)4 * nb * sizeof(double2)).p;
  const std::string key = key_of("msddf", {p, px, U1, Z1, AP, AX, partial, T.d_blk.p},
                                 {(double)Np, (double)h->threads, (double)nb}) + coef_bits(c);
  run_graph(h, key, st, [&](cudaStream_t s2) {
    void* in[2] = {p, px};
    float4* t0[2] = {U2, Z2};
    launch_split<2>(in, t0, (size_t)h->n, s2);
    df_dispatch(h, [&](auto ch, auto kk) {
      constexpr bool CH = decltype(ch)::value;
      constexpr int KK = decltype(kk)::value;
      const DfEll<CH> H = df_ell_of<CH>(h);
      const int4* tab = (const int4*)T.d_tab4.p;
      DfMsd B;
      B.p = (double2*)p;
      B.px = (double2*)px;
      B.u1 = U2;
      B.z1 = Z2;
      B.u2 = B.z2 = nullptr;
      B.uo = U1;
      B.zo = Z1;
      B.accp = AP;
      B.accx = AX;
      auto orders = [&](auto uh) {
        constexpr bool UH = decltype(uh)::value && !CH;  // one common hopping: no hop array read
        k_msd_evolve_df<CH, KK, 0, UH><<<nb, h->threads, smem, s2>>>(H, tab, B, terms_of<float2>(c, 1), partial, nb, 0);
        check_launch("k_msd_evolve_df(0)");
        if (Np <= 2) {
          k_msd_evolve_df<CH, KK, 3, UH><<<nb, h->threads, smem, s2>>>(H, tab, B, EvoTerms<float2>{}, partial, nb, 2);
          check_launch("k_msd_evolve_df(3)");
          return;
        }
        for (int m = 2; m < Np; ++m) {
          B.u1 = (m - 1) % 2 == 1 ? U1 : U2;
          B.z1 = (m - 1) % 2 == 1 ? Z1 : Z2;
          B.uo = (m % 2 == 1) ? U1 : U2;
          B.zo = (m % 2 == 1) ? Z1 : Z2;
          B.u2 = B.uo;
          B.z2 = B.zo;
          size_t pe = prof_begin(s2);
          if (m == Np - 1)
            launch_chain(true, k_msd_evolve_df<CH, KK, 2, UH>, nb, h->threads, smem, s2, H, tab, B, terms_of<float2>(c, m), partial,
                                                                         nb, 2);
          else
            launch_chain(true, k_msd_evolve_df<CH, KK, 1, UH>, nb, h->threads, smem, s2, H, tab, B, terms_of<float2>(c, m), partial,
                                                                         nb, 2);
          check_launch("k_msd_evolve_df");
          prof_end(pe, 4, s2);
        }
      };
      if (h->hop_uniform)
        orders(std::true_type());
      else
        orders(std::false_type());
    });
    launch_slot_sums(partial, nb, 1, (const int*)T.d_seg_blk.p, h->nseg, 0, 4, -1, s2);
    k_norm_check_msd<<<1, 256, 0, s2>>>(partial, nb, 1, (const int*)T.d_seg_blk.p, h->nseg, 1e-10,
                                        (int*)h->d_flag.p);
    check_launch("k_norm_check_msd");
  });
}

// Coefficients of an expansion that fits the cluster kernels' argument.
ClusterCoefs cluster_coefs(const std::vector<double2>& c) {
  ClusterCoefs k = {};
  k.n = (int)c.size();
  for (int m = 0; m < k.n; ++m) k.c[m] = coef_part(c, m);
  return k;
}

// Small systems: every order of an evolution (or of an MSD time step) in one launch on a
// thread-block cluster, for FP64 handles with one vector and one segment, expansions of up to CL_ORDERS
// orders and systems of up to 512 sites per CTA, where cluster rows are on.
bool cluster_evo_applies(const gqt_ham* h, int R, int Np) {
  return h->use_cluster && h->prec == GQT_FP64 && R == 1 && h->nseg == 1 && Np <= CL_ORDERS &&
         (h->K == 2 || h->K == 3 || h->K == 4 || h->K == 6) && h->n <= 16 * 512;
}

template <int NSET>
bool launch_evolve_cluster(gqt_ham* h, void* const* psi, const std::vector<double2>& c, cudaStream_t st,
                           double* d_norms) {
  if (!cluster_evo_applies(h, 1, (int)c.size())) return false;
  const ClusterCoefs co = cluster_coefs(c);
  bool done = false;
  df_dispatch(h, [&](auto ch, auto kk) {
    constexpr bool CH = decltype(ch)::value;
    auto kern = k_evolve_cluster<CH, NSET, decltype(kk)::value>;
    ClusterSets<NSET> A;
    for (int q = 0; q < NSET; ++q) A.psi[q] = (double2*)psi[q];
    done = cluster1_launch(
        kern, h->n, st,
        [](int chunk, int) { return (size_t)2 * NSET * chunk * sizeof(double2) + 18 * 2 * NSET * sizeof(double); },
        [&](const cudaLaunchConfig_t& cfg, int chunk) {
          check_cuda(cudaLaunchKernelEx(&cfg, kern, ell_of<true, CH>(h), chunk, A, co, 1e-10, d_norms,
                                        (int*)h->d_flag.p),
                     "k_evolve_cluster");
          check_launch("k_evolve_cluster");
        });
  });
  return done;
}

bool launch_msd_cluster(gqt_ham* h, void* p, void* px, const std::vector<double2>& c, cudaStream_t st) {
  if (!cluster_evo_applies(h, 1, (int)c.size())) return false;
  const ClusterCoefs co = cluster_coefs(c);
  bool done = false;
  df_dispatch(h, [&](auto ch, auto kk) {
    constexpr bool CH = decltype(ch)::value;
    auto kern = k_msd_cluster<CH, decltype(kk)::value>;
    done = cluster1_launch(
        kern, h->n, st, [](int chunk, int) { return (size_t)4 * chunk * sizeof(double2) + 18 * 3 * sizeof(double); },
        [&](const cudaLaunchConfig_t& cfg, int chunk) {
          check_cuda(cudaLaunchKernelEx(&cfg, kern, ell_of<true, CH>(h), chunk, (double2*)p, (double2*)px, co, 1e-10,
                                        (int*)h->d_flag.p),
                     "k_msd_cluster");
          check_launch("k_msd_cluster");
        });
  });
  return done;
}

// Grid of a storage-precision wavefront kernel: its resident CTAs.
template <class K>
int wave_grid(const gqt_ham* h, K kern, size_t smem) {
  if (h->blocks_per_sm > 0) return h->blocks_per_sm;
  return std::min(16, occupancy_of((const void*)kern, h->threads, smem));
}

// Vectors per lane: two FP32 ones (one 16-byte load) for R >= 2, where the caller's
// vectors are 16-byte aligned.
template <class F>
void with_width(const gqt_ham* h, int R, bool aligned, F&& f) {
  dispatch(h, [&](auto H) {
    using Tr = EllTraits<decltype(H)>;
    if constexpr (!Tr::fp64) {
      if (R >= 2 && aligned) {
        f(H, std::integral_constant<int, 2>());
        return;
      }
    }
    f(H, std::integral_constant<int, 1>());
  });
}

}  // namespace

template <int NSET>
void gqt::launch_evolve_sets(gqt_ham* h, void* const* psi, int R, const std::vector<double2>& c, cudaStream_t st,
                             double* d_norms) {
  if (R == 1 && launch_evolve_cluster<NSET>(h, psi, c, st, d_norms)) return;
  if (df_evo_applies(h, R)) {
    launch_evolve_df<NSET>(h, psi, c, st, d_norms);
    return;
  }
  const int Np = (int)c.size();
  const bool wave = wave_evo_applies(h);
  bool aligned = true;
  for (int q = 0; q < NSET; ++q) aligned = aligned && (uintptr_t)psi[q] % 16 == 0;
  const size_t smem = smem_bytes(h, R, 4);
  int occ = 0;
  if (wave)
    with_width(h, R, aligned, [&](auto H, auto vw) {
      using Tr = EllTraits<decltype(H)>;
      with_K(h->K, [&](auto kk) {
        occ = wave_grid(h, k_evolve_w<NSET, Tr::fp64, Tr::ch, decltype(vw)::value, decltype(kk)::value>, smem);
      });
    });
  const BlockTable& T = h->table(R, occ);
  const int nb = T.nblocks, rs = rshift_of(R);
  const size_t vb = h->vec_bytes(R);
  void* W1[NSET];
  void* W2[NSET];
  double2* ACC[NSET];
  for (int q = 0; q < NSET; ++q) {
    W1[q] = h->ws(WS_E1 + 2 * q, vb).p;
    W2[q] = h->ws(WS_E1 + 2 * q + 1, vb).p;
    ACC[q] = (double2*)h->ws(WS_ACC0 + q, (size_t)h->n * R * sizeof(double2)).p;
  }
  double2* partial = (double2*)h->ws(WS_PARTIAL_EVO, (size_t)(2 * NSET) * nb * R * sizeof(double2)).p;
  const std::string key = key_of("evo", {psi[0], psi[NSET - 1], W1[0], W2[0], ACC[0], partial, d_norms, T.d_blk.p},
                                 {(double)NSET, (double)R, (double)Np, (double)h->threads, (double)wave, (double)nb}) +
                          coef_bits(c);
  run_graph(h, key, st, [&](cudaStream_t s2) {
    with_width(h, R, aligned, [&](auto H, auto vw) {
      using Tr = EllTraits<decltype(H)>;
      using V = typename Tr::V;
      constexpr int VW = decltype(vw)::value;
      EvoSets<NSET, Tr::fp64> A;
      for (int q = 0; q < NSET; ++q) {
        A.t1[q] = (const V*)psi[q];
        A.t2[q] = nullptr;
        A.out[q] = (V*)W1[q];
        A.acc[q] = ACC[q];
        A.fin[q] = (V*)psi[q];
      }
      // one launch: order m (phases 0, 1, 2), or the finish (phase 3)
      auto order = [&](int m, int phase, int slot) {
        if (wave) {
          const EvoTerms<double> t = phase == 3 ? EvoTerms<double>{} : terms_of<double>(c, m);
          with_K(h->K, [&](auto kk) {
            k_evolve_w<NSET, Tr::fp64, Tr::ch, VW, decltype(kk)::value><<<nb, h->threads, smem, s2>>>(
                H, (const int4*)T.d_tab4.p, R, rs - (VW - 1), A, t, phase, partial, nb, slot);
          });
        } else if constexpr (VW == 1 || !Tr::fp64) {
          const double2 zero = make_double2(0.0, 0.0);
          const double2 c0 = phase == 0 ? c[0] : (phase == 3 ? zero : c[m]);
          k_evolve<NSET, Tr::fp64, Tr::ch><<<nb, h->threads, smem, s2>>>(H, (const int*)T.d_blk.p, R, rs, A, c0,
                                                                         phase == 0 && Np > 1 ? c[1] : zero, phase,
                                                                         partial, nb, slot);
        }
        check_launch("k_evolve");
      };
      order(1, 0, 0);
      if (Np <= 2) {
        order(0, 3, NSET);
        return;
      }
      for (int m = 2; m < Np; ++m) {
        for (int q = 0; q < NSET; ++q) {
          V* w1 = (V*)W1[q];
          V* w2 = (V*)W2[q];
          A.t1[q] = (m - 1) % 2 == 1 ? w1 : w2;
          V* o = (m % 2 == 1) ? w1 : w2;
          A.t2[q] = (m == 2) ? (const V*)psi[q] : o;
          A.out[q] = o;
        }
        const size_t pe = prof_begin(s2);
        order(m, m == Np - 1 ? 2 : 1, NSET);
        prof_end(pe, 1 + NSET, s2);
      }
    });
    const double tol = h->prec == GQT_FP64 ? 1e-10 : 1e-5;
    launch_slot_sums(partial, nb, R, (const int*)T.d_seg_blk.p, h->nseg, 0, 2 * NSET, -1, s2);
    k_norm_check<<<1, 256, 0, s2>>>(partial, NSET, nb, R, (const int*)T.d_seg_blk.p, h->nseg, tol, d_norms,
                                    (int*)h->d_flag.p);
    check_launch("k_norm_check");
  });
}

template void gqt::launch_evolve_sets<1>(gqt_ham*, void* const*, int, const std::vector<double2>&, cudaStream_t,
                                         double*);
template void gqt::launch_evolve_sets<2>(gqt_ham*, void* const*, int, const std::vector<double2>&, cudaStream_t,
                                         double*);

void gqt::launch_msd_step(gqt_ham* h, void* p, void* px, int R, const std::vector<double2>& c, cudaStream_t st) {
  if (R == 1 && launch_msd_cluster(h, p, px, c, st)) return;
  if (df_evo_applies(h, R)) {
    launch_msd_df(h, p, px, c, st);
    return;
  }
  const int Np = (int)c.size();
  const bool wave = wave_evo_applies(h);
  const bool aligned = ((uintptr_t)p | (uintptr_t)px) % 16 == 0;
  const size_t smem = smem_bytes(h, R, 4);
  int occ = 0;
  if (wave)
    with_width(h, R, aligned, [&](auto H, auto vw) {
      using Tr = EllTraits<decltype(H)>;
      with_K(h->K, [&](auto kk) {
        occ = wave_grid(h, k_msd_evolve_w<Tr::fp64, Tr::ch, decltype(vw)::value, decltype(kk)::value>, smem);
      });
    });
  const BlockTable& T = h->table(R, occ);
  const int nb = T.nblocks, rs = rshift_of(R);
  const size_t vb = h->vec_bytes(R);
  void* U1 = h->ws(WS_E1, vb).p;
  void* U2 = h->ws(WS_E1 + 1, vb).p;
  void* Z1 = h->ws(WS_E1 + 2, vb).p;
  void* Z2 = h->ws(WS_E1 + 3, vb).p;
  double2* AP = (double2*)h->ws(WS_ACC0, (size_t)h->n * R * sizeof(double2)).p;
  double2* AX = (double2*)h->ws(WS_ACC0 + 1, (size_t)h->n * R * sizeof(double2)).p;
  double2* partial = (double2*)h->ws(WS_PARTIAL_EVO, (size_t)4 * nb * R * sizeof(double2)).p;
  const std::string key = key_of("msd", {p, px, U1, Z1, AP, AX, partial, T.d_blk.p},
                                 {(double)R, (double)Np, (double)h->threads, (double)wave, (double)nb}) + coef_bits(c);
  run_graph(h, key, st, [&](cudaStream_t s2) {
    with_width(h, R, aligned, [&](auto H, auto vw) {
      using Tr = EllTraits<decltype(H)>;
      using V = typename Tr::V;
      constexpr int VW = decltype(vw)::value;
      MsdBufs<Tr::fp64> B;
      B.u1 = (const V*)p;
      B.z1 = (const V*)px;
      B.u2 = nullptr;
      B.z2 = nullptr;
      B.uo = (V*)U1;
      B.zo = (V*)Z1;
      B.accp = AP;
      B.accx = AX;
      B.p = (V*)p;
      B.px = (V*)px;
      auto order = [&](int m, int phase, int slot) {
        if (wave) {
          const EvoTerms<double> t = phase == 3 ? EvoTerms<double>{} : terms_of<double>(c, m);
          with_K(h->K, [&](auto kk) {
            k_msd_evolve_w<Tr::fp64, Tr::ch, VW, decltype(kk)::value><<<nb, h->threads, smem, s2>>>(
                H, (const int4*)T.d_tab4.p, R, rs - (VW - 1), B, t, phase, partial, nb, slot);
          });
        } else {
          const double2 zero = make_double2(0.0, 0.0);
          const double2 c0 = phase == 0 ? c[0] : (phase == 3 ? zero : c[m]);
          k_msd_evolve<Tr::fp64, Tr::ch><<<nb, h->threads, smem, s2>>>(H, (const int*)T.d_blk.p, R, rs, B, c0,
                                                                       phase == 0 && Np > 1 ? c[1] : zero, phase,
                                                                       partial, nb, slot);
        }
        check_launch("k_msd_evolve");
      };
      order(1, 0, 0);
      if (Np <= 2) {
        order(0, 3, 2);
        return;
      }
      for (int m = 2; m < Np; ++m) {
        B.u1 = (m - 1) % 2 == 1 ? (const V*)U1 : (const V*)U2;
        B.z1 = (m - 1) % 2 == 1 ? (const V*)Z1 : (const V*)Z2;
        V* uo = (m % 2 == 1) ? (V*)U1 : (V*)U2;
        V* zo = (m % 2 == 1) ? (V*)Z1 : (V*)Z2;
        B.u2 = (m == 2) ? (const V*)p : uo;
        B.z2 = (m == 2) ? (const V*)px : zo;
        B.uo = uo;
        B.zo = zo;
        const size_t pe = prof_begin(s2);
        order(m, m == Np - 1 ? 2 : 1, 2);
        prof_end(pe, 4, s2);
      }
    });
    // only |U p| vs |p| is a unitarity check; the px norm changes by construction.
    const double tol = h->prec == GQT_FP64 ? 1e-10 : 1e-5;
    launch_slot_sums(partial, nb, R, (const int*)T.d_seg_blk.p, h->nseg, 0, 4, -1, s2);
    k_norm_check_msd<<<1, 256, 0, s2>>>(partial, nb, R, (const int*)T.d_seg_blk.p, h->nseg, tol, (int*)h->d_flag.p);
    check_launch("k_norm_check_msd");
  });
}
