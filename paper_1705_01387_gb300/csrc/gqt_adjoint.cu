// gqt_adjoint.cu -- reverse-mode gradients of VAC-moment losses: the adjoint of the
// Chebyshev recursion, its kernels and gqt_vac_loss_grad.

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <type_traits>
#include <vector>

#include "gqt_host.cuh"

using namespace gqt;

namespace gqt {

// ------------------------------------------------------------ K9: adjoint
//
// Reverse-mode derivative of J = Re sum_{m<P} coef_m <lam| T_m(H~) |r> with
// u_m = T_m r (not in the paper; it differentiates Eqs. 17, 21 and 29).  The
// adjoint vectors obey the transposed recurrence
//   w_m = conj(coef_m) lam + 2 H~ w_{m+1} - w_{m+2},   w_P = w_{P+1} = 0,
// and dJ = Re sum_ij conj(G_ij) dH~_ij with G = w_1 u_0^+ + 2 sum_{m>=2} w_m u_{m-1}^+,
// needed only on the diagonal and the ELL slots.

// The H~ row of site i, unrolled for the neighbour counts KK = 2, 3, 4, 6; KK = 0 reads
// it slot by slot.
template <class E, int KK>
struct AdjRow {
  int idx[KK > 0 ? KK : 1];
  typename E::HT hv[KK > 0 ? KK : 1];
  typename E::S dg;
  __device__ __forceinline__ AdjRow(const E& H, int i) {
#pragma unroll
    for (int k = 0; k < KK; ++k) {
      const size_t s = (size_t)k * H.n + i;
      idx[k] = __ldg(H.idx + s);
      hv[k] = __ldg(H.hop2 + s);
    }
    dg = __ldg(H.diag2 + i);
  }
  // acc + 2H~ x at the site, diagonal first, then the slots in order
  template <class V>
  __device__ __forceinline__ V apply(const E& H, int i, const V* __restrict__ x, V acc) const {
    V nb[KK > 0 ? KK : 1];
    const V own = __ldg(x + i);
#pragma unroll
    for (int k = 0; k < KK; ++k) nb[k] = __ldg(x + idx[k]);
    acc = cmul_acc(acc, dg, own);
#pragma unroll
    for (int k = 0; k < KK; ++k) acc = cmul_acc(acc, hv[k], nb[k]);
    if (KK == 0)
      for (int k = 0; k < H.K; ++k) {
        const size_t s = (size_t)k * H.n + i;
        acc = cmul_acc(acc, __ldg(H.hop2 + s), __ldg(x + __ldg(H.idx + s)));
      }
    return acc;
  }
};

__device__ __forceinline__ double2 widen(float2 a) { return make_double2(f2d(a.x), f2d(a.y)); }
__device__ __forceinline__ double2 widen(double2 a) { return a; }

// acc += c x (im = 0) or i c x: the coefficients of the moment rows are real, those of
// the evolution real at even and imaginary at odd orders, so a term costs two FP64
// multiply-adds instead of four.
template <class V>
__device__ __forceinline__ void adj_term(double2& acc, double c, int im, V xv) {
  V u;  // the operands are chosen, not the operations (see evo_term)
  u.x = im ? xv.y : xv.x;
  u.y = im ? xv.x : xv.y;
  const double2 x = widen(u);
  acc.x = fma(im ? -c : c, x.x, acc.x);
  acc.y = fma(c, x.y, acc.y);
}

// The terms of an accumulator that is touched every third order (as in the evolution):
// c[j] multiplies T_{m-2+j}, times i where bit j of im is set.
struct AdjTerms {
  double c[3];
  int im, on, acc_in;
};

// Order m of the forward recursion, one site per thread: out = 2H~ t1 - t2 (first: out =
// H~ t1) and, where on, the accumulator's terms up to it.  t2 and out may be one buffer
// (each element is read and written by its thread only).  FP64 pipe bound (8 + 2
// multiply-adds per site), so the grid is as fine as the sites allow: 1024 CTAs of 128
// at 131,072 sites leave 4% of the SM time idle, 256 of 256 with two sites a thread 16%.
template <bool FP64, bool CH, int KK>
__global__ void __launch_bounds__(128) k_recur(Ell<FP64, CH> H, const typename Prec<FP64>::V* __restrict__ t1,
                                               const typename Prec<FP64>::V* t2, typename Prec<FP64>::V* out,
                                               double2* __restrict__ acc, AdjTerms t, int first) {
  using V = typename Prec<FP64>::V;
  using S = typename Prec<FP64>::S;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= H.n) return;
  const AdjRow<Ell<FP64, CH>, KK> row(H, i);
  V tm2, y;
  tm2.x = tm2.y = 0;
  if (!first) tm2 = t2[i];
  y = row.apply(H, i, t1, first ? tm2 : cneg(tm2));
  if (first) y = cscale(y, (S)0.5);
  out[i] = y;
  if (t.on) {
    double2 a = t.acc_in ? acc[i] : make_double2(0.0, 0.0);
    if (!first) adj_term(a, t.c[0], t.im & 1, tm2);
    adj_term(a, t.c[1], t.im & 2, __ldg(t1 + i));
    adj_term(a, t.c[2], t.im & 4, y);
    acc[i] = a;
  }
}

// One adjoint order m: w_m = lc lam + 2H~ w1 - w2 (w1 = w_{m+1}, w2 = w_{m+2}, w_m
// overwrites w2; lc = c or i c) and G += f w_m conj(u_{m-1}) on the diagonal (gdiag,
// real part) and on the slots (gslot [K][n]).  f = (m == 1 ? 1 : 2) / dE.  f multiplies
// w_m once and the products are accumulated directly: 26 FP64 operations per site with
// three real slots (34 before), the kernel's bound.
template <bool FP64, bool CH, int KK>
__global__ void __launch_bounds__(128) k_adj_step(Ell<FP64, CH> H, const typename Prec<FP64>::V* __restrict__ w1,
                                                  typename Prec<FP64>::V* w2,
                                                  const typename Prec<FP64>::V* __restrict__ lam, double c, int im,
                                                  const typename Prec<FP64>::V* __restrict__ u, double f,
                                                  double* __restrict__ gdiag, double2* __restrict__ gslot) {
  using V = typename Prec<FP64>::V;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= H.n) return;
  const AdjRow<Ell<FP64, CH>, KK> row(H, i);
  const V lv = __ldg(lam + i), ui = __ldg(u + i);
  V un[KK > 0 ? KK : 1];
  double2 g[KK > 0 ? KK : 1];
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    un[k] = __ldg(u + row.idx[k]);
    g[k] = gslot[(size_t)k * H.n + i];
  }
  double gd = gdiag[i];
  double2 wd = widen(row.apply(H, i, w1, cneg(w2[i])));
  adj_term(wd, c, im, lv);
  const V w = from_d2<V>(wd);
  w2[i] = w;
  wd = widen(w);
  wd.x *= f;
  wd.y *= f;
  const double2 ud = widen(ui);
  gdiag[i] = fma(wd.x, ud.x, fma(wd.y, ud.y, gd));
  auto add = [&](double2& q, V uv) {  // q += f w conj(uv)
    const double2 x = widen(uv);
    q.x = fma(wd.x, x.x, fma(wd.y, x.y, q.x));
    q.y = fma(wd.y, x.x, fma(-wd.x, x.y, q.y));
  };
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    add(g[k], un[k]);
    gslot[(size_t)k * H.n + i] = g[k];
  }
  if (KK == 0)
    for (int k = 0; k < H.K; ++k) {
      const size_t s = (size_t)k * H.n + i;
      double2 q = gslot[s];
      add(q, __ldg(u + __ldg(H.idx + s)));
      gslot[s] = q;
    }
}

// rbar = lc0 lam + H~ w1 - w2 (Clenshaw end, = sum_m conj(coef_m) T_m lam); w1 may be null (P = 1).
template <bool FP64, bool CH>
__global__ void k_adj_final(Ell<FP64, CH> H, const int* __restrict__ blk, const typename Prec<FP64>::V* __restrict__ w1,
                            const typename Prec<FP64>::V* __restrict__ w2, const typename Prec<FP64>::V* __restrict__ lam,
                            double2 lc0, typename Prec<FP64>::V* __restrict__ rbar) {
  using V = typename Prec<FP64>::V;
  using S = typename Prec<FP64>::S;
  const int b = blockIdx.x;
  for (int i = blk[b] + threadIdx.x; i < blk[b + 1]; i += blockDim.x) {
    double2 acc = cfma_d(make_double2(0.0, 0.0), lc0, __ldg(lam + i));
    if (w1) {
      V zero;
      zero.x = 0;
      zero.y = 0;
      V y = cscale(apply2h<FP64, CH>(H, w1, i, 0, 0, zero), (S)0.5);
      const double2 yd = to_d2(y), w2d = to_d2(__ldg(w2 + i));
      acc.x += yd.x - w2d.x;
      acc.y += yd.y - w2d.y;
    }
    rbar[i] = from_d2<V>(acc);
  }
}

__device__ __forceinline__ double2 hop_d(double2 h) { return h; }
__device__ __forceinline__ double2 hop_d(float2 h) { return to_d2(h); }
__device__ __forceinline__ double hop_d(double h) { return h; }
__device__ __forceinline__ double hop_d(float h) { return (double)h; }

// Velocity part of the gradient: l = V x with V_ij = i dx_ij H_ij (unscaled H), so
// G_ij += lbar_i (-i dx_ij) conj(x_j) (slots only; V has no diagonal).
template <bool FP64, bool CH, class LB>
__global__ void k_vel_adj(Ell<FP64, CH> H, const int* __restrict__ blk, const LB* __restrict__ lbar,
                          const typename Prec<FP64>::V* __restrict__ x, double2* __restrict__ gslot) {
  const int b = blockIdx.x;
  for (int i = blk[b] + threadIdx.x; i < blk[b + 1]; i += blockDim.x) {
    const double2 lb = to_d2(lbar[i]);
    for (int k = 0; k < H.K; ++k) {
      const size_t s = (size_t)k * H.n + i;
      const double2 xj = to_d2(__ldg(x + __ldg(H.idx + s)));
      const double d = (double)__ldg(H.dx + s);
      // lbar * (-i d) * conj(xj) = -i d (lb.x + i lb.y)(xj.x - i xj.y)
      const double re = lb.x * xj.x + lb.y * xj.y, im = lb.y * xj.x - lb.x * xj.y;
      double2 g = gslot[s];
      g.x += d * im;
      g.y += -d * re;
      gslot[s] = g;
    }
  }
}

// y += V x for a double2 accumulator y (x storage precision), V = i dE sum dx H~.
template <bool FP64, bool CH>
__global__ void k_vel_acc(Ell<FP64, CH> H, const int* __restrict__ blk, double half_dE,
                          const double2* __restrict__ x, typename Prec<FP64>::V* __restrict__ y) {
  using V = typename Prec<FP64>::V;
  const int b = blockIdx.x;
  for (int i = blk[b] + threadIdx.x; i < blk[b + 1]; i += blockDim.x) {
    double2 a = make_double2(0.0, 0.0);
    for (int k = 0; k < H.K; ++k) {
      const size_t s = (size_t)k * H.n + i;
      const int j = __ldg(H.idx + s);
      const double d = (double)__ldg(H.dx + s);
      a = cmul_acc(a, hop_d(__ldg(H.hop2 + s)), cscale(x[j], d));
    }
    double2 yo = to_d2(y[i]);
    yo.x += -a.y * half_dE;
    yo.y += a.x * half_dE;
    y[i] = from_d2<V>(yo);
  }
}

// Re <l|x> partial sums per CTA (x double2).
template <class V>
__global__ void k_dot_re(const int* __restrict__ blk, const V* __restrict__ l, const double2* __restrict__ x,
                         double* __restrict__ partial) {
  __shared__ double sh[32];
  const int b = blockIdx.x;
  double s = 0.0;
  for (int i = blk[b] + threadIdx.x; i < blk[b + 1]; i += blockDim.x) {
    const double2 lv = to_d2(l[i]);
    const double2 xv = x[i];
    s += lv.x * xv.x + lv.y * xv.y;
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    partial[b] = t;
  }
}

// y += x (storage precision).
template <class V>
__global__ void k_axpy(const int* __restrict__ blk, V* __restrict__ y, const V* __restrict__ x) {
  const int b = blockIdx.x;
  for (int i = blk[b] + threadIdx.x; i < blk[b + 1]; i += blockDim.x) {
    V a = y[i];
    const V c = x[i];
    a.x += c.x;
    a.y += c.y;
    y[i] = a;
  }
}

// Slot-major [K][n] double2 -> row-major [n][K] double2; diagonal copied.
static __global__ void k_grad_out(int n, int K, const double2* __restrict__ gslot, const double* __restrict__ gdiag,
                           double2* __restrict__ out_slot, double* __restrict__ out_diag) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < (size_t)n * K; t += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(t / K), k = (int)(t % K);
    out_slot[t] = gslot[(size_t)k * n + i];
    if (k == 0) out_diag[i] = gdiag[i];
  }
}

}  // namespace gqt

namespace {

template <class F>
void with_K(int K, F&& f) {
  switch (K) {
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    default: f(std::integral_constant<int, 0>()); break;
  }
}

// Bytes of forward vectors a gradient call may keep instead of recomputing them.
constexpr size_t ADJ_KEEP = (size_t)4 << 30;

// The part of a coefficient that is not zero, and whether it is the imaginary one (the
// moment weights are real, the evolution coefficients real or imaginary).
double part_of(double2 c, int& im) {
  im = c.x == 0.0 && c.y != 0.0;
  return im ? c.y : c.x;
}

// Adds to (gdiag, gslot) the gradient of J = Re sum_{m<P} coef_m <lam|T_m(H~)|r>
// (coefficients real or imaginary) and writes rbar = sum_m conj(coef_m) T_m lam (dJ = Re
// <rbar|dr>).  If lbar is non-null it receives sum_m coef_m T_m r (FP64).  The u_m = T_m r
// of the forward pass are kept (stride >= P) or recomputed from checkpoint pairs (u_c,
// u_{c+1}) taken every `stride` orders.
template <class HT>
void poly_adjoint(gqt_ham* h, const HT& H, const void* r, const void* lam, const std::vector<double2>& coef,
                  int stride, void* rbar, double2* lbar, double* gdiag, double2* gslot, cudaStream_t st) {
  using Tr = EllTraits<HT>;
  using V = typename Tr::V;
  const int P = (int)coef.size(), last = P - 1;
  const BlockTable& T = h->table(1);
  const int nb = T.nblocks;
  const int* blk = (const int*)T.d_blk.p;
  const size_t vb = h->vec_bytes(1);
  const int s = std::max(2, std::min(stride, std::max(P, 2)));
  const bool keep = s >= P;  // u_m, m < P, all stay in seg
  const int nck = (P + s - 1) / s;
  char* ck = keep ? nullptr : (char*)h->ws(WS_ADJ0, (size_t)2 * nck * vb).p;
  char* seg = (char*)h->ws(WS_ADJ0 + 1, (size_t)s * vb).p;
  V* WA = (V*)h->ws(WS_ADJ0 + 2, vb).p;
  V* WB = (V*)h->ws(WS_ADJ0 + 3, vb).p;
  auto ckp = [&](int j, int q) { return (V*)(ck + ((size_t)2 * j + q) * vb); };
  auto kept = [&](int m) { return (V*)(seg + (size_t)m * vb); };
  const int thr = h->threads, grid = (int)((h->n + 127) / 128);
  std::vector<double> cdata(2 * coef.size());
  for (size_t q = 0; q < coef.size(); ++q) {
    cdata[2 * q] = coef[q].x;
    cdata[2 * q + 1] = coef[q].y;
  }
  // lbar's terms at order m >= 1: the last order and every third one before it, down to
  // m0 = 2, 3 or 4; the orders below m0 - 2 (all, for P <= 2) at m = 1
  const int m0 = last >= 2 ? 2 + (last - 2) % 3 : 0;
  auto terms = [&](int m) {
    AdjTerms t = {};
    if (!lbar) return t;
    auto put = [&](int j, int q) {
      int im = 0;
      t.c[j] = q < P ? part_of(coef[q], im) : 0.0;
      t.im |= im << j;
    };
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
  };
  const std::string key = key_of("padj", {r, lam, rbar, lbar, gdiag, gslot, ck, seg, WA, WB, blk},
                                 {(double)P, (double)s, (double)thr});
  run_graph(h, key, st, [&](cudaStream_t s2) {
    with_K(h->K, [&](auto kk) {
      constexpr int KK = decltype(kk)::value;
      auto recur = [&](const V* t1, const V* t2, V* out, const AdjTerms& t) {
        k_recur<Tr::fp64, Tr::ch, KK><<<grid, 128, 0, s2>>>(H, t1, t2, out, lbar, t, t2 == nullptr);
        check_launch("k_recur");
      };
      auto copy = [&](V* d, const void* src) {
        check_cuda(cudaMemcpyAsync(d, src, vb, cudaMemcpyDeviceToDevice, s2), "checkpoint");
      };
      // forward pass: u_m kept, or checkpoints; and lbar
      const V* rv = (const V*)r;
      if (keep) {
        if (P > 1 || lbar) recur(rv, nullptr, kept(1), terms(1));
        for (int m = 2; m < P; ++m) recur(kept(m - 1), m == 2 ? rv : kept(m - 2), kept(m), terms(m));
      } else {
        copy(ckp(0, 0), r);
        if (P > 1 || lbar) recur(rv, nullptr, WA, terms(1));
        if (P > 1 && 1 % s == 1) copy(ckp(0, 1), WA);
        const V* um2 = rv;
        V* um1 = WA;
        for (int m = 2; m < P; ++m) {
          V* out = (m == 2) ? WB : const_cast<V*>(um2);
          recur(um1, um2, out, terms(m));
          if (m % s == 0) copy(ckp(m / s, 0), out);
          if (m % s == 1) copy(ckp(m / s, 1), out);
          um2 = um1;
          um1 = out;
        }
      }
      // backward pass
      check_cuda(cudaMemsetAsync(WA, 0, vb, s2), "memset");
      check_cuda(cudaMemsetAsync(WB, 0, vb, s2), "memset");
      V* X = WA;  // w_{m+1}
      V* Y = WB;  // w_{m+2} -> w_m
      auto back = [&](int m, const V* u) {  // u = u_{m-1}
        int im = 0;
        const double2 cc = make_double2(coef[m].x, -coef[m].y);
        const double c = part_of(cc, im), f = (m == 1 ? 1.0 : 2.0) / h->dE;
        k_adj_step<Tr::fp64, Tr::ch, KK><<<grid, 128, 0, s2>>>(H, X, Y, (const V*)lam, c, im, u, f, gdiag, gslot);
        check_launch("k_adj_step");
        std::swap(X, Y);
      };
      if (keep) {
        for (int m = P - 1; m >= 1; --m) back(m, m == 1 ? rv : kept(m - 1));
      } else {
        for (int j = nck - 1; j >= 0; --j) {
          const int c = j * s;
          const int len = std::min(s, P - c);
          std::vector<const V*> useg(len);
          for (int q = 0; q < len; ++q) {
            if (q < 2) {
              useg[q] = ckp(j, q);
            } else {
              recur(useg[q - 1], useg[q - 2], kept(q), AdjTerms{});
              useg[q] = kept(q);
            }
          }
          for (int m = std::min(c + len, P - 1); m >= c + 1; --m) back(m, useg[m - 1 - c]);
        }
      }
      const double2 lc0 = make_double2(coef[0].x, -coef[0].y);
      k_adj_final<Tr::fp64, Tr::ch><<<nb, thr, 0, s2>>>(H, blk, P > 1 ? X : nullptr, Y, (const V*)lam, lc0, (V*)rbar);
      check_launch("k_adj_final");
    });
  }, &cdata);
}

}  // namespace

extern "C" gqt_status gqt_vac_loss_grad(gqt_ham* h, const void* d_phi, const double* dt, const int* Np, int Nt,
                                        int M, const double* beta, int stride, double* loss, double* d_g_onsite,
                                        double* d_g_slot, void* stream) {
  API_BEGIN
  check_common(h, 1);
  require(d_phi && dt && beta && loss && d_g_onsite && d_g_slot && Nt >= 1 && M >= 1, "gqt_vac_loss_grad: bad argument");
  require(h->nseg == 1, "gqt_vac_loss_grad: single-segment handles only");
  cudaStream_t st = (cudaStream_t)stream;
  reset_flag(h, st);
  const int64_t n = h->n;
  const int K = h->K;
  const size_t vb = h->vec_bytes(1);
  const BlockTable& T = h->table(1);
  const int nb = T.nblocks;
  const int* blk = (const int*)T.d_blk.p;
  const int thr = h->threads;
  std::vector<double> hbeta;
  if (!is_host_ptr(beta)) {  // device weights: one copy to the host (they become kernel arguments)
    hbeta.resize((size_t)Nt * M);
    check_cuda(cudaMemcpy(hbeta.data(), beta, hbeta.size() * sizeof(double), cudaMemcpyDeviceToHost), "beta");
    beta = hbeta.data();
  }
  char* A = (char*)h->ws(WS_ADJ0 + 4, (size_t)Nt * vb).p;
  char* B = (char*)h->ws(WS_ADJ0 + 5, (size_t)Nt * vb).p;
  double* gdiag = (double*)h->ws(WS_ADJ0 + 6, (size_t)n * sizeof(double)).p;
  double2* gslot = (double2*)h->ws(WS_ADJ0 + 7, (size_t)n * K * sizeof(double2)).p;
  void* abar = h->ws(WS_ADJ0 + 8, vb).p;
  void* bbar = h->ws(WS_ADJ0 + 9, vb).p;
  double2* LB = (double2*)h->ws(WS_ADJ0 + 10, (size_t)n * sizeof(double2)).p;
  void* tmp = h->ws(WS_ADJ0 + 11, vb).p;
  void* l = h->ws(WS_L, vb).p;
  double* dpart = (double*)h->ws(WS_ADJ0 + 12, (size_t)Nt * nb * sizeof(double)).p;  // loss partials per row
  // orders between checkpoints: the caller's, else all orders are kept where they fit
  // ADJ_KEEP and a quarter of the memory that is free once the buffers above are there
  // (the rest of the call takes a dozen vectors, or as much as it would with checkpoints),
  // and sqrt of the orders is the rule
  auto spacing = [&](int orders) {
    const int root = std::max(2, (int)std::ceil(std::sqrt((double)orders)));
    if (stride > 0) return root;
    size_t free_b = 0, total_b = 0;
    const size_t need = (size_t)orders * vb, have = h->ws(WS_ADJ0 + 1, vb).bytes;
    if (need > have) {
      check_cuda(cudaMemGetInfo(&free_b, &total_b), "cudaMemGetInfo");
      if (need > ADJ_KEEP || need > free_b / 4) return root;
    }
    return std::max(2, orders);
  };
  std::vector<int> nps(Nt);
  int most = M;  // orders of the longest expansion: its vectors are allocated first
  for (int k = 0; k < Nt; ++k) {
    nps[k] = resolve_np(h, dt[k], Np ? Np[k] : 0);
    if (k + 1 < Nt) most = std::max(most, nps[k]);
  }
  const SpareInUse used(h->spare_in_use, WS_ADJ0 + 1);
  if (spacing(most) >= most) h->ws(WS_ADJ0 + 1, (size_t)std::max(2, most) * vb);
  const int row_stride = stride > 0 ? stride : spacing(M);
  auto Ak = [&](int k) { return (void*)(A + (size_t)k * vb); };
  auto Bk = [&](int k) { return (void*)(B + (size_t)k * vb); };
  // forward states a_k = U(-t_k) phi, b_k = U(-t_k) V phi
  launch_velocity(h, d_phi, Bk(0), Ak(0), 1, st);
  for (int k = 0; k + 1 < Nt; ++k) {
    check_cuda(cudaMemcpyAsync(Ak(k + 1), Ak(k), vb, cudaMemcpyDeviceToDevice, st), "copy");
    check_cuda(cudaMemcpyAsync(Bk(k + 1), Bk(k), vb, cudaMemcpyDeviceToDevice, st), "copy");
    void* sets[2] = {Ak(k + 1), Bk(k + 1)};
    launch_evolve_sets<2>(h, sets, 1, evolve_coefs(h->dE * dt[k], -1, nps[k]), st, nullptr);
  }
  check_cuda(cudaMemsetAsync(gdiag, 0, (size_t)n * sizeof(double), st), "memset");
  check_cuda(cudaMemsetAsync(gslot, 0, (size_t)n * K * sizeof(double2), st), "memset");
  check_cuda(cudaMemsetAsync(abar, 0, vb, st), "memset");
  check_cuda(cudaMemsetAsync(bbar, 0, vb, st), "memset");
  std::vector<double> hpart((size_t)Nt * nb);
  double total = 0.0;
  dispatch(h, [&](auto H) {
    using Tr = EllTraits<decltype(H)>;
    using V = typename Tr::V;
    for (int k = Nt - 1; k >= 0; --k) {
      if (k + 1 < Nt) {
        const auto c = evolve_coefs(h->dE * dt[k], -1, nps[k]);
        poly_adjoint(h, H, Ak(k), abar, c, spacing((int)c.size()), tmp, nullptr,
                     gdiag, gslot, st);
        std::swap(abar, tmp);
        poly_adjoint(h, H, Bk(k), bbar, c, spacing((int)c.size()), tmp, nullptr,
                     gdiag, gslot, st);
        std::swap(bbar, tmp);
      }
      launch_velocity(h, Ak(k), l, nullptr, 1, st);
      std::vector<double2> bc(M);
      for (int m = 0; m < M; ++m) bc[m] = make_double2(beta[(size_t)k * M + m], 0.0);
      poly_adjoint(h, H, Bk(k), l, bc, row_stride, tmp, LB, gdiag, gslot, st);
      k_axpy<V><<<nb, thr, 0, st>>>(blk, (V*)bbar, (const V*)tmp);
      check_launch("k_axpy");
      k_dot_re<V><<<nb, thr, 0, st>>>(blk, (const V*)l, LB, dpart + (size_t)k * nb);
      check_launch("k_dot_re");
      k_vel_adj<Tr::fp64, Tr::ch, double2><<<nb, thr, 0, st>>>(H, blk, LB, (const V*)Ak(k), gslot);
      check_launch("k_vel_adj");
      k_vel_acc<Tr::fp64, Tr::ch><<<nb, thr, 0, st>>>(H, blk, 0.5 * h->dE, LB, (V*)abar);
      check_launch("k_vel_acc");
    }
    k_vel_adj<Tr::fp64, Tr::ch, V><<<nb, thr, 0, st>>>(H, blk, (const V*)bbar, (const V*)d_phi, gslot);
    check_launch("k_vel_adj");
  });
  const size_t tot = (size_t)n * K;
  k_grad_out<<<(int)std::min<size_t>((tot + 255) / 256, 8192), 256, 0, st>>>((int)n, K, gslot, gdiag,
                                                                            (double2*)d_g_slot, d_g_onsite);
  check_launch("k_grad_out");
  check_cuda(cudaMemcpyAsync(hpart.data(), dpart, hpart.size() * sizeof(double), cudaMemcpyDeviceToHost, st), "loss");
  check_cuda(cudaStreamSynchronize(st), "loss");
  for (int k = Nt - 1; k >= 0; --k)  // the order the rows were summed before: last row first
    for (int b = 0; b < nb; ++b) total += hpart[(size_t)k * nb + b];
  *loss = total;
  return finish_call(h, st, "gqt_vac_loss_grad");
  API_END
}

