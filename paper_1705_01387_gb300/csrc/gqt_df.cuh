// gqt_df.cuh -- FP64-storage moment rows and evolution orders computed on the FP32 pipes.
//
// GB300 issues about 2 FP64 fused multiply-adds per clock per SM and 128 FP32
// ones, so the FP64 moment kernels (k_cheb_pair_w, k_cheb_dbl_w) are bound by
// the FP64 pipe, well below the HBM roofline.  These kernels keep FP64-sized
// storage (16 bytes per complex element) and FP64-level results, but do the
// arithmetic of the recursion (Eq. 21) and of the moment dots (Eqs. 28-30) on
// unevaluated pairs of FP32 numbers ("double-float": x = hi + lo with
// |lo| <= ulp(hi)/2, about 48 significant bits), using the error-free
// transformations of Dekker (1971) and Knuth (TwoSum), with TwoProduct by the
// fused multiply-add (Ogita, Rump and Oishi 2005):
//   TwoProduct(a, b): p = fl(a b), e = fma(a, b, -p), a b = p + e exactly;
//   TwoSum(a, b):     s = fl(a + b), v = s - a, e = (a - (s - v)) + (b - v),
//                     a + b = s + e exactly.
// A product of two pairs keeps p and e + a_hi b_lo + a_lo b_hi (the a_lo b_lo
// term is below 2^-48 of the product); sums keep the TwoSum error in the low
// word and renormalise once per element.  Every operation is written with the
// _rn intrinsics, which the compiler never contracts into fused multiply-adds
// (a contraction would break the error-free transformations).
//
// Storage: the chain vectors T_k are float4 per complex element
// (re.hi, im.hi, re.lo, im.lo); the caller's input vectors stay complex128 and
// are split once per row or evolution.  The Hamiltonian's 2H~ (real hoppings:
// float2 (hi, lo) per slot; complex: float4 (re.hi, re.lo, im.hi, im.lo)) and 2U/dE
// (float2) are split once per handle from its FP64 arrays.  Moment partial sums leave
// each thread as FP64 (hi + lo) and are reduced in FP64 as in the FP64 kernels, into
// the same partial slots, so k_reduce_dbl combines them unchanged.
#pragma once

#include "gqt_kernels.cuh"

namespace gqt {

template <bool CH>
struct DfHop;
template <>
struct DfHop<false> {
  using T = float2;  // (hi, lo) of a real 2H~_ij
};
template <>
struct DfHop<true> {
  using T = float4;  // (re.hi, re.lo, im.hi, im.lo) of a complex 2H~_ij
};

template <bool CH>
struct DfEll {
  int n = 0;
  int K = 0;
  const int* idx = nullptr;                    // [K][n]
  const typename DfHop<CH>::T* hop = nullptr;  // [K][n]
  const float2* diag = nullptr;                // [n]
  const uint16_t* cls = nullptr;    // row classes (row_neighbours)
  const int* cls_off = nullptr;
  const typename DfHop<CH>::T* xhop = nullptr;  // [K][n] 2[X,H~]_ij = -dx_ij 2H~_ij (commutator orders)
  float2 h0 = {0.f, 0.f};  // the common 2H~_ij of handles whose slots all hold one real hopping
};

// ---------------------------------------------------------------- pair arithmetic

// An FP64 value as a pair (the first order reads the caller's FP64 vectors).
__device__ __forceinline__ float2 df_split(double x) {
  const float h = __double2float_rn(x);
  return make_float2(h, __double2float_rn(x - (double)h));
}
// A complex FP64 element as a chain element (re.hi, im.hi, re.lo, im.lo).
__device__ __forceinline__ float4 df_split(double2 z) {
  const float2 a = df_split(z.x), b = df_split(z.y);
  return make_float4(a.x, b.x, a.y, b.y);
}
// df_split by integer operations: the FP64 pipe (four operations a value) took 1.9 ms
// for two vectors of 16.8M elements and their neighbours.  hi is x rounded to 24 bits
// (half up; the pair's sum is the same where a tie rounds the other way), the rest a
// signed integer of 29 bits, rounded to FP32 and scaled.  Values outside 2^-73 .. 2^126,
// whose parts could leave the normal FP32 range, take df_split.
__device__ __forceinline__ float2 df_split_int(double x) {
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  const uint32_t top = (uint32_t)(u >> 32), ex = (top >> 20) & 0x7FFu;
  if (ex - 950u > 199u) return (u << 1) == 0 ? make_float2(0.f, 0.f) : df_split(x);
  const uint32_t sign = top & 0x80000000u, low = (uint32_t)u & 0x1FFFFFFFu;
  const uint64_t m = (u & 0x7FFFFFFFFFFFFFFFull) + (1u << 28);
  const float hi = __uint_as_float((uint32_t)((m >> 29) - (896u << 23)) | sign);
  const int r = (int)low - ((low >> 28) ? (1 << 29) : 0);
  const float lo = __fmul_rn((float)r, __uint_as_float(((ex - 948u) << 23) | sign));
  return make_float2(hi, lo);
}

// A complex FP64 coefficient as (re.hi, re.lo, im.hi, im.lo).
__device__ __forceinline__ float4 df_split_coef(double2 z) {
  const float2 a = df_split(z.x), b = df_split(z.y);
  return make_float4(a.x, a.y, b.x, b.y);
}
// A float widened to double with integer operations (exact), as the conversion
// instruction does on the FP64 pipe at 1/64 of the FP32 rate; zeros, denormals,
// infinities and NaNs take the instruction (in a function of its own, so that it is
// not executed under a predicate for every value).
static __device__ __noinline__ double f2d_special(float x) { return (double)x; }
__device__ __forceinline__ double f2d(float x) {
  const uint32_t u = __float_as_uint(x);
  if (((u >> 23) + 1u & 0xFFu) < 2u) return f2d_special(x);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double df_value(float h, float l) { return f2d(h) + f2d(l); }

// Operations on the (re, im) words, each rounded to nearest.
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) {
  return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) {
  return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}
__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) {
  return make_float2(__fmaf_rn(a.x, b.x, c.x), __fmaf_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) {
  return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y));
}
__device__ __forceinline__ float2 f2_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 f2_both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 f2_hi(float4 x) { return make_float2(x.x, x.y); }
__device__ __forceinline__ float2 f2_lo(float4 x) { return make_float2(x.z, x.w); }

// Product of pairs: p = fl(ah bh), e its error and the cross terms.
__device__ __forceinline__ void df_prod(float2& p, float2& e, float2 ah, float2 al, float2 bh, float2 bl) {
  p = f2_mul(ah, bh);
  e = f2_fma(ah, bh, f2_neg(p));
  e = f2_fma(ah, bl, e);
  e = f2_fma(al, bh, e);
}

// Complex accumulator (h: re.hi, im.hi; l: re.lo, im.lo), unnormalised: l collects the
// TwoSum errors and the low parts of the products.
struct DfC {
  float2 h, l;
};

__device__ __forceinline__ DfC dfc_zero() { return DfC{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ DfC dfc_of(float4 a) { return DfC{f2_hi(a), f2_lo(a)}; }

// a += (ah, al) * (bh, bl)
__device__ __forceinline__ void df_mac(DfC& a, float2 ah, float2 al, float2 bh, float2 bl) {
  float2 p, e;
  df_prod(p, e, ah, al, bh, bl);
  const float2 s = f2_add(a.h, p);
  const float2 v = f2_sub(s, a.h);
  const float2 t = f2_add(f2_sub(a.h, f2_sub(s, v)), f2_sub(p, v));
  a.h = s;
  a.l = f2_add(a.l, f2_add(t, e));
}

// a = (ah, al) * (bh, bl) - x, as df_mac on an accumulator holding -x
__device__ __forceinline__ DfC df_mul_sub(float2 ah, float2 al, float2 bh, float2 bl, float4 x) {
  float2 p, e;
  df_prod(p, e, ah, al, bh, bl);
  const float2 xh = f2_hi(x);
  const float2 s = f2_sub(p, xh);
  const float2 v = f2_add(s, xh);
  const float2 t = f2_sub(f2_sub(p, v), f2_add(xh, f2_sub(s, v)));
  return DfC{s, f2_sub(f2_add(t, e), f2_lo(x))};
}

// a += x (TwoSum of the high words, the low words and the TwoSum error added into l)
__device__ __forceinline__ void df_add(DfC& a, float4 x) {
  const float2 xh = f2_hi(x);
  const float2 s = f2_add(a.h, xh);
  const float2 v = f2_sub(s, a.h);
  const float2 t = f2_add(f2_sub(a.h, f2_sub(s, v)), f2_sub(xh, v));
  a.h = s;
  a.l = f2_add(a.l, f2_add(f2_lo(x), t));
}

// acc += c * x, c real pair
__device__ __forceinline__ void dfc_mac(DfC& a, float2 c, float4 x) {
  df_mac(a, f2_both(c.x), f2_both(c.y), f2_hi(x), f2_lo(x));
}
// acc += i c * x, c real pair: (re, im) += c (-im, re)
__device__ __forceinline__ void dfc_mac_i(DfC& a, float2 c, float4 x) {
  df_mac(a, make_float2(-c.x, c.x), make_float2(-c.y, c.y), make_float2(x.y, x.x), make_float2(x.w, x.z));
}
// acc += c * x, c complex pair (re.hi, re.lo, im.hi, im.lo)
__device__ __forceinline__ void dfc_mac(DfC& a, float4 c, float4 x) {
  dfc_mac(a, make_float2(c.x, c.y), x);
  dfc_mac_i(a, make_float2(c.z, c.w), x);
}

// Normalised pairs of an accumulator (TwoSum of the two words).
__device__ __forceinline__ float4 dfc_out(const DfC& a, bool half) {
  float2 s = f2_add(a.h, a.l);
  const float2 v = f2_sub(s, a.h);
  float2 t = f2_add(f2_sub(a.h, f2_sub(s, v)), f2_sub(a.l, v));
  if (half) {  // exact scaling of both words (T_1 = H~ T_0 from 2H~)
    s = f2_mul(s, make_float2(0.5f, 0.5f));
    t = f2_mul(t, make_float2(0.5f, 0.5f));
  }
  return make_float4(s.x, s.y, t.x, t.y);
}

__device__ __forceinline__ void df_mac1(float& sh, float& sl, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  const float s = __fadd_rn(sh, p);
  const float v = __fsub_rn(s, sh);
  const float t = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, v)), __fsub_rn(p, v));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(t, e));
}
// Per-thread real dot accumulator: sum of Re conj(a) b or |a|^2 over the thread's
// elements, as one unnormalised pair; FP64 once per thread.  (Separate pairs for the
// real and imaginary products cost the l = r orders their registers: 15.0 -> 18.4 us
// at 1M sites of a square lattice.)
struct DfDot {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add_re(float4 a, float4 b) {
    df_mac1(h, l, a.x, a.z, b.x, b.z);
    df_mac1(h, l, a.y, a.w, b.y, b.w);
  }
  __device__ __forceinline__ void add_norm(float4 a) { add_re(a, a); }
  __device__ __forceinline__ double get() const { return df_value(h, l); }
};

// ---------------------------------------------------------------- split of H~

// 2H~ and 2U/dE of an FP64 handle as pairs (once per handle).
template <bool CH>
__global__ void k_split_hamiltonian(long long nslots, const void* __restrict__ hop64, int n,
                                    const double* __restrict__ diag64, void* __restrict__ hop_df,
                                    float2* __restrict__ diag_df) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < nslots; s += stride) {
    if (CH)
      ((float4*)hop_df)[s] = df_split_coef(((const double2*)hop64)[s]);
    else
      ((float2*)hop_df)[s] = df_split(((const double*)hop64)[s]);
  }
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += stride)
    diag_df[i] = df_split(diag64[i]);
}

// 2[X,H~] slot values -dx_ij 2H~_ij (Eq. 34 with [X,H]_ij = -dx_ij H_ij) as pairs,
// formed in FP64 and split once per handle.
template <bool CH>
__global__ void k_split_xhop(long long nslots, const void* __restrict__ hop64, const double* __restrict__ dx,
                             void* __restrict__ xhop_df) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < nslots; s += stride) {
    const double d = -dx[s];
    if (CH) {
      const double2 h = ((const double2*)hop64)[s];
      ((float4*)xhop_df)[s] = df_split_coef(make_double2(d * h.x, d * h.y));
    } else {
      ((float2*)xhop_df)[s] = df_split(d * ((const double*)hop64)[s]);
    }
  }
}

// FP64 vectors as pairs, once per row or evolution (T_0 of the chains).
template <int NV>
struct DfSplit {
  const double2* in[NV];
  float4* out[NV];
};
template <int NV>
__global__ void __launch_bounds__(256) k_split_vec(DfSplit<NV> A, size_t n) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const double2 z = A.in[q][e];
      const float2 a = df_split_int(z.x), b = df_split_int(z.y);
      A.out[q][e] = make_float4(a.x, b.x, a.y, b.y);
    }
}

// ---------------------------------------------------------------- moment rows

// T_m = 2H~ T_{m-1} - T_{m-2} at element i of a pair chain (T_1 = H~ T_0 when
// FIRST); own = T_{m-1}[i], nb[k] = T_{m-1}[idx[k][i]].
template <bool FIRST>
__device__ __forceinline__ DfC df_start(float2 dg, float4 own, float4 tm2) {
  if (FIRST) {
    DfC a;
    df_prod(a.h, a.l, f2_both(dg.x), f2_both(dg.y), f2_hi(own), f2_lo(own));
    return a;
  }
  return df_mul_sub(f2_both(dg.x), f2_both(dg.y), f2_hi(own), f2_lo(own), tm2);
}
template <bool CH, int KK, bool FIRST>
__device__ __forceinline__ float4 df_step(const typename DfHop<CH>::T (&hv)[KK], float2 dg, float4 own,
                                          const float4 (&nb)[KK], float4 tm2) {
  DfC a = df_start<FIRST>(dg, own, tm2);
#pragma unroll
  for (int k = 0; k < KK; ++k) dfc_mac(a, hv[k], nb[k]);
  return dfc_out(a, FIRST);
}

// a += h0 * (sum_k nb[k]) for a real pair h0: the neighbour values are summed as
// pairs first, so one product with h0 replaces KK.
template <int KK>
__device__ __forceinline__ void dfc_mac_sum(DfC& a, float2 h0, const float4 (&nb)[KK]) {
  DfC s = dfc_of(nb[0]);
#pragma unroll
  for (int k = 1; k < KK; ++k) df_add(s, nb[k]);
  df_mac(a, f2_both(h0.x), f2_both(h0.y), s.h, s.l);
}

// T_m at one element when every hopping equals h0 (a real 2H~ value), as
// df_step (T_1 = H~ T_0 when FIRST).
template <int KK, bool FIRST = false>
__device__ __forceinline__ float4 df_step_uh(float2 h0, float2 dg, float4 own, const float4 (&nb)[KK], float4 tm2) {
  DfC a = df_start<FIRST>(dg, own, tm2);
  dfc_mac_sum<KK>(a, h0, nb);
  return dfc_out(a, FIRST);
}

// T_m with the hoppings of the slots (hv) or, when UH, the common value H.h0.
template <bool CH, int KK, bool FIRST, bool UH>
__device__ __forceinline__ float4 df_step_any(const DfEll<CH>& H, const typename DfHop<CH>::T (&hv)[KK], float2 dg,
                                              float4 own, const float4 (&nb)[KK], float4 tm2) {
  if constexpr (UH)
    return df_step_uh<KK, FIRST>(H.h0, dg, own, nb, tm2);
  else
    return df_step<CH, KK, FIRST>(hv, dg, own, nb, tm2);
}

// VAC rows by two recurrences (the pair form of k_cheb_pair_w): chain A from l,
// chain B from r, A_k = T_k l, B_k = T_k r; step m writes A_m, B_m and adds
// Re <A_{m-1}|B_{m-1}> (moment slot 2m-2) and Re <A_{m-1}|B_m> (slot 2m-1); the
// first step also adds |l|^2 and |r|^2 (slot_norm).  l and r are split before it
// (k_split_vec).  R = 1, wavefront CTA order, one element per thread.
template <bool CH, int KK, bool FIRST, bool UH>
__global__ void __launch_bounds__(256, 3) k_cheb_pair_df(DfEll<CH> H, const int4* __restrict__ tab,
                                                         const float4* am1,
                                                         const float4* bm1, const float4* am2,
                                                         const float4* bm2, float4* aout, float4* bout,
                                                         double2* __restrict__ partial, int nblocks, int m,
                                                         int slot_norm) {
  using HT = typename DfHop<CH>::T;
  double2* smem = dyn_smem();
  const int b = blockIdx.x;
  const int4 tb = tab[b];
  chain_wait();
  const size_t segb = (size_t)tb.x, sege = (size_t)tb.y;
  const size_t step = (size_t)tb.w * blockDim.x;
  DfDot d0, d1, nl, nr;
  for (size_t e = segb + (size_t)tb.z * blockDim.x + threadIdx.x; e < sege; e += step) {
    const int i = (int)e;
    int idx[KK];
    HT hv[KK];
    row_neighbours<KK>(H.idx, H.cls, H.cls_off, H.n, i, row_class(H.cls, i), idx);
    if (!UH)
#pragma unroll
      for (int k = 0; k < KK; ++k) hv[k] = __ldg(H.hop + (size_t)k * H.n + i);
    const float2 dg = __ldg(H.diag + i);
    const float4 ao = am1[e], bo = bm1[e];
    float4 a2 = make_float4(0.f, 0.f, 0.f, 0.f), b2 = a2;
    if (!FIRST) {
      a2 = am2[e];
      b2 = bm2[e];
    }
    float4 na[KK], nbv[KK];
#pragma unroll
    for (int k = 0; k < KK; ++k) {
      na[k] = am1[idx[k]];
      nbv[k] = bm1[idx[k]];
    }
    const float4 a = df_step_any<CH, KK, FIRST, UH>(H, hv, dg, ao, na, a2);
    const float4 bb = df_step_any<CH, KK, FIRST, UH>(H, hv, dg, bo, nbv, b2);
    aout[e] = a;
    bout[e] = bb;
    d0.add_re(ao, bo);
    d1.add_re(ao, bb);
    if (FIRST) {
      nl.add_norm(ao);
      nr.add_norm(bo);
    }
  }
  const int k0 = 2 * m - 2;
  if (FIRST) {
    double v[4] = {d0.get(), d1.get(), nl.get(), nr.get()};
    block_reduce_rx<4>(v, 1, (double*)smem);
    if (threadIdx.x == 0) {
      partial[(size_t)k0 * nblocks + b] = make_double2(v[0], 0.0);
      partial[(size_t)(k0 + 1) * nblocks + b] = make_double2(v[1], 0.0);
      partial[(size_t)slot_norm * nblocks + b] = make_double2(v[2], v[3]);
    }
  } else {
    double v[2] = {d0.get(), d1.get()};
    block_reduce_rx<2>(v, 1, (double*)smem);
    if (threadIdx.x == 0) {
      partial[(size_t)k0 * nblocks + b] = make_double2(v[0], 0.0);
      partial[(size_t)(k0 + 1) * nblocks + b] = make_double2(v[1], 0.0);
    }
  }
}

// l = r rows (DOS, MSD) by the doubling identities (the pair form of
// k_cheb_dbl_w): step m writes u_m and adds <u_{m-1}|u_{m-1}> (slot 2m-2) and
// Re <u_m|u_{m-1}> (slot 2m-1).  R = 1, wavefront CTA order, U elements in flight
// per thread.
template <bool CH, int KK, int U, bool FIRST, bool UH>
__global__ void __launch_bounds__(256, U == 1 && UH ? 4 : 3) k_cheb_dbl_df(DfEll<CH> H, const int4* __restrict__ tab,
                                                        const float4* tm1, const float4* tm2,
                                                        float4* tout, double2* __restrict__ partial, int nblocks,
                                                        int m) {
  using HT = typename DfHop<CH>::T;
  double2* smem = dyn_smem();
  const int b = blockIdx.x;
  const int4 tb = tab[b];
  chain_wait();
  const size_t segb = (size_t)tb.x, sege = (size_t)tb.y;
  const size_t step = (size_t)tb.w * blockDim.x;
  DfDot a0, a1;
  // a row's class is asked for one iteration ahead (as the index array would be by U = 2
  // elements in flight): the neighbours' addresses then depend on no load from memory
  const size_t first_e = segb + (size_t)tb.z * blockDim.x + threadIdx.x;
  int cl[U];
#pragma unroll
  for (int u = 0; u < U; ++u) cl[u] = first_e + u * step < sege ? row_class(H.cls, (int)(first_e + u * step)) : 0;
  for (size_t e0 = first_e; e0 < sege; e0 += (size_t)U * step) {
    int idx[U][KK];
    HT hv[U][KK];
    float2 dg[U];
    float4 own[U], t2[U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const size_t e = e0 + u * step;
      ok[u] = e < sege;
      const size_t ee = ok[u] ? e : e0;
      const int i = (int)ee;
      row_neighbours<KK>(H.idx, H.cls, H.cls_off, H.n, i, ok[u] ? cl[u] : cl[0], idx[u]);
      if (!UH)
#pragma unroll
        for (int k = 0; k < KK; ++k) hv[u][k] = __ldg(H.hop + (size_t)k * H.n + i);
      dg[u] = __ldg(H.diag + i);
      own[u] = tm1[ee];
      t2[u] = FIRST ? make_float4(0.f, 0.f, 0.f, 0.f) : tm2[ee];
    }
    float4 nb[U][KK];
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int k = 0; k < KK; ++k) nb[u][k] = tm1[idx[u][k]];
      const size_t en = e0 + (size_t)(U + u) * step;
      cl[u] = en < sege ? row_class(H.cls, (int)en) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float4 a = df_step_any<CH, KK, FIRST, UH>(H, hv[u], dg[u], own[u], nb[u], t2[u]);
      if (ok[u]) {
        const size_t e = e0 + u * step;
        tout[e] = a;
        a0.add_norm(own[u]);
        a1.add_re(a, own[u]);
      }
    }
  }
  double v[2] = {a0.get(), a1.get()};
  block_reduce_rx<2>(v, 1, (double*)smem);
  if (threadIdx.x == 0) {
    const int k0 = 2 * m - 2;
    partial[(size_t)k0 * nblocks + b] = make_double2(v[0], 0.0);
    partial[(size_t)(k0 + 1) * nblocks + b] = make_double2(v[1], 0.0);
  }
}

}  // namespace gqt
