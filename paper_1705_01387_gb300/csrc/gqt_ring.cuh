// gqt_ring.cuh -- two Chebyshev orders per launch on honeycomb lattices with the rows
// in shared memory (temporal blocking of the paired-FP32 rows, Eq. 21).
//
// The built-in honeycomb layout: site 2(c1 + L1 c2) + s, periodic; A(c1,c2) is bonded to
// B(c1,c2), B(c1+1,c2-1), B(c1,c2-1), and B(c1,c2) to A(c1,c2), A(c1-1,c2+1),
// A(c1,c2+1).  A CTA owns a band of BW cells and the rows y0 .. y0 + S - 1, a thread one
// site of a band row.  In iteration t it computes
//   - T_{m+1} = 2H~T_m - T_{m-1} on row y0 - 1 + t, and
//   - T_{m+2} = 2H~T_{m+1} - T_m on row y0 + t - 3, from the rows of T_{m+1} it made one to
//     three iterations before,
// so that per two orders a site's T_m, T_{m-1} and 2U/dE come from DRAM once and the two
// outputs go there once (NC chains: 64 NC + 8 bytes; hop array besides where the
// hoppings are not all one real number; no index array).  A single-order launch moves
// 140 (two chains) or 92 bytes per order.
//
// Every operand that more than one thread uses is in shared memory: the rows of T_m come
// in by bulk copies into a ring of six, two rows ahead of their first use, and T_{m+1} is
// handed on through a ring of four.  A thread's own T_{m-1} and 2U/dE are loaded one row
// ahead into registers.  What is left is the issue of instructions: the pair arithmetic
// runs two-wide on (re, im), the band width is a compile-time constant (shared-memory
// offsets are immediates), the neighbours of a site lie in its own row and in one
// other (below for A, above for B), and the steady iterations carry no conditions.
// N = 16.8M, one common hopping: a VAC pass takes 449 us (5.1 TB/s on its own 136 bytes,
// 0.75 of HBM), 520 with T_{m+1} staged through L2 instead of shared memory; an l = r
// pass at N = 4.2M 73.4 us (0.61), 79 before.  With the scalar operations the VAC pass is
// at 484, with a band width read at run time at 460, with bands of 64 at 494; of the
// 320 instructions per site of an l = r pass (450 of a VAC pass) 152 are arithmetic.
//
// Ring rows hold the cells B1 - 1 .. B1 + BW (entry 0: sublattice A of the left halo
// cell).  T_{m+1} at the two halo sites that T_{m+2} needs (A left, B right) is computed
// in a prologue for all rows of the piece, from global memory.
//
// Work split: one CTA per band and segment of rows, the segments as many as the
// resident CTAs allow.  With more bands than resident CTAs the band rows, band-major, are
// cut into gridDim.x equal ranges instead; a range that crosses a band's end, or is
// longer than RG_ROWS, is walked in pieces.
//
// The waits for the copies are bounded (gqt_set_wait_limit).  One that runs out sets bit
// 16 of the status word and goes on as a drain of RG_DRAIN polls: a slot may be filled
// again only when its row has landed, and no CTA may end with a copy in flight.  If the
// drain runs out too (bit 32), the thread that issues the copies leaves, so that none
// follows, and the others go through the remaining rows without waiting.  All of it is in
// the path of a poll that failed: a flag looked at before each row is asked for costs 5%
// of an l = r pass.
#pragma once

#include "gqt_tile.cuh"

namespace gqt {

// Band width for L1 cells: the largest of 128, 64, 32 dividing it (0: none).
__host__ __device__ inline int tl_band_width(int L1) {
  return L1 % 128 == 0 ? 128 : L1 % 64 == 0 ? 64 : L1 % 32 == 0 ? 32 : 0;
}

constexpr int RG_X = 6;       // rows of T_m in shared memory: four in use, two on their way
constexpr int RG_Z = 4;       // rows of T_{m+1}
constexpr int RG_ROWS = 256;  // rows of a piece at most (its halo columns are kept)
constexpr int RG_DRAIN = 1 << 24;  // polls of a drain

__host__ __device__ constexpr int ring_row(int bw) { return 2 * bw + 4; }  // entries of a ring row
inline size_t ring_smem(int bw, int nc, int rows) {
  return (size_t)nc * ((RG_X + RG_Z) * ring_row(bw) + 2 * (rows + 2)) * sizeof(float4) + RG_X * 8 + 16 + 4 * 8 * 8;
}

__device__ __forceinline__ uint32_t rg_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool rg_poll(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// What a CTA's waits share.
struct RingWait {
  int* err;    // status word
  int limit;   // polls of a wait
  int dead;    // a drain has run out
};
// The rest of a wait whose first poll failed.
__device__ __noinline__ void rg_wait_slow(uint32_t bar, uint32_t parity, volatile RingWait* w) {
  const bool issuer = threadIdx.x == 0;
  const int limit = w->limit;
  for (int it = 0; it < limit; ++it) {
    if (rg_poll(bar, parity)) return;
    if (w->dead && !issuer) return;
  }
  atomicOr(w->err, 16);
  for (int it = 0; it < RG_DRAIN; ++it) {
    if (rg_poll(bar, parity)) return;
    if (w->dead && !issuer) return;
  }
  w->dead = 1;
  atomicOr(w->err, 32);
  if (issuer) asm volatile("exit;");
}
__device__ __forceinline__ void rg_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ float4 rg_ld(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void rg_st(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}

// ---------------------------------------------------------------- two-wide pair arithmetic
// The operations of gqt_df.cuh on (re, im) as packed instructions; a - b is fma(b, -1, a)
// and a sign change a product with -1 (both exact), since the packed instructions
// take no signs on their operands.
__device__ __forceinline__ float2 p2_sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ void p2_prod(float2& p, float2& e, float2 ah, float2 al, float2 bh, float2 bl) {
  p = __fmul2_rn(ah, bh);
  e = __ffma2_rn(ah, bh, __fmul2_rn(p, make_float2(-1.f, -1.f)));
  e = __ffma2_rn(ah, bl, e);
  e = __ffma2_rn(al, bh, e);
}
__device__ __forceinline__ void p2_mac(DfC& a, float2 ah, float2 al, float2 bh, float2 bl) {
  float2 p, e;
  p2_prod(p, e, ah, al, bh, bl);
  const float2 s = __fadd2_rn(a.h, p);
  const float2 v = p2_sub(s, a.h);
  const float2 t = __fadd2_rn(p2_sub(a.h, p2_sub(s, v)), p2_sub(p, v));
  a.h = s;
  a.l = __fadd2_rn(a.l, __fadd2_rn(t, e));
}
__device__ __forceinline__ DfC p2_mul_sub(float2 ah, float2 al, float4 b, float4 x) {
  float2 p, e;
  p2_prod(p, e, ah, al, f2_hi(b), f2_lo(b));
  const float2 xh = f2_hi(x);
  const float2 s = p2_sub(p, xh);
  const float2 v = __fadd2_rn(s, xh);
  const float2 t = p2_sub(p2_sub(p, v), __fadd2_rn(xh, p2_sub(s, v)));
  return DfC{s, p2_sub(__fadd2_rn(t, e), f2_lo(x))};
}
__device__ __forceinline__ void p2_add(DfC& a, float4 x) {
  const float2 xh = f2_hi(x);
  const float2 s = __fadd2_rn(a.h, xh);
  const float2 v = p2_sub(s, a.h);
  const float2 t = __fadd2_rn(p2_sub(a.h, p2_sub(s, v)), p2_sub(xh, v));
  a.h = s;
  a.l = __fadd2_rn(a.l, __fadd2_rn(f2_lo(x), t));
}
__device__ __forceinline__ float4 p2_out(const DfC& a) {
  const float2 s = __fadd2_rn(a.h, a.l);
  const float2 v = p2_sub(s, a.h);
  const float2 t = __fadd2_rn(p2_sub(a.h, p2_sub(s, v)), p2_sub(a.l, v));
  return make_float4(s.x, s.y, t.x, t.y);
}
// sum of the products of the (re, im) words, kept apart until the end
__device__ __forceinline__ void p2_dot(DfC& d, float4 a, float4 b) { p2_mac(d, f2_hi(a), f2_lo(a), f2_hi(b), f2_lo(b)); }
__device__ __forceinline__ double p2_total(const DfC& d) { return df_value(d.h.x, d.l.x) + df_value(d.h.y, d.l.y); }

// T_{m+1} at a site from T_m (own, nb) and T_{m-1} (prev).
template <bool CH, bool UH>
__device__ __forceinline__ float4 rg_step(float2 h0h, float2 h0l, const typename DfHop<CH>::T (&hv)[3], float2 dg,
                                          float4 own, const float4 (&nb)[3], float4 prev) {
  DfC a = p2_mul_sub(f2_both(dg.x), f2_both(dg.y), own, prev);
  if constexpr (UH) {
    DfC s = dfc_of(nb[0]);
    p2_add(s, nb[1]);
    p2_add(s, nb[2]);
    p2_mac(a, h0h, h0l, s.h, s.l);
  } else {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      p2_mac(a, f2_both(hv[k].x), f2_both(hv[k].y), f2_hi(nb[k]), f2_lo(nb[k]));
      if constexpr (CH)
        p2_mac(a, make_float2(-hv[k].z, hv[k].z), make_float2(-hv[k].w, hv[k].w), make_float2(nb[k].y, nb[k].x),
               make_float2(nb[k].w, nb[k].z));
    }
  }
  return p2_out(a);
}

// The operands of one order at a site: H~ row, own value, the three neighbours
// and the order before, for NC chains.
template <bool CH, int NC>
struct TlSite {
  typename DfHop<CH>::T hv[3];
  float2 dg;
  float4 own[NC], nb[NC][3], prev[NC];
};

// Loads for site i with neighbours j[3]: in = the order the step multiplies,
// pv = the order before.
template <bool CH, int NC, bool UH>
__device__ __forceinline__ void tl_load(TlSite<CH, NC>& S, const DfEll<CH>& H, int i, const int (&j)[3],
                                        const float4* __restrict__ in0, const float4* __restrict__ in1,
                                        const float4* __restrict__ pv0, const float4* __restrict__ pv1) {
  if (!UH) {
#pragma unroll
    for (int k = 0; k < 3; ++k) S.hv[k] = __ldg(H.hop + (size_t)k * H.n + i);
  }
  S.dg = __ldg(H.diag + i);
#pragma unroll
  for (int ch = 0; ch < NC; ++ch) {
    const float4* in = ch ? in1 : in0;
    S.own[ch] = __ldg(in + i);
#pragma unroll
    for (int k = 0; k < 3; ++k) S.nb[ch][k] = __ldg(in + j[k]);
    S.prev[ch] = __ldg((ch ? pv1 : pv0) + i);
  }
}

// UH: every hopping is the real value H.h0 (no hop array is read).
template <bool CH, int NC, bool UH>
__device__ __forceinline__ void tl_compute(const TlSite<CH, NC>& S, const DfEll<CH>& H, float4 (&v)[NC]) {
#pragma unroll
  for (int ch = 0; ch < NC; ++ch) {
    if (UH)
      v[ch] = df_step_uh<3>(H.h0, S.dg, S.own[ch], S.nb[ch], S.prev[ch]);
    else
      v[ch] = df_step<CH, 3, false>(S.hv, S.dg, S.own[ch], S.nb[ch], S.prev[ch]);
  }
}

// hop slot of each neighbour type (0: same cell, 1: the neighbouring column, 2: the other
// row's same column) per sublattice
struct RingHop {
  int slot[2][3];
};

template <bool CH, int NC, bool UH, int BW>
__global__ void __launch_bounds__(2 * BW, (NC == 1 && UH ? 3 : 2) * (128 / BW)) k_cheb2_honey_df(
    DfEll<CH> H, Honey G, RingHop hs, int nseg, int max_rows, const float4* __restrict__ xa,
    const float4* __restrict__ ya, const float4* __restrict__ xb, const float4* __restrict__ yb,
    float4* __restrict__ za, float4* __restrict__ wa, float4* __restrict__ zb, float4* __restrict__ wb,
    double2* __restrict__ pout, int ostride, int nzero, int* __restrict__ err, int limit) {
  using HT = typename DfHop<CH>::T;
  constexpr int RW = ring_row(BW), RB = RW * 16;   // a ring row: entries, bytes
  constexpr int XCH = RG_X * RB, ZCH = RG_Z * RB;  // a chain's rings in bytes
  extern __shared__ __align__(128) unsigned char rg_sm[];
  const int tid = (int)threadIdx.x;
  const int zs = max_rows + 2;
  float4* const zh = reinterpret_cast<float4*>(rg_sm + NC * (XCH + ZCH));  // [NC][2][max_rows + 2]
  uint64_t* const full = reinterpret_cast<uint64_t*>(zh + NC * 2 * zs);
  volatile RingWait* const rw = reinterpret_cast<volatile RingWait*>(full + RG_X);
  double* const rsm = reinterpret_cast<double*>(full + RG_X + 2);
  const uint32_t xr = rg_addr(rg_sm), zr = xr + NC * XCH, bar = rg_addr(full);
  if (tid == 0) {
    for (int q = 0; q < RG_X; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar + 8 * q), "r"(1));
    asm volatile("fence.mbarrier_init.release.cluster;");
    rw->err = err;
    rw->limit = limit;
    rw->dead = 0;
    if (limit == 0) atomicOr(err, 16);  // gives up whatever its first polls say
  }
  __syncthreads();
  // the thread's site and its neighbours: own entry 2 + tid, the same cell's other site
  // (own ^ 1) in its own row and in the other row, and the neighbouring column's site
  const int s = tid & 1;
  const uint32_t oo = 16u * (2 + tid), o1 = 16u * ((2 + tid) ^ 1), o2 = 16u * (s ? tid - 1 : tid + 5);
  const float2 h0h = f2_both(H.h0.x), h0l = f2_both(H.h0.y);
  const int nbands = G.L1 / BW, r2 = 2 * G.L1;
  size_t hoff[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) hoff[k] = UH ? 0 : (size_t)(s ? hs.slot[1][k] : hs.slot[0][k]) * H.n;
  long long r_beg, r_end;  // band rows, band-major
  if (nseg > 0) {
    const int band = (int)blockIdx.x % nbands, seg = (int)blockIdx.x / nbands;
    r_beg = (long long)band * G.L2 + (long long)G.L2 * seg / nseg;
    r_end = (long long)band * G.L2 + (long long)G.L2 * (seg + 1) / nseg;
  } else {
    const long long total = (long long)nbands * G.L2;
    r_beg = total * blockIdx.x / gridDim.x;
    r_end = total * (blockIdx.x + 1) / gridDim.x;
  }
  DfC q0 = dfc_zero(), q1 = q0, q2 = q0, q3 = q0;
  int sw = 0;       // ring slot of the next row to wait for, and its parity
  uint32_t pw = 0;
  for (long long p = r_beg; p < r_end;) {
    const int band = (int)(p / G.L2), y0 = (int)(p % G.L2);
    const int S = (int)min(min((long long)(G.L2 - y0), r_end - p), (long long)max_rows);
    p += S;
    const int B1 = band * BW;
    const int cl = B1 == 0 ? G.L1 - 1 : B1 - 1, cr = B1 + BW == G.L1 ? 0 : B1 + BW;
    int si = sw, yi = y0 >= 2 ? y0 - 2 : y0 - 2 + G.L2;  // next row to ask for (thread 0)
    auto issue = [&]() {
      const size_t b = (size_t)r2 * yi;
      const uint32_t fb = bar + 8 * si;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"((uint32_t)(NC * RB))
                   : "memory");
#pragma unroll
      for (int ch = 0; ch < NC; ++ch) {
        const float4* x = (ch ? xb : xa) + b;
        const uint32_t d = xr + ch * XCH + si * RB;
        rg_copy(d, x + 2 * cl, 32, fb);
        rg_copy(d + 32, x + 2 * B1, 2 * BW * 16, fb);
        rg_copy(d + 32 + 2 * BW * 16, x + 2 * cr, 32, fb);
      }
      si = si + 1 == RG_X ? 0 : si + 1;
      yi = yi + 1 == G.L2 ? 0 : yi + 1;
    };
    if (tid == 0)
      for (int u = 0; u < 4; ++u) issue();
    // T_{m+1} on the halo columns (A at cell B1 - 1, B at cell B1 + BW) of rows y0 - 1 .. y0 + S
    for (int q = tid; q < 2 * (S + 2); q += 2 * BW) {
      const int right = q & 1;
      const TlCols C(G, right ? cr : cl, right);
      int j[3];
      const int i = C.at(G, y0 - 1 + (q >> 1), j);
      TlSite<CH, NC> T;
      tl_load<CH, NC, UH>(T, H, i, j, xa, xb, ya, yb);
      float4 v[NC];
      tl_compute<CH, NC, UH>(T, H, v);
#pragma unroll
      for (int ch = 0; ch < NC; ++ch) zh[(ch * 2 + right) * zs + (q >> 1)] = v[ch];
    }
    // own-site streams one row ahead: T_{m-1} and 2U/dE of the row yn (site index in)
    int yn = y0 == 0 ? G.L2 - 1 : y0 - 1;
    const size_t col = (size_t)(2 * B1 + tid);
    size_t in = (size_t)r2 * yn + col, ic = in;  // of the next and of the current row
    float4 ny[NC];
    float2 nd, d1 = make_float2(0.f, 0.f), d2 = d1;  // 2U/dE of the next row, of rows t - 1 and t - 2
    auto fetch = [&]() {
      ny[0] = __ldg(ya + in);
      if (NC == 2) ny[NC - 1] = __ldg(yb + in);
      nd = __ldg(H.diag + in);
    };
    fetch();
    size_t wi = (size_t)r2 * y0 + col;  // T_{m+2}'s site
    int sx = sw;                        // ring slot of row u = t (lattice row y0 - 2 + t)
    int waited = 0;
    auto wait_row = [&]() {
      if (!rg_poll(bar + 8 * sw, pw)) rg_wait_slow(bar + 8 * sw, pw, rw);
      sw = sw + 1 == RG_X ? 0 : sw + 1;
      pw ^= sw == 0 ? 1u : 0u;
      ++waited;
    };
    for (int u = 0; u < 3; ++u) wait_row();
    __syncthreads();
    // iteration t; FAST: both orders, on rows that are the CTA's own
    auto iterate = [&](int t, auto fast) {
      constexpr bool FAST = decltype(fast)::value;
      const bool first = FAST || t <= S + 1, own = FAST || (t >= 1 && t <= S), second = FAST || t >= 3;
      if (tid == 0 && t + 4 <= S + 3) issue();
      float4 yc[NC];
#pragma unroll
      for (int ch = 0; ch < NC; ++ch) yc[ch] = ny[ch];
      const float2 dc = nd;
      HT hv[3], hw[3];
      if (!UH) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (first) hv[k] = __ldg(H.hop + hoff[k] + in);
          if (second) hw[k] = __ldg(H.hop + hoff[k] + wi);
        }
      }
      ic = in;
      if (FAST || t + 1 <= S + 1) {
        yn = yn + 1 == G.L2 ? 0 : yn + 1;
        in = (size_t)r2 * yn + col;
        fetch();
      }
      const int sp1 = sx + 1 >= RG_X ? sx + 1 - RG_X : sx + 1;
      if (second) {
        // T_{m+2} on row y0 + t - 3: T_{m+1} of the rows t - 3 .. t - 1, T_m of row u = t - 1
        const int sm1 = sx == 0 ? RG_X - 1 : sx - 1;
        const uint32_t za_ = zr + ((t + 2) & (RG_Z - 1)) * RB;
        const uint32_t zo = zr + ((s ? t + 3 : t + 1) & (RG_Z - 1)) * RB;
        const uint32_t xp = xr + sm1 * RB + oo;
        float4 o[NC], v[NC];
#pragma unroll
        for (int ch = 0; ch < NC; ++ch) {
          o[ch] = rg_ld(za_ + oo + ch * ZCH);
          const float4 nb[3] = {rg_ld(za_ + o1 + ch * ZCH), rg_ld(zo + o2 + ch * ZCH), rg_ld(zo + o1 + ch * ZCH)};
          v[ch] = rg_step<CH, UH>(h0h, h0l, hw, d2, o[ch], nb, rg_ld(xp + ch * XCH));
        }
        wa[wi] = v[0];
        if (NC == 2) wb[wi] = v[NC - 1];
        if (NC == 2) {
          p2_dot(q2, o[0], o[NC - 1]);
          p2_dot(q3, o[0], v[NC - 1]);
        } else {
          p2_dot(q2, o[0], o[0]);
          p2_dot(q3, v[0], o[0]);
        }
        wi += r2;
      }
      if (first) {
        // T_{m+1} on row y0 - 1 + t: T_m of the rows u = t .. t + 2
        const int sp2 = sp1 + 1 >= RG_X ? sp1 + 1 - RG_X : sp1 + 1;
        const uint32_t xo = xr + sp1 * RB, xn = xr + (s ? sp2 : sx) * RB;
        const uint32_t zt = zr + (t & (RG_Z - 1)) * RB;
        float4 o[NC], v[NC];
#pragma unroll
        for (int ch = 0; ch < NC; ++ch) {
          o[ch] = rg_ld(xo + oo + ch * XCH);
          const float4 nb[3] = {rg_ld(xo + o1 + ch * XCH), rg_ld(xn + o2 + ch * XCH), rg_ld(xn + o1 + ch * XCH)};
          v[ch] = rg_step<CH, UH>(h0h, h0l, hv, dc, o[ch], nb, yc[ch]);
        }
#pragma unroll
        for (int ch = 0; ch < NC; ++ch) {
          rg_st(zt + oo + ch * ZCH, v[ch]);
          if (tid < 2) rg_st(zt + (tid == 0 ? 0 : 16 * (2 * BW + 3)) + ch * ZCH, zh[(ch * 2 + tid) * zs + t]);
        }
        if (own) {
          za[ic] = v[0];
          if (NC == 2) zb[ic] = v[NC - 1];
          if (NC == 2) {
            p2_dot(q0, o[0], o[NC - 1]);
            p2_dot(q1, o[0], v[NC - 1]);
          } else {
            p2_dot(q0, o[0], o[0]);
            p2_dot(q1, v[0], o[0]);
          }
        }
      }
      d2 = d1;
      d1 = dc;
      sx = sp1;
      // the next iteration's last row of T_m; one warp waits for everybody
      if (tid < 32 && (FAST || waited < S + 4)) wait_row();
      __syncthreads();
    };
    int t = 0;
    for (; t < 3; ++t) iterate(t, std::false_type());
    for (; t <= S; ++t) iterate(t, std::true_type());
    for (; t <= S + 2; ++t) iterate(t, std::false_type());
    // warps 1 .. follow the waiting warp's position
    if (tid >= 32) {
      for (; waited < S + 4; ++waited) {
        sw = sw + 1 == RG_X ? 0 : sw + 1;
        pw ^= sw == 0 ? 1u : 0u;
      }
    }
  }
  double r[4] = {p2_total(q0), p2_total(q1), p2_total(q2), p2_total(q3)};
  block_reduce_rx<4>(r, 1, rsm);
  if (tid == 0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) pout[(size_t)j * ostride + blockIdx.x] = make_double2(r[j], 0.0);
  }
  for (int b = blockIdx.x + gridDim.x; b < nzero; b += gridDim.x)
    if (tid < 4) pout[(size_t)tid * ostride + b] = make_double2(0.0, 0.0);
}

}  // namespace gqt
