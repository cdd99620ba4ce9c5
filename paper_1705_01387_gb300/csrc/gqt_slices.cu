// gqt_slices.cu -- FP64 matrix products on the tcgen05 tensor cores, by exact integer
// slices.
//
// GB300 multiplies FP64 numbers at 0.63e12 multiply-adds a second and FP16 ones at
// about 1e15, so a dense FP64 contraction is split into small integers (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with
// fixed-point slices): every row is scaled by a power of two to below 1 in magnitude
// and cut into SL = 7 signed base-256 digits d_0 .. d_6 (FP16 holds them exactly),
//   x = 2^e sum_i d_i 2^(-7-8i) + r,  |r| <= 2^(e-56),
// so that a product sum becomes sum_l 2^(-14-8l) V_l with V_l the sum of d_i d_j over
// the contraction and over i + j = l.  Levels l = 0 .. 6 are kept (28 digit products);
// the first one left out is 2^-56 of the rows' maxima, where the FP64 accumulation of
// such a sum rounds at 2^-53 of its partial sums.  |d_i d_j| <= 2^14 and at most 7
// pairs share a level, so 8 stages of 16 elements stay below 2^24 and accumulate
// without rounding in the FP32 accumulators of tensor memory; they are then added up
// as 64-bit integers.
//
// What is left out is at most 2^-53 of the product of the rows' largest elements for
// every element of the contraction (six digit pairs of the first level left out and two
// remainders, 2^-56 each), typically 2^-56 times the root of their number; a chain of
// FP64 multiply-adds rounds by 2^-54 of its partial sums.  For rows of about even
// magnitude the slices are the more exact of the two: simulated for normal values with the
// largest at 2^e, 512 complex elements a chain, their error is 0.3, 0.6, 1.2 and 4 times
// the multiply-adds' at 2^e = 6, 8, 12 and 24 standard deviations (2048 elements: 0.3,
// 0.3, 0.7 and 3.9), which is the bound SLICE_SPREAD on the rows' spreads.  Whole Lambda
// (chains in 64 bits) of random vectors against 80-bit arithmetic, sums of squares:
// 2.5e-16 at M = 12 and N R = 24 (3.0e-16 on the FP64 pipe), 8e-16 at M = 100 and N R =
// 800 (1.4e-15), 8e-16 at M = 120 and N R = 1600 (1.0e-15).
//
// One CTA: a 128 x 64 tile of one product, seven accumulators of 64 columns.  Stages of
// 16 contraction elements (7 slices of both operands, 42 KB) come in by two bulk tensor
// copies into a ring of five buffers; one thread issues the copies and the 28 products
// of a stage; eight warps empty the accumulators every eighth stage.  Bound: the
// products (28 x 128 x 64 x 16 per stage, the shared-memory reads of a 64-column
// product taking 1.5 times its tensor time).  Lambda at M = 256, N R = 18432: 0.42 ms
// (643 TFLOP/s of digit products, 0.31 of the FP16 rate) and 0.15 ms for the slices,
// against 8.15 ms for the same contraction on the FP64 pipe at 0.99 of its rate.
//
// Every wait is bounded: after `limit` polls (0: at once) a role gives up, the issuing
// thread drains what it has in flight (SLICE_WAIT polls a wait), tensor memory is freed,
// and the error word gets bit 16 (32 if the drain gave up as well).

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>
#include <string>

#include "gqt_internal.h"
#include "gqt_slices.h"

namespace gqt {
namespace {

constexpr int SL = SLICES;
constexpr int SG_M = 128, SG_N = 64, SG_K = 16;
constexpr int SG_ASLICE = SG_M * SG_K * 2, SG_BSLICE = SG_N * SG_K * 2;  // 4 KB, 2 KB
constexpr int SG_STAGE = SL * (SG_ASLICE + SG_BSLICE);                    // 42 KB
constexpr int SG_NBUF = 5;
constexpr int SG_GROUP = 8;  // stages per emptying of the accumulators
constexpr int SG_THREADS = 288;
constexpr int SG_SMEM = SG_NBUF * SG_STAGE + 1024 + 256;

static_assert(SL * SG_GROUP * SG_K * (1 << 14) < (1 << 24), "a level's sum must stay exact in FP32");

__device__ __forceinline__ uint32_t sg_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool sg_poll(uint64_t* bar, uint32_t parity) {
  uint32_t done = 0;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(sg_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// Bounded wait; gives up early once another role has.
__device__ __forceinline__ bool sg_wait(uint64_t* bar, uint32_t parity, int limit, volatile int* stop) {
  for (int it = 0; it < limit; ++it) {
    if (sg_poll(bar, parity)) return true;
    if (*stop) return false;
  }
  return false;
}
__device__ __forceinline__ bool sg_drain(uint64_t* bar, uint32_t parity) {
  for (int it = 0; it < SLICE_WAIT; ++it)
    if (sg_poll(bar, parity)) return true;
  return false;
}

// K-major operand, rows of 32 B (16 FP16 values), 32-B swizzle, 8-row groups 256 B apart.
__device__ __forceinline__ uint64_t sg_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(256 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
}

// kind::f16, FP16 operands, FP32 accumulator, K-major, M = 128, N = 64; bit 13 negates A.
constexpr uint32_t SG_IDESC = (1u << 4) | ((uint32_t)(SG_N >> 3) << 17) | ((uint32_t)(SG_M >> 4) << 24);
__device__ __forceinline__ void sg_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void sg_load(uint32_t dst, const CUtensorMap* map, int row, int chunk, int slice,
                                        uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(chunk), "r"(slice), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void sg_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sg_addr(bar))
               : "memory");
}

__device__ __forceinline__ void sg_tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Tile (blockIdx.x: 128 rows of A; blockIdx.y: part and 64 rows of B; blockIdx.z: split
// of the contraction).  Part p sums its `terms` products A-plane . B-plane (negated
// where neg).  out[split][part][rowsA][rowsB], scaled rows (the caller applies 2^(eA +
// eB)); add: on top of what it holds.
__global__ void __launch_bounds__(SG_THREADS, 1)
    k_slice_gemm(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, SliceParts parts,
                 int rows_a, int rows_b, int nchunk, int per_split, double* __restrict__ out, int add,
                 int* __restrict__ err, int limit) {
  extern __shared__ __align__(1024) unsigned char sg_raw[];
  const uint32_t raw = sg_addr(sg_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = sg_raw + (base - raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + SG_NBUF * SG_STAGE);
  uint64_t* done = full + SG_NBUF;
  uint64_t* acc_full = done + SG_NBUF;
  uint64_t* acc_free = acc_full + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(acc_free + 1);
  volatile int* stop = reinterpret_cast<volatile int*>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ntile_b = (rows_b + SG_N - 1) / SG_N;
  const int part = (int)blockIdx.y / ntile_b;
  const int m0 = blockIdx.x * SG_M, n0 = ((int)blockIdx.y % ntile_b) * SG_N;
  const int c0 = (int)blockIdx.z * per_split, c1 = min(nchunk, c0 + per_split);
  const int terms = parts.terms;
  const int nst = max(0, c1 - c0) * terms;
  const int groups = (nst + SG_GROUP - 1) / SG_GROUP;
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sg_addr(tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int b = 0; b < SG_NBUF; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sg_addr(&full[b])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sg_addr(&done[b])), "r"(1));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sg_addr(acc_full)), "r"(1));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sg_addr(acc_free)), "r"(8));
    asm volatile("fence.mbarrier_init.release.cluster;");
    *stop = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  if (warp == 8) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
      auto issue = [&](int s) {
        const int b = s % SG_NBUF, term = s % terms, chunk = c0 + s / terms;
        const uint32_t st = base + b * SG_STAGE, fb = sg_addr(&full[b]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(SG_STAGE) : "memory");
        sg_load(st, &map_a, m0, chunk, parts.a[part][term] * SL, fb);
        sg_load(st + SL * SG_ASLICE, &map_b, n0, chunk, parts.b[part][term] * SL, fb);
      };
      int issued = 0, landed = 0, committed = 0;
      bool ok = true;
      for (; issued < nst && issued < SG_NBUF; ++issued) issue(issued);
      for (int s = 0; s < nst && ok; ++s) {
        const int b = s % SG_NBUF, g = s / SG_GROUP;
        const bool fresh = s % SG_GROUP == 0;
        if (fresh && g > 0) ok = sg_wait(acc_free, (uint32_t)((g - 1) & 1), limit, stop);
        ok = ok && sg_wait(&full[b], (uint32_t)((s / SG_NBUF) & 1), limit, stop);
        if (!ok) break;
        landed = s + 1;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t sa = base + b * SG_STAGE, sb = sa + SL * SG_ASLICE;
        const uint32_t idesc = SG_IDESC | (parts.neg[part][s % terms] ? (1u << 13) : 0u);
#pragma unroll
        for (int l = 0; l < SL; ++l)
#pragma unroll
          for (int i = 0; i <= l; ++i)
            sg_mma(tmem + l * SG_N, sg_desc(sa + i * SG_ASLICE), sg_desc(sb + (l - i) * SG_BSLICE), idesc,
                   fresh && i == 0 ? 0u : 1u);
        sg_commit(&done[b]);
        if (s % SG_GROUP == SG_GROUP - 1 || s == nst - 1) sg_commit(acc_full);
        committed = s + 1;
        // the products of stage s - 1 have read their buffer: refill it while those of
        // stage s run
        if (s >= 1 && issued < nst) {
          const int p = s - 1;
          if (!sg_wait(&done[p % SG_NBUF], (uint32_t)((p / SG_NBUF) & 1), limit, stop)) {
            ok = false;
            break;
          }
          issue(issued++);
        }
      }
      if (!ok) {
        *stop = 1;
        bool drained = true;
        if (committed > 0)
          drained = sg_drain(&done[(committed - 1) % SG_NBUF], (uint32_t)(((committed - 1) / SG_NBUF) & 1));
        for (int s = landed; s < issued; ++s)
          drained = sg_drain(&full[s % SG_NBUF], (uint32_t)((s / SG_NBUF) & 1)) && drained;
        atomicOr(err, drained ? 16 : (16 | 32));
      }
    }
    __syncwarp();
  } else {
    // warp w: rows 32 (w % 4) .. + 31 of the tile (tensor-memory lanes), columns
    // 32 (w / 4) .. + 31
    const int quarter = warp & 3, col = (warp >> 2) * 32;
    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + col;
    long long hi[32], lo[32];  // sum V_l 2^(24 - 8l), l < 4, and sum V_l 2^(48 - 8l), l >= 4
#pragma unroll
    for (int j = 0; j < 32; ++j) hi[j] = lo[j] = 0;
    bool ok = true;
    for (int g = 0; g < groups; ++g) {
      ok = sg_wait(acc_full, (uint32_t)(g & 1), limit, stop);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int l = 0; l < SL; ++l) {
        uint32_t v[32];
        sg_tmem_ld32(taddr + l * SG_N, v);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int t = __float2int_rn(__uint_as_float(v[j]));
          if (l < 4)
            hi[j] += (long long)t * (1 << (24 - 8 * l));
          else
            lo[j] += (long long)t * (1 << (48 - 8 * l));
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sg_addr(acc_free)) : "memory");
    }
    if (ok) {
      const int m = m0 + quarter * 32 + lane;
      if (m < rows_a) {
        double* dst = out + (((size_t)blockIdx.z * parts.n + part) * rows_a + m) * rows_b + n0 + col;
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (n0 + col + j < rows_b) {
            double v = (double)hi[j] * 0x1p-38 + (double)lo[j] * 0x1p-62;
            if (add) v += dst[j];
            dst[j] = v;
          }
      }
    } else if (lane == 0) {
      *stop = 1;
      atomicOr(err, 16);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 8) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---------------------------------------------------------------- slicing

// Binary exponent e with |x| < 2^e for the biased exponent field ex of a row's largest
// element (0: the row is zero or denormal and taken as zero).
__device__ __forceinline__ int row_exp(int ex) { return ex - 1022; }

// Digits of 8 consecutive values of a row, as 8 FP16 numbers per slice.
struct Digits {
  uint32_t z0[8], z1[8];  // low and high words of round(x 2^(55 - e)) + sum_i 128 256^i
  __device__ __forceinline__ void set(int k, double x, int e) {
    const long long bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7FF);
    long long y = 0;
    if (ex != 0) {
      const long long m = (bits & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll;
      const int sh = ex - 1020 - e;  // x 2^(55 - e) = m 2^sh, sh <= 2
      if (sh >= 0)
        y = m << sh;
      else if (sh > -54)
        y = (m + (1ll << (-sh - 1))) >> -sh;
      if (bits < 0) y = -y;
    }
    y += 0x0080808080808080ll;
    z0[k] = (uint32_t)y;
    z1[k] = (uint32_t)(y >> 32);
  }
  // slice i (digit i, 0 the leading one) of the 8 values
  __device__ __forceinline__ uint4 slice(int i) const {
    uint32_t w[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      uint32_t a, b;
      const int sh = 8 * (SL - 1 - i);  // bit of the digit
      if (i == 0) {
        a = z1[2 * p] >> 16;
        b = z1[2 * p + 1] >> 16;
      } else if (sh >= 32) {
        a = (z1[2 * p] >> (sh - 32)) & 0xFFu;
        b = (z1[2 * p + 1] >> (sh - 32)) & 0xFFu;
      } else {
        a = (z0[2 * p] >> sh) & 0xFFu;
        b = (z0[2 * p + 1] >> sh) & 0xFFu;
      }
      // FP16 1024 + v is 0x6400 | v; minus 1152 leaves v - 128
      const uint32_t u = 0x64006400u | a | (b << 16);
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&u), __half2half2(__ushort_as_half(0x6480)));
      w[p] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
};

// Largest biased exponent of each row of x [rows][k] times the weights w [k] over elements
// [blockIdx.y * span, ..); 2047 (infinity or NaN) stays and marks the row.  exps must hold
// zeros.
__global__ void __launch_bounds__(256) k_row_exps(const double* __restrict__ x, size_t k, const double* __restrict__ w,
                                                  size_t span, int* __restrict__ exps) {
  const double* row = x + (size_t)blockIdx.x * k;
  const size_t e0 = (size_t)blockIdx.y * span, e1 = min(k, e0 + span);
  int top = 0;
  for (size_t e = e0 + threadIdx.x; e < e1; e += blockDim.x)
    top = max(top, (int)((__double_as_longlong(row[e] * w[e]) >> 52) & 0x7FF));
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0 && top > 0) atomicMax(exps + blockIdx.x, top);
}

// What k_row_spreads knows of a part of a row: its largest biased exponent, how many values
// are not zero (nor denormal), and the sum of the squares of their leading 16 bits at the
// scale of 2^(top - 1022) (a value v adds (2^16 v)^2 < 2^32).  Integers, so that the sum
// does not load the FP64 pipe and, in a fixed tree, has the same bits each time.
struct RowSpread {
  unsigned long long sum;
  unsigned int count;
  int top;
  __device__ __forceinline__ void rescale(int to) {
    const int d = 2 * (to - top);
    sum = d < 64 ? sum >> d : 0;
    top = to;
  }
  __device__ __forceinline__ void add(RowSpread o) {
    const int t = max(top, o.top);
    rescale(t);
    o.rescale(t);
    sum += o.sum;
    count += o.count;
  }
  __device__ __forceinline__ void warp() {
    for (int off = 16; off > 0; off >>= 1) {
      RowSpread o;
      o.sum = __shfl_down_sync(0xffffffffu, sum, off);
      o.count = __shfl_down_sync(0xffffffffu, count, off);
      o.top = __shfl_down_sync(0xffffffffu, top, off);
      add(o);
    }
  }
};

// Elements [blockIdx.y * span, ..) of row blockIdx.x of x0 and x1, `rows` rows each, into
// part[row][blockIdx.y].  Nothing but denormals has top 0 and a count of 1.
__global__ void __launch_bounds__(256) k_row_spreads(const double2* __restrict__ x0, const double2* __restrict__ x1,
                                                     int rows, size_t k, size_t span, RowSpread* __restrict__ part) {
  __shared__ RowSpread sh[8];
  const int r = blockIdx.x;
  const double2* row = r < rows ? x0 + (size_t)r * k : x1 + (size_t)(r - rows) * k;
  const size_t e0 = (size_t)blockIdx.y * span, e1 = min(k, e0 + span);
  RowSpread a = {0, 0, 0};
  bool tiny = false;
  auto add = [&](double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v) & 0x7FFFFFFFu;
    const int ex = (int)(hi >> 20);
    if (ex > a.top) a.rescale(ex);
    if (ex == 0) {
      tiny = tiny || v != 0.0;
      return;
    }
    const uint32_t m = (((hi & 0xFFFFFu) | 0x100000u) >> 5) >> min(31, a.top - ex);
    a.sum += (unsigned long long)m * m;
    ++a.count;
  };
#pragma unroll 4
  for (size_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const double2 v = row[e];
    add(v.x);
    add(v.y);
  }
  if (a.top == 0) a.count = tiny;
  a.warp();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) a.add(sh[w]);
    part[(size_t)blockIdx.x * gridDim.y + blockIdx.y] = a;
  }
}

// One warp a row: its parts in a fixed tree, its exponent and its spread.
__global__ void __launch_bounds__(128) k_row_spread_of(const RowSpread* __restrict__ part, int rows, int ny, size_t k,
                                                       double chunk, int* __restrict__ exps,
                                                       float* __restrict__ spread) {
  const int r = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  RowSpread a = {0, 0, 0};
  for (int y = lane; y < ny; y += 32) a.add(part[(size_t)r * ny + y]);
  a.warp();
  if (lane != 0) return;
  exps[r] = a.top;
  float g = 1e-30f;  // a row of zeros: exact in any way
  if (a.top == 2047 || (a.top == 0 && a.count > 0)) {
    g = CUDART_INF_F;
  } else if (a.count > 0) {
    const double n = fmax(1.0, chunk * (double)a.count / (2.0 * (double)k));
    g = (float)(65536.0 * sqrt((double)a.count / fmax(1.0, (double)a.sum) / sqrt(n)));
  }
  spread[r] = g;
}

// Slices of elements [k0, k0 + 16 nchunk) of every row (zeros past k), COMP planes:
// out[plane * SL + slice][chunk][row][16].  Two threads a chunk and row, eight elements
// each, rows fastest, so that a warp's stores are contiguous.
template <int COMP>
__global__ void __launch_bounds__(128) k_slice_rows(const double* __restrict__ x, size_t stride, size_t k, size_t k0,
                                                    const double* __restrict__ w, int rows, int nchunk,
                                                    const int* __restrict__ exps, __half* __restrict__ out) {
  const size_t total = (size_t)nchunk * rows * 2;
  const size_t plane = (size_t)nchunk * rows * SG_K;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int half = (int)(t & 1);
    const size_t rc = t >> 1;
    const int row = (int)(rc % rows), chunk = (int)(rc / rows);
    const int ex = exps[row];
    const int e = row_exp(ex);
    const size_t kb = k0 + (size_t)chunk * SG_K + half * 8;
    const double* src = x + (size_t)row * stride * COMP;
    Digits d[COMP];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const size_t kk = kb + q;
#pragma unroll
      for (int c = 0; c < COMP; ++c) {
        double v = (kk < k && ex > 0 && ex < 2047) ? src[kk * COMP + c] : 0.0;
        if (w && kk < k) v *= w[kk];
        d[c].set(q, v, e);
      }
    }
    __half* dst = out + ((size_t)chunk * rows + row) * SG_K + half * 8;
#pragma unroll
    for (int c = 0; c < COMP; ++c)
#pragma unroll
      for (int i = 0; i < SL; ++i) *reinterpret_cast<uint4*>(dst + (c * SL + i) * plane) = d[c].slice(i);
  }
}

// Slices of the Chebyshev table cos(n th_e), x_e = E_e / dE = cos th_e, rows e, n < m
// (zeros past it, and in rows with |x_e| >= 1), scaled by 2^0: out[slice][chunk][e][16].
// A thread runs through 64 orders of one energy by rotations of th, from a first angle
// n0 th whose rounding is taken into account to first order.  M = 500, NE = 1001: 54 us,
// the FP64 pipe's (4 multiply-adds an entry, an angle every 64); the table in memory, one
// acos and cosine an entry, took 874.
__global__ void __launch_bounds__(128) k_cos_slices(const double* __restrict__ E, int ne, double dE, int m,
                                                    int nchunk, __half* __restrict__ out) {
  const int groups = (nchunk + 3) / 4;
  const size_t total = (size_t)groups * ne, plane = (size_t)nchunk * ne * SG_K;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int e = (int)(t % ne), g = (int)(t / ne);
    const double x = E[e] / dE;  // as the energy factor has it: an ulp of x is n ulp / sin th of an angle
    const bool in = fabs(x) < 1.0;
    const double th = in ? acos(x) : 0.0, sx = in ? sqrt((1.0 - x) * (1.0 + x)) : 0.0;
    const double n0 = 64.0 * g, a = n0 * th, da = fma(n0, th, -a);
    double sn, cn;
    sincos(a, &sn, &cn);
    const double c0 = cn;
    cn = fma(-da, sn, cn);
    sn = fma(da, c0, sn);
    for (int c = 4 * g; c < min(nchunk, 4 * g + 4); ++c)
      for (int half = 0; half < 2; ++half) {
        Digits d;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int n = c * SG_K + half * 8 + q;
          d.set(q, in && n < m ? fmin(1.0, fmax(-1.0, cn)) : 0.0, 0);
          const double v = fma(cn, x, -sn * sx);
          sn = fma(sn, x, cn * sx);
          cn = v;
        }
        __half* dst = out + ((size_t)c * ne + e) * SG_K + half * 8;
#pragma unroll
        for (int i = 0; i < SL; ++i) *reinterpret_cast<uint4*>(dst + i * plane) = d.slice(i);
      }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
    return (e == cudaSuccess && q == cudaDriverEntryPointSuccess) ? (PFN_cuTensorMapEncodeTiled_v12000)p : nullptr;
  }();
  if (!fn) throw Error(GQT_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
  return fn;
}

CUtensorMap slice_map(const SliceOperand& o, int nchunk, int box_rows) {
  CUtensorMap map;
  const cuuint64_t dims[4] = {(cuuint64_t)SG_K, (cuuint64_t)o.rows, (cuuint64_t)nchunk, (cuuint64_t)o.planes * SL};
  const cuuint64_t strides[3] = {(cuuint64_t)SG_K * 2, (cuuint64_t)o.rows * SG_K * 2,
                                 (cuuint64_t)nchunk * o.rows * SG_K * 2};
  const cuuint32_t box[4] = {(cuuint32_t)SG_K, (cuuint32_t)box_rows, 1, (cuuint32_t)SL}, estr[4] = {1, 1, 1, 1};
  const CUresult r = encoder()(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(o.data), dims, strides, box,
                               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw Error(GQT_ECUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return map;
}

}  // namespace

size_t slice_bytes(int rows, int planes, int nchunk) { return (size_t)planes * SL * nchunk * rows * SG_K * 2; }

// CTAs a row: a few per SM in all, at least 4096 elements each
static size_t row_parts(int rows, size_t k) {
  const size_t want = std::max<size_t>(1, (size_t)sm_count() * 8 / rows);
  return std::min<size_t>(want, (k + 4095) / 4096);
}
void launch_row_exps(const double* x, int rows, size_t k, const double* w, int* exps, cudaStream_t st) {
  check_cuda(cudaMemsetAsync(exps, 0, (size_t)rows * sizeof(int), st), "row exponents");
  const size_t ny = row_parts(rows, k), span = (k + ny - 1) / ny;
  k_row_exps<<<dim3(rows, (unsigned)ny), 256, 0, st>>>(x, k, w, span, exps);
  check_launch("k_row_exps");
}

size_t row_spread_bytes(int rows, size_t k) {
  return (size_t)2 * rows * row_parts(2 * rows, k) * sizeof(RowSpread);
}

void launch_row_spreads(const double* x0, const double* x1, int rows, size_t k, double chunk, void* scratch, int* exps,
                        float* spread, cudaStream_t st) {
  const size_t ny = row_parts(2 * rows, k), span = (k + ny - 1) / ny;
  k_row_spreads<<<dim3(2 * rows, (unsigned)ny), 256, 0, st>>>((const double2*)x0, (const double2*)x1, rows, k, span,
                                                              (RowSpread*)scratch);
  check_launch("k_row_spreads");
  k_row_spread_of<<<(2 * rows + 3) / 4, 128, 0, st>>>((const RowSpread*)scratch, 2 * rows, (int)ny, k, chunk, exps,
                                                      spread);
  check_launch("k_row_spread_of");
}

void launch_slice_rows(const double* x, int comp, int rows, size_t stride, size_t k, size_t k0, const double* w,
                       int nchunk, const int* exps, void* out, cudaStream_t st) {
  const size_t total = (size_t)nchunk * rows * 2;
  const int grid = (int)std::min<size_t>((total + 127) / 128, (size_t)sm_count() * 32);
  if (comp == 2)
    k_slice_rows<2><<<grid, 128, 0, st>>>(x, stride, k, k0, w, rows, nchunk, exps, (__half*)out);
  else
    k_slice_rows<1><<<grid, 128, 0, st>>>(x, stride, k, k0, w, rows, nchunk, exps, (__half*)out);
  check_launch("k_slice_rows");
}

void launch_cos_slices(const double* E, int ne, double dE, int m, int nchunk, void* out, cudaStream_t st) {
  const size_t total = (size_t)((nchunk + 3) / 4) * ne;
  k_cos_slices<<<(int)std::min<size_t>((total + 127) / 128, (size_t)sm_count() * 32), 128, 0, st>>>(
      E, ne, dE, m, nchunk, (__half*)out);
  check_launch("k_cos_slices");
}

int slice_splits(int rows_a, int rows_b, int parts, int nchunk) {
  // splits of the contraction: at least 16 chunks each; among the counts up to four
  // waves of one CTA per SM, the one with the least work per SM (a chunk's products and
  // about five chunks' worth of start, finish and result traffic per CTA)
  const long long tiles = (long long)((rows_a + SG_M - 1) / SG_M) * ((rows_b + SG_N - 1) / SG_N) * parts;
  const long long sms = sm_count();
  const long long top = std::max<long long>(1, std::min<long long>((nchunk + 15) / 16, (4 * sms + tiles - 1) / tiles));
  long long best = 1;
  double cost = 1e300;
  for (long long s = 1; s <= top; ++s) {
    const long long per = (nchunk + s - 1) / s, used = (nchunk + per - 1) / per;
    const double c = (double)((tiles * used + sms - 1) / sms) * (double)(per + 5);
    if (c < cost * (1 - 1e-9)) cost = c, best = used;
  }
  return (int)best;
}

void launch_slice_gemm(const SliceOperand& a, const SliceOperand& b, const SliceParts& parts, int nchunk, int splits,
                       double* out, bool add, int* err, int limit, cudaStream_t st) {
  const CUtensorMap ma = slice_map(a, nchunk, SG_M), mb = slice_map(b, nchunk, SG_N);
  check_cuda(cudaFuncSetAttribute(k_slice_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM),
             "smem attribute");
  const int per = (nchunk + splits - 1) / splits;
  const dim3 grid((a.rows + SG_M - 1) / SG_M, (unsigned)((b.rows + SG_N - 1) / SG_N) * parts.n, splits);
  k_slice_gemm<<<grid, SG_THREADS, SG_SMEM, st>>>(ma, mb, parts, a.rows, b.rows, nchunk, per, out, add ? 1 : 0, err,
                                              limit);
  check_launch("k_slice_gemm");
}

}  // namespace gqt
