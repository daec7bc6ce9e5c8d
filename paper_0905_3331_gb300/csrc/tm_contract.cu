// tm_contract.cu -- meson contraction of a point-source propagator (tm_meson_contract).
//
// The correlators of Sec. 4.3 (one-end trick) are, for a point source at the origin,
//   C_PG(t) = sum_{x, x_t = t} tr[ G(x,0)^dag G(x,0) G~ ]  with G~ = Gamma gamma5 on source spin,
// where G(x,0) is the 12 x 12 spin-colour propagator (column j = the solution for the source
// of spin-colour j).  This file computes the timeslice sums of its Gram matrix
//   A_t[j][k] = sum_{x, x_t = t} <psi^(j)(x), psi^(k)(x)>   (conjugate on j),
// from which every C_PG(t) follows as a 12 x 12 trace (tm_correlator, below).  Deterministic.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "tm_dslash_fx.cuh"
#include "tm_internal.cuh"

namespace tmq {

// The contraction is a Gram matrix per timeslice, 24 x 24 real (12 propagators x re, im) over the 12
// spatial components of every site.  In FP64 it is 3744 multiply-adds per site against 2304 bytes: 5.5 ms
// on 24^3 x 48 at 75% of the FP64 units, 24 times the time of its bytes.  GB300's tensor cores have no
// FP64 rate to speak of, so it runs on the fp16 ones with the operands split into exact digits (the
// scheme of Ozaki, Ogita, Oishi and Rump 2012):
//   a real is v 2^(E - 1077), v a 55-bit integer (rounded), E one exponent per propagator (at least one
//   above the largest real of the tiles it serves, and at most four where it is set anew, so that those
//   reals keep 51 to 53 bits and smaller ones what lies above the same place); v = sum_i d_i 256^(6 - i), seven balanced digits
//   -128 <= d_i < 128, each exact in fp16;
//   sum_k v_r v_c = sum_{i + j <= 7} 256^(12 - i - j) sum_k d_i(r, k) d_j(c, k),
// every inner sum an integer below 1024 2^14 = 2^24, exact in FP32, over at most CK = 1024 components;
// the left-out products i + j > 7 come to ~2^-62 of the largest real squared per component.  The sums are
// drained to 64-bit integers, combined, and added in FP64 with the exponents.
// One tcgen05.mma of 128 x 176 x 16 takes all digits of all rows against each other: operand row
// 24 i + 2 j + part holds digit i of propagator j's re or im part, A is rows 0..127 and B rows 0..175 of
// the same tile in shared memory (K-major, no swizzle: core matrices of 8 rows x 16 bytes).  Digits i > 3
// of A would repeat, transposed, what B's columns hold: the drain reads rows 0..95 only.
// A tile is CT components.  Bulk copies bring the raw tiles into shared memory two ahead; the block
// converts one while the tensor core works on its last one and the other resident block's (two blocks
// per SM: 106 kB of shared memory and 256 TMEM columns each).
// Relative error of A against 113-bit arithmetic on 4 x 10^3, FP64 sums and this: Gaussian propagators
// 2.6e-16, 7.2e-17; decaying in time 3.2e-16, 7.2e-17; peaked at a point source 7.0e-16, 1.6e-16.
constexpr int NPAIR = 78;              // pairs j <= k of 12 indices
constexpr int CT = 128;                // components per tile: 16 groups of 8
constexpr int CNT = 24 * (CT / 8);     // threads: one per operand row and 8 components
constexpr int CK = 1024;               // components per exact sum
constexpr int C_ROWG = 22;             // row groups of 8: 176 operand rows
constexpr int C_LBO = C_ROWG * 128;    // bytes between k groups; 128 between row groups
constexpr int C_RED = 4 * 24 * 24 * 3 * 8;  // the drained sums, in the operand tile's place
constexpr int C_OPER = CT / 8 * C_LBO > C_RED ? CT / 8 * C_LBO : C_RED;
constexpr int C_ROWP = CT * 16 + 32;   // bytes per propagator of a raw tile (padded: conflict-free reads)
constexpr int C_RAW = 12 * C_ROWP;
constexpr int C_SMEM = C_OPER + 2 * C_RAW;
constexpr int C_COLS = 256;            // TMEM columns per block

__device__ __forceinline__ void pair_of(int p, int* j, int* k) {
  int jj = 0, n = 12;
  while (p >= n) {
    p -= n;
    ++jj;
    --n;
  }
  *j = jj;
  *k = jj + p;
}

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major, no swizzle
__device__ __forceinline__ unsigned long long c_desc(unsigned addr) {
  return (unsigned long long)((addr & 0x3ffff) >> 4) | ((unsigned long long)(C_LBO >> 4) << 16) |
         ((unsigned long long)(128 >> 4) << 32) | (1ull << 46);
}
// kind::f16: FP32 accumulators, fp16 operands, both K-major, M = 128, N = 176
constexpr unsigned C_IDESC = (1u << 4) | ((8u * C_ROWG / 8) << 17) | ((128u / 16) << 24);

__device__ __forceinline__ void c_mma(unsigned tmem, unsigned long long a, unsigned long long b, bool add) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(tmem), "l"(a), "l"(b), "r"(C_IDESC), "r"((int)add)
      : "memory");
}

// Bounded wait for a phase of the barrier: false if it did not complete (~0.1 s and more; a tile takes ~2 us).
__device__ __forceinline__ bool c_wait(unsigned bar, unsigned parity) {
  for (int n = 0; n < (1 << 20); ++n) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (n > (1 << 14)) __nanosleep(100);
  }
  return false;
}

// |x| as an integer of exponent E, v 2^(E - 1077), rounded, with 128 added to each of its seven balanced
// digits
__device__ __forceinline__ unsigned long long c_digits(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int sh = E - (int)((hi >> 20) & 0x7ffu);  // >= 1; zero and denormal reals are shifted out
  const unsigned long long w =
      ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 35) | ((unsigned long long)lo << 3);
  unsigned long long q;
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(w), "r"(sh));  // PTX clamps shifts above 63: 0
  return (q + (2 * 0x80808080808080ull + 1)) >> 1;
}

// Eight reals of one operand row: the seven digit rows' 16 bytes each.  The digits of |x| take x's sign in
// the fp16 operation that removes their offset.
__device__ __forceinline__ void c_store_row(char* tile, int row, const double x[8], int E) {
  unsigned d[7][4];  // digit i: components 2 m, 2 m + 1 in word m
  const __half2 off = __half2half2(__ushort_as_half(0xe480));  // -1152
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const unsigned long long a = c_digits(x[2 * m], E), b = c_digits(x[2 * m + 1], E);
    const unsigned w[2][2] = {{(unsigned)a, (unsigned)b}, {(unsigned)(a >> 32), (unsigned)(b >> 32)}};
    const unsigned sb = (__byte_perm(__double2hiint(x[2 * m]), __double2hiint(x[2 * m + 1]), 0x7632) & 0x80008000u) | 0x3c003c00u;
    const __half2 sgn = *reinterpret_cast<const __half2*>(&sb), soff = __hmul2(sgn, off);  // +-1, -+1152
#pragma unroll
    for (int byte = 0; byte < 7; ++byte) {
      // bytes (a.b, b.b) of two digits, then 0x64 above each: the halves 1024 + digit + 128
      const unsigned g = __byte_perm(w[byte / 4][0], w[byte / 4][1], (byte & 2) ? 0x7362 : 0x5140);
      const unsigned h = __byte_perm(g, 0x64646464u, (byte & 1) ? 0x4342 : 0x4140);
      const __half2 v = __hfma2(*reinterpret_cast<const __half2*>(&h), sgn, soff);
      d[6 - byte][m] = *reinterpret_cast<const unsigned*>(&v);
    }
  }
#pragma unroll
  for (int i = 0; i < 7; ++i) *reinterpret_cast<uint4*>(tile + (24 * i + row) * 16) = make_uint4(d[i][0], d[i][1], d[i][2], d[i][3]);
}

// s += a b in 64 bits
__device__ __forceinline__ void c_mad(long long& s, int a, int b) {
  unsigned lo = (unsigned)s, hi = (unsigned)((unsigned long long)s >> 32);
  asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(b));
  s = (long long)(((unsigned long long)hi << 32) | lo);
}

// partial[t][bx][pair] (complex): block bx of timeslice t sums its tiles of components.
// 24^3 x 48: 5.53 -> 0.72 ms (1.53 GB: 225 us of HBM).  With two barriers per tile, the next tile read after
// them, it was 0.77; conflict-free raw rows and the sign taken in fp16 (an eighth of the instructions)
// brought 0.05.  Bound by the latency of a block's steps, which the other resident block covers in part:
// issue 43% active, ALU 45%, tensor core 22%, DRAM 27%; a third of a block's clocks go into the drains (one
// per eight tiles), half into conversion and reading, the rest into the barrier and the waits.
__global__ void __launch_bounds__(CNT, 2) contract_kernel(const double* __restrict__ props, size_t V, int spatial,
                                                          int nbx, double* __restrict__ partial) {
  extern __shared__ __align__(128) char smem[];
  __shared__ int tmax[2][4][12];  // largest biased exponents of a tile (by parity): per quarter of it and propagator
  __shared__ int Es[12];
  __shared__ __align__(8) unsigned long long bar, full[2];
  __shared__ unsigned taddr;
  const int t = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // this thread's operand row, part prt of propagator j, and its 8 components of a tile: 16 m + kp.  (Which
  // of a tile's components sits where along K does not matter.)  The eight lanes of a store phase write
  // the eight rows of a core matrix.
  const int prt = lane & 1, j = 4 * (warp % 3) + ((lane >> 1) & 3), kp = 4 * (warp / 3) + (lane >> 3);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&taddr)), "n"(C_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (unsigned long long* b : {&bar, &full[0], &full[1]})
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(b)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 12) Es[tid] = 0;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = taddr;

  // outputs: thread 2 p + part < 156 owns the re (part 0) or im sum of pair p
  int pj = 0, pk = 0;
  const int part = tid & 1;
  if (tid < 2 * NPAIR) pair_of(tid >> 1, &pj, &pk);
  double acc = 0.0;

  const int ncomp = spatial * 12, ntile = (ncomp + CT - 1) / CT;
  // warp 11: raw tile tl to buffer b, lane r propagator r
  auto fetch = [&](int tl, int b) {
    const unsigned bytes = 16u * (unsigned)min(CT, ncomp - tl * CT);
    if (lane == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&full[b])), "r"(12 * bytes)
                   : "memory");
    __syncwarp();
    if (lane < 12)
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              smem_addr(smem + C_OPER + b * C_RAW + lane * C_ROWP)),
          "l"(props + (((size_t)lane * V + (size_t)t * spatial) * 12 + (size_t)tl * CT) * 2), "r"(bytes),
          "r"(smem_addr(&full[b]))
          : "memory");
  };
  if (warp == 11)
    for (int n = 0; n < 2; ++n)
      if ((int)blockIdx.x + n * nbx < ntile) fetch(blockIdx.x + n * nbx, n);
  int E = 0;          // the exponent of propagator j in the sums
  int summed = 0;     // components in the sums
  unsigned phase = 0; // commits waited for
  bool pending = false, ok = true;
  double x[8];        // this thread's components of the tile in hand
  int e = 0;          // their warp's largest exponent
  bool bad = false;   // the tile has a real that the sums cannot take
  // tile number n of this block, from its raw buffer
  auto take = [&](int tl, int n) {
    ok = c_wait(smem_addr(&full[n & 1]), (n >> 1) & 1) && ok;
    const char* raw = smem + C_OPER + (n & 1) * C_RAW + j * C_ROWP + 8 * prt + 16 * kp;
    if ((tl + 1) * CT <= ncomp) {  // uniform
#pragma unroll
      for (int m = 0; m < 8; ++m) x[m] = *reinterpret_cast<const double*>(raw + 256 * m);
    } else {
#pragma unroll
      for (int m = 0; m < 8; ++m)
        x[m] = tl * CT + kp + 16 * m < ncomp ? *reinterpret_cast<const double*>(raw + 256 * m) : 0.0;
    }
    unsigned u = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) u = max(u, (unsigned)__double2hiint(x[m]) & 0x7fffffffu);
    e = (int)(u >> 20);
    bool zero = false;
    if (u == 0) {
      unsigned any = 0;
#pragma unroll
      for (int m = 0; m < 8; ++m) any |= (unsigned)__double2loint(x[m]);
      zero = any == 0;
    }
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 8));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
    if ((lane & 25) == 0) tmax[n & 1][warp / 3][j] = e;
    bad = e > FX_EMAX || (!zero && e < FX_EMIN);
  };
  // one barrier per tile: the operand tile is written, and the next tile is in registers (its raw buffer
  // is free) and known to fit the exponents or not
  take(blockIdx.x, 0);
  bool flag = __syncthreads_or(bad || e != 0) != 0;
  if (warp == 11 && (int)blockIdx.x + 2 * nbx < ntile) fetch(blockIdx.x + 2 * nbx, 0);
  int n = 0;
  for (int tl = blockIdx.x;; tl += nbx, ++n) {  // one more round drains
    const bool last = tl >= ntile;
    bool direct = false, drain = last || summed + CT > CK;
    if (flag || drain) {
      direct = __syncthreads_or(!last && bad) != 0;  // the tile in FP64, outside the sums
      drain = last || !direct;
      if (!last) {
#pragma unroll
        for (int m = 0; m < 4; ++m) e = max(e, tmax[n & 1][m][j]);
      }
    }
    if (drain) {
      // ---- drain the sums
      if (pending) {
        ok = c_wait(smem_addr(&bar), phase & 1) && ok;
        phase ^= 1;
        pending = false;
      }
      if (summed > 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        long long* red = reinterpret_cast<long long*>(smem);  // [i][24][24][hi, lo, z]
        const int quad = warp & 3;
        if (quad < 3) {  // TMEM lanes 32 quad ..: row = 24 i + r; columns 24 j + c0 .. c0 + 3
          const int row = 32 * quad + lane, i = row / 24, r = row % 24;
#pragma unroll 1
          for (int c0 = 8 * (warp >> 2), c1 = c0 + 8; c0 < c1; c0 += 4) {
            long long hi[4], lo[4], z[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) hi[c] = lo[c] = z[c] = 0;
            unsigned d[7][4];
#pragma unroll
            for (int jj = 0; jj < 7; ++jj)
              asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                           : "=r"(d[jj][0]), "=r"(d[jj][1]), "=r"(d[jj][2]), "=r"(d[jj][3])
                           : "r"(tmem + ((unsigned)(32 * quad) << 16) + 24 * jj + c0));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int jj = 0; jj < 7; ++jj) {
              const int w = i + jj;
              const int mh = w <= 2 ? 1 << (8 * (2 - w)) : 0;              // hi: weights 256^(2 - w)
              const int ml = (w >= 4 && w <= 7) ? 1 << (8 * (7 - w)) : 0;  // lo: 256^(7 - w)
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const int v = __float2int_rn(__uint_as_float(d[jj][c]));
                if (jj < 3) c_mad(hi[c], v, mh);
                c_mad(lo[c], v, ml);
                if (jj < 4 && w == 3) lo[c] += (long long)v << 32;
                if (jj >= 4) c_mad(z[c], v, ml);  // (i, jj) stands for (jj, i) of the transposed entry too
              }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              long long* q = red + ((i * 24 + r) * 24 + c0 + c) * 3;
              q[0] = hi[c];
              q[1] = lo[c];
              q[2] = z[c];
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (tid < 2 * NPAIR) {
          // G[r][c] = Y[r][c] + Z[c][r]; re = G[2j][2k] + G[2j+1][2k+1], im = G[2j][2k+1] - G[2j+1][2k]
          long long h = 0, l = 0;
#pragma unroll
          for (int n = 0; n < 2; ++n) {
            const int r = 2 * pj + n, c = 2 * pk + (n ^ part);
            long long hs = 0, ls = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const long long* q = red + ((i * 24 + r) * 24 + c) * 3;
              hs += q[0];
              ls += q[1] + red[((i * 24 + c) * 24 + r) * 3 + 2];
            }
            h += (n && part) ? -hs : hs;
            l += (n && part) ? -ls : ls;
          }
          // units 256^5 2^(Ej - 1077) 2^(Ek - 1077)
          const double v = fma((double)h, 0x1p40, (double)l);
          const int ej = Es[pj], ek = Es[pk];
          if (ej > 0 && ek > 0)
            acc = fma(v * __hiloint2double((ej - 54 + 20) << 20, 0), __hiloint2double((ek - 54 + 20) << 20, 0), acc);
        }
        summed = 0;
      }
      __syncthreads();
      if (!last) {
        // raised when a real does not fit, lowered only when three bits too high: the largest real of a
        // tile moves between two binades, and an exponent that followed it would drain at every tile
        if (e != 0 && (e >= E || e + 4 < E)) E = e + 1;
        if ((lane & 25) == 0 && warp < 3) Es[j] = E;
      }
    }
    if (last) break;
    if (direct) {  // a non-finite real, or one outside the exponent range: this tile in FP64
      if (tid < 2 * NPAIR) {
        const double2* a = reinterpret_cast<const double2*>(props) + ((size_t)pj * V + (size_t)t * spatial) * 12;
        const double2* b = reinterpret_cast<const double2*>(props) + ((size_t)pk * V + (size_t)t * spatial) * 12;
        for (int k = tl * CT; k < min(ncomp, (tl + 1) * CT); ++k) {
          const double2 p = a[k], q = b[k];
          acc = part ? fma(p.x, q.y, fma(-p.y, q.x, acc)) : fma(p.x, q.x, fma(p.y, q.y, acc));
        }
      }
    } else {
      // ---- the tile's digits, once the tensor core has read the last ones
      if (pending) {
        ok = c_wait(smem_addr(&bar), phase & 1) && ok;
        phase ^= 1;
      }
      c_store_row(smem + kp * C_LBO, 2 * j + prt, x, E == 0 ? FX_BAD : E);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    e = 0;
    bad = false;
    if (tl + nbx < ntile) take(tl + nbx, n + 1);
    flag = __syncthreads_or(bad || (e >= E && e != 0)) != 0;
    if (warp == 11 && tl + 3 * nbx < ntile) fetch(tl + 3 * nbx, (n + 1) & 1);
    if (direct) continue;
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned a = smem_addr(smem);
#pragma unroll
      for (int k = 0; k < CT / 16; ++k) {
        const unsigned long long d = c_desc(a + k * 2 * C_LBO);
        c_mma(tmem, d, d, summed > 0 || k > 0);
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(&bar))
                   : "memory");
    }
    pending = true;
    summed += CT;
  }
  if (tid < 2 * NPAIR)
    partial[(((size_t)t * nbx + blockIdx.x) * NPAIR + (tid >> 1)) * 2 + part] =
        ok ? acc : __longlong_as_double(0x7ff8000000000000ll);  // NaN if a wait ran out
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(C_COLS) : "memory");
}

// out[t][j][k] = sum over bx of partial[t][bx][pair]; out[t][k][j] = its conjugate.  One warp per (t, pair):
// lane l adds partials l, l + 32, ..., then a fixed shuffle tree (24^3 x 48: 10 -> 3 us against one thread
// adding all of them in turn, whose roundings also piled up when the partials are alike).
__global__ void __launch_bounds__(128) contract_finish_kernel(const double* __restrict__ partial, int nbx, int T,
                                                              double* __restrict__ out) {
  const int i = (blockIdx.x * 128 + threadIdx.x) >> 5, lane = threadIdx.x & 31;  // (t, pair)
  if (i >= T * NPAIR) return;
  const int t = i / NPAIR, p = i % NPAIR;
  double re = 0.0, im = 0.0;
  for (int b = lane; b < nbx; b += 32) {
    const double* q = partial + (((size_t)t * nbx + b) * NPAIR + p) * 2;
    re += q[0];
    im += q[1];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_down_sync(0xffffffffu, re, o);
    im += __shfl_down_sync(0xffffffffu, im, o);
  }
  if (lane != 0) return;
  int j, k;
  pair_of(p, &j, &k);
  double* o = out + (size_t)t * 12 * 12 * 2;
  o[(j * 12 + k) * 2] = re;
  o[(j * 12 + k) * 2 + 1] = im;
  o[(k * 12 + j) * 2] = re;
  o[(k * 12 + j) * 2 + 1] = j == k ? im : -im;
}

// C[g][t] = tr[A_t (X_g (x) 1_colour)] = sum_{s, s', c} A_t[3s+c][3s'+c] X_g[s'][s]: one thread
// per (g, t), the 48 complex products summed in the order s, s', c (FP64, deterministic).
__global__ void correlator_kernel(const double* __restrict__ A, const double* __restrict__ X, int T, int ngamma,
                                  double* __restrict__ C) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // (g, t)
  if (i >= T * ngamma) return;
  const int g = i / T, t = i % T;
  const double* a = A + (size_t)t * 144 * 2;
  const double* x = X + (size_t)g * 16 * 2;
  double re = 0.0, im = 0.0;
  for (int s = 0; s < 4; ++s)
    for (int sp = 0; sp < 4; ++sp) {
      const double xr = x[(sp * 4 + s) * 2], xi = x[(sp * 4 + s) * 2 + 1];
      for (int c = 0; c < 3; ++c) {
        const int jk = (3 * s + c) * 12 + (3 * sp + c);
        const double ar = a[jk * 2], ai = a[jk * 2 + 1];
        re = fma(ar, xr, fma(-ai, xi, re));
        im = fma(ar, xi, fma(ai, xr, im));
      }
    }
  C[(size_t)i * 2] = re;
  C[(size_t)i * 2 + 1] = im;
}

}  // namespace tmq

using namespace tmq;

extern "C" tm_status tm_correlator(tm_lattice lat, const double* A, const double* X, int ngamma, double* C,
                                   void* stream) {
  if (!lat || !A || !X || !C || ngamma < 1 || ngamma > 1024)
    return set_error(TM_ERR_ARG, "tm_correlator: NULL argument or ngamma not in 1..1024");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int T = lat->T;
  tm_status st;
  const double* dA = static_cast<const double*>(stage_in(lat, WS_STAGE_IN, A, (size_t)T * 144 * 2 * sizeof(double), s, &st));
  if (st != TM_OK) return st;
  const double* dX = static_cast<const double*>(stage_in(lat, WS_GAMMA, X, (size_t)ngamma * 16 * 2 * sizeof(double), s, &st));
  if (st != TM_OK) return st;
  const size_t out_bytes = (size_t)ngamma * T * 2 * sizeof(double);
  double* dC = static_cast<double*>(stage_out(lat, WS_STAGE_OUT, C, out_bytes, &st));
  if (st != TM_OK) return st;
  const int n = T * ngamma;
  correlator_kernel<<<(n + 127) / 128, 128, 0, s>>>(dA, dX, T, ngamma, dC);
  count_launch();
  if ((st = cuda_check(cudaGetLastError(), "tm_correlator")) != TM_OK) return st;
  return stage_out_finish(C, dC, out_bytes, s);
}

extern "C" tm_status tm_meson_contract(tm_lattice lat, const double* props, double* out, void* stream) {
  if (!lat || !props || !out) return set_error(TM_ERR_ARG, "tm_meson_contract: NULL argument");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t V = lat->V;
  const int spatial = lat->L * lat->L * lat->L;
  const int T = lat->T;
  tm_status st;
  const double* dp = static_cast<const double*>(stage_in(lat, WS_STAGE_IN, props, 12 * V * 24 * sizeof(double), s, &st));
  if (st != TM_OK) return st;
  if (reinterpret_cast<uintptr_t>(dp) % 16 != 0)
    return set_error(TM_ERR_ARG, "tm_meson_contract: device props must be 16-byte aligned");
  const size_t out_bytes = (size_t)T * 12 * 12 * 2 * sizeof(double);
  double* dout = static_cast<double*>(stage_out(lat, WS_STAGE_OUT, out, out_bytes, &st));
  if (st != TM_OK) return st;
  // two blocks per SM over all timeslices (one wave); each block loops over its tiles.  Rounded down: above 152
  // timeslices one block each, which leaves up to half of the slots empty (160 x 12^3 544 us; 48 x 24^3, 2.4 times
  // the sites, 726)
  const int ntile = (spatial * 12 + CT - 1) / CT;
  const int nbx = std::max(1, std::min(ntile, 2 * 152 / T));
  double* partial =
      static_cast<double*>(workspace(lat, WS_X0 + 1, (size_t)T * nbx * NPAIR * 2 * sizeof(double), &st));
  if (st != TM_OK) return st;
  if ((st = cuda_check(cudaFuncSetAttribute(contract_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C_SMEM),
                       "tm_meson_contract: shared memory")) != TM_OK)
    return st;
  contract_kernel<<<dim3(nbx, T), CNT, C_SMEM, s>>>(dp, V, spatial, nbx, partial);
  count_launch();
  const int n = T * NPAIR;
  contract_finish_kernel<<<(n + 3) / 4, 128, 0, s>>>(partial, nbx, T, dout);
  count_launch();
  if ((st = cuda_check(cudaGetLastError(), "tm_meson_contract")) != TM_OK) return st;
  return stage_out_finish(out, dout, out_bytes, s);
}
