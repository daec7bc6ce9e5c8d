// tm_dslash_fx.cuh -- the hopping sum of FP64 spinors and 18-real links in 64-bit fixed point on the
// integer units.
//
// GB300 retires 1.6 FP64 FMAs per clock and SM, but ~23-47 32x32+64-bit integer multiply-adds
// (IMAD.WIDE) and ~55 64-bit adds or 32-bit shifts (measured).  In FP64 the sum takes 888 FP64
// instructions per output site, ~550 clocks of that pipe; here it takes 1728 IMAD.WIDE and ~4500 other
// instructions.  One launch (hopping only, warm): 16^3 x 32 125 -> 45 us, 32^3 x 64 1600 -> 560 us; with
// the input already in FX form 32^3 x 64 ~425 us.  It is bound by latency now: issue 40% active, no pipe
// above 35%, DRAM 43% (ncu, 24^3 x 48).
//
// Numbers.  A link real u (|u| <= 1) is stored as v = round(u 2^62) in two signed 32-bit limbs,
// v = uh 2^32 + ul (LinkRecon<double, double, 18>).  A spinor site is 24 integers of a common exponent
// e (a biased FP64 exponent: every real is below 2^(e - 1022)), real = V 2^(e - 1081), |V| < 2^59: the
// site's largest real has six bits more than in FP64, and the others keep every bit down to the same
// absolute place.  Half fields in this form are called FX here; FP64 fields are brought
// to it as they are read.  The sum has an exponent E of its own, at least e + 1 of every neighbour
// added: a neighbour is shifted right by E - e, and the sum when E grows.  A projected real h so
// shifted, |h| < 2^59, is hh 2^32 + hl, hl signed, and
//   u h / 2^64 = uh hh + (uh hl + ul hh) / 2^32 (+ ul hl / 2^64, dropped),
// so the sum is kept in units of 4 2^(E - 1081) = 2^(E - 1079).  Sizes, by Cauchy-Schwarz with the unit
// rows of U: the middle sum of a colour row is below sqrt(6) 2^30 2^31 + 6 2^31 2^27 < 2^62.7, the
// result of a hop below sqrt(6) 2^57, eight hops below 2^61.3.  The dropped terms and the rounding of
// the middle sum come to ~0.4 units per hop (rms), 2^-57 of the largest neighbour real over all eight,
// far below the final rounding to FP64.  Measured against 113-bit arithmetic (4^4, 6^3 x 8, 6^3 x 10):
// relative error of the sum 5.0e-17 on Gaussian fields (FP64 arithmetic: 1.3e-16), 3.9-5.6e-17 on point
// sources, 5.5e-17 with time slices a factor e^1.5 apart, 6-8e-17 with sites of random size over e^40.
// These are relative to the norm.  Entry by entry the error is relative to the largest neighbour real: a
// component 2^-k below its site's largest enters with 59 - k bits (FP64: 53), and not at all from k = 59
// on.  That shows only where links do not mix colours (unit or diagonal links) or the spins of the other
// lane stay apart.  12- and 8-real links keep FP64 arithmetic, and so do the fields that solvers return.
//
// A neighbour read from an FP64 field that has a non-finite real, or whose largest real is outside
// [2^-894, 2^978) without being zero throughout, has no FX form (exponent FX_BAD): its output site takes
// the FP64 form (hop_f64_general).  A site that a solver stores in FX form is held at the lowest exponent
// if its largest real is below 2^-894 (to 2^-953; at least 2^370 below anything that a norm in FP64
// sees), and is NaN to its readers if it has a non-finite real or one from 2^978 on, whose squares have
// left FP64 as well.
#pragma once

#include "tm_internal.cuh"

namespace tmq {

typedef long long fx;

constexpr int FX_EMIN = 128, FX_EMAX = 2000;  // biased exponents of the fixed-point form
constexpr int FX_BAD = 0x7fff;                // exponent of a site without a fixed-point form
constexpr size_t FX_SITE_BYTES = 196;         // FX half field: longlong2 blocks [12][h], then int e[h]

__device__ __forceinline__ const int* fx_exps(const char* base, int h) {
  return reinterpret_cast<const int*>(base + (size_t)192 * h);
}

// The FP64 number with words (lo, hi) times 2^(1081 - E), truncated towards zero; E at least its exponent.
__device__ __forceinline__ fx fx_from(unsigned lo, unsigned hi, int E) {
  const int sh = E - (int)((hi >> 20) & 0x7ffu);  // zero and denormal reals have sh >= 128: shifted out
  const unsigned long long w =
      ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 38) | ((unsigned long long)lo << 6);
  unsigned long long q;
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(w), "r"(sh));  // PTX clamps shifts above 63: 0
  const fx s = (fx)((int)hi >> 31);
  return ((fx)q ^ s) - s;
}

// The exponent of N complex numbers from their words, 0 if all are zero, FX_BAD without a fixed-point form.
template <int N>
__device__ __forceinline__ int fx_exponent(const uint4 w[N]) {
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) m = max(m, max(w[k].y & 0x7fffffffu, w[k].w & 0x7fffffffu));
  const int e = (int)(m >> 20);
  if (e >= FX_EMIN && e <= FX_EMAX) return e;
  unsigned any = m;
#pragma unroll
  for (int k = 0; k < N; ++k) any |= w[k].x | w[k].z;
  return any != 0 ? FX_BAD : 0;
}

// The same of the 2 N numbers of a lane pair, called by whole warps; TINY: the exponent where the largest is below 2^-894.
template <int N, int TINY = FX_BAD>
__device__ __forceinline__ int fx_pair_exponent(const uint4 w[N]) {
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) m = max(m, max(w[k].y & 0x7fffffffu, w[k].w & 0x7fffffffu));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
  const int e = (int)(m >> 20);
  if (e >= FX_EMIN && e <= FX_EMAX) return e;
  unsigned any = m;  // both lanes of the pair come here
#pragma unroll
  for (int k = 0; k < N; ++k) any |= w[k].x | w[k].z;
  any |= __shfl_xor_sync(3u << (threadIdx.x & 30), any, 1);
  return any == 0 ? 0 : (e > FX_EMAX ? FX_BAD : TINY);
}

// The exponent to convert at: that of a zero site (0) shifts everything out.
__device__ __forceinline__ int fx_shift_exponent(int e) { return e == 0 ? FX_BAD : e; }

// The unit 2^(e - 1081) of a site's integers.
__device__ __forceinline__ double fx_stored_unit(int e) {
  return e == FX_BAD ? __longlong_as_double(0x7ff8000000000000ll) : (e == 0 ? 0.0 : __hiloint2double((e - 58) << 20, 0));
}

// What the hopping sum reads: an FP64 half field, an FX half field, or a canonical FP64 field.
constexpr int FXS_HALF = 0, FXS_FX = 1, FXS_CANON = 2;
// Canonical input: (t + z + y + parity) & 1 of the output site, that is the parity of its x (its
// neighbours' sum is the same across t, z and y, the other across x), gamma5 applied or not, and whether
// the field is 16-byte aligned.
struct FxCanon {
  int b, g5;
  bool al;
};

// Six complex numbers at blocks ja .. ja + 2 and jb .. jb + 2 of site i (canonical: its lexicographic
// index), as integers, and the site's exponent.
template <int SRC>
__device__ __forceinline__ int fx_load(const char* in, int h, int i, int ja, int jb, cpx<fx> v[6], const FxCanon& canon) {
  uint4 w[6];
  if (SRC == FXS_CANON) {
    const double* p = reinterpret_cast<const double*>(in) + (size_t)i * 24;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const double2 d = canon_load(p + 2 * (k < 3 ? ja + k : jb + k - 3), canon.al);
      const unsigned m = (k >= 3 && canon.g5) ? 0x80000000u : 0u;  // the partner is a lower spin
      w[k] = make_uint4((unsigned)__double2loint(d.x), (unsigned)__double2hiint(d.x) ^ m, (unsigned)__double2loint(d.y),
                        (unsigned)__double2hiint(d.y) ^ m);
    }
  } else {
    const uint4* p = reinterpret_cast<const uint4*>(in) + i;
#pragma unroll
    for (int k = 0; k < 3; ++k) w[k] = __ldg(p + (size_t)(ja + k) * h);
#pragma unroll
    for (int k = 0; k < 3; ++k) w[3 + k] = __ldg(p + (size_t)(jb + k) * h);
  }
  int e;
  if (SRC == FXS_FX) {
    e = __ldg(fx_exps(in, h) + i);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      v[k] = mk<fx>((fx)(((unsigned long long)w[k].y << 32) | w[k].x), (fx)(((unsigned long long)w[k].w << 32) | w[k].z));
  } else {
    e = fx_pair_exponent<6>(w);  // the site's: its twelve components are the lane pair's
    const int es = fx_shift_exponent(e);
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = mk<fx>(fx_from(w[k].x, w[k].y, es), fx_from(w[k].z, w[k].w, es));
  }
  return e;
}

// Exponent of N FP64 complex numbers, and the one to store the 2 N of a lane pair with.
template <int N>
__device__ __forceinline__ void fx_words(const cpx<double> v[N], uint4 w[N]) {
#pragma unroll
  for (int k = 0; k < N; ++k)
    w[k] = make_uint4((unsigned)__double2loint(v[k].re), (unsigned)__double2hiint(v[k].re),
                      (unsigned)__double2loint(v[k].im), (unsigned)__double2hiint(v[k].im));
}
template <int N>
__device__ __forceinline__ int fx_exponent_f64(const cpx<double> v[N]) {
  uint4 w[N];
  fx_words<N>(v, w);
  return fx_exponent<N>(w);
}
template <int N>
__device__ __forceinline__ int fx_stored_exponent(const cpx<double> v[N]) {
  uint4 w[N];
  fx_words<N>(v, w);
  return fx_pair_exponent<N, FX_EMIN>(w);
}
__device__ __forceinline__ longlong2 fx_pack(cpx<double> v, int e) {
  e = fx_shift_exponent(e);
  return make_longlong2(fx_from((unsigned)__double2loint(v.re), (unsigned)__double2hiint(v.re), e),
                        fx_from((unsigned)__double2loint(v.im), (unsigned)__double2hiint(v.im), e));
}
// x = hi 2^32 + lo, lo signed
struct FxLimbs {
  int hi, lo;
};
__device__ __forceinline__ FxLimbs fx_split(fx x) {
  const unsigned lo = (unsigned)x, hi = (unsigned)((unsigned long long)x >> 32);
  return {(int)(hi + (lo >> 31)), (int)lo};
}
// A 64-bit sum in two words, s += a b.  The mad.lo.cc / madc.hi pair becomes one IMAD.WIDE; written as
// a 64-bit product and sum (or mad.wide) the compiler emits the product and two adds (measured: 1.4
// instructions per multiply-add against 1.9 with mad.wide and 3.1 from C).
struct FxSum {
  unsigned lo, hi;
};
__device__ __forceinline__ void fx_mad(FxSum& s, int a, int b) {
  asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+r"(s.lo), "+r"(s.hi) : "r"(a), "r"(b));
}
__device__ __forceinline__ FxSum fx_mul(int a, int b) {
  unsigned long long p;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
  return {(unsigned)p, (unsigned)(p >> 32)};
}
// The number 1 in a register that the compiler does not know: s += hi * one is one IMAD.WIDE where the
// sign-extended 64-bit add takes three instructions.
__device__ __forceinline__ int fx_one() {
  int v;
  asm("mov.u32 %0, 1;" : "=r"(v));
  return v;
}
__device__ __forceinline__ fx fx_value(FxSum s) { return (fx)(((unsigned long long)s.hi << 32) | s.lo); }
// a + (m ? -x : x), m = 0 or -1
__device__ __forceinline__ fx fx_addsgn(fx a, fx x, int m) { return a + (x ^ (fx)m) + (fx)(m & 1); }

constexpr int FX_LINK_BYTES = 18 * 8;  // a link's 9 complex entries, words (re.lo, re.hi, im.lo, im.hi)

// u = U h (S > 0) or U^dag h for a colour vector, h >> sh, in units of 2^(E - 1079)
template <int S, class Link>
__device__ __forceinline__ void fx_su3(Link U, const cpx<fx> h[3], int sh, int one, cpx<fx> u[3]) {
  FxLimbs hr[3], hi[3], hn[3];  // re, im, and -im (U h) or -re (U^dag h)
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const fx re = h[c].re >> sh, im = h[c].im >> sh;
    hr[c] = fx_split(re);
    hi[c] = fx_split(im);
    hn[c] = fx_split(-(S > 0 ? im : re));  // (negated limbs would miss lo = -2^31)
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    FxSum p[2], m[2] = {{0x80000000u, 0}, {0x80000000u, 0}};  // re, im: uh hh; the middle sum from half a unit
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int k = S > 0 ? 3 * a + b : 3 * b + a;
      const uint4 w = U(k);
      const FxLimbs ur = {(int)w.y, (int)w.x}, ui = {(int)w.w, (int)w.z};
      const FxLimbs xr = S > 0 ? hn[b] : hi[b], xi = S > 0 ? hr[b] : hn[b];  // ui's partners
      if (b == 0) {
        p[0] = fx_mul(ur.hi, hr[b].hi);
        p[1] = fx_mul(ur.hi, hi[b].hi);
      } else {
        fx_mad(p[0], ur.hi, hr[b].hi);
        fx_mad(p[1], ur.hi, hi[b].hi);
      }
      fx_mad(m[0], ur.hi, hr[b].lo);
      fx_mad(m[1], ur.hi, hi[b].lo);
      fx_mad(m[0], ur.lo, hr[b].hi);
      fx_mad(m[1], ur.lo, hi[b].hi);
      fx_mad(p[0], ui.hi, xr.hi);
      fx_mad(p[1], ui.hi, xi.hi);
      fx_mad(m[0], ui.hi, xr.lo);
      fx_mad(m[1], ui.hi, xi.lo);
      fx_mad(m[0], ui.lo, xr.hi);
      fx_mad(m[1], ui.lo, xi.hi);
    }
    fx_mad(p[0], (int)m[0].hi, one);
    fx_mad(p[1], (int)m[1].hi, one);
    u[a] = mk<fx>(fx_value(p[0]), fx_value(p[1]));
  }
}

// A site's sum in two lanes, one per component q = 0, 1 of the projected spinors: lane q sums its upper
// spin q, and what its component adds to the lower spins, s = spin 2 + q (t, z hops) and o = spin 3 - q
// (x, y hops): 36 registers of sums where one thread for both components had 48 (168 registers in all,
// 12 warps per SM, latency bound; with two lanes 128 registers and 16 warps).
struct FxAcc {
  cpx<fx> up[3], s[3], o[3];
  int E;
  bool bad;
};

// acc += one hop of direction mu: v the neighbour's component q and its partner, of exponent e, link(k) the
// entry k of the hop's link.  E grows to the neighbour's exponent, acc is shifted right then.  Component
// q of (1 + S gamma_mu) v is v_q - S z v_partner for q = 0 and v_1 - S sigma z v_partner for q = 1,
// z = 1 (t, y) or i (x, z), sigma = -1 for y and z; the hop adds conj(-S sigma z) u to the partner's
// spin.
template <int S, class Link>
__device__ __forceinline__ void fx_hop_apply(int mu, int q, int one, FxAcc& A, const cpx<fx> v[6], int e, Link link,
                                             bool negate) {
  if (e >= A.E && e <= FX_EMAX && e != 0) {  // to e + 1: a later neighbour has to be twice as large to grow it again
    const int sh = min(e + 1 - A.E, 63);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      A.up[k] = mk<fx>(A.up[k].re >> sh, A.up[k].im >> sh);
      A.s[k] = mk<fx>(A.s[k].re >> sh, A.s[k].im >> sh);
      A.o[k] = mk<fx>(A.o[k].re >> sh, A.o[k].im >> sh);
    }
    A.E = e + 1;
  }
  A.bad = A.bad || e == FX_BAD;
  const int m1 = S > 0 ? (q ? 0 : -1) : (q ? -1 : 0);  // y, z: mask of -S sigma
  cpx<fx> hh[3], u[3];
  if (mu == 0) {
#pragma unroll
    for (int c = 0; c < 3; ++c) hh[c] = S > 0 ? v[c] - v[3 + c] : v[c] + v[3 + c];
    if (negate) {  // the antiperiodic time boundary
#pragma unroll
      for (int c = 0; c < 3; ++c) hh[c] = mk<fx>(-hh[c].re, -hh[c].im);
    }
  } else if (mu == 1) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      hh[c] = S > 0 ? mk<fx>(v[c].re + v[3 + c].im, v[c].im - v[3 + c].re)
                    : mk<fx>(v[c].re - v[3 + c].im, v[c].im + v[3 + c].re);
  } else if (mu == 2) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      hh[c] = mk<fx>(fx_addsgn(v[c].re, v[3 + c].re, m1), fx_addsgn(v[c].im, v[3 + c].im, m1));
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      hh[c] = mk<fx>(fx_addsgn(v[c].re, v[3 + c].im, ~m1), fx_addsgn(v[c].im, v[3 + c].re, m1));
  }
  fx_su3<S>(link, hh, min(max(A.E - e, 0), 63), one, u);  // a zero or FX_BAD neighbour: any shift
#pragma unroll
  for (int a = 0; a < 3; ++a) A.up[a] = A.up[a] + u[a];
  if (mu == 0) {
#pragma unroll
    for (int a = 0; a < 3; ++a) A.s[a] = S > 0 ? A.s[a] - u[a] : A.s[a] + u[a];
  } else if (mu == 1) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
      A.o[a] = S > 0 ? mk<fx>(A.o[a].re - u[a].im, A.o[a].im + u[a].re) : mk<fx>(A.o[a].re + u[a].im, A.o[a].im - u[a].re);
  } else if (mu == 2) {
#pragma unroll
    for (int a = 0; a < 3; ++a) A.o[a] = mk<fx>(fx_addsgn(A.o[a].re, u[a].re, m1), fx_addsgn(A.o[a].im, u[a].im, m1));
  } else {
#pragma unroll
    for (int a = 0; a < 3; ++a) A.s[a] = mk<fx>(fx_addsgn(A.s[a].re, u[a].im, m1), fx_addsgn(A.s[a].im, u[a].re, ~m1));
  }
}

// One hop read into registers and applied.
template <int SRC, int S>
__device__ __forceinline__ void fx_hop(int mu, int q, int one, FxAcc& A, const char* in, int h, int nbi, const char* slab,
                                       int li, bool negate, const FxCanon& canon) {
  const RawWords<FX_LINK_BYTES> U = load_raw<FX_LINK_BYTES>(slab, h, li);
  const bool tz = mu == 0 || mu == 3;
  cpx<fx> v[6];
  const int e = fx_load<SRC>(in, h, SRC == FXS_CANON ? 2 * nbi + (mu == 1 ? 1 - canon.b : canon.b) : nbi, 3 * q,
                       tz ? 6 + 3 * q : 9 - 3 * q, v, canon);
  fx_hop_apply<S>(mu, q, one, A, v, e,
                  [&](int k) { return make_uint4(U.w[4 * k], U.w[4 * k + 1], U.w[4 * k + 2], U.w[4 * k + 3]); }, negate);
}

// The two neighbours of direction mu, and whether they lie across the lattice's edge.
__device__ __forceinline__ void fx_neighbours(const Geom& g, int cb, const SiteCoord& c, int mu, int& nf, int& nb, bool& wf,
                                              bool& wb) {
  if (mu == 1) {
    const int xp = c.x == g.L - 1 ? 0 : c.x + 1, xm = c.x == 0 ? g.L - 1 : c.x - 1;
    const int row = cb - (c.x >> 1);
    nf = row + (xp >> 1);
    nb = row + (xm >> 1);
    wf = wb = false;
  } else {
    const int co = mu == 0 ? c.t : (mu == 2 ? c.y : c.z);
    const int ext = mu == 0 ? g.T : g.L;
    const int st = mu == 0 ? g.st : (mu == 2 ? g.sy : g.sz);
    wf = co == ext - 1;
    wb = co == 0;
    nf = wf ? cb - (ext - 1) * st : cb + st;
    nb = wb ? cb + (ext - 1) * st : cb - st;
  }
}

// The hops of directions [d0, d1) of a site in lane q, A in units of 2^(E - 1079).  Whole warps call it, lanes
// past the last site with that site: its shuffles and warp barriers name every lane.  The directions run
// as one loop over the same code (what differs between them are signs and uniform branches): unrolled,
// the sum was ~100 kB of instructions and the kernel waited for instruction fetch (16^3 x 32
// 97-130 us, 4^4 38 us).
template <int SRC>
__device__ __forceinline__ void fx_hops(FxAcc& A, int q, const Geom& g, int cb, const SiteCoord& c, const char* in,
                                        const char* lf, const char* lo, int d0, int d1, const FxCanon& canon = {0, 0, true}) {
  const size_t slab = (size_t)FX_LINK_BYTES * g.h;
  const int one = fx_one();
#pragma unroll 1
  for (int mu = d0; mu < d1; ++mu) {
    int nf, nb;
    bool wf, wb;
    fx_neighbours(g, cb, c, mu, nf, nb, wf, wb);
    fx_hop<SRC, +1>(mu, q, one, A, in, g.h, nf, lf + mu * slab, cb, mu == 0 && wf, canon);
    fx_hop<SRC, -1>(mu, q, one, A, in, g.h, nb, lo + mu * slab, nb, mu == 0 && wb, canon);
  }
}

// The same for FX input with the next hop's neighbour and link copied to shared memory (cp.async) while
// this hop is computed: in registers the two hops in flight would be 42 more of them.  For launches that
// fill the chip (the full operator with one pair per site); the solvers' hopping launches on smaller
// lattices lost 6 % with it (16^3 x 32, a CG of FP64 12.0 -> 12.7 ms), so they read into registers.
// stage: FX_STAGE 16-byte slots per site and hop, slot k of the block's S sites at stage[k * S ..], two
// hops.  Lane q's components are its own; lane 1 keeps them at site s ^ 4, so that the two lanes of four
// sites (a shared-memory phase) use different banks.
constexpr int FX_STAGE = 21;  // 9 link entries, 12 components
__device__ __forceinline__ void fx_copy16(uint4* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
template <int SITES>
__device__ __forceinline__ void fx_stage_hop(uint4* st, int site, int q, int h, const char* in, int nbi, const char* slab, int li,
                                             int jb, int& e) {
  const char* lp = slab + (size_t)li * 16;
  const char* vp = in + (size_t)nbi * 16;
  const size_t hb = (size_t)h * 16;
#pragma unroll
  for (int k = 0; k < 5; ++k) {  // link entries 0, 2, .. 8 by lane 0; 1, 3, 5, 7 by lane 1
    const int n = 2 * k + q;
    if (n < 9) fx_copy16(st + n * SITES + site, lp + n * hb);
  }
  uint4* const sv = st + (9 + 6 * q) * SITES + (site ^ (4 * q));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    fx_copy16(sv + k * SITES, vp + (3 * q + k) * hb);
    fx_copy16(sv + (3 + k) * SITES, vp + (jb + k) * hb);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  e = __ldg(fx_exps(in, h) + nbi);
}
template <int SITES, int S>
__device__ __forceinline__ void fx_apply_staged(const uint4* st, int site, int mu, int q, int one, FxAcc& A, int e, bool negate) {
  cpx<fx> v[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const uint4 w = st[(9 + 6 * q + k) * SITES + (site ^ (4 * q))];
    v[k] = mk<fx>((fx)(((unsigned long long)w.y << 32) | w.x), (fx)(((unsigned long long)w.w << 32) | w.z));
  }
  fx_hop_apply<S>(mu, q, one, A, v, e, [&](int k) { return st[k * SITES + site]; }, negate);
}
template <int SITES>
__device__ __forceinline__ void fx_hops_staged(FxAcc& A, int q, const Geom& g, int cb, const SiteCoord& c, const char* in,
                                               const char* lf, const char* lo, int d0, int d1, uint4* stage, int site) {
  const size_t slab = (size_t)FX_LINK_BYTES * g.h;
  const int one = fx_one();
  uint4* const s1 = stage + FX_STAGE * SITES;
  int nf, nb, e0, e1 = 0;
  bool wf, wb;
  fx_neighbours(g, cb, c, d0, nf, nb, wf, wb);
  fx_stage_hop<SITES>(stage, site, q, g.h, in, nf, lf + d0 * slab, cb, (d0 == 0 || d0 == 3) ? 6 + 3 * q : 9 - 3 * q, e0);
#pragma unroll 1
  for (int mu = d0; mu < d1; ++mu) {
    const int jb = (mu == 0 || mu == 3) ? 6 + 3 * q : 9 - 3 * q;
    fx_stage_hop<SITES>(s1, site, q, g.h, in, nb, lo + mu * slab, nb, jb, e1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    fx_apply_staged<SITES, +1>(stage, site, mu, q, one, A, e0, mu == 0 && wf);
    __syncwarp();
    const bool wrap = mu == 0 && wb;
    if (mu + 1 < d1) {
      fx_neighbours(g, cb, c, mu + 1, nf, nb, wf, wb);
      fx_stage_hop<SITES>(stage, site, q, g.h, in, nf, lf + (mu + 1) * slab, cb,
                          (mu + 1 == 3) ? 6 + 3 * q : 9 - 3 * q, e0);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    fx_apply_staged<SITES, -1>(s1, site, mu, q, one, A, e1, wrap);
    __syncwarp();
  }
}

// 2^(E - 1079), the unit of a sum with exponent E (1 for the empty sum)
__device__ __forceinline__ double fx_unit(int E) { return E == 0 ? 1.0 : __hiloint2double((E - 56) << 20, 0); }

}  // namespace tmq
