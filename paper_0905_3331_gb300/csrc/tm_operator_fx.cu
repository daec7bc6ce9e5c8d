// tm_operator_fx.cu -- the full operator M of eq. eo0 on canonical FP64 fields, in two launches: the
// canonical field to the FX form (tm_dslash_fx.cuh) of its two parities, then the hopping sum of both
// parities with the site term, written in canonical order.
//
// The first form packed each parity, ran one hopping launch per parity on half fields and unpacked
// each: six launches, and 192-byte records read and written by single threads (a quarter of the time on
// 32^3 x 64).  Here the canonical records pass through shared memory (padded to 13 x 16 bytes: conflict
// free), so that global accesses are whole 192-byte runs.  Both together, on 32^3 x 64: 1781 -> 1226 us a
// call (most of it the hopping launch, latency bound as in tm_dslash_fx.cuh; 2.0 GB a call are 297 us of
// HBM); 8^4 41 -> 16 us (two launches instead of six).
//
// The hopping launch takes the next hop's neighbour and link into shared memory (cp.async) while it
// computes this one (fx_hops_staged): 32^3 x 64 1226 -> 1112 us, two fields of 20 x 14^3 79.9 -> 77.5;
// with the real part of the site term as a sign, not a product, 1089 and 73.6; with whole warps in the loop
// and constant masks 1067 and 71.7.
//
// Small lattices take one launch, which converts the canonical neighbours as it reads them: 8^4 16 -> 10
// us (the rule and its figures are at CANON_SITES).
#include <algorithm>

#include "tm_hop_fx.cuh"

namespace tmq {

// Sites lex [128 b, 128 b + 128) -- cb [64 b, 64 b + 64) of both parities -- of right-hand side y.
__global__ void __launch_bounds__(128) full_to_fx_kernel(const Geom g, const double* __restrict__ in, char* __restrict__ out,
                                                         size_t out_stride, int g5, bool al) {
  __shared__ double2 tile[128 * CANON_TILE];
  const size_t V = 2 * (size_t)g.h, first = (size_t)blockIdx.x * 128;
  const int n = (int)min((size_t)128, V - first);
  const double* src = in + ((size_t)blockIdx.y * V + first) * 24;
  for (int i = threadIdx.x; i < n * 12; i += 128) canon_to_shared(&tile[i / 12 * CANON_TILE + i % 12], src + 2 * (size_t)i, al);
  canon_wait();
  __syncthreads();
  if ((int)threadIdx.x >= n) return;
  const size_t lex = first + threadIdx.x;
  const int cb = (int)(lex / 2);
  const int r = cb / g.Lh, y = r % g.L, z = (r / g.L) % g.L, t = r / (g.L * g.L);
  const int p = (int)((lex + t + z + y) & 1);
  cpx<double> v[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const double2 a = tile[threadIdx.x * CANON_TILE + k];
    v[k] = (g5 && k >= 6) ? mk(-a.x, -a.y) : mk(a.x, a.y);
  }
  const int e = fx_exponent_f64<12>(v);
  char* o = out + blockIdx.y * out_stride + p * fx_field_bytes(g.h);
  longlong2* q = reinterpret_cast<longlong2*>(o) + cb;
#pragma unroll
  for (int k = 0; k < 12; ++k) q[(size_t)k * g.h] = fx_pack(v[k], e);
  const_cast<int*>(fx_exps(o, g.h))[cb] = e;
}

// out = d H in + e in (d, e: coef's, d real) on both parities (blockIdx.y) of right-hand side blockIdx.z.  CANON: the
// hopping sum reads the canonical field itself, with P thread pairs per site; otherwise its FX form fxin,
// staged, with one.
template <int P, bool CANON>
__global__ void __launch_bounds__(fx_nt(P), HOP_FX_WARPS * 32 / fx_nt(P))
    full_fx_kernel(const Geom g, const char* __restrict__ links, const char* __restrict__ fxin, size_t fx_stride,
                   const double* __restrict__ in, double* __restrict__ out, const EpiCoef coef, int g5, bool al_in,
                   bool al_out) {
  constexpr int SPB = fx_spb(P), NT = fx_nt(P), WPP = NT / 32 / P;
  static_assert(CANON || P == 1);
  constexpr int TILE = SPB * CANON_TILE * 16, SUMS = P > 1 ? P * SPB * 2 * 19 * 8 : 0;
  constexpr int STAGE = CANON ? 0 : SPB * 2 * FX_STAGE * 16;
  constexpr int SMEM = STAGE > TILE ? STAGE : (SUMS > TILE ? SUMS : TILE);
  // the staged hops or the parts' sums, then the results
  __shared__ __align__(16) char smem[SMEM];
  double2* const tile = reinterpret_cast<double2*>(smem);
  const int warp = threadIdx.x >> 5;
  const int part = P == 1 ? 0 : warp / WPP;
  const int lane2 = P == 1 ? (int)threadIdx.x : (warp % WPP) * 32 + (int)(threadIdx.x & 31);
  const int q = lane2 & 1, site = lane2 >> 1;
  const int parity = blockIdx.y;
  const int cb = blockIdx.x * SPB + site;
  const bool active = cb < g.h;
  const size_t V24 = 48 * (size_t)g.h;
  const double* inr = in + blockIdx.z * V24;
  const size_t slab = (size_t)FX_LINK_BYTES * g.h;
  const char* lf = links + (size_t)(parity * 4) * slab;
  const char* lo = links + (size_t)((1 - parity) * 4) * slab;
  const char* src = fxin + blockIdx.z * fx_stride + (1 - parity) * fx_field_bytes(g.h);
  FxAcc A;
#pragma unroll
  for (int k = 0; k < 3; ++k) A.up[k] = A.s[k] = A.o[k] = mk<fx>(0, 0);
  A.E = 0;
  A.bad = false;
  const int cbs = min(cb, g.h - 1);
  const SiteCoord c = site_of(g, cbs, parity);
  if constexpr (CANON)
    fx_hops<FXS_CANON>(A, q, g, cbs, c, reinterpret_cast<const char*>(inr), lf, lo, part * (4 / P), (part + 1) * (4 / P),
                       FxCanon{(c.t + c.z + c.y + parity) & 1, g5, al_in});
  else
    fx_hops_staged<SPB>(A, q, g, cbs, c, src, lf, lo, 0, 4, reinterpret_cast<uint4*>(smem), site);
  if constexpr (P > 1) fx_merge<P, SPB>(A, part, lane2, reinterpret_cast<fx*>(smem));
  __syncthreads();
  if (part == 0) {
    cpx<double> acc[6];
    double unit;
    fx_finish(A, q, active, g, parity, cb, CanonInput{inr, 1 - parity, g5}, lf, lo, acc, unit);
    if (active) {
      // e = +-1 + i e_im: 6 FP64 instructions a component (80 clocks of the unit each) with the conversions
      const double cu = coef.d_up_re * unit, cl = coef.d_lo_re * unit;
      const int mu = __double2hiint(coef.e_up_re) & 0x80000000, ml = __double2hiint(coef.e_lo_re) & 0x80000000;
      const double* y = inr + lex_of_cb(g, cb, parity) * 24;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const int blk = (k < 3 ? 3 * q : 6 + 3 * q) + k % 3;
        const double2 t = canon_load(y + 2 * blk, al_in);
        const int m = k < 3 ? mu : ml;
        const double im = k < 3 ? coef.e_up_im : coef.e_lo_im, d = k < 3 ? cu : cl;
        const double sx = __hiloint2double(__double2hiint(t.x) ^ m, __double2loint(t.x));
        const double sy = __hiloint2double(__double2hiint(t.y) ^ m, __double2loint(t.y));
        tile[site * CANON_TILE + blk] =
            make_double2(fma(d, acc[k].re, fma(-im, t.y, sx)), fma(d, acc[k].im, fma(im, t.x, sy)));
      }
    }
  }
  __syncthreads();
  double* dst = out + blockIdx.z * V24;
  for (int i = threadIdx.x; i < SPB * 12; i += NT) {
    const int s = i / 12, k = i % 12, c2 = blockIdx.x * SPB + s;
    if (c2 >= g.h) break;
    double* o = dst + lex_of_cb(g, c2, parity) * 24 + 2 * k;
    canon_store(o, tile[s * CANON_TILE + k], al_out);
  }
}

// Which form of the second launch, from the sites of both parities and all right-hand sides, by
// measurement (one field unless said; us, FX form | canonical form with 1, 2, 4 pairs per site):
//   4^4 13.7 | 14.8 10.3 10.3      8^4 15.6 | 16.4 12.3 10.3      8^3 x 16 17.3 | 16.4 14.3 12.3
//   10^3 x 16 22.5 | 20.5 18.5 21.8            3 fields of 8^3 x 16 26.7 | 24.6 25.7 30.4
//   12^3 x 24 37.8 | 36.9 36.6 44.4            14^3 x 20 45.1 | 42.6 44.4 55.4
//   2 fields of 14^3 x 20 73.8 | 76.0 80.0 104.5      16^3 x 32 90.1 | 97.5 102.6 129.0
// (both a few per cent less since the site term's real part became a sign).
// Small: the launch and the pass over the FX form cost more than converting each neighbour as it is read,
// eight times over.  The pairs per site are as many as one field fits on the chip in a wave of 16 warps
// per SM, so that a field's bits do not depend on the right-hand sides beside it.  With one pair both forms
// give the same bits; the FX form has no kernel with two or four, so there the canonical form serves any
// number of fields, also where one pair on the FX form would be quicker (3 fields of 8^3 x 16).
constexpr size_t CANON_SITES = 65536;
constexpr size_t WAVE_LANES = 152 * 16 * 32;
// The FX form of as many fields at a time as fit in 256 MiB (1.4 million sites), at least one.  Smaller chunks
// end in more last waves: 12 fields of 24 x 16^3 596 us with 1.4 million sites, 614 with 1.0, 629 with 0.5,
// 686 with 0.25; of 20 x 14^3 336, 336, 350, 369.
constexpr size_t FULL_FX_BYTES = (size_t)256 << 20;
constexpr int MAX_FIELDS = 65535;  // of a launch: they are its gridDim.z (gridDim.y in the FX pass)

static int full_pairs(tm_lattice lat) {
  if (hop_tps_fixed(lat, TM_F64, 18)) return lat->hop_tps[TM_F64][link_index(18)];
  return lat->V * 8 <= WAVE_LANES ? 4 : (lat->V * 4 <= WAVE_LANES ? 2 : 1);
}

int full_fx_fields(tm_lattice lat, int nrhs) {
  return full_pairs(lat) > 1 || (size_t)std::min(nrhs, MAX_FIELDS) * lat->V <= CANON_SITES
             ? 0
             : (int)std::max<size_t>(1, FULL_FX_BYTES / full_fx_bytes(lat->h));
}

tm_status apply_full(tm_lattice lat, double* out, const double* in, int f, int g5, int nrhs, void* scratch, int per,
                     cudaStream_t s) {
  tm_status st = ensure_links(lat, TM_F64, 18, s);
  if (st != TM_OK) return st;
  const Geom& g = lat->geom;
  EpiCoef c = epi_full_M(lat->kappa, 2.0 * lat->kappa * lat->mu, f);
  if (g5) {  // gamma5 M gamma5: the lower spins of the result, and of the site term's input, change sign
    c.d_lo_re = -c.d_lo_re;
    c.e_lo_re = -c.e_lo_re;
    c.e_lo_im = -c.e_lo_im;
  }
  c.e_up_re *= c.d_up_re;  // D (c H + E) multiplied out, D real
  c.e_up_im *= c.d_up_re;
  c.e_lo_re *= c.d_lo_re;
  c.e_lo_im *= c.d_lo_re;
  c.d_up_re *= c.c;
  c.d_lo_re *= c.c;
  const char* links = static_cast<const char*>(lat->links[TM_F64][link_index(18)]);
  char* fxs = static_cast<char*>(scratch);
  const size_t stride = full_fx_bytes(lat->h);
  const bool al_in = canon_aligned(in), al_out = canon_aligned(out);
  const int pairs = full_pairs(lat);
  for (int r = 0, n; r < nrhs; r += n) {
    n = std::min(nrhs - r, MAX_FIELDS);
    const bool canon = per == 0 || pairs > 1 || (size_t)n * lat->V <= CANON_SITES;
    if (!canon) n = (n + (n + per - 1) / per - 1) / ((n + per - 1) / per);  // equal chunks of at most `per`
    const double* src = in + (size_t)r * lat->V * 24;
    double* dst = out + (size_t)r * lat->V * 24;
#define TM_FULL_ARGS g, links, fxs, stride, src, dst, c, g5, al_in, al_out
#define TM_FULL(P)                                                                                         \
  full_fx_kernel<P, true><<<dim3((g.h + fx_spb(P) - 1) / fx_spb(P), 2, n), fx_nt(P), 0, s>>>(TM_FULL_ARGS)
    if (canon) {
      if (pairs == 2)
        TM_FULL(2);
      else if (pairs == 4)
        TM_FULL(4);
      else
        TM_FULL(1);
    } else {
      full_to_fx_kernel<<<dim3((unsigned)((lat->V + 127) / 128), n), 128, 0, s>>>(g, src, fxs, stride, g5, al_in);
      count_launch();
      full_fx_kernel<1, false><<<dim3((g.h + fx_spb(1) - 1) / fx_spb(1), 2, n), fx_nt(1), 0, s>>>(TM_FULL_ARGS);
    }
#undef TM_FULL
#undef TM_FULL_ARGS
    count_launch();
    if ((st = cuda_check(cudaGetLastError(), "operator kernel launch")) != TM_OK) return st;
  }
  return TM_OK;
}

}  // namespace tmq
