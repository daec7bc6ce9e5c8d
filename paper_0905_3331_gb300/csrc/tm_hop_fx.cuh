// tm_hop_fx.cuh -- the hopping kernel of FP64 fields and 18-real links: the fixed-point sum of
// tm_dslash_fx.cuh with the fused epilogues and reductions of tm_dslash.cuh.
//
// Two lanes per output site, one per projected spin component (lane q holds spins q and 2 + q of the
// result), times P direction parts in different warps (P = 1, 2, 4 for 1, 2, 4 "threads per site").
#pragma once

#include "tm_dslash.cuh"

namespace tmq {

// Sites and threads per block: 64 sites with 128 threads (P = 1), 32 with 128 (2) or 256 (4).
constexpr int fx_spb(int P) { return P == 1 ? 64 : 32; }
constexpr int fx_nt(int P) { return fx_spb(P) * 2 * P; }

// Where the FP64 input of a launch is: an FP64 half field, or the sites of parity p of a canonical full
// field, gamma5 applied if g5.
struct HalfInput {
  const char* in;
  __device__ __forceinline__ bool valid() const { return in != nullptr; }
  __device__ __forceinline__ void load(const Geom& g, int i, cpx<double> v[12]) const {
    SpinorFmt<TM_F64>::load(in, g.h, i, v);
  }
};
struct CanonInput {
  const double* in;
  int p, g5;
  __device__ __forceinline__ bool valid() const { return true; }
  __device__ __forceinline__ void load(const Geom& g, int i, cpx<double> v[12]) const {
    const double* q = in + lex_of_cb(g, i, p) * 24;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const cpx<double> t = mk(__ldg(q + 2 * k), __ldg(q + 2 * k + 1));
      v[k] = (g5 && k >= 6) ? mk(-t.re, -t.im) : t;
    }
  }
};

// The FP64 form of one output site, for the sites whose neighbours have no fixed-point form.  A real
// call, so that its registers are not the caller's.
template <class Input>
static __device__ __noinline__ void hop_f64_general(const Geom& g, int out_parity, int cb, const Input in,
                                                    const char* lf, const char* lo, double out[24]) {
  const SiteCoord c = site_of(g, cb, out_parity);
  int nb[8];
  neighbours(g, cb, c, nb);
  const size_t slab = link_bytes(TM_F64, 18) * (size_t)g.h;
  cpx<double> acc[12], p[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = mk(0.0, 0.0);
#define TM_GENERAL_HOP(MU, S, I, SLAB, LI, NEG)                                                       \
  in.load(g, nb[I], p);                                                                               \
  hop_apply<TM_F64, 18, MU, S>(acc, load_raw<18 * 8>((SLAB) + MU * slab, g.h, LI), p, 1.0, NEG);
  TM_GENERAL_HOP(0, +1, 0, lf, cb, c.t == g.T - 1)
  TM_GENERAL_HOP(0, -1, 4, lo, nb[4], c.t == 0)
  TM_GENERAL_HOP(1, +1, 1, lf, cb, false)
  TM_GENERAL_HOP(1, -1, 5, lo, nb[5], false)
  TM_GENERAL_HOP(2, +1, 2, lf, cb, false)
  TM_GENERAL_HOP(2, -1, 6, lo, nb[6], false)
  TM_GENERAL_HOP(3, +1, 3, lf, cb, false)
  TM_GENERAL_HOP(3, -1, 7, lo, nb[7], false)
#undef TM_GENERAL_HOP
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    out[2 * k] = acc[k].re;
    out[2 * k + 1] = acc[k].im;
  }
}

// |x| == 1, on the words
__device__ __forceinline__ bool fx_is_one(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) == 0x3ff00000u && __double2loint(x) == 0;
}

// acc = this lane's six components (spins q and 2 + q) of the sum A in FP64, with unit folded in by the
// caller: real = acc unit.  All lanes of the warp call it (shuffles between the two lanes of a site).
// in64: the FP64 input, if there is one.
template <class Input>
__device__ __forceinline__ void fx_finish(const FxAcc& A, int q, bool active, const Geom& g, int out_parity, int cb,
                                          const Input in64, const char* lf, const char* lo, cpx<double> acc[6],
                                          double& unit) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {  // the other lane's share of this lane's lower spin 2 + q
    const fx re = A.s[k].re + __shfl_xor_sync(0xffffffffu, A.o[k].re, 1);
    const fx im = A.s[k].im + __shfl_xor_sync(0xffffffffu, A.o[k].im, 1);
    acc[k] = mk<double>((double)A.up[k].re, (double)A.up[k].im);
    acc[3 + k] = mk<double>((double)re, (double)im);
  }
  unit = fx_unit(A.E);
  if (A.bad && active) {
    unit = 1.0;
    if (in64.valid()) {
      double v[24];
      hop_f64_general(g, out_parity, cb, in64, lf, lo, v);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        acc[k] = mk<double>(v[6 * q + 2 * k], v[6 * q + 2 * k + 1]);
        acc[3 + k] = mk<double>(v[12 + 6 * q + 2 * k], v[13 + 6 * q + 2 * k]);
      }
    } else {
      const double nan = fx_stored_unit(FX_BAD);
#pragma unroll
      for (int k = 0; k < 6; ++k) acc[k] = mk<double>(nan, nan);
    }
  }
}

// The whole sum of a site in its two lanes, as FP64.
template <bool XIN>
__device__ __forceinline__ void fx_site(cpx<double> acc[6], int q, bool active, const Geom& g, int out_parity, int cb,
                                        const char* in, const char* in64, const char* lf, const char* lo) {
  FxAcc A;
#pragma unroll
  for (int k = 0; k < 3; ++k) A.up[k] = A.s[k] = A.o[k] = mk<fx>(0, 0);
  A.E = 0;
  A.bad = false;
  const int site = min(cb, g.h - 1);
  fx_hops<XIN>(A, q, g, site, site_of(g, site, out_parity), in, lf, lo, 0, 4);
  double unit;
  fx_finish(A, q, active, g, out_parity, cb, HalfInput{in64}, lf, lo, acc, unit);
#pragma unroll
  for (int k = 0; k < 6; ++k) acc[k] = unit * acc[k];
}

// The P direction parts' sums meet in part 0, at the largest of their exponents (called by the block).
template <int P, int SPB>
__device__ __forceinline__ void fx_merge(FxAcc& A, int part, int lane2, fx* part_sum) {
  fx* mine = part_sum + (part * SPB * 2 + lane2) * 19;
  if (part > 0) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      mine[2 * k] = A.up[k].re;
      mine[2 * k + 1] = A.up[k].im;
      mine[6 + 2 * k] = A.s[k].re;
      mine[7 + 2 * k] = A.s[k].im;
      mine[12 + 2 * k] = A.o[k].re;
      mine[13 + 2 * k] = A.o[k].im;
    }
    mine[18] = A.bad ? -1 : A.E;
  }
  __syncthreads();
  if (part == 0) {
#pragma unroll
    for (int p = 1; p < P; ++p) {
      const fx* o = part_sum + (p * SPB * 2 + lane2) * 19;
      const int Ep = (int)o[18];
      if (Ep < 0) {
        A.bad = true;
        continue;
      }
      const int sa = Ep > A.E ? min(Ep - A.E, 63) : 0, so = A.E > Ep ? min(A.E - Ep, 63) : 0;
      A.E = max(A.E, Ep);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        A.up[k] = mk<fx>((A.up[k].re >> sa) + (o[2 * k] >> so), (A.up[k].im >> sa) + (o[2 * k + 1] >> so));
        A.s[k] = mk<fx>((A.s[k].re >> sa) + (o[6 + 2 * k] >> so), (A.s[k].im >> sa) + (o[7 + 2 * k] >> so));
        A.o[k] = mk<fx>((A.o[k].re >> sa) + (o[12 + 2 * k] >> so), (A.o[k].im >> sa) + (o[13 + 2 * k] >> so));
      }
    }
  }
}

// The body: output sites [bid SPB, (bid + 1) SPB) of right-hand side rhs; arguments and modes as
// hop_sites (tm_dslash.cuh).  XIN: `in` is an FX half field; fxa: the other FX fields.
template <bool HAS_Y, int MODE, int P, bool XIN, class Blk>
__device__ __forceinline__ void hop_sites_fx(const Geom g, const int out_parity, const char* __restrict__ links,
                                             const void* in, size_t in_stride, void* out, size_t out_stride,
                                             const void* y, size_t y_stride, const EpiCoef coef,
                                             const CGState* alpha_src, const double alpha_sign, const Reduce red,
                                             const Blk B, const FxArgs fxa) {
  constexpr int SPB = fx_spb(P), NT = fx_nt(P);
  constexpr int WPP = NT / 32 / P;  // warps per part
  __shared__ double sh[NT / 32];
  __shared__ fx part_sum[P > 1 ? P * SPB * 2 * 19 : 1];
  const int warp = threadIdx.x >> 5;
  const int part = P == 1 ? 0 : warp / WPP;
  const int lane2 = P == 1 ? (int)threadIdx.x : (warp % WPP) * 32 + (int)(threadIdx.x & 31);  // 2 site + q
  const int q = lane2 & 1;
  const int rhs = B.rhs();
  const int cb = B.bid() * SPB + (lane2 >> 1);
  const bool active = cb < g.h;
  FxAcc A;
#pragma unroll
  for (int k = 0; k < 3; ++k) A.up[k] = A.s[k] = A.o[k] = mk<fx>(0, 0);
  A.E = 0;
  A.bad = false;
  const char* inr = static_cast<const char*>(in) + (size_t)rhs * in_stride;
  const size_t slab = (size_t)FX_LINK_BYTES * g.h;
  const char* lf = links + (size_t)(out_parity * 4) * slab;        // U_mu(x), x of this parity
  const char* lo = links + (size_t)((1 - out_parity) * 4) * slab;  // U_mu(y), y of the other parity
  const int site = min(cb, g.h - 1);
  fx_hops<XIN>(A, q, g, site, site_of(g, site, out_parity), inr, lf, lo, part * (4 / P), (part + 1) * (4 / P));
  if constexpr (P > 1) fx_merge<P, SPB>(A, part, lane2, part_sum);
  double nrm = 0.0;
  if (part == 0) {
    cpx<double> acc[6];
    double unit;
    fx_finish(A, q, active, g, out_parity, cb, HalfInput{XIN ? nullptr : inr}, lf, lo, acc,
              unit);
    // epilogue: o_s = D_s (c acc_s + E_s y_s) as (D_s c unit) acc_s + (D_s E_s) y_s; a real D c (every
    // coefficient set but the inverse site term) takes half the products.  An FP64 instruction of a warp
    // takes 80 clocks of its quarter of the SM, so the units and MODE 2's -alpha go into the coefficients
    // and r is where the chains begin: K4 on 12^3 x 24 31.0 -> 28.6 us (20 of them without an epilogue).
    const double m = MODE == 2 ? -(alpha_src ? alpha_sign * alpha_src[rhs].alpha : alpha_sign) : 1.0;
    const double cc = coef.c * unit;
    const cpx<double> Du = MODE == 2 ? mk(m * coef.d_up_re, m * coef.d_up_im) : mk(coef.d_up_re, coef.d_up_im);
    const cpx<double> Dl = MODE == 2 ? mk(m * coef.d_lo_re, m * coef.d_lo_im) : mk(coef.d_lo_re, coef.d_lo_im);
    const bool real_d = coef.d_up_im == 0.0 && coef.d_lo_im == 0.0;
    const int kq[2] = {3 * q, 6 + 3 * q};  // this lane's blocks: kq[half] + k
    char* outr = static_cast<char*>(out) + (size_t)rhs * out_stride;
    cpx<double> o[6];
    if (MODE == 2) {
#pragma unroll
      for (int k = 0; k < 6; ++k) o[k] = mk(0.0, 0.0);
      if (active) {
        const double2* p = reinterpret_cast<const double2*>(outr) + cb;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const double2 t = p[(size_t)(kq[k / 3] + k % 3) * g.h];
          o[k] = mk(t.x, t.y);
        }
      }
    }
    if (HAS_Y) {
      cpx<double> Eu = mk(coef.e_up_re, coef.e_up_im), El = mk(coef.e_lo_re, coef.e_lo_im);
      cpx<double> yv[6];  // in units of yu
#pragma unroll
      for (int k = 0; k < 6; ++k) yv[k] = mk(0.0, 0.0);
      if (active) {
        const char* yr = static_cast<const char*>(y) + (size_t)rhs * y_stride;
        if (fxa.flags & FX_Y) {  // uniform
          const double yu = fx_stored_unit(__ldg(fx_exps(yr, g.h) + cb));
          Eu = yu * Eu;
          El = yu * El;
          const longlong2* p = reinterpret_cast<const longlong2*>(yr) + cb;
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const longlong2 t = __ldg(p + (size_t)(kq[k / 3] + k % 3) * g.h);
            yv[k] = mk((double)t.x, (double)t.y);
          }
        } else {
          const double2* p = reinterpret_cast<const double2*>(yr) + cb;
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const double2 t = __ldg(p + (size_t)(kq[k / 3] + k % 3) * g.h);
            yv[k] = mk(t.x, t.y);
          }
        }
      }
      if (MODE == 3) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const cpx<double> t = cc * acc[k] + (k < 3 ? Eu : El) * yv[k];
          o[k] = (k < 3 ? Du : Dl) * t;
          const cpx<double> M = k < 3 ? mk(coef.m_up_re, coef.m_up_im) : mk(coef.m_lo_re, coef.m_lo_im);
          nrm += norm2(t - M * o[k]);
        }
      } else {
        const cpx<double> DEu = real_d ? Du.re * Eu : Du * Eu, DEl = real_d ? Dl.re * El : Dl * El;
        // the Schur operator's D E = +-1 + i e_im on an FP64 y: the real part is a sign
        const bool sign_re = MODE != 2 && fx_is_one(DEu.re) && fx_is_one(DEl.re);  // uniform
        const int mu = __double2hiint(DEu.re) & 0x80000000, ml = __double2hiint(DEl.re) & 0x80000000;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const cpx<double> DE = k < 3 ? DEu : DEl;
          double re, im;
          if (MODE == 2) {
            re = fma(DE.re, yv[k].re, o[k].re);
            im = fma(DE.re, yv[k].im, o[k].im);
          } else if (sign_re) {
            const int m = k < 3 ? mu : ml;
            re = __hiloint2double(__double2hiint(yv[k].re) ^ m, __double2loint(yv[k].re));
            im = __hiloint2double(__double2hiint(yv[k].im) ^ m, __double2loint(yv[k].im));
          } else {
            re = DE.re * yv[k].re;
            im = DE.re * yv[k].im;
          }
          o[k] = mk(fma(-DE.im, yv[k].im, re), fma(DE.im, yv[k].re, im));
        }
      }
    }
    if (MODE != 3) {
      if (real_d) {
        const double du = Du.re * cc, dl = Dl.re * cc;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const double d = k < 3 ? du : dl;
          o[k] = HAS_Y ? mk(fma(d, acc[k].re, o[k].re), fma(d, acc[k].im, o[k].im)) : mk(d * acc[k].re, d * acc[k].im);
        }
      } else {
        const cpx<double> DCu = mk(Du.re * cc, Du.im * cc), DCl = mk(Dl.re * cc, Dl.im * cc);
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = HAS_Y ? o[k] + (k < 3 ? DCu : DCl) * acc[k] : (k < 3 ? DCu : DCl) * acc[k];
      }
    }
    if (MODE == 1 || MODE == 2) {
      if (active) {
#pragma unroll
        for (int k = 0; k < 6; ++k) nrm = fma(o[k].im, o[k].im, fma(o[k].re, o[k].re, nrm));
      }
    }
    if (MODE == 2) {
      if (active) {
        double2* p = reinterpret_cast<double2*>(outr) + cb;
#pragma unroll
        for (int k = 0; k < 6; ++k) p[(size_t)(kq[k / 3] + k % 3) * g.h] = make_double2(o[k].re, o[k].im);
      }
    } else {
      if (fxa.flags & FX_OUT) {  // uniform
        const int e = fx_stored_exponent<6>(o);  // the site's (a lane's six may be out of range by themselves)
        if (active) {
          longlong2* p = reinterpret_cast<longlong2*>(outr) + cb;
#pragma unroll
          for (int k = 0; k < 6; ++k) p[(size_t)(kq[k / 3] + k % 3) * g.h] = fx_pack(o[k], e);
          if (q == 0) const_cast<int*>(fx_exps(outr, g.h))[cb] = e;
        }
      } else if (active) {
        double2* p = reinterpret_cast<double2*>(outr) + cb;
#pragma unroll
        for (int k = 0; k < 6; ++k) p[(size_t)(kq[k / 3] + k % 3) * g.h] = make_double2(o[k].re, o[k].im);
      }
    }
  }
  if (MODE >= 1) {
    const double bs = block_sum<NT>(nrm, sh);
    grid_reduce<NT>(red, rhs, B.nblocks(), B.bid(), bs, sh);
  }
}

#ifndef HOP_FX_WARPS
#define HOP_FX_WARPS 16
#endif
// 16 warps per SM (128 registers)
template <bool HAS_Y, int MODE, int P, bool XIN>
__global__ void __launch_bounds__(fx_nt(P), HOP_FX_WARPS * 32 / fx_nt(P))
    hop_fx_kernel(const Geom g, const int out_parity, const char* __restrict__ links, const void* in, size_t in_stride,
                  void* out, size_t out_stride, const void* y, size_t y_stride, const EpiCoef coef,
                  const CGState* alpha_src, const double alpha_sign, const Reduce red, const int* skip,
                  const FxArgs fxa) {
  pdl_wait();
  pdl_allow();
  if (skip != nullptr && *skip != 0) return;
  hop_sites_fx<HAS_Y, MODE, P, XIN>(g, out_parity, links, in, in_stride, out, out_stride, y, y_stride, coef, alpha_src,
                                    alpha_sign, red, GridBlock{}, fxa);
}

template <int P, bool XIN>
tm_status hop_fx_launch_p(tm_lattice lat, const HopArgs& a, cudaStream_t s) {
  const Geom& g = lat->geom;
  constexpr int SPB = fx_spb(P), NT = fx_nt(P);
  dim3 grid((g.h + SPB - 1) / SPB, a.nrhs);
  const char* links = static_cast<const char*>(lat->links[TM_F64][link_index(18)]);
  const bool has_y = a.y != nullptr;
#define TM_FX_LAUNCH(HY, MD)                                                                                       \
  launch_pdl(hop_fx_kernel<HY, MD, P, XIN>, grid, dim3(NT), s, g, a.out_parity, links, a.in, a.in_stride, a.out,  \
             a.out_stride, a.y, a.y_stride, a.coef, a.alpha_src, a.alpha_sign, a.red, a.skip, a.fx)
  if (!has_y && a.mode == 0)
    TM_FX_LAUNCH(false, 0);
  else if (!has_y && a.mode == 1)
    TM_FX_LAUNCH(false, 1);
  else if (has_y && a.mode == 0)
    TM_FX_LAUNCH(true, 0);
  else if (has_y && a.mode == 1)
    TM_FX_LAUNCH(true, 1);
  else if (has_y && a.mode == 2)
    TM_FX_LAUNCH(true, 2);
  else if (has_y && a.mode == 3)
    TM_FX_LAUNCH(true, 3);
  else
    return set_error(TM_ERR_ARG, "hopping: unsupported epilogue combination");
#undef TM_FX_LAUNCH
  count_launch();
  return cuda_check(cudaGetLastError(), "hopping kernel launch");
}

template <bool XIN>
tm_status hop_fx_launch_t(tm_lattice lat, const HopArgs& a, cudaStream_t s) {
  switch (lat->hop_tps[TM_F64][link_index(18)]) {
    case 2:
      return hop_fx_launch_p<2, XIN>(lat, a, s);
    case 4:
      return hop_fx_launch_p<4, XIN>(lat, a, s);
    default:
      return hop_fx_launch_p<1, XIN>(lat, a, s);
  }
}

}  // namespace tmq
