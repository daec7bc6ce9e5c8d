// tm_fields.cu -- conversions between the canonical FP64 spinor order (t, z, y, x, spin,
// colour; Sec. 4.7.2) and the device half-field layouts, precision conversions, and the
// site-diagonal operator (M_ee^f)^{-1} = (1 - i f mu~ gamma5) / (1 + mu~^2) of eq. eo3.
#include "tm_internal.cuh"

namespace tmq {

constexpr int FNT = 128;

template <typename R>
__device__ __forceinline__ void apply_g5(cpx<R> s[12]) {
#pragma unroll
  for (int k = 6; k < 12; ++k) s[k] = R(-1) * s[k];
}

// Canonical records <-> a device half field, FNT sites per block through shared memory.  FULL: the sites
// of parity p of a canonical full field (times gamma5 if g5), else a canonical half field [rhs][cb].
// Bound by HBM: packing and unpacking two FP32 fields on 24^3 x 48 (382 MB) 163 -> 73 us (36 each); with a
// record read or written by one thread, unpacking alone took 115 us.  Packing copies asynchronously: through
// registers its guarded loads followed one another (52 us, long scoreboard 24 cycles an issue).
// Double-float is bound by the FP64 units (24 splits or sums a site) and gains nothing from the tile where
// the L2 takes what a record's accesses leave open: there a thread takes a whole record (!TILED).  Two
// fields, tile and whole records: packing 16^3 x 32 28.9 and 27.0 us, 24^3 x 48 124 and 121; unpacking 12^3 x
// 24 12.5 and 10.6, 16^3 x 32 22.7 and 20.8, but 24^3 x 48 92 and 122.
template <bool FULL>
__device__ __forceinline__ void tile_index(const Geom& g, int first, int n, int p, unsigned* lex) {
  if (FULL && (int)threadIdx.x < n) lex[threadIdx.x] = (unsigned)lex_of_cb(g, first + threadIdx.x, p);
}
template <bool FULL>
__device__ __forceinline__ size_t tile_offset(int first, int i, const unsigned* lex) {  // double2 i of the tile
  return 24 * (FULL ? (size_t)lex[i / 12] : (size_t)(first + i / 12)) + 2 * (i % 12);
}

template <int PREC, bool FULL, bool TILED>
__global__ void __launch_bounds__(FNT) pack_kernel(const Geom g, const double* __restrict__ src, char* __restrict__ dst,
                                                   size_t dstride, int p, int g5, bool al) {
  __shared__ double2 tile[TILED ? FNT * CANON_TILE : 1];
  __shared__ unsigned lex[FULL && TILED ? FNT : 1];
  const int first = blockIdx.x * FNT, n = min(FNT, g.h - first), cb = first + threadIdx.x;
  const double* in = src + (size_t)blockIdx.y * g.h * 24;
  cpx<double> s[12];
  if constexpr (!TILED) {
    if ((int)threadIdx.x >= n) return;
    const double* rec = in + 24 * (FULL ? lex_of_cb(g, cb, p) : (size_t)cb);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const double2 v = canon_load(rec + 2 * k, al);
      s[k] = mk(v.x, v.y);
    }
    if (FULL && g5) apply_g5(s);
    SpinorFmt<PREC>::store(dst + blockIdx.y * dstride, g.h, cb, s);
    return;
  }
  if (FULL) {
    tile_index<FULL>(g, first, n, p, lex);
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < 12; ++j) {
    const int i = j * FNT + threadIdx.x;
    if (i < n * 12) canon_to_shared(&tile[i / 12 * CANON_TILE + i % 12], in + tile_offset<FULL>(first, i, lex), al);
  }
  canon_wait();
  __syncthreads();
  if ((int)threadIdx.x >= n) return;
#pragma unroll
  for (int k = 0; k < 12; ++k) s[k] = mk(tile[threadIdx.x * CANON_TILE + k].x, tile[threadIdx.x * CANON_TILE + k].y);
  if (FULL && g5) apply_g5(s);
  SpinorFmt<PREC>::store(dst + blockIdx.y * dstride, g.h, cb, s);
}

template <int PREC, bool FULL, bool TILED>
__global__ void __launch_bounds__(FNT) unpack_kernel(const Geom g, const char* __restrict__ src, size_t sstride,
                                                     double* __restrict__ dst, int p, int g5, bool al) {
  __shared__ double2 tile[TILED ? FNT * CANON_TILE : 1];
  __shared__ unsigned lex[FULL && TILED ? FNT : 1];
  const int first = blockIdx.x * FNT, n = min(FNT, g.h - first), cb = first + threadIdx.x;
  double* out = dst + (size_t)blockIdx.y * g.h * 24;
  if (FULL && TILED) tile_index<FULL>(g, first, n, p, lex);
  if ((int)threadIdx.x < n) {
    cpx<double> s[12];
    SpinorFmt<PREC>::load(src + blockIdx.y * sstride, g.h, cb, s);
    if (FULL && g5) apply_g5(s);
    if constexpr (!TILED) {  // (16-byte stores were no faster than the tile)
      double* rec = out + 24 * (FULL ? lex_of_cb(g, cb, p) : (size_t)cb);
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        rec[2 * k] = s[k].re;
        rec[2 * k + 1] = s[k].im;
      }
      return;
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) tile[threadIdx.x * CANON_TILE + k] = make_double2(s[k].re, s[k].im);
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 12; ++j) {
    const int i = j * FNT + threadIdx.x;
    if (i < n * 12) canon_store(out + tile_offset<FULL>(first, i, lex), tile[i / 12 * CANON_TILE + i % 12], al);
  }
}

template <int PIN, int POUT>
__global__ void convert_kernel(int h, const char* __restrict__ src, char* __restrict__ dst) {
  const int cb = blockIdx.x * FNT + threadIdx.x;
  if (cb >= h) return;
  typedef typename SpinorFmt<PIN>::real R;
  cpx<R> s[12];
  SpinorFmt<PIN>::load(src, h, cb, s);
  SpinorFmt<POUT>::store(dst, h, cb, s);
}

// out = diag(Du, Du, Dl, Dl) in, site by site (in == out allowed)
template <int PREC>
__global__ void diag_kernel(int h, const char* in, size_t istride, char* out, size_t ostride, double dur,
                            double dui, double dlr, double dli) {
  const int cb = blockIdx.x * FNT + threadIdx.x, r = blockIdx.y;
  if (cb >= h) return;
  typedef typename SpinorFmt<PREC>::real R;
  cpx<R> s[12];
  SpinorFmt<PREC>::load(in + r * istride, h, cb, s);
  const cpx<R> Du = mk<R>((R)dur, (R)dui), Dl = mk<R>((R)dlr, (R)dli);
#pragma unroll
  for (int k = 0; k < 12; ++k) s[k] = ((k < 6) ? Du : Dl) * s[k];
  SpinorFmt<PREC>::store(out + r * ostride, h, cb, s);
}

#define TM_PREC_SWITCH(prec, F)        \
  switch (prec) {                      \
    case TM_F64: {                     \
      constexpr int P = TM_F64;        \
      F;                               \
    } break;                           \
    case TM_F32: {                     \
      constexpr int P = TM_F32;        \
      F;                               \
    } break;                           \
    case TM_DF64: {                    \
      constexpr int P = TM_DF64;       \
      F;                               \
    } break;                           \
    default: {                         \
      constexpr int P = TM_F16;        \
      F;                               \
    } break;                           \
  }

tm_status pack_full_parity(tm_lattice lat, int prec, void* dst, const double* src_full, int parity, int g5,
                           cudaStream_t s) {
  const Geom& g = lat->geom;
  const unsigned nb = (unsigned)((g.h + FNT - 1) / FNT);
  TM_PREC_SWITCH(prec, (pack_kernel<P, true, P != TM_DF64><<<nb, FNT, 0, s>>>(g, src_full, static_cast<char*>(dst), 0, parity, g5,
                                                         canon_aligned(src_full))));
  count_launch();
  return cuda_check(cudaGetLastError(), "pack kernel");
}

tm_status unpack_full_parity(tm_lattice lat, int prec, double* dst_full, const void* src, int parity, int g5,
                             cudaStream_t s) {
  const Geom& g = lat->geom;
  const unsigned nb = (unsigned)((g.h + FNT - 1) / FNT);
  TM_PREC_SWITCH(prec, (unpack_kernel<P, true, true><<<nb, FNT, 0, s>>>(g, static_cast<const char*>(src), 0, dst_full, parity,
                                                           g5, canon_aligned(dst_full))));
  count_launch();
  return cuda_check(cudaGetLastError(), "unpack kernel");
}

tm_status convert_half(tm_lattice lat, int prec_out, void* dst, int prec_in, const void* src, cudaStream_t s) {
  const int h = lat->geom.h;
  const unsigned nb = (unsigned)((h + FNT - 1) / FNT);
  const char* in = static_cast<const char*>(src);
  char* out = static_cast<char*>(dst);
#define TM_CONV(A, B) \
  if (prec_in == A && prec_out == B) convert_kernel<A, B><<<nb, FNT, 0, s>>>(h, in, out);
  TM_CONV(TM_F64, TM_F64)
  TM_CONV(TM_F64, TM_F32)
  TM_CONV(TM_F64, TM_F16)
  TM_CONV(TM_F32, TM_F64)
  TM_CONV(TM_F32, TM_F32)
  TM_CONV(TM_F32, TM_F16)
  TM_CONV(TM_F16, TM_F64)
  TM_CONV(TM_F16, TM_F32)
  TM_CONV(TM_F16, TM_F16)
  TM_CONV(TM_F64, TM_DF64)
  TM_CONV(TM_DF64, TM_F64)
  TM_CONV(TM_DF64, TM_F32)
  TM_CONV(TM_F32, TM_DF64)
  TM_CONV(TM_DF64, TM_DF64)
#undef TM_CONV
  count_launch();
  return cuda_check(cudaGetLastError(), "convert kernel");
}

tm_status diag_apply(tm_lattice lat, int prec, void* out, const void* in, int nrhs, double dur, double dui,
                     double dlr, double dli, cudaStream_t s) {
  const int h = lat->geom.h;
  const size_t stride = spinor_bytes_per_site(prec) * lat->h;
  dim3 grid((h + FNT - 1) / FNT, nrhs);
  TM_PREC_SWITCH(prec, (diag_kernel<P><<<grid, FNT, 0, s>>>(h, static_cast<const char*>(in), stride,
                                                              static_cast<char*>(out), stride, dur, dui, dlr,
                                                              dli)));
  count_launch();
  return cuda_check(cudaGetLastError(), "diagonal kernel");
}

// Staging of host buffers: returns a device pointer holding (or receiving) `bytes`.
const void* stage_in(tm_lattice lat, int slot, const void* src, size_t bytes, cudaStream_t s, tm_status* st) {
  *st = TM_OK;
  if (is_device_pointer(src)) return src;
  void* d = workspace(lat, slot, bytes, st);
  if (*st != TM_OK) return nullptr;
  *st = cuda_check(cudaMemcpyAsync(d, src, bytes, cudaMemcpyHostToDevice, s), "host-to-device copy");
  return d;
}
void* stage_out(tm_lattice lat, int slot, void* dst, size_t bytes, tm_status* st) {
  *st = TM_OK;
  if (is_device_pointer(dst)) return dst;
  return workspace(lat, slot, bytes, st);
}
tm_status stage_out_finish(void* dst, const void* dev, size_t bytes, cudaStream_t s) {
  if (dst == dev) return TM_OK;
  return cuda_check(cudaMemcpyAsync(dst, dev, bytes, cudaMemcpyDeviceToHost, s), "device-to-host copy");
}

}  // namespace tmq

using namespace tmq;

extern "C" {

tm_status tm_pack_half(tm_lattice lat, tm_prec prec, void* dst, const double* src, int nrhs, void* stream) {
  if (!lat || !dst || !src || nrhs < 1) return set_error(TM_ERR_ARG, "tm_pack_half: bad argument");
  if (prec < TM_F64 || prec > TM_DF64) return set_error(TM_ERR_ARG, "tm_pack_half: precision %d", (int)prec);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  tm_status st;
  const void* d = stage_in(lat, WS_STAGE_IN, src, (size_t)nrhs * lat->h * 24 * sizeof(double), s, &st);
  if (st != TM_OK) return st;
  const int h = lat->geom.h;
  dim3 grid((h + FNT - 1) / FNT, nrhs);
  const size_t stride = spinor_bytes_per_site(prec) * lat->h;
  TM_PREC_SWITCH(prec, (pack_kernel<P, false, P != TM_DF64><<<grid, FNT, 0, s>>>(lat->geom, static_cast<const double*>(d),
                                                                   static_cast<char*>(dst), stride, 0, 0,
                                                                   canon_aligned(d))));
  count_launch();
  return cuda_check(cudaGetLastError(), "tm_pack_half");
}

tm_status tm_unpack_half(tm_lattice lat, tm_prec prec, double* dst, const void* src, int nrhs, void* stream) {
  if (!lat || !dst || !src || nrhs < 1) return set_error(TM_ERR_ARG, "tm_unpack_half: bad argument");
  if (prec < TM_F64 || prec > TM_DF64) return set_error(TM_ERR_ARG, "tm_unpack_half: precision %d", (int)prec);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  tm_status st;
  const size_t bytes = (size_t)nrhs * lat->h * 24 * sizeof(double);
  void* d = stage_out(lat, WS_STAGE_OUT, dst, bytes, &st);
  if (st != TM_OK) return st;
  const int h = lat->geom.h;
  dim3 grid((h + FNT - 1) / FNT, nrhs);
  const size_t stride = spinor_bytes_per_site(prec) * lat->h;
  const char* in = static_cast<const char*>(src);
  const bool al = canon_aligned(d);
  // double-float fields that the L2 holds beside their canonical form (129 MB): whole records
  if (prec == TM_DF64 && 2 * stride * nrhs <= ((size_t)126 << 20))
    unpack_kernel<TM_DF64, false, false><<<grid, FNT, 0, s>>>(lat->geom, in, stride, static_cast<double*>(d), 0, 0, al);
  else
    TM_PREC_SWITCH(prec, (unpack_kernel<P, false, true><<<grid, FNT, 0, s>>>(lat->geom, in, stride,
                                                                       static_cast<double*>(d), 0, 0, al)));
  count_launch();
  st = cuda_check(cudaGetLastError(), "tm_unpack_half");
  if (st != TM_OK) return st;
  return stage_out_finish(dst, d, bytes, s);
}

tm_status tm_apply_Mee_inv(tm_lattice lat, void* out, const void* in, int flavour, tm_prec prec, int nrhs,
                           void* stream) {
  if (!lat || !out || !in || nrhs < 1) return set_error(TM_ERR_ARG, "tm_apply_Mee_inv: bad argument");
  if (flavour != 1 && flavour != -1) return set_error(TM_ERR_ARG, "tm_apply_Mee_inv: flavour must be +1 or -1");
  if (prec < TM_F64 || prec > TM_DF64) return set_error(TM_ERR_ARG, "tm_apply_Mee_inv: precision %d", (int)prec);
  const double mut = 2.0 * lat->kappa * lat->mu;
  const double n = 1.0 / (1.0 + mut * mut);
  return diag_apply(lat, prec, out, in, nrhs, n, -flavour * mut * n, n, flavour * mut * n,
                    static_cast<cudaStream_t>(stream));
}

}  // extern "C"
