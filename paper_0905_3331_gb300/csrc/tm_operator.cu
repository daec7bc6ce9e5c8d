// tm_operator.cu -- the operator entry points: the hopping matrix H_{p,1-p} between half
// fields (eq. eo2 blocks) and the full operator M of eq. eo0 on canonical fields.
#include "tm_internal.cuh"

namespace tmq {

static bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const char* x = static_cast<const char*>(a);
  const char* y = static_cast<const char*>(b);
  return x < y + nb && y < x + na;
}

}  // namespace tmq

using namespace tmq;

extern "C" {

tm_status tm_apply_hopping_eo(tm_lattice lat, int out_parity, void* out, const void* in, tm_prec prec,
                              tm_link link, int nrhs, void* stream) {
  if (!lat || !out || !in || nrhs < 1) return set_error(TM_ERR_ARG, "tm_apply_hopping_eo: bad argument");
  if (out_parity != 0 && out_parity != 1)
    return set_error(TM_ERR_ARG, "tm_apply_hopping_eo: out_parity must be 0 or 1");
  if (prec < TM_F64 || prec > TM_DF64) return set_error(TM_ERR_ARG, "tm_apply_hopping_eo: precision %d", (int)prec);
  if (link != TM_LINK18 && link != TM_LINK12 && link != TM_LINK8)
    return set_error(TM_ERR_ARG, "tm_apply_hopping_eo: link format %d", (int)link);
  const size_t fb = tm_half_field_bytes(lat, prec);
  if (overlap(out, fb * nrhs, in, fb * nrhs)) return set_error(TM_ERR_ARG, "tm_apply_hopping_eo: out overlaps in");
  HopArgs a{};
  a.out_parity = out_parity;
  a.prec = prec;
  a.nreal = (int)link;
  a.nrhs = nrhs;
  a.in = in;
  a.in_stride = fb;
  a.out = out;
  a.out_stride = fb;
  a.coef = epi_plain();
  a.mode = 0;
  return hop_launch(lat, a, static_cast<cudaStream_t>(stream));
}

tm_status tm_apply_D(tm_lattice lat, double* out, const double* in, int flavour, int dagger, int nrhs,
                     void* stream) {
  if (!lat || !out || !in || nrhs < 1) return set_error(TM_ERR_ARG, "tm_apply_D: bad argument");
  if (flavour != 1 && flavour != -1) return set_error(TM_ERR_ARG, "tm_apply_D: flavour must be +1 or -1");
  if (!lat->has_gauge) return set_error(TM_ERR_NO_GAUGE, "tm_apply_D: no gauge field");
  const size_t fbytes = lat->V * 24 * sizeof(double);
  if (overlap(out, fbytes * nrhs, in, fbytes * nrhs)) return set_error(TM_ERR_ARG, "tm_apply_D: out overlaps in");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  tm_status st;
  const double* din = static_cast<const double*>(stage_in(lat, WS_STAGE_IN, in, fbytes * nrhs, s, &st));
  if (st != TM_OK) return st;
  double* dout = static_cast<double*>(stage_out(lat, WS_STAGE_OUT, out, fbytes * nrhs, &st));
  if (st != TM_OK) return st;
  // the FX form of a fixed number of fields, whatever nrhs is: a buffer sized by nrhs would be freed and
  // allocated anew by a call with more of them, under the feet of a captured one
  if ((st = ensure_links(lat, TM_F64, 18, s)) != TM_OK) return st;
  int per = full_fx_fields(lat, nrhs);
  if (per > 0 && lat->ws[WS_FULL_FX] == nullptr) {  // nothing is allocated in a capture: the form without a buffer, same bits
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();
    if (cap != cudaStreamCaptureStatusNone) per = 0;
  }
  void* w = nullptr;
  if (per > 0) w = workspace(lat, WS_FULL_FX, full_fx_bytes(lat->h) * per, &st);
  if (st != TM_OK) return st;
  // M^dag = g5 M(-f) g5
  if ((st = apply_full(lat, dout, din, dagger ? -flavour : flavour, dagger ? 1 : 0, nrhs, w, per, s)) != TM_OK) return st;
  return stage_out_finish(out, dout, fbytes * nrhs, s);
}

}  // extern "C"
