// Fixed-point passes of the FP64 2D node levels (fx2d.cuh): operator set-up and dispatch.
#include <string.h>

#include "fx2d.cuh"

namespace mg {
namespace d2 {

namespace {

bool fx_args(fx2::Args &a, const Level &L, int smoother, double omega, bool corr) {
  memset(&a, 0, sizeof a);
  // stages of the longest pass: two sweeps
  const int stages = smoother == 0 ? 4 : 2;
  return fx2::set_operator(a, L.c[0] * L.inv_h2, L.c[1] * L.inv_h2, 0.0, 2, omega, corr, stages);
}

}  // namespace

bool fx_ok(const Level &L, int smoother, double omega) {
  fx2::Args a;
  return L.dim == 2 && L.dtype == F64 && !L.kf[0] && L.n >= kFxMinN && fx_args(a, L, smoother, omega, true);
}

cudaError_t fx_pass(const Level &L, const Level *C, int smoother, double omega, int nu, const void *uin, void *uout,
                    bool zero, const void *ec, void *fc, double *partials, int *nparts, int rows, cudaStream_t s) {
  fx2::Args a;
  if (!fx_args(a, L, smoother, omega, ec != nullptr)) return cudaErrorInvalidValue;
  a.uin = (const double *)uin;
  a.f = (const double *)L.f;
  a.uout = (double *)uout;
  a.ec = (const double *)ec;
  a.fc = (double *)fc;
  a.partials = partials;
  a.max_parts = kMaxPartials;
  a.n = L.n;
  a.pitch = L.pitch;
  if (C) {
    a.nc = C->n;
    a.pitchc = C->pitch;
  }
  const int out = fc ? fx2::kRestrict : partials ? fx2::kNorm : fx2::kNone;
  const bool corr = ec != nullptr;
  return fx2::run(a, false, smoother != 0, rows, nu, zero, corr, out, nparts, s);
}

}  // namespace d2
}  // namespace mg
