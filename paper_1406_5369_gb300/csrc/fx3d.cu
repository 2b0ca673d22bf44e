// Fixed-point passes of the FP64 3D node levels (fx3d.cuh): operator set-up and dispatch.
#include <string.h>

#include "fx3d.cuh"

namespace mg {
namespace d3 {

namespace {

bool fx_args(fx3::Args &a, const Level &L, int smoother, double omega, bool corr) {
  memset(&a, 0, sizeof a);
  const double k[3] = {L.c[0] * L.inv_h2, L.c[1] * L.inv_h2, L.c[2] * L.inv_h2};
  return fx3::set_operator(a, k, omega, corr, smoother == 0 ? 2 : 1);
}

}  // namespace

bool fx_ok(const Level &L, int smoother, double omega) {
  fx3::Args a;
  return L.dim == 3 && L.dtype == F64 && !L.kf[0] && L.n >= kFxMinN && L.n <= kFxMaxN &&
         fx_args(a, L, smoother, omega, true);
}

cudaError_t fx_pass(const Level &L, const Level *C, int smoother, double omega, const void *uin, void *uout, bool zero,
                    const void *ec, void *fc, double *partials, int *nparts, cudaStream_t s) {
  fx3::Args a;
  if (!fx_args(a, L, smoother, omega, ec != nullptr)) return cudaErrorInvalidValue;
  a.uin = (const double *)uin;
  a.f = (const double *)L.f;
  a.uout = (double *)uout;
  a.ec = (const double *)ec;
  a.fc = (double *)fc;
  a.partials = partials;
  a.n = L.n;
  a.pitch = L.pitch;
  a.plane = L.plane;
  if (C) {
    a.nc = C->n;
    a.pitchc = C->pitch;
    a.planec = C->plane;
  }
  const bool gen = a.has_p[0] || a.has_p[1] || a.has_p[2];
  auto run = smoother == 0 ? (gen ? fx3::rbgs_gen : fx3::rbgs_iso) : (gen ? fx3::jacobi_gen : fx3::jacobi_iso);
  return run(a, zero, ec != nullptr, fc ? fx3::kRestrict : partials ? fx3::kNorm : fx3::kNone, nparts, s);
}

}  // namespace d3
}  // namespace mg
