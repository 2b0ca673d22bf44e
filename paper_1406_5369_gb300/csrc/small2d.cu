// Launcher of the FP64 cluster V-cycle of the small 2D levels (small2d.cuh).
#include "small2d.cuh"

#include <string.h>

#include "perdevice.h"

namespace mg {

namespace {

// One more than the blocks per cluster the device places with the most shared
// memory a block can have (16, a non-portable size, 8, or none).
PerDevice g_nctas;
int nctas() {
  // asked by small2d_probe only: not inside a stream capture
  return (int)per_device(g_nctas, [] { return 0LL; }) - 1;
}

template <bool CELL> void config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &at, size_t smem, int nctas, cudaStream_t s) {
  memset(&cfg, 0, sizeof cfg);
  memset(&at, 0, sizeof at);
  cfg.gridDim = dim3(nctas, 1, 1);
  cfg.blockDim = dim3(sm2::kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = nctas;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
}

constexpr size_t kMaxSmem = 226 * 1024;  // 1 KB less than a block can have: static shared memory

template <bool CELL> int probe() {
  auto kernel = sm2::k_small2d<CELL>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess) return 0;
  const bool big = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  for (int nctas : {16, 8}) {
    if (nctas > 8 && !big) continue;
    int clusters = 0;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    config<CELL>(cfg, at, kMaxSmem, nctas, 0);
    if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters >= 1) return nctas;
  }
  return 0;
}

// Fills the arguments; returns the shared memory per block, 0 when the
// hierarchy does not fit.
size_t fill(const Small2D &d, int nctas, sm2::Args &a) {
  memset(&a, 0, sizeof a);
  if (d.nlev < 2 || d.lg > sm2::kTopLog || d.lg < d.nlev - 1) return 0;
  int nd = d.lg - sm2::kLocalLog;
  if (nd < 0) nd = 0;
  if (nd > 0 && nctas < 2) return 0;
  if (d.nlev - nd < 1 || d.nlev - nd > sm2::kMaxLocal) return 0;
  a.nctas = nd ? nctas : 1;
  a.nd = nd;
  a.nl = d.nlev - nd;
  const double k = d.kx > d.ky ? d.kx : d.ky;
  if (!(k > 1e-200 && k < 1e200)) return 0;  // 1 / k is used; the general kernels take the others
  a.px = d.kx / k;
  a.py = d.ky / k;
  a.gamma = 1.0 - d.omega;
  a.edge = d.edge;
  a.jacobi = d.smoother != 0;
  a.nu1 = d.nu1;
  a.nu2 = d.nu2;
  a.polish = !d.polish ? 0 : d.nu2 > 0 ? 1 : 2;
  a.zero_top = d.zero;
  a.f_top = d.f;
  a.u_top = d.u;
  a.pitch_top = d.pitch;
  a.kinv = 1.0 / k;
  a.k = k;
  a.norm_out = d.norm_out;
  a.uh = d.uh;
  a.fc = d.fc;
  a.pitchc = d.pitchc;
  a.kc = 0.25 * k;
  auto rows = [&](int l) { return (1 << (d.lg - l)) - (d.cell ? 0 : 1); };
  if (nd > 0) {
    const int m = rows(nd);
    for (int r = 0; r <= a.nctas; r++) a.band[nd][r] = 1 + r * m / a.nctas;
    for (int l = nd - 1; l >= 0; l--) {
      a.band[l][0] = 1;
      for (int r = 1; r < a.nctas; r++) a.band[l][r] = 2 * a.band[l + 1][r] - (d.cell ? 1 : 0);
      a.band[l][a.nctas] = rows(l) + 1;
    }
  }
  size_t elems = 0;
  auto take = [&](size_t e) {
    const size_t at = elems;
    elems += e;
    return (int)at;
  };
  double kl = k;
  for (int l = 0; l < d.nlev; l++, kl *= 0.25) {
    sm2::Lev &L = a.lv[l];
    L.lg = d.lg - l;
    L.m = rows(l);
    int R = L.m;
    if (l < nd) {
      R = 0;
      for (int r = 0; r < a.nctas; r++) {
        const int b = a.band[l][r + 1] - a.band[l][r];
        if (b < 1) return 0;
        if (b > R) R = b;
      }
    }
    const size_t pitch = L.m + 2;
    L.u = take((R + 2) * pitch);
    L.v = a.jacobi ? take((R + 2) * pitch) : L.u;
    L.f = take(R * pitch);
    L.r = take((R + 1) * pitch);
    L.s = d.sigma / kl;
    for (int c = 0; c < 4; c++) {
      const double dx = (c & 1) ? d.edge : 2, dy = (c & 2) ? d.edge : 2;
      L.w[c] = d.omega / (L.s + a.px * dx + a.py * dy);
    }
    a.dense_k = kl;
  }
  a.dense = d.dense;
  a.one = 1.0 / (2.0 * (a.px + a.py));
  a.total = (int)elems;
  const size_t smem = elems * sizeof(double);
  return smem <= kMaxSmem ? smem : 0;
}

template <bool CELL> cudaError_t launch(const sm2::Args &a, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  config<CELL>(cfg, at, smem, a.nctas, s);
  cudaError_t e = cudaLaunchKernelEx(&cfg, sm2::k_small2d<CELL>, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

void small2d_probe() {
  per_device(g_nctas, [] {
    const int node = probe<false>(), cell = probe<true>();
    cudaGetLastError();  // a refused query leaves no sticky error behind
    return 1LL + (node < cell ? node : cell);
  });
}

bool small2d_ok(const Small2D &d) {
  sm2::Args a;
  const int n = nctas();
  return n > 0 && fill(d, n, a) != 0;
}

cudaError_t small2d_cycle(const Small2D &d, cudaStream_t s) {
  sm2::Args a;
  const int n = nctas();
  const size_t smem = n > 0 ? fill(d, n, a) : 0;
  if (!smem) return cudaErrorInvalidValue;
  return d.cell ? launch<true>(a, smem, s) : launch<false>(a, smem, s);
}

}  // namespace mg
