// Cell-centred multigrid (include/mg_cc.h): the cell-centred grid type of
// the paper's feature model (Table 1) with Neumann or Dirichlet boundary
// faces, cell-centred restriction and constant interpolation (Sec. 4), on
// the FP64 operator sigma u - sum_d c_d d^2u/dx_d^2 (finite volumes).
//
// Layout: level l has n_l = n / 2^l cells per dimension, four FP64 fields
// u[0], u[1] (Jacobi ping-pong), f, r with rows padded to 128 bytes (pitch =
// n_l rounded up to 16 doubles), x fastest, no ghost cells: the kernels read
// a neighbour only across an interior face and apply the boundary rule
// (zero flux, or the ghost -u_p of a homogeneous Dirichlet face) in
// registers. One thread per cell (per cell of the swept colour for
// red-black Gauss-Seidel), rows on blockIdx.y, planes on blockIdx.z, so a
// warp reads consecutive doubles of one row.
#include <math.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <cuda_runtime.h>

#include "fx2d.cuh"
#include "mg_cc.h"
#include "mg_internal.h"
#include "stepgraph.h"

namespace mg {
namespace cc {

constexpr int kMaxLev = 16;
constexpr int kCoarseMax = 64;  // unknowns of the largest coarsest grid (4^3)
constexpr int kThreads = 256;
constexpr int kNormBlocks = 4096;  // enough blocks to hide FP64 latency on every level

struct Geo {
  int n;
  long long sy, sz;  // row and plane strides (elements)
};

// FP64 runs at 1/64 of the FP32 rate on this GPU, so the kernels are bound
// by FP64 issue, not by memory: the operator is written to need few FP64
// instructions per cell. A boundary face uses a ghost value (u_p for a
// Neumann face, -u_p for a Dirichlet one), so every face is one subtraction
// u_p - u_q (exactly 0 or 2 u_p at the boundary, as the operator defines),
// and the smoothers multiply by omega / diag_p from a table instead of
// dividing: diag_p depends only on which faces of the cell are boundary
// faces, class a_d = [x_d == 0] + [x_d == n-1] per axis, 3^dim classes.
struct Coef {
  double k[3];        // c_d / h^2 = c_d n^2 (exact scaling: n is a power of two)
  double sigma, ih2;  // ih2 = 1/h^2 = n^2
  int neumann;        // ghost value u_p (Neumann) or -u_p (Dirichlet)
  double wd[27];      // omega / diag by boundary class a_0 + 3 a_1 + 9 a_2
};

// (A u)_p of cell (i, j, k) at index p (the operator of mg_cc.h); cls gets
// the cell's boundary class.
template <int DIM>
__device__ __forceinline__ double apply(const double *__restrict__ u, long long p, int i, int j, int k,
                                        const Geo &g, const Coef &s, int &cls) {
  const double u0 = u[p], gh = s.neumann ? u0 : -u0;
  const int x[3] = {i, j, k};
  const long long st[3] = {1, g.sy, g.sz};
  const int mul[3] = {1, 3, 9};
  double acc = 0.0;
  cls = 0;
#pragma unroll
  for (int d = 0; d < DIM; d++) {
    const bool lo = x[d] == 0, hi = x[d] == g.n - 1;
    const double um = lo ? gh : u[p - st[d]];
    const double up = hi ? gh : u[p + st[d]];
    acc += s.k[d] * ((u0 - um) + (u0 - up));
    cls += mul[d] * ((int)lo + (int)hi);
  }
  return s.sigma * u0 + acc;
}

struct Cell {
  int i, j, k;
  long long p;
  bool ok;
};

template <int DIM> __device__ __forceinline__ Cell cell_of(const Geo &g, int i) {
  Cell c;
  c.i = i;
  c.j = blockIdx.y;
  c.k = DIM == 3 ? (int)blockIdx.z : 0;
  c.p = (long long)c.k * g.sz + (long long)c.j * g.sy + i;
  c.ok = i < g.n;
  return c;
}

// Half-sweep of red-black Gauss-Seidel: thread t of a row takes the t-th
// cell of the colour ((i + j + k) % 2 == color) in that row.
template <int DIM>
__global__ void k_rbgs_half(double *__restrict__ u, const double *__restrict__ f, Geo g, Coef s, int color) {
  const int j = blockIdx.y, k = DIM == 3 ? (int)blockIdx.z : 0;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  Cell c = cell_of<DIM>(g, 2 * t + ((color + j + k) & 1));
  if (!c.ok) return;
  int cls;
  const double Au = apply<DIM>(u, c.p, c.i, c.j, c.k, g, s, cls);
  u[c.p] = u[c.p] + s.wd[cls] * (f[c.p] - Au);
}

template <int DIM>
__global__ void k_jacobi(const double *__restrict__ uin, double *__restrict__ uout, const double *__restrict__ f,
                         Geo g, Coef s) {
  Cell c = cell_of<DIM>(g, blockIdx.x * blockDim.x + threadIdx.x);
  if (!c.ok) return;
  int cls;
  const double Au = apply<DIM>(uin, c.p, c.i, c.j, c.k, g, s, cls);
  uout[c.p] = uin[c.p] + s.wd[cls] * (f[c.p] - Au);
}

template <int DIM>
__global__ void k_residual(const double *__restrict__ u, const double *__restrict__ f, double *__restrict__ r,
                           Geo g, Coef s) {
  Cell c = cell_of<DIM>(g, blockIdx.x * blockDim.x + threadIdx.x);
  if (!c.ok) return;
  int cls;
  r[c.p] = f[c.p] - apply<DIM>(u, c.p, c.i, c.j, c.k, g, s, cls);
}

// Coarse cell (I, J, K): mean of its 2^DIM fine cells (2I+a, 2J+b, 2K+e).
template <int DIM>
__global__ void k_restrict(const double *__restrict__ rf, Geo gf, double *__restrict__ fc, Geo gc) {
  Cell c = cell_of<DIM>(gc, blockIdx.x * blockDim.x + threadIdx.x);
  if (!c.ok) return;
  double acc = 0.0;
#pragma unroll
  for (int e = 0; e < (DIM == 3 ? 2 : 1); e++)
#pragma unroll
    for (int b = 0; b < 2; b++) {
      const double *row = rf + (long long)(2 * c.k + e) * gf.sz + (long long)(2 * c.j + b) * gf.sy + 2 * c.i;
      acc += row[0];
      acc += row[1];
    }
  fc[c.p] = (DIM == 3 ? 0.125 : 0.25) * acc;
}

// Constant interpolation and correction: u_p += e_{parent(p)}.
template <int DIM>
__global__ void k_prolong(const double *__restrict__ ec, Geo gc, double *__restrict__ uf, Geo gf) {
  Cell c = cell_of<DIM>(gf, blockIdx.x * blockDim.x + threadIdx.x);
  if (!c.ok) return;
  uf[c.p] += ec[(long long)(c.k >> 1) * gc.sz + (long long)(c.j >> 1) * gc.sy + (c.i >> 1)];
}

// Fixed-order norm: block b sums r^2 over rows b, b + gridDim, ... (thread t
// over cells t, t + 256, ... of each row), then a fixed-shape tree; no 64-bit
// index division per cell.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double buf[kThreads];
  buf[threadIdx.x] = v;
  __syncthreads();
  for (int s = kThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) buf[threadIdx.x] += buf[threadIdx.x + s];
    __syncthreads();
  }
  return buf[0];
}

template <int DIM>
__global__ void k_norm_partials(const double *__restrict__ u, const double *__restrict__ f, Geo g, Coef s,
                                double *__restrict__ partials) {
  const int n = g.n, rows = DIM == 3 ? n * n : n;
  double acc = 0.0;
  for (int row = blockIdx.x; row < rows; row += gridDim.x) {
    const int j = row % n, k = DIM == 3 ? row / n : 0;
    const long long base = (long long)k * g.sz + (long long)j * g.sy;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      int cls;
      const double r = f[base + i] - apply<DIM>(u, base + i, i, j, k, g, s, cls);
      acc += r * r;
    }
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

__global__ void k_norm_final(const double *__restrict__ partials, int count, double *__restrict__ out) {
  double a = 0.0;
  for (int i = threadIdx.x; i < count; i += kThreads) a += partials[i];
  a = block_sum(a);
  if (threadIdx.x == 0) out[0] = sqrt(a);
}

// Cell t of the coarsest grid in lexicographic order (x fastest).
template <int DIM> __device__ __forceinline__ void coarse_cell(int t, int n, int &i, int &j, int &k) {
  i = t % n;
  j = DIM == 3 ? (t / n) % n : t / n;
  k = DIM == 3 ? t / (n * n) : 0;
}

// ------------------------------------------------------------------------
// Kernels of the V-cycle on levels that neither fx2d.cuh nor small2d.cuh takes
// (3D grids). FP64 instructions bound them (2.1 M cells: 3.5 us each), so the
// sweep is u' = gamma u + wd (f + sum_d k_d (um + up)), a missing neighbour
// counting as zero (7 instructions; the operator's difference
// form and a correction take 15), and the residual is restricted without being
// stored: the mean over a coarse cell needs the differences across its outer
// faces only, since what crosses an inner face cancels (7 per fine cell
// against 15). Blocks are 32 x 8 cells of a plane.
constexpr int kBX = 32, kBY = 8;

// f_p + sum_d k_d (um + up), one FMA per neighbour (an FP64 addition issues
// slower than an FMA here: 76 cycles of a scheduler against 64).
template <int DIM>
__device__ __forceinline__ double neighbours(const double *__restrict__ u, double f, long long p, int i, int j, int k,
                                             const Geo &g, const Coef &s, int &cls) {
  const int x[3] = {i, j, k};
  const long long st[3] = {1, g.sy, g.sz};
  const int mul[3] = {1, 3, 9};
  cls = 0;
#pragma unroll
  for (int d = 0; d < DIM; d++) {
    const bool lo = x[d] == 0, hi = x[d] == g.n - 1;
    f = fma(s.k[d], lo ? 0.0 : u[p - st[d]], f);
    f = fma(s.k[d], hi ? 0.0 : u[p + st[d]], f);
    cls += mul[d] * ((int)lo + (int)hi);
  }
  return f;
}

// POLISH: the difference form u + wd (f - A u), for the finest level of cycles
// that may be near the rounding floor. It rounds the solution once; the sum of
// neighbours rounds values of the size of diag u several times, and a solve that
// went on with it came to rest at 2 to 2.7 times the residual (3D, 8^3 to 128^3).
// With it in every cycle's last sweep a solve of 128^3, V(2,2), took 3.59 ms,
// without 3.33: solves take it when near_floor says so, then in all
// post-smoothing sweeps; a cycle called by itself, in its last one.
template <int DIM, bool POLISH>
__global__ void __launch_bounds__(kBX * kBY) kv_rbgs_half(double *u, const double *__restrict__ f, Geo g, Coef s,
                                                          double gamma, int color) {
  const int j = blockIdx.y * kBY + threadIdx.y, k = DIM == 3 ? (int)blockIdx.z : 0;
  const int i = 2 * (blockIdx.x * kBX + threadIdx.x) + ((color + j + k) & 1);
  if (i >= g.n || j >= g.n) return;
  const long long p = (long long)k * g.sz + (long long)j * g.sy + i;
  int cls;
  if (POLISH) {
    const double r = f[p] - apply<DIM>(u, p, i, j, k, g, s, cls);
    u[p] = fma(s.wd[cls], r, u[p]);
    return;
  }
  const double b = neighbours<DIM>(u, f[p], p, i, j, k, g, s, cls);
  const double v = s.wd[cls] * b;
  u[p] = gamma != 0.0 ? fma(gamma, u[p], v) : v;
}

template <int DIM, bool POLISH>
__global__ void __launch_bounds__(kBX * kBY) kv_jacobi(const double *__restrict__ uin, double *__restrict__ uout,
                                                       const double *__restrict__ f, Geo g, Coef s, double gamma) {
  const int i = blockIdx.x * kBX + threadIdx.x, j = blockIdx.y * kBY + threadIdx.y;
  const int k = DIM == 3 ? (int)blockIdx.z : 0;
  if (i >= g.n || j >= g.n) return;
  const long long p = (long long)k * g.sz + (long long)j * g.sy + i;
  int cls;
  if (POLISH) {
    const double r = f[p] - apply<DIM>(uin, p, i, j, k, g, s, cls);
    uout[p] = fma(s.wd[cls], r, uin[p]);
    return;
  }
  const double b = neighbours<DIM>(uin, f[p], p, i, j, k, g, s, cls);
  const double v = s.wd[cls] * b;
  uout[p] = gamma != 0.0 ? fma(gamma, uin[p], v) : v;
}

// Mean of the residuals of the fine cells of coarse cell x (nc per dimension);
// uh (may be NULL) receives their values of u.
template <int DIM>
__device__ __forceinline__ double restricted(const double *__restrict__ u, const double *__restrict__ f, const Geo &g,
                                             const Coef &s, const int (&x)[3], int nc, double *__restrict__ uh) {
  const long long st[3] = {1, g.sy, g.sz};
  const long long p = (long long)(2 * x[2]) * g.sz + (long long)(2 * x[1]) * g.sy + 2 * x[0];
  constexpr int N = 1 << DIM;
  double v[N], r = 0.0, su = 0.0;
#pragma unroll
  for (int c = 0; c < N; c++) {
    const long long q = p + (c & 1) + ((c >> 1) & 1) * g.sy + (c >> 2) * g.sz;
    v[c] = u[q];
    r += f[q];
    su += v[c];
    if (uh) uh[q] = v[c];
  }
  r = fma(-s.sigma, su, r);
#pragma unroll
  for (int d = 0; d < DIM; d++) {
    const bool lo = x[d] == 0, hi = x[d] == nc - 1;
    double t = 0.0;
#pragma unroll
    for (int c = 0; c < N; c++) {
      const long long q = p + (c & 1) + ((c >> 1) & 1) * g.sy + (c >> 2) * g.sz;
      const bool up = (c >> d) & 1;  // the cell's outer face on this axis
      const bool edge = up ? hi : lo;
      const double gh = s.neumann ? v[c] : -v[c];
      t += v[c] - (edge ? gh : u[up ? q + st[d] : q - st[d]]);
    }
    r = fma(-s.k[d], t, r);
  }
  return r * (DIM == 3 ? 0.125 : 0.25);
}

// u of a cell after the first sweep (first = 1: Jacobi) or red half-sweep (2)
// from zero, else 0.
template <int DIM>
__device__ __forceinline__ double first_sweep(double f, const Coef &s, const int (&x)[3], int n, int first) {
  const int mul[3] = {1, 3, 9};
  int cls = 0;
#pragma unroll
  for (int d = 0; d < DIM; d++) cls += mul[d] * ((int)(x[d] == 0) + (int)(x[d] == n - 1));
  return first == 1 || (first == 2 && ((x[0] + x[1] + x[2]) & 1) == 0) ? s.wd[cls] * f : 0.0;
}

// Coarse cell: f = mean of its fine cells' residuals; u = first_sweep. uh: see restricted.
template <int DIM>
__global__ void __launch_bounds__(kBX * kBY)
    kv_restrict(const double *__restrict__ u, const double *__restrict__ f, Geo g, Coef s, double *__restrict__ fc,
                double *__restrict__ uc, Geo gc, Coef sc, int first, double *__restrict__ uh) {
  const int x[3] = {(int)(blockIdx.x * kBX + threadIdx.x), (int)(blockIdx.y * kBY + threadIdx.y),
                    DIM == 3 ? (int)blockIdx.z : 0};
  if (x[0] >= gc.n || x[1] >= gc.n) return;
  const double r = restricted<DIM>(u, f, g, s, x, gc.n, uh);
  const long long P = (long long)x[2] * gc.sz + (long long)x[1] * gc.sy + x[0];
  fc[P] = r;
  uc[P] = first_sweep<DIM>(r, sc, x, gc.n, first);
}

// V-cycle of the 3D levels of at most 8^3 cells in one block, one thread per
// cell of the largest: some 10 launches of 2 us per level otherwise.
constexpr int kSmall3 = 8, kSmall3Lev = 4, kSmall3Threads = kSmall3 * kSmall3 * kSmall3;
struct Small3 {
  int nl, nu1, nu2, jacobi, start;  // start: as general_cycle's
  int polish;                       // level 0's post-smoothing (without any: pre-smoothing) in difference form
  double gamma;
  Coef s[kSmall3Lev];
  int n[kSmall3Lev];
  const double *f, *ainv;
  double *u;
  Geo g;  // of the top level's global fields
  double *uh, *fc;  // finest level: its pre-smoothed u and the next level's f, kept for the fields (else NULL)
  Geo gc;
};
__global__ void __launch_bounds__(kSmall3Threads) kv_small3(const __grid_constant__ Small3 a) {
  __shared__ double U[2][kSmall3Lev][kSmall3Threads], F[kSmall3Lev][kSmall3Threads];
  const int t = threadIdx.x;
  int cur[kSmall3Lev];
  auto cell = [&](int l, int (&x)[3]) {
    const int n = a.n[l];
    x[0] = t % n;
    x[1] = (t / n) % n;
    x[2] = t / (n * n);
    return t < n * n * n;
  };
  auto smooth = [&](int l, int sweeps, bool begun, bool polish) {
    const Geo g = {a.n[l], a.n[l], (long long)a.n[l] * a.n[l]};
    int x[3];
    const bool mine = cell(l, x);
    for (int h = begun ? 1 : 0; h < (a.jacobi ? sweeps : 2 * sweeps); h++) {
      const double *u = U[cur[l]][l];
      double *out = U[a.jacobi ? cur[l] ^ 1 : cur[l]][l];
      if (mine && (a.jacobi || ((x[0] + x[1] + x[2]) & 1) == (h & 1))) {
        int cls;
        if (polish) {
          const double r = F[l][t] - apply<3>(u, t, x[0], x[1], x[2], g, a.s[l], cls);
          out[t] = fma(a.s[l].wd[cls], r, u[t]);
        } else {
          const double b = neighbours<3>(u, F[l][t], t, x[0], x[1], x[2], g, a.s[l], cls);
          out[t] = fma(a.gamma, u[t], a.s[l].wd[cls] * b);
        }
      }
      if (a.jacobi) cur[l] ^= 1;
      __syncthreads();
    }
  };
  const int first = a.nu1 == 0 ? 0 : a.jacobi ? 1 : 2;
#pragma unroll
  for (int l = 0; l < kSmall3Lev; l++) cur[l] = 0;
  int x[3];
  long long top = 0;
  if (cell(0, x)) {
    top = (long long)x[2] * a.g.sz + (long long)x[1] * a.g.sy + x[0];
    F[0][t] = a.f[top];
    U[0][0][t] = a.start == 0 ? first_sweep<3>(F[0][t], a.s[0], x, a.n[0], first) : a.u[top];
  }
  __syncthreads();
#pragma unroll
  for (int l = 0; l < kSmall3Lev - 1; l++) {
    if (l + 1 >= a.nl) break;
    smooth(l, a.nu1, a.nu1 > 0 && (l > 0 || a.start >= 0), a.polish && l == 0 && a.nu2 == 0);
    if (cell(l + 1, x)) {
      const Geo g = {a.n[l], a.n[l], (long long)a.n[l] * a.n[l]};
      const double r = restricted<3>(U[cur[l]][l], F[l], g, a.s[l], x, a.n[l + 1], nullptr);
      F[l + 1][t] = r;
      U[0][l + 1][t] = l + 2 == a.nl ? 0.0 : first_sweep<3>(r, a.s[l + 1], x, a.n[l + 1], first);
      if (l == 0 && a.fc) a.fc[(long long)x[2] * a.gc.sz + (long long)x[1] * a.gc.sy + x[0]] = r;
    }
    if (l == 0 && a.uh && cell(0, x)) a.uh[top] = U[cur[0]][0][t];
    __syncthreads();
  }
  {
    const int l = a.nl - 1, N = a.n[l] * a.n[l] * a.n[l];
    if (t < N) {
      double acc = 0.0;
      for (int q = 0; q < N; q++) acc += a.ainv[q * N + t] * F[l][q];
      U[0][l][t] = acc;
    }
    __syncthreads();
  }
#pragma unroll
  for (int l = kSmall3Lev - 2; l >= 0; l--) {
    if (l + 1 >= a.nl) continue;
    if (cell(l, x)) {
      const int m = a.n[l + 1];
      U[cur[l]][l][t] += U[cur[l + 1]][l + 1][((x[2] >> 1) * m + (x[1] >> 1)) * m + (x[0] >> 1)];
    }
    __syncthreads();
    smooth(l, a.nu2, false, a.polish && l == 0);
  }
  if (cell(0, x)) a.u[top] = U[cur[0]][0][t];
}

// One block: assembles the coarsest operator over its N = n^DIM cells
// (row t: diag_t, and -c_d/h^2 for each neighbour across an interior face)
// and inverts it in place by Gauss-Jordan elimination without pivoting (A
// is symmetric positive definite: sigma > 0 or Dirichlet faces). A
// Dirichlet face adds 2 c_d/h^2 to the diagonal, a Neumann face nothing.
template <int DIM>
__global__ void k_dense_inverse(double *a, Geo g, Coef s) {
  __shared__ double colk[kCoarseMax];
  __shared__ double rpiv;
  const int n = g.n, N = DIM == 3 ? n * n * n : n * n;
  for (int e = threadIdx.x; e < N * N; e += blockDim.x) a[e] = 0.0;
  __syncthreads();
  for (int t = threadIdx.x; t < N; t += blockDim.x) {
    int x[3];
    coarse_cell<DIM>(t, n, x[0], x[1], x[2]);
    const int ts[3] = {1, n, n * n};
    double w = 0.0;
    for (int d = 0; d < DIM; d++) {
      if (x[d] > 0) {
        a[t * N + t - ts[d]] = -s.k[d];
        w += s.k[d];
      } else if (!s.neumann) {
        w += 2.0 * s.k[d];
      }
      if (x[d] < n - 1) {
        a[t * N + t + ts[d]] = -s.k[d];
        w += s.k[d];
      } else if (!s.neumann) {
        w += 2.0 * s.k[d];
      }
    }
    a[t * N + t] = s.sigma + w;
  }
  __syncthreads();
  for (int k = 0; k < N; k++) {
    if (threadIdx.x == 0) rpiv = 1.0 / a[k * N + k];
    for (int i = threadIdx.x; i < N; i += blockDim.x) colk[i] = a[i * N + k];
    __syncthreads();
    for (int j = threadIdx.x; j < N; j += blockDim.x) a[k * N + j] = (j == k ? 1.0 : a[k * N + j]) * rpiv;
    __syncthreads();
    for (int e = threadIdx.x; e < N * N; e += blockDim.x) {
      const int i = e / N, j = e % N;
      if (i == k) continue;
      a[e] = (j == k ? 0.0 : a[e]) - colk[i] * a[k * N + j];
    }
    __syncthreads();
  }
}

// One block: u += A^{-1} (f - A u) on the coarsest grid.
template <int DIM>
__global__ void k_coarse_solve(double *__restrict__ u, const double *__restrict__ f, Geo g, Coef s,
                               const double *__restrict__ ainv) {
  __shared__ double r[kCoarseMax];
  const int n = g.n, N = DIM == 3 ? n * n * n : n * n;
  for (int t = threadIdx.x; t < N; t += blockDim.x) {
    int i, j, k;
    coarse_cell<DIM>(t, n, i, j, k);
    const long long p = (long long)k * g.sz + (long long)j * g.sy + i;
    int cls;
    r[t] = f[p] - apply<DIM>(u, p, i, j, k, g, s, cls);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < N; t += blockDim.x) {
    double acc = 0.0;
    for (int q = 0; q < N; q++) acc += ainv[q * N + t] * r[q];
    int i, j, k;
    coarse_cell<DIM>(t, n, i, j, k);
    u[(long long)k * g.sz + (long long)j * g.sy + i] += acc;
  }
}

struct Lev {
  int n, pitch;
  long long plane, count;
  double *u[2], *f, *r;
  int cur;
};

}  // namespace cc
}  // namespace mg

using namespace mg::cc;

struct mg_cc_ctx {
  mg_cc_params p;
  int nl;
  Lev lv[kMaxLev];
  double *ainv;      // coarsest grid inverse, N x N
  double *partials;  // kNormBlocks norm partial sums
  double *norm_out;  // the norm (and its square)
  cudaStream_t s;
  int polish;        // sweeps in difference form that this cycle's finest level ends with: 0, 1, or 2 for a phase's all
  // The fields that a V-cycle leaves besides level 0's u (r of level 0; u, f and r
  // of the others) are formed when a call needs them (settle): the cycle keeps the
  // finest level's pre-smoothed u in its r, and the next level's f.
  bool unsettled;
  mg::StepGraphs graphs;
};

namespace {

thread_local char g_cc_err[256];

mg_status ccfail(mg_status st, const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_cc_err, sizeof g_cc_err, fmt, ap);
  va_end(ap);
  mg::set_error_message(g_cc_err);
  return st;
}

#define CCK(call)                                                                       \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) return ccfail(MG_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

bool pow2(int n) { return n >= 1 && (n & (n - 1)) == 0; }

mg_status check_params(const mg_cc_params *p) {
  if (!p) return ccfail(MG_EINVAL, "params are NULL");
  if (p->dim != 2 && p->dim != 3) return ccfail(MG_EINVAL, "dim must be 2 or 3 (got %d)", p->dim);
  if (!pow2(p->n) || p->n > (p->dim == 2 ? 16384 : 1024))
    return ccfail(MG_EINVAL, "n must be a power of two, at most %d in %dD (got %d)", p->dim == 2 ? 16384 : 1024,
                  p->dim, p->n);
  for (int d = 0; d < p->dim; d++)
    if (!(p->c[d] > 0.0)) return ccfail(MG_EINVAL, "axis coefficients must be > 0");
  if (p->bc != MG_CC_NEUMANN && p->bc != MG_CC_DIRICHLET) return ccfail(MG_EINVAL, "unknown boundary kind");
  if (!(p->sigma >= 0.0) || !isfinite(p->sigma)) return ccfail(MG_EINVAL, "sigma must be finite and >= 0");
  if (p->bc == MG_CC_NEUMANN && !(p->sigma > 0.0))
    return ccfail(MG_EINVAL, "sigma must be > 0 with Neumann faces (constants are a null space otherwise)");
  if (p->smoother != MG_RBGS && p->smoother != MG_JACOBI) return ccfail(MG_EINVAL, "unknown smoother");
  if (!(p->omega > 0.0 && p->omega < 2.0)) return ccfail(MG_EINVAL, "omega must lie in (0, 2)");
  if (p->nu1 < 0 || p->nu2 < 0 || p->nu1 > 8 || p->nu2 > 8 || p->nu1 + p->nu2 == 0)
    return ccfail(MG_EINVAL, "nu1, nu2 must lie in 0..8 with a positive sum");
  if (p->coarsest_n != 1 && p->coarsest_n != 2 && p->coarsest_n != 4)
    return ccfail(MG_EINVAL, "coarsest_n must be 1, 2 or 4 (got %d)", p->coarsest_n);
  if (p->coarsest_n > p->n) return ccfail(MG_EINVAL, "coarsest_n (%d) exceeds n (%d)", p->coarsest_n, p->n);
  if (p->maxit < 0) return ccfail(MG_EINVAL, "maxit must be >= 0");
  return MG_OK;
}

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

// Lays out the context's buffers from `base` (NULL: sizing only).
size_t layout(mg_cc_ctx *c, char *base) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = align256(off);
    void *q = base ? base + off : nullptr;
    off += bytes;
    return (double *)q;
  };
  const int dim = c->p.dim;
  c->nl = 0;
  for (int n = c->p.n; n >= c->p.coarsest_n; n /= 2) {
    Lev &L = c->lv[c->nl++];
    L.n = n;
    L.pitch = (n + 15) / 16 * 16;
    L.plane = (long long)L.pitch * n;
    L.count = L.plane * (dim == 3 ? n : 1);
    L.cur = 0;
    size_t bytes = (size_t)L.count * sizeof(double);
    L.u[0] = take(bytes);
    L.u[1] = take(bytes);
    L.f = take(bytes);
    L.r = take(bytes);
    if (n == c->p.coarsest_n) break;
  }
  const int nc = c->lv[c->nl - 1].n;
  const size_t N = (size_t)nc * nc * (dim == 3 ? nc : 1);
  c->ainv = take(N * N * sizeof(double));
  c->partials = take(kNormBlocks * sizeof(double));
  c->norm_out = take(sizeof(double));  // the rounding up to 256 bytes below leaves room for its square beside it
  return align256(off);
}

Geo geo_of(const Lev &L) { return Geo{L.n, (long long)L.pitch, L.plane}; }

Coef coef_of(const mg_cc_ctx *c, const Lev &L) {
  Coef s;
  memset(&s, 0, sizeof s);
  s.sigma = c->p.sigma;
  s.ih2 = (double)L.n * (double)L.n;
  for (int d = 0; d < 3; d++) s.k[d] = c->p.c[d] * s.ih2;
  const bool neumann = c->p.bc == MG_CC_NEUMANN;
  s.neumann = neumann;
  // diag of each boundary class: per axis, a_d boundary faces (a_d = 2 only
  // for a single cell) weigh 0 (Neumann) or 2 (Dirichlet), interior faces 1
  const int dim = c->p.dim;
  for (int cls = 0; cls < 27; cls++) {
    int a[3] = {cls % 3, (cls / 3) % 3, cls / 9};
    bool valid = true;
    double w = 0.0;
    for (int d = 0; d < 3; d++) {
      if (d >= dim) {
        valid = valid && a[d] == 0;
        continue;
      }
      if (a[d] == 2 && L.n != 1) valid = false;
      w += c->p.c[d] * ((2 - a[d]) + (neumann ? 0 : 2 * a[d]));
    }
    s.wd[cls] = valid ? c->p.omega / (s.sigma + w * s.ih2) : 0.0;
  }
  return s;
}

dim3 grid_of(const Lev &L, int cells_per_row) {
  return dim3((unsigned)((cells_per_row + kThreads - 1) / kThreads), (unsigned)L.n,
              L.count > L.plane ? (unsigned)L.n : 1u);
}

#define DIMCALL(dim, kern, grid, block, ...)                                    \
  do {                                                                          \
    if ((dim) == 2) kern<2><<<grid, block, 0, c->s>>>(__VA_ARGS__);             \
    else kern<3><<<grid, block, 0, c->s>>>(__VA_ARGS__);                        \
    CCK(cudaGetLastError());                                                    \
  } while (0)

mg_status op_smooth(mg_cc_ctx *c, int l, int sweeps) {
  Lev &L = c->lv[l];
  const Geo g = geo_of(L);
  const Coef s = coef_of(c, L);
  for (int it = 0; it < sweeps; it++) {
    if (c->p.smoother == MG_RBGS) {
      for (int color = 0; color < 2; color++)
        DIMCALL(c->p.dim, k_rbgs_half, grid_of(L, (L.n + 1) / 2), kThreads, L.u[L.cur], L.f, g, s, color);
    } else {
      DIMCALL(c->p.dim, k_jacobi, grid_of(L, L.n), kThreads, L.u[L.cur], L.u[L.cur ^ 1], L.f, g, s);
      L.cur ^= 1;
    }
  }
  return MG_OK;
}

mg_status op_residual(mg_cc_ctx *c, int l) {
  Lev &L = c->lv[l];
  DIMCALL(c->p.dim, k_residual, grid_of(L, L.n), kThreads, L.u[L.cur], L.f, L.r, geo_of(L), coef_of(c, L));
  return MG_OK;
}

mg_status op_restrict(mg_cc_ctx *c, int l) {
  Lev &F = c->lv[l], &C = c->lv[l + 1];
  DIMCALL(c->p.dim, k_restrict, grid_of(C, C.n), kThreads, F.r, geo_of(F), C.f, geo_of(C));
  return MG_OK;
}

mg_status op_prolong(mg_cc_ctx *c, int l) {
  Lev &F = c->lv[l], &C = c->lv[l + 1];
  DIMCALL(c->p.dim, k_prolong, grid_of(F, F.n), kThreads, C.u[C.cur], geo_of(C), F.u[F.cur], geo_of(F));
  return MG_OK;
}

mg_status op_coarse(mg_cc_ctx *c) {
  Lev &L = c->lv[c->nl - 1];
  DIMCALL(c->p.dim, k_coarse_solve, 1, 64, L.u[L.cur], L.f, geo_of(L), coef_of(c, L), c->ainv);
  return MG_OK;
}

mg_status norm_final(mg_cc_ctx *c, int nparts) {
  k_norm_final<<<1, kThreads, 0, c->s>>>(c->partials, nparts, c->norm_out);
  CCK(cudaGetLastError());
  return MG_OK;
}

mg_status op_norm(mg_cc_ctx *c, int l) {
  Lev &L = c->lv[l];
  DIMCALL(c->p.dim, k_norm_partials, kNormBlocks, kThreads, L.u[L.cur], L.f, geo_of(L), coef_of(c, L),
          c->partials);
  return norm_final(c, kNormBlocks);
}

mg_status read_norm(mg_cc_ctx *c, double *out) {
  CCK(cudaMemcpyAsync(out, c->norm_out, sizeof(double), cudaMemcpyDeviceToHost, c->s));
  CCK(cudaStreamSynchronize(c->s));
  return MG_OK;
}

// 2D levels of at least this size run on the fixed-point passes of fx2d.cuh:
// one launch per smoothing phase in place of 6 or more.
constexpr int kFxMinN = 64;

// The passes hold a strip's values as multiples of one unit, 54 to 57 bits below
// the largest. With a reaction term the solution may decay by e^-a per cell, a =
// sqrt(sigma / k); where that adds up to more than 2^-10 over the columns of a
// strip and the rows of a chunk the finest level, whose values are the result,
// stays in FP64 (its last digits would go first: sigma h^2 = 0.05, 512^2, solved to
// the rounding floor, had relative errors of 5e-12 in place of 5e-14 where the
// solution had fallen to 4e-12). A chunk is 8 rows or n^2 / 52 / 2432: one wave of
// warps, 52 columns each.
bool decays(const mg_cc_ctx *c, const Lev &L) {
  const double ih2 = (double)L.n * (double)L.n;
  const double rows = fmax(8.0, ih2 / (52.0 * 2432.0));
  const double a = mg::fx2::kCols * sqrt(c->p.sigma / (c->p.c[0] * ih2)) + rows * sqrt(c->p.sigma / (c->p.c[1] * ih2));
  return a > 10.0 * M_LN2;
}

// Level l's pass constants; false: the level keeps the kernels above.
bool fx_args(const mg_cc_ctx *c, int l, bool corr, mg::fx2::Args &a) {
  const Lev &L = c->lv[l];
  if (c->p.dim != 2 || L.n < kFxMinN || l + 1 >= c->nl || c->p.nu1 < 1 || c->p.nu2 < 1) return false;
  if (l == 0 && decays(c, L)) return false;
  memset(&a, 0, sizeof a);
  const double ih2 = (double)L.n * (double)L.n;
  return mg::fx2::set_operator(a, c->p.c[0] * ih2, c->p.c[1] * ih2, c->p.sigma, c->p.bc == MG_CC_NEUMANN ? 1 : 3,
                               c->p.omega, corr, c->p.smoother == MG_RBGS ? 4 : 2);
}
bool level_fx(const mg_cc_ctx *c, int l) {
  mg::fx2::Args a;
  return fx_args(c, l, true, a);
}

// One pass of level l: nu (1 or 2) sweeps from `in` (or zero) to `out`; before
// them the coarse correction (corr), after them the restricted residual (restr)
// or the partial sums of its square (nparts).
mg_status fx_pass(mg_cc_ctx *c, int l, const double *in, double *out_u, int nu, bool zero, bool corr, bool restr,
                  int *nparts) {
  Lev &L = c->lv[l], &C = c->lv[l + 1];
  mg::fx2::Args a;
  if (!fx_args(c, l, corr, a)) return ccfail(MG_EINVAL, "level %d has no fixed-point pass", l);
  a.uin = in;
  a.uout = out_u;
  a.f = L.f;
  a.ec = corr ? C.u[C.cur] : nullptr;
  a.fc = restr ? C.f : nullptr;
  a.partials = nparts ? c->partials : nullptr;
  a.max_parts = kNormBlocks;
  a.n = L.n;
  a.pitch = L.pitch;
  a.nc = C.n;
  a.pitchc = C.pitch;
  const int out = restr ? mg::fx2::kRestrict : nparts ? mg::fx2::kNorm : mg::fx2::kNone;
  CCK(mg::fx2::run(a, true, c->p.smoother != MG_RBGS, 0, nu, zero, corr, out, nparts, c->s));
  return MG_OK;
}

// The cluster V-cycle of levels l .. nl-1 (small2d.cuh); lg = 0 when the level does not take it.
mg::Small2D small_desc(const mg_cc_ctx *c, int l, bool zero) {
  mg::Small2D d;
  memset(&d, 0, sizeof d);
  const Lev &L = c->lv[l];
  if (c->p.dim != 2 || L.n > (1 << mg::kSmallTopLog) || l + 1 >= c->nl) return d;
  while ((1 << d.lg) < L.n) d.lg++;
  const double ih2 = (double)L.n * (double)L.n;
  d.cell = true;
  d.nlev = c->nl - l;
  d.kx = c->p.c[0] * ih2;
  d.ky = c->p.c[1] * ih2;
  d.sigma = c->p.sigma;
  d.edge = c->p.bc == MG_CC_NEUMANN ? 1 : 3;
  d.smoother = (int)c->p.smoother;
  d.nu1 = c->p.nu1;
  d.nu2 = c->p.nu2;
  d.omega = c->p.omega;
  d.zero = zero;
  d.polish = l == 0 && c->polish;
  d.f = L.f;
  d.u = L.u[L.cur];
  d.pitch = L.pitch;
  d.dense = c->ainv;
  if (l == 0) {
    d.uh = L.r;
    d.fc = c->lv[1].f;
    d.pitchc = c->lv[1].pitch;
  }
  return d;
}

dim3 tiles(const mg_cc_ctx *c, int nx, int n) {
  return dim3((unsigned)((nx + kBX - 1) / kBX), (unsigned)((n + kBY - 1) / kBY), c->p.dim == 3 ? (unsigned)n : 1u);
}

// A cycle that leaves the residual norm itself in c->norm_out sets *nparts to this.
constexpr int kNormDone = -1;
mg_status vcycle_rec(mg_cc_ctx *c, int l, bool zero = false, int *nparts = nullptr);

#define DIMCALL2(dim, flag, kern, grid, block, ...)                                  \
  do {                                                                               \
    if ((dim) == 2) {                                                                \
      if (flag) kern<2, true><<<grid, block, 0, c->s>>>(__VA_ARGS__);                \
      else kern<2, false><<<grid, block, 0, c->s>>>(__VA_ARGS__);                    \
    } else {                                                                         \
      if (flag) kern<3, true><<<grid, block, 0, c->s>>>(__VA_ARGS__);                \
      else kern<3, false><<<grid, block, 0, c->s>>>(__VA_ARGS__);                    \
    }                                                                                \
    CCK(cudaGetLastError());                                                         \
  } while (0)

// Sweeps of level l; begun: the first sweep (Jacobi) or red half-sweep is in u;
// polish: none, the last or all of them in difference form.
mg_status general_smooth(mg_cc_ctx *c, int l, int sweeps, bool begun, int polish) {
  const int fast = polish == 0 ? sweeps : polish == 1 ? sweeps - 1 : 0;
  Lev &L = c->lv[l];
  const Geo g = geo_of(L);
  const Coef s = coef_of(c, L);
  const double gamma = 1.0 - c->p.omega;
  const dim3 block(kBX, kBY);
  if (c->p.smoother == MG_RBGS) {
    for (int h = begun ? 1 : 0; h < 2 * sweeps; h++)
      DIMCALL2(c->p.dim, h >= 2 * fast, kv_rbgs_half, tiles(c, (L.n + 1) / 2, L.n), block, L.u[L.cur], L.f, g, s, gamma, h & 1);
  } else {
    for (int h = begun ? 1 : 0; h < sweeps; h++) {
      DIMCALL2(c->p.dim, h >= fast, kv_jacobi, tiles(c, L.n, L.n), block, L.u[L.cur], L.u[L.cur ^ 1], L.f, g, s, gamma);
      L.cur ^= 1;
    }
  }
  return MG_OK;
}

// One level of Algorithm 1 on the kv_ kernels. start: -1 u as it is, 0 from
// zero, 1 u holds the first (half-)sweep from zero.
mg_status general_cycle(mg_cc_ctx *c, int l, int start) {
  mg_status st;
  Lev &L = c->lv[l], &C = c->lv[l + 1];
  if (c->p.dim == 3 && L.n <= kSmall3 && c->nl - l <= kSmall3Lev) {
    Small3 a;
    memset(&a, 0, sizeof a);
    a.nl = c->nl - l;
    for (int i = 0; i < a.nl; i++) {
      a.s[i] = coef_of(c, c->lv[l + i]);
      a.n[i] = c->lv[l + i].n;
    }
    a.nu1 = c->p.nu1;
    a.nu2 = c->p.nu2;
    a.jacobi = c->p.smoother != MG_RBGS;
    a.start = start;
    a.polish = l == 0 && c->polish;
    a.gamma = 1.0 - c->p.omega;
    a.f = L.f;
    a.u = L.u[L.cur];
    a.g = geo_of(L);
    if (l == 0) {
      a.uh = L.r;
      a.fc = C.f;
      a.gc = geo_of(C);
    }
    a.ainv = c->ainv;
    kv_small3<<<1, kSmall3Threads, 0, c->s>>>(a);
    CCK(cudaGetLastError());
    return MG_OK;
  }
  if (start == 0) CCK(cudaMemsetAsync(L.u[L.cur], 0, (size_t)L.count * sizeof(double), c->s));
  if ((st = general_smooth(c, l, c->p.nu1, start == 1 && c->p.nu1 > 0, l == 0 && c->p.nu2 == 0 ? c->polish : 0))) return st;
  // the next level: u from its first sweep unless it solves, or starts by itself
  const bool last = l + 2 == c->nl, own = !last && (small_desc(c, l + 1, true).lg > 0 || level_fx(c, l + 1));
  const int first = last || own || c->p.nu1 == 0 ? 0 : c->p.smoother == MG_RBGS ? 2 : 1;
  DIMCALL(c->p.dim, kv_restrict, tiles(c, C.n, C.n), dim3(kBX, kBY), L.u[L.cur], L.f, geo_of(L), coef_of(c, L), C.f,
          C.u[C.cur], geo_of(C), coef_of(c, C), first, l == 0 ? L.r : nullptr);
  if (last) st = op_coarse(c);
  else if (own) st = vcycle_rec(c, l + 1, true);
  else st = general_cycle(c, l + 1, 1);
  if (st || (st = op_prolong(c, l))) return st;
  return general_smooth(c, l, c->p.nu2, false, l == 0 ? c->polish : 0);
}

// Algorithm 1 from level l down; coarse levels start from zero (`zero`: u_l
// counts as zero whatever its buffer holds). nparts (finest level, may be
// NULL): the number of partial sums of the squared residual that the last
// pass left in c->partials, 0 if it left none.
mg_status vcycle_rec(mg_cc_ctx *c, int l, bool zero, int *nparts) {
  mg_status st;
  Lev &L = c->lv[l];
  if (nparts) *nparts = 0;
  {
    mg::Small2D d = small_desc(c, l, zero);
    if (d.lg > 0 && mg::small2d_ok(d)) {
      if (nparts) {
        d.norm_out = c->norm_out;
        *nparts = kNormDone;
      }
      CCK(mg::small2d_cycle(d, c->s));
      return MG_OK;
    }
  }
  if (level_fx(c, l)) {
    // passes of at most two sweeps; more of them are passes of their own. The
    // pre-smoothed solution goes to r, where it stays.
    int left = c->p.nu1;
    if (zero && left > 2) {
      CCK(cudaMemsetAsync(L.u[L.cur], 0, (size_t)L.count * sizeof(double), c->s));
      zero = false;
    }
    for (; left > 2; left -= 2, L.cur ^= 1)
      if ((st = fx_pass(c, l, L.u[L.cur], L.u[L.cur ^ 1], 2, false, false, false, nullptr))) return st;
    if ((st = fx_pass(c, l, L.u[L.cur], L.r, left, zero, false, true, nullptr))) return st;
    if ((st = vcycle_rec(c, l + 1, true))) return st;
    left = c->p.nu2;
    const int first = left > 2 ? 2 : left;
    left -= first;
    if ((st = fx_pass(c, l, L.r, L.u[L.cur], first, false, true, false, left ? nullptr : nparts))) return st;
    for (; left > 0; left -= 2, L.cur ^= 1)
      if ((st = fx_pass(c, l, L.u[L.cur], L.u[L.cur ^ 1], left > 2 ? 2 : left, false, false, false, nullptr))) return st;
    return MG_OK;
  }
  if (l == c->nl - 1) {
    if (zero) CCK(cudaMemsetAsync(L.u[L.cur], 0, (size_t)L.count * sizeof(double), c->s));
    return op_coarse(c);
  }
  return general_cycle(c, l, zero ? 0 : -1);
}

// The finest level has sweeps in difference form (the fixed-point passes round
// once anyway).
bool polishes(const mg_cc_ctx *c) {
  const mg::Small2D d = small_desc(c, 0, false);
  return (d.lg > 0 && mg::small2d_ok(d)) || !level_fx(c, 0);
}

// Algorithm 1 on level l, one operator at a time: every level keeps its u, f and r.
mg_status plain_cycle(mg_cc_ctx *c, int l) {
  mg_status st;
  if (l == c->nl - 1) return op_coarse(c);
  if ((st = op_smooth(c, l, c->p.nu1))) return st;
  if ((st = op_residual(c, l))) return st;
  if ((st = op_restrict(c, l))) return st;
  Lev &C = c->lv[l + 1];
  CCK(cudaMemsetAsync(C.u[C.cur], 0, (size_t)C.count * sizeof(double), c->s));
  if ((st = plain_cycle(c, l + 1))) return st;
  if ((st = op_prolong(c, l))) return st;
  return op_smooth(c, l, c->p.nu2);
}

// Forms what the last V-cycle leaves on every level: the finest residual from the
// pre-smoothed solution kept in r, and the coarser levels by their part of the
// cycle, from level 1's right-hand side and zero.
mg_status settle(mg_cc_ctx *c) {
  if (!c->unsettled) return MG_OK;
  c->unsettled = false;
  Lev &L = c->lv[0], &C = c->lv[1];
  double *uh = L.u[L.cur ^ 1];
  CCK(cudaMemcpyAsync(uh, L.r, (size_t)L.count * sizeof(double), cudaMemcpyDeviceToDevice, c->s));
  DIMCALL(c->p.dim, k_residual, grid_of(L, L.n), kThreads, uh, L.f, L.r, geo_of(L), coef_of(c, L));
  CCK(cudaMemsetAsync(C.u[C.cur], 0, (size_t)C.count * sizeof(double), c->s));
  return plain_cycle(c, 1);
}

// Step k of a solve: a V-cycle and the residual norm.
mg_status solve_step(mg_cc_ctx *c, int k) {
  int status = 0;
  CCK(mg::step(
      c->graphs, k, c->s,
      [&] {
        unsigned b = c->polish ? 1u << 31 : 0u;
        for (int l = 0; l < c->nl; l++) b |= (unsigned)c->lv[l].cur << l;
        return b;
      },
      [&](unsigned b) {
        for (int l = 0; l < c->nl; l++) c->lv[l].cur = (b >> l) & 1u;
      },
      [&]() -> int {
        int np = 0;
        mg_status st = vcycle_rec(c, 0, false, &np);
        return st || np == kNormDone ? st : np ? norm_final(c, np) : op_norm(c, 0);
      },
      &status));
  c->unsettled = c->nl > 1;
  return (mg_status)status;
}

mg_status level_ok(const mg_cc_ctx *c, int level, bool need_coarser) {
  if (!c) return ccfail(MG_EINVAL, "NULL context");
  if (level < 0 || level >= c->nl - (need_coarser ? 1 : 0))
    return ccfail(MG_EINVAL, "level %d out of range", level);
  return MG_OK;
}

}  // namespace

extern "C" {

void mg_cc_default_params(mg_cc_params *p) {
  if (!p) return;
  memset(p, 0, sizeof *p);
  p->dim = 2;
  p->n = 2;
  p->c[0] = p->c[1] = p->c[2] = 1.0;
  p->sigma = 1.0;
  p->bc = MG_CC_NEUMANN;
  p->smoother = MG_RBGS;
  p->omega = 1.0;
  p->nu1 = 2;
  p->nu2 = 1;
  p->coarsest_n = 1;
  p->maxit = 50;
}

size_t mg_cc_workspace_bytes(const mg_cc_params *p) {
  if (check_params(p)) return 0;
  mg_cc_ctx tmp;
  memset(&tmp, 0, sizeof tmp);
  tmp.p = *p;
  return layout(&tmp, nullptr);
}

mg_status mg_cc_create(const mg_cc_params *p, void *arena, size_t arena_bytes, mg_cc_ctx **out) {
  if (!out) return ccfail(MG_EINVAL, "out is NULL");
  *out = nullptr;
  mg_status st = check_params(p);
  if (st) return st;
  if (!arena) return ccfail(MG_EINVAL, "arena is NULL");
  if ((uintptr_t)arena % 256) return ccfail(MG_EINVAL, "arena must be 256-byte aligned");
  mg_cc_ctx *c = (mg_cc_ctx *)calloc(1, sizeof(mg_cc_ctx));
  if (!c) return ccfail(MG_ENOMEM, "host allocation of the context failed");
  c->p = *p;
  c->s = (cudaStream_t)p->stream;
  if (p->dim == 2) mg::small2d_probe();
  size_t need = layout(c, nullptr);
  if (arena_bytes < need) {
    free(c);
    return ccfail(MG_ENOMEM, "arena has %zu bytes, %zu needed", arena_bytes, need);
  }
  layout(c, (char *)arena);
  cudaError_t e = cudaMemsetAsync(arena, 0, need, c->s);
  if (e == cudaSuccess) {
    Lev &Z = c->lv[c->nl - 1];
    if (p->dim == 2) k_dense_inverse<2><<<1, kThreads, 0, c->s>>>(c->ainv, geo_of(Z), coef_of(c, Z));
    else k_dense_inverse<3><<<1, kThreads, 0, c->s>>>(c->ainv, geo_of(Z), coef_of(c, Z));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->s);
  if (e != cudaSuccess) {
    free(c);
    return ccfail(MG_ECUDA, "creation: %s", cudaGetErrorString(e));
  }
  *out = c;
  return MG_OK;
}

mg_status mg_cc_destroy(mg_cc_ctx *c) {
  if (c) mg::drop(c->graphs);
  free(c);
  return MG_OK;
}

int mg_cc_num_levels(const mg_cc_ctx *c) { return c ? c->nl : -1; }

int mg_cc_level_size(const mg_cc_ctx *c, int level) {
  if (!c || level < 0 || level >= c->nl) return -1;
  return c->lv[level].n;
}

mg_status mg_cc_set_field(mg_cc_ctx *c, int level, int field, const double *src) {
  mg_status st = level_ok(c, level, false);
  if (st) return st;
  if (!src) return ccfail(MG_EINVAL, "src is NULL");
  if (field < 0 || field > 2) return ccfail(MG_EINVAL, "field must be 0 (u), 1 (f) or 2 (r)");
  if ((level > 0 || field == 2) && (st = settle(c))) return st;
  Lev &L = c->lv[level];
  double *dst = field == 0 ? L.u[L.cur] : (field == 1 ? L.f : L.r);
  const size_t rows = (size_t)L.n * (c->p.dim == 3 ? L.n : 1);
  CCK(cudaMemcpy2DAsync(dst, (size_t)L.pitch * 8, src, (size_t)L.n * 8, (size_t)L.n * 8, rows, cudaMemcpyDefault,
                        c->s));
  return MG_OK;
}

mg_status mg_cc_get_field(mg_cc_ctx *c, int level, int field, double *dst) {
  mg_status st = level_ok(c, level, false);
  if (st) return st;
  if (!dst) return ccfail(MG_EINVAL, "dst is NULL");
  if (field < 0 || field > 2) return ccfail(MG_EINVAL, "field must be 0 (u), 1 (f) or 2 (r)");
  if ((level > 0 || field == 2) && (st = settle(c))) return st;
  Lev &L = c->lv[level];
  const double *src = field == 0 ? L.u[L.cur] : (field == 1 ? L.f : L.r);
  const size_t rows = (size_t)L.n * (c->p.dim == 3 ? L.n : 1);
  CCK(cudaMemcpy2DAsync(dst, (size_t)L.n * 8, src, (size_t)L.pitch * 8, (size_t)L.n * 8, rows, cudaMemcpyDefault,
                        c->s));
  CCK(cudaStreamSynchronize(c->s));
  return MG_OK;
}

mg_status mg_cc_smooth(mg_cc_ctx *c, int level, int sweeps) {
  mg_status st = level_ok(c, level, false);
  if (st) return st;
  if (sweeps < 0) return ccfail(MG_EINVAL, "sweeps must be >= 0");
  return (st = settle(c)) ? st : op_smooth(c, level, sweeps);
}

mg_status mg_cc_residual(mg_cc_ctx *c, int level) {
  mg_status st = level_ok(c, level, false);
  return st || (st = settle(c)) ? st : op_residual(c, level);
}

mg_status mg_cc_restrict(mg_cc_ctx *c, int level) {
  mg_status st = level_ok(c, level, true);
  return st || (st = settle(c)) ? st : op_restrict(c, level);
}

mg_status mg_cc_prolongate(mg_cc_ctx *c, int level) {
  mg_status st = level_ok(c, level, true);
  return st || (st = settle(c)) ? st : op_prolong(c, level);
}

mg_status mg_cc_coarse_solve(mg_cc_ctx *c) {
  if (!c) return ccfail(MG_EINVAL, "NULL context");
  mg_status st = settle(c);
  return st ? st : op_coarse(c);
}

mg_status mg_cc_vcycle(mg_cc_ctx *c) {
  if (!c) return ccfail(MG_EINVAL, "NULL context");
  c->polish = polishes(c) ? 1 : 0;  // how near the floor this cycle is, is not known here
  c->unsettled = c->nl > 1;
  return vcycle_rec(c, 0);
}

mg_status mg_cc_residual_norm(mg_cc_ctx *c, int level, double *out) {
  mg_status st = level_ok(c, level, false);
  if (st) return st;
  if (!out) return ccfail(MG_EINVAL, "out is NULL");
  if (level > 0 && (st = settle(c))) return st;
  if ((st = op_norm(c, level))) return st;
  return read_norm(c, out);
}

mg_status mg_cc_solve(mg_cc_ctx *c, double tol, int *iters, double *relres, double *history) {
  if (!c) return ccfail(MG_EINVAL, "NULL context");
  if (!(tol >= 0.0)) return ccfail(MG_EINVAL, "tol must be >= 0");
  mg_status st;
  double r0;
  if ((st = op_norm(c, 0)) || (st = read_norm(c, &r0))) return st;
  if (history) history[0] = 1.0;
  if (!isfinite(r0)) return ccfail(MG_ENOCONV, "initial residual is not finite");
  int k = 0;
  double rho = r0 > 0.0 ? 1.0 : 0.0, last = INFINITY;
  while (r0 > 0.0 && rho > tol && k < c->p.maxit) {
    c->polish = polishes(c) && mg::near_floor(rho, last) ? 2 : 0;
    if ((st = solve_step(c, k))) return st;
    double rk;
    if ((st = read_norm(c, &rk))) return st;
    last = rho;
    rho = rk / r0;
    k++;
    if (history) history[k] = rho;
    if (!isfinite(rho)) break;
  }
  if (iters) *iters = k;
  if (relres) *relres = rho;
  if (!isfinite(rho)) return ccfail(MG_ENOCONV, "residual is not finite after %d cycles", k);
  if (rho > tol) return ccfail(MG_ENOCONV, "relative residual %.3e above tol %.3e after %d cycles", rho, tol, k);
  return MG_OK;
}

}  // extern "C"
