// FP64 V-cycle of the small 2D levels in one thread-block cluster (Algorithm 1
// from a level of at most 2^kTopLog cells per dimension down to the exact
// coarsest solve): node-based or cell-centred constant-stencil grids,
// red-black Gauss-Seidel or omega-Jacobi.
//
// These levels are bound by latency: one kernel launch per operator and level
// costs 2 .. 3 us each, one SM alone is short of FP64 units (two lanes), and a
// grid-wide barrier costs more than a cluster's. A cluster of 16 blocks (8
// where the device cannot place 16) keeps every level in shared memory. Block
// r owns a band of rows of each level with one halo row above and below; the
// bands of consecutive levels are nested, so transfers read own and halo rows
// only (node grids: one residual row comes from the block above). The thread
// that updates a node in a band's first or last row also stores it into the
// neighbour's halo row, and a cluster barrier ends the half-sweep: the
// neighbour, still in the same half-sweep, reads only the other colour of its
// halo row (Jacobi: the other buffer). Levels of at most 2^kLocalLog cells run
// in block 0 alone, with block barriers.
//
// Arithmetic is FP64 with few instructions per node: the right-hand side is
// held as f' = f / k (k the larger axis coefficient over h^2; the restriction
// to the next level multiplies by 4, exactly, since k does), so that
//   u' = W (f' + px (uw + ue) + py (us + un)) + gamma u,  max(px, py) = 1,
// W = omega / diag k by boundary class, and
//   r' = f' - [px ((u - uw) + (u - ue)) + py (...) + s u].
// Interior nodes (cells) have indices 1 .. m in both directions; indices 0
// and m + 1 hold the boundary nodes' values, or zero beside a cell grid,
// whose boundary faces then only change the diagonal (weights kx, ky = edge
// instead of 2 on u).
//
// Measured per V(2,1) cycle from 129^2, with the residual norm: 57 us, one
// launch, in place of 232 us in seven (block tiles for 129^2 and 65^2, the
// single-block cycle below, the norm). About 20 us are barriers (0.5 us each),
// the rest FP64 issue: 33^2 on all blocks instead of block 0 saved 5 us, a level
// of 257^2 taken along would add 40 us where the streaming passes take 35.
//
// Every block executes the same sequence of cluster barriers (the loop bounds
// are kernel arguments), and no block touches another's shared memory after
// the last one.
#pragma once

#include <cooperative_groups.h>

#include "mg_internal.h"

namespace mg {
namespace sm2 {

namespace cg = cooperative_groups;

constexpr int kThreads = 512;
constexpr int kMaxCTAs = 16;
constexpr int kTopLog = 8;    // largest level: 2^8 cells (257 nodes) per dimension
constexpr int kLocalLog = 4;  // levels up to 2^4 cells run in block 0
constexpr int kMaxDist = kTopLog - kLocalLog, kMaxLocal = kLocalLog + 1;

struct Lev {
  int lg, m;         // 2^lg cells per dimension; interior rows and columns
  int u, v, f, r;    // element offsets in shared memory (v: Jacobi's second buffer, else u)
  double s;          // sigma / k
  double w[4];       // W by boundary class: (row at the edge) * 2 + (column at the edge)
};

struct Args {
  int nctas, nd, nl;                    // blocks; distributed levels; local levels
  int band[kMaxDist + 1][kMaxCTAs + 1]; // level l, block r: rows [band[l][r], band[l][r + 1]); l = nd: first local level
  Lev lv[kMaxDist + kMaxLocal];
  double px, py, gamma, edge;           // edge: weight of u at a boundary face's axis (cells)
  int jacobi, nu1, nu2;
  int polish;        // top level's last sweep in difference form: 0 no, 1 the last post-smoothing, 2 pre-smoothing
  int zero_top;
  const double *f_top;
  double *u_top;
  int pitch_top;
  double kinv;       // 1 / k of the top level
  const double *dense;  // inverse of the coarsest operator, NULL for one node
  double dense_k;       // coarsest k: the inverse acts on f = f' k
  double one;           // one node: u = f' one
  double *norm_out;     // norm of the top residual and its square (NULL: none)
  double k;             // top k
  double *uh, *fc;      // the top level's pre-smoothed u, the next level's right-hand side (NULL: not stored)
  int pitchc;
  double kc;            // k of the next level
  int total;            // elements of shared memory
};

// A level as one block sees it: rows b0 .. b0 + R - 1, row q of U at global
// row b0 - 1 + q, row q of F at b0 + q, row q of the residual at b0 - 1 + q.
struct View {
  double *U, *V, *F, *T;
  int lg, m, pitch, b0, R;
};

template <bool LOCAL> __device__ __forceinline__ void barrier(cg::cluster_group &cl) {
  if (LOCAL) __syncthreads();
  else cl.sync();
}

__device__ __forceinline__ View view(const Args &a, double *sm, int l, int r) {
  const Lev &L = a.lv[l];
  View x;
  x.U = sm + L.u;
  x.V = sm + L.v;
  x.F = sm + L.f;
  x.T = sm + L.r;
  x.lg = L.lg;
  x.m = L.m;
  x.pitch = L.m + 2;
  x.b0 = l < a.nd ? a.band[l][r] : 1;
  x.R = l < a.nd ? a.band[l][r + 1] - x.b0 : L.m;
  return x;
}

template <bool CELL> __device__ __forceinline__ double weight(const Lev &L, int i, int j) {
  if (!CELL) return L.w[0];
  const bool ei = i == 1 || i == L.m, ej = j == 1 || j == L.m;
  return ej ? (ei ? L.w[3] : L.w[2]) : (ei ? L.w[1] : L.w[0]);
}

template <bool CELL>
__device__ __forceinline__ double resid(const Args &a, const Lev &L, const View &x, int jl, int i) {
  const int p = (jl + 1) * x.pitch + i, j = x.b0 + jl;
  const double u = x.U[p];
  double tx = (u - x.U[p - 1]) + (u - x.U[p + 1]), ty = (u - x.U[p - x.pitch]) + (u - x.U[p + x.pitch]);
  double r = x.F[jl * x.pitch + i];
  if (CELL) {
    // zero neighbours beside the grid: the two differences count 2 u
    if (i == 1 || i == x.m) tx += (x.m == 1 ? 2.0 : 1.0) * (a.edge - 2.0) * u;
    if (j == 1 || j == x.m) ty += (x.m == 1 ? 2.0 : 1.0) * (a.edge - 2.0) * u;
    r = fma(-L.s, u, r);
  }
  return r - fma(a.py, ty, a.px * tx);
}

// Sweeps of level l; returns with the result in x.U (Jacobi swaps the buffers
// and the caller's copy of the view with them). POLISH: as u + W r with the
// residual's differences, which rounds the solution once: the last sweep on the
// finest level. The sum of neighbours rounds several times, and a solve that ended
// with it came to rest at up to 2.5 times the residual (17^2 to 129^2). Ten V(2,1)
// cycles of 129^2: 677 us, 668 without.
template <bool CELL, bool LOCAL, bool POLISH>
__device__ __forceinline__ void sweep(const Args &a, cg::cluster_group &cl, double *sm, int l, int r, View &x,
                                      int sweeps) {
  const Lev &L = a.lv[l];
  const int pitch = x.pitch, rows = x.R;
  // the neighbours' bands start where this one ends: halo row indices there
  const bool up = !LOCAL && r > 0, dn = !LOCAL && r < a.nctas - 1;
  const int uprow = up ? x.b0 - a.band[l][r - 1] + 1 : 0;
  const int lgq = a.jacobi ? x.lg : x.lg - 1;  // threads per row, a power of two
  for (int st = 0; st < (a.jacobi ? sweeps : 2 * sweeps); st++) {
    const int color = st & 1;
    double *src = x.U, *dst = a.jacobi ? x.V : x.U;
    double *pu = up ? cl.map_shared_rank(dst, r - 1) + uprow * pitch : nullptr;
    double *pd = dn ? cl.map_shared_rank(dst, r + 1) : nullptr;
    for (int q = threadIdx.x; q < (rows << lgq); q += kThreads) {
      const int jl = q >> lgq, kk = q & ((1 << lgq) - 1), j = x.b0 + jl;
      const int i = a.jacobi ? kk + 1 : 2 * kk + 1 + ((color + j + 1) & 1);
      if (i > x.m) continue;
      const int p = (jl + 1) * pitch + i;
      const double u = src[p];
      double v;
      if (POLISH) {
        v = fma(weight<CELL>(L, i, j), resid<CELL>(a, L, x, jl, i), u);
      } else {
        const double sx = src[p - 1] + src[p + 1], sy = src[p - pitch] + src[p + pitch];
        v = weight<CELL>(L, i, j) * fma(a.py, sy, fma(a.px, sx, x.F[jl * pitch + i]));
        if (a.gamma != 0.0) v = fma(a.gamma, u, v);
      }
      dst[p] = v;
      if (jl == 0 && up) pu[i] = v;
      if (jl == rows - 1 && dn) pd[i] = v;
    }
    if (a.jacobi) {
      x.V = src;
      x.U = dst;
    }
    barrier<LOCAL>(cl);
  }
}

// The same, the last sweep polished where asked.
template <bool CELL, bool LOCAL>
__device__ __forceinline__ void smooth(const Args &a, cg::cluster_group &cl, double *sm, int l, int r, View &x,
                                       int sweeps, bool polish) {
  sweep<CELL, LOCAL, false>(a, cl, sm, l, r, x, polish ? sweeps - 1 : sweeps);
  if (polish) sweep<CELL, LOCAL, true>(a, cl, sm, l, r, x, 1);
}

// Residual rows of level l (node grids: the last row also to the block below).
// uh (may be NULL): the level's solution goes there.
template <bool CELL, bool LOCAL>
__device__ __forceinline__ void residual(const Args &a, cg::cluster_group &cl, int l, int r, const View &x, double *uh) {
  const Lev &L = a.lv[l];
  const int off = CELL ? 1 : 0;
  double *pd = !CELL && !LOCAL && r < a.nctas - 1 ? cl.map_shared_rank(x.T, r + 1) : nullptr;
  for (int q = threadIdx.x; q < (x.R << x.lg); q += kThreads) {
    const int jl = q >> x.lg, i = (q & ((1 << x.lg) - 1)) + 1;
    if (i > x.m) continue;
    const double v = resid<CELL>(a, L, x, jl, i);
    if (uh) uh[(long long)(x.b0 + jl - off) * a.pitch_top + i - off] = x.U[(jl + 1) * x.pitch + i];
    x.T[(jl + 1) * x.pitch + i] = v;
    if (pd && jl == x.R - 1) pd[i] = v;
  }
  if (!CELL) barrier<LOCAL>(cl);
  else __syncthreads();
}

// f' of the next level on rows [B0, B0 + RC): the restricted residual times 4
// (k falls by 4 from level to level). dst row of coarse row J: (J - row0). g
// (may be NULL): the level's global right-hand side f = f' kc.
template <bool CELL>
__device__ __forceinline__ void restrict_rows(const View &x, double *dst, int row0, int B0, int RC, double *g,
                                              int pitchc, double kc) {
  const int lgc = x.lg - 1, mc = CELL ? x.m / 2 : (x.m - 1) / 2, pc = mc + 2, p = x.pitch;
  for (int q = threadIdx.x; q < (RC << lgc); q += kThreads) {
    const int J = B0 + (q >> lgc), I = (q & ((1 << lgc) - 1)) + 1;
    if (I > mc) continue;
    double v;
    if (CELL) {
      const double *t = x.T + (2 * J - 1 - x.b0 + 1) * p + 2 * I - 1;
      v = (t[0] + t[1]) + (t[p] + t[p + 1]);
    } else {
      const double *t = x.T + (2 * J - x.b0 + 1) * p + 2 * I;
      const double e = (t[-p - 1] + t[-p + 1]) + (t[p - 1] + t[p + 1]);
      const double c = (t[-p] + t[p]) + (t[-1] + t[1]);
      v = 0.25 * fma(2.0, c, e) + t[0];
    }
    dst[(J - row0) * pc + I] = v;
    if (g) g[(long long)(J - (CELL ? 1 : 0)) * pitchc + I - (CELL ? 1 : 0)] = v * kc;
  }
}

// Correction of rows b0 - 1 .. b0 + R (halo rows with the same sums as their
// owners) by the coarse solution E, coarse row J at E + (J - row0) * pc.
template <bool CELL>
__device__ __forceinline__ void prolong_rows(const View &x, const double *E, int row0) {
  const int mc = CELL ? x.m / 2 : (x.m - 1) / 2, pc = mc + 2;
  for (int q = threadIdx.x; q < ((x.R + 2) << x.lg); q += kThreads) {
    const int jl = q >> x.lg, i = (q & ((1 << x.lg) - 1)) + 1, j = x.b0 - 1 + jl;
    if (i > x.m || j < 1 || j > x.m) continue;
    double v;
    if (CELL) {
      v = E[((j + 1) / 2 - row0) * pc + (i + 1) / 2];
    } else {
      const double *e = E + (j / 2 - row0) * pc + i / 2;
      v = (i & 1) ? 0.5 * (e[0] + e[1]) : e[0];
      if (j & 1) v = 0.5 * (v + ((i & 1) ? 0.5 * (e[pc] + e[pc + 1]) : e[pc]));
    }
    x.U[jl * x.pitch + i] += v;
  }
}

// Block 0's levels nd .. nd + nl - 1; the first one's f' is in place.
template <bool CELL> __device__ __forceinline__ void local_cycle(const Args &a, cg::cluster_group &cl, double *sm) {
  const int first = a.nd, last = a.nd + a.nl - 1;
  for (int l = first; l < last; l++) {
    View x = view(a, sm, l, 0);
    smooth<CELL, true>(a, cl, sm, l, 0, x, a.nu1, l == 0 && a.polish == 2);
    residual<CELL, true>(a, cl, l, 0, x, l == 0 ? a.uh : nullptr);
    const View c = view(a, sm, l + 1, 0);
    restrict_rows<CELL>(x, c.F, 1, 1, c.R, l == 0 ? a.fc : nullptr, a.pitchc, a.kc);
    __syncthreads();
  }
  {
    const View z = view(a, sm, last, 0);
    if (!a.dense) {
      if (threadIdx.x == 0) z.U[z.pitch + 1] = z.F[1] * a.one;
    } else {
      const int N = z.m * z.m;
      for (int t = threadIdx.x; t < N; t += kThreads) {
        double acc = 0.0;
        for (int q = 0; q < N; q++) acc += a.dense[(long long)q * N + t] * (z.F[(q / z.m) * z.pitch + q % z.m + 1] * a.dense_k);
        z.U[(t / z.m + 1) * z.pitch + t % z.m + 1] = acc;
      }
    }
    __syncthreads();
  }
  for (int l = last - 1; l >= first; l--) {
    View x = view(a, sm, l, 0);
    // Jacobi: the pre-smoothing left the solution in the buffer that an odd
    // number of sweeps swaps to; the coarser level's post-smoothing likewise
    if (a.jacobi && (a.nu1 & 1)) { double *t = x.U; x.U = x.V; x.V = t; }
    const View c = view(a, sm, l + 1, 0);
    const bool swapped = a.jacobi && l + 1 < last && ((a.nu1 + a.nu2) & 1);
    prolong_rows<CELL>(x, swapped ? c.V : c.U, 0);
    __syncthreads();
    smooth<CELL, true>(a, cl, sm, l, 0, x, a.nu2, l == 0 && a.polish == 1);
  }
}

template <bool CELL> __global__ void __launch_bounds__(kThreads, 1) k_small2d(const __grid_constant__ Args a) {
  cg::cluster_group cl = cg::this_cluster();
  const int r = (int)cl.block_rank();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *sm = (double *)smem_raw;
  for (int p = threadIdx.x; p < a.total; p += kThreads) sm[p] = 0.0;
  __syncthreads();
  const int off = CELL ? 1 : 0;  // global index of interior index i: i - off
  if (a.nd > 0 || r == 0) {
    const View x = view(a, sm, 0, r);
    for (int q = threadIdx.x; q < (x.R << x.lg); q += kThreads) {
      const int jl = q >> x.lg, i = (q & ((1 << x.lg) - 1)) + 1;
      if (i <= x.m) x.F[jl * x.pitch + i] = a.f_top[(long long)(x.b0 + jl - off) * a.pitch_top + i - off] * a.kinv;
    }
    if (!a.zero_top) {
      for (int q = threadIdx.x; q < (x.R + 2) * x.pitch; q += kThreads) {
        const int jl = q / x.pitch, i = q - jl * x.pitch, j = x.b0 - 1 + jl;
        if (CELL && (i < 1 || i > x.m || j < 1 || j > x.m)) continue;
        const double v = a.u_top[(long long)(j - off) * a.pitch_top + i - off];
        x.U[q] = v;
        x.V[q] = v;  // Jacobi: boundary values in both buffers
      }
    }
  }
  // every block has set up its shared memory before any block stores into it
  cl.sync();
  for (int l = 0; l < a.nd; l++) {
    View x = view(a, sm, l, r);
    smooth<CELL, false>(a, cl, sm, l, r, x, a.nu1, l == 0 && a.polish == 2);
    residual<CELL, false>(a, cl, l, r, x, l == 0 ? a.uh : nullptr);
    const int B0 = a.band[l + 1][r], RC = a.band[l + 1][r + 1] - B0;
    double *G = sm + a.lv[l + 1].f;
    double *g = l == 0 ? a.fc : nullptr;
    if (l + 1 < a.nd) restrict_rows<CELL>(x, G, B0, B0, RC, g, a.pitchc, a.kc);
    else restrict_rows<CELL>(x, cl.map_shared_rank(G, 0), 1, B0, RC, g, a.pitchc, a.kc);
    __syncthreads();
  }
  if (a.nd > 0) cl.sync();
  if (r == 0) local_cycle<CELL>(a, cl, sm);
  if (a.nd > 0) cl.sync();
  View x = view(a, sm, 0, r);
  const bool top_swapped = a.jacobi && ((a.nu1 + a.nu2) & 1);  // a smoothed level's solution after a cycle
  for (int l = a.nd - 1; l >= 0; l--) {
    x = view(a, sm, l, r);
    if (a.jacobi && (a.nu1 & 1)) { double *t = x.U; x.U = x.V; x.V = t; }
    const Lev &C = a.lv[l + 1];
    if (l + 1 < a.nd) {
      prolong_rows<CELL>(x, sm + (top_swapped ? C.v : C.u), a.band[l + 1][r] - 1);
    } else {
      const bool swapped = top_swapped && a.nl > 1;  // not the coarsest level
      prolong_rows<CELL>(x, cl.map_shared_rank(sm + (swapped ? C.v : C.u), 0), 0);
    }
    cl.sync();
    smooth<CELL, false>(a, cl, sm, l, r, x, a.nu2, l == 0 && a.polish == 1);
  }
  if (a.nd == 0 && top_swapped && a.nl > 1) { double *t = x.U; x.U = x.V; x.V = t; }
  __shared__ double sums[kMaxCTAs];  // block 0: every block's sum of squares
  if (a.nd > 0 || r == 0) {
    double acc = 0.0;
    for (int q = threadIdx.x; q < (x.R << x.lg); q += kThreads) {
      const int jl = q >> x.lg, i = (q & ((1 << x.lg) - 1)) + 1;
      if (i > x.m) continue;
      a.u_top[(long long)(x.b0 + jl - off) * a.pitch_top + i - off] = x.U[(jl + 1) * x.pitch + i];
      if (a.norm_out) {
        const double v = resid<CELL>(a, a.lv[0], x, jl, i) * a.k;
        acc += v * v;
      }
    }
    if (a.norm_out) {
      __shared__ double part[kThreads / 32];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
      if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
      __syncthreads();
      if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kThreads / 32; w++) t += part[w];
        *cl.map_shared_rank(&sums[r], 0) = t;
      }
    }
  }
  cl.sync();
  if (a.norm_out && r == 0 && threadIdx.x == 0) {
    double t = 0.0;
    for (int b = 0; b < a.nctas; b++) t += sums[b];
    a.norm_out[0] = sqrt(t);
    a.norm_out[1] = t;
  }
}

}  // namespace sm2
}  // namespace mg
