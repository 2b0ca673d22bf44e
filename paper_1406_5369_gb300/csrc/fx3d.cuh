// Fixed-point passes of the FP64 constant-stencil 3D levels (the arithmetic of
// fx2d.cuh).
//
// One sweep per pass, optionally with the coarse correction before it and the
// restricted residual or its norm after it. A block of 16 warps owns a column
// of 64 x 32 nodes (2 columns per lane, 2 rows per warp) of which the outer
// kHalo on each side are recomputed, and marches through a chunk of planes:
//
//   step t:  plane t is converted (and corrected); stage h (a half-sweep, or
//            the Jacobi sweep) runs on plane t - h; the smoothed plane t - S is
//            written; the residual is formed on plane t - S - 1.
//
// A thread keeps its own columns of the planes t .. t - S - 2 in registers; the
// rows beside its own come from shared memory, where every warp publishes the
// planes (a red-black half-sweep rewrites its colour in place, which nobody
// reads in that step), x-neighbours from shuffles. u and f are staged by
// cp.async a plane ahead; f stays staged and is converted where it is used (12
// registers per node less than keeping it). One block barrier per step; it
// also publishes each warp's largest exponent of the next plane, from which
// all threads take the same scale E. Rescaling (block-uniform, rare) shifts
// registers and the published planes. A block whose data the fixed point
// cannot hold starts again in FP64.
//
// Bound: integer issue (the ALU at 61 to 68 % while a block runs, 16 warps per SM)
// on 1.5 to 2 times the nodes, since the tiles' recomputed edges count: 257^3,
// V(2,2) red-black, one cycle's level in us, FP64 half-sweeps, residual,
// restriction and norm one by one -> these: 971 -> 717 (pre), 740 + 265 -> 841
// (post with the norm; 831 when it was that of the unrounded values).
#pragma once

#include "fx2d.cuh"

namespace mg {
namespace fx3 {

using fx2::expo;
using fx2::F64;
using fx2::Fix;
using fx2::fraction;
using fx2::kGen;
using fx2::kIso;
using fx2::kMaxE;
using fx2::kMinE;
using fx2::kNone;
using fx2::kNorm;
using fx2::kRestrict;
using fx2::Mul;
using fx2::mul62;
using fx2::shdn;
using fx2::shup;
using fx2::to_dbl;
using fx2::to_fix;

constexpr int kWarps = 16, kThreads = 32 * kWarps;
constexpr int kRows = 2 * kWarps, kCols = 64;
constexpr int kLo = 18;        // extra bits of f' (64 weights of the restriction fit an int)
constexpr int kRes = kLo + 6;  // low bits of a residual whose high part is r' / 64
constexpr int kPlaneB = kRows * kCols * 8;
constexpr int kFSlots = 6, kUSlots = 2, kPSlots = 4;

struct Args {
  const double *uin, *f, *ec;
  double *uout, *fc, *partials;
  int n, pitch, nc, pitchc;
  long long plane, planec;
  int ntx, nty, zc;  // blocks in x and y, planes per chunk (even)
  int P, fexp, fbound;
  double fscale, fpow;
  int has_p[3], has_gamma;
  Mul p[3], gamma, w;
  double k, dp[3], dgamma, dw;
  double km;  // k = km 2^ke
  int ke;
};

// fx2::stored on the integer pipe, 13 instructions: the warps of a block run in
// step, so the two conversions (128 cycles a value) add to every step (257^3,
// V(2,2): 15.16 ms a solve with them, 14.57 with this, 14.44 without any).
__device__ __forceinline__ long long stored(long long x) {
  const int hi = (int)(x >> 32);
  // bits beyond 53; -2^k counts one bit less than 2^k and loses none
  const int k = max(11 - __clz(hi ^ (hi >> 31)), 0);
  const unsigned m = (1u << k) - 1;
  const unsigned odd = __funnelshift_r((unsigned)x, (unsigned)hi, k) & m & 1u;
  return (x + (m >> 1) + odd) & ~(long long)m;
}

template <class A, int KIND>
__device__ __forceinline__ typename A::N relax(const Args &a, typename A::N u, typename A::N f, typename A::N sx,
                                               typename A::N sy, typename A::N sz) {
  if constexpr (A::fixed) {
    if (KIND == kGen) {
      if (a.has_p[0]) sx = mul62(sx, a.p[0]);
      if (a.has_p[1]) sy = mul62(sy, a.p[1]);
      if (a.has_p[2]) sz = mul62(sz, a.p[2]);
    }
    long long v = f + (sx + sy) + sz;
    if (KIND == kIso) {
      // gamma = 1 - 6 W: one multiplication does
      if (a.has_gamma) return u + mul62(v - 6 * u, a.w);
      return mul62(v, a.w);
    }
    v = mul62(v, a.w);
    if (a.has_gamma) {
      const long long g = mul62(u, a.gamma);
      v = a.dgamma < 0.0 ? v - g : v + g;
    }
    return v;
  } else {
    return a.dw * (f + a.dp[0] * sx + a.dp[1] * sy + a.dp[2] * sz) + a.dgamma * u;
  }
}

template <class A, bool JAC, int KIND, bool ZERO, bool CORR, int OUT>
__device__ __forceinline__ bool column(const Args &a, unsigned char *smem, double &acc) {
  typedef typename A::N N;
  constexpr bool FX = A::fixed;
  constexpr int S = JAC ? 1 : 2;
  // recomputed nodes on each side: one per stage, for the residual, its restriction
  // (nodes) and the interpolation, whose last column lacks its right neighbour
  constexpr int kNeed = S + (OUT != kNone) + (OUT == kRestrict) + (CORR);
  constexpr int kHalo = (kNeed + 1) / 2 * 2;
  constexpr int WU = S + 3;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = a.n, P = a.P;
  const int lo = 1, hi = n - 2;  // relaxed indices
  const int bx = blockIdx.x % a.ntx, by = blockIdx.x / a.ntx;
  const int c0 = bx * (kCols - 2 * kHalo) - kHalo + 2 * lane, y0 = by * (kRows - 2 * kHalo) - kHalo + 2 * w;
  const int z0 = blockIdx.y * a.zc, z1 = min(z0 + a.zc, n);
  const int tstart = max(z0 - 4, 0);  // even
  const int tend = OUT == kNone ? z1 - 1 + S : z1 + S + (OUT == kRestrict ? 1 : 0);
  const bool xout = lane >= kHalo / 2 && lane < 32 - kHalo / 2, yout = w >= kHalo / 2 && w < kWarps - kHalo / 2;
  bool in[2][2];  // [row][column]: relaxed on inner planes
#pragma unroll
  for (int r = 0; r < 2; r++)
#pragma unroll
    for (int q = 0; q < 2; q++) in[r][q] = y0 + r >= lo && y0 + r <= hi && c0 + q >= lo && c0 + q <= hi;
  auto plane_in = [&](int z) { return z >= lo && z <= hi; };

  // shared memory: published planes, staged f and u, restriction exchange, exponents
  N *pub = (N *)smem;
  unsigned char *sf = smem + kPSlots * kPlaneB, *su = sf + kFSlots * kPlaneB;
  N *xh = (N *)(su + kUSlots * kPlaneB);
  int *xl = (int *)(xh + kThreads);
  int *se = xl + kThreads;  // [2][kWarps]
  const int own = (2 * w) * kCols + 2 * lane;  // row A of this thread inside a plane; row B at + kCols

  N U[WU][2][2], Old[2][2], Z[2][2], Ec[2], xa = 0, xb = 0;
  int ZL[2][2], la = 0, lb = 0;
  double ne[2] = {0.0, 0.0};  // coarse values loaded for the next plane
#pragma unroll
  for (int r = 0; r < 2; r++) {
    Ec[r] = 0;
#pragma unroll
    for (int q = 0; q < 2; q++) {
      Old[r][q] = 0;
      Z[r][q] = 0;
      ZL[r][q] = 0;
#pragma unroll
      for (int i = 0; i < WU; i++) U[i][r][q] = 0;
    }
  }
  int E = kMinE;
  acc = 0.0;
  // Slots of the published planes: red-black p mod 4; Jacobi keeps the values
  // before (0, 1) and after (2, 3) the sweep.
  auto slot_of = [](int p, bool after) { return JAC ? (after ? 2 : 0) + (p & 1) : p & 3; };
  for (int i = 0; i < kPSlots; i++) {
    *(longlong2 *)(pub + i * (kRows * kCols) + own) = make_longlong2(0, 0);
    *(longlong2 *)(pub + i * (kRows * kCols) + own + kCols) = make_longlong2(0, 0);
  }
  xh[threadIdx.x] = 0;
  xl[threadIdx.x] = 0;

  const long long rowoff = (long long)y0 * a.pitch + c0;
  bool rowok[2];
#pragma unroll
  for (int r = 0; r < 2; r++) rowok[r] = c0 >= 0 && c0 < a.pitch && y0 + r >= 0 && y0 + r < n;
  // f of plane p stays in slot p mod kFSlots; fslot is plane t's
  int fslot = tstart % kFSlots;
  auto slot_at = [&](int d) {  // of plane t + d, -4 < d < 3
    const int v = fslot + d;
    return v < 0 ? v + kFSlots : v >= kFSlots ? v - kFSlots : v;
  };
  const double *pf = a.f + (long long)tstart * a.plane + rowoff, *pu = ZERO ? pf : a.uin + (long long)tstart * a.plane + rowoff;
  auto issue = [&](int t, int slot) {  // planes in turn
    const bool pok = t < n && t <= tend;
#pragma unroll
    for (int r = 0; r < 2; r++) {
      const bool ok = rowok[r] && pok;
      const int at = (own + r * kCols) * 8;
      fz::cp_async16(sf + slot * kPlaneB + at, ok ? pf + r * a.pitch : a.f, ok);
      if (!ZERO) fz::cp_async16(su + (t & 1) * kPlaneB + at, ok ? pu + r * a.pitch : a.uin, ok);
    }
    fz::cp_async_commit();
    pf += a.plane;
    pu += a.plane;
  };
  // f of plane t at this thread's nodes, zero where it is not part of the problem
  auto load_f = [&](int t, int slot, double (&fd)[2][2]) {
    const bool pin = plane_in(t);
#pragma unroll
    for (int r = 0; r < 2; r++) {
      const double2 v = *(const double2 *)(sf + slot * kPlaneB + (own + r * kCols) * 8);
      fd[r][0] = pin && in[r][0] ? v.x : 0.0;
      fd[r][1] = pin && in[r][1] ? v.y : 0.0;
    }
  };
  // Coarse values for plane t, where it brings a coarse plane: rows y0 / 2 and
  // y0 / 2 + 1 of plane (t + 1) / 2 (t odd, or t = tstart: of t / 2).
  auto load_e = [&](int K) {
    const int I = c0 >> 1, J = y0 >> 1;
#pragma unroll
    for (int r = 0; r < 2; r++) {
      const bool ok = c0 >= 0 && I < a.nc && y0 >= 0 && J + r < a.nc && K < a.nc;
      ne[r] = ok ? a.ec[(long long)K * a.planec + (long long)(J + r) * a.pitchc + I] : 0.0;
    }
  };
  // Largest exponent of plane t's staged values (and of ne) over the warp.
  auto publish_exponent = [&](int t, int slot, bool e) {
    int mu = 0, mf = 0;
    double fd[2][2];
    load_f(t, slot, fd);
#pragma unroll
    for (int r = 0; r < 2; r++) {
      mf = max(mf, max(__double2hiint(fd[r][0]) & 0x7fffffff, __double2hiint(fd[r][1]) & 0x7fffffff));
      if (!ZERO) {
        const double2 v = *(const double2 *)(su + (t & 1) * kPlaneB + (own + r * kCols) * 8);
        mu = max(mu, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
      }
      if (CORR && e) mu = max(mu, __double2hiint(ne[r]) & 0x7fffffff);
    }
    mf >>= 20;
    if (mf) mf = mf == 2047 ? 2047 + kMaxE : max(mf + a.fbound, 1);
    const int m = __reduce_max_sync(0xffffffffu, max(mu >> 20, mf));
    if (lane == 0) se[(t & 1) * kWarps + w] = m;
  };
  // Takes the block's largest exponent of plane t into the scale.
  auto take = [&](int t) -> bool {
    int e = 0;
#pragma unroll
    for (int i = 0; i < kWarps; i += 4) {
      const int4 v = *(const int4 *)(se + (t & 1) * kWarps + i);
      e = max(e, max(max(v.x, v.y), max(v.z, v.w)));
    }
    if (e <= E) return !(E == kMinE && e > 0);
    if (e > kMaxE) return false;
    if constexpr (FX) {
      for (int left = E == kMinE ? 0 : e - E; left > 0; left -= 30) {
        const int d = min(left, 30);
#pragma unroll
        for (int r = 0; r < 2; r++) {
#pragma unroll
          for (int q = 0; q < 2; q++) {
#pragma unroll
            for (int i = 0; i < WU; i++) U[i][r][q] >>= d;
            if (JAC) Old[r][q] >>= d;
            if (OUT == kRestrict) fx2::shift_pair(Z[r][q], ZL[r][q], kRes, d);
          }
          Ec[r] >>= d;
          for (int i = 0; i < kPSlots; i++) {
            longlong2 *p = (longlong2 *)(pub + i * (kRows * kCols) + own + r * kCols);
            *p = make_longlong2(p->x >> d, p->y >> d);
          }
        }
        if (OUT == kRestrict) {
          fx2::shift_pair(xa, la, kRes, d);
          fx2::shift_pair(xb, lb, kRes, d);
          xh[threadIdx.x] = xb;
          xl[threadIdx.x] = lb;
        }
      }
      __syncthreads();
    }
    E = e;
    return true;
  };
  // The neighbour in y of row r, column q that the adjacent warp published (only
  // that word: the other column may be written meanwhile, by a half-sweep).
  auto yother = [&](int slot, int r, int q) -> N {
    const int at = (r == 0 ? own - kCols : own + 2 * kCols) + q;
    const bool have = r == 0 ? w > 0 : w < kWarps - 1;
    return have ? pub[slot * (kRows * kCols) + at] : (N)0;
  };

  issue(tstart, fslot);
  if (CORR) load_e(tstart >> 1);
  fz::cp_async_wait<0>();
  bool good = true;
  if constexpr (FX) publish_exponent(tstart, fslot, true);
  issue(tstart + 1, slot_at(1));
  __syncthreads();

  auto step = [&](auto kc, const int t) -> bool {
    constexpr int K = decltype(kc)::value;  // parity of t
    if constexpr (FX) {
      if (!take(t)) return false;
    }
    // what the stages read of earlier steps' shared memory, all at once (the
    // latency is then paid once; none of it is written before they use it)
    double fs[S][2][2];
    N ys[S][2][2];
#pragma unroll
    for (int h = 1; h <= S; h++) {
      load_f(t - h, slot_at(-h), fs[h - 1]);
#pragma unroll
      for (int r = 0; r < 2; r++) {
        if (JAC) {
          ys[h - 1][r][0] = yother(slot_of(t - h, false), r, 0);
          ys[h - 1][r][1] = yother(slot_of(t - h, false), r, 1);
        } else {
          const int q = (h - 1 + r + K + h) & 1;
          ys[h - 1][r][q] = yother(slot_of(t - h, false), r, q);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 2; r++)
#pragma unroll
      for (int q = 0; q < 2; q++)
#pragma unroll
        for (int i = WU - 1; i > 0; i--) U[i][r][q] = U[i - 1][r][q];
    // ---- plane t
#pragma unroll
    for (int r = 0; r < 2; r++) {
      const double2 v = ZERO ? make_double2(0.0, 0.0) : *(const double2 *)(su + (t & 1) * kPlaneB + (own + r * kCols) * 8);
      if constexpr (FX) {
        U[0][r][0] = ZERO ? 0 : to_fix(v.x, E, P);
        U[0][r][1] = ZERO ? 0 : to_fix(v.y, E, P);
      } else {
        U[0][r][0] = v.x;
        U[0][r][1] = v.y;
      }
    }
    if (CORR) {
      // e[r]: correction at column c0 of coarse row J + r, plane t
      N e[2] = {Ec[0], Ec[1]};
      const bool fresh = K == 1 || t == tstart;
      if (fresh) {
#pragma unroll
        for (int r = 0; r < 2; r++) {
          if constexpr (FX) Ec[r] = to_fix(ne[r], E, P);
          else Ec[r] = ne[r];
        }
      }
      const bool pin = plane_in(t);
      N v[2][2];
      {
#pragma unroll
        for (int r = 0; r < 2; r++) {
          if constexpr (FX) e[r] = K == 1 ? (e[r] + Ec[r] + 1) >> 1 : Ec[r];
          else e[r] = K == 1 ? 0.5 * (e[r] + Ec[r]) : Ec[r];
        }
        if constexpr (FX) e[1] = (e[0] + e[1] + 1) >> 1;
        else e[1] = 0.5 * (e[0] + e[1]);
#pragma unroll
        for (int r = 0; r < 2; r++) {
          v[r][0] = e[r];
          if constexpr (FX) v[r][1] = (e[r] + shdn(e[r]) + 1) >> 1;
          else v[r][1] = 0.5 * (e[r] + shdn(e[r]));
        }
      }
#pragma unroll
      for (int r = 0; r < 2; r++)
#pragma unroll
        for (int q = 0; q < 2; q++)
          if (pin && in[r][q]) U[0][r][q] += v[r][q];
      // the next plane's coarse values, used at the end of this step
      if (K == 0) load_e((t + 2) >> 1);
    }
    issue(t + 2, slot_at(2));  // its staging slots held u of plane t and f of plane t - 4
    // ---- stage h on plane t - h
#pragma unroll
    for (int h = 1; h <= S; h++) {
      const int z = t - h;
      const bool pin = plane_in(z);
      double (&fd)[2][2] = fs[h - 1];
      if (a.fscale != 1.0) {
#pragma unroll
        for (int r = 0; r < 2; r++)
#pragma unroll
          for (int q = 0; q < 2; q++) fd[r][q] *= a.fscale;
      }
      N nv[2][2];
#pragma unroll
      for (int r = 0; r < 2; r++) {
        if (JAC) {
          const N left = shup(U[h][r][1]), right = shdn(U[h][r][0]);
#pragma unroll
          for (int q = 0; q < 2; q++) {
            N f;
            if constexpr (FX) f = to_fix(fd[r][q], E - a.fexp, P);
            else f = fd[r][q] * a.fpow;
            nv[r][q] = relax<A, KIND>(a, U[h][r][q], f, q == 0 ? left + U[h][r][1] : U[h][r][0] + right,
                                            ys[h - 1][r][q] + U[h][1 - r][q],
                                            Old[r][q] + U[h - 1][r][q]);
          }
        } else {
          // colour (h - 1) & 1 at columns with (c + y + z) of that parity; c0 and y0 are even
          const int q = (h - 1 + r + K + h) & 1;  // z = t - h has parity K + h
          N f;
          if constexpr (FX) f = to_fix(fd[r][q], E - a.fexp, P);
          else f = fd[r][q] * a.fpow;
          const N sx = q == 0 ? shup(U[h][r][1]) + U[h][r][1] : U[h][r][0] + shdn(U[h][r][0]);
          nv[r][q] = relax<A, KIND>(a, U[h][r][q], f, sx, ys[h - 1][r][q] + U[h][1 - r][q],
                                          U[h + 1][r][q] + U[h - 1][r][q]);
          nv[r][1 - q] = U[h][r][1 - q];
        }
      }
      if constexpr (FX && OUT == kNorm) {  // the norm is that of the stored solution
#pragma unroll
        for (int r = 0; r < 2; r++)
#pragma unroll
          for (int q = 0; q < 2; q++)
            if (JAC || q == ((h - 1 + r + K + h) & 1)) nv[r][q] = stored(nv[r][q]);
      }
#pragma unroll
      for (int r = 0; r < 2; r++) {
        if (JAC) {
#pragma unroll
          for (int q = 0; q < 2; q++) {
            Old[r][q] = U[h][r][q];  // before the sweep, for plane z + 1
            if (pin && in[r][q]) U[h][r][q] = nv[r][q];
          }
          N *p = pub + slot_of(z, true) * (kRows * kCols) + own + r * kCols;
          p[0] = U[h][r][0];
          p[1] = U[h][r][1];
        } else {
          const int q = (h - 1 + r + K + h) & 1;
          if (pin && in[r][q]) U[h][r][q] = nv[r][q];
          pub[slot_of(z, false) * (kRows * kCols) + own + r * kCols + q] = U[h][r][q];
        }
      }
    }
    // ---- plane t published as it is before its first stage
#pragma unroll
    for (int r = 0; r < 2; r++) {
      N *p = pub + slot_of(t, false) * (kRows * kCols) + own + r * kCols;
      p[0] = U[0][r][0];
      p[1] = U[0][r][1];
    }
    // ---- the smoothed plane t - S
    {
      const int z = t - S;
      if (z >= z0 && z < z1 && xout && yout) {
        const bool pin = plane_in(z);
#pragma unroll
        for (int r = 0; r < 2; r++) {
          if (y0 + r >= n) continue;
          double v[2];
#pragma unroll
          for (int q = 0; q < 2; q++) {
            if constexpr (FX) v[q] = to_dbl(U[S][r][q], E, P);
            else v[q] = U[S][r][q];
          }
          const long long off = (long long)z * a.plane + rowoff + (long long)r * a.pitch;
          if (pin && in[r][0] && in[r][1]) {
            *(double2 *)(a.uout + off) = make_double2(v[0], v[1]);
          } else {
            // boundary nodes keep their values
#pragma unroll
            for (int q = 0; q < 2; q++)
              if (c0 + q < n) a.uout[off + q] = pin && in[r][q] ? v[q] : ZERO ? 0.0 : a.uin[off + q];
          }
        }
      }
    }
    // ---- residual of plane t - S - 1
    if (OUT != kNone) {
      const int z = t - S - 1;
      constexpr int sc = S + 1;
      const bool pin = plane_in(z);
      double fd[2][2];
      load_f(z, slot_at(-S - 1), fd);
      N R[2][2];
      int RL[2][2];
#pragma unroll
      for (int r = 0; r < 2; r++) {
        const N left = shup(U[sc][r][1]), right = shdn(U[sc][r][0]);
#pragma unroll
        for (int q = 0; q < 2; q++) {
          const N u = U[sc][r][q];
          const N sx = q == 0 ? left + U[sc][r][1] : U[sc][r][0] + right;
          const N sy = yother(slot_of(z, true), r, q) + U[sc][1 - r][q], sz = U[sc - 1][r][q] + U[sc + 1][r][q];
          const bool ok = pin && in[r][q];
          if constexpr (FX) {
            int l;
            const double fs = a.fscale != 1.0 ? fd[r][q] * a.fscale : fd[r][q];
            const N f = fx2::to_fix2<kLo>(fs, E - a.fexp, P, l);
            if (KIND == kIso) {
              R[r][q] = f + (sx + sy) + sz - 6 * u;
            } else {
              long long tx = 2 * u - sx, ty = 2 * u - sy, tz = 2 * u - sz;
              if (a.has_p[0]) tx = mul62<kLo>(tx, a.p[0], l);
              if (a.has_p[1]) ty = mul62<kLo>(ty, a.p[1], l);
              if (a.has_p[2]) tz = mul62<kLo>(tz, a.p[2], l);
              R[r][q] = f - (tx + ty) - tz;
            }
            if (!ok) {
              R[r][q] = 0;
              l = 0;
            }
            RL[r][q] = l;
            if (OUT == kRestrict) {
              RL[r][q] = (((int)R[r][q] & 63) << kLo) + l;
              R[r][q] >>= 6;
            }
          } else {
            const double f = fd[r][q] * a.fscale * a.fpow;
            R[r][q] = ok ? f - (a.dp[0] * (2 * u - sx) + a.dp[1] * (2 * u - sy) + a.dp[2] * (2 * u - sz))
                         : 0.0;
            RL[r][q] = 0;
          }
        }
      }
      if constexpr (OUT == kNorm) {
        if (z >= z0 && z < z1 && xout && yout) {
          if constexpr (FX) {
            unsigned long long m = 0;
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
              for (int q = 0; q < 2; q++) m |= (unsigned long long)(R[r][q] ^ (R[r][q] >> 63));
            const int sh = min(max(__clzll((long long)m) - 2, 0), 40);
            unsigned long long sq = 0;
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
              for (int q = 0; q < 2; q++) {
                const long long l = sh >= kLo ? (long long)RL[r][q] << (sh - kLo) : (long long)(RL[r][q] >> (kLo - sh));
                const long long v = (R[r][q] << sh) + l;
                sq += (unsigned long long)__mul64hi(v, v);
              }
            const double d = __ull2double_rn(sq);
            const int ex = 64 - 2 * sh + 2 * (E - 1022 - P + a.ke) + (__double2hiint(d) >> 20);
            if (sq) acc += ex <= 0 ? 0.0
                           : ex >= 2047 ? __hiloint2double(0x7ff00000, 0)
                                        : __hiloint2double((ex << 20) | (__double2hiint(d) & 0xfffff),
                                                           __double2loint(d));
          } else {
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
              for (int q = 0; q < 2; q++) {
                const double v = R[r][q] * a.k;
                acc += v * v;
              }
          }
        }
      }
      if constexpr (OUT == kRestrict) {
        constexpr bool zodd = ((K + S + 1) & 1) != 0;  // parity of z
        const int I = c0 >> 1, J = y0 >> 1;
        const bool cin = xout && yout && I >= 1 && I <= a.nc - 2 && J >= 1 && J <= a.nc - 2;
        auto emit = [&](N v, int l, int Kc) {
          if (!(cin && Kc >= 1 && Kc <= a.nc - 2 && 2 * Kc >= z0 && 2 * Kc < z1)) return;
          double *dst = a.fc + (long long)Kc * a.planec + (long long)J * a.pitchc + I;
          if constexpr (FX) {
            const int sh = min(max(__clzll(v ^ (v >> 63)) - 2, 0), kRes);
            *dst = to_dbl((v << sh) + (l >> (kRes - sh)), E - sh, P) * a.k;
          } else {
            *dst = v * (a.k / 64.0);
          }
        };
        if (!zodd) {
          // the step after the odd plane z - 1: row y0 - 1's sum from the warp above
          const N up = w > 0 ? xh[threadIdx.x - 32] : 0;
          const int ul = w > 0 ? xl[threadIdx.x - 32] : 0;
          emit(up + 2 * xa + xb, ul + 2 * la + lb, (z - 2) >> 1);
        }
        if (!zodd) {
#pragma unroll
          for (int r = 0; r < 2; r++)
#pragma unroll
            for (int q = 0; q < 2; q++) {
              Z[r][q] += 2 * R[r][q];
              ZL[r][q] += 2 * RL[r][q];
            }
        } else {
          N xs[2];
          int ls[2];
#pragma unroll
          for (int r = 0; r < 2; r++) {
            const N s0 = Z[r][0] + R[r][0], s1 = Z[r][1] + R[r][1];
            const int m0 = ZL[r][0] + RL[r][0], m1 = ZL[r][1] + RL[r][1];
            xs[r] = shup(s1) + 2 * s0 + s1;
            ls[r] = shup(m1) + 2 * m0 + m1;
#pragma unroll
            for (int q = 0; q < 2; q++) {
              Z[r][q] = R[r][q];
              ZL[r][q] = RL[r][q];
            }
          }
          xa = xs[0];
          la = ls[0];
          xb = xs[1];
          lb = ls[1];
          xh[threadIdx.x] = xb;
          xl[threadIdx.x] = lb;
        }
      }
    }
    // ---- plane t + 1 has landed: its exponents
    fz::cp_async_wait<1>();
    if constexpr (FX) publish_exponent(t + 1, slot_at(1), K == 0);
    fslot = slot_at(1);
    __syncthreads();
    return true;
  };

#pragma unroll 1
  for (int t = tstart; t <= tend; t += 2) {
    if (!step(std::integral_constant<int, 0>{}, t) || !step(std::integral_constant<int, 1>{}, t + 1)) {
      good = false;
      break;
    }
  }
  fz::cp_async_wait<0>();
  __syncthreads();
  return good;
}

constexpr size_t kSmem = (size_t)(kPSlots + kFSlots + kUSlots) * kPlaneB + kThreads * 12 + 2 * kWarps * 4;

template <bool JAC, int KIND, bool ZERO, bool CORR, int OUT>
__global__ void __launch_bounds__(kThreads, 1) k_fx3d(const __grid_constant__ Args a) {
  extern __shared__ __align__(16) unsigned char smem[];
  double acc;
  const bool good = column<Fix, JAC, KIND, ZERO, CORR, OUT>(a, smem, acc);
  if (!good) column<F64, JAC, kGen, ZERO, CORR, OUT>(a, smem, acc);
  if constexpr (OUT == kNorm) {
    double *part = (double *)smem;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int i = 0; i < kWarps; i++) t += part[i];
      a.partials[(long long)blockIdx.y * gridDim.x + blockIdx.x] = good ? t * (a.km * a.km) : t;
    }
  }
}

// ------------------------------------------------------------------------
// Host side (fx2d.cuh: set_operator, launch, dispatch).

inline bool set_operator(Args &a, const double (&k)[3], double omega, bool corr, int stages) {
  a.k = fmax(k[0], fmax(k[1], k[2]));
  a.dgamma = 1.0 - omega;
  if (!(a.k > 1e-200 && a.k < 1e200)) return false;
  for (int d = 0; d < 3; d++) {
    a.dp[d] = k[d] / a.k;
    if (!(a.dp[d] > 1e-3)) return false;
    a.has_p[d] = a.dp[d] != 1.0;
    a.p[d] = fraction(a.has_p[d] ? k[d] : 0.0, a.k);
  }
  a.has_gamma = a.dgamma != 0.0;
  a.gamma = fraction(fabs(a.dgamma), 1.0);
  int ke;
  const double km = frexp(a.k, &ke);
  a.km = km;
  a.ke = ke;
  a.fexp = 0;
  a.fscale = 1.0;
  if (km == 0.5 && ke - 1 >= -40 && ke - 1 <= 40) {
    a.fexp = a.fbound = 1 - ke;
  } else {
    a.fscale = 1.0 / a.k;
    a.fbound = 2 - ke;
  }
  a.fpow = ldexp(1.0, a.fexp);
  const double sum = 2.0 * (a.dp[0] + a.dp[1] + a.dp[2]), diag = 2.0 * (k[0] + k[1] + k[2]);
  a.dw = omega * a.k / diag;
  if (!(a.dw < 1.0)) return false;
  a.w = fraction(omega * a.k, diag);
  double m = corr ? 2.0 : 1.0;
  for (int st = 0; st < stages; st++) m = fmax(m, fabs(a.dgamma) * m + a.dw * (1.0 + sum * m));
  const double bound = 1.0 + 2.0 * sum * m;
  int be;
  frexp(bound, &be);
  a.P = 62 - be < 57 ? 62 - be : 57;
  return a.P >= 54;
}

template <bool JAC, int KIND, bool ZERO, bool CORR, int OUT>
cudaError_t launch(Args a, int *nparts, cudaStream_t s) {
  auto kernel = k_fx3d<JAC, KIND, ZERO, CORR, OUT>;
  constexpr int S = JAC ? 1 : 2, kNeed = S + (OUT != kNone) + (OUT == kRestrict) + (CORR);
  constexpr int kHalo = (kNeed + 1) / 2 * 2;
  static PerDevice counts;  // SMs (or minus an error)
  const long long sms = per_device(counts, [&]() -> long long {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return -(long long)e;
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
  });
  if (sms < 0) return (cudaError_t)-sms;
  const int ox = kCols - 2 * kHalo, oy = kRows - 2 * kHalo;
  a.ntx = (a.n + ox - 1) / ox;
  a.nty = (a.n + oy - 1) / oy;
  // planes per chunk, even: the fewest plane steps of the longest-running SM
  // (waves of one block per SM, each walking its chunk and the planes around it)
  const long long cols = (long long)a.ntx * a.nty;
  long long best = -1;
  for (int nz = 1; nz <= 64; nz++) {
    int zc = (a.n + nz - 1) / nz;
    zc += zc & 1;
    const int chunks = (a.n + zc - 1) / zc;
    if (nz > 1 && (zc < 4 || cols * chunks > kMaxPartials)) break;
    const long long cost = (cols * chunks + sms - 1) / sms * (zc + 4 + kNeed);
    if (best < 0 || cost < best) {
      best = cost;
      a.zc = zc;
    }
  }
  const int chunks = (a.n + a.zc - 1) / a.zc;
  if (OUT == kNorm && cols * chunks > kMaxPartials) return cudaErrorInvalidValue;
  if (nparts) *nparts = (int)(cols * chunks);
  kernel<<<dim3((unsigned)cols, (unsigned)chunks), kThreads, kSmem, s>>>(a);
  return cudaGetLastError();
}

template <bool JAC, int KIND>
cudaError_t dispatch(const Args &a, bool zero, bool corr, int out, int *nparts, cudaStream_t s) {
#define FX3_CASE(Z, C, O) \
  if (zero == Z && corr == C && out == O) return launch<JAC, KIND, Z, C, O>(a, nparts, s)
  FX3_CASE(true, false, kNone);
  FX3_CASE(true, false, kRestrict);
  FX3_CASE(false, false, kNone);
  FX3_CASE(false, false, kRestrict);
  FX3_CASE(false, false, kNorm);
  FX3_CASE(false, true, kNone);
  FX3_CASE(false, true, kNorm);
#undef FX3_CASE
  return cudaErrorInvalidValue;
}

#define FX3_RUN(name) cudaError_t name(const Args &a, bool zero, bool corr, int out, int *nparts, cudaStream_t s)
FX3_RUN(rbgs_iso);
FX3_RUN(rbgs_gen);
FX3_RUN(jacobi_iso);
FX3_RUN(jacobi_gen);

}  // namespace fx3
}  // namespace mg
