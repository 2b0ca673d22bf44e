// Fused 2D passes of the FP64 levels on the integer pipes.
//
// This GPU issues FP64 at 1/64 of its FP32 rate: the FP64 form of one V(2,2)
// pass over a 4097^2 level needs about 40 FP64 instructions per node (2 ms),
// its memory traffic 60 us. So the sweeps, the residual and the transfers
// below run in 64-bit fixed point, with more bits than FP64 keeps:
//
//   A warp streams down a strip of the level (the decomposition of
//   fused2d.cuh with 64 columns, 2 per lane: rows in groups of 4 through a
//   cp.async ring, a register window of the last rows). It holds every value as an
//   integer multiple of 2^(E - 1022 - P), where E is the largest biased
//   exponent of u, f' = f / k (k the largest axis coefficient) and the coarse
//   correction among the rows read so far, so that every loaded |X| <= 2^P.
//   When a row with a larger exponent arrives the window is shifted right
//   (warp-uniform, rare). P (54 .. 57) is chosen on the host from a bound on
//   the growth of the values over the sweeps and on the residual
//   (set_operator), so no sum below can overflow, whatever the data. u loses
//   nothing within a factor 2^(P - 53) of the largest value and is cut at 2^-P
//   of it otherwise, half to a sixteenth of an FP64 unit in that value's last
//   place. f' carries 22 more bits (FL), used by the
//   residual: h^2 f is far smaller than u, and its relative precision decides
//   that of the solution.
//   Sweep: u' = W (f' + px (uw + ue) + py (us + un)) + gamma u, max(px, py)
//   = 1, W = omega / diag * k; an isotropic stencil with omega = 1 needs no
//   multiplication (W = 1/4). Other constants are 62-bit fractions.
//   Residual: r' = f' - [px (2u - uw - ue) + py (2u - us - un) + s u], exact
//   up to the multiplications; it is rounded once, after the restriction.
//
// A strip that meets Inf or NaN, or whose exponents leave 128 .. 1900, is
// done again in FP64 arithmetic by the same code (Arith = F64).
//
// Bound: integer issue (the ALU at 59 to 63 % while a warp runs, the FP64 pipe, on
// which the conversions issue, at 35 to 54 % and 70 to 74 % in the passes with a
// norm; 64 columns of which 52 are written and the rows before a chunk are 1.3
// times the minimal work), then HBM (430 MB at 6.7 TB/s: 64 us). 4097^2, V(2,2),
// one cycle's level in us, FP64 kernels -> these: red-black omega = 1, fused FP64
// passes and norm 1062 -> 193 (pre), 654 + 378 -> 257 (post with the norm; 234 when
// it was that of the unrounded values); Jacobi, one kernel per operator, 1453 ->
// 231, 1294 + 398 -> 307 (283).
//
// The same pass serves node-based grids (values on boundary nodes stay, full
// weighting, bilinear interpolation) and cell-centred ones (a missing
// neighbour counts as zero and the diagonal has the face's weight: 0 for
// zero flux, 2 for a fixed value; mean restriction, constant interpolation),
// red-black Gauss-Seidel and omega-Jacobi.
#pragma once

#include <math.h>

#include "fused2d.cuh"
#include "mg_internal.h"
#include "perdevice.h"

namespace mg {
namespace fx2 {

using fz::cp_async16;
using fz::cp_async_commit;
using fz::cp_async_wait;
using fz::kGroup;
using fz::kRing;

constexpr int kVec = 2;                  // columns per lane
constexpr int kCols = 32 * kVec;         // columns per strip (loaded)
constexpr int kHalo = 6;                 // halo columns on each side: four stages, residual, restriction
constexpr int kOut = kCols - 2 * kHalo;  // columns written per strip
constexpr int kWarps = 2;                // warps per block
constexpr int kBlocks = 8;               // resident blocks asked of the register allocator
constexpr int kLoBits = 22;   // extra bits of f'
constexpr int kResBits = 26;  // bits of a residual's low part (its high part is r' / 16)
constexpr int kMinE = 128, kMaxE = 1900;

// A constant as a fixed-point multiplier: value 2^62 = hi 2^32 + lo, lo signed.
struct Mul {
  int hi, lo;
};

struct Args {
  const double *uin, *f, *ec;
  double *uout, *fc, *partials;  // kNorm: one partial sum per warp
  int n, pitch, nc, pitchc;
  int R, nstrips, nchunks;
  int max_parts;       // room for the partial sums of kNorm
  int P;               // bits of the largest loaded value
  int fexp, fbound;    // f' = (f fscale) 2^fexp, one of the two trivial; the exponent of f' is at most f's + fbound
  double fscale, fpow; // fpow = 2^fexp
  int has_px, has_py, has_gamma, has_s;
  Mul px, py, gamma, s;  // 62-bit fractions (gamma: its magnitude)
  Mul w[4];              // the same by boundary class (row is edge) * 2 + (column is edge)
  int edge;              // cells: weight 2u loses or gains at an edge: 1 (zero flux) or 3 (fixed value) in place of 2
  double k;              // residual = r' k
  double km;             // k = km 2^ke, km in [1/2, 1)
  int ke;
  double dpx, dpy, dgamma, ds, dw[4];
};

// What one pass does with the strip.
enum { kNone = 0, kRestrict = 1, kNorm = 2 };

// X m / 2^62, rounded to nearest, for a fraction 0 <= m < 2^62 and |X| < 2^62
// (the product of the low words is dropped: 2^-30 units).
__device__ __forceinline__ long long mul62(long long x, Mul m) {
  const int xh = (int)(x >> 32);
  const unsigned xl = (unsigned)x;
  const long long mid =
      (long long)((unsigned long long)xl * (unsigned)m.hi + (1ull << 29)) + (long long)xh * m.lo;
  return (((long long)xh * m.hi) << 2) + (mid >> 30);
}

// X m / 2^62 for a residual: returns the product's integer part and takes
// its next BITS bits off lo (no bias: a one-sided error of one unit in
// every residual would grow by n^2 / 16 in the solution).
template <int BITS>
__device__ __forceinline__ long long mul62(long long x, Mul m, int &lo) {
  const int xh = (int)(x >> 32);
  const unsigned xl = (unsigned)x;
  const long long mid = (long long)((unsigned long long)xl * (unsigned)m.hi) + (long long)xh * m.lo +
                        (((long long)xl * m.lo) >> 32);
  lo -= (int)(((unsigned)mid & 0x3fffffffu) >> (30 - BITS));
  return (((long long)xh * m.hi) << 2) + (mid >> 30);
}

// Shifts whose count may reach 64 and more (PTX clamps it).
__device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}

// Significand of x (53 bits, for a normal x) << a.
__device__ __forceinline__ unsigned long long significand(double x, int a) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  return (((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << a;
}
__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// trunc(x 2^(P + 1022 - E)); values with a biased exponent above E do not occur.
__device__ __forceinline__ long long to_fix(double x, int E, int P) {
  const long long v = (long long)shr64(significand(x, P - 53), (unsigned)(E - expo(x)));
  const long long sg = (long long)(__double2hiint(x) >> 31);
  return (v ^ sg) - sg;
}
// The same with BITS further bits in lo (same sign as x).
template <int BITS>
__device__ __forceinline__ long long to_fix2(double x, int E, int P, int &lo) {
  const unsigned long long y = significand(x, P - 53);
  const int t = E - expo(x), t2 = t - BITS;
  const unsigned q = t2 >= 0 ? (unsigned)shr64(y, (unsigned)t2) : (unsigned)y << -t2;
  const int sg = __double2hiint(x) >> 31;
  const long long v = (long long)shr64(y, (unsigned)t);
  lo = ((int)(q & ((1u << BITS) - 1)) ^ sg) - sg;
  return (v ^ (long long)sg) - (long long)sg;
}
// x 2^(E - 1022 - P), rounded to nearest. The conversion instruction issues
// on the FP64 pipe, which this pass leaves idle otherwise.
__device__ __forceinline__ double to_dbl(long long x, int E, int P) {
  const double d = __ll2double_rn(x);
  const int hi = __double2hiint(d) + ((E - 1022 - P) << 20);
  return __hiloint2double(x == 0 ? 0 : hi, __double2loint(d));
}

// x as to_dbl stores it: rounded to 53 bits. A pass that forms the norm rounds
// each node's last update with it, so that the norm is that of the stored
// solution: the bits beyond FP64 would hide its rounding (2049^2, smooth data,
// at the rounding floor: 0.09 of the residual of what was returned). Both
// conversions issue on the FP64 pipe.
__device__ __forceinline__ long long stored(long long x) { return __double2ll_rn(__ll2double_rn(x)); }

__device__ __forceinline__ long long shup(long long v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ long long shdn(long long v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ int shup(int v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double shup(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double shdn(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// Shifts (hi, lo / 2^bits) right by d <= 30.
__device__ __forceinline__ void shift_pair(long long &hi, int &lo, int bits, int d) {
  const long long part = ((hi & ((1LL << d) - 1)) << bits) + lo;
  hi >>= d;
  lo = (int)(part >> d);
}

// Arithmetic of the pass: fixed point (N = int64) or FP64.
struct Fix {
  typedef long long N;
  static constexpr bool fixed = true;
};
struct F64 {
  typedef double N;
  static constexpr bool fixed = false;
};

// What the stencil's constants look like: kQuarter: px = py = 1, W = 1/4,
// gamma = 0 (isotropic node grids with omega = 1); kIso: px = py = 1; kGen:
// any. One instance each, since the code of a pass has to stay in the
// instruction cache.
enum { kQuarter = 0, kIso = 1, kGen = 2 };

template <class A, bool CELL, int KIND>
__device__ __forceinline__ typename A::N relax(const Args &a, typename A::N u, typename A::N f, typename A::N sx,
                                               typename A::N sy, int cls) {
  if constexpr (A::fixed) {
    if (KIND == kQuarter) return (f + sx + sy + 2) >> 2;
    if (KIND == kGen && a.has_px) sx = mul62(sx, a.px);
    if (KIND == kGen && a.has_py) sy = mul62(sy, a.py);
    const Mul w = !CELL || cls == 0 ? a.w[0] : cls == 1 ? a.w[1] : cls == 2 ? a.w[2] : a.w[3];
    // node grids: gamma = 1 - 4 W, so that one multiplication does
    if (KIND == kIso && !CELL) return u + mul62(f + sx + sy - 4 * u, w);
    long long v = mul62(f + sx + sy, w);
    if (a.has_gamma) {
      const long long g = mul62(u, a.gamma);
      v = a.dgamma < 0.0 ? v - g : v + g;
    }
    return v;
  } else {
    return a.dw[cls] * (f + a.dpx * sx + a.dpy * sy) + a.dgamma * u;
  }
}

// One strip. JAC: omega-Jacobi instead of red-black sweeps. ZERO: u = 0 on
// entry. CORR: coarse correction first. OUT: what follows the sweeps. Returns
// false when the fixed-point arithmetic cannot hold the data.
//
// The window is held by age: index j is row t - j, and each row moves
// everything up by one. The loop is unrolled by two rows only (the moves that
// remain cost 5 %): with a ring unrolled by its 8 rows the code of one pass
// (70 KB and more) missed the instruction cache and ran at half the speed or
// less (Jacobi pass of 4097^2: 600 us, 42 % of the fetches hit).
template <class A, bool CELL, bool JAC, int KIND, int NU, bool ZERO, bool CORR, int OUT, bool CHECK>
__device__ __forceinline__ bool strip(const Args &a, unsigned char *ring, int lane, int s, int ch, double &acc) {
  typedef typename A::N N;
  constexpr bool FX = A::fixed;
  constexpr int S = JAC ? NU : 2 * NU;  // stages: stage h runs on row t - h
  constexpr int LB = kVec * 8;
  constexpr int WU = S + 3, WF = S + 2, WR = OUT == kRestrict ? 3 : 1, WO = JAC ? NU + 1 : 1;
  const int n = a.n, P = a.P;
  const int lo = CELL ? 0 : 1, hi = CELL ? n - 1 : n - 2;  // rows and columns that are relaxed
  const int c0 = s * kOut - kHalo + kVec * lane;
  const bool col_ok = c0 >= 0 && c0 < a.pitch;
  const int J0 = c0 >> 1;
  const bool ccol_ok = c0 >= 0 && J0 < a.nc;
  const bool out_lane = lane >= kHalo / kVec && lane < 32 - kHalo / kVec && col_ok;
  const int r0 = ch * a.R, r1 = min(r0 + a.R, n);
  const int tstart = max(r0 - kHalo, 0);
  const int tend = OUT == kNone ? r1 - 1 + S : r1 + S;
  unsigned char *su = ring + lane * LB;
  unsigned char *sf = su + (ZERO ? 0 : kRing * 32 * LB);
  unsigned char *se = ring + (ZERO ? 1 : 2) * kRing * 32 * LB + lane * 8;
  auto in = [&](int c) { return !CHECK || (c >= lo && c <= hi); };

  N U[WU][kVec], F[WF][kVec], Rr[WR][kVec], Old[WO][kVec], Ec = 0;  // Ec: coarse row t / 2
  int FL[WF][kVec], RL[WR][kVec];
#pragma unroll
  for (int q = 0; q < kVec; q++) {
#pragma unroll
    for (int i = 0; i < WU; i++) U[i][q] = 0;
#pragma unroll
    for (int i = 0; i < WF; i++) { F[i][q] = 0; FL[i][q] = 0; }
#pragma unroll
    for (int i = 0; i < WR; i++) { Rr[i][q] = 0; RL[i][q] = 0; }
#pragma unroll
    for (int i = 0; i < WO; i++) Old[i][q] = 0;
  }
  int E = kMinE;  // scale exponent (fixed point)
  bool good = true;
  acc = 0.0;

  // Window values from scale E to E + d (all of them are zero at kMinE).
  auto rescale = [&](int d) {
    if constexpr (FX) {
      for (int left = E == kMinE ? 0 : d; left > 0; left -= 30) {
        const int e = min(left, 30);
#pragma unroll
        for (int q = 0; q < kVec; q++) {
#pragma unroll
          for (int i = 0; i < WU; i++) U[i][q] >>= e;
#pragma unroll
          for (int i = 0; i < WF; i++) shift_pair(F[i][q], FL[i][q], kLoBits, e);
          if (OUT == kRestrict) {
#pragma unroll
            for (int i = 0; i < WR; i++) shift_pair(Rr[i][q], RL[i][q], kResBits, e);
          }
          if (JAC) {
#pragma unroll
            for (int i = 0; i < WO; i++) Old[i][q] >>= e;
          }
        }
        Ec >>= e;
      }
    }
    E += d;
  };
  // Takes a largest biased exponent e (over the warp) into the scale.
  auto take = [&](int e) {
    e = __reduce_max_sync(0xffffffffu, e);
    if (e > E) {
      if (e > kMaxE) good = false;
      else rescale(e - E);
    } else if (E == kMinE && e > 0) {
      good = false;  // magnitudes too small for the exponent range
    }
  };

  auto issue_group = [&](int tg) {
#pragma unroll
    for (int K = 0; K < kGroup; K++) {
      const int row = tg + K, slot = row & (kRing - 1);
      const bool ok = col_ok && row < n && row <= tend;
      const long long off = (long long)row * a.pitch + c0;
      if (!ZERO) cp_async16(su + slot * 32 * LB, ok ? a.uin + off : a.uin, ok);
      cp_async16(sf + slot * 32 * LB, ok ? a.f + off : a.f, ok);
      if (CORR) {
        // nodes: coarse row (row + 1) / 2 comes with an odd fine row, coarse
        // row 0 with fine row 0; cells: row / 2 with an even one
        const int I = CELL ? ((K & 1) ? -1 : row >> 1) : ((K & 1) ? (row + 1) >> 1 : (row == 0 ? 0 : -1));
        const bool cok = ccol_ok && row <= tend && I >= 0 && I < a.nc;
        if (CELL ? (K & 1) == 0 : (K & 1) != 0 || K == 0)
          fz::cp_async8(se + slot * 32 * 8, cok ? a.ec + (long long)I * a.pitchc + J0 : a.ec, cok);
      }
    }
    cp_async_commit();
  };

  if (CORR && !CELL && tstart > 0) {
    // coarse row tstart / 2 precedes the window
    const int I = tstart >> 1;
    const double e0 = ccol_ok && I < a.nc ? a.ec[(long long)I * a.pitchc + J0] : 0.0;
    if constexpr (FX) {
      take(expo(e0));
      if (good) Ec = to_fix(e0, E, P);
    } else {
      Ec = e0;
    }
  }

  // Row t, of parity K.
  auto row = [&](auto kc, const int t) {
    constexpr int K = decltype(kc)::value;
    const int slot = t & (kRing - 1);
    const bool rowin = !CHECK || (t >= lo && t <= hi);
#pragma unroll
    for (int q = 0; q < kVec; q++) {
#pragma unroll
      for (int i = WU - 1; i > 0; i--) U[i][q] = U[i - 1][q];
#pragma unroll
      for (int i = WF - 1; i > 0; i--) {
        F[i][q] = F[i - 1][q];
        FL[i][q] = FL[i - 1][q];
      }
      if (OUT == kRestrict) {
#pragma unroll
        for (int i = WR - 1; i > 0; i--) {
          Rr[i][q] = Rr[i - 1][q];
          RL[i][q] = RL[i - 1][q];
        }
      }
    }
    // ---- values and conversion; interpolation and correction
    {
      const double2 uv = ZERO ? make_double2(0.0, 0.0) : *(const double2 *)(su + slot * 32 * LB);
      const double2 fv = *(const double2 *)(sf + slot * 32 * LB);
      const double ud[kVec] = {uv.x, uv.y};
      double fd[kVec] = {fv.x, fv.y};
      if (CHECK) {
        // the right-hand side of boundary nodes and of padding is not part of the problem
#pragma unroll
        for (int q = 0; q < kVec; q++)
          if (!(rowin && in(c0 + q))) fd[q] = 0.0;
      }
      if (KIND != kQuarter && a.fscale != 1.0) {
#pragma unroll
        for (int q = 0; q < kVec; q++) fd[q] *= a.fscale;
      }
#pragma unroll
      for (int q = 0; q < kVec; q++) {
        if constexpr (FX) {
          U[0][q] = ZERO ? 0 : to_fix(ud[q], E, P);
          F[0][q] = to_fix2<kLoBits>(fd[q], E - a.fexp, P, FL[0][q]);
        } else {
          U[0][q] = ud[q];
          F[0][q] = fd[q] * a.fpow;
        }
      }
      if (CORR) {
        const bool firstE = !CELL && CHECK && t == 0;
        N e0 = Ec;
        if ((CELL ? K == 0 : K == 1) || firstE) {
          const double ed = *(const double *)(se + slot * 32 * 8);
          if constexpr (FX) Ec = to_fix(ed, E, P);
          else Ec = ed;
          if (CELL || firstE) e0 = Ec;
        }
        N v[kVec];
        if (CELL) {
          v[0] = v[1] = e0;
        } else if constexpr (FX) {
          if (K == 1) e0 = (e0 + Ec + 1) >> 1;
          v[0] = e0;
          v[1] = (e0 + shdn(e0) + 1) >> 1;
        } else {
          if (K == 1) e0 = 0.5 * (e0 + Ec);
          v[0] = e0;
          v[1] = 0.5 * (e0 + shdn(e0));
        }
#pragma unroll
        for (int q = 0; q < kVec; q++)
          if (rowin && in(c0 + q)) U[0][q] += v[q];
      }
    }
    // ---- stage h on row t - h
    auto cls_of = [&](int r, int c) {
      return CELL && CHECK ? (r == 0 || r == n - 1 ? 2 : 0) + (c == 0 || c == n - 1 ? 1 : 0) : 0;
    };
#pragma unroll
    for (int h = 1; h <= S; h++) {
      const int r = t - h;
      const bool rin = !CHECK || (r >= lo && r <= hi);
      if (JAC) {
        const N left = shup(U[h][1]), right = shdn(U[h][0]);
        N nv[kVec];
#pragma unroll
        for (int q = 0; q < kVec; q++)
          nv[q] = relax<A, CELL, KIND>(a, U[h][q], F[h][q], q == 0 ? left + U[h][1] : U[h][0] + right,
                                       Old[JAC ? h : 0][q] + U[h - 1][q], cls_of(r, c0 + q));
#pragma unroll
        for (int q = 0; q < kVec; q++) {
          if constexpr (FX && OUT == kNorm)
            if (h == S) nv[q] = stored(nv[q]);
          Old[JAC ? h : 0][q] = U[h][q];  // the row's values before this sweep, for the row below
          if (rin && in(c0 + q)) U[h][q] = nv[q];
        }
      } else {
        // colour (h - 1) & 1; c0 is even and t has parity K: column q with the parity of
        constexpr int q = (K + 1) & 1;
        const N sx = q == 0 ? shup(U[h][1]) + U[h][1] : U[h][0] + shdn(U[h][0]);
        N nv = relax<A, CELL, KIND>(a, U[h][q], F[h][q], sx, U[h + 1][q] + U[h - 1][q], cls_of(r, c0 + q));
        if constexpr (FX && OUT == kNorm)
          if (h > S - 2) nv = stored(nv);  // the last red and the last black half-sweep
        if (rin && in(c0 + q)) U[h][q] = nv;
      }
    }
    // ---- the smoothed row t - S
    {
      const int r = t - S;
      if (r >= r0 && r < r1 && out_lane) {
        double v[kVec];
#pragma unroll
        for (int q = 0; q < kVec; q++) {
          if constexpr (FX) v[q] = to_dbl(U[S][q], E, P);
          else v[q] = U[S][q];
        }
        double *dst = a.uout + (long long)r * a.pitch + c0;
        if (!CHECK) {
          *(double2 *)dst = make_double2(v[0], v[1]);
        } else {
          // boundary nodes keep their values
#pragma unroll
          for (int q = 0; q < kVec; q++)
            if (c0 + q < n)
              dst[q] = r >= lo && r <= hi && in(c0 + q) ? v[q]
                       : ZERO                           ? 0.0
                                                        : a.uin[(long long)r * a.pitch + c0 + q];
        }
      }
    }
    // ---- residual of row t - S - 1
    if (OUT != kNone) {
      const int r = t - S - 1;
      constexpr int sc = S + 1;
      const bool rin = !CHECK || (r >= lo && r <= hi);
      const N left = shup(U[sc][1]), right = shdn(U[sc][0]);
      N rr[kVec];
      int rl[kVec] = {0, 0};
#pragma unroll
      for (int q = 0; q < kVec; q++) {
        const int c = c0 + q;
        const N u = U[sc][q], uw = q == 0 ? left : U[sc][0], ue = q == 0 ? U[sc][1] : right;
        const N us = U[sc + 1][q], un = U[sc - 1][q];
        int kx = 2, ky = 2;
        if (CELL && CHECK) {
          if (c == 0 || c == n - 1) kx = a.edge;
          if (r == 0 || r == n - 1) ky = a.edge;
        }
        const bool ok = rin && in(c);
        if constexpr (FX) {
          int lo2 = FL[sc][q];
          if (KIND != kGen) {
            rr[q] = F[sc][q] + (uw + ue) + (us + un) - (kx + ky) * u;
          } else {
            long long tx = kx * u - (uw + ue), ty = ky * u - (us + un);
            if (a.has_px) tx = mul62<kLoBits>(tx, a.px, lo2);
            if (a.has_py) ty = mul62<kLoBits>(ty, a.py, lo2);
            rr[q] = F[sc][q] - (tx + ty);
          }
          if (CELL && a.has_s) rr[q] -= mul62<kLoBits>(u, a.s, lo2);
          if (ok) rl[q] = lo2;
        } else {
          const N tx = (u - uw) + (u - ue) + (kx - 2) * u, ty = (u - us) + (u - un) + (ky - 2) * u;
          rr[q] = F[sc][q] - (a.dpx * tx + a.dpy * ty) - a.ds * u;
        }
        if (!ok) rr[q] = 0;
        if constexpr (FX && OUT == kRestrict) {
          RL[0][q] = (((int)rr[q] & 15) << kLoBits) + rl[q];
          Rr[0][q] = rr[q] >> 4;
        }
        if constexpr (!FX && OUT == kRestrict) Rr[0][q] = rr[q];
      }
      if constexpr (OUT == kNorm) {
        if (r >= r0 && r < r1 && out_lane) {
          if constexpr (FX) {
            // squares of the lane's residuals, normalised to the larger
            const unsigned long long m = (unsigned long long)((rr[0] ^ (rr[0] >> 63)) | (rr[1] ^ (rr[1] >> 63)));
            const int sh = min(max(__clzll((long long)m) - 2, 0), 40);
            unsigned long long sq = 0;
#pragma unroll
            for (int q = 0; q < kVec; q++) {
              const long long l = sh >= kLoBits ? (long long)rl[q] << (sh - kLoBits)
                                                : (long long)(rl[q] >> (kLoBits - sh));
              const long long v = (rr[q] << sh) + l;
              sq += (unsigned long long)__mul64hi(v, v);
            }
            // sq 2^(64 - 2 sh) units squared, a unit is 2^(E - 1022 - P); with k's power
            // of two, since the square of r' or of k alone may leave FP64's range
            const double d = __ull2double_rn(sq);
            const int ex = 64 - 2 * sh + 2 * (E - 1022 - P + a.ke) + (__double2hiint(d) >> 20);
            if (sq) acc += ex <= 0 ? 0.0
                           : ex >= 2047 ? __hiloint2double(0x7ff00000, 0)
                                        : __hiloint2double((ex << 20) | (__double2hiint(d) & 0xfffff),
                                                           __double2loint(d));
          } else {
            const double v0 = rr[0] * a.k, v1 = rr[1] * a.k;
            acc += v0 * v0 + v1 * v1;
          }
        }
      }
      // ---- restriction once the row below the coarse row is there (r odd)
      if constexpr (OUT == kRestrict && ((K + S + 1) & 1) != 0) {
        const int I = (r - 1) >> 1;
        constexpr int b = WR > 1 ? 1 : 0, top = WR > 2 ? 2 : 0;
        N v;
        int l = 0;
        if (CELL) {
          v = (Rr[b][0] + Rr[b][1]) + (Rr[0][0] + Rr[0][1]);
          if constexpr (FX) l = (RL[b][0] + RL[b][1]) + (RL[0][0] + RL[0][1]);
        } else {
          // vertical weights first, so that one shuffle serves the three rows
          const N w0 = Rr[top][0] + 2 * Rr[b][0] + Rr[0][0], w1 = Rr[top][1] + 2 * Rr[b][1] + Rr[0][1];
          v = shup(w1) + 2 * w0 + w1;
          if constexpr (FX) {
            const int l0 = RL[top][0] + 2 * RL[b][0] + RL[0][0], l1 = RL[top][1] + 2 * RL[b][1] + RL[0][1];
            l = shup(l1) + 2 * l0 + l1;
          }
        }
        const int clo = CELL ? 0 : 1, chi = CELL ? a.nc - 1 : a.nc - 2;
        if (out_lane && 2 * I >= r0 && 2 * I < r1 && I >= clo && I <= chi && J0 >= clo && J0 <= chi) {
          double *dst = a.fc + (long long)I * a.pitchc + J0;
          if constexpr (FX) {
            // v + l / 2^26, with as many bits of l as there is room for
            const int sh = min(max(__clzll(v ^ (v >> 63)) - 2, 0), kResBits);
            *dst = to_dbl((v << sh) + (l >> (kResBits - sh)), E - sh + (CELL ? 2 : 0), P) * a.k;
          } else {
            *dst = v * ((CELL ? 0.25 : 0.0625) * a.k);
          }
        }
      }
    }
  };

  issue_group(tstart);
  for (int tg = tstart; tg <= tend && good; tg += kGroup) {
    issue_group(tg + kGroup);
    cp_async_wait<1>();  // group tg has landed; the next one may be in flight
    if constexpr (FX) {
      // the scale takes in the rows that have landed
      int mu = 0, mf = 0;
#pragma unroll
      for (int g = 0; g < kGroup; g++) {
        const int slot = (tg + g) & (kRing - 1);
        const bool rg = !CHECK || (tg + g >= lo && tg + g <= hi);
#pragma unroll
        for (int q = 0; q < kVec; q++) {
          if (!ZERO) mu = max(mu, *(const int *)(su + slot * 32 * LB + 8 * q + 4) & 0x7fffffff);
          if (rg && in(c0 + q)) mf = max(mf, *(const int *)(sf + slot * 32 * LB + 8 * q + 4) & 0x7fffffff);
        }
        if (CORR && (CELL ? (g & 1) == 0 : (g & 1) != 0 || (CHECK && tg == 0 && g == 0)))
          mu = max(mu, *(const int *)(se + slot * 32 * 8 + 4) & 0x7fffffff);
      }
      mf >>= 20;
      // an Inf or NaN stays one whatever the shift
      if (mf) mf = mf == 2047 ? 2047 + kMaxE : max(mf + a.fbound, 1);
      take(max(mu >> 20, mf));
      if (!good) break;
    }
#pragma unroll 1
    for (int t = tg; t < tg + kGroup; t += 2) {
      row(std::integral_constant<int, 0>{}, t);
      row(std::integral_constant<int, 1>{}, t + 1);
    }
  }
  cp_async_wait<0>();
  return good;
}

template <bool CELL, bool JAC, int KIND, int NU, bool ZERO, bool CORR, int OUT>
__global__ void __launch_bounds__(32 * kWarps, kBlocks) k_fx2d(const __grid_constant__ Args a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int S = JAC ? NU : 2 * NU;
  constexpr int WB = kRing * 32 * (kVec * 8 * (ZERO ? 1 : 2) + (CORR ? 8 : 0));
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const long long gw = (long long)blockIdx.x * kWarps + wib;
  if (gw >= (long long)a.nstrips * a.nchunks) return;
  const int s = (int)(gw % a.nstrips), ch = (int)(gw / a.nstrips);
  const int x0 = s * kOut - kHalo, r0 = ch * a.R, r1 = min(r0 + a.R, a.n);
  const int tstart = max(r0 - kHalo, 0), tend = r1 + S;
  const int tlast = tstart + ((tend - tstart) / kGroup + 1) * kGroup - 1;
  const bool interior = x0 >= 1 && x0 + kCols - 1 <= a.n - 2 && tstart - S - 2 >= 1 && tlast <= a.n - 2;
  unsigned char *ring = smem + (size_t)wib * WB;
  double acc;
  const bool good = interior ? strip<Fix, CELL, JAC, KIND, NU, ZERO, CORR, OUT, false>(a, ring, lane, s, ch, acc)
                             : strip<Fix, CELL, JAC, KIND, NU, ZERO, CORR, OUT, true>(a, ring, lane, s, ch, acc);
  if (!good) strip<F64, CELL, JAC, kGen, NU, ZERO, CORR, OUT, true>(a, ring, lane, s, ch, acc);
  if constexpr (OUT == kNorm) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) a.partials[gw] = good ? acc * (a.km * a.km) : acc;
  }
}

// ------------------------------------------------------------------------
// Host side.

// num / den < 1 as a multiplier, rounded to 2^-61: the quotient's FP64 rounding
// error is added back (a constant that is off by 2^-54 shows in the solution).
inline Mul fraction(double num, double den) {
  const double q = num / den, one = 4611686018427387904.0;  // 2^62
  const long long k = (long long)(q * one) + (long long)(fma(-q, den, num) / den * one);
  Mul m;
  m.lo = (int)(unsigned)(k & 0xffffffffLL);
  m.hi = (int)((k - m.lo) >> 32);
  return m;
}

// The pass's constants for axis coefficients kx, ky (c_d / h^2), reaction
// sigma and edge weight `edge` (2: node grids), and P. False: this operator
// stays on the FP64 kernels (coefficients of very different size, sigma h^2
// not small, or omega so large that the growth bound leaves too few bits).
inline bool set_operator(Args &a, double kx, double ky, double sigma, int edge, double omega, bool corr, int stages) {
  a.k = kx > ky ? kx : ky;
  a.dpx = kx / a.k;
  a.dpy = ky / a.k;
  a.ds = sigma / a.k;
  a.dgamma = 1.0 - omega;
  a.edge = edge;
  if (!(a.dpx > 1e-3 && a.dpy > 1e-3 && a.ds < 0.99 && a.k > 1e-200 && a.k < 1e200)) return false;
  a.has_px = a.dpx != 1.0;
  a.has_py = a.dpy != 1.0;
  a.has_s = a.ds != 0.0;
  a.has_gamma = a.dgamma != 0.0;
  int ke;
  const double km = frexp(a.k, &ke);  // k = km 2^ke
  a.km = km;
  a.ke = ke;
  a.fexp = 0;
  a.fscale = 1.0;
  if (km == 0.5 && ke - 1 >= -40 && ke - 1 <= 40) {
    a.fexp = a.fbound = 1 - ke;
  } else {
    a.fscale = 1.0 / a.k;
    a.fbound = 1 - ke + 1;  // 1 / k < 2^(1 - ke)
  }
  a.fpow = ldexp(1.0, a.fexp);
  a.px = fraction(a.has_px ? kx : 0.0, a.k);
  a.py = fraction(a.has_py ? ky : 0.0, a.k);
  a.s = fraction(sigma, a.k);
  a.gamma = fraction(fabs(a.dgamma), 1.0);
  // Growth: loaded values (with the correction added) are at most m = 1 or 2
  // units of 2^P; each stage gives at most |gamma| m + W (1 + weights m). The
  // residual is at most 1 + (4 px + 4 py + s) m, and every sum of a sweep is
  // below that; it has to stay below 2^62.
  double m = corr ? 2.0 : 1.0;
  for (int c = 0; c < 4; c++) {
    const double dx = (c & 1) ? edge : 2, dy = (c & 2) ? edge : 2;
    const double diag = sigma + kx * dx + ky * dy;
    a.dw[c] = omega * a.k / diag;
    if (!(a.dw[c] < 1.0)) return false;
    a.w[c] = fraction(omega * a.k, diag);
  }
  for (int st = 0; st < stages; st++) {
    double g = m;
    for (int c = 0; c < 4; c++) {
      const double nx = edge != 2 && (c & 1) ? 1 : 2, ny = edge != 2 && (c & 2) ? 1 : 2;
      g = fmax(g, fabs(a.dgamma) * m + a.dw[c] * (1.0 + (nx * a.dpx + ny * a.dpy) * m));
    }
    m = g;
  }
  const double bound = 1.0 + (4.0 * (a.dpx + a.dpy) + a.ds) * m;
  int be;
  frexp(bound, &be);  // bound < 2^be
  a.P = 62 - be < 57 ? 62 - be : 57;
  return a.P >= 54;
}

// Rows per chunk: one wave of resident warps, an even number (multiples of 8
// left 6 % of the resident warps without a chunk at 4097^2).
inline int chunk_rows(int n, int nstrips, long long warps) {
  long long chunks = warps / nstrips;
  if (chunks < 1) chunks = 1;
  const int R = ((int)((n + chunks - 1) / chunks) + 1) / 2 * 2;
  return R < 8 ? 8 : R;
}

template <bool CELL, bool JAC, int KIND, int NU, bool ZERO, bool CORR, int OUT>
cudaError_t launch(Args a, int rows, int *nparts, cudaStream_t s) {
  auto kernel = k_fx2d<CELL, JAC, KIND, NU, ZERO, CORR, OUT>;
  constexpr int smem = kWarps * kRing * 32 * (kVec * 8 * (ZERO ? 1 : 2) + (CORR ? 8 : 0));
  // warps of one wave (or minus an error)
  static PerDevice waves;
  const long long wave = per_device(waves, [&]() -> long long {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return -(long long)e;
    int dev = 0, sms = 0, blocks = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, 32 * kWarps, smem);
    return (long long)(sms > 0 ? sms : 1) * (blocks > 0 ? blocks : 1) * kWarps;
  });
  if (wave < 0) return (cudaError_t)-wave;
  a.nstrips = (a.n + kOut - 1) / kOut;
  a.R = rows > 0 ? (rows + 7) / 8 * 8 : chunk_rows(a.n, a.nstrips, wave);
  if (OUT == kNorm)  // one partial sum per warp
    while ((long long)a.nstrips * ((a.n + a.R - 1) / a.R) > a.max_parts) a.R += 8;
  a.nchunks = (a.n + a.R - 1) / a.R;
  const long long warps = (long long)a.nstrips * a.nchunks;
  if (nparts) *nparts = (int)warps;
  kernel<<<(unsigned)((warps + kWarps - 1) / kWarps), 32 * kWarps, smem, s>>>(a);
  return cudaGetLastError();
}

// nparts (may be NULL): the partial sums a kNorm pass leaves.
template <bool CELL, bool JAC, int KIND>
cudaError_t dispatch(const Args &a, int rows, int nu, bool zero, bool corr, int out, int *nparts,
                     cudaStream_t s) {
#define FX2_CASE(NU, Z, C, O) \
  if (nu == NU && zero == Z && corr == C && out == O) return launch<CELL, JAC, KIND, NU, Z, C, O>(a, rows, nparts, s)
  FX2_CASE(1, true, false, kRestrict);
  FX2_CASE(2, true, false, kRestrict);
  FX2_CASE(1, false, false, kRestrict);
  FX2_CASE(2, false, false, kRestrict);
  FX2_CASE(1, false, true, kNone);
  FX2_CASE(2, false, true, kNone);
  FX2_CASE(1, false, true, kNorm);
  FX2_CASE(2, false, true, kNorm);
  FX2_CASE(1, false, false, kNone);
  FX2_CASE(2, false, false, kNone);
#undef FX2_CASE
  return cudaErrorInvalidValue;
}

// The instances (fx2d_*.cu).
#define FX2_RUN(name)                                                                                   \
  cudaError_t name(const Args &a, int rows, int nu, bool zero, bool corr, int out, int *nparts, cudaStream_t s)
FX2_RUN(node_rbgs_quarter);
FX2_RUN(node_rbgs_iso);
FX2_RUN(node_rbgs_gen);
FX2_RUN(node_jacobi_iso);
FX2_RUN(node_jacobi_gen);
FX2_RUN(cell_rbgs_iso);
FX2_RUN(cell_rbgs_gen);
FX2_RUN(cell_jacobi_iso);
FX2_RUN(cell_jacobi_gen);

// The instance for set_operator's constants.
inline cudaError_t run(const Args &a, bool cell, bool jacobi, int rows, int nu, bool zero, bool corr, int out,
                       int *nparts, cudaStream_t s) {
  const bool gen = a.has_px || a.has_py;
  auto f = cell ? (jacobi ? (gen ? cell_jacobi_gen : cell_jacobi_iso) : (gen ? cell_rbgs_gen : cell_rbgs_iso))
           : jacobi ? (gen ? node_jacobi_gen : node_jacobi_iso)
           : gen    ? node_rbgs_gen
                    : (a.has_gamma || a.fscale != 1.0 ? node_rbgs_iso : node_rbgs_quarter);
  return f(a, rows, nu, zero, corr, out, nparts, s);
}

}  // namespace fx2
}  // namespace mg
