// Residual of the FP64 outer problem with a variable 2D stencil (defect
// correction): r = f - h^-2 sum_f k_f (u_p - u_q), written as the inner
// defect, and its squares summed.
//
// In FP64 the pass is bound by 11 FP64 instructions per node (64 to 76 cycles
// of a scheduler each). Here a warp streams down a strip of 64 columns (60
// written, 2 per lane) and a chunk of rows with u as integer multiples of
// 2^(E - 1022 - P), E the largest biased exponent read so far (the scale of
// fx2d.cuh): the differences u_p - u_q are exact integers, a face's flux is one
// 64-bit high product with the significand of its coefficient, formed once
// for its two nodes (the left one comes by shuffle, the upper one from the row
// before), and a node's four fluxes are added after alignment to the largest
// exponent among its coefficients. Only the last step is FP64: the sum's
// conversion, r = f - h^-2 (...) and r^2.
//
// Precision: a flux is cut at a quarter of the unit 2^(E - 1022 - P) of u times
// the largest coefficient of the node, P = 56, an eighth of the FP64 spacing
// of the largest u; FP64 keeps 2^-53 of each flux. u itself is rounded to that
// FP64 spacing, which moves the residual eight times as much, so the solution
// reached is the same. Chunks with non-finite or out-of-range values, and
// coefficients that are negative or not finite, are done in FP64.
//
// Bound: the FP64 pipe (57 %) and the integer ALU (54 %) together. 12 problems of
// 513^2 and 1025^2 (7.9 M nodes): 95 us; 290 MB, 43 us of HBM. The FP64 kernel took
// 4.9 ms for 1021 problems of 33^2 to 1025^2, 174 us for 8.4 M nodes in proportion.
#pragma once

#include "fx2d.cuh"
#include "kernels.cuh"
#include "outer2d.cuh"

namespace mg {
namespace dv2 {

constexpr int kWarps = 4, kThreads = 32 * kWarps;
constexpr int kOut = 60;   // columns written per strip
// Rows per chunk of a batch's problems. A warp walks its chunk alone (0.7 us a
// row), so problems with few strips take short ones; the largest (1025^2) has a
// chunk for each of its 512 warps. Below kBatchMinN a problem's rows are too few
// to hide a chunk's latency, and beside smaller problems, which keep the FP64
// kernel, it costs a launch of its own (solves of a few 33^2 to 257^2 problems:
// 3.45 ms on the FP64 kernel, 3.53 ms with 257^2 here; 40 of them: 5.07 and 5.06;
// four of 513^2: 6.15 and 6.04 ms).
constexpr int kBatchMinN = 513;
__host__ __device__ constexpr int batch_rows(int n) { return n <= 513 ? 16 : 40; }
// A problem alone: short chunks, or too few warps; below 1025^2 the FP64 kernel's
// one node per thread is as fast (129^2: 738 us a solve, 750 us with this one).
constexpr int kAloneMinN = 1025;
constexpr int alone_rows(int n) { return n <= 1025 ? 8 : n <= 2049 ? 16 : 40; }
constexpr int kP = 56;

struct Prob {
  const double *u, *f, *kx, *ky;
  void *d;  // inner defect (may be NULL)
  double ih2;
  int n;
  long long sy, syi;  // row strides of the FP64 fields and of the defect
  int rows;           // per chunk
};

__device__ __forceinline__ int tasks(const Prob &a) { return ((a.n + kOut - 1) / kOut) * ((a.n - 2 + a.rows - 1) / a.rows); }

// Flux of a difference through a face with coefficient k >= 0: x k / 2^(e -
// 1023) * 4, e its biased exponent (of the product of the low words only the
// carry is dropped). A zero or subnormal k counts as 2^-1023: e = 0 shifts it
// out beside any other coefficient.
__device__ __forceinline__ long long flux(long long x, double k, int &e) {
  const unsigned hi = (unsigned)__double2hiint(k), klo = (unsigned)__double2loint(k);
  e = (int)(hi >> 20);
  // significand << 9 = mh 2^32 + ml, ml signed
  const int ml = (int)(klo << 9);
  const int mh = (int)__funnelshift_l(klo, (hi & 0xfffffu) | 0x100000u, 9) + (int)((unsigned)ml >> 31);
  const int xh = (int)(x >> 32);
  const unsigned xl = (unsigned)x;
  const long long mid = (long long)((unsigned long long)xl * (unsigned)mh) + (long long)xh * ml;
  return (((long long)xh * mh) << 5) + (mid >> 27);
}

__device__ __forceinline__ long long sar(long long v, int n) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));  // counts of 64 and more leave the sign
  return r;
}

template <typename Ti, bool RN> __device__ __forceinline__ void put(Ti *p, double r) {
  st(p, RN ? (float)r : oz::d2f_bits(r));
}

// Task t of the problem; returns the lane's sum of squares.
template <typename Ti, bool RN> __device__ __forceinline__ double task(const Prob &a, int t, int lane) {
  const int n = a.n, strips = (n + kOut - 1) / kOut;
  const int c0 = (t % strips) * kOut - 2 + 2 * lane;
  const int R = a.rows, r0 = 1 + (t / strips) * R, r1 = min(r0 + R, n - 1);  // rows r0 .. r1 - 1
  const bool out = lane >= 1 && lane < 31;
  const bool ok0 = out && c0 >= 1 && c0 <= n - 2, ok1 = out && c0 + 1 >= 1 && c0 + 1 <= n - 2;
  const bool ld_ok = c0 >= 0 && c0 < n;  // rows are padded to an even number of columns
  Ti *d = (Ti *)a.d;
  // -h^-2 2^(-1022 - P - 2 - 1023): high word, low word, exponent
  const int ihm = __double2hiint(-a.ih2), ihl = __double2loint(a.ih2);
  const int ihe = ((ihm >> 20) & 0x7ff) - 1022 - kP - 2 - 1023;
  const double2 zero = make_double2(0.0, 0.0);
  auto load = [&](const double *p, int row) {
    return ld_ok ? __ldg((const double2 *)(p + (long long)row * a.sy + c0)) : zero;
  };
  int E = fx2::kMinE;
  bool good = true;
  double acc = 0.0;
  // row above: u, x-fluxes, f; the y-fluxes into it
  long long X[2] = {0, 0}, Fx[2] = {0, 0}, Fy[2] = {0, 0};
  int ex[2] = {0, 0}, ey[2] = {0, 0};
  double2 fr = zero, kyr = zero;
  double2 un = load(a.u, r0 - 1), kxn = load(a.kx, r0 - 1), kyn = load(a.ky, r0 - 1), fn = zero;
  for (int row = r0 - 1; row <= r1; row++) {
    const double2 u = un, kx = kxn, ky = kyn, f = fn;
    if (row < r1) {
      un = load(a.u, row + 1);
      kxn = load(a.kx, row + 1);
      kyn = load(a.ky, row + 1);
      fn = load(a.f, row + 1);
    }
    // the scale; a coefficient that is negative, Inf or NaN ends the integer pass
    const int m = max(__double2hiint(u.x) & 0x7fffffff, __double2hiint(u.y) & 0x7fffffff) >> 20;
    // as unsigned numbers, negative coefficients exceed all others too
    const unsigned mk = max(max((unsigned)__double2hiint(kx.x), (unsigned)__double2hiint(kx.y)),
                            max((unsigned)__double2hiint(ky.x), (unsigned)__double2hiint(ky.y)));
    const int e = __reduce_max_sync(0xffffffffu, mk >= 0x7ff00000u ? fx2::kMaxE + 1 : m);
    if (e > E) {
      if (e > fx2::kMaxE) {
        good = false;
        break;
      }
      if (E != fx2::kMinE) {
        const int sh = min(e - E, 63);
#pragma unroll
        for (int q = 0; q < 2; q++) {
          X[q] >>= sh;
          Fx[q] >>= sh;
          Fy[q] >>= sh;
        }
      }
      E = e;
    } else if (E == fx2::kMinE && e > 0) {
      good = false;
      break;
    }
    const long long Y[2] = {fx2::to_fix(u.x, E, kP), fx2::to_fix(u.y, E, kP)};
    if (row >= r0) {
      // flux from the row above into this one
      int en[2];
      const long long Fn[2] = {flux(X[0] - Y[0], kyr.x, en[0]), flux(X[1] - Y[1], kyr.y, en[1])};
      if (row > r0) {
        // residual of the row above: its fluxes right, left, down and up
        const long long left = fx2::shup(Fx[1]);
        const int eleft = fx2::shup(ex[1]);
        const long long r = row - 1;
        double rv[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
          const long long fl = q == 0 ? left : Fx[0];
          const int el = q == 0 ? eleft : ex[0];
          const int em = max(max(ex[q], el), max(en[q], ey[q]));
          auto al = [&](long long v, int ev) { return sar(v, em - ev); };
          const long long S = (al(Fx[q], ex[q]) - al(fl, el)) + (al(Fn[q], en[q]) - al(Fy[q], ey[q]));
          // r = f - h^-2 S 2^(E - 1022 - P - 2 + em - 1023), the power inside the factor
          const int ec = ihe + E + em;
          const double c = ec < 1 ? 0.0 : __hiloint2double((ihm & 0x800fffff) | (min(ec, 2046) << 20), ihl);
          rv[q] = fma(c, __ll2double_rn(S), q == 0 ? fr.x : fr.y);
        }
        if (ok0) {
          acc = fma(rv[0], rv[0], acc);
          if (d) put<Ti, RN>(d + r * a.syi + c0, rv[0]);
        }
        if (ok1) {
          acc = fma(rv[1], rv[1], acc);
          if (d) put<Ti, RN>(d + r * a.syi + c0 + 1, rv[1]);
        }
      }
      Fy[0] = Fn[0];
      Fy[1] = Fn[1];
      ey[0] = en[0];
      ey[1] = en[1];
    }
    // x-fluxes of this row: column c to c + 1
    const long long right = fx2::shdn(Y[0]);
    Fx[0] = flux(Y[0] - Y[1], kx.x, ex[0]);
    Fx[1] = flux(Y[1] - right, kx.y, ex[1]);
    X[0] = Y[0];
    X[1] = Y[1];
    kyr = ky;
    fr = f;
  }
  if (good) return acc;
  // FP64, node by node
  acc = 0.0;
  for (int row = r0; row < r1; row++)
#pragma unroll
    for (int q = 0; q < 2; q++) {
      if (!(q == 0 ? ok0 : ok1)) continue;
      const long long p = (long long)row * a.sy + c0 + q;
      const double u0 = a.u[p];
      const double s = a.kx[p] * (u0 - a.u[p + 1]) + a.kx[p - 1] * (u0 - a.u[p - 1]) + a.ky[p] * (u0 - a.u[p + a.sy]) +
                       a.ky[p - a.sy] * (u0 - a.u[p - a.sy]);
      const double r = a.f[p] - s * a.ih2;
      acc += r * r;
      if (d) put<Ti, RN>(d + (long long)row * a.syi + c0 + q, r);
    }
  return acc;
}

// One problem by the blocks of a grid row; the block's sum of squares, valid in thread 0.
template <typename Ti, bool RN> __device__ __forceinline__ double residual(const Prob &a) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, count = tasks(a);
  double acc = 0.0;
  for (int t = blockIdx.x * kWarps + w; t < count; t += gridDim.x * kWarps) acc += task<Ti, RN>(a, t, lane);
  return block_sum(acc);
}

}  // namespace dv2
}  // namespace mg
