// Device helpers shared by the tiled pair kernel (dh_kernels.cu) and the list
// kernel (dh_list.cu): float32 primitives, the branch-free counting step,
// double-float arithmetic and the binary64 definition.  Not part of the ABI.
#pragma once

#include <math.h>
#include <stdint.h>

#include "dh_internal.h"

namespace dh {

// Order-preserving map float -> int32 (for atomicMin/atomicMax on floats).
__device__ __forceinline__ int32_t ord_of(float f) {
  int32_t i = __float_as_int(f);
  return i >= 0 ? i : (i ^ 0x7FFFFFFF);
}
__device__ __forceinline__ float float_of_ord(int32_t k) {
  return __int_as_float(k >= 0 ? k : (k ^ 0x7FFFFFFF));
}

constexpr float kMagicRound = 12582912.0f;  // 1.5 * 2^23: fma(x, s, M) - M = nint_even(x*s), |x*s| < 2^22
constexpr float kMagicFloor = 8388608.0f;   // 2^23: fadd.rd(t, 2^23) - 2^23 = floor(t), 0 <= t < 2^23
constexpr unsigned kFull = 0xffffffffu;

// Relative error bound assumed for sqrt.approx.ftz.f32 (checked exhaustively
// over two binades by the GPU test suite).
constexpr double kSqrtRelErr = 8.0 / 16777216.0;  // 8 * 2^-24

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// IEEE minimum that propagates NaN (masked pairs carry NaN and must stay NaN).
__device__ __forceinline__ float min_nan(float a, float b) {
  float y;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}
__device__ __forceinline__ float nint_scaled(float x, float s) {
  return __fadd_rn(__fmaf_rn(x, s, kMagicRound), -kMagicRound);
}
__device__ __forceinline__ float nint_f(float x) {
  return __fadd_rn(__fadd_rn(x, kMagicRound), -kMagicRound);
}

// ---- packed float32 arithmetic: two pairs per instruction (FFMA2/FADD2/FMUL2)

__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Guard words on each side of a shared-memory histogram copy: the increments
// of pairs outside [lo, hi) land there (see count_or_defer).
constexpr int kGuard = 36;

// Count one pair, branch free.  With sm = s_c + 1.5*2^23 (s_c the clamped root,
// bits(sm) - bits(1.5*2^23) = its nearest integer n) and the residual
// e = n^2 - q (e > 0: t < n, so floor(t) = n - 1; e < 0: floor(t) = n), the
// bin relative to the sweep is v - kb1 with v = bits(sm) + signbit(e), and the
// shared-memory address is 4 v + hbase (a shift and an add, which stay off the
// FMA pipe that the packed float32 arithmetic keeps busy; a multiply-add by 4
// measured 1-2 % slower).  Every pair increments that word.  The
// clamp of s_c to [lo - lane, hi + 1 + lane] (integers below 2^22) keeps the
// relative bin in [-1 - lane, width + 1 + lane]: pairs outside the sweep, and
// NaN pairs (s_c = hi + 1 + lane, e NaN with a clear sign bit: bin width + lane),
// land in the guard words, spread over the lanes.  A clamped pair that is
// decided is decided right: e > bound means t lies within the clamp's integer
// and the one below, e < -bound that t lies above it, out of the sweep (and
// the converse at the lower clamp).  A pair with |e| <= bound (false for NaN)
// also sets the bit `bit` of dmask: it is counted provisionally and re-decided
// by the drain, which moves its count to the exact bin when the two differ.
__device__ __forceinline__ void count_or_defer(float sm, float e, float bound, uint32_t hbase, uint32_t bit,
                                               uint32_t& dmask) {
  asm volatile(
      "{\n\t.reg .pred pn;\n\t.reg .u32 eb, sg, v, addr;\n\t.reg .f32 ae;\n\t"
      "mov.b32 eb, %2;\n\t"
      "shr.u32 sg, eb, 31;\n\t"
      "add.u32 v, %1, sg;\n\t"
      "shl.b32 addr, v, 2;\n\t"
      "add.u32 addr, addr, %4;\n\t"
      "abs.f32 ae, %2;\n\t"
      "setp.gtu.f32 pn, ae, %3;\n\t"
      "@!pn or.b32 %0, %0, %5;\n\t"
      "red.shared.add.u32 [addr], 1;\n\t"
      "}"
      : "+r"(dmask)
      : "r"(__float_as_uint(sm)), "f"(e), "f"(bound), "r"(hbase), "r"(bit));
}

// ---- double-float middle tier

struct DF {
  float h, l;  // unevaluated sum h + l
};

__device__ __forceinline__ DF two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
// The multiple of the grid (a power of two) nearest to v (|v| < 2^22 steps).
__device__ __forceinline__ float on_grid(float v, float grid) {
  const float m = kMagicRound * grid;
  return __fsub_rn(__fadd_rn(v, m), m);
}
__device__ __forceinline__ DF two_prod(float a, float b) {
  float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
// v - k (bh + bl) for an integer k, renormalised: after a large image is
// taken off, the low part of v (the rounding error of a difference of large
// coordinates) can be far above an ulp of the small result, and the products
// of df_norm2 are accurate only for a normalised pair (|l| <= ulp(h) / 2)
__device__ __forceinline__ DF df_sub_kb(DF v, float k, float bh, float bl) {
  DF p = two_prod(k, bh);
  DF s = two_sum(v.h, -p.h);
  float low = __fmaf_rn(-k, bl, __fsub_rn(__fadd_rn(v.l, s.l), p.l));
  return two_sum(s.h, low);
}
__device__ __forceinline__ DF df_norm2(DF x, DF y, DF z) {
  DF ax = two_prod(x.h, x.h), ay = two_prod(y.h, y.h), az = two_prod(z.h, z.h);
  DF s1 = two_sum(ax.h, ay.h);
  DF s2 = two_sum(s1.h, az.h);
  float low = __fadd_rn(__fadd_rn(__fadd_rn(ax.l, ay.l), __fadd_rn(az.l, s1.l)), s2.l);
  low = __fmaf_rn(__fadd_rn(x.h, x.h), x.l, low);
  low = __fmaf_rn(__fadd_rn(y.h, y.h), y.l, low);
  low = __fmaf_rn(__fadd_rn(z.h, z.h), z.l, low);
  low = __fmaf_rn(x.l, x.l, __fmaf_rn(y.l, y.l, __fmaf_rn(z.l, z.l, low)));
  return {s2.h, low};
}

// xj - xi for binary64 values, as a double-float: each value split into float32
// high and low parts (x = h + l to about 2^-48 |x|), the high parts subtracted
// exactly and the low parts added to the error term.
__device__ __forceinline__ DF df_diff64(double xj, double xi) {
  const float hj = __double2float_rn(xj), hi = __double2float_rn(xi);
  const float lj = __double2float_rn(__dsub_rn(xj, (double)hj)), li = __double2float_rn(__dsub_rn(xi, (double)hi));
  DF s = two_sum(hj, -hi);
  return two_sum(s.h, __fadd_rn(s.l, __fsub_rn(lj, li)));  // renormalised (see df_sub_kb)
}

// ---- binary64 last resort

// The displacement of the definition's nearest image in binary64 (Alg. 1, Eq. 5),
// the same operations in the same order; for boxes with the image search, the
// image the 27 neighbouring shifts start from.  The coordinates are the caller's
// (float32 promoted exactly, or binary64).
template <int V>
__device__ __forceinline__ double3 exact_image(const FrameDev& F, double3 pi, double3 pj) {
  double dx = __dsub_rn(pj.x, pi.x);
  double dy = __dsub_rn(pj.y, pi.y);
  double dz = __dsub_rn(pj.z, pi.z);
  const double* B = F.B;
  if (V == V_ORTHO) {
    double kx = rint(__dmul_rn(dx, F.Linv[0]));
    double ky = rint(__dmul_rn(dy, F.Linv[1]));
    double kz = rint(__dmul_rn(dz, F.Linv[2]));
    dx = __fma_rn(-kx, B[0], dx);
    dy = __fma_rn(-ky, B[4], dy);
    dz = __fma_rn(-kz, B[8], dz);
  } else if (V == V_TRIC || V == V_TRIC_SEARCH) {
    const double ax = B[0], bx = B[1], cx = B[2], by = B[4], cy = B[5], cz = B[8];
    double sz = __ddiv_rn(dz, cz);
    double sy = __ddiv_rn(__dsub_rn(dy, __dmul_rn(cy, sz)), by);
    double sx = __ddiv_rn(__dsub_rn(__dsub_rn(dx, __dmul_rn(bx, sy)), __dmul_rn(cx, sz)), ax);
    double kx = rint(sx), ky = rint(sy), kz = rint(sz);
    dx = __dsub_rn(__dsub_rn(__dsub_rn(dx, __dmul_rn(ax, kx)), __dmul_rn(bx, ky)), __dmul_rn(cx, kz));
    dy = __dsub_rn(__dsub_rn(dy, __dmul_rn(by, ky)), __dmul_rn(cy, kz));
    dz = __dsub_rn(dz, __dmul_rn(cz, kz));
  }
  return make_double3(dx, dy, dz);
}

// Squared minimum-image distance in binary64: exact_image, then the 27
// neighbouring shifts where the definition's minimum needs them.
template <int V>
__device__ double exact_r2(const FrameDev& F, double3 pi, double3 pj) {
  const double3 d = exact_image<V>(F, pi, pj);
  const double dx = d.x, dy = d.y, dz = d.z;
  if (V == V_TRIC_SEARCH) {
    // Below half the plane spacing (V_TRIC: r_max <= (1 - 2^-8) h_min / 2) the
    // shift m = 0 is the minimum of the 27 for every pair inside r_max: the
    // sequential rounding is Babai's nearest plane in the upper-triangular
    // basis, exact for vectors shorter than half its smallest Gram-Schmidt
    // length (cz, by, ax >= h_min), and every other shift is longer than
    // h_min - r_max > r_max.  Its value is the m = 0 term of the loop, bit for
    // bit (adding the zero products changes nothing); a pair beyond r_max stays
    // beyond it under any shift.  So the binary64 bin is the definition's.
    const double* B = F.B;
    const double ax = B[0], bx = B[1], cx = B[2], by = B[4], cy = B[5], cz = B[8];
    double best = INFINITY;
#pragma unroll 1
    for (int mx = -1; mx <= 1; ++mx)
#pragma unroll 1
      for (int my = -1; my <= 1; ++my)
#pragma unroll 1
        for (int mz = -1; mz <= 1; ++mz) {
          double ex = __dadd_rn(__dadd_rn(__dadd_rn(dx, __dmul_rn(ax, (double)mx)), __dmul_rn(bx, (double)my)),
                                __dmul_rn(cx, (double)mz));
          double ey = __dadd_rn(__dadd_rn(dy, __dmul_rn(by, (double)my)), __dmul_rn(cy, (double)mz));
          double ez = __dadd_rn(dz, __dmul_rn(cz, (double)mz));
          double r2 = __fma_rn(ez, ez, __fma_rn(ey, ey, __dmul_rn(ex, ex)));
          if (r2 < best) best = r2;
        }
    return best;
  }
  return __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx)));
}

// Bin of a binary64 r^2 from the threshold table: the largest k with T[k] <= r2
// (T[0] = 0, T nondecreasing; 0 for NaN).  The float32 estimate S sqrt(r2) is
// within a bin or two of it; the two walks make the result exact whatever the
// estimate, with one or two dependent loads instead of a binary search's
// log2(nbins).
__device__ __forceinline__ int bin_from_thresholds(const double* __restrict__ T, float S, int nbins, double r2) {
  if (!(r2 >= 0.0)) return 0;
  int k = (int)fminf(__fmul_rn(sqrtf(__double2float_rn(r2)), S), (float)nbins);
  while (k > 0 && __ldg(T + k) > r2) --k;
  while (k < nbins && __ldg(T + k + 1) <= r2) ++k;
  return k;
}

// The caller's coordinates of particle i of a frame, in binary64.
__device__ __forceinline__ double3 coords64(const FrameDev& F, int i) {
  if (F.X64) {
    double4 p = F.X64[i];
    return make_double3(p.x, p.y, p.z);
  }
  float4 p = __ldg(F.X + i);
  return make_double3((double)p.x, (double)p.y, (double)p.z);
}

}  // namespace dh
