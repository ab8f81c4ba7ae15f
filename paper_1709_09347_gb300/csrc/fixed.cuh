// Fixed-point arithmetic of the complex128 operator apply.
//
// This part has 1.6-1.9 FP64 lanes per clock and SM but 64 lanes of 32x32+64-bit integer
// multiply-add and of 64-bit addition (measured: 59 each), so the complex128 stencil and
// projector sums run on integers.  The values of one (system, column) share one power-of-two
// scale taken from the column's largest component:
//     x ~ xi * 2^(ex - Q),   |component| < 2^ex,   Q <= 59,
// the sums of neighbours are exact 64-bit integer sums, the finite-difference coefficients
// enter as the integers n_k of c_k = +-n_k / den, and every product keeps both words of both
// factors, so an output is rounded once, when it is converted back to FP64.  The error of an
// output is about 2^(ex - Q) / 4 times the root of the sum of the squared weights; the FP64
// kernels' is about 2^-53 of the local partial sums, of each part for itself.  The fixed-point one is
// no larger where the real parts over a point and its nearest neighbours hold one of at least 2^53
// units, and the imaginary parts too (k_gather_fixed has its own test, on the terms of its sums).
// A point without them (one of a real field, say), a column whose largest component is zero, not
// finite or extreme, and a system whose twist or energy is out of range take the FP64 formula
// instead, point by point.  Inside BiCG and its residual check the moduli are looked at: its updates
// with complex scalars round a part against the larger of the two.
#pragma once

#include "tails.cuh"

namespace cbs {

constexpr int kFixMaxQ = 59;
constexpr int kFixSmallWord = 1 << (53 - 32);   // high word of the smallest value that counts

// Columns of which too many points would leave fixed point take the FP64 formula as a whole: point
// by point the fixed-point sums are paid as well, and a warp pays for an FP64 output whatever its
// active lanes (32x32x16 cell, 32 systems of 32 columns: fixed point 0.9 ms, FP64 3.0, point by
// point on localised columns 4.5).  At one point in 24, two warps in three hold one and the two
// cost about the same; 32 points of each column are looked at.  An FP64 warp covers 32 columns, so
// one such column takes the 32 along.
constexpr int kFixSamples = 32, kFixPoor = 2, kFixRoute = 32;

// Exponents of one (system, column).
struct FixScale {
  int ok;     // 0: FP64 formula for every point of the column
  int Q, ex;  // unit of the vector components: 2^(ex - Q)
  int sa;     // y = (A 2^62 + B 2^31 + C) products >> (62 - sa), in units 2^uy
  int uy;
  int sp;     // projector products (A 2^58 + B 2^29 + C) enter y as >> (58 - sp)
  int fd;     // projector coefficients are stored as D * 2^fd
};

__device__ __forceinline__ int float_exp_above(float f) {   // 2^r > f for a positive normal f
  return (int)((__float_as_uint(f) >> 23) & 255u) - 126;
}

// maxhi: largest high word of |component| over the column.
__device__ __forceinline__ FixScale fix_scale(const HamView &H, const VlocUnit &u, double2 w, double2 wi, double E,
                                              unsigned maxhi) {
  FixScale s;
  const float a = fmaxf(fmaxf(fabsf((float)w.x), fabsf((float)w.y)), fmaxf(fabsf((float)wi.x), fabsf((float)wi.y)));
  const double de = fabs(E - H.diag_kin) + u.vmax;
  s.ex = (int)(maxhi >> 20) - 1022;
  // (a NaN would pass through fmaxf: the products with zero are NaN for it)
  const bool finite = w.x * 0.0 + w.y * 0.0 + wi.x * 0.0 + wi.y * 0.0 == 0.0;
  s.ok = u.ew == H.fx_ew && finite && a < 8.0f && s.ex > -700 && s.ex < 700 && __double2hiint(de) < ((1023 + H.fx_ew) << 20) && de >= 0.0;
  if (!s.ok) {
    s.Q = kFixMaxQ; s.ex = 0; s.sa = 0; s.uy = 0; s.sp = 0; s.fd = 0;
    return s;
  }
  // modulus of the larger of w and 1/w, and what twisted values can reach (larger twists would
  // leave the projector coefficients, bounded with tw^2, too few bits)
  const float wm = fmaxf(1.0f, sqrtf(fmaxf((float)w.x * (float)w.x + (float)w.y * (float)w.y,
                                            (float)wi.x * (float)wi.x + (float)wi.y * (float)wi.y)) * 1.0001f);
  const float tw = 1.4143f * wm;
  s.Q = min(kFixMaxQ, 63 - float_exp_above(4.0f + 2.0f * tw));
  const float yb = H.fx_wxy + H.fx_wz * tw + exp2f((float)H.fx_ew) * 1.0001f + H.fx_pb * tw * tw;
  const int lb = float_exp_above(yb * 1.0001f);
  s.sa = min(24, 66 + H.fx_ew - s.Q - lb);
  s.uy = s.ex - s.Q + H.fx_ew + 4 - s.sa;
  // the coefficients (and their twisted images) in 57 bits
  s.sp = H.fx_db > 0 ? max(0, 1 + float_exp_above(H.fx_db * tw * tw * 1.0001f) + s.ex - H.fx_fp - s.uy) : 0;
  s.fd = 58 - H.fx_fp - s.sp - s.uy;
  s.ok = s.sa >= 0 && s.sp <= 24 && wm < 4.5f;
  return s;
}

// floor(x * 2^(Q - ex)) for |x| < 2^ex; base = 1086 + ex - Q.  The significand, left-justified
// with its hidden bit, is shifted down and one's-complemented for a negative x, which is the
// floor (values below one unit, zero among them, give 1 or -2).
// word collects the high words of the magnitudes.
__device__ __forceinline__ long long to_fixed(double x, int base, int &word) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int e = (int)(((unsigned)hi << 1) >> 21);
  const unsigned mh = __funnelshift_l((unsigned)lo, (unsigned)hi, 11) | 0x80000000u;
  const unsigned ml = (unsigned)lo << 11;
  const unsigned long long m = ((unsigned long long)mh << 32) | ml;
  const unsigned long long v = m >> min((unsigned)(base - e), 63u);
  const long long sg = hi >> 31;
  word |= (int)(v >> 32);
  return (long long)v ^ sg;
}
__device__ __forceinline__ long long to_fixed(double x, int base) {
  int word = 0;
  return to_fixed(x, base, word);
}

// v * 2^k in FP64 (one rounding); |k| well inside the exponent range
__device__ __forceinline__ double from_fixed(long long v, int k) {
  const double d = (double)v;
  return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (k << 20), __double2loint(d));
}

// rint(d * 2^k)
__device__ __forceinline__ long long round_fixed(double d, int k) {
  // two factors: 2^k itself may leave the exponent range when d is small
  const int k1 = k / 2, k2 = k - k1;
  return __double2ll_rn(d * __hiloint2double((1023 + k1) << 20, 0) * __hiloint2double((1023 + k2) << 20, 0));
}

// c += a * b, 32 x 32 + 64 bits, one instruction.  A factor cut out of a 64-bit value must be
// hidden from the compiler (opaque): seen through, its extension to 64 bits is not that of a
// plain int any more and the product becomes a full 64-bit multiplication.
__device__ __forceinline__ void madw(long long &c, int a, int b) { c += (long long)a * b; }
__device__ __forceinline__ void madwu(unsigned long long &c, unsigned a, unsigned b) {
  c += (unsigned long long)a * b;
}
__device__ __forceinline__ int opaque(int a) {
  asm("" : "+r"(a));
  return a;
}

__device__ __forceinline__ int hi31(long long x) { return opaque((int)(x >> 31)); }
__device__ __forceinline__ int lo31(long long x) { return opaque((int)x & 0x7fffffff); }

// v = hi 2^29 + lo with -2^28 <= lo < 2^28
__host__ __device__ __forceinline__ int balanced_hi(long long v) { return (int)((v + (1 << 28)) >> 29); }
__host__ __device__ __forceinline__ int balanced_lo(long long v) {
  return (int)((v + (1 << 28)) & 0x1fffffff) - (1 << 28);
}

// high word of a fixed-point component's magnitude (of |v| - 1 for a negative one)
__device__ __forceinline__ int absword(long long v) {
  const int h = (int)(v >> 32);
  return h ^ (h >> 31);
}

// -lim <= h < lim
__device__ __forceinline__ bool within(int h, int lim) { return (unsigned)(h + lim) < 2u * (unsigned)lim; }

// What one (system, column) needs besides its vector.
struct ColumnScale {
  FixScale f;
  int base;        // exponent offset of to_fixed
  long long ef;    // E - diag_kin in the unit of the weights
  long long skip;  // 1: the column takes no part (its output is not written); 2: it takes the FP64 formula
  double2 w, wi;   // the twist and its inverse
};
static_assert(sizeof(ColumnScale) % 16 == 0, "ColumnScale is read in 16-byte pieces");

__device__ __forceinline__ ColumnScale column_scale(const HamView &H, double2 w, double E, unsigned maxhi, bool skip) {
  ColumnScale o;
  o.w = w;
  o.wi = cdiv(make_double2(1.0, 0.0), w);
  const VlocUnit u = *H.fx_u;
  o.f = fix_scale(H, u, w, o.wi, E, maxhi);
  o.base = 1086 + o.f.ex - o.f.Q;
  o.ef = o.f.ok ? round_fixed(E, 58 - H.fx_ew) - H.fx_diag : 0;
  o.skip = skip;
  return o;
}

// The same apply with the columns' scales already in place (fixed_scales of the scratch), for
// callers that know the maxima; with `dot`, the stencil also sums (p~, q) over the columns of
// the first dot->n systems, p~ the input of system n + s, and its last block per system forms
// alpha.
struct FixedDot {
  int n = 0;
  double *part = nullptr;   // [n][fixed_dot_parts][L][2]
  AlphaTail tail;
};
ColumnScale *fixed_scales(const HamView &H, int n_sys, int L, void *ws);
int fixed_dot_parts(const HamView &H, int n_sys, int L);
cbs_status apply_fixed_scaled(const HamView &H, int n_sys, int L, const double2 *X, double2 *Y, const double *E,
                              void *ws, const int *sys_active, cudaStream_t st, bool parts, const FixedDot *dot);

}  // namespace cbs
