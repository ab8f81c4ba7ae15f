// The rotation of one-sided Jacobi (host and device, so that its accuracy can be checked on either).
#pragma once

#include "common.cuh"

namespace cbs {

// Rotation that makes two columns orthogonal, from their squared norms al, be and inner product
// g: with g = |g| e^{i phi}, zeta = (be - al)/(2|g|), t the smaller root of
// t^2 + 2 zeta t - 1 = 0,
//   a_p' = c a_p - s e^{-i phi} a_q,  a_q' = s e^{i phi} a_p + c a_q,   sp = s e^{i phi}.
// False where the pair is orthogonal to tolj.  It stands alone on every round's critical path,
// so it avoids the divisions and hypot of the textbook form (about 150 dependent FP64
// operations): t starts in single precision and takes two Newton steps, whose slope in single
// precision is enough (after one, sp is off by up to 2e-14; after two it is as good as the textbook's).
__host__ __device__ __forceinline__ bool pair_rotation(double al, double be, double gx, double gy, double tolj,
                                                       double &c, double2 &sp) {
  const double g2 = fma(gx, gx, gy * gy), ab = al * be;
  if (al == 0.0 || be == 0.0) return false;
  if (!(g2 > 1e-270 && g2 < 1e270 && ab > 1e-270 && ab < 1e270)) {
    const double g = hypot(gx, gy);
    if (!(g > tolj * (sqrt(al) * sqrt(be)))) return false;
    const double zeta = (be - al) / (2.0 * g);
    const double t = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
    c = 1.0 / sqrt(1.0 + t * t);
    sp = make_double2(c * t * (gx / g), c * t * (gy / g));
    return true;
  }
  if (!(g2 > tolj * tolj * ab)) return false;
  const double ig = rsqrt(g2);
  const double zeta = 0.5 * (be - al) * ig, az = fabs(zeta);
  double t;
  if (az < 1e15) {
    const float zf = (float)az, t0 = 1.0f / (zf + sqrtf(fmaf(zf, zf, 1.0f)));
    const double h = (double)(0.5f / (t0 + zf)), z2 = 2.0 * az;
    t = (double)t0;
    t = fma(-fma(z2, t, fma(t, t, -1.0)), h, t);
    t = fma(-fma(z2, t, fma(t, t, -1.0)), h, t);
  } else {
    t = 0.5 / az;
  }
  c = rsqrt(fma(t, t, 1.0));
  const double s = copysign(c * t, zeta) * ig;
  sp = make_double2(s * gx, s * gy);
  return true;
}

}  // namespace cbs
