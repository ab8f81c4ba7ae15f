// The complex128 operator apply Y = E X - H(w) X in fixed point (see fixed.cuh for the
// arithmetic and apply.cu for the operator).  Four kernels:
//   k_column_max     the largest |component| of every (system, column) over chunks of points,
//   k_fix_scales     from it the column's scale, with its twist and energy,
//   k_gather_fixed   D_a = h_a F_a(1/w)^T X per atom, as FP64 and as fixed-point images
//                    D, w D, w^{-1} D,
//   k_stencil_fixed  the stencil and the projector scatter.
// Scratch: D [n_sys][n_atoms][L][4] FP64, then the images [n_sys][3][n_atoms][4][L] as
// (high, low) word pairs of both components (images of wrap -1, 0, +1), then the scales
// [n_sys][L], then the chunk maxima [n_sys][chunks][L].
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "fixed.cuh"

namespace cbs {

// Bound by memory: 44 us for 268 MB (32 systems of the 32x32x16 cell, L = 32), 6.1 TB/s.
// maxhi[s][chunk][c] = max over the chunk's points of the high word of |re|, |im| (the order of
// non-negative doubles)
__global__ void k_column_max(int64_t N, int L, int chunk_pts, const double2 *__restrict__ X,
                             unsigned *__restrict__ maxhi, const int *__restrict__ sys_active) {
  extern __shared__ unsigned smax[];   // [py][L]
  const int s = blockIdx.y, c = threadIdx.x, ly = threadIdx.y, py = blockDim.y;
  if (sys_active && !sys_active[s]) return;
  const int64_t i0 = (int64_t)blockIdx.x * chunk_pts, i1 = min(N, i0 + chunk_pts);
  const double2 *Xs = X + (int64_t)s * N * L;
  unsigned m = 0;
#pragma unroll 4
  for (int64_t i = i0 + ly; i < i1; i += py) {
    const double2 v = Xs[i * L + c];
    m = max(m, max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu));
  }
  smax[ly * L + c] = m;
  __syncthreads();
  if (ly == 0) {
    for (int y = 1; y < py; ++y) m = max(m, smax[y * L + c]);
    maxhi[((int64_t)s * gridDim.x + blockIdx.x) * L + c] = m;
  }
}

// Sample k of a cell of n points: hashed, since steps that divide the grid's would meet one corner of
// it only.
__device__ __forceinline__ int sample_point(int k, int64_t n) {
  return (int)(((unsigned long long)((k + 1) * 0x9e3779b9u) * (unsigned long long)n) >> 32);
}

// High words of the magnitudes of both components of a point.
__device__ __forceinline__ uint2 point_words(const double2 *Xc, int L, int i) {
  const double2 v = Xc[(int64_t)i * L];
  return make_uint2((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
}

// The larger of these over point i and its nearest neighbours, in a column whose first element is Xc.
__device__ __forceinline__ uint2 words_around(const HamView &H, const double2 *Xc, int L, int i) {
  const int nx = H.nx, ny = H.ny, nz = H.nz, sz = nx * ny;
  const int ix = i % nx, iy = i / nx % ny, iz = i / sz;
  const int step[6] = {ix + 1 < nx ? 1 : 1 - nx, ix > 0 ? -1 : nx - 1,        iy + 1 < ny ? nx : nx - sz,
                       iy > 0 ? -nx : sz - nx,   iz + 1 < nz ? sz : sz - sz * nz, iz > 0 ? -sz : sz * nz - sz};
  uint2 m = point_words(Xc, L, i);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const uint2 v = point_words(Xc, L, i + step[k]);
    m.x = max(m.x, v.x);
    m.y = max(m.y, v.y);
  }
  return m;
}

// One block of (L, lanes) per system: the FP64 work of the scales (a division, the conversions) is
// done here once instead of by every thread of the kernels that use them.  The lanes share the
// chunks and the samples of a column; bound by latency, so the samples are loaded beside the maxima.
// Without `parts` no column is sent to the FP64 formula as a whole.
__global__ void __launch_bounds__(1024) k_fix_scales(const __grid_constant__ HamView H, int L, int chunks,
                                                     const unsigned *__restrict__ maxhi, const double2 *__restrict__ X,
                                                     const double2 *__restrict__ twist, int per_col,
                                                     const double *__restrict__ E, ColumnScale *__restrict__ scales,
                                                     const int *__restrict__ sys_active, bool parts) {
  extern __shared__ unsigned smax[];   // [lanes][L], lim [L], poor [L]
  __shared__ int bad[256 / kFixRoute];
  const int s = blockIdx.x, c = threadIdx.x, ly = threadIdx.y, ry = blockDim.y;
  if (sys_active && !sys_active[s]) return;
  const double2 *Xc = X + (int64_t)s * H.n * L + c;
  unsigned m = 0;
  for (int k = ly; k < chunks; k += ry) m = max(m, maxhi[((int64_t)s * chunks + k) * L + c]);
  double2 w = make_double2(1, 0);
  double energy = 0;
  if (ly == 0) {
    w = twist[per_col ? (int64_t)s * L + c : s];
    energy = E[s];
  }
  constexpr int U = kFixSamples / 4;   // at least 4 lanes
  unsigned word[U];                    // the smaller part's
#pragma unroll
  for (int j = 0; j < U; ++j) {
    word[j] = ~0u;
    if (parts && ly + j * ry < kFixSamples) {
      const uint2 v = words_around(H, Xc, L, sample_point(ly + j * ry, H.n));
      word[j] = min(v.x, v.y);
    }
  }
  smax[ly * L + c] = m;
  unsigned *lim = smax + ry * L, *poor = lim + L;
  __syncthreads();
  ColumnScale o;
  if (ly == 0) {
    for (int y = 1; y < min(ry, chunks); ++y) m = max(m, smax[y * L + c]);
    o = column_scale(H, w, energy, m, false);
    lim[c] = o.f.ok ? (unsigned)(o.f.ex - o.f.Q + 53 + 1023) << 20 : 0u;
    poor[c] = 0;
    if (c % kFixRoute == 0) bad[c / kFixRoute] = 0;
  }
  __syncthreads();
  const unsigned lm = lim[c];
  int p = 0;
#pragma unroll
  for (int j = 0; j < U; ++j) p += word[j] < lm;
  if (p) atomicAdd(&poor[c], (unsigned)p);
  __syncthreads();
  if (parts && ly == 0 && (!o.f.ok || poor[c] >= kFixPoor)) bad[c / kFixRoute] = 1;
  __syncthreads();
  if (ly) return;
  if (bad[c / kFixRoute]) o.skip = 2;
  scales[(int64_t)s * L + c] = o;
}

// FP64 sums of one image of one atom over the entries t0, t0 + step, ... in gather order: the columns
// that fixed point does not serve.  Bound by FP64 issue, as k_proj_gather is.
__device__ __noinline__ void gather_entries_fp64(const HamView *H, int t0, int t1, int step, int L, const double2 *Xc,
                                                 double2 *out) {
  double2 acc[4];
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) acc[mu] = make_double2(0, 0);
  const int np = H->n_proj;
  constexpr int U = 4;   // rows in flight
  for (int tb = t0; tb < t1; tb += U * step) {
    double2 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = tb + u * step < t1 ? Xc[(int64_t)H->fx_gi[tb + u * step] * L] : make_double2(0, 0);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (tb + u * step >= t1) break;
      const double *p = H->sup_val + (int64_t)H->fx_gt[tb + u * step] * np;
#pragma unroll
      for (int mu = 0; mu < 4; ++mu)
        if (mu < np) {
          acc[mu].x = fma(p[mu], x[u].x, acc[mu].x);
          acc[mu].y = fma(p[mu], x[u].y, acc[mu].y);
        }
    }
  }
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) out[mu] = acc[mu];
}

// Bound by the latency of its integer products and of the gathered rows at 16 warps per SM (it issues
// on 38 per cent of the cycles): 32 systems of the 32x32x16 cell (40 atoms, L = 32) take 194 us (175
// without PARTS); the FP64 gather, at FP64 issue, 550 us.  About 90 instructions per entry and
// column, 24 of them products.
// One block per (atom, system, group of columns); threadIdx.x a column, threadIdx.y a lane over
// the atom's support entries.  Per entry: one 16-byte load, two conversions and 3 word
// products per projector and component.  The projector words are balanced (the low word is
// signed), so the product of the two low words, left out but for its mean (which depends on the
// projector alone), is below 2^-58 of the largest product per entry.
// A sum is about as accurate as the FP64 one where one of its larger projector values (a quarter of the
// largest, at least six of them) meets a component of at least 2^54 units.  PARTS: each projector is watched for that, the
// real and the imaginary parts for themselves, and a column without it over the atom is summed in
// FP64.  BiCG, which mixes the parts, has the moduli over the atom looked at.
constexpr int kGatherU = 8;      // entries in flight per thread
constexpr int kGatherCarry = 2;  // steps of kGatherU entries between carries: |B| grows by less
                                 // than 2^58.4 per entry
template <bool PARTS>
__global__ void __launch_bounds__(256, 2) k_gather_fixed(const __grid_constant__ HamView H, int L,
                                                      const double2 *__restrict__ X,
                                                      const ColumnScale *__restrict__ scales,
                                                      double2 *__restrict__ D, int4 *__restrict__ Df,
                                                      const int *__restrict__ sys_active) {
  extern __shared__ long long gsm[];
  const int a = blockIdx.x, s = blockIdx.y;
  if (sys_active && !sys_active[s]) return;
  const int cg = blockDim.x, ly = threadIdx.y, py = blockDim.y;
  const int cx = threadIdx.x;
  const int c = min((int)(blockIdx.z * cg) + cx, L - 1);
  const bool own = (int)(blockIdx.z * cg) + cx < L;
  long long *redA = gsm;                                   // [py][8][cg]
  long long *redB = redA + (size_t)py * 8 * cg;            // [py][8][cg]
  double2 *sums = (double2 *)(redB + (size_t)py * 8 * cg); // [4][cg] F_a(1/w)^T X
  int *seen = (int *)(sums + 4 * cg);                      // [2][cg] large components met
  const ColumnScale *sc = scales + (int64_t)s * L + c;
  const FixScale f = sc->f;
  const int base = sc->base;
  const double2 *Xc = X + (int64_t)s * H.n * L + c;
  const char *Xb = (const char *)(X + (int64_t)s * H.n * L);
  const unsigned row = (unsigned)L * (unsigned)sizeof(double2), col = (unsigned)c * (unsigned)sizeof(double2);
  const int *gp = H.fx_gptr + 4 * a;
  if (ly == 0) {
    seen[cx] = seen[cg + cx] = 0;
    for (int mu = 0; mu < 4; ++mu) sums[mu * cg + cx] = make_double2(0, 0);
  }
  // a warp pays for its FP64 sums whatever its active lanes: one column without a scale takes the
  // block's others along
  const bool all64 = __syncthreads_or(sc->skip != 1 && (!f.ok || sc->skip == 2));
  int met01 = 0, met23 = 0;   // PARTS: a byte per projector and part, else high words
  for (int img = 0; img < 3 && !all64; ++img) {
    const int t0 = gp[img], t1 = gp[img + 1];
    if (t0 == t1) continue;
    long long A[8], B[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) A[k] = B[k] = 0;
    const int *gi = H.fx_gi + t0 + ly;
    const int4 *pw = H.fx_gp + 2 * (t0 + ly);
    const int2 *pm = H.fx_gm + t0 + ly;
    int left = (t1 - t0 - ly + py - 1) / py;     // this thread's entries
    auto fetch = [&](int u) -> double2 { return *(const double2 *)(Xb + ((unsigned)gi[u * py] * row + col)); };
    auto take = [&](double2 x, const int4 *p, const int2 *large) {
      const int4 p01 = p[0], p23 = p[1];
      int wr = 0, wi = 0;
      const long long xr = to_fixed(x.x, base, wr), xi = to_fixed(x.y, base, wi);
      if constexpr (PARTS) {
        const int2 m = *large;
        const int met = __byte_perm((wr >> 22) | (wi >> 22) << 8, 0, 0x1010);
        met01 |= met & m.x;
        met23 |= met & m.y;
      } else {
        met01 |= wr | wi;
      }
      const int r1 = opaque((int)(xr >> 29)), r0 = opaque((int)xr & 0x1fffffff);
      const int i1 = opaque((int)(xi >> 29)), i0 = opaque((int)xi & 0x1fffffff);
      const int p1[4] = {p01.x, p01.z, p23.x, p23.z}, p0[4] = {p01.y, p01.w, p23.y, p23.w};
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        madw(A[2 * mu], r1, p1[mu]);
        madw(B[2 * mu], r1, p0[mu]);
        madw(B[2 * mu], r0, p1[mu]);
        madw(A[2 * mu + 1], i1, p1[mu]);
        madw(B[2 * mu + 1], i1, p0[mu]);
        madw(B[2 * mu + 1], i0, p1[mu]);
      }
    };
    auto carry = [&]() {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        A[k] += B[k] >> 29;
        B[k] &= 0x1fffffff;
      }
    };
    int step = 0;
    for (; left >= kGatherU; left -= kGatherU) {
      double2 xv[kGatherU];
#pragma unroll
      for (int u = 0; u < kGatherU; ++u) xv[u] = fetch(u);
#pragma unroll
      for (int u = 0; u < kGatherU; ++u) take(xv[u], pw + 2 * u * py, pm + u * py);
      gi += kGatherU * py;
      pw += 2 * kGatherU * py;
      pm += kGatherU * py;
      if (++step % kGatherCarry == 0) carry();
    }
    carry();
    for (; left > 0; --left) {
      take(fetch(0), pw, pm);
      gi += py;
      pw += 2 * py;
      pm += py;
    }
    carry();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      redA[((size_t)ly * 8 + k) * cg + cx] = A[k];
      redB[((size_t)ly * 8 + k) * cg + cx] = B[k];
    }
    __syncthreads();
    // projector mu of column cx: the image's sum, times w^{-m}
    for (int mu = ly; mu < 4; mu += py) {
      // the mean of the products of the low words, 2^28 times the sum of the projector's
      const long long low = H.fx_gc[(a * 3 + img) * 4 + mu];
      long long ar = 0, br = low, ai = 0, bi = low;
      for (int y = 0; y < py; ++y) {
        ar += redA[((size_t)y * 8 + 2 * mu) * cg + cx];
        br += redB[((size_t)y * 8 + 2 * mu) * cg + cx];
        ai += redA[((size_t)y * 8 + 2 * mu + 1) * cg + cx];
        bi += redB[((size_t)y * 8 + 2 * mu + 1) * cg + cx];
      }
      // (A 2^58 + B 2^29) 2^(ex - Q - fp)
      const double unit = __hiloint2double((1023 + f.ex - f.Q - H.fx_fp + 29) << 20, 0);
      double2 v = make_double2(fma((double)ar, 536870912.0, (double)br) * unit,
                               fma((double)ai, 536870912.0, (double)bi) * unit);
      if (img != 1) v = cmul(img == 2 ? sc->wi : sc->w, v);
      sums[mu * cg + cx] = cadd(sums[mu * cg + cx], v);
    }
    __syncthreads();
  }
  if (met01) atomicOr(&seen[cx], met01);
  if (met23) atomicOr(&seen[cg + cx], met23);
  __syncthreads();
  // columns out of range, or with a sum of nothing but small terms: FP64 sums
  bool redo = all64;
  if (PARTS)
    for (int k = 0; k < 2 * H.n_proj; ++k) redo |= !(seen[k / 4 * cg + cx] >> (k % 4 * 8) & 255);
  else
    redo |= seen[cx] < kFixSmallWord;
  redo &= sc->skip != 1;
  if (__syncthreads_or(redo)) {
    double2 *red = (double2 *)gsm;                         // [py][4][cg], the space of redA
    if (redo && ly == 0)
      for (int mu = 0; mu < 4; ++mu) sums[mu * cg + cx] = make_double2(0, 0);
    for (int img = 0; img < 3; ++img) {
      const int t0 = gp[img], t1 = gp[img + 1];   // empty ones too: w may not be finite
      if (redo) {
        double2 part[4];
        gather_entries_fp64(&H, t0 + ly, t1, py, L, Xc, part);
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) red[((size_t)ly * 4 + mu) * cg + cx] = part[mu];
      }
      __syncthreads();
      if (redo)
        for (int mu = ly; mu < 4; mu += py) {
          double2 v = make_double2(0, 0);
          for (int y = 0; y < py; ++y) v = cadd(v, red[((size_t)y * 4 + mu) * cg + cx]);
          if (img != 1) v = cmul(img == 2 ? sc->wi : sc->w, v);
          sums[mu * cg + cx] = cadd(sums[mu * cg + cx], v);
        }
      __syncthreads();
    }
  }
  const double *ha = H.h + (int64_t)a * H.n_proj * H.n_proj;
  if (!own) return;
  for (int mu = ly; mu < 4; mu += py) {
    double2 d = make_double2(0, 0);
    if (mu < H.n_proj)
      for (int nu = 0; nu < H.n_proj; ++nu) {
        const double hv = ha[mu * H.n_proj + nu];
        const double2 v = sums[nu * cg + cx];
        d.x = fma(hv, v.x, d.x);
        d.y = fma(hv, v.y, d.y);
      }
    D[(((int64_t)s * H.n_atoms + a) * L + c) * 4 + mu] = d;
    if (!f.ok || sc->skip) continue;
    const double2 im[3] = {cmul(sc->wi, d), d, cmul(sc->w, d)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const long long vr = round_fixed(im[k].x, f.fd), vi = round_fixed(im[k].y, f.fd);
      Df[((((int64_t)s * 3 + k) * H.n_atoms + a) * 4 + mu) * L + c] =
          make_int4(balanced_hi(vr), balanced_lo(vr), balanced_hi(vi), balanced_lo(vi));
    }
  }
}

// One output of the FP64 formula (the arithmetic of k_apply_zm<double>).
__device__ __noinline__ double2 output_fp64(const HamView *H, const double2 *Xc, int L, int ix, int iy, int iz,
                                            double2 w, double2 wi, double E, const double2 *Dc) {
  const int nx = H->nx, ny = H->ny, nz = H->nz, nxy = nx * ny;
  const int pt = (iz * ny + iy) * nx + ix;
  const double2 x0 = Xc[(int64_t)pt * L];
  const double dd = (E - H->diag_kin) - H->vloc[pt];
  double2 acc = make_double2(dd * x0.x, dd * x0.y);
  for (int k = 1; k <= H->m; ++k) {
    const int xp = (ix + k) % nx, xm = (ix - k % nx + nx) % nx, yp = (iy + k) % ny, ym = (iy - k % ny + ny) % ny;
    const double2 a1 = Xc[(int64_t)(pt - ix + xp) * L], a2 = Xc[(int64_t)(pt - ix + xm) * L];
    const double2 b1 = Xc[(int64_t)(pt + (yp - iy) * nx) * L], b2 = Xc[(int64_t)(pt + (ym - iy) * nx) * L];
    const int up = iz + k, dn = iz - k;
    double2 z1 = Xc[(int64_t)(pt + (k - (up >= nz ? nz : 0)) * nxy) * L];
    double2 z2 = Xc[(int64_t)(pt + ((dn < 0 ? nz : 0) - k) * nxy) * L];
    if (up >= nz) z1 = cmul(w, z1);
    if (dn < 0) z2 = cmul(wi, z2);
    acc.x = fma(-H->wx[k], a1.x + a2.x, acc.x);
    acc.y = fma(-H->wx[k], a1.y + a2.y, acc.y);
    acc.x = fma(-H->wy[k], b1.x + b2.x, acc.x);
    acc.y = fma(-H->wy[k], b1.y + b2.y, acc.y);
    acc.x = fma(-H->wz[k], z1.x + z2.x, acc.x);
    acc.y = fma(-H->wz[k], z1.y + z2.y, acc.y);
  }
  if (Dc)
    for (int64_t q = H->pt_ptr[pt]; q < H->pt_ptr[pt + 1]; ++q) {
      const int2 aw = H->pt_aw[q];
      const int64_t t = H->pt_ent[q];
      const double2 *Da = Dc + (int64_t)aw.x * L * 4;
      double2 v = make_double2(0, 0);
      for (int mu = 0; mu < H->n_proj; ++mu) {
        const double p = H->sup_val[t * H->n_proj + mu];
        v.x = fma(p, Da[mu].x, v.x);
        v.y = fma(p, Da[mu].y, v.y);
      }
      if (aw.y) v = cmul(aw.y > 0 ? w : wi, v);
      acc = csub(acc, v);
    }
  return acc;
}

// A block's share of a group of columns that takes the FP64 formula throughout: the blocks of the
// group's columns split the lines of their tile, columns innermost (the march of
// k_apply_zm<double>, at FP64 issue: 2.35 ms on 32 systems of the 32x32x16 cell, L = 32).
template <int MH, int CG, int TX, int TY>
__device__ __noinline__ void tile_fp64(const HamView &H, int L, int groups, int tiles_x, int z_chunk, const double2 *X,
                                       double2 *Y, const double *E, const ColumnScale *scales, const double2 *D) {
  const int nx = H.nx, ny = H.ny, nz = H.nz, nxy = nx * ny;
  const int s = blockIdx.z, g = blockIdx.x % groups, tb = blockIdx.x / groups;
  const int bx = (tb % tiles_x) * TX, by = (tb / tiles_x) * TY;
  const int z0 = blockIdx.y * z_chunk, z1 = min(nz, z0 + z_chunk);
  const double2 *Xs = X + (int64_t)s * H.n * L;
  double2 *Ys = Y + (int64_t)s * H.n * L;
  scales += (int64_t)s * L;
  D += (int64_t)s * H.n_atoms * L * 4;
  const int c0 = g * CG / kFixRoute * kFixRoute, cols = min(kFixRoute, L - c0);
  const int blocks = (cols + CG - 1) / CG, per = CG * TX * TY / cols;
  const int tid = threadIdx.x, c = c0 + tid % cols;
  if (tid >= per * cols) return;
  const double2 w = scales[c].w, wi = scales[c].wi;
  const double ed = E[s] - H.diag_kin;
  for (int ln = tid / cols + per * (g - c0 / CG); ln < TX * TY; ln += per * blocks) {
    const int ix = bx + ln % TX, iy = by + ln / TX;
    if (ix >= nx || iy >= ny) continue;
    const int line = iy * nx + ix;
    auto fold = [](int j, int n) {
      while (j >= n) j -= n;
      while (j < 0) j += n;
      return j;
    };
    int ox_p[MH + 1], ox_m[MH + 1], oy_p[MH + 1], oy_m[MH + 1];
#pragma unroll
    for (int k = 1; k <= MH; ++k) {
      ox_p[k] = (fold(ix + k, nx) - ix) * L;
      ox_m[k] = (fold(ix - k, nx) - ix) * L;
      oy_p[k] = (fold(iy + k, ny) - iy) * nx * L;
      oy_m[k] = (fold(iy - k, ny) - iy) * nx * L;
    }
    auto bloch = [&](int p) -> double2 {
      if (p >= nz) return cmul(w, Xs[((p - nz) * nxy + line) * L + c]);
      if (p < 0) return cmul(wi, Xs[((p + nz) * nxy + line) * L + c]);
      return Xs[(p * nxy + line) * L + c];
    };
    double2 q[2 * MH + 1];
#pragma unroll
    for (int d = 0; d < 2 * MH; ++d) q[d] = bloch(z0 + d - MH);
    for (int iz = z0; iz < z1; ++iz) {
      const int pt = iz * nxy + line, b = pt * L + c;
      int e0 = 0, e1 = 0;
      if (H.n_atoms) { e0 = (int)H.pt_ptr[pt]; e1 = (int)H.pt_ptr[pt + 1]; }
      q[2 * MH] = bloch(iz + MH);
      const double2 x0 = q[MH];
      const double dd = ed - H.vloc[pt];
      double2 acc = make_double2(dd * x0.x, dd * x0.y);
#pragma unroll
      for (int k = 1; k <= MH; ++k) {
        const double2 a1 = Xs[b + ox_p[k]], a2 = Xs[b + ox_m[k]], b1 = Xs[b + oy_p[k]], b2 = Xs[b + oy_m[k]];
        const double2 z1 = q[MH + k], z2 = q[MH - k];
        acc.x = fma(-H.wx[k], a1.x + a2.x, acc.x);
        acc.y = fma(-H.wx[k], a1.y + a2.y, acc.y);
        acc.x = fma(-H.wy[k], b1.x + b2.x, acc.x);
        acc.y = fma(-H.wy[k], b1.y + b2.y, acc.y);
        acc.x = fma(-H.wz[k], z1.x + z2.x, acc.x);
        acc.y = fma(-H.wz[k], z1.y + z2.y, acc.y);
      }
      for (int e = e0; e < e1; ++e) {
        const int2 aw = H.pt_aw[e];
        const double *p = H.sup_val + (int64_t)H.pt_ent[e] * H.n_proj;
        const double2 *Da = D + ((int64_t)aw.x * L + c) * 4;
        if (aw.y == 0) {
          for (int mu = 0; mu < H.n_proj; ++mu) {
            const double2 d = Da[mu];
            acc.x = fma(-p[mu], d.x, acc.x);
            acc.y = fma(-p[mu], d.y, acc.y);
          }
        } else {
          double2 v = make_double2(0, 0);
          for (int mu = 0; mu < H.n_proj; ++mu) {
            const double2 d = Da[mu];
            v.x = fma(p[mu], d.x, v.x);
            v.y = fma(p[mu], d.y, v.y);
          }
          const double2 t = aw.y > 0 ? w : wi;
          acc = cfma(make_double2(-t.x, -t.y), v, acc);
        }
      }
      Ys[b] = acc;
#pragma unroll
      for (int d = 0; d < 2 * MH; ++d) q[d] = q[d + 1];
    }
  }
}

struct Fixed2 { long long re, im; };

// sum_k +-n_k s_k as two words: even k enter negative (the signs of c_k alternate).  The sums s_k stay
// below 2^63 by the choice of Q, and sum_k n_k below 2^(fx_st - 1), so shifted(fx_st) stays below 2^62:
// what Product::add, which cuts its factor at 31 bits, can hold.
struct WeightedSum {
  long long hi = 0;
  unsigned long long plus = 0, minus = 0;
  __device__ __forceinline__ void add(int k, int nk, long long s) {
    const int s1 = opaque((int)(s >> 32));
    const unsigned s0 = (unsigned)opaque((int)s);
    if (k & 1) {
      madw(hi, s1, nk);
      madwu(plus, s0, nk);
    } else {
      madw(hi, s1, -nk);
      madwu(minus, s0, nk);
    }
  }
  __device__ __forceinline__ long long shifted(int st) const {   // the sum >> st
    const long long lo = (long long)(plus - minus);
    const long long h = hi + (lo >> 32);
    return (h << (32 - st)) | (long long)((unsigned)lo >> st);
  }
};

// The products x * g in words of 31 bits: A 2^62 + B 2^31 + C
struct Product {
  long long A = 0, B = 0;
  unsigned long long C = 0;
  __device__ __forceinline__ void add(long long x, int g1, int g0) {
    const int x1 = hi31(x), x0 = lo31(x);
    madw(A, x1, g1);
    madw(B, x1, g0);
    madw(B, x0, g1);
    madwu(C, x0, g0);
  }
  __device__ __forceinline__ long long shifted(int sa) const {   // >> (62 - sa)
    return (A << sa) + ((B + (long long)(C >> 31)) >> (31 - sa));
  }
};

// Projector products in balanced words of 29 bits: A 2^58 + B 2^29 (the product of the low
// words, of zero mean and below 2^-57 of the largest, is left out).  One entry (4 projectors)
// adds less than 2^58.6 to |B|: 16 entries between carries.
struct Scatter {
  long long A = 0, B = 0;
  __device__ __forceinline__ void add(int d1, int d0, int p1, int p0) {
    madw(A, d1, p1);
    madw(B, d1, p0);
    madw(B, d0, p1);
  }
  __device__ __forceinline__ void carry() {
    A += B >> 29;
    B &= 0x1fffffff;
  }
  __device__ __forceinline__ long long shifted(int sp) const {   // >> (58 - sp)
    return (A << sp) + (B >> (29 - sp));
  }
};

// Stencil and projector scatter: 677 us on 32 systems of the 32x32x16 cell (L = 32, 16.8 M
// outputs), of which the stencil is 360; k_apply_zm<double>, at FP64 issue, 2400 us.  About 480
// instructions per output for the stencil and 110 per covering entry; they issue on 48 per cent of
// the cycles, bound by the latency of dependent products, shared-memory reads and the scatter's loads
// and by the barriers (16 warps per SM at 128 registers, of which the z queue takes 36; the widest
// stencils, of half-width 5 and 6, spill 30 to 270 bytes per thread).
// 8 x 8 x 4 tiles of 256 threads beat 16 x 8 x 4 of 512 (two blocks per SM
// cover each other's barriers) and 8 x 4 x 8; the columns are cut in fours because the halo,
// converted once per tile, shrinks with the tile's x-y extent.  A block covers TX x TY lines of CG
// columns and walks the planes z0 .. z1-1; the plane it is on lies in shared memory with its x-y
// halo, as fixed-point pairs (two buffers, one barrier per plane), and each thread keeps the
// 2 MH + 1 z neighbours of its point in registers.  The next plane's halo and the plane MH ahead
// are loaded while the current one is computed.  Offsets inside a plane are 32-bit byte offsets
// from a base that all threads share.  PARTS: the real and the imaginary parts to the FP64 kernels'
// accuracy; else the moduli, as BiCG's iterations and its residual check apply it (with (p~, q) over
// the first dot.n systems).
template <int MH, int CG, int TX, int TY, bool ISO, bool PARTS>
__global__ void __launch_bounds__(CG *TX *TY, 512 / (CG * TX * TY))
    k_stencil_fixed(const __grid_constant__ HamView H, int L, int groups, int tiles_x, int z_chunk,
                    const double2 *__restrict__ X, double2 *__restrict__ Y, const double *__restrict__ E,
                    const ColumnScale *__restrict__ scales,
                    const double2 *__restrict__ D, const int4 *__restrict__ Df,
                    const int *__restrict__ sys_active, const FixedDot dot) {
  constexpr int WX = TX + 2 * MH, WY = TY + 2 * MH, THREADS = CG * TX * TY;
  constexpr int HALO = 2 * MH * (TX + TY) * CG;
  constexpr int SLOTS = (HALO + THREADS - 1) / THREADS;
  constexpr int PLANE = WX * WY * CG;
  extern __shared__ Fixed2 tile[];   // [2][WY][WX][CG]
  const int s = blockIdx.z;
  if (sys_active && !sys_active[s]) return;
  const int nx = H.nx, ny = H.ny, nz = H.nz;
  const int g = blockIdx.x % groups, tb = blockIdx.x / groups;
  if (PARTS && scales[(int64_t)s * L + g * CG].skip) {   // the same for the columns of the block
    tile_fp64<MH, CG, TX, TY>(H, L, groups, tiles_x, z_chunk, X, Y, E, scales, D);
    return;
  }
  const int bx = (tb % tiles_x) * TX, by = (tb / tiles_x) * TY;
  const int z0 = blockIdx.y * z_chunk, z1 = min(nz, z0 + z_chunk);
  const int tid = threadIdx.x;
  const int cl = tid % CG, lx = (tid / CG) % TX, ly = tid / (CG * TX);
  const int c = min(g * CG + cl, L - 1);
  const int ix = (bx + lx) % nx, iy = (by + ly) % ny;
  const int line = iy * nx + ix;
  const int64_t plane_bytes = (int64_t)nx * ny * L * sizeof(double2);
  const char *Xs = (const char *)(X + (int64_t)s * H.n * L);
  char *Ys = (char *)(Y + (int64_t)s * H.n * L);
  const unsigned mine = (unsigned)(line * L + c) * (unsigned)sizeof(double2);
  auto load = [&](int p, unsigned off) -> double2 { return *(const double2 *)(Xs + p * plane_bytes + off); };

  const ColumnScale *sc = scales + (int64_t)s * L + c;
  const FixScale f = sc->f;
  const int base = sc->base;
  const bool own = g * CG + cl < L && bx + lx < nx && by + ly < ny && !sc->skip;
  // (p~, q): this thread's share, for primal systems
  const bool dotted = !PARTS && s < dot.n;
  const char *Xd = Xs + (!PARTS ? (int64_t)dot.n * H.n * L * (int64_t)sizeof(double2) : 0);
  double dx = 0, dy = 0;
  auto add_dot = [&](double2 pd, double2 q) {
    dx = fma(pd.x, q.x, fma(pd.y, q.y, dx));
    dy = fma(pd.x, q.y, fma(-pd.y, q.x, dy));
  };
  const double2 w0 = sc->w, wi0 = sc->wi;
  // In the widest stencils the twist is read again where it is used (the last planes, the FP64
  // formula): kept, it would hold 8 registers through the march (13x10x6 cell, order 12, with the
  // neighbours of the test below: 21.4 -> 19.4 us; at order 8 the loads cost more, 677 -> 687).
  auto twist = [&](bool inverse) -> double2 {
    if constexpr (MH > 4) {
      const ColumnScale *t = sc;
      asm volatile("" : "+l"(t));
      return inverse ? t->wi : t->w;
    }
    return inverse ? wi0 : w0;
  };
  const long long ef = sc->ef;
  auto conv = [&](double2 v) -> Fixed2 { return Fixed2{to_fixed(v.x, base), to_fixed(v.y, base)}; };
  // this thread's value in plane p of the Bloch-extended field, -nz <= p < 2 nz
  auto raw = [&](int p) -> double2 { return load(p >= nz ? p - nz : (p < 0 ? p + nz : p), mine); };
  // halo elements tid, tid + THREADS, ...: 2 MH rows of TX, then 2 MH columns of TY (THREADS is
  // a multiple of CG, so an element's column is its thread's own)
  unsigned hoff[SLOTS];
  int hat[SLOTS];
#pragma unroll
  for (int k = 0; k < SLOTS; ++k) {
    const int h = tid + k * THREADS;
    const int hp = min(h, HALO - CG + cl) / CG;
    int px, py;
    if (hp < 2 * MH * TX) {
      const int r = hp / TX;
      px = hp % TX + MH;
      py = r < MH ? r : r + TY;
    } else {
      const int r = (hp - 2 * MH * TX) / TY;
      py = (hp - 2 * MH * TX) % TY + MH;
      px = r < MH ? r : r + TX;
    }
    int gx = (bx + px - MH) % nx, gy = (by + py - MH) % ny;
    if (gx < 0) gx += nx;
    if (gy < 0) gy += ny;
    hoff[k] = (unsigned)((gy * nx + gx) * L + c) * (unsigned)sizeof(double2);
    hat[k] = (py * WX + px) * CG + cl;
  }
  const int self = ((ly + MH) * WX + lx + MH) * CG + cl;

  Fixed2 q[2 * MH + 1];
#pragma unroll
  for (int d = 0; d < 2 * MH; ++d) {
    double2 v = raw(z0 + d - MH);
    if (d < MH && z0 < MH) {
      const double2 t = cmul(wi0, v);
      if (z0 + d - MH < 0) v = t;
    }
    if (d > MH && z0 + MH > nz) {
      const double2 t = cmul(w0, v);
      if (z0 + d - MH >= nz) v = t;
    }
    q[d] = conv(v);
  }
  double2 head = raw(z0 + MH);
  tile[self] = q[MH];
#pragma unroll
  for (int k = 0; k < SLOTS; ++k) tile[hat[k]] = conv(load(z0, hoff[k]));
  const bool proj = H.n_atoms > 0;
  const char *Ds = (const char *)(Df + (int64_t)s * 3 * H.n_atoms * L * 4);
  const unsigned d_mu = (unsigned)L * (unsigned)sizeof(int4), d_mine = (unsigned)c * (unsigned)sizeof(int4);
  // the line's tables: entry ranges and V_loc of its planes, one after the other
  const int *ptr = H.fx_ptr + (int64_t)line * (nz + 1) + z0;
  const long long *vl = H.fx_v + (int64_t)line * nz + z0;
  int e0 = 0, e1 = proj ? ptr[0] : 0, e2 = proj ? ptr[1] : 0;
  // the first entry not yet used (the tables have one spare entry at the end)
  int img = 0;
  int4 np01 = make_int4(0, 0, 0, 0), np23 = np01;
  if (proj) {
    img = H.fx_img[e1];
    np01 = H.fx_p[2 * e1];
    np23 = H.fx_p[2 * e1 + 1];
  }
  long long vnext = vl[0];
  unsigned long long redo = 0;   // planes whose output is left to the FP64 formula
  // one plane; `twisted`: the plane MH ahead lies in the next cell
  auto plane = [&](int iz, auto twisted) {
    const Fixed2 *mid = tile + ((iz - z0) & 1) * PLANE + self;
    Fixed2 *next = tile + ((iz - z0 + 1) & 1) * PLANE;
    const bool more = iz + 1 < z1;
    e0 = e1;
    e1 = e2;
    const long long dd = ef - vnext;
    q[2 * MH] = conv(twisted ? cmul(twist(false), head) : head);
    double2 hv[SLOTS];
    if (more) {
      head = raw(iz + 1 + MH);
#pragma unroll
      for (int k = 0; k < SLOTS; ++k) hv[k] = load(iz + 1, hoff[k]);
      if (proj) e2 = ptr[iz - z0 + 2];
      vnext = vl[iz - z0 + 1];
    }
    __syncthreads();
    const Fixed2 x0 = q[MH];
    if (!PARTS && max(absword(x0.re), absword(x0.im)) < kFixSmallWord) {
      // small at the point: its nearest neighbours decide (the moduli, since BiCG mixes the parts: its
      // updates round each against the larger one)
      const Fixed2 n[6] = {mid[CG], mid[-CG], mid[WX * CG], mid[-WX * CG], q[MH + 1], q[MH - 1]};
      int m = 0;
#pragma unroll
      for (int k = 0; k < 6; ++k) m = max(m, max(absword(n[k].re), absword(n[k].im)));
      if (m < kFixSmallWord) redo |= 1ull << (iz - z0);
    }
    Product yr, yi;
    {
      const int d1 = hi31(dd), d0 = lo31(dd);
      yr.add(x0.re, d1, d0);
      yi.add(x0.im, d1, d0);
    }
    int near_re = 0, near_im = 0;   // high words of the sums over the nearest neighbours
    if (ISO) {
      WeightedSum tr, ti;
#pragma unroll
      for (int k = 1; k <= MH; ++k) {
        const Fixed2 a1 = mid[k * CG], a2 = mid[-k * CG], b1 = mid[k * WX * CG], b2 = mid[-k * WX * CG];
        const long long sr = (a1.re + a2.re + b1.re) + (b2.re + q[MH + k].re + q[MH - k].re);
        const long long si = (a1.im + a2.im + b1.im) + (b2.im + q[MH + k].im + q[MH - k].im);
        if (k == 1) { near_re = (int)(sr >> 32); near_im = (int)(si >> 32); }
        tr.add(k, H.fx_nk[k], sr);
        ti.add(k, H.fx_nk[k], si);
      }
      yr.add(tr.shifted(H.fx_st), H.fx_c1[0], H.fx_c0[0]);
      yi.add(ti.shifted(H.fx_st), H.fx_c1[0], H.fx_c0[0]);
    } else {
#pragma unroll
      for (int dir = 0; dir < 3; ++dir) {
        WeightedSum tr, ti;
#pragma unroll
        for (int k = 1; k <= MH; ++k) {
          const Fixed2 a = dir == 0 ? mid[k * CG] : dir == 1 ? mid[k * WX * CG] : q[MH + k];
          const Fixed2 b = dir == 0 ? mid[-k * CG] : dir == 1 ? mid[-k * WX * CG] : q[MH - k];
          if (k == 1) { near_re += (int)((a.re + b.re) >> 32); near_im += (int)((a.im + b.im) >> 32); }
          tr.add(k, H.fx_nk[k], a.re + b.re);
          ti.add(k, H.fx_nk[k], a.im + b.im);
        }
        yr.add(tr.shifted(H.fx_st), H.fx_c1[dir], H.fx_c0[dir]);
        yi.add(ti.shifted(H.fx_st), H.fx_c1[dir], H.fx_c0[dir]);
      }
    }
    if (PARTS && ((within((int)(x0.re >> 32), kFixSmallWord) && within(near_re, 8 * kFixSmallWord)) ||
                  (within((int)(x0.im >> 32), kFixSmallWord) && within(near_im, 8 * kFixSmallWord)))) {
      // a part that is small at the point, and may be at its nearest neighbours: their sum, which
      // is at hand, is then below 6 times the limit (seldom otherwise)
      const Fixed2 *at = mid;
      if constexpr (MH > 4) asm volatile("" : "+l"(at));   // read again, as the twist
      const Fixed2 n[6] = {at[CG], at[-CG], at[WX * CG], at[-WX * CG], q[MH + 1], q[MH - 1]};
      int mr = absword(x0.re), mi = absword(x0.im);
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        mr = max(mr, absword(n[k].re));
        mi = max(mi, absword(n[k].im));
      }
      if (min(mr, mi) < kFixSmallWord) redo |= 1ull << (iz - z0);
    }
    long long vr = yr.shifted(f.sa), vi = yi.shifted(f.sa);
    if (e0 < e1) {
      Scatter pr, pi;
      int e = e0;
      while (true) {
        const int stop = min(e1, e + 16);
#pragma unroll 1
        for (; e < stop; ++e) {
          const char *Da = Ds + ((unsigned)img * 4 * d_mu + d_mine);
          const int4 da = *(const int4 *)Da, db = *(const int4 *)(Da + d_mu), dc = *(const int4 *)(Da + 2 * d_mu),
                     de = *(const int4 *)(Da + 3 * d_mu);
          const int4 p01 = np01, p23 = np23;
          // the next entry (of this plane or of the next one with entries)
          np01 = H.fx_p[2 * (e + 1)];
          np23 = H.fx_p[2 * (e + 1) + 1];
          img = H.fx_img[e + 1];
          pr.add(da.x, da.y, p01.x, p01.y);
          pi.add(da.z, da.w, p01.x, p01.y);
          pr.add(db.x, db.y, p01.z, p01.w);
          pi.add(db.z, db.w, p01.z, p01.w);
          pr.add(dc.x, dc.y, p23.x, p23.y);
          pi.add(dc.z, dc.w, p23.x, p23.y);
          pr.add(de.x, de.y, p23.z, p23.w);
          pi.add(de.z, de.w, p23.z, p23.w);
        }
        if (e == e1) break;
        pr.carry();
        pi.carry();
      }
      vr -= pr.shifted(f.sp);
      vi -= pi.shifted(f.sp);
    }
    if (own) {
      const double2 out = make_double2(from_fixed(vr, f.uy), from_fixed(vi, f.uy));
      *(double2 *)(Ys + iz * plane_bytes + mine) = out;
      if (dotted && f.ok && !((redo >> (iz - z0)) & 1)) add_dot(*(const double2 *)(Xd + iz * plane_bytes + mine), out);
    }
#pragma unroll
    for (int d = 0; d < 2 * MH; ++d) q[d] = q[d + 1];
    if (more) {
      next[self] = q[MH];
#pragma unroll
      for (int k = 0; k < SLOTS; ++k) next[hat[k]] = conv(hv[k]);
    }
  };
  int iz = z0;
  for (; iz < min(z1, nz - MH); ++iz) plane(iz, std::false_type());
  for (; iz < z1; ++iz) plane(iz, std::true_type());
  if (!f.ok) redo = ~0ull;
  if (own && redo)
    for (iz = z0; iz < z1; ++iz)
      if ((redo >> (iz - z0)) & 1) {
        const double2 out = output_fp64(&H, (const double2 *)Xs + c, L, ix, iy, iz, twist(false), twist(true), E[s],
                                        proj ? D + ((int64_t)s * H.n_atoms * L + c) * 4 : nullptr);
        *(double2 *)(Ys + iz * plane_bytes + mine) = out;
        if (dotted) add_dot(*(const double2 *)(Xd + iz * plane_bytes + mine), out);
      }
  if (dotted) {
    // the block's sum per column, lines in order of the shuffles: fixed for a given grid
    double *red = (double *)tile;   // [warps][CG][2]
    for (int o = CG; o < 32; o <<= 1) {
      dx += __shfl_xor_sync(0xffffffffu, dx, o);
      dy += __shfl_xor_sync(0xffffffffu, dy, o);
    }
    __syncthreads();
    if (tid % 32 < CG) {
      red[(tid / 32 * CG + cl) * 2] = dx;
      red[(tid / 32 * CG + cl) * 2 + 1] = dy;
    }
    __syncthreads();
    const int tiles = gridDim.x / groups, parts = tiles * gridDim.y;
    if (tid < CG && g * CG + tid < L) {
      for (int k = 1; k < THREADS / 32; ++k) {
        dx += red[(k * CG + tid) * 2];
        dy += red[(k * CG + tid) * 2 + 1];
      }
      double *o = dot.part + (((int64_t)s * parts + blockIdx.y * tiles + tb) * L + g * CG + tid) * 2;
      o[0] = dx;
      o[1] = dy;
    }
    if (last_block(dot.tail.count + s, gridDim.x * gridDim.y))
      alpha_tail<2>(dot.tail, dot.part, s, L, parts, tid, THREADS, (double *)tile);
  }
}

size_t apply_coef_bytes(const HamView &H, int n_sys, int L, int dtype) {
  const size_t csz = dtype == CBS_C128 ? sizeof(double2) : sizeof(float2);
  return (size_t)n_sys * (H.n_atoms ? H.n_atoms : 1) * H.np4 * L * csz;
}

// points per chunk of k_column_max: enough chunks to fill the GPU, at most 64 per system
static int max_chunks(const HamView &H, int n_sys, int L, int64_t *pts) {
  const int py = (int)col_block(L).y;
  int64_t p = std::max<int64_t>((int64_t)py * 16, ceil_div(H.n, 64));
  while (ceil_div(H.n, p) * (int64_t)n_sys > 152 * 16 && p < (int64_t)py * 256) p *= 2;
  *pts = p;
  return ceil_div(H.n, p);
}

size_t apply_ws_bytes(const HamView &H, int n_sys, int L, int dtype) {
  const size_t d = apply_coef_bytes(H, n_sys, L, dtype);
  if (dtype != CBS_C128 || !H.fx_ok || L < 1) return d;
  int64_t pts;
  const size_t cols = (size_t)n_sys * L;
  return (H.n_atoms ? 4 * d : 0) + cols * sizeof(ColumnScale) +
         cols * max_chunks(H, n_sys, L, &pts) * sizeof(unsigned) + 256;
}

bool fixed_serves(const HamView &H, int n_sys, int L, size_t ws_bytes) {
  // offsets inside a system's block and inside its coefficients are 32-bit byte offsets
  return H.fx_ok && L <= 256 && H.n * L < ((int64_t)1 << 28) &&
         (int64_t)3 * H.n_atoms * L < ((int64_t)1 << 26) && ws_bytes >= apply_ws_bytes(H, n_sys, L, CBS_C128);
}

ColumnScale *fixed_scales(const HamView &H, int n_sys, int L, void *ws) {
  return (ColumnScale *)((char *)ws + (H.n_atoms ? 4 * apply_coef_bytes(H, n_sys, L, CBS_C128) : 0));
}

// 8 x 8 lines of 4 columns (64-byte pieces of a point's row)
constexpr int kFixCG = 4, kFixTX = 8, kFixTY = 8;
struct FixGrid { int groups, tiles_x, tiles, z_chunk, z_blocks; };
static FixGrid fix_grid(const HamView &H, int n_sys, int L) {
  FixGrid g;
  g.groups = ceil_div(L, kFixCG);
  g.tiles_x = ceil_div(H.nx, kFixTX);
  g.tiles = g.tiles_x * ceil_div(H.ny, kFixTY);
  // planes per block: all of them unless that leaves SMs idle
  int zc = 1;
  while (zc < 8 && (int64_t)g.groups * g.tiles * n_sys * zc < 152 && H.nz / (zc * 2) >= 2) zc *= 2;
  g.z_chunk = std::min(64, ceil_div(H.nz, zc));   // a block marks its planes in 64 bits
  g.z_blocks = ceil_div(H.nz, g.z_chunk);
  return g;
}

// Fixed point takes three launches without projectors, the FP64 stencil one, and its tiles of 8 x 8
// lines and 4 columns are padded where the cell or the block is narrower.  The times of both in
// microseconds, fitted to 900 cells without projectors (4..96 x 4..96 x 4..32, orders 2..12, 1..64
// columns and systems, up to 4 M outputs; 9 and 5 per cent off in the mean).  The FP64 march is
// bound by the latency of a line, in rounds of the blocks that the SMs hold (by registers), or by the
// FP64 issue of the fullest SM; fixed point by its rounds of two blocks per SM.  A microsecond on top
// is the host's for two more launches.  The choice was 0.6 per cent from the better of the two in
// the mean, one of the 900 more than a twentieth slower than the FP64 stencil (62x9x16, order 2,
// one column of 14 systems: 16.5 against 34 us; 8x8x4, order 4, 16 columns: 10 against 17; but
// 47x14x6, order 8, 14 columns: 35 against 23).
bool fp64_quicker(const HamView &H, int n_sys, int L) {
  const double outputs = (double)n_sys * H.n * L;
  if (H.n_atoms || outputs > 4e6) return false;
  static const int resident[kMaxHalf + 1] = {0, 5, 4, 3, 2, 2, 2};   // blocks of the FP64 stencil per SM
  const int lines = std::max(1, 256 / L), across = ceil_div(H.nx, lines);
  const double blocks64 = (double)across * H.ny * n_sys;
  const int widest = ceil_div((int64_t)std::min(H.nx, lines) * L, 32);   // warps of the fullest block
  const int last = ceil_div((int64_t)(H.nx - (across - 1) * lines) * L, 32);
  const double mean = across > 1 ? (double)((across - 1) * widest + last) / across : widest;
  const double latency = H.nz * (0.033 + 0.542 * H.m) * std::max(1.0, blocks64 / (152 * resident[H.m]));
  const double warps = std::max(ceil(blocks64 / 152) * mean, blocks64 <= 152 ? (double)widest : 0.0);
  const double fp64 = 4.85 + std::max(latency, warps * H.nz * (2 + 12 * H.m) * 0.0124);
  const FixGrid g = fix_grid(H, n_sys, L);
  const int64_t blocks = (int64_t)g.groups * g.tiles * g.z_blocks * n_sys, rest = blocks % 304;
  const double rounds = 1.64 * (double)(blocks / 304) + (rest == 0 ? 0.0 : rest <= 152 ? 1.0 : 1.64);
  const double fixed = 10.8 + (g.z_chunk + 2.5) * (0.21 + 0.2 * H.m) * rounds + 7.3e-6 * outputs;
  return fp64 < fixed + 1;
}

int fixed_dot_parts(const HamView &H, int n_sys, int L) {
  const FixGrid g = fix_grid(H, n_sys, L);
  return g.tiles * g.z_blocks;
}

cbs_status apply_fixed_scaled(const HamView &H, int n_sys, int L, const double2 *X, double2 *Y, const double *E,
                              void *ws, const int *sys_active, cudaStream_t st, bool parts, const FixedDot *dot) {
  double2 *D = (double2 *)ws;
  int4 *Df = (int4 *)((char *)ws + (H.n_atoms ? apply_coef_bytes(H, n_sys, L, CBS_C128) : 0));
  const ColumnScale *scales = fixed_scales(H, n_sys, L, ws);
  if (H.n_atoms) {
    const int groups = ceil_div(L, 32), cg = ceil_div(L, groups);
    const int py = 256 / cg > 32 ? 32 : 256 / cg;
    const dim3 blk((unsigned)cg, (unsigned)py, 1), grd((unsigned)H.n_atoms, (unsigned)n_sys, (unsigned)groups);
    const size_t sm = (size_t)py * 16 * cg * sizeof(long long) + 4 * cg * sizeof(double2) + 2 * cg * sizeof(int);
    if (parts) k_gather_fixed<true><<<grd, blk, sm, st>>>(H, L, X, scales, D, Df, sys_active);
    else k_gather_fixed<false><<<grd, blk, sm, st>>>(H, L, X, scales, D, Df, sys_active);
    count_launches(1);
    CBS_CUDA(cudaGetLastError());
  }
  const FixGrid g = fix_grid(H, n_sys, L);
  const dim3 grd((unsigned)(g.groups * g.tiles), (unsigned)g.z_blocks, (unsigned)n_sys);
  const size_t sm = (size_t)2 * (kFixTX + 2 * H.m) * (kFixTY + 2 * H.m) * kFixCG * sizeof(Fixed2);
  const FixedDot d = dot ? *dot : FixedDot();
#define FK(MH, ISO, PARTS)                                                                                 \
  do {                                                                                                     \
    if (sm > 48 * 1024)                                                                                    \
      CBS_CUDA(cudaFuncSetAttribute(k_stencil_fixed<MH, kFixCG, kFixTX, kFixTY, ISO, PARTS>,               \
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));                \
    k_stencil_fixed<MH, kFixCG, kFixTX, kFixTY, ISO, PARTS><<<grd, kFixCG * kFixTX * kFixTY, sm, st>>>(    \
        H, L, g.groups, g.tiles_x, g.z_chunk, X, Y, E, scales, D, Df, sys_active, d);                      \
  } while (0)
#define FM(MH)                        \
  case MH:                            \
    if (H.fx_iso) {                   \
      if (parts) FK(MH, true, true);  \
      else FK(MH, true, false);       \
    } else {                          \
      if (parts) FK(MH, false, true); \
      else FK(MH, false, false);      \
    }                                 \
    break
  switch (H.m) {
    FM(1); FM(2); FM(3); FM(4); FM(5); FM(6);
    default: set_error("apply: FD half-width must be 1..6"); return CBS_EINVAL;
  }
#undef FM
#undef FK
  count_launches(1);
  CBS_CUDA(cudaGetLastError());
  return CBS_OK;
}

cbs_status apply_fixed(const HamView &H, int n_sys, int L, const double2 *X, double2 *Y,
                       const double2 *twist, bool per_col, const double *E, void *ws,
                       const int *sys_active, cudaStream_t st, bool parts) {
  ColumnScale *scales = fixed_scales(H, n_sys, L, ws);
  unsigned *maxhi = (unsigned *)(scales + (size_t)n_sys * L);
  int64_t pts;
  const int chunks = max_chunks(H, n_sys, L, &pts);
  const dim3 blk = col_block(L);
  k_column_max<<<dim3((unsigned)chunks, (unsigned)n_sys, 1), blk, (size_t)blk.x * blk.y * sizeof(unsigned), st>>>(
      H.n, L, (int)pts, X, maxhi, sys_active);
  const dim3 sblk((unsigned)L, (unsigned)std::min(kFixSamples, 1024 / L), 1);
  k_fix_scales<<<n_sys, sblk, (size_t)(sblk.y + 2) * L * sizeof(unsigned), st>>>(H, L, chunks, maxhi, X, twist, per_col ? 1 : 0,
                                                                               E, scales, sys_active, parts);
  count_launches(2);
  CBS_CUDA(cudaGetLastError());
  return apply_fixed_scaled(H, n_sys, L, X, Y, E, ws, sys_active, st, parts, nullptr);
}

}  // namespace cbs
