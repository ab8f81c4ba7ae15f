// Cell Hamiltonian set-up (the layout step of the path): FD weights, local potential,
// the projector table and its transpose, and the exact Frobenius norms of H+, H- and the
// pieces of ||H0 - E||_F used by the residual check.
//
// Paper §2, Eq. (2): the cell block H0 = H_{n,n} and the couplings H+ = H_{n,n+1},
// H- = H_{n,n-1} = H+^T of a real-space Hamiltonian (-1/2 FD Laplacian + V_loc +
// separable projectors); §4 uses a nine-point (order 8) central FD Laplacian.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <vector>

#include "fixed.cuh"

namespace cbs {

// Central second-derivative weights of order 2m, closed form:
// c_k = 2 (-1)^{k+1} (m!)^2 / (k^2 (m-k)! (m+k)!),  c_0 = -2 sum_k c_k.
static void fd_weights(int order, double *c) {
  int m = order / 2;
  double s = 0.0;
  for (int k = 1; k <= m; ++k) {
    // (m!)^2 / ((m-k)! (m+k)!) = prod_{j=1..k} (m-k+j)/(m+j)
    double r = 1.0;
    for (int j = 1; j <= k; ++j) r *= (double)(m - k + j) / (double)(m + j);
    c[k] = 2.0 * ((k % 2) ? 1.0 : -1.0) * r / ((double)k * k);
    s += c[k];
  }
  c[0] = -2.0 * s;
}

// ------------------------------------------------------------------ Frobenius norms
// One warp per row i.  The row's entries are the merged FD stencil (block l, column j,
// weight) and, for every atom a covering i (entry s), the values (h_a p_s) . p_t at
// columns i_t of all entries t of a, in block l = m_s - m_t.  Entries that coincide in
// (l, j) are summed before squaring, so the result is the exact Frobenius norm.  The lanes
// share the stencil's entries, then each atom's (one thread per row, walking some 1500 of them
// with its lists in local memory, took 29 ms on the 32x32x16 cell).
constexpr int kMaxCover = 64;
constexpr int kMaxSten = 1 + 6 * kMaxHalf;
constexpr int kFroWarps = 4;

struct FroRow {
  int64_t sc[kMaxSten];
  double sw[kMaxSten];
  double cq[kMaxCover][kMaxProj];
  int sl[kMaxSten], ns;
  int ca[kMaxCover], cm[kMaxCover];
};

__global__ void __launch_bounds__(32 * kFroWarps) k_frobenius(HamView H, double *part, int *err) {
  __shared__ FroRow rows[kFroWarps];
  __shared__ double red[kFroWarps][5];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * kFroWarps + warp;
  FroRow &R = rows[warp];
  double acc[5] = {0, 0, 0, 0, 0};  // off-diag l=0, l=+1, l=-1, diag, diag^2
  if (i < H.n) {
    const int64_t nxy = (int64_t)H.nx * H.ny;
    const int ix = (int)(i % H.nx), iy = (int)((i / H.nx) % H.ny), iz = (int)(i / nxy);
    if (lane == 0) {
      int ns = 0;
      auto add = [&](int l, int64_t col, double w) {
        for (int q = 0; q < ns; ++q)
          if (R.sl[q] == l && R.sc[q] == col) { R.sw[q] += w; return; }
        R.sl[ns] = l; R.sc[ns] = col; R.sw[ns] = w; ++ns;
      };
      add(0, i, H.diag_kin + H.vloc[i]);
      for (int k = 1; k <= H.m; ++k) {
        for (int sg = -1; sg <= 1; sg += 2) {
          int jx = ((ix + sg * k) % H.nx + H.nx) % H.nx;
          add(0, i - ix + jx, H.wx[k]);
          int jy = ((iy + sg * k) % H.ny + H.ny) % H.ny;
          add(0, i + (int64_t)(jy - iy) * H.nx, H.wy[k]);
          int pz = iz + sg * k;
          int l = pz >= H.nz ? 1 : (pz < 0 ? -1 : 0);
          int jz = pz - l * H.nz;
          add(l, i + (int64_t)(jz - iz) * nxy, H.wz[k]);
        }
      }
      R.ns = ns;
    }
    // covering entries of row i
    const int np = H.n_proj;
    int nc = 0;
    if (H.n_atoms) {
      const int64_t e0 = H.pt_ptr[i];
      int64_t e1 = H.pt_ptr[i + 1];
      if (e1 - e0 > kMaxCover) { atomicExch(err, 1); e1 = e0 + kMaxCover; }
      nc = (int)(e1 - e0);
      for (int q = lane; q < nc; q += 32) {
        const int t = H.pt_ent[e0 + q], a = H.pt_atom[e0 + q];
        R.ca[q] = a;
        R.cm[q] = H.sup_wrap[t];
        const double *ha = H.h + (int64_t)a * np * np;
        for (int mu = 0; mu < np; ++mu) {
          double v = 0;
          for (int nu = 0; nu < np; ++nu) v += ha[mu * np + nu] * H.sup_val[(int64_t)t * np + nu];
          R.cq[q][mu] = v;
        }
      }
    }
    __syncwarp();
    const int ns = R.ns;
    // Non-local value at (l, j) from covering entries with index >= from; *earlier is set
    // when a covering entry with index < from also contributes at (l, j).
    auto nl_value = [&](int l, int64_t j, int from, bool *earlier) {
      double v = 0;
      if (earlier) *earlier = false;
      int64_t f0 = H.pt_ptr[j], f1 = H.pt_ptr[j + 1];
      for (int64_t f = f0; f < f1; ++f) {
        int a2 = H.pt_atom[f], u = H.pt_ent[f];
        int mu_w = H.sup_wrap[u];
        for (int q = 0; q < nc; ++q) {
          if (R.ca[q] != a2 || mu_w != R.cm[q] - l) continue;
          if (q < from) { if (earlier) *earlier = true; continue; }
          double dot = 0;
          for (int mu = 0; mu < np; ++mu) dot += R.cq[q][mu] * H.sup_val[(int64_t)u * np + mu];
          v += dot;
        }
      }
      return v;
    };
    for (int q = lane; q < ns; q += 32) {
      double val = R.sw[q] + (nc ? nl_value(R.sl[q], R.sc[q], 0, nullptr) : 0.0);
      if (R.sl[q] == 0 && R.sc[q] == i) { acc[3] += val; acc[4] += val * val; }
      else acc[R.sl[q] == 0 ? 0 : (R.sl[q] == 1 ? 1 : 2)] += val * val;
    }
    for (int q = 0; q < nc; ++q) {
      const int a = R.ca[q];
      for (int64_t t = H.sup_ptr[a] + lane; t < H.sup_ptr[a + 1]; t += 32) {
        const int64_t j = H.sup_idx[t];
        const int l = R.cm[q] - H.sup_wrap[t];
        if (l < -1 || l > 1) { atomicExch(err, 2); continue; }
        bool in_st = false;
        for (int r = 0; r < ns; ++r)
          if (R.sl[r] == l && R.sc[r] == j) { in_st = true; break; }
        if (in_st) continue;
        bool earlier;
        double val = nl_value(l, j, q, &earlier);
        if (earlier) continue;
        acc[l == 0 ? 0 : (l == 1 ? 1 : 2)] += val * val;
      }
    }
  }
  for (int k = 0; k < 5; ++k) {
    for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if (lane == 0) red[warp][k] = acc[k];
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    double t = 0;
    for (int w = 0; w < kFroWarps; ++w) t += red[w][threadIdx.x];
    part[(int64_t)blockIdx.x * 5 + threadIdx.x] = t;
  }
}

// Cells without projectors: the off-diagonal entries are the merged stencil's, the same in every row
// but for the cell faces, so their squares have a closed form (stencil_norms); what is left is the
// sum of the diagonal and of its square.  part as above, with zeros in the other places.
__global__ void k_diag_sums(int64_t n, double diag, const double *__restrict__ vloc, double *part) {
  __shared__ double red[8][2];
  double s = 0, s2 = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double d = diag + vloc[i];
    s += d;
    s2 = fma(d, d, s2);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = s;
    red[threadIdx.x >> 5][1] = s2;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    double t = 0;
    for (int w = 0; w < 8 && threadIdx.x >= 3; ++w) t += red[w][threadIdx.x - 3];
    part[(int64_t)blockIdx.x * 5 + threadIdx.x] = t;
  }
}

// Squares of the merged stencil entries over all rows, by block (l = 0 off the diagonal, l = +1; l = -1
// has the same), and what arms that wrap onto their own point add to the diagonal.
static void stencil_norms(const HamView &v, double *off0, double *plus, double *diag) {
  *diag = 0;
  double row = 0;
  auto wrapped = [&](int n, const double *w) {   // arms along x or y
    std::vector<double> at(std::min(n, 2 * v.m + 1), 0.0);
    for (int k = 1; k <= v.m; ++k)
      for (int sg = -1; sg <= 1; sg += 2) {
        const int o = n > 2 * v.m ? (sg > 0 ? k : v.m + k) : ((sg * k) % n + n) % n;   // apart where nothing coincides
        at[o] += w[k];
      }
    *diag += at[0];
    for (size_t o = 1; o < at.size(); ++o) row += at[o] * at[o];
  };
  wrapped(v.nx, v.wx);
  wrapped(v.ny, v.wy);
  const double nxy = (double)v.nx * v.ny;
  *off0 = row * (double)v.n;
  *plus = 0;
  for (int k = 1; k <= v.m; ++k) {   // arms along z are apart: k <= nz
    *off0 += nxy * 2.0 * (v.nz - k) * v.wz[k] * v.wz[k];
    *plus += nxy * k * v.wz[k] * v.wz[k];
  }
}

__global__ void k_sum_parts(const double *part, int nparts, double *out) {
  // one block, 128 lanes per sum, the lanes' sums added in order
  __shared__ double lanes[128][5];
  double s[5] = {0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nparts; b += 128)
    for (int k = 0; k < 5; ++k) s[k] += part[(int64_t)b * 5 + k];
  for (int k = 0; k < 5; ++k) lanes[threadIdx.x][k] = s[k];
  __syncthreads();
  if (threadIdx.x < 5) {
    double t = 0;
    for (int y = 0; y < 128; ++y) t += lanes[y][threadIdx.x];
    out[threadIdx.x] = t;
  }
}

// V_loc in the fixed-point unit 2^(ew - 58), line by line, and that unit for the applies
__global__ void k_fixed_vloc(int64_t n, int nz, VlocUnit u, const double *v, VlocUnit *du, long long *fv) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *du = u;
  if (u.ew == kNoUnit) return;
  const double up = ldexp(1.0, 58 - u.ew);
  const int64_t nxy = n / nz;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    fv[(i % nxy) * nz + i / nxy] = __double2ll_rn(v[i] * up);
}

// Integer form of the FD coefficients, |c_k| = n_k / den.
static int64_t fd_integers(int m, int *nk) {
  static const int den[kMaxHalf + 1] = {0, 1, 12, 180, 5040, 25200, 831600};
  static const int num[kMaxHalf + 1][kMaxHalf] = {
      {0}, {1}, {16, 1}, {270, 27, 2}, {8064, 1008, 128, 9}, {42000, 6000, 1000, 125, 8},
      {1425600, 222750, 44000, 7425, 864, 50}};
  for (int k = 0; k <= kMaxHalf; ++k) nk[k] = (k >= 1 && k <= m) ? num[m][k - 1] : 0;
  return den[m];
}

// The parts of the fixed-point tables that follow the range of V_loc: the common exponent of
// the weights, the kinetic factors and V_loc in that unit.  Where a range does not fit, fx_ok stays 0
// (the FP64 kernels then serve the cell) and captured applies are told by kNoUnit.
static cbs_status fixed_weights(cbs_hamiltonian *h, double vmax) {
  HamView &v = h->v;
  v.fx_ok = 0;
  if (v.n_atoms && v.np4 != 4) return CBS_OK;
  const int64_t den = fd_integers(v.m, v.fx_nk);
  int64_t sum = 0;
  for (int k = 1; k <= v.m; ++k) sum += v.fx_nk[k];
  v.fx_st = 1;   // sum < 2^(fx_st - 1), not just 2^fx_st: Product::add takes the sums' upper words as ints
  while (((int64_t)1 << (v.fx_st - 1)) <= sum) ++v.fx_st;
  const double hh[3] = {h->hx, h->hy, h->hz};
  double top = 2.0 * (fabs(v.diag_kin) + vmax), c[3];
  for (int d = 0; d < 3; ++d) {
    c[d] = ldexp(1.0, v.fx_st) / (2.0 * hh[d] * hh[d] * (double)den);
    top = std::max(top, c[d]);
  }
  const bool fits = top < 1e50 && top > 1e-50;
  if (fits) {
    v.fx_ew = ilogb(top) + 1;
    for (int d = 0; d < 3; ++d) {
      const long long f = llrint(ldexp(c[d], 58 - v.fx_ew));
      v.fx_c1[d] = (int)(f >> 31);
      v.fx_c0[d] = (int)(f & 0x7fffffff);
    }
    // The neighbours' coefficients n_k c differ from the FP64 weights by up to half an ulp each.
    // What a constant field sees of the difference goes onto the diagonal: left out, the operator
    // is shifted by up to some 8e-15 of energy, and the gradient of a 12x10x6 cell's ring objective
    // at tol 1e-14 is 5.5e-14 from that of the FP64 weights instead of 1.5e-14 (the FP64
    // kernels': 2.1e-14).
    double shift = 0;
    for (int d = 0; d < 3; ++d) {
      const long long f = ((long long)v.fx_c1[d] << 31) + v.fx_c0[d];
      const double fh = (double)f, fl = (double)(f - (long long)fh);   // f = fh + fl
      const double *w = d == 0 ? v.wx : d == 1 ? v.wy : v.wz;
      for (int k = 1; k <= v.m; ++k) {
        const double n = ldexp(k & 1 ? 1.0 : -1.0, v.fx_ew - 58 - v.fx_st) * v.fx_nk[k];
        shift += 2 * (fma(fh, n, w[k]) + fl * n);   // w_k = -n_k c: what is left of it
      }
    }
    v.fx_diag = llrint(ldexp(v.diag_kin, 58 - v.fx_ew)) + llrint(ldexp(shift, 58 - v.fx_ew));
  }
  v.fx_iso = h->hx == h->hy && h->hy == h->hz;
  double sxy = 0, sz = 0;
  for (int k = 1; k <= v.m; ++k) {
    sxy += 2 * (fabs(v.wx[k]) + fabs(v.wy[k]));
    sz += 2 * fabs(v.wz[k]);
  }
  v.fx_wxy = (float)(sxy * 1.001);
  v.fx_wz = (float)(sz * 1.001);
  const VlocUnit unit = {fits ? v.fx_ew : kNoUnit, vmax};
  k_fixed_vloc<<<(unsigned)std::min<int64_t>(1024, (v.n + 255) / 256), 256>>>(
      v.n, v.nz, unit, v.vloc, const_cast<VlocUnit *>(v.fx_u), const_cast<long long *>(v.fx_v));
  count_launches(1);
  CBS_CUDA(cudaGetLastError());
  v.fx_ok = fits && h->fx_proj_ok;
  return CBS_OK;
}

static cbs_status dalloc(cbs_hamiltonian *h, void **p, size_t bytes) {
  if (bytes == 0) bytes = 16;
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    set_error("cudaMalloc failed in cbs_create_hamiltonian");
    return CBS_ENOMEM;
  }
  h->allocs[h->n_allocs++] = *p;
  return CBS_OK;
}

template <typename T>
static cbs_status upload(cbs_hamiltonian *h, const T *src, size_t count, const T **dst) {
  void *p = nullptr;
  cbs_status s = dalloc(h, &p, count * sizeof(T));
  if (s != CBS_OK) return s;
  if (count) CBS_CUDA(cudaMemcpy(p, src, count * sizeof(T), cudaMemcpyHostToDevice));
  *dst = (const T *)p;
  return CBS_OK;
}

}  // namespace cbs

using namespace cbs;

extern "C" void cbs_hamiltonian_free(cbs_hamiltonian *h) {
  if (!h) return;
  for (int k = 0; k < h->n_allocs; ++k) cudaFree(h->allocs[k]);
  if (h->scratch) cudaFree(h->scratch);
  free(h);
}

extern "C" int64_t cbs_hamiltonian_size(const cbs_hamiltonian *h) { return h ? h->v.n : 0; }

extern "C" cbs_status cbs_hamiltonian_norms(const cbs_hamiltonian *h, double E, double *np_,
                                            double *n0, double *nm) {
  if (!h) { set_error("null hamiltonian"); return CBS_EINVAL; }
  double n = (double)h->v.n;
  double a2 = h->fro_off0 + h->diag_sum2 - 2.0 * E * h->diag_sum + n * E * E;
  if (np_) *np_ = sqrt(h->fro_p2);
  if (n0) *n0 = sqrt(a2 > 0 ? a2 : 0.0);
  if (nm) *nm = sqrt(h->fro_m2);
  return CBS_OK;
}

// Exact Frobenius norms of H+, H- and the pieces of ||H0 - E||_F, on the device.
static cbs_status compute_norms(cbs_hamiltonian *h) {
  HamView &v = h->v;
  // exact Frobenius norms on the device
  const bool bare = v.n_atoms == 0;
  const int nb = bare ? std::min(304, ceil_div(v.n, 256)) : ceil_div(v.n, kFroWarps);
  double off0 = 0, plus = 0, diag = 0;
  double *part = nullptr, *out = nullptr;
  int *err = nullptr;
  CBS_CUDA(cudaMalloc(&part, ((size_t)nb * 5 + 6) * sizeof(double)));
  out = part + (size_t)nb * 5;
  err = (int *)(out + 5);
  CBS_CUDA(cudaMemset(err, 0, sizeof(int)));
  if (bare) {
    stencil_norms(v, &off0, &plus, &diag);
    k_diag_sums<<<nb, 256>>>(v.n, v.diag_kin + diag, v.vloc, part);
  } else {
    k_frobenius<<<nb, 32 * kFroWarps>>>(v, part, err);
  }
  cbs::count_launches(1);
  k_sum_parts<<<1, 128>>>(part, nb, out); cbs::count_launches(1);
  double res[5];
  int herr = 0;
  cudaError_t e1 = cudaMemcpy(res, out, sizeof(res), cudaMemcpyDeviceToHost);
  cudaError_t e2 = cudaMemcpy(&herr, err, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(part);
  if (e1 != cudaSuccess) return cuda_fail(e1, "Frobenius norm kernel");
  if (e2 != cudaSuccess) return cuda_fail(e2, "Frobenius norm kernel");
  if (herr == 1) { set_error("more than 64 atoms cover one grid point"); return CBS_EINVAL; }
  if (herr == 2) { set_error("projector coupling beyond the neighbouring cells"); return CBS_EINVAL; }
  h->fro_off0 = res[0] + off0; h->fro_p2 = res[1] + plus; h->fro_m2 = res[2] + plus;
  h->diag_sum = res[3]; h->diag_sum2 = res[4];
  return CBS_OK;
}

// Projector tables of the kernels that march along lines: the entries in line order (single
// precision and fixed point) and in gather order (fixed point: per atom, entries of image -1,
// then 0, then +1), and the bounds that size the fixed-point sums.
static cbs_status line_projectors(cbs_hamiltonian *h, const cbs_projectors *P, const std::vector<int64_t> &pt_ptr,
                                   const std::vector<int32_t> &pt_ent, const std::vector<int32_t> &pt_atom) {
  HamView &v = h->v;
  const int na = P->n_atoms, np = P->n_proj;
  const int64_t nnz = P->sup_ptr[na];
  double pmax = 0, l1max = 0, dmax = 0;
  for (int a = 0; a < na; ++a) {
    double l1[4] = {0, 0, 0, 0};
    for (int64_t t = P->sup_ptr[a]; t < P->sup_ptr[a + 1]; ++t)
      for (int mu = 0; mu < np; ++mu) {
        const double p = fabs(P->sup_val[t * np + mu]);
        pmax = std::max(pmax, p);
        l1[mu] += p;
      }
    for (int mu = 0; mu < np; ++mu) {
      double d = 0;
      for (int nu = 0; nu < np; ++nu) d += fabs(P->h[((int64_t)a * np + mu) * np + nu]) * l1[nu];
      dmax = std::max(dmax, d);
      l1max = std::max(l1max, l1[mu]);
    }
  }
  double cover = 0;
  for (int64_t i = 0; i < v.n; ++i) {
    double c = 0;
    for (int64_t q = pt_ptr[i]; q < pt_ptr[i + 1]; ++q)
      for (int mu = 0; mu < np; ++mu) c += fabs(P->sup_val[(int64_t)pt_ent[q] * np + mu]);
    cover = std::max(cover, c);
  }
  if (pmax == 0) pmax = l1max = 1;
  // (the kernels count the two words of an entry's values in 32 bits)
  h->fx_proj_ok = nnz < (int64_t)1 << 30 && pmax > 1e-50 && l1max < 1e50 && dmax < 1e30 && cover * dmax < 1e30;
  // |p| 2^fp < 2^56, and a thread's sum of high words times 2^30 below 2^62
  v.fx_fp = h->fx_proj_ok ? std::min(56 - (ilogb(pmax) + 1), 61 - (ilogb(l1max) + 1)) : 0;
  v.fx_db = (float)(dmax * 1.001);
  v.fx_pb = (float)(cover * dmax * 1.001);
  const double unit = ldexp(1.0, v.fx_fp);
  auto words = [&](int64_t t, int4 *out) {
    int w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int mu = 0; mu < (h->fx_proj_ok ? np : 0); ++mu) {
      const long long f = llrint(P->sup_val[t * np + mu] * unit);
      w[2 * mu] = balanced_hi(f);
      w[2 * mu + 1] = balanced_lo(f);
    }
    out[0] = make_int4(w[0], w[1], w[2], w[3]);
    out[1] = make_int4(w[4], w[5], w[6], w[7]);
  };
  auto single = [&](int64_t t) {
    float pv[4] = {0, 0, 0, 0};
    for (int mu = 0; mu < np; ++mu) pv[mu] = (float)P->sup_val[t * np + mu];
    return make_float4(pv[0], pv[1], pv[2], pv[3]);
  };
  // one host buffer, one allocation and one copy for all tables: on small cells those are what they cost
  const int64_t nxy = (int64_t)v.nx * v.ny;
  size_t bytes = 0;
  auto place = [&](size_t count, size_t size) {
    const size_t at = bytes;
    bytes += (count * size + 255) & ~(size_t)255;
    return at;
  };
  const size_t n1 = (size_t)nnz + 1;   // a spare entry after the last of the line order
  const size_t a_pp = place(2 * n1, sizeof(int4)), a_p32 = place(n1, sizeof(float4)), a_img = place(n1, sizeof(int)),
               a_ptr = place((size_t)nxy * (v.nz + 1), sizeof(int)), a_gp = place(2 * (size_t)nnz, sizeof(int4)),
               a_gp32 = place(nnz, sizeof(float4)), a_gi = place(nnz, sizeof(int)), a_gt = place(nnz, sizeof(int)),
               a_gm = place(nnz, sizeof(int2)), a_gc = place((size_t)na * 12, sizeof(long long)),
               a_gptr = place((size_t)na * 4, sizeof(int));
  std::vector<unsigned char> host(bytes, 0);
  unsigned char *hb = host.data();
  int4 *pp = (int4 *)(hb + a_pp), *gp = (int4 *)(hb + a_gp);
  float4 *p32 = (float4 *)(hb + a_p32), *gp32 = (float4 *)(hb + a_gp32);
  int2 *gm = (int2 *)(hb + a_gm);
  long long *gc = (long long *)(hb + a_gc);
  int *img = (int *)(hb + a_img), *ptr = (int *)(hb + a_ptr), *gi = (int *)(hb + a_gi), *gt = (int *)(hb + a_gt),
      *gptr = (int *)(hb + a_gptr);
  std::vector<int> at(nnz);   // place of an entry in gather order
  int64_t o = 0;
  std::vector<double> size;
  for (int a = 0; a < na; ++a) {
    // the larger values of each projector: a quarter of the largest, at least six of them (a narrow
    // projector has one or two, and an ordinary column often something small there)
    double large[4] = {0, 0, 0, 0}, top[4] = {0, 0, 0, 0};
    const int64_t t0 = P->sup_ptr[a], entries = P->sup_ptr[a + 1] - t0;
    for (int mu = 0; mu < np && entries > 0; ++mu) {
      size.resize(entries);
      for (int64_t t = 0; t < entries; ++t) size[t] = fabs(P->sup_val[(t0 + t) * np + mu]);
      const int64_t sixth = std::min<int64_t>(6, entries) - 1;
      std::nth_element(size.begin(), size.begin() + sixth, size.end(), std::greater<double>());
      top[mu] = *std::max_element(size.begin(), size.begin() + sixth + 1);
      large[mu] = std::min(size[sixth], top[mu] / 4);
    }
    for (int m = -1; m <= 2; ++m) {
      gptr[(size_t)a * 4 + m + 1] = (int)o;
      if (m == 2) break;
      for (int64_t t = t0; t < t0 + entries; ++t)
        if (P->sup_wrap[t] == m) {
          gi[o] = P->sup_idx[t];
          gt[o] = (int)t;
          at[t] = (int)o;
          words(t, &gp[2 * o]);
          const int4 w0 = gp[2 * o], w1 = gp[2 * o + 1];
          const int low[4] = {w0.y, w0.w, w1.y, w1.w};
          for (int mu = 0; mu < 4; ++mu) gc[((size_t)a * 3 + m + 1) * 4 + mu] += low[mu];
          gp32[o] = single(t);
          for (int mu = 0; mu < np; ++mu) {
            const double p = fabs(P->sup_val[t * np + mu]);
            if (p >= large[mu] && (p > 0 || top[mu] == 0)) (mu < 2 ? gm[o].x : gm[o].y) |= mu % 2 ? (int)0xffff0000 : 0xffff;
          }
          ++o;
        }
    }
  }
  for (int64_t k = 0; k < (int64_t)na * 12; ++k) gc[k] /= 2;   // 2^28 of the 2^29 that a low word stands for
  o = 0;
  for (int64_t line = 0; line < nxy; ++line) {
    for (int iz = 0; iz < v.nz; ++iz) {
      const int64_t i = (int64_t)iz * nxy + line;
      ptr[line * (v.nz + 1) + iz] = (int)o;
      for (int64_t q = pt_ptr[i]; q < pt_ptr[i + 1]; ++q, ++o) {
        const int64_t g = at[pt_ent[q]];
        pp[2 * o] = gp[2 * g];
        pp[2 * o + 1] = gp[2 * g + 1];
        p32[o] = gp32[g];
        img[o] = ((int)P->sup_wrap[pt_ent[q]] + 1) * na + pt_atom[q];
      }
    }
    ptr[line * (v.nz + 1) + v.nz] = (int)o;
  }
  const unsigned char *dev = nullptr;
  const cbs_status s = upload(h, hb, bytes, &dev);
  if (s != CBS_OK) return s;
  v.fx_p = (const int4 *)(dev + a_pp);
  v.ln_p32 = (const float4 *)(dev + a_p32);
  v.fx_img = (const int *)(dev + a_img);
  v.fx_ptr = (const int *)(dev + a_ptr);
  v.fx_gp = (const int4 *)(dev + a_gp);
  v.fx_gp32 = (const float4 *)(dev + a_gp32);
  v.fx_gi = (const int *)(dev + a_gi);
  v.fx_gt = (const int *)(dev + a_gt);
  v.fx_gm = (const int2 *)(dev + a_gm);
  v.fx_gc = (const long long *)(dev + a_gc);
  v.fx_gptr = (const int *)(dev + a_gptr);
  return CBS_OK;
}

static cbs_status create_impl(const cbs_grid *g, const double *v_loc, const cbs_projectors *P,
                              cbs_hamiltonian *h) {
  HamView &v = h->v;
  if (g->nx < 1 || g->ny < 1 || g->nz < 1 || !(g->hx > 0) || !(g->hy > 0) || !(g->hz > 0)) {
    set_error("grid sizes and spacings must be positive");
    return CBS_EINVAL;
  }
  if (g->fd_order < 2 || g->fd_order > 2 * kMaxHalf || g->fd_order % 2) {
    set_error("fd_order must be even, 2..12");
    return CBS_EINVAL;
  }
  const int m = g->fd_order / 2;
  if (m > g->nz) {
    set_error("fd_order/2 must not exceed nz (nearest-cell coupling only)");
    return CBS_EINVAL;
  }
  if (!v_loc) { set_error("v_loc is NULL"); return CBS_EINVAL; }
  v.nx = g->nx; v.ny = g->ny; v.nz = g->nz; v.m = m;
  v.n = (int64_t)g->nx * g->ny * g->nz;
  if (v.n > (int64_t)1 << 31) { set_error("grid larger than 2^31 points"); return CBS_EINVAL; }
  h->hx = g->hx; h->hy = g->hy; h->hz = g->hz; h->fd_order = g->fd_order;
  fd_weights(g->fd_order, h->fd_c);
  v.diag_kin = -0.5 * h->fd_c[0] * (1.0 / (g->hx * g->hx) + 1.0 / (g->hy * g->hy) + 1.0 / (g->hz * g->hz));
  for (int k = 0; k <= kMaxHalf; ++k) {
    double c = (k >= 1 && k <= m) ? h->fd_c[k] : 0.0;
    v.wx[k] = -0.5 * c / (g->hx * g->hx);
    v.wy[k] = -0.5 * c / (g->hy * g->hy);
    v.wz[k] = -0.5 * c / (g->hz * g->hz);
    v.w32[0][k] = (float)v.wx[k];
    v.w32[1][k] = (float)v.wy[k];
    v.w32[2][k] = (float)v.wz[k];
  }
  v.diag_kin32 = (float)v.diag_kin;
  const size_t N = (size_t)v.n;
  for (size_t i = 0; i < N; ++i)
    if (!isfinite(v_loc[i])) { set_error("v_loc contains a non-finite value"); return CBS_EINVAL; }
  // V_loc in FP64 and in fixed point with its unit: one allocation (on small cells they are what
  // creation costs)
  void *pv = nullptr;
  cbs_status s = dalloc(h, &pv, 2 * N * sizeof(double) + sizeof(VlocUnit));
  if (s != CBS_OK) return s;
  CBS_CUDA(cudaMemcpy(pv, v_loc, N * sizeof(double), cudaMemcpyHostToDevice));
  v.vloc = (const double *)pv;
  v.fx_v = (const long long *)((double *)pv + N);
  v.fx_u = (const VlocUnit *)(v.fx_v + N);
  std::vector<float> v32(v_loc, v_loc + N);
  s = upload(h, v32.data(), N, &v.vloc32);
  if (s != CBS_OK) return s;

  double vmax = 0;
  for (size_t i = 0; i < N; ++i) vmax = std::max(vmax, fabs(v_loc[i]));
  // projectors
  v.n_atoms = 0; v.n_proj = 0; h->nnz = 0; v.np4 = 4;
  h->fx_proj_ok = 1;
  std::vector<int64_t> pt_ptr(N + 1, 0);
  if (P && P->n_atoms > 0) {
    if (P->n_proj < 1 || P->n_proj > kMaxProj) { set_error("n_proj must be 1..8"); return CBS_EINVAL; }
    if (!P->sup_ptr || !P->sup_idx || !P->sup_wrap || !P->sup_val || !P->h) {
      set_error("projector table has a NULL array");
      return CBS_EINVAL;
    }
    const int na = P->n_atoms, np = P->n_proj;
    if (P->sup_ptr[0] != 0) { set_error("sup_ptr[0] must be 0"); return CBS_EINVAL; }
    for (int a = 0; a < na; ++a)
      if (P->sup_ptr[a + 1] < P->sup_ptr[a]) { set_error("sup_ptr must be non-decreasing"); return CBS_EINVAL; }
    const int64_t nnz = P->sup_ptr[na];
    if (nnz > INT32_MAX) { set_error("projector table too large"); return CBS_EINVAL; }
    std::vector<int> stamp(N, -1);
    for (int a = 0; a < na; ++a) {
      bool has_m = false, has_p = false;
      for (int64_t t = P->sup_ptr[a]; t < P->sup_ptr[a + 1]; ++t) {
        int32_t i = P->sup_idx[t];
        int w = P->sup_wrap[t];
        if (i < 0 || (size_t)i >= N) { set_error("sup_idx out of range"); return CBS_EINVAL; }
        if (w < -1 || w > 1) { set_error("sup_wrap must be -1, 0 or +1"); return CBS_EINVAL; }
        has_m |= (w == -1); has_p |= (w == 1);
        if (stamp[i] == a) { set_error("a grid point is covered twice by one atom"); return CBS_EINVAL; }
        stamp[i] = a;
        for (int mu = 0; mu < np; ++mu)
          if (!isfinite(P->sup_val[t * np + mu])) { set_error("sup_val not finite"); return CBS_EINVAL; }
        pt_ptr[i + 1]++;
      }
      if (has_m && has_p) {
        set_error("an atom covers points with wraps -1 and +1: support longer than the cell along z");
        return CBS_EINVAL;
      }
      for (int mu = 0; mu < np; ++mu)
        for (int nu = 0; nu < np; ++nu) {
          double x = P->h[((int64_t)a * np + mu) * np + nu], y = P->h[((int64_t)a * np + nu) * np + mu];
          if (!isfinite(x) || fabs(x - y) > 1e-12 * (fabs(x) + fabs(y) + 1e-300)) {
            set_error("h blocks must be finite and symmetric");
            return CBS_EINVAL;
          }
        }
    }
    for (size_t i = 0; i < N; ++i) pt_ptr[i + 1] += pt_ptr[i];
    std::vector<int32_t> pt_ent(nnz), pt_atom(nnz);
    std::vector<int64_t> fill(pt_ptr.begin(), pt_ptr.end() - 1);
    for (int a = 0; a < na; ++a)
      for (int64_t t = P->sup_ptr[a]; t < P->sup_ptr[a + 1]; ++t) {
        int64_t q = fill[P->sup_idx[t]]++;
        pt_ent[q] = (int32_t)t;
        pt_atom[q] = a;
      }
    v.n_atoms = na; v.n_proj = np; h->nnz = nnz;
    if ((s = upload(h, P->sup_ptr, (size_t)na + 1, &v.sup_ptr)) != CBS_OK) return s;
    if ((s = upload(h, P->sup_idx, (size_t)nnz, &v.sup_idx)) != CBS_OK) return s;
    if ((s = upload(h, P->sup_wrap, (size_t)nnz, &v.sup_wrap)) != CBS_OK) return s;
    if ((s = upload(h, P->sup_val, (size_t)nnz * np, &v.sup_val)) != CBS_OK) return s;
    std::vector<float> sv32(P->sup_val, P->sup_val + (size_t)nnz * np);
    if ((s = upload(h, sv32.data(), sv32.size(), &v.sup_val32)) != CBS_OK) return s;
    if ((s = upload(h, P->h, (size_t)na * np * np, &v.h)) != CBS_OK) return s;
    std::vector<float> h32(P->h, P->h + (size_t)na * np * np);
    if ((s = upload(h, h32.data(), h32.size(), &v.h32)) != CBS_OK) return s;
    if ((s = upload(h, pt_ptr.data(), N + 1, &v.pt_ptr)) != CBS_OK) return s;
    if ((s = upload(h, pt_ent.data(), (size_t)nnz, &v.pt_ent)) != CBS_OK) return s;
    if ((s = upload(h, pt_atom.data(), (size_t)nnz, &v.pt_atom)) != CBS_OK) return s;
    // packed per-entry records (point order)
    v.np4 = np <= 4 ? 4 : 8;
    std::vector<int2> aw(nnz);
    for (int64_t q = 0; q < nnz; ++q) aw[q] = make_int2(pt_atom[q], (int)P->sup_wrap[pt_ent[q]]);
    if ((s = upload(h, aw.data(), (size_t)nnz, &v.pt_aw)) != CBS_OK) return s;
    if (np <= 4 && (s = line_projectors(h, P, pt_ptr, pt_ent, pt_atom)) != CBS_OK) return s;
  } else {
    if ((s = upload(h, pt_ptr.data(), N + 1, &v.pt_ptr)) != CBS_OK) return s;
  }
  if ((s = fixed_weights(h, vmax)) != CBS_OK) return s;
  return compute_norms(h);
}

extern "C" cbs_status cbs_create_hamiltonian(const cbs_grid *grid, const double *v_loc,
                                             const cbs_projectors *proj, cbs_hamiltonian **out) {
  if (!grid || !out) { set_error("null argument"); return CBS_EINVAL; }
  *out = nullptr;
  cbs_hamiltonian *h = (cbs_hamiltonian *)calloc(1, sizeof(cbs_hamiltonian));
  if (!h) { set_error("host allocation failed"); return CBS_ENOMEM; }
  cbs_status s = create_impl(grid, v_loc, proj, h);
  if (s != CBS_OK) { cbs_hamiltonian_free(h); return s; }
  *out = h;
  return CBS_OK;
}

namespace cbs {
// V_loc in single precision from the FP64 copy, a flag if any value is not finite, and
// max |V_loc| (as bits: the order of non-negative doubles).
__global__ void k_vloc32(int64_t n, const double *v, float *v32, int *bad, unsigned long long *vmax) {
  int b = 0;
  unsigned long long m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double x = v[i];
    v32[i] = (float)x;
    b |= !isfinite(x);
    m = max(m, (unsigned long long)__double_as_longlong(fabs(x)));
  }
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0 && m) atomicMax(vmax, m);
  if (__syncthreads_or(b) && threadIdx.x == 0) atomicOr(bad, 1);
}
}  // namespace cbs

extern "C" cbs_status cbs_hamiltonian_set_vloc(cbs_hamiltonian *h, const double *v_loc) {
  if (!h || !v_loc) { set_error("cbs_hamiltonian_set_vloc: null argument"); return CBS_EINVAL; }
  HamView &v = h->v;
  const size_t N = (size_t)v.n;
  int *bad = nullptr;
  double *tmp = nullptr;
  CBS_CUDA(cudaMalloc(&tmp, N * sizeof(double) + 256));
  bad = (int *)((char *)tmp + ((N * sizeof(double) + 127) & ~(size_t)127));
  unsigned long long *dmax = (unsigned long long *)(bad + 2);
  cbs_status s = CBS_OK;
  cudaError_t e = cudaMemcpy(tmp, v_loc, N * sizeof(double), cudaMemcpyDefault);
  if (e == cudaSuccess) e = cudaMemset(bad, 0, 2 * sizeof(int) + sizeof(unsigned long long));
  if (e == cudaSuccess) {
    // check into a scratch copy first, so a rejected V_loc leaves the handle unchanged
    k_vloc32<<<std::min<int64_t>(1024, ((int64_t)N + 255) / 256), 256>>>((int64_t)N, tmp,
                                                                         const_cast<float *>(v.vloc32), bad, dmax);
    cbs::count_launches(1);
    e = cudaGetLastError();
  }
  int hb = 0;
  double hmax = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&hb, bad, sizeof(int), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(&hmax, dmax, sizeof(double), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) s = cuda_fail(e, "cbs_hamiltonian_set_vloc");
  else if (hb) {
    // restore the single-precision copy from the unchanged FP64 one
    k_vloc32<<<std::min<int64_t>(1024, ((int64_t)N + 255) / 256), 256>>>((int64_t)N, v.vloc,
                                                                         const_cast<float *>(v.vloc32), bad, dmax);
    cbs::count_launches(1);
    cudaDeviceSynchronize();
    set_error("v_loc contains a non-finite value");
    s = CBS_EINVAL;
  } else {
    e = cudaMemcpy(const_cast<double *>(v.vloc), tmp, N * sizeof(double), cudaMemcpyDeviceToDevice);
    if (e != cudaSuccess) s = cuda_fail(e, "cbs_hamiltonian_set_vloc copy");
  }
  cudaFree(tmp);
  if (s != CBS_OK) return s;
  if ((s = fixed_weights(h, hmax)) != CBS_OK) return s;
  return compute_norms(h);
}
