// Shared helpers for libcbs: complex arithmetic on interleaved pairs, error plumbing,
// and the device-side view of the cell Hamiltonian.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/cbs.h"

namespace cbs {

// ---------------------------------------------------------------- complex types
template <typename R> struct CT;
template <> struct CT<double> { typedef double2 T; };
template <> struct CT<float> { typedef float2 T; };

template <typename R> __host__ __device__ __forceinline__ typename CT<R>::T mk(R a, R b) {
  typename CT<R>::T r; r.x = a; r.y = b; return r;
}
__host__ __device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// conj(a) * b
__host__ __device__ __forceinline__ double2 cmulc(double2 a, double2 b) {
  return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
__host__ __device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
__host__ __device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__host__ __device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__host__ __device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__host__ __device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__host__ __device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }
__host__ __device__ __forceinline__ float cabs2(float2 a) { return a.x * a.x + a.y * a.y; }
// a += s * b  (s complex)
__host__ __device__ __forceinline__ double2 cfma(double2 s, double2 b, double2 a) {
  a.x = fma(s.x, b.x, a.x); a.x = fma(-s.y, b.y, a.x);
  a.y = fma(s.x, b.y, a.y); a.y = fma(s.y, b.x, a.y);
  return a;
}
__host__ __device__ __forceinline__ float2 cfma(float2 s, float2 b, float2 a) {
  a.x = fmaf(s.x, b.x, a.x); a.x = fmaf(-s.y, b.y, a.x);
  a.y = fmaf(s.x, b.y, a.y); a.y = fmaf(s.y, b.x, a.y);
  return a;
}
__host__ __device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  // One reciprocal and a correction by the residual a - q b where both moduli are well inside the range
  // (a division is some 20 dependent FP64 operations, and the scalars of an iteration wait for
  // theirs; the correction is 5, and the error at most 1.9 half ulps of the modulus, Smith's 2.7,
  // without the correction 4.3), else Smith's algorithm.
  const double b2 = fma(b.x, b.x, b.y * b.y), a1 = fabs(a.x) + fabs(a.y);
  if (b2 > 1e-200 && b2 < 1e200 && a1 > 1e-150 && a1 < 1e150) {
    const double i = 1.0 / b2;
    const double qx = fma(a.x, b.x, a.y * b.y) * i, qy = fma(a.y, b.x, -(a.x * b.y)) * i;
    const double rx = fma(-qx, b.x, fma(qy, b.y, a.x)), ry = fma(-qx, b.y, fma(-qy, b.x, a.y));
    return make_double2(fma(fma(rx, b.x, ry * b.y), i, qx), fma(fma(ry, b.x, -(rx * b.y)), i, qy));
  }
  if (fabs(b.x) >= fabs(b.y)) {
    double r = b.y / b.x, d = b.x + b.y * r;
    return make_double2((a.x + a.y * r) / d, (a.y - a.x * r) / d);
  } else {
    double r = b.x / b.y, d = b.y + b.x * r;
    return make_double2((a.x * r + a.y) / d, (a.y * r - a.x) / d);
  }
}
__host__ __device__ __forceinline__ double2 to_d(float2 a) { return make_double2(a.x, a.y); }
__host__ __device__ __forceinline__ double2 to_d(double2 a) { return a; }
template <typename R> __host__ __device__ __forceinline__ typename CT<R>::T from_d(double2 a);
template <> __host__ __device__ __forceinline__ double2 from_d<double>(double2 a) { return a; }
template <> __host__ __device__ __forceinline__ float2 from_d<float>(double2 a) {
  return make_float2((float)a.x, (float)a.y);
}

// ---------------------------------------------------------------- Hamiltonian
constexpr int kMaxHalf = 6;   // fd_order <= 12
constexpr int kMaxProj = 8;

// The unit that the device table fx_v holds V_loc in, and the range of V_loc.  V_loc may be replaced in
// place, so these lie in device memory: an apply captured in a graph with another unit takes the
// FP64 formula (column_scale), which reads V_loc itself.
struct VlocUnit {
  int ew;        // fx_v holds V_loc * 2^(58 - ew); kNoUnit: it does not fit
  double vmax;   // max |V_loc|
};
constexpr int kNoUnit = -(1 << 30);

// Device view, passed by value to kernels.
struct HamView {
  int nx, ny, nz, m;        // grid and FD half-width
  int64_t n;                // nx*ny*nz
  double diag_kin;          // -1/2 c0 (1/hx^2 + 1/hy^2 + 1/hz^2)
  double wx[kMaxHalf + 1], wy[kMaxHalf + 1], wz[kMaxHalf + 1];  // -1/2 c_k / h^2 (k >= 1)
  float w32[3][kMaxHalf + 1];   // the same weights in single precision (x, y, z)
  float diag_kin32;
  const double *vloc;
  const float *vloc32;
  // projector table and its transpose (grid point -> covering entries)
  int n_atoms, n_proj;
  const int64_t *sup_ptr;   // [n_atoms+1]
  const int32_t *sup_idx;   // [nnz]
  const int8_t *sup_wrap;   // [nnz]
  const double *sup_val;    // [nnz][n_proj]
  const float *sup_val32;
  const double *h;          // [n_atoms][n_proj][n_proj]
  const float *h32;
  const int64_t *pt_ptr;    // [n+1]
  const int32_t *pt_ent;    // [nnz] support entry index
  const int32_t *pt_atom;   // [nnz] atom of that entry
  int np4;                  // projector slots per entry in D: 4 (n_proj <= 4) or 8
  const int2 *pt_aw;        // [nnz] (atom, wrap) of each covering entry, point order
  // stencil launch shape chosen by cbs_autotune_apply, per precision ([0] complex128,
  // [1] complex64): a block covers tune_py x-lines of tune_pz rows (0 = default: 256 /
  // threads per line x-lines of one row) and, for complex64, whether the
  // two-columns-per-thread kernel is used (1 = yes, 0 = default, -1 = no)
  int tune_py[2], tune_pz[2];
  int tune_x2;
  // fixed-point tables of the complex128 apply (fixed.cuh); fx_ok = 0: FP64 kernels only
  int fx_ok, fx_iso;        // fx_iso: hx = hy = hz
  int fx_fp;                // projector values as p * 2^fx_fp
  int fx_ew;                // weights (diagonal, kinetic factors) are stored as g * 2^(58 - fx_ew)
  int fx_st;                // sum_k n_k < 2^(fx_st - 1): half the range, see WeightedSum
  int fx_nk[kMaxHalf + 1];  // n_k: |c_k| = n_k / den
  int fx_c1[3], fx_c0[3];   // 2^fx_st / (2 h^2 den) per direction, high and low 31-bit words
  float fx_wxy, fx_wz;      // sums of |weights| of the x and y arms and of the z arms
  float fx_db, fx_pb;       // bounds: largest |D| per unit component, largest projector term
  long long fx_diag;        // kinetic diagonal in the unit of the weights
  const VlocUnit *fx_u;
  // tables in line order (x-y line by line, along z inside a line), the projectors' for at most
  // 4 per atom
  const float4 *ln_p32;     // [nnz+1] projector values of the entries, zero-padded to 4
  const long long *fx_v;    // [n] V_loc * 2^(58 - fx_u->ew)
  const int *fx_ptr;        // [nx ny][nz + 1] entries of each point of a line
  const int4 *fx_p;         // [nnz+1][2] projector values of the entries: high and low 29-bit words of 4
  const int *fx_img;        // [nnz+1] (wrap + 1) * n_atoms + atom of the entries
  const int4 *fx_gp;        // projector values in gather order: per atom, by image -1, 0, +1
  const int2 *fx_gm;        // [nnz] gather order: ones in the 16 bits of projector mu where |p| is one of the
                            // atom's larger (a quarter of the largest, at least six of them)
  const long long *fx_gc;   // [n_atoms][3][4] half the sum of the low words of the projector values of each image
  const float4 *fx_gp32;    // [nnz] projector values in gather order, zero-padded to 4
  const int *fx_gi;         // [nnz] grid point, gather order
  const int *fx_gt;         // [nnz] support entry, gather order
  const int *fx_gptr;       // [n_atoms][4] first entry of each image, gather order
};

}  // namespace cbs

struct cbs_hamiltonian {
  cbs::HamView v;
  double hx, hy, hz;
  int fd_order;
  int64_t nnz;
  double fd_c[cbs::kMaxHalf + 1];
  // Frobenius pieces: ||H+||^2, ||H-||^2, off-diagonal part of ||H0||^2, sum d_i, sum d_i^2
  double fro_p2, fro_m2, fro_off0, diag_sum, diag_sum2;
  int fx_proj_ok;   // the projector values fit the fixed-point tables
  // scratch of one-call applies, kept between calls: taken by one call at a time (scratch_busy)
  void *scratch;
  size_t scratch_bytes;
  int scratch_busy;
  // device allocations owned by the handle
  void *allocs[32];
  int n_allocs;
};

namespace cbs {

// ---------------------------------------------------------------- errors
void set_error(const std::string &msg);
cbs_status cuda_fail(cudaError_t e, const char *what);

// kernel-launch accounting (cbs_kernel_launches)
void count_launches(uint64_t n);
void uncount_launches(uint64_t n);   // kernels recorded into a graph, not run
uint64_t launches_so_far();
uint64_t thread_launches();   // this thread's share of launches_so_far()

#define CBS_STR2(x) #x
#define CBS_STR(x) CBS_STR2(x)
#define CBS_CUDA(call)                                                               \
  do {                                                                               \
    cudaError_t _e = (call);                                                         \
    if (_e != cudaSuccess) return cbs::cuda_fail(_e, __FILE__ ":" CBS_STR(__LINE__) ": " #call); \
  } while (0)

inline int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// Thread-block shape for [N][L] blocks: x = columns, y = point lanes.
inline dim3 col_block(int L) {
  int py = 256 / L;
  if (py < 1) py = 1;
  return dim3((unsigned)L, (unsigned)py, 1);
}

// ---------------------------------------------------------------- kernels (launchers)
// apply.cu
template <typename R>
cbs_status launch_proj_gather(const HamView &H, int n_sys, int L, const typename CT<R>::T *X,
                              const double2 *twist, bool per_col, typename CT<R>::T *D,
                              const int *sys_active, cudaStream_t st);
template <typename R>
cbs_status launch_apply(const HamView &H, int n_sys, int L, const typename CT<R>::T *X,
                        typename CT<R>::T *Y, const double2 *twist, bool per_col,
                        const double *E, const typename CT<R>::T *D, const int *sys_active,
                        cudaStream_t st);
// Whether the operator apply supports L columns of element type dtype on this cell:
// complex128 up to 256 columns; complex64 up to 256, or up to 512 with an even L and at
// most 4 projectors (two columns per thread).  Sets the error message when it does not.
bool apply_supported(const HamView &H, int L, int dtype, const char *who);
// Bytes of scratch of apply_P.  The first apply_coef_bytes of it hold the projector
// coefficients D; complex128 scratch of only that size is served by the FP64 kernels.
size_t apply_coef_bytes(const HamView &H, int n_sys, int L, int dtype);
size_t apply_ws_bytes(const HamView &H, int n_sys, int L, int dtype);
// Y = P(w) X for n_sys systems; ws: scratch of ws_bytes.  parts: complex128 results are as accurate as
// the FP64 kernels' in the real and the imaginary part, else in the modulus (as BiCG applies it: its
// residual check sees the same operator)
template <typename R>
cbs_status apply_P(const HamView &H, int n_sys, int L, const typename CT<R>::T *X,
                   typename CT<R>::T *Y, const double2 *twist, bool per_col, const double *E,
                   void *ws, size_t ws_bytes, const int *sys_active, cudaStream_t st, bool parts = true);
// apply_fixed.cu: complex128 through fixed point
bool fixed_serves(const HamView &H, int n_sys, int L, size_t ws_bytes);
// whether the FP64 stencil takes about as long or less on a cell without projectors
bool fp64_quicker(const HamView &H, int n_sys, int L);
cbs_status apply_fixed(const HamView &H, int n_sys, int L, const double2 *X, double2 *Y,
                       const double2 *twist, bool per_col, const double *E, void *ws,
                       const int *sys_active, cudaStream_t st, bool parts);

}  // namespace cbs
