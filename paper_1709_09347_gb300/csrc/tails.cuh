// Work that follows a grid-wide reduction, done by the last block of a system to finish instead
// of by a kernel of its own (on the small cells a launch costs as much as the sums themselves).
// No block waits for another: each one counts itself done and the one that completes the
// count carries on.
#pragma once

#include "common.cuh"

namespace cbs {

// True in every thread of the block that is the last of `total` to arrive; what the others wrote
// before is then visible (read it with __ldcg).  The counter is left at zero.
__device__ __forceinline__ bool last_block(unsigned *count, unsigned total) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    const unsigned before = atomicAdd(count, 1u);
    last = before == total - 1;
    if (last) *count = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// alpha = rho / (p~, q) of one system's columns from the partial sums of (p~, q).
struct AlphaTail {
  unsigned *count = nullptr;                   // [n] blocks done
  const double2 *rho = nullptr;                // [n][L]
  double2 *alpha = nullptr;
  int *active = nullptr, *flags = nullptr;
  unsigned long long *sys_apply = nullptr;     // systems that went through an apply (profiling)
};

// part: [n][parts][L][ST] sums (re, im first); thread t of nt serves column t % L.  smem: 2 nt
// doubles.  All threads of the block take part; nt >= L.
template <int ST>
__device__ __forceinline__ void alpha_tail(const AlphaTail &a, const double *part, int s, int L, int parts, int t, int nt,
                                           double *smem) {
  const int c = t % L, ly = t / L, ry = min(nt / L, parts);   // no lane without a part
  const int64_t k0 = (int64_t)s * L + c;
  const double2 rho = ly == 0 ? a.rho[k0] : make_double2(0, 0);   // before the sums
  double gx = 0, gy = 0;
  if (ly < ry) {
#pragma unroll 4
    for (int k = ly; k < parts; k += ry) {
      const double *p = part + (((int64_t)s * parts + k) * L + c) * ST;
      gx += __ldcg(p);
      gy += __ldcg(p + 1);
    }
  }
  __syncthreads();
  smem[2 * t] = gx;
  smem[2 * t + 1] = gy;
  __syncthreads();
  if (ly != 0) return;
  for (int y = 1; y < ry; ++y) {
    gx += smem[2 * (y * L + c)];
    gy += smem[2 * (y * L + c) + 1];
  }
  if (c == 0 && a.sys_apply) atomicAdd(a.sys_apply, 1ull);   // system s went through this apply
  const int64_t k = (int64_t)s * L + c;
  double2 al = make_double2(0, 0);
  if (a.active[k]) {
    const double2 g = make_double2(gx, gy);
    const double g2 = cabs2(g);
    if (!(g2 > 0) || !isfinite(g2)) {
      a.flags[k] |= 2;
      a.active[k] = 0;
    } else {
      al = cdiv(rho, g);
    }
  }
  a.alpha[k] = al;
}

}  // namespace cbs
