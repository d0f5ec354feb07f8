// CFL terms of a cell and the reductions of their maxima: per block into part
// (fixed layout, maxima are independent of the order), per instance in k_finalize.
#pragma once

#include "physics.cuh"

namespace amrvac {

// CFL terms of a conserved cell: running max of sum_d (|v_d| + c_f,d)/dx_d and
// of |v_d| + c_f,d.  1/rho, a^2 = gamma p/rho and the components B_i^2/rho are shared
// by the directions; b_t^2 is the sum of its two.  (As b^2 - B_d^2/rho it is as long,
// but for a field along d with a = b its rounding error stands alone under the inner
// root: 5e-9 of c_f in double, 1.2e-4 in float.)
template <class T, int DIM>
__device__ __forceinline__ void cfl_terms(const T* u, double gammad, T g, bool ff, float gm1f,
                                          const T* idx, T& smx, T& cmx) {
  T w[NV];
  cons2prim(gammad, u, w, ff, gm1f);
  const T ir = rcp_T(w[0]);
  const T a2 = g * w[4] * ir;
  const T b2[3] = {w[5] * w[5] * ir, w[6] * w[6] * ir, w[7] * w[7] * ir};
  const T byz = b2[1] + b2[2], bb = b2[0] + byz;
  const T dd = a2 - bb, sab = a2 + bb;
  T s = T(0);
#pragma unroll
  for (int d = 0; d < DIM; d++) {
    const T bt2 = d == 0 ? byz : b2[0] + b2[3 - d];
    const T cf = sqrt_T(T(0.5) * (sab + sqrt_T(dd * dd + T(4) * a2 * bt2)));
    const T spd = fabs(w[1 + d]) + cf;
    s += spd * idx[d];
    cmx = fmax(cmx, spd);
  }
  smx = fmax(smx, s);
}

// Per-warp maxima of the owners' two CFL terms merged into part_b[0..1] with
// atomicMax on the bit patterns (order-independent for values >= 0; NaN is
// dropped as fmax drops it).  part_b[0..1] are zeroed before the block's first
// barrier, the atomics come after its last one.
__device__ __forceinline__ void warp_max2_atomic(double smax, double cmax, double* part_b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    cmax = fmax(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (smax == smax)
      atomicMax((unsigned long long*)&part_b[0], (unsigned long long)__double_as_longlong(smax));
    if (cmax == cmax)
      atomicMax((unsigned long long*)&part_b[1], (unsigned long long)__double_as_longlong(cmax));
  }
}

// the same of the two CFL terms for a number of dimensions known at run time
template <class T>
__device__ __forceinline__ void cfl_terms_nd(int nd, const T* u, double gammad, T g, bool ff,
                                             float gm1f, const T* idx, T& smx, T& cmx) {
  if (nd == 3) cfl_terms<T, 3>(u, gammad, g, ff, gm1f, idx, smx, cmx);
  else if (nd == 2) cfl_terms<T, 2>(u, gammad, g, ff, gm1f, idx, smx, cmx);
  else cfl_terms<T, 1>(u, gammad, g, ff, gm1f, idx, smx, cmx);
}

// CTA maximum of the two CFL terms (every thread of the CTA takes part): thread 0
// stores it to part_b[0..1], or merges it there when several CTAs share a block
// (merge: part_b zeroed before; values >= 0, NaN dropped as fmax drops it)
__device__ __forceinline__ void cta_max2(double smax, double cmax, bool merge, double* part_b) {
  __shared__ double sh[32][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    cmax = fmax(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
  }
  if (lane == 0) {
    sh[warp][0] = smax;
    sh[warp][1] = cmax;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); w++) {
      smax = fmax(smax, sh[w][0]);
      cmax = fmax(cmax, sh[w][1]);
    }
    if (!merge) {
      part_b[0] = smax;
      part_b[1] = cmax;
    } else {
      if (smax == smax)
        atomicMax((unsigned long long*)&part_b[0], (unsigned long long)__double_as_longlong(smax));
      if (cmax == cmax)
        atomicMax((unsigned long long*)&part_b[1], (unsigned long long)__double_as_longlong(cmax));
    }
  }
  __syncthreads();  // sh is reused
}

}  // namespace amrvac
