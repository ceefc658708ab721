// The cross-pair energy sums of one fragment, by one CTA of 256 threads.
#pragma once

#include "rimp2_internal.cuh"

namespace rimp2 {

// s + c += x with the rounding error of s kept in c
__device__ __forceinline__ void comp_add(double& s, double& c, double x) {
  const double t = s + x, b = t - s;
  c += (s - (t - b)) + (x - b);
  s = t;
}

// E = sum of n pair energies and (epos given) its opposite-spin part, both with compensated
// (TwoSum) sums in a fixed order: per thread, then over the lanes, then over the warps, the
// two side by side.  Only as many warps as have four values a lane take part: a sum across the
// lanes of one warp is 70 FP64 issues of 16 clocks, the SM's pipe takes one at a time.
// Copies the pair energies to epair where it is given; writes energy[idx], energy_os[idx] and
// the spin-component-scaled energy.
__device__ __forceinline__ void fragment_energy(const double* ep, const double* epos, long long n,
                                                double* epair, int idx, const Bases& bs) {
  __shared__ double sh[8][4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = n > 512 ? 8 : n > 256 ? 4 : n > 128 ? 2 : 1;
  double s = 0.0, c = 0.0, so = 0.0, co = 0.0;
  if (nw == 1 && warp != 0) return;
  for (long long e = threadIdx.x; warp < nw && e < n; e += 32 * nw) {
    const double y = __ldcg(ep + e);
    comp_add(s, c, y);
    if (epos) comp_add(so, co, __ldcg(epos + e));
    if (epair) epair[e] = y;
  }
  if (warp < nw) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double a = __shfl_xor_sync(0xffffffffu, s, off), b = __shfl_xor_sync(0xffffffffu, c, off);
      const double ao = __shfl_xor_sync(0xffffffffu, so, off), bo = __shfl_xor_sync(0xffffffffu, co, off);
      comp_add(s, c, a);
      comp_add(so, co, ao);
      c += b;
      co += bo;
    }
  }
  if (nw > 1) {
    if (lane == 0 && warp < nw) { sh[warp][0] = s; sh[warp][1] = c; sh[warp][2] = so; sh[warp][3] = co; }
    __syncthreads();
    if (warp != 0) return;
    const int w = lane & (nw - 1);
    s = sh[w][0]; c = sh[w][1]; so = sh[w][2]; co = sh[w][3];
    for (int off = nw / 2; off > 0; off >>= 1) {
      const double a = __shfl_xor_sync(0xffffffffu, s, off), b = __shfl_xor_sync(0xffffffffu, c, off);
      const double ao = __shfl_xor_sync(0xffffffffu, so, off), bo = __shfl_xor_sync(0xffffffffu, co, off);
      comp_add(s, c, a);
      comp_add(so, co, ao);
      c += b;
      co += bo;
    }
  }
  if (lane != 0) return;
  const double e = s + c;
  bs.energy[idx] = e;
  if (!epos) return;
  const double eos = so + co;
  if (bs.energy_os) bs.energy_os[idx] = eos;
  // spin-component scaling: c_os E_OS + c_ss E_SS with E_SS = E - E_OS
  if (bs.energy_scs) bs.energy_scs[idx] = bs.scs_os * eos + bs.scs_ss * (e - eos);
}

}  // namespace rimp2
