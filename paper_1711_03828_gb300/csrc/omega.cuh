// omega.cuh -- the two-type field update of one cell (Eq. omega-fields), shared
// by the field kernels and the resident sweep, which evaluates it where it
// gathers; the roundings are written out so that every use gives the same bits.
#pragma once

#include "common.cuh"

namespace soma {

// omega_A (B false) or omega_B of a cell with packed counts v:
//   K^0: kappa_0 (phi_A + phi_B - 1) -/+ chi_0/2 (phi_A - phi_B)
//   K^1: kappa_0 (phi_A + phi_B - 1) + chi_0 phi_k of the other type k
__device__ __forceinline__ float omega_of(uint32_t v, bool B, float inv_rho, float kappa0,
                                          float half_chi0, int hamiltonian) {
  const float a = (float)(v & 0xFFFFu), b = (float)(v >> 16);
  const float phiA = __fmul_rn(a, inv_rho), phiB = __fmul_rn(b, inv_rho);
  if (hamiltonian) {
    const float comp = __fmul_rn(kappa0, __fsub_rn(__fadd_rn(phiA, phiB), 1.f));
    return __fmaf_rn(__fmul_rn(2.f, half_chi0), B ? phiA : phiB, comp);
  }
  const float d = __fmul_rn(half_chi0, __fmaf_rn(a, inv_rho, -phiB));
  return __fmaf_rn(kappa0, __fsub_rn(__fmaf_rn(a, inv_rho, phiB), 1.f), B ? d : -d);
}

// The same with the external potential and closed cells of f, as stored (WT).
template <typename WT>
__device__ __forceinline__ float omega_stored(const FieldArgs& f, uint32_t v, uint32_t c, bool B) {
  float w = omega_of(v, B, f.inv_rho, f.kappa0, f.half_chi0, f.hamiltonian);
  if (f.ext) w += f.ext[B ? f.g.cells + c : c];
  if (f.forbidden && f.forbidden[c]) w = __int_as_float(0x7F800000);   // +inf
  return load_cvt<WT>(store_cvt<WT>(w));
}

}  // namespace soma
