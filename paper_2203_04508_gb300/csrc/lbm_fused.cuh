// Device code shared by the fused step and the separate passes.
#pragma once
#include "lbm_device.cuh"

namespace lbmgb {

// psi(rho_s) (1 + c_w) of a solid-layer node whose density is rho_s (pseudopotential force)
template <typename real>
__device__ __forceinline__ real psi_wall(const Lattice<real>& L, int n, real rs) {
  const int b = L.body[n];
  const double cw = b < L.n_cyl ? L.cyl[4 * b + 3] : L.cw_walls;
  return psi_of(L, rs) * (real(1) + (real)cw);
}

}  // namespace lbmgb
