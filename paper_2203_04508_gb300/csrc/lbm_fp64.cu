// The FP64 step (chemical-potential force, an equation of state, two lattices): four kernels that
// start early (programmatic dependent launch) -- chemical potential, collision, links, and the new
// state's density with its solid layers -- instead of a fork and a join of seven.
//
// GB300 has two FP64 lanes an SM and clock, so a warp's FP64 instruction takes 16 clocks: a node's
// some 220 (collision 150, BGK 105, density and psi' 53, chemical potential 18) are what a large lattice
// costs (512 x 512 BGK: 101 us a step, of which 80 are FP64 issue), and on a small one what counts is that they spread over all SMs and
// that nothing waits in between.  Hence one node a thread everywhere, in blocks of 128 (a 128 x 128
// lattice gives 128 of the 152 SMs a block, where tiles of 256 nodes gave 64: collision 19 -> 8 us),
// no halo formed twice (a fused tile would evaluate psi' or collide 1.7 times a node), stencils from
// the L1 cache instead of shared memory (the load units idle), and every load whose producer is two
// kernels back issued before the wait.  128 x 128: 52 -> 26 us a step, 512 x 512: 174 -> 101,
// 1024 x 1024 (MRT): 568 -> 410.
#include "lbm_device.cuh"
#include "lbm_fused.cuh"
#include "lbm_internal.h"
#include "lbm_phases.cuh"

namespace lbmgb {

namespace {

constexpr int D_BLOCK = 128;    // nodes of a block, along a row
constexpr int DC_X = 32;        // the collision's blocks: 32 x 4 nodes
constexpr int DB_BLOCK = 32;    // boundary nodes of a block

// Eq. 12 from the density and psi' of this state
__global__ void __launch_bounds__(D_BLOCK) k64_mu(const __grid_constant__ Lattice<double> L, int per_row) {
  const int y = blockIdx.x / per_row, x = (blockIdx.x - y * per_row) * D_BLOCK + threadIdx.x, n = y * L.pitch + x;
  const bool live = x < L.nx && L.kind[n] == KIND_FLUID;
  grid_wait();
  grid_launch();
  if (!live) return;
  const Stencil s = stencil_at(L, x, y);
  const double* r = L.rho;
  const double lap = lap4_of(r[n], r[s.xp1], r[s.xm1], r[s.xp2], r[s.xm2], r[s.yp1], r[s.ym1], r[s.yp2], r[s.ym2]);
  L.mu[n] = mu_of(L, L.psip[n], lap);
}

// force, collision and streaming.  Density and populations are complete when the chemical
// potential's kernel has started: they are fetched before the wait.
__global__ void __launch_bounds__(D_BLOCK) k64_collide(const __grid_constant__ Lattice<double> L, int cur, int per_row) {
  const int by = blockIdx.x / per_row, bx = blockIdx.x - by * per_row;
  const int x = bx * DC_X + threadIdx.x % DC_X, y = by * (D_BLOCK / DC_X) + threadIdx.x / DC_X;
  const int n = y * L.pitch + x;
  const bool live = x < L.nx && y < L.ny && L.kind[n] == KIND_FLUID;
  double fl[9], drx = 0.0, dry = 0.0;
  Stencil s{};
  if (live) {
    const double* f = L.f[cur];
#pragma unroll
    for (int i = 0; i < 9; ++i) fl[i] = f[i * L.plane + n];
    s = stencil_at(L, x, y);
    diff4(L.rho, s, drx, dry);
  }
  grid_wait();
  grid_launch();
  if (!live) return;
  const double* m = L.mu;
  const double dmx = diff4_of(m[s.xp1], m[s.xm1], m[s.xp2], m[s.xm2]), dmy = diff4_of(m[s.yp1], m[s.ym1], m[s.yp2], m[s.ym2]);
  collide_loaded(L, cur, x, y, fl, [&](double r, double& Fx, double& Fy) {
    Fx = force_cp(r, L.gx, dmx, drx);
    Fy = force_cp(r, L.gy, dmy, dry);
  });
}

__global__ void __launch_bounds__(DB_BLOCK) k64_links(const __grid_constant__ Lattice<double> L, int cur) {
  links<false, false>(L, cur, blockIdx.x * DB_BLOCK + threadIdx.x);
}

// The new state: the solid layers from the boundary nodes' densities in the first blocks, then
// density and psi' of the fluid nodes of lattice `cur`.
__global__ void __launch_bounds__(D_BLOCK) k64_state(const __grid_constant__ Lattice<double> L, int cur, int blocks2, int blocks1,
                                                     int per_row) {
  const int b = (int)blockIdx.x - (blocks2 + blocks1 + 1);
  if (b < 0) {
    solids<false, D_BLOCK>(L, blockIdx.x, blocks2, blocks1, 1);
    return;
  }
  const int y = b / per_row, x = (b - y * per_row) * D_BLOCK + threadIdx.x, n = y * L.pitch + x;
  const bool live = x < L.nx && L.kind[n] == KIND_FLUID;
  grid_wait();
  grid_launch();
  if (!live) return;
  const double* f = L.f[cur] + n;
  double v[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) v[i] = f[i * L.plane];
  const double r = density_of(L, v);
  L.rho_next[n] = r;
  L.psip[n] = psi_prime_shifted(L, r);
}

}  // namespace

int launches_fp64(const Lattice<double>& L) { return 3 + (L.n_bnodes > 0); }

cudaError_t launch_fp64_mu(const Lattice<double>& L, cudaStream_t s) {
  const int per_row = (L.nx + D_BLOCK - 1) / D_BLOCK;
  return launch_after(k64_mu, dim3((unsigned)(per_row * L.ny)), D_BLOCK, 0, s, L, per_row);
}

cudaError_t launch_fp64_step(const Lattice<double>& Lt, double* rho_next, int cur, cudaStream_t s, unsigned parts) {
  Lattice<double> L = Lt;
  L.rho_next = rho_next;
  const auto blocks = [](int n, int per) { return (n + per - 1) / per; };
  const int per_row = blocks(L.nx, D_BLOCK), b2 = blocks(8 * L.n_s2, D_BLOCK), b1 = blocks(L.n_s1, D_BLOCK);
  cudaError_t e = parts & PART_MU ? launch_fp64_mu(L, s) : cudaSuccess;
  const int across = blocks(L.nx, DC_X), grid = across * blocks(L.ny, D_BLOCK / DC_X);
  if (e == cudaSuccess && (parts & PART_PASS)) e = launch_after(k64_collide, dim3((unsigned)grid), D_BLOCK, 0, s, L, cur, across);
  if (e == cudaSuccess && L.n_bnodes > 0 && (parts & PART_LINKS))
    e = launch_after(k64_links, dim3((unsigned)blocks(L.n_bnodes, DB_BLOCK)), DB_BLOCK, 0, s, L, cur);
  if (e == cudaSuccess && (parts & PART_LAYERS))
    e = launch_after(k64_state, dim3((unsigned)(b2 + b1 + 1 + per_row * L.ny)), D_BLOCK, 0, s, L, cur ^ 1, b2, b1, per_row);
  return e;
}

}  // namespace lbmgb
