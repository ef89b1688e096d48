// Code shared by the fused step, the FP64 step and the separate passes.
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

// Programmatic dependent launch: a kernel of the step may start while the one before it still runs
// (grid_launch there), and reads or writes nothing that one touches before grid_wait, which waits
// for it to finish.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// a launch that may overlap the end of the one before it in the stream
template <typename... P, typename... A>
inline cudaError_t launch_after(void (*k)(P...), dim3 grid, int block, int smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = (size_t)smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = s ? 1 : 0;
  return cudaLaunchKernelEx(&c, k, P(args)...);
}
// Cut links of one boundary node a thread (phase_bc's arithmetic; the force from the planes the
// pass left, or PLANES false: formed again).  Latency is all it costs: what does not depend on the
// collision is done before the wait -- the node's record, set up with the geometry, and, PLANES false,
// its state and the links' force terms (FP64: 31.7 -> 29.6 us a step of 128 x 128; with PLANES the
// state's loads come after the wait: before it they delay the pass they overlap, 600 x 1200 800 -> 835
// us for 50 steps) -- and the loads behind it make one round.  The node's own populations stay in
// registers for its density.  Leaves one compensation sum per warp, which solids
// adds up.
template <bool PSEUDO, bool PLANES, int AA = 0, typename real>
__device__ __forceinline__ void links(const Lattice<real>& L, int cur, int b) {
  const bool live = b < L.n_bnodes;
  const int2 nd = live ? L.bnd[b] : make_int2(0, 0);
  const unsigned mask = live ? L.bmask[b] : 0u;
  real q[8];
#pragma unroll
  for (int i = 1; i < 9; ++i) q[i - 1] = mask & (1u << (i - 1)) ? L.bq[(i - 1) * (long long)L.bcap + b] : real(0);
  const int n = nd.x, x = nd.y;
  const real* fin = L.f[cur];
  real fl[9], ux = real(0), uy = real(0), r = real(1), inv_r = real(1), Fx = real(0), Fy = real(0);
  double carry = 0.0;
  auto load_state = [&]() {
    if constexpr (AA != 0) {
      // (the collision has overwritten the populations: the moments the step before left)
#pragma unroll
      for (int i = 0; i < 3; ++i) fl[i] = L.bmom[3 * b + i];
    } else {
#pragma unroll
      for (int i = 0; i < 9; ++i) fl[i] = fin[i * L.plane + n];
    }
    carry = L.carry[b];
  };
  real F[8];   // the links' force terms
  auto terms = [&]() {
    real drho, jx, jy;
    if constexpr (AA != 0) {
      drho = fl[0];
      jx = fl[1];
      jy = fl[2];
    } else {
      moments(fl, drho, jx, jy);
    }
    r = L.rho_ref + drho;
    if constexpr (!PLANES) force_at<real, PSEUDO>(L, x, n / L.pitch, r, Fx, Fy);
    inv_r = real(1) / r;
    ux = mul_rn(jx, inv_r);
    uy = mul_rn(jy, inv_r);
    const real dux = mul_rn(Fx, inv_r), duy = mul_rn(Fy, inv_r);
#pragma unroll
    for (int i = 1; i < 9; ++i) F[i - 1] = mask & (1u << (i - 1)) ? edm_term<real>(i, r, ux, uy, dux, duy) : real(0);
  };
  if (!PLANES && live) {
    load_state();
    terms();
  }
  grid_wait();
  grid_launch();
  double sum = 0.0;
  if (live) {
    real* fout = L.f[cur ^ 1];
    // offsets to the neighbours (periodic in x, and in y without walls)
    const int xm = x == 0 ? L.nx - 1 : -1, xp = x == L.nx - 1 ? 1 - L.nx : 1;
    const int ym = !L.walls && n < L.pitch ? L.plane - L.pitch : -L.pitch;
    const int yp = !L.walls && n >= L.plane - L.pitch ? L.pitch - L.plane : L.pitch;
    auto nb = [&](int dx, int dy) { return n + (dx < 0 ? xm : dx > 0 ? xp : 0) + (dy < 0 ? ym : dy > 0 ? yp : 0); };
    real g[9], a[8], cc[8];
    // Slots of the new state: f_i(x) in slot i of x, or (AA 1: the step from the natural order)
    // slot opp(i) of x - e_i
    auto own = [&](int i) { return AA == 1 ? opp(i) * L.plane + nb(-ex(i), -ey(i)) : i * L.plane + n; };
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = fout[own(i)];
    if constexpr (PLANES) {
      load_state();
      Fx = L.fx[n];
      Fy = L.fy[n];
    }
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      a[i - 1] = cc[i - 1] = real(0);
      if (mask & (1u << (i - 1))) {
        a[i - 1] = fout[AA == 1 ? opp(i) * L.plane + n : i * L.plane + nb(ex(i), ey(i))];
        cc[i - 1] = fout[AA == 1 ? i * L.plane + n : opp(i) * L.plane + nb(-ex(i), -ey(i))];
      }
    }
    if constexpr (PLANES) terms();
    real v[8];
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      if (!(mask & (1u << (i - 1)))) continue;
      v[i - 1] = link_rule<real>(L.bc, q[i - 1], (mask >> (i + 7)) & 1u, a[i - 1], g[i], cc[i - 1], F[i - 1]);
      sum += (double)a[i - 1] - (double)v[i - 1];
    }
    // (no link reads a slot another link of the node writes: b2 counts only where x2 is fluid)
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      if (!(mask & (1u << (i - 1)))) continue;
      g[opp(i)] = v[i - 1];
      fout[own(opp(i))] = v[i - 1];
    }
    if (L.bc == BC_PRESENT || L.bc == BC_MIBC) {
      const double t = (double)g[0] + sum + carry;
      g[0] = (real)t;
      L.carry[b] = t - (double)g[0];
      fout[n] = g[0];
    } else {
      sum = 0.0;
    }
    if constexpr (AA != 0) moments(g, L.bmom[3 * b], L.bmom[3 * b + 1], L.bmom[3 * b + 2]);
    const real rn = density_of(L, g);
    L.rho_b[b] = rn;
    L.rho_next[n] = PSEUDO ? psi_of(L, rn) : rn;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) L.partials[b >> 5] = sum;
}

// Both solid layers from the boundary nodes' densities in rho_b (every fluid neighbour of a
// first-layer node is a boundary node), into the density plane (psi with the wall factor into the
// psi plane).  A second-layer node forms its first-layer neighbours' densities again, one a lane of
// its eight lanes, and adds them in phase_solid's order.  The last block adds the links'
// compensation sums in the order of k_bc's two-level sum, and steps the counter; steps == 0 leaves
// that out (the layers of a new state).
template <bool PSEUDO, int BLOCK, typename real>
__device__ __forceinline__ void solids(const Lattice<real>& L, int blk, int blocks2, int blocks1, int steps) {
  __shared__ double red[32];
  auto first = [&](unsigned m, real winv, const int (&nb)[8]) {
    real acc = real(0);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (m & (1u << i)) acc = fma_rn((real)wgt(i + 1), L.rho_b[nb[i]], acc);
    return acc * winv;
  };
  auto record = [&](int k, unsigned& m, real& winv, int (&nb)[8]) {
    m = L.s1mask[k];
    winv = L.s1winv[k];
    const int4 u = *reinterpret_cast<const int4*>(L.s1nb + 8 * k), w = *reinterpret_cast<const int4*>(L.s1nb + 8 * k + 4);
    nb[0] = u.x; nb[1] = u.y; nb[2] = u.z; nb[3] = u.w;
    nb[4] = w.x; nb[5] = w.y; nb[6] = w.z; nb[7] = w.w;
  };
  if (blk < blocks2) {
    const int t = blk * BLOCK + threadIdx.x, k = t >> 3, lane = t & 7;
    unsigned m2 = 0, m = 0;
    real winv2 = real(0), winv = real(0);
    int nb[8], n = 0;
    if (k < L.n_s2) {
      m2 = L.s2mask[k];
      winv2 = L.s2winv[k];
      n = L.s2node[k];
      if (m2 & (1u << lane)) record(L.s2nb[8 * k + lane], m, winv, nb);
    }
    grid_wait();
    grid_launch();
    const real v = first(m, winv, nb);
    real acc = real(0);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const real vi = __shfl_sync(0xffffffffu, v, i, 8);
      if (m2 & (1u << i)) acc = fma_rn((real)wgt(i + 1), vi, acc);
    }
    const real rs = acc * winv2;
    if (k < L.n_s2 && lane == 0) L.rho_next[n] = PSEUDO ? psi_wall(L, n, rs) : rs;
  } else if (blk < blocks2 + blocks1) {
    const int k = (blk - blocks2) * BLOCK + threadIdx.x;
    unsigned m = 0;
    real winv = real(0);
    int nb[8], n = 0;
    if (k < L.n_s1) {
      n = L.s1node[k];
      record(k, m, winv, nb);
    }
    grid_wait();
    grid_launch();
    const real rs = first(m, winv, nb);
    if (k < L.n_s1) L.rho_next[n] = PSEUDO ? psi_wall(L, n, rs) : rs;
  } else {
    grid_wait();
    grid_launch();
    if (steps) {
      // k_bc's blocks of eight warps: their warps' sums in block_sum's tree, then the blocks'
      const int warps = (L.n_bnodes + 31) / 32, chunks = (warps + 7) / 8;
      constexpr int SUM_BLOCK = 256, PARTS = SUM_BLOCK / BLOCK;   // k_bc's last block; each thread's share of it
      static_assert(PARTS == 1 || PARTS == 2, "block_sum's tree over 8 warps begins with pairs (j, j + 4)");
      double v[PARTS];
#pragma unroll
      for (int p = 0; p < PARTS; ++p) {
        v[p] = 0.0;
        for (int k = threadIdx.x + p * BLOCK; k < chunks; k += SUM_BLOCK) {
          double w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) w[j] = 8 * k + j < warps ? L.partials[8 * k + j] : 0.0;
          v[p] += ((w[0] + w[4]) + (w[2] + w[6])) + ((w[1] + w[5]) + (w[3] + w[7]));
        }
        if constexpr (PARTS == 2) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v[p] += __shfl_down_sync(0xffffffffu, v[p], o);
        }
      }
      double mine = v[0];
      if constexpr (PARTS == 2) mine = (threadIdx.x & 31) == 0 ? v[0] + v[1] : 0.0;
      const double total = block_sum(mine, red);
      if (threadIdx.x == 0) {
        const unsigned long long st = *L.step_ctr;
        L.dM_ring[st % DM_RING] = total;
        L.dM_ring[DM_RING] = total;
        *L.step_ctr = st + 1;
      }
    }
  }
}

}  // namespace lbmgb
