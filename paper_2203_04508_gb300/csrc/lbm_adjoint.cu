// Reverse (adjoint) mode of one time step, and the droplet objective it is seeded from.
//
// Forward step t (lbm_phases.cuh):  f^t -> rho -> (Eq. 15) solid rho -> (Eq. 12) mu -> (Eq. 9) F
//   -> collision + exact-difference forcing (Eq. 4, 13) -> streaming (Eq. 5) -> cut links
//   (Eqs. 16-17) -> compensation (Eq. 18) -> f^{t+1}.
// Given lambda^{t+1} = dJ/df^{t+1} this file produces lambda^t = dJ/df^t and adds the step's
// share of dJ/d(wall chemical potential) and dJ/d(cylinder centre) (the centre enters only
// through the cut fractions q: |x1 + q e - c|^2 = r^2 gives dq/dc = p / (p . e) with
// p = x1 + q e - c).  The reverse phases run in the opposite order of the forward ones:
//   adj_bc      links and Eq. 18 (per boundary node; the post-collision values a, b2, c the
//               links used are read back from f^{t+1}, where the step left them)
//   adj_collide streaming (pulled) + collision + forcing, per fluid node
//   adj_force   Eq. 9: the force's dependence on mu and rho at the stencil neighbours (gather)
//   adj_mu      Eq. 12: mu's dependence on rho (gather); wall mu -> dJ/d(offset)
//   adj_solid   Eq. 15, second layer then first layer (scatter, atomics)
// FP64 runs them as six kernels, FP32 as four: k_adj_links, k_adj_nodes, k_adj_fields (adj_force and
// adj_mu) and k_adj_layers.
// The density's share of lambda^t, Lrho (one value per node, the same for all nine
// populations), is not added to the nine planes: lambda^t is kept as (nine planes, Lrho) and the
// next reverse step adds Lrho where it reads lambda.  The forward quantities of step t (rho,
// solid rho, mu) are those the recomputation of the segment stored for that step.
#include "lbm_fused.cuh"
#include "lbm_internal.h"
#include "lbm_phases.cuh"

namespace lbmgb {

constexpr int ADJ_BLOCK = 256;

template <typename real>
__device__ __forceinline__ bool is_field_node(uint8_t k) {
  return k == KIND_FLUID || k == KIND_SOLID1 || k == KIND_SOLID2;
}

// dpsi'/drho = (dp0/drho) / rho (Eq. 7)
template <typename real>
__device__ __forceinline__ real psi_second(const Lattice<real>& L, real r) {
  if (L.eos == EOS_CS) {
    const real eta = L.b * r * real(0.25), om = real(1) - eta;
    const real om2 = om * om;
    const real h1 = (real(1) + eta * (real(4) + eta * (real(4) + eta * (real(-4) + eta)))) / (om2 * om2);
    return L.RT * h1 / r - real(2) * L.a;
  }
  const real x = L.b * r, om = real(1) - x;
  const real D = real(1) + real(2) * x - x * x;
  return L.RT / (r * om * om) - L.aalpha * (real(2) + real(2) * x) / (D * D);
}

// Adjoint of collide_node at one node: lt = dJ/d(post-collision populations); adds
// dJ/d(populations) (direct part) to lf, and dJ/d(delta rho), dJ/dj, dJ/dF to the scalars.
template <typename real>
__device__ __forceinline__ void collide_adjoint(const Lattice<real>& L, real r, real jx, real jy, real Fx, real Fy,
                                                const real (&lt)[9], real (&lf)[9], real& lrho, real& ljx, real& ljy,
                                                real& lFx, real& lFy) {
  const real ir = real(1) / r, ir2 = ir * ir;
  // the equilibrium depends on lt only through its moments with the weights: sum w lt, sum w e lt,
  // sum w e e lt (w e_x^2 and w e_y^2 share the diagonals)
  const real s13 = lt[1] + lt[3], s24 = lt[2] + lt[4], s57 = lt[5] + lt[7], s68 = lt[6] + lt[8];
  const real d13 = lt[1] - lt[3], d24 = lt[2] - lt[4], d57 = lt[5] - lt[7], d68 = lt[6] - lt[8];
  const real w1 = real(1.0 / 9.0), w5 = real(1.0 / 36.0);
  const real sd = w5 * (s57 + s68);
  const real S0 = real(4.0 / 9.0) * lt[0] + w1 * (s13 + s24) + sd;
  const real Sx = w1 * d13 + w5 * (d57 - d68), Sy = w1 * d24 + w5 * (d57 + d68);
  const real Sxx = w1 * s13 + sd, Syy = w1 * s24 + sd, Sxy = w5 * (s57 - s68);
  // sum w lt (1 + ...) at momentum (mx, my): its derivatives by rho and by the momentum
  auto eq_adjoint = [&](real mx, real my, real& gr, real& gx, real& gy) {
    const real vx = mx * ir, vy = my * ir;
    gr = S0 * (real(1) + real(1.5) * (vx * vx + vy * vy)) - real(4.5) * (Sxx * vx * vx + real(2) * (Sxy * vx * vy) + Syy * vy * vy);
    gx = real(3) * (Sx - vx * S0) + real(9) * (vx * Sxx + vy * Sxy);
    gy = real(3) * (Sy - vy * S0) + real(9) * (vx * Sxy + vy * Syy);
  };
  // equilibrium at J' = j + F (the exact-difference term folded in)
  {
    real gr, gx, gy;
    eq_adjoint(jx + Fx, jy + Fy, gr, gx, gy);
    lrho += gr;
    ljx += gx;
    ljy += gy;
    lFx += gx;
    lFy += gy;
  }
  if (L.coll == COLL_MRT) {
    // moment-space adjoint of M^-1 (I - S) (M f - m_eq): nu_k = (M lt)_k / D_k (1 - s_k)
    const real me = (real(-4) * lt[0] - (s13 + s24) + real(2) * (s57 + s68)) * real(1.0 / 36.0) * (real(1) - L.s_e);
    const real mp = (real(4) * lt[0] - real(2) * (s13 + s24) + (s57 + s68)) * real(1.0 / 36.0) * (real(1) - L.s_eps);
    const real mqx = (real(-2) * d13 + (d57 - d68)) * real(1.0 / 12.0) * (real(1) - L.s_q);
    const real mqy = (real(-2) * d24 + (d57 + d68)) * real(1.0 / 12.0) * (real(1) - L.s_q);
    const real mxx = (s13 - s24) * real(0.25) * (real(1) - L.s_nu);
    const real mxy = (s57 - s68) * real(0.25) * (real(1) - L.s_nu);
    // M^T nu
    const real ax = -me - real(2) * mp, dg = real(2) * me + mp, qp = mqx + mqy, qm = mqx - mqy;
    lf[0] += real(4) * (mp - me);
    lf[1] += ax - real(2) * mqx + mxx;
    lf[2] += ax - real(2) * mqy - mxx;
    lf[3] += ax + real(2) * mqx + mxx;
    lf[4] += ax + real(2) * mqy - mxx;
    lf[5] += dg + qp + mxy;
    lf[6] += dg - qm - mxy;
    lf[7] += dg - qp + mxy;
    lf[8] += dg + qm - mxy;
    // minus the equilibrium moments' dependence on (delta rho, j)
    const real j2 = jx * jx + jy * jy;
    lrho -= me * (real(-2) - real(3) * j2 * ir2) + mp * (real(1) + real(3) * j2 * ir2) -
            mxx * (jx * jx - jy * jy) * ir2 - mxy * jx * jy * ir2;
    const real ep = real(6) * ir * (me - mp);
    ljx -= ep * jx - mqx + mxx * real(2) * jx * ir + mxy * jy * ir;
    ljy -= ep * jy - mqy - mxx * real(2) * jy * ir + mxy * jx * ir;
  } else {
    const real keep = real(1) - L.omega;
    real gr, gx, gy;
    eq_adjoint(jx, jy, gr, gx, gy);
    lrho -= keep * gr;
    ljx -= keep * gx;
    ljy -= keep * gy;
#pragma unroll
    for (int i = 0; i < 9; ++i) lf[i] += keep * lt[i];
  }
}

// populations, moments and force of node n of the stored state (the forward arithmetic)
template <typename real>
__device__ __forceinline__ void node_state(const Lattice<real>& L, int x, int y, real (&f)[9], real& r, real& drho,
                                           real& jx, real& jy, real& Fx, real& Fy) {
  const int n = y * L.pitch + x;
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = L.f[0][i * L.plane + n];
  moments(f, drho, jx, jy);
  r = L.rho_ref + drho;
  force_at(L, x, y, r, Fx, Fy);
}

// ---- adj_bc: one thread per boundary node -------------------------------------------------
template <typename real>
__global__ void __launch_bounds__(ADJ_BLOCK) k_adj_bc(Lattice<real> L, AdjBuffers A) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= L.n_bnodes) return;
  const int n = L.bnode[b];
  const int x = n % L.pitch, y = n / L.pitch;
  const real* lin = static_cast<const real*>(A.lam_in);
  const real lrn = static_cast<const real*>(A.Lrho)[n];   // density share of lambda^{t+1} at x1
  real* lbc = static_cast<real*>(A.lam_bc);
  real f[9], r, drho, jx, jy, Fx, Fy;
  node_state(L, x, y, f, r, drho, jx, jy, Fx, Fy);
  // f^{t+1} holds the post-collision values the links used: a = f~_i(x1) parked in the solid
  // node's slot, b2 = f~_i(x2) streamed into x1, c = f~_ibar(x1) streamed into x2 (the link
  // phase overwrites none of them where they are used)
  const real* __restrict__ fn = L.f[1];
  const bool comp = L.bc == BC_PRESENT || L.bc == BC_MIBC;
  const real wF = L.bc == BC_PRESENT ? real(1) : real(0);
  const real l0 = comp ? lin[n] + lrn : real(0);
  const real ir = real(1) / r;
  real lrho = 0, ljx = 0, ljy = 0, lFx = 0, lFy = 0;
  for (int l = L.bstart[b]; l < L.bstart[b + 1]; ++l) {
    const int i = L.ldir[l];
    const int ib = opp(i);
    const real q = L.lq[l];
    const int x2 = node_at(L, x - ex(i), y - ey(i));
    const int xs = node_at(L, x + ex(i), y + ey(i));
    const real a = fn[i * L.plane + xs], c = fn[ib * L.plane + x2];
    const real exi = real(ex(i)), eyi = real(ey(i));
    const real eF = exi * Fx + eyi * Fy, ej = exi * jx + eyi * jy, eJ = ej + eF;
    const real Jx = jx + Fx, Jy = jy + Fy;
    const real Fi = real(wgt(i)) * (real(3) * eF + real(4.5) * (eJ * eJ - ej * ej) * ir -
                                    real(1.5) * ((Jx * Jx + Jy * Jy) - (jx * jx + jy * jy)) * ir);
    const real lR = (lin[ib * L.plane + n] + lrn) - l0;
    real dA = 0, dB = 0, dC = 0, dF = 0, dQ = 0;
    if (L.bc == BC_HBB || (q < real(0.5) && !L.lx2f[l])) {
      dA = 1;
    } else if (q < real(0.5)) {
      const real b2 = fn[i * L.plane + n];
      dA = real(2) * q;
      dB = real(1) - real(2) * q;
      dF = wF * (real(1) - real(2) * q);
      dQ = real(2) * a - real(2) * b2 - real(2) * wF * Fi;
    } else {
      const real i2q = real(1) / (real(2) * q);
      dA = i2q;
      dC = (real(2) * q - real(1)) * i2q;
      dF = wF * dC;
      dQ = (c - a + wF * Fi) * i2q * i2q * real(2);
    }
    atomicAdd(&lbc[i * L.plane + n], dA * lR + l0);
    if (dB != real(0)) atomicAdd(&lbc[i * L.plane + x2], dB * lR);
    if (dC != real(0)) atomicAdd(&lbc[ib * L.plane + n], dC * lR);
    // F_i = w [3 e.F + 4.5 ((e.J')^2 - (e.j)^2)/rho - 1.5 (|J'|^2 - |j|^2)/rho], J' = j + F
    const real lFi = dF * lR;
    if (lFi != real(0)) {
      const real w = real(wgt(i)) * lFi;
      lFx += w * (real(3) * exi + real(9) * eJ * exi * ir - real(3) * Jx * ir);
      lFy += w * (real(3) * eyi + real(9) * eJ * eyi * ir - real(3) * Jy * ir);
      ljx += w * (real(9) * eF * exi - real(3) * Fx) * ir;
      ljy += w * (real(9) * eF * eyi - real(3) * Fy) * ir;
      lrho -= w * (real(4.5) * (eJ * eJ - ej * ej) - real(1.5) * ((Jx * Jx + Jy * Jy) - (jx * jx + jy * jy))) * ir * ir;
    }
    // dJ/dq -> dJ/dc of the cylinder this link cuts
    const int bd = L.body[xs];
    if (bd >= 0 && bd < A.n_cyl && dQ != real(0)) {
      const double gq = (double)dQ * (double)lR;
      const double px = (double)x - L.cyl[4 * bd] + (double)q * ex(i);
      const double py = (double)y - L.cyl[4 * bd + 1] + (double)q * ey(i);
      const double pe = px * ex(i) + py * ey(i);
      atomicAdd(&A.grad[A.n_cyl + 1 + 2 * bd], gq * px / pe);
      atomicAdd(&A.grad[A.n_cyl + 2 + 2 * bd], gq * py / pe);
    }
  }
  real* lrj = static_cast<real*>(A.lrj);
  lrj[n] = lrho;
  lrj[L.plane + n] = ljx;
  lrj[2 * L.plane + n] = ljy;
  real* lF = static_cast<real*>(A.lamF);
  lF[n] = lFx;
  lF[L.plane + n] = lFy;
}

// ---- adj_collide: one thread per fluid node ---------------------------------------------
template <typename real>
__global__ void __launch_bounds__(ADJ_BLOCK) k_adj_collide(Lattice<real> L, AdjBuffers A) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= L.nx) return;
  const int n = y * L.pitch + x;
  if (L.kind[n] != KIND_FLUID) return;
  const real* lin = static_cast<const real*>(A.lam_in);
  const real* lrp = static_cast<const real*>(A.Lrho);   // density share of lambda^{t+1}
  real* lout = static_cast<real*>(A.lam_out);
  real* lbc = static_cast<real*>(A.lam_bc);
  real* lrj = static_cast<real*>(A.lrj);
  real* lF = static_cast<real*>(A.lamF);
  real f[9], r, drho, jx, jy, Fx, Fy;
  node_state(L, x, y, f, r, drho, jx, jy, Fx, Fy);
  // adjoint of the post-collision populations: pulled back from where they streamed to
  real lt[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int yy = y + ey(i);
    real v = real(0);
    if (!L.walls || (yy >= 0 && yy < L.ny)) {
      const int m = node_at(L, x + ex(i), yy);
      if (L.kind[m] == KIND_FLUID) v = lin[i * L.plane + m] + lrp[m];
    }
    lt[i] = v;
  }
  real lrho = 0, ljx = 0, ljy = 0, lFx = 0, lFy = 0;
  const uint8_t t = A.bct[n];
  if (t & 1) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      lt[i] += lbc[i * L.plane + n];
      lbc[i * L.plane + n] = real(0);
    }
  }
  if (t & 2) {
    lrho = lrj[n];
    ljx = lrj[L.plane + n];
    ljy = lrj[2 * L.plane + n];
    lFx = lF[n];
    lFy = lF[L.plane + n];
  }
  real lf[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) lf[i] = real(0);
  collide_adjoint(L, r, jx, jy, Fx, Fy, lt, lf, lrho, ljx, ljy, lFx, lFy);
#pragma unroll
  for (int i = 0; i < 9; ++i) lout[i * L.plane + n] = lf[i] + lrho + real(ex(i)) * ljx + real(ey(i)) * ljy;
  lF[n] = lFx;
  lF[L.plane + n] = lFy;
}

// ---- adj_force: Eq. 9, gathered at every node that carries rho or mu ------------------------
template <typename real>
__global__ void __launch_bounds__(ADJ_BLOCK) k_adj_force(Lattice<real> L, AdjBuffers A) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= L.nx) return;
  const int n = y * L.pitch + x;
  const uint8_t k = L.kind[n];
  if (!is_field_node<real>(k)) return;
  const real* lF = static_cast<const real*>(A.lamF);
  const real* lFy = lF + L.plane;
  real* Lmu = static_cast<real*>(A.Lmu);
  real* Lrho = static_cast<real*>(A.Lrho);
  real lm = 0, lr = 0;
  if (L.eos != EOS_NONE) {
    // gradient coefficients c_{+1} = 8/12, c_{+2} = -1/12, c_{-d} = -c_d; the neighbour m - d
    // sees this node at offset +d.  Only fluid neighbours carry a force (and so dJ/dF); the
    // density plane holds no value at deep solid nodes, so they are skipped, not multiplied
    // by zero.
    const real c1 = real(8.0 / 12.0), c2 = real(-1.0 / 12.0), cs2 = real(1.0 / 3.0);
    const int dd[4] = {1, -1, 2, -2};
    const real cc[4] = {c1, -c1, c2, -c2};
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) {
      const int yy = y - dd[k2];
      if (!L.walls || (yy >= 0 && yy < L.ny)) {
        const int m = node_at(L, x, yy);
        if (L.kind[m] == KIND_FLUID) {
          const real ly = lFy[m];
          lm -= cc[k2] * (L.rho[m] * ly);
          lr += cs2 * cc[k2] * ly;
        }
      }
      const int mx = node_at(L, x - dd[k2], y);
      if (L.kind[mx] == KIND_FLUID) {
        const real lx = lF[mx];
        lm -= cc[k2] * (L.rho[mx] * lx);
        lr += cs2 * cc[k2] * lx;
      }
    }
  }
  if (k == KIND_FLUID) {
    real gmx = 0, gmy = 0;
    if (L.eos != EOS_NONE) {
      Stencil s = stencil_at(L, x, y);
      grad4(L.mu, s, gmx, gmy);
    }
    lr += lF[n] * (L.gx - gmx) + lFy[n] * (L.gy - gmy);
  }
  Lmu[n] = lm;
  Lrho[n] = lr;
}

// ---- adj_mu: Eq. 12 gathered; wall chemical potential -> dJ/d(offset) ------------------------
template <typename real>
__global__ void __launch_bounds__(ADJ_BLOCK) k_adj_mu(Lattice<real> L, AdjBuffers A) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= L.nx) return;
  const int n = y * L.pitch + x;
  const uint8_t k = L.kind[n];
  if (!is_field_node<real>(k) || L.eos == EOS_NONE) return;
  const real* Lmu = static_cast<const real*>(A.Lmu);
  real* Lrho = static_cast<real*>(A.Lrho);
  // mu_m = k^2 psi'(rho_m) - kappa sum_d l_d rho_{m+d}; l_0 = -60/12 (both axes), l_{+-1} =
  // 16/12, l_{+-2} = -1/12; only fluid m carry this dependence
  real acc = 0;
  const int dd[4] = {1, -1, 2, -2};
  const real ll[4] = {real(16.0 / 12.0), real(16.0 / 12.0), real(-1.0 / 12.0), real(-1.0 / 12.0)};
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) {
    const int yy = y - dd[k2];
    if (!L.walls || (yy >= 0 && yy < L.ny)) {
      const int m = node_at(L, x, yy);
      if (L.kind[m] == KIND_FLUID) acc += ll[k2] * Lmu[m];
    }
    const int mx = node_at(L, x - dd[k2], y);
    if (L.kind[mx] == KIND_FLUID) acc += ll[k2] * Lmu[mx];
  }
  real lr = Lrho[n] - L.kappa * acc;
  if (k == KIND_FLUID) {
    lr += -L.kappa * real(-60.0 / 12.0) * Lmu[n] + L.k2 * psi_second(L, L.rho[n]) * Lmu[n];
  } else {
    const int bd = L.body[n];
    atomicAdd(&A.grad[bd >= 0 && bd < A.n_cyl ? bd : A.n_cyl], (double)Lmu[n]);
  }
  Lrho[n] = lr;
}

// ---- adj_solid: Eq. 15 in reverse (second layer, then first) -------------------------------
template <typename real>
__global__ void __launch_bounds__(ADJ_BLOCK) k_adj_solid(Lattice<real> L, AdjBuffers A, int layer) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= (layer == 1 ? L.n_s1 : L.n_s2)) return;
  const int n = layer == 1 ? L.s1node[j] : L.s2node[j];
  const uint8_t m = layer == 1 ? L.s1mask[j] : L.s2mask[j];
  const real winv = layer == 1 ? L.s1winv[j] : L.s2winv[j];
  real* Lrho = static_cast<real*>(A.Lrho);
  const real v = Lrho[n] * winv;
  const int x = n % L.pitch, y = n / L.pitch;
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (m & (1u << (i - 1))) atomicAdd(&Lrho[node_at(L, x + ex(i), y + ey(i))], real(wgt(i)) * v);
}

// ---------------------------------------------------------------------------------------
// FP32: four kernels a reverse step that start early (programmatic dependent launch).  Whatever the
// recomputation left -- populations, density, chemical potential -- and the geometry is complete
// before the sweep of a segment begins, so each kernel fetches its share before it waits for the
// one it follows, and only lambda is read behind the wait.  They replace a chain of six whose
// latency was what a 512 x 512 lattice paid for: 100 steps with their recomputation took 6.3 ms and take 3.0.

// adds v to grad[k] (k < 0: nothing); a warp whose nodes all belong to one body adds once
__device__ __forceinline__ void add_by_body(double* grad, int k, double v) {
  const unsigned any = __ballot_sync(0xffffffffu, k >= 0);
  if (!any) return;
  const int lead = __shfl_sync(0xffffffffu, k, __ffs(any) - 1);
  if (__all_sync(0xffffffffu, k < 0 || k == lead)) {
    if (k < 0) v = 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&grad[lead], v);
  } else if (k >= 0) {
    atomicAdd(&grad[k], v);
  }
}

// k_adj_bc with the links by node (as the fused step's): one round of loads instead of one a link
constexpr int AL_BLOCK = 32;
__global__ void __launch_bounds__(AL_BLOCK) k_adj_links(const __grid_constant__ Lattice<float> L,
                                                        const __grid_constant__ AdjBuffers A) {
  const int b = blockIdx.x * AL_BLOCK + threadIdx.x;
  const bool live = b < L.n_bnodes;
  const int2 nd = live ? L.bnd[b] : make_int2(0, 0);
  const unsigned mask = live ? L.bmask[b] : 0u;
  const int n = nd.x, x = nd.y, y = n / L.pitch;
  const int xm = x == 0 ? L.nx - 1 : -1, xp = x == L.nx - 1 ? 1 - L.nx : 1;
  const int ym = !L.walls && y == 0 ? L.plane - L.pitch : -L.pitch;
  const int yp = !L.walls && y == L.ny - 1 ? L.pitch - L.plane : L.pitch;
  auto nb = [&](int dx, int dy) { return n + (dx < 0 ? xm : dx > 0 ? xp : 0) + (dy < 0 ? ym : dy > 0 ? yp : 0); };
  // f^{t+1} holds the post-collision values the links used (see k_adj_bc): a, b2, c
  const float* __restrict__ fn = L.f[1];
  float q[8], a[8], b2[8], cc[8], f[9];
  int bd[8];
  double2 dc[8];   // q's derivative by the cylinder's centre (k_adj_geometry)
  float r = 1.f, drho = 0.f, jx = 0.f, jy = 0.f, Fx = 0.f, Fy = 0.f;
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const bool on = mask & (1u << (i - 1));
    q[i - 1] = on ? L.bq[(i - 1) * (long long)L.bcap + b] : 0.f;
    a[i - 1] = on ? fn[i * L.plane + nb(ex(i), ey(i))] : 0.f;
    b2[i - 1] = on ? fn[i * L.plane + n] : 0.f;
    cc[i - 1] = on ? fn[opp(i) * L.plane + nb(-ex(i), -ey(i))] : 0.f;
    bd[i - 1] = on && A.n_cyl > 0 ? L.body[nb(ex(i), ey(i))] : -1;
    dc[i - 1] = bd[i - 1] >= 0 && bd[i - 1] < A.n_cyl ? A.dqdc[(i - 1) * (long long)L.bcap + b] : make_double2(0.0, 0.0);
  }
  if (live) node_state(L, x, y, f, r, drho, jx, jy, Fx, Fy);
  grid_wait();
  grid_launch();
  if (!live) return;
  const float* lin = static_cast<const float*>(A.lam_in);
  const float lrn = static_cast<const float*>(A.Lrho)[n];   // density share of lambda^{t+1} at x1
  float* lbc = static_cast<float*>(A.lam_bc);
  const bool comp = L.bc == BC_PRESENT || L.bc == BC_MIBC;
  const float wF = L.bc == BC_PRESENT ? 1.f : 0.f;
  float li[8];
#pragma unroll
  for (int i = 1; i < 9; ++i) li[i - 1] = mask & (1u << (i - 1)) ? lin[opp(i) * L.plane + n] : 0.f;
  const float l0 = comp ? lin[n] + lrn : 0.f;
  const float ir = 1.0f / r, Jx = jx + Fx, Jy = jy + Fy;
  const float dJ2 = (Jx * Jx + Jy * Jy) - (jx * jx + jy * jy);
  float lrho = 0, ljx = 0, ljy = 0, lFx = 0, lFy = 0, own[9];
  int body = -1;
  double gx = 0.0, gy = 0.0;
  auto flush = [&]() {
    if (body < 0) return;
    atomicAdd(&A.grad[A.n_cyl + 1 + 2 * body], gx);
    atomicAdd(&A.grad[A.n_cyl + 2 + 2 * body], gy);
  };
#pragma unroll
  for (int i = 0; i < 9; ++i) own[i] = 0.f;
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    if (!(mask & (1u << (i - 1)))) continue;
    const float qi = q[i - 1];
    const float exi = float(ex(i)), eyi = float(ey(i));
    const float eF = exi * Fx + eyi * Fy, ej = exi * jx + eyi * jy, eJ = ej + eF;
    const float Fi = float(wgt(i)) * (3.f * eF + 4.5f * (eJ * eJ - ej * ej) * ir - 1.5f * dJ2 * ir);
    const float lR = (li[i - 1] + lrn) - l0;
    float dA = 0, dB = 0, dC = 0, dF = 0, dQ = 0;
    if (L.bc == BC_HBB || (qi < 0.5f && !((mask >> (i + 7)) & 1u))) {
      dA = 1;
    } else if (qi < 0.5f) {
      dA = 2.f * qi;
      dB = 1.f - 2.f * qi;
      dF = wF * dB;
      dQ = 2.f * a[i - 1] - 2.f * b2[i - 1] - 2.f * wF * Fi;
    } else {
      const float i2q = 1.0f / (2.f * qi);
      dA = i2q;
      dC = (2.f * qi - 1.f) * i2q;
      dF = wF * dC;
      dQ = (cc[i - 1] - a[i - 1] + wF * Fi) * i2q * i2q * 2.f;
    }
    own[i] += dA * lR + l0;
    own[opp(i)] += dC * lR;
    if (dB != 0.f) atomicAdd(&lbc[i * L.plane + nb(-ex(i), -ey(i))], dB * lR);
    // F_i = w [3 e.F + 4.5 ((e.J')^2 - (e.j)^2)/rho - 1.5 (|J'|^2 - |j|^2)/rho], J' = j + F
    const float w = float(wgt(i)) * (dF * lR);
    lFx += w * (3.f * exi + 9.f * eJ * exi * ir - 3.f * Jx * ir);
    lFy += w * (3.f * eyi + 9.f * eJ * eyi * ir - 3.f * Jy * ir);
    ljx += w * (9.f * eF * exi - 3.f * Fx) * ir;
    ljy += w * (9.f * eF * eyi - 3.f * Fy) * ir;
    lrho -= w * (4.5f * (eJ * eJ - ej * ej) - 1.5f * dJ2) * ir * ir;
    // dJ/dq -> dJ/dc of the cylinder this link cuts (a node's links rarely cut two)
    const int c = bd[i - 1];
    if (c >= 0 && c < A.n_cyl && dQ != 0.f) {
      if (c != body) {
        flush();
        body = c;
        gx = gy = 0.0;
      }
      const double g = (double)dQ * (double)lR;
      gx += g * dc[i - 1].x;
      gy += g * dc[i - 1].y;
    }
  }
  flush();
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (own[i] != 0.f) atomicAdd(&lbc[i * L.plane + n], own[i]);
  float* lrj = static_cast<float*>(A.lrj);
  lrj[n] = lrho;
  lrj[L.plane + n] = ljx;
  lrj[2 * L.plane + n] = ljy;
  float* lF = static_cast<float*>(A.lamF);
  lF[n] = lFx;
  lF[L.plane + n] = lFy;
}

// k_adj_collide: a node a thread.  Latency and its loads are what it costs: sixteen blocks an SM (32
// registers instead of 40: a 512 x 512 lattice is one wave instead of 1.1), and what the geometry says
// of a node in one word (MOVES_) instead of ten bytes: 100 reverse steps of 512 x 512 with their
// recomputation 3.17 -> 2.96 ms.
constexpr int AC_BLOCK = 128;
constexpr unsigned MOVES_BC = 1u << 9, MOVES_BNODE = 1u << 10, MOVES_FLUID = 1u << 11;   // bits 0-8: directions that stream to a fluid node
__global__ void __launch_bounds__(AC_BLOCK, 16) k_adj_nodes(const __grid_constant__ Lattice<float> L,
                                                        const __grid_constant__ AdjBuffers A) {
  const int x = blockIdx.x * AC_BLOCK + threadIdx.x, y = blockIdx.y, n = y * L.pitch + x;
  const unsigned to = x < L.nx ? A.moves[n] : 0u;
  const bool live = to & MOVES_FLUID;
  const int xm = x == 0 ? L.nx - 1 : -1, xp = x == L.nx - 1 ? 1 - L.nx : 1;
  const int ym = !L.walls && y == 0 ? L.plane - L.pitch : -L.pitch;
  const int yp = !L.walls && y == L.ny - 1 ? L.pitch - L.plane : L.pitch;
  auto nb = [&](int i) { return n + (ex(i) < 0 ? xm : ex(i) > 0 ? xp : 0) + (ey(i) < 0 ? ym : ey(i) > 0 ? yp : 0); };
  float f[9], r = 1.f, drho = 0.f, jx = 0.f, jy = 0.f, Fx = 0.f, Fy = 0.f;
  if (live) node_state(L, x, y, f, r, drho, jx, jy, Fx, Fy);
  grid_wait();
  grid_launch();
  if (!live) return;
  const float* lin = static_cast<const float*>(A.lam_in);
  const float* lrp = static_cast<const float*>(A.Lrho);   // density share of lambda^{t+1}
  float* lout = static_cast<float*>(A.lam_out);
  float* lbc = static_cast<float*>(A.lam_bc);
  float* lF = static_cast<float*>(A.lamF);
  float lt[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) lt[i] = to & (1u << i) ? lin[i * L.plane + nb(i)] + lrp[nb(i)] : 0.f;
  float lrho = 0, ljx = 0, ljy = 0, lFx = 0, lFy = 0;
  if (to & MOVES_BC) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      lt[i] += lbc[i * L.plane + n];
      lbc[i * L.plane + n] = 0.f;
    }
  }
  if (to & MOVES_BNODE) {
    const float* lrj = static_cast<const float*>(A.lrj);
    lrho = lrj[n];
    ljx = lrj[L.plane + n];
    ljy = lrj[2 * L.plane + n];
    lFx = lF[n];
    lFy = lF[L.plane + n];
  }
  float lf[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) lf[i] = 0.f;
  collide_adjoint(L, r, jx, jy, Fx, Fy, lt, lf, lrho, ljx, ljy, lFx, lFy);
#pragma unroll
  for (int i = 0; i < 9; ++i) lout[i * L.plane + n] = lf[i] + lrho + float(ex(i)) * ljx + float(ey(i)) * ljy;
  lF[n] = lFx;
  lF[L.plane + n] = lFy;
}

// Force and chemical potential in reverse (k_adj_force, k_adj_mu) in one pass.  A block takes AT_X =
// 64 columns, 56 of them its own, and AT_H rows of its own: from dJ/dF at its nodes and the four
// rows and columns around them it forms dJ/dmu at the two around, then dJ/drho at its own.
constexpr int AT_X = 64, AT_HX = 4, AT_OUT = AT_X - 2 * AT_HX, AT_H = 16, AT_THREADS = 512;
constexpr int AT_FR = AT_H + 8;            // dJ/dF rows: four each side
constexpr int AT_MR = AT_H + 4;            // dJ/dmu and chemical-potential rows: two each side
constexpr int AT_STEP = AT_THREADS / AT_X;
static_assert(AT_FR % AT_STEP == 0 && AT_H % AT_STEP == 0, "rows of a block");
struct AdjTile {
  float fx[AT_FR][AT_X], fy[AT_FR][AT_X], px[AT_FR][AT_X], py[AT_FR][AT_X];   // dJ/dF and rho dJ/dF (0 off the fluid)
  float mu[AT_MR][AT_X];
  float lmu[AT_MR][AT_X];                                                     // dJ/dmu at fluid nodes
  uint8_t kind[AT_FR][AT_X];
};

__global__ void __launch_bounds__(AT_THREADS) k_adj_fields(const __grid_constant__ Lattice<float> L,
                                                           const __grid_constant__ AdjBuffers A, int strips) {
  __shared__ AdjTile S;
  const int band = blockIdx.x / strips, strip = blockIdx.x - band * strips;
  const int ya = band * AT_H, yb = min(ya + AT_H, L.ny);
  const int c = threadIdx.x % AT_X, t = threadIdx.x / AT_X;   // this thread's column; rows t, t + AT_STEP, ...
  const int x = strip * AT_OUT - AT_HX + c;
  int xw = x % L.nx;
  if (xw < 0) xw += L.nx;
  const bool own_col = c >= AT_HX && c < AT_X - AT_HX && x < L.nx;
  auto row_in = [&](int y) { return !L.walls || (y >= 0 && y < L.ny); };
  // (rows reach four beyond the lattice, which has five or more)
  auto row = [&](int y) { return (y < 0 ? y + L.ny : y >= L.ny ? y - L.ny : y) * L.pitch; };
  constexpr int PER = AT_FR / AT_STEP;
  float rho[PER];
  unsigned fluid = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int r = t + k * AT_STEP, y = ya - 4 + r;
    const bool in = row_in(y) && y < yb + 4;
    const uint8_t kd = in ? L.kind[row(y) + xw] : (uint8_t)KIND_DEEP;
    S.kind[r][c] = kd;
    rho[k] = kd == KIND_FLUID ? L.rho[row(y) + xw] : 0.f;
    if (kd == KIND_FLUID) fluid |= 1u << k;
    if (r >= 2 && r < AT_FR - 2 && in) S.mu[r - 2][c] = L.mu[row(y) + xw];
  }
  grid_wait();
  grid_launch();
  const float* lF = static_cast<const float*>(A.lamF);
  float* Lrho = static_cast<float*>(A.Lrho);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int r = t + k * AT_STEP, m = row(ya - 4 + r) + xw;
    const float lx = fluid & (1u << k) ? lF[m] : 0.f, ly = fluid & (1u << k) ? lF[L.plane + m] : 0.f;
    S.fx[r][c] = lx;
    S.fy[r][c] = ly;
    S.px[r][c] = rho[k] * lx;
    S.py[r][c] = rho[k] * ly;
  }
  __syncthreads();
  // ---- Eq. 9: gradient coefficients c_{+1} = 8/12, c_{+2} = -1/12, c_{-d} = -c_d; the neighbour m - d
  // sees this node at offset +d
  const float c1 = 8.0f / 12.0f, c2 = -1.0f / 12.0f;
  const bool eos = L.eos != EOS_NONE;
  // sum over d of c_d v(m - d), along x of the first array and along y of the second
  auto grad_t = [&](const float (*vx)[AT_X], const float (*vy)[AT_X], int r) {
    return c1 * (vx[r][c - 1] - vx[r][c + 1]) + c2 * (vx[r][c - 2] - vx[r][c + 2]) + c1 * (vy[r - 1][c] - vy[r + 1][c]) +
           c2 * (vy[r - 2][c] - vy[r + 2][c]);
  };
  for (int r = t; r < AT_MR; r += AT_STEP) {
    const int y = ya - 2 + r;
    const uint8_t k = S.kind[r + 2][c];
    float lm = 0.f;
    if (eos && c >= 2 && c < AT_X - 2 && is_field_node<float>(k)) lm = -grad_t(S.px, S.py, r + 2);
    // the wall chemical potential's gradient
    int to = -1;
    if (eos && own_col && y >= ya && y < yb && (k == KIND_SOLID1 || k == KIND_SOLID2)) {
      const int bd = L.body[row(y) + xw];
      to = bd >= 0 && bd < A.n_cyl ? bd : A.n_cyl;
    }
    add_by_body(A.grad, to, (double)lm);
    S.lmu[r][c] = k == KIND_FLUID ? lm : 0.f;
  }
  __syncthreads();
  // ---- dJ/drho: Eq. 9 directly, and Eq. 12 (mu_m = k^2 psi'(rho_m) - kappa sum_d l_d rho_{m+d}; l_0 =
  // -60/12, l_{+-1} = 16/12, l_{+-2} = -1/12)
  for (int r = t; r < AT_H; r += AT_STEP) {
    const int y = ya + r;
    const uint8_t k = S.kind[r + 4][c];
    if (!own_col || y >= yb || !is_field_node<float>(k)) continue;
    float lr = 0.f;
    if (eos) lr = (1.0f / 3.0f) * grad_t(S.fx, S.fy, r + 4);
    if (k == KIND_FLUID) {
      float gmx = 0.f, gmy = 0.f;
      if (eos) {
        const float* z = &S.mu[r + 2][c];
        gmx = diff4_of(z[1], z[-1], z[2], z[-2]) * (1.0f / 12.0f);
        gmy = diff4_of(z[AT_X], z[-AT_X], z[2 * AT_X], z[-2 * AT_X]) * (1.0f / 12.0f);
      }
      lr += S.fx[r + 4][c] * (L.gx - gmx) + S.fy[r + 4][c] * (L.gy - gmy);
    }
    if (eos) {
      const int m = r + 2;
      const float acc = (16.0f / 12.0f) * ((S.lmu[m][c - 1] + S.lmu[m][c + 1]) + (S.lmu[m - 1][c] + S.lmu[m + 1][c])) -
                        (1.0f / 12.0f) * ((S.lmu[m][c - 2] + S.lmu[m][c + 2]) + (S.lmu[m - 2][c] + S.lmu[m + 2][c]));
      lr -= L.kappa * acc;
      if (k == KIND_FLUID) {
        const float l = S.lmu[m][c];
        lr += L.kappa * (60.0f / 12.0f) * l + L.k2 * psi_second(L, L.rho[row(y) + xw]) * l;
      }
    }
    Lrho[row(y) + xw] = lr;
  }
}

// Eq. 15 in reverse: a first-layer node's share is its own and what its second-layer neighbours
// hand it (winv: 1 / sum of their weights, by node); it passes it on to its fluid neighbours.
__global__ void __launch_bounds__(ADJ_BLOCK) k_adj_layers(const __grid_constant__ Lattice<float> L,
                                                          const __grid_constant__ AdjBuffers A) {
  float* Lrho = static_cast<float*>(A.Lrho);
  const float* winv = static_cast<const float*>(A.winv);
  const int j = blockIdx.x * ADJ_BLOCK + threadIdx.x;
  int n = 0, x = 0, y = 0;
  unsigned m = 0, outer = 0;
  float w1 = 0.f, w2[8];
  if (j < L.n_s1) {
    n = L.s1node[j];
    m = L.s1mask[j];
    w1 = L.s1winv[j];
    x = n % L.pitch;
    y = n / L.pitch;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const int yy = y - ey(i);
      if (L.walls && (yy < 0 || yy >= L.ny)) continue;
      const int q = node_at(L, x - ex(i), yy);
      if (L.kind[q] == KIND_SOLID2) {
        outer |= 1u << (i - 1);
        w2[i - 1] = winv[q];
      }
    }
  }
  grid_wait();
  grid_launch();
  if (j >= L.n_s1) return;
  float v = Lrho[n];
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (outer & (1u << (i - 1))) v += float(wgt(i)) * (Lrho[node_at(L, x - ex(i), y - ey(i))] * w2[i - 1]);
  v *= w1;
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (m & (1u << (i - 1))) atomicAdd(&Lrho[node_at(L, x + ex(i), y + ey(i))], float(wgt(i)) * v);
}
// What every reverse step needs of the geometry, formed once a sweep: 1 / sum of the weights of each
// second-layer node's Eq. 15, by node; p / (p . e) of each link into a cylinder (its FP64 division is
// several microseconds a step on a GPU with few FP64 units).
__global__ void k_adj_geometry(Lattice<float> L, float* winv, double2* dqdc, int n_cyl) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < L.n_s2) winv[L.s2node[j]] = L.s2winv[j];
  if (j >= L.n_bnodes || n_cyl == 0) return;
  const int n = L.bnode[j], x = n % L.pitch, y = n / L.pitch;
  for (int l = L.bstart[j]; l < L.bstart[j + 1]; ++l) {
    const int i = L.ldir[l], c = L.body[node_at(L, x + ex(i), y + ey(i))];
    if (c < 0 || c >= n_cyl) continue;
    const double q = (double)L.lq[l];
    const double px = (double)x - L.cyl[4 * c] + q * ex(i);
    const double py = (double)y - L.cyl[4 * c + 1] + q * ey(i);
    const double pe = px * ex(i) + py * ey(i);
    dqdc[(i - 1) * (long long)L.bcap + j] = make_double2(px / pe, py / pe);
  }
}

// moves of every node, once a sweep
__global__ void __launch_bounds__(ADJ_BLOCK) k_adj_moves(Lattice<float> L, const uint8_t* bct, uint16_t* moves) {
  const long long n = (long long)blockIdx.x * ADJ_BLOCK + threadIdx.x;
  if (n >= L.plane) return;
  const int y = (int)(n / L.pitch), x = (int)(n - (long long)y * L.pitch);
  unsigned m = 0;
  if (x < L.nx && L.kind[n] == KIND_FLUID) {
    m = MOVES_FLUID | (bct[n] & 1 ? MOVES_BC : 0u) | (bct[n] & 2 ? MOVES_BNODE : 0u);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const bool in = !L.walls || (y + ey(i) >= 0 && y + ey(i) < L.ny);
      if (in && L.kind[node_at(L, x + ex(i), y + ey(i))] == KIND_FLUID) m |= 1u << i;
    }
  }
  moves[n] = (uint16_t)m;
}

// ---- set-up, objective, seeds ------------------------------------------------------------
// bct bit 0: node may receive boundary contributions to its post-collision adjoint (x1 or x2 of
// a cut link); bit 1: boundary node (local moment and force adjoints from its links)
template <typename real>
__global__ void k_adj_flags_x2(Lattice<real> L, uint8_t* bct) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= L.n_bnodes) return;
  const int n = L.bnode[b];
  const int x = n % L.pitch, y = n / L.pitch;
  for (int l = L.bstart[b]; l < L.bstart[b + 1]; ++l) {
    const int i = L.ldir[l];
    if (L.lx2f[l]) bct[node_at(L, x - ex(i), y - ey(i))] = 1;
  }
}

template <typename real>
__global__ void k_adj_flags_x1(Lattice<real> L, uint8_t* bct) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= L.n_bnodes) return;
  bct[L.bnode[b]] = 3;
}

// touch[n] = 1 at fluid nodes with a cut link into body `body`
template <typename real>
__global__ void k_touch(Lattice<real> L, uint8_t* touch, int body) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= L.n_bnodes) return;
  const int n = L.bnode[b];
  const int x = n % L.pitch, y = n / L.pitch;
  uint8_t t = 0;
  for (int l = L.bstart[b]; l < L.bstart[b + 1]; ++l) {
    const int i = L.ldir[l];
    if (L.body[node_at(L, x + ex(i), y + ey(i))] == body) t = 1;
  }
  touch[n] = t;
}

// Sums of the droplet objective over the fluid nodes of lattice `cur`, one set per block
// (red[4 b + k]; the host adds the blocks in order, so the result does not depend on timing):
//   k = 0: sum (rho - rho_g), 1: sum (rho - rho_g) y,
//   2: sum over touching nodes of (rho - rho_g)/(rho_l - rho_g), 3: their number.
template <typename real>
__global__ void k_objective_sums(Lattice<real> L, int cur, const uint8_t* touch, double* red, double rg, double rl) {
  __shared__ double sm[32];
  double s0 = 0, s1 = 0, s2 = 0, s3 = 0;
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < L.plane; n += gridDim.x * blockDim.x) {
    if (L.kind[n] != KIND_FLUID) continue;
    real fl[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) fl[i] = L.f[cur][i * L.plane + n];
    const double r = (double)L.rho_ref + (double)density_sum(fl);
    const double y = (double)(n / L.pitch);
    s0 += r - rg;
    s1 += (r - rg) * y;
    if (touch[n]) {
      s2 += (r - rg) / (rl - rg);
      s3 += 1.0;
    }
  }
  double* out = red + 4 * blockIdx.x;
  double t;
  t = block_sum(s0, sm); if (threadIdx.x == 0) out[0] = t;
  t = block_sum(s1, sm); if (threadIdx.x == 0) out[1] = t;
  t = block_sum(s2, sm); if (threadIdx.x == 0) out[2] = t;
  t = block_sum(s3, sm); if (threadIdx.x == 0) out[3] = t;
}

// dJ/drho of the objective at every node (row-major nx x ny; zero off the fluid)
template <typename real>
__global__ void k_objective_seed(Lattice<real> L, const uint8_t* touch, double y_cm, double S, double wcoef, real* out) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= L.nx) return;
  const int n = y * L.pitch + x;
  double g = 0.0;
  if (L.kind[n] == KIND_FLUID) g = ((double)y - y_cm) / S + (touch[n] ? wcoef : 0.0);
  out[(long long)y * L.nx + x] = (real)g;
}

// lambda = dJ/df of the last state from dJ/drho (row-major nx x ny) and dJ/df (9 such arrays),
// either may be null
template <typename real>
__global__ void k_adj_seed(Lattice<real> L, real* lam, const real* drho, const real* df) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= L.nx) return;
  const int n = y * L.pitch + x;
  const long long c = (long long)y * L.nx + x, dn = (long long)L.nx * L.ny;
  const bool fl = L.kind[n] == KIND_FLUID;
  const real g = fl && drho ? drho[c] : real(0);
#pragma unroll
  for (int i = 0; i < 9; ++i) lam[i * L.plane + n] = fl ? g + (df ? df[i * dn + c] : real(0)) : real(0);
}

// lambda of the first state (nine planes plus the density share), row-major (9 arrays of
// nx x ny; zero off the fluid)
template <typename real>
__global__ void k_adj_export(Lattice<real> L, const real* lam, const real* Lrho, real* out) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= L.nx) return;
  const int n = y * L.pitch + x;
  const long long c = (long long)y * L.nx + x, dn = (long long)L.nx * L.ny;
  const bool fl = L.kind[n] == KIND_FLUID;
  const real lr = fl ? Lrho[n] : real(0);
#pragma unroll
  for (int i = 0; i < 9; ++i) out[i * dn + c] = fl ? lam[i * L.plane + n] + lr : real(0);
}

// ---- launchers -------------------------------------------------------------------------------
template <typename real>
static dim3 adj_grid(const Lattice<real>& L) { return dim3((unsigned)((L.nx + ADJ_BLOCK - 1) / ADJ_BLOCK), (unsigned)L.ny); }
static unsigned list_grid(int n) { return (unsigned)(n > 0 ? (n + ADJ_BLOCK - 1) / ADJ_BLOCK : 1); }

template <typename real>
cudaError_t adj_flags(const Lattice<real>& L, uint8_t* bct, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(bct, 0, (size_t)L.plane, s);
  if (e != cudaSuccess || L.n_bnodes == 0) return e;
  k_adj_flags_x2<real><<<list_grid(L.n_bnodes), ADJ_BLOCK, 0, s>>>(L, bct);
  k_adj_flags_x1<real><<<list_grid(L.n_bnodes), ADJ_BLOCK, 0, s>>>(L, bct);
  return cudaGetLastError();
}

unsigned objective_blocks(long long plane) {
  const long long b = (plane + ADJ_BLOCK - 1) / ADJ_BLOCK;
  return (unsigned)(b < (long long)mass_blocks() ? b : (long long)mass_blocks());
}

template <typename real>
cudaError_t objective_sums(const Lattice<real>& L, int cur, int body, uint8_t* touch, double* red, double rg,
                           double rl, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(touch, 0, (size_t)L.plane, s);
  if (e != cudaSuccess) return e;
  if (L.n_bnodes > 0) k_touch<real><<<list_grid(L.n_bnodes), ADJ_BLOCK, 0, s>>>(L, touch, body);
  k_objective_sums<real><<<objective_blocks(L.plane), ADJ_BLOCK, 0, s>>>(L, cur, touch, red, rg, rl);
  return cudaGetLastError();
}

template <typename real>
cudaError_t objective_seed(const Lattice<real>& L, const uint8_t* touch, double y_cm, double S, double wcoef,
                           real* out, cudaStream_t s) {
  k_objective_seed<real><<<adj_grid(L), ADJ_BLOCK, 0, s>>>(L, touch, y_cm, S, wcoef, out);
  return cudaGetLastError();
}

template <typename real>
cudaError_t adj_seed(const Lattice<real>& L, real* lam, const real* drho, const real* df, cudaStream_t s) {
  k_adj_seed<real><<<adj_grid(L), ADJ_BLOCK, 0, s>>>(L, lam, drho, df);
  return cudaGetLastError();
}

template <typename real>
cudaError_t adj_export(const Lattice<real>& L, const real* lam, const real* Lrho, real* out, cudaStream_t s) {
  k_adj_export<real><<<adj_grid(L), ADJ_BLOCK, 0, s>>>(L, lam, Lrho, out);
  return cudaGetLastError();
}

cudaError_t adj_geometry(const Lattice<float>& L, const uint8_t* bct, float* winv, double2* dqdc, uint16_t* moves, int n_cyl,
                         cudaStream_t s) {
  k_adj_moves<<<(unsigned)((L.plane + ADJ_BLOCK - 1) / ADJ_BLOCK), ADJ_BLOCK, 0, s>>>(L, bct, moves);
  const int n = L.n_s2 > L.n_bnodes ? L.n_s2 : L.n_bnodes;
  if (n > 0) k_adj_geometry<<<list_grid(n), ADJ_BLOCK, 0, s>>>(L, winv, dqdc, n_cyl);
  return cudaGetLastError();
}

// One reverse step.  L.f[0] holds f^t and L.rho / L.mu the density and chemical potential of
// step t; lambda^{t+1} is (A.lam_in, A.Lrho); leaves lambda^t as (A.lam_out, A.Lrho).
template <typename real>
cudaError_t adj_step(const Lattice<real>& L, const AdjBuffers& A, cudaStream_t s) {
  if constexpr (sizeof(real) == 4) {
    cudaError_t e = cudaSuccess;
    const auto blocks = [](int n, int per) { return dim3((unsigned)((n + per - 1) / per)); };
    bool first = A.first;   // the step's first kernel follows other work: an ordinary launch
    if (L.n_bnodes > 0) {
      if (first) k_adj_links<<<blocks(L.n_bnodes, AL_BLOCK), AL_BLOCK, 0, s>>>(L, A);
      else e = launch_after(k_adj_links, blocks(L.n_bnodes, AL_BLOCK), AL_BLOCK, 0, s, L, A);
      first = false;
    }
    const dim3 nodes((unsigned)((L.nx + AC_BLOCK - 1) / AC_BLOCK), (unsigned)L.ny);
    if (first) k_adj_nodes<<<nodes, AC_BLOCK, 0, s>>>(L, A);
    else if (e == cudaSuccess) e = launch_after(k_adj_nodes, nodes, AC_BLOCK, 0, s, L, A);
    const int strips = (L.nx + AT_OUT - 1) / AT_OUT, bands = (L.ny + AT_H - 1) / AT_H;
    if (e == cudaSuccess) e = launch_after(k_adj_fields, dim3((unsigned)(strips * bands)), AT_THREADS, 0, s, L, A, strips);
    if (e == cudaSuccess && L.n_s1 > 0) e = launch_after(k_adj_layers, blocks(L.n_s1, ADJ_BLOCK), ADJ_BLOCK, 0, s, L, A);
    return e == cudaSuccess ? cudaGetLastError() : e;
  } else {
    if (L.n_bnodes > 0) k_adj_bc<real><<<list_grid(L.n_bnodes), ADJ_BLOCK, 0, s>>>(L, A);
    k_adj_collide<real><<<adj_grid(L), ADJ_BLOCK, 0, s>>>(L, A);
    k_adj_force<real><<<adj_grid(L), ADJ_BLOCK, 0, s>>>(L, A);
    k_adj_mu<real><<<adj_grid(L), ADJ_BLOCK, 0, s>>>(L, A);
    if (L.n_s2 > 0) k_adj_solid<real><<<list_grid(L.n_s2), ADJ_BLOCK, 0, s>>>(L, A, 2);
    if (L.n_s1 > 0) k_adj_solid<real><<<list_grid(L.n_s1), ADJ_BLOCK, 0, s>>>(L, A, 1);
    return cudaGetLastError();
  }
}

#define LBMGB_ADJ_INSTANTIATE(real)                                                                        \
  template cudaError_t adj_flags<real>(const Lattice<real>&, uint8_t*, cudaStream_t);                     \
  template cudaError_t objective_sums<real>(const Lattice<real>&, int, int, uint8_t*, double*, double,    \
                                            double, cudaStream_t);                                        \
  template cudaError_t objective_seed<real>(const Lattice<real>&, const uint8_t*, double, double, double, \
                                            real*, cudaStream_t);                                         \
  template cudaError_t adj_seed<real>(const Lattice<real>&, real*, const real*, const real*, cudaStream_t); \
  template cudaError_t adj_export<real>(const Lattice<real>&, const real*, const real*, real*, cudaStream_t); \
  template cudaError_t adj_step<real>(const Lattice<real>&, const AdjBuffers&, cudaStream_t);
LBMGB_ADJ_INSTANTIATE(float)
LBMGB_ADJ_INSTANTIATE(double)

}  // namespace lbmgb
