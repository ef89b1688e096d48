// The fused step (FP32, two population lattices, an equation of state): chemical potential, force,
// collision, streaming and the next state's density in ONE pass over the populations (k_walk on
// large lattices, k_tile on the others), then the cut links (k_bc_fused) and the solid layers
// (k_solids), instead of a density, a chemical-potential, a collide, a boundary and two layer
// kernels and a scatter that hand planes to one another through memory.  The values are those of
// the separate passes, bit for bit.
//
// A warp works on rows of FW = 64 columns, two adjacent ones a lane, in sm_103a's packed FP32
// arithmetic (float2: the separate collide kernel was bound by instruction issue as much as by
// bytes).  It forms what the OUT = 56 inner columns receive: the columns beyond belong to the
// neighbouring strips and are collided again here, so that every store is an aligned pair of its
// own (the shifted directions go through the neighbouring lane) and each node's density can be
// summed from registers as the populations streaming into it are formed.  That costs 64/56 = 14 %
// of the arithmetic and of the L2 traffic, nothing of the DRAM traffic: 36 + 36 bytes of
// populations, 4 + 4 of density and the node's class are read and written once.
//
// Slots of boundary nodes whose source is solid are left to k_bc_fused, which finds the force of
// those nodes in two planes (the pass stores it in the rows next to solids).  The densities of
// boundary nodes come from k_bc_fused, those of the solid layers from k_solids.
//
// On the 2048 x 4096 impact lattice a step takes 0.147 ms against 0.192 ms for the separate passes
// (2048 x 2048 84 against 110 us, 1024 x 1024 with 16 drops 33 against 45, 131 x 97 9.0 against 29);
// the pass itself 0.13 ms, 661 MB of DRAM traffic.  What bounds a walk is instruction issue: twelve
// warps an SM (three in each quarter, which is what their registers allow) issue 0.6 instructions a
// clock and scheduler, a third of them integer work and constants' moves; DRAM is at 55 %.  What was
// tried on the way there: the density formed from the populations at the start of the same pass
// instead of the end of the previous one (72 instead of 80 bytes a node, but the populations of four
// more rows wait in shared memory for their collision: 0.19 ms); 8-byte cp.async through L1 instead
// of 16-byte ones past it (the L1 lines left beside 200 KB of shared memory bound the loads in
// flight: 0.20 against 0.15 ms); two rows an iteration with a second path for rows that hold solids
// (0.143 ms on 2048 x 4096, but 1.6 times the code, which the instruction cache pays for: 92 against
// 82 us on 1672 x 2453, 0.137 against 0.128 ms with the pseudopotential), and with three paths 0.175;
// four columns a lane (half the shared-memory and store instructions, but 7 warps an SM: 0.20 ms);
// sixteen warps of 128 registers (0.153 ms).
//
// Batches run the same kernels over flat lists of all instances' tiles (walks, where the instances
// are large), links and layers, each block with its instance's descriptor in shared memory: 64
// lattices of 128..768 take 368 us a step against 590 us for the persistent kernel (k_batch: six grid
// barriers a step, 890 instructions a node), 256 of 64..128 119 against 217 us.
#include <algorithm>
#include <vector>

#include "lbm_fused.cuh"

#include "lbm_internal.h"
#include "lbm_phases.cuh"

namespace lbmgb {

namespace {

constexpr int FW = 64;                 // columns a warp holds
constexpr int FD = 4;                  // rows of populations in shared memory
constexpr int AHEAD = 3;               // rows of populations and densities requested ahead
constexpr int ROW_F = 9 * FW * 4;      // bytes of one row's populations in shared memory
constexpr int HX = 4;                  // columns held on each side of the strip's outputs
constexpr int OUT = FW - 2 * HX;       // output columns
constexpr int SP = FW / 2 + 4;         // pairs of a density or chemical-potential row: two more each side
constexpr int RHO_ROWS = 8, MU_ROWS = 4;   // rows of the two rings (psi: RHO_ROWS)
constexpr int RHO_CHUNKS = SP / 2;     // 16-byte pieces of a density row

// LEAD: rows between the newest density row and the collision
template <bool PSEUDO> struct Reach {
  static constexpr int LEAD = PSEUDO ? 1 : 4;
  static constexpr int BYTES = FD * ROW_F + (RHO_ROWS + (PSEUDO ? 0 : MU_ROWS)) * SP * 8;
};

__device__ __forceinline__ void cp4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// column c of a lattice of nx columns, wrapped (c within one lattice of the range, or clamped)
__device__ __forceinline__ int wrap_col(int c, int nx) {
  c %= nx;
  return c < 0 ? c + nx : c;
}

// The walk: one warp takes a strip up through a band of rows.  At row r it forms the chemical
// potential of row r - 2, whose stencil is complete then, collides row r - 4 and completes the
// density of row r - 5.  Rows arrive by cp.async three rows ahead; densities and chemical potentials
// live in rings in shared memory that no other warp reads, so one __syncwarp a row is all the
// synchronisation.  All rows take one path, whose only branches are warp-wide: solid nodes' chemical
// potential is chosen, not branched for, and the classes that decide are fetched two rows early.
//
// One warp: the populations streaming into the output columns of strip `strip` in rows [ya, yb),
// and those nodes' density (psi), from the state in lattice `cur`.
template <bool PSEUDO, int AA = 0>
__device__ __forceinline__ void walk(const Lattice<float>& L, int cur, int strip, int ya, int yb, char* smem) {
  using R = Reach<PSEUDO>;
  constexpr int LEAD = R::LEAD;
  const int lane = threadIdx.x & 31;
  const int x0 = strip * OUT, c = x0 - HX + 2 * lane;   // this lane's columns c, c + 1
  const bool mine = lane >= HX / 2 && lane < 32 - HX / 2;
  // (with nx odd the last pair's second column is the row's padding, which nothing reads)
  const bool out1 = mine && c < L.nx;
  const int ca = wrap_col(c, L.nx), cb = wrap_col(c + 1, L.nx);   // inside the lattice
  // Rows arrive in 16-byte pieces of four columns, straight into shared memory (not through L1,
  // which would bound the rows in flight).  With nx a multiple of four a wrapped piece stays one
  // aligned piece; otherwise the strips at the edges (split) load their columns one by one.
  const bool split = (L.nx & 3) != 0 && (x0 - 2 * HX < 0 || x0 + OUT + 2 * HX > L.nx);
  const int p4 = wrap_col(x0 - HX + 4 * (lane & 15), L.nx);                 // this lane's piece of a population row
  const int q4 = wrap_col(x0 - 2 * HX + 4 * lane, L.nx);                    // ... of a density row (18 lanes)
  const float* __restrict__ fin = L.f[cur];
  float* __restrict__ fout = L.f[cur ^ 1];
  float* const fone = L.f[0];                              // (AA: the one lattice)
  const float* __restrict__ rin = PSEUDO ? L.mu : L.rho;   // the state's density (psi)
  float* __restrict__ rout = L.rho_next;                   // the next state's
  const float2* const fs = reinterpret_cast<const float2*>(smem) + lane;          // own pair: + (row, i) * 32
  float2* const rs = reinterpret_cast<float2*>(smem + FD * ROW_F) + HX / 2 + lane;   // density (psi): + row * SP
  float2* const ms = rs + RHO_ROWS * SP;                                          // chemical potential
  const int cm = c == 0 ? L.nx - 1 : c - 1, c1 = c + 1 == L.nx ? 0 : c + 1, c2 = c1 + 1 == L.nx ? 0 : c1 + 1;   // (AA 2)
  // AA: this lane's part of aa_edge if it holds an outermost column with a strip beside it
  float* edge = nullptr;
  if (AA && lane == HX / 2 && strip > 0) edge = L.aa_edge + (strip - 1) * 16ll * L.ny + 8;
  if (AA && lane == 31 - HX / 2 && x0 + OUT < L.nx) edge = L.aa_edge + strip * 16ll * L.ny;
  auto rslot = [](int r) { return (r & (RHO_ROWS - 1)) * SP; };
  auto mslot = [](int r) { return (r & (MU_ROWS - 1)) * SP; };
  auto fslot = [](int y) { return (y & (FD - 1)) * (9 * 32); };

  // row r inside the lattice: wrapped, or (walls) clamped to a wall row, whose values no fluid
  // node's stencil reaches
  auto row_of = [&](int r) {
    if (L.walls) return min(max(r, 0), L.ny - 1);
    return r < 0 ? r + L.ny : (r >= L.ny ? r - L.ny : r);
  };
  auto load_rho = [&](int r) {
    const int n = row_of(r) * L.pitch;
    char* const d = smem + FD * ROW_F + rslot(r) * 8;
    if (!split) {
      if (lane < RHO_CHUNKS) cp16(d + 16 * lane, reinterpret_cast<const char*>(rin) + 4u * (unsigned)(n + q4));
    } else {
      for (int e = lane; e < 4 * RHO_CHUNKS; e += 32) cp4(d + 4 * e, rin + n + wrap_col(x0 - 2 * HX + e, L.nx));
    }
  };
  auto load_f = [&](int y) {
    const int n = row_of(y) * L.pitch;
    char* const d = smem + fslot(y) * 8;
    if constexpr (AA == 2) {
      // direction i from plane opp(i), row y - e_y
      const int nm = row_of(y - 1) * L.pitch, np = row_of(y + 1) * L.pitch;
      auto from = [&](int i) { return fin + opp(i) * (long long)L.plane + (ey(i) == 0 ? n : ey(i) > 0 ? nm : np); };
      if (!split) {
#pragma unroll
        for (int k = 0; k < 4; ++k) cp16(d + 512 * k + 16 * lane, (lane & 16 ? from(2 * k + 1) : from(2 * k)) + p4);
        if (lane < 16) cp16(d + 2048 + 16 * lane, from(8) + p4);
      } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          cp4(d + 256 * i + 8 * lane, from(i) + ca);
          cp4(d + 256 * i + 8 * lane + 4, from(i) + cb);
        }
      }
    } else if (!split) {
      // a warp's 32 pieces are two directions' rows
      const char* base = reinterpret_cast<const char*>(fin + (lane >> 4) * (long long)L.plane) + 4u * (unsigned)(n + p4);
#pragma unroll
      for (int k = 0; k < 4; ++k) cp16(d + 512 * k + 16 * lane, base + 8ll * k * L.plane);
      if (lane < 16) cp16(d + 2048 + 16 * lane, base + 32ll * L.plane);
    } else {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        cp4(d + 256 * i + 8 * lane, fin + i * L.plane + n + ca);
        cp4(d + 256 * i + 8 * lane + 4, fin + i * L.plane + n + cb);
      }
    }
  };
  // rows collided: ya - 1 .. yb (AA: the band's own); the newest density row r runs from rb to re
  const int ylo = AA ? ya : ya - 1, yhi = AA ? yb - 1 : yb;
  const int rb = ylo + (PSEUDO ? 1 : 0), re = yhi + LEAD;
  // density row r + AHEAD and the populations of the row AHEAD above the one collided with row r
  auto request = [&](int r) {
    if (r + AHEAD <= re) load_rho(r + AHEAD);
    const int y = r - LEAD + AHEAD;
    if (y >= ylo && y <= yhi) load_f(y);
    cp_commit();
  };
  // The classes of columns c and c + 1 of a row.  (Two registers that nothing touches before the row's
  // turn: combining them at once would wait for the loads.)
  struct Kinds { unsigned a, b; };
  auto kind_row = [&](int r) -> Kinds {
    const uint8_t* k = L.kind + row_of(r) * L.pitch;
    return {k[ca], k[cb]};
  };
  // bit 0 / 1: column c / c + 1 is fluid
  auto fluid_bits = [](Kinds k) { return (k.a == KIND_FLUID ? 1u : 0u) | (k.b == KIND_FLUID ? 2u : 0u); };
  auto load_pops = [&](int y, float2 (&v)[9]) {
    const float2* d = fs + fslot(y);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if (AA == 2 && ex(i) != 0) {
        const float* p = reinterpret_cast<const float*>(d + i * 32) - ex(i);
        v[i] = make_float2(p[0], p[1]);
      } else {
        v[i] = d[i * 32];
      }
    }
  };
  // the undivided x differences of Eq. 9 from a pair and its neighbour pairs
  auto dx_of = [](float2 l, float2 C, float2 g) {
    return fma_rn(splat<float2>(8.0f), make_float2(sub_rn(C.y, l.y), sub_rn(g.x, C.x)), sub_rn(l, g));
  };
  // mu from the densities of its row (left, own, right pair) and of the rows around it
  auto mu_at = [&](float2 l, float2 C, float2 g, float2 u1, float2 u2, float2 d1, float2 d2) {
    // (x+1 - c) + (x-1 - c): within the pair the two differences are +-(C.y - C.x)
    const float t = sub_rn(C.y, C.x);
    const float2 x1 = make_float2(add_rn(t, sub_rn(l.y, C.x)), add_rn(sub_rn(g.x, C.y), -t));
    const float2 lap = lap4_diff(x1, add_rn(sub_rn(C, g), sub_rn(C, l)), add_rn(sub_rn(u1, C), sub_rn(d1, C)),
                                 add_rn(sub_rn(C, u2), sub_rn(C, d2)));
    return mu_of(L, psi_prime_shifted(L, C), lap);
  };
  auto force_pp_at = [&](float2 rho, int y, float2& Fx, float2& Fy) {
    const float2* u = rs + rslot(y + 1);
    const float2* q = rs + rslot(y);
    const float2* d = rs + rslot(y - 1);
    const float2 C = q[0], U = u[0], D = d[0];
    float2 ax, ay;
    pp_sums(make_float2(C.y, q[1].x), U, make_float2(q[-1].y, C.x), D, make_float2(U.y, u[1].x), make_float2(u[-1].y, U.x),
            make_float2(d[-1].y, D.x), make_float2(D.y, d[1].x), ax, ay);
    Fx = force_pp(rho, L.gx, C, ax);
    Fy = force_pp(rho, L.gy, C, ay);
  };
  // What the rows collided so far stream into row y (the next one collided) and the row below it:
  // that row's density is complete once row y is collided.
  struct Incoming {
    float2 c0, s13;          // row y - 1: at rest, and along x
    float2 d2, d5, d6;       // into row y - 1 from row y - 2
    float2 e2, e5, e6;       // into row y from row y - 1
  } in;
  {
    const float2 z = make_float2(0.f, 0.f);
    in = {z, z, z, z, z, z, z, z};
  }
  struct {
    float h, o1, o5, n5;     // AA, outermost columns: received and sent along x in row y - 1; sent into
  } out = {0.f, 0.f, 0.f, 0.f};   // the column beside in row y - 1 and row y from the row below each
  // Streaming of row y's post-collision populations: every pair of outputs receives columns c - 1, c
  // (moving right) or c + 1, c + 2 (moving left) through the neighbouring lane, so that all stores
  // are aligned pairs.  Slots whose source is solid get a meaningless value; the boundary phase
  // rewrites those of fluid nodes, nothing reads the others.
  // fl: this lane's fluid bits of the row
  auto stream_row = [&](const float2 (&v)[9], int y, unsigned fl) {
    auto right = [](float2 a) { return make_float2(__shfl_up_sync(0xffffffffu, a.y, 1), a.x); };
    auto left = [](float2 a) { return make_float2(a.y, __shfl_down_sync(0xffffffffu, a.x, 1)); };
    const float2 r1 = right(v[1]), r5 = right(v[5]), r8 = right(v[8]);
    const float2 l3 = left(v[3]), l6 = left(v[6]), l7 = left(v[7]);
    // row y - 1: density_sum's order
    const float2 sum = add_rn(in.c0, add_rn(add_rn(in.s13, add_rn(in.d2, v[4])),
                                            add_rn(add_rn(in.d5, l7), add_rn(in.d6, r8))));
    float2 q = add_rn(splat<float2>(L.rho_ref), sum);
    if (PSEUDO) q = psi_of(L, q);
    const int n = y * L.pitch + c;
    const bool mid = y >= ya && y < yb, up = y + 1 < yb, dn = y > ya;   // rows the band does not own are left
    if constexpr (AA != 0) {
      // (the density of a band's outermost rows and a strip's outermost columns: k_layers_aa)
      if (y >= ya + 2 && out1) {
        const bool first = c == x0, last = c + 1 == x0 + OUT - 1 || c + 1 == L.nx - 1;
        float* const p = rout + n - L.pitch;
        if (!first && !last) *reinterpret_cast<float2*>(p) = q;
        else if (!first) *p = q.x;
        else if (!last) p[1] = q.y;
      }
      if (edge) {
        // row y - 1's record: what the outermost column has received from the strip, and what it
        // has sent into the column beside it
        const bool lo = lane == HX / 2;
        auto at = [&](float2 a, float2 b) { return lo ? a.x : b.y; };
        const float2 f24 = add_rn(in.d2, v[4]);
        if (y >= ya + 2) {
          float4* const p = reinterpret_cast<float4*>(edge + 16 * (y - 1));
          p[0] = make_float4(at(in.c0, in.c0), out.h, at(f24, f24), at(in.d6, in.d5));
          p[1] = make_float4(at(l7, r8), out.o1, out.o5, at(v[7], v[8]));
        }
        out.o5 = out.n5;
        out.h = at(l3, r1);
        out.o1 = at(v[3], v[1]);
        out.n5 = at(v[6], v[5]);
      }
      if constexpr (AA == 1) {
        // each node's own slot opp(i)
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          float* const p = fone + opp(i) * (long long)L.plane + n;
          if (out1) *reinterpret_cast<float2*>(p) = v[i];
        }
      } else {
        // slot i of x + e_i: the slots read
        const int nm = row_of(y - 1) * L.pitch, n0 = y * L.pitch, np = row_of(y + 1) * L.pitch;
        const bool w0 = out1 && (fl & 1u), w1 = out1 && (fl & 2u) && c + 1 < L.nx;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          float* const p = fone + i * (long long)L.plane + (ey(i) == 0 ? n0 : ey(i) > 0 ? np : nm);
          if (w0) p[ex(i) == 0 ? c : ex(i) > 0 ? c1 : cm] = v[i].x;
          if (w1) p[ex(i) == 0 ? c1 : ex(i) > 0 ? c2 : c] = v[i].y;
        }
      }
    } else if (out1) {
      auto put = [&](float* plane, int at, float2 a) { *reinterpret_cast<float2*>(plane + at) = a; };
      if (mid) {
        put(fout, n, v[0]);
        put(fout + 1ll * L.plane, n, r1);
        put(fout + 3ll * L.plane, n, l3);
      }
      if (up) {
        put(fout + 2ll * L.plane, n + L.pitch, v[2]);
        put(fout + 5ll * L.plane, n + L.pitch, r5);
        put(fout + 6ll * L.plane, n + L.pitch, l6);
      }
      if (dn) {
        put(fout + 4ll * L.plane, n - L.pitch, v[4]);
        put(fout + 7ll * L.plane, n - L.pitch, l7);
        put(fout + 8ll * L.plane, n - L.pitch, r8);
        put(rout, n - L.pitch, q);
      }
    }
    in.c0 = v[0];
    in.s13 = add_rn(r1, l3);
    in.d2 = in.e2;
    in.d5 = in.e5;
    in.d6 = in.e6;
    in.e2 = v[2];
    in.e5 = r5;
    in.e6 = l6;
  };

  // density rows below rb, then the first requests
#pragma unroll 1
  for (int k = 1; k <= (PSEUDO ? 2 : 4); ++k) load_rho(rb - k);
#pragma unroll 1
  for (int k = AHEAD; k >= 1; --k) request(rb - k);
  Kinds k0 = kind_row(rb), k1 = kind_row(rb + 1);   // of rows r, r + 1
  unsigned bits = 0;                   // fluid bits of this lane, two per row, the newest row lowest
  unsigned solid = 0, none = 0;        // per row: some column of the warp is not fluid / none is
  // the constant chemical potential of a row's solid nodes
  auto walls_of = [&](int r, unsigned fl) {
    float2 w = make_float2(0.f, 0.f);
    const float* m = L.mu + row_of(r) * L.pitch;
    if (!PSEUDO && !(fl & 1u)) w.x = m[ca];
    if (!PSEUDO && !(fl & 2u)) w.y = m[cb];
    return w;
  };
  // Rows r - 2 and r - 1 came before the loop: their classes and walls (w2, w1).  Own pairs of density
  // rows r - 5, r - 6 and chemical-potential rows r - 5, r - 6 stay in registers: no neighbour needs
  // them, and the rings get by with 8 and 4 rows.
  float2 w2, w1, p5, p6, m5, m6;
  p5 = p6 = m5 = m6 = make_float2(0.f, 0.f);
  {
    const unsigned f2 = fluid_bits(kind_row(rb - 2)), f1 = fluid_bits(kind_row(rb - 1));
    bits = (f2 << 2) | f1;
    solid = (__all_sync(0xffffffffu, f2 == 3u) ? 0u : 2u) | (__all_sync(0xffffffffu, f1 == 3u) ? 0u : 1u);
    none = (__any_sync(0xffffffffu, f2 != 0u) ? 0u : 2u) | (__any_sync(0xffffffffu, f1 != 0u) ? 0u : 1u);
    w2 = walls_of(rb - 2, f2);
    w1 = walls_of(rb - 1, f1);
  }
#pragma unroll 1
  for (int r = rb; r <= re; ++r) {
    const int y = r - LEAD;
    const unsigned fl = fluid_bits(k0);
    bits = (bits << 2) | fl;
    solid = (solid << 1) | (__all_sync(0xffffffffu, fl == 3u) ? 0u : 1u);
    none = (none << 1) | (__any_sync(0xffffffffu, fl != 0u) ? 0u : 1u);
    k0 = k1;
    k1 = kind_row(min(r + 2, re));
    cp_wait<AHEAD - 1>();              // density row r and population row y are in
    __syncwarp();
    request(r);
    const float2 wn = walls_of(r, fl);
    // chemical potential of row r - 2, the walls' where solid
    float2 p4, p3, p2, mu;
    auto chem = [&]() {
      const float2* q = rs + rslot(r - 2);
      const float2 p1 = rs[rslot(r - 1)], t0 = rs[rslot(r)];
      p4 = rs[rslot(r - 4)];
      p3 = rs[rslot(r - 3)];
      p2 = q[0];
      mu = mu_at(q[-1], p2, q[1], p1, t0, p3, p4);
      if (!(bits & 16u)) mu.x = w2.x;
      if (!(bits & 32u)) mu.y = w2.y;
      ms[mslot(r - 2)] = mu;
    };
    if (y < ylo || (none & (1u << LEAD))) {
      // nothing to collide
      if (!PSEUDO) {
        chem();
        m6 = m5;
        m5 = ms[mslot(r - 4)];
      }
    } else {
      float2 v[9];
      load_pops(y, v);
      float2 drho, jx, jy, Fx, Fy;
      moments(v, drho, jx, jy);
      const float2 rho = add_rn(splat<float2>(L.rho_ref), drho);
      if constexpr (PSEUDO) {
        force_pp_at(rho, y, Fx, Fy);
      } else {
        chem();
        const float2* q = rs + rslot(r - 4);
        const float2* z = ms + mslot(r - 4);
        const float2 m4 = z[0], m3 = ms[mslot(r - 3)];
        Fx = force_cp(rho, L.gx, dx_of(z[-1], m4, z[1]), dx_of(q[-1], p4, q[1]));
        Fy = force_cp(rho, L.gy, diff4_of(m3, m5, mu, m6), diff4_of(p3, p5, p2, p6));
        m6 = m5;
        m5 = m4;
      }
      const unsigned fy = (bits >> (2 * LEAD)) & 3u;
      if (solid & (7u << (LEAD - 1))) {
        // next to a solid: the force for the boundary phase
        const int n = y * L.pitch + c;
        if (out1 && y >= ya && y < yb) {
          if (fy & 1u) { L.fx[n] = Fx.x; L.fy[n] = Fy.x; }
          if (fy & 2u) { L.fx[n + 1] = Fx.y; L.fy[n + 1] = Fy.y; }
        }
      }
      collide_node(L, v, rho, drho, jx, jy, Fx, Fy);
      stream_row(v, y, fy);
    }
    p6 = p5;
    p5 = p4;
    w2 = w1;
    w1 = wn;
  }
  cp_wait<0>();
}

// (A limit of 152 registers, of which the variants take 128 to 148: twelve warps an SM with or without
// it, and the schedule the compiler finds within it is 2 to 4 % faster than the one it finds alone.)
template <bool PSEUDO, int AA = 0>
__global__ void __maxnreg__(152) k_walk(const __grid_constant__ Lattice<float> L, int cur, int strips, int rows) {
  extern __shared__ __align__(16) char smem[];
  const int band = blockIdx.x / strips, strip = blockIdx.x - band * strips;
  const int ya = band * rows, yb = min(ya + rows, L.ny);
  grid_wait();
  grid_launch();
  walk<PSEUDO, AA>(L, cur, strip, ya, yb, smem);
}

// The descriptor of a batch's instance in shared memory, copied by the block's threads (the tables
// are constant: this runs before grid_wait).
__device__ __forceinline__ void take_lattice(Lattice<float>& L, const Lattice<float>* lat, int k) {
  static_assert(sizeof(Lattice<float>) % 4 == 0, "descriptor size");
  const int* s = reinterpret_cast<const int*>(lat + k);
  int* d = reinterpret_cast<int*>(&L);
  for (int i = threadIdx.x; i < (int)(sizeof(Lattice<float>) / 4); i += blockDim.x) d[i] = s[i];
}
// a batch: item blockIdx.x is (instance, strip, first row, rows)
__global__ void __launch_bounds__(32) k_walk_batch(const Lattice<float>* lat, const int4* items, int cur) {
  extern __shared__ __align__(16) char smem[];
  __shared__ __align__(16) Lattice<float> L;
  const int4 it = items[blockIdx.x];
  take_lattice(L, lat, it.x);
  __syncwarp();
  grid_wait();
  grid_launch();
  walk<false>(L, cur, it.y, it.z, it.z + it.w, smem);
}

// ---------------------------------------------------------------------------------------
// The same pass by tiles: a block of W warps takes the OUT output columns of a strip in H rows; its
// density rows (five more on each side) and population rows (one more) arrive together, then all
// chemical-potential rows, all collisions and all densities are formed side by side.

// the tile shapes: output rows at most, warps a block, blocks an SM
constexpr int TH_M = 14, TW_M = 8, TB_M = 3;
constexpr int TH_L = 10, TW_L = 4, TB_L = 5;

template <bool PSEUDO, int H>
struct Tile {
  static constexpr int MR = PSEUDO ? 0 : 3;              // chemical-potential rows beyond the outputs
  static constexpr int RR = PSEUDO ? 2 : 5;              // density (psi) rows beyond the outputs
  static constexpr int NC = H + 2, NM = H + 2 * MR, NR = H + 2 * RR;
  static constexpr int F = 0, RHO = NC * ROW_F, MU = RHO + NR * SP * 8, FLAGS = MU + (PSEUDO ? 0 : NM * SP * 8);
  static constexpr int BYTES = FLAGS + (H + 6) * 4;
};

// One population lattice in AA order (AA: the state's slot order plus one, pop_index): a tile collides
// its own nodes only.  Each reads and writes nine slots that no other node touches -- its own
// (natural order), or slot opp(i) of x - e_i (shifted), from aligned rows in shared memory read one
// column aside -- but what streams into the tile's outermost rows and columns comes from other
// tiles, so the density of those nodes is left to k_layers_aa.
template <bool PSEUDO, int H, int W, int AA = 0>
__device__ __forceinline__ void tile(const Lattice<float>& L, int cur, int strip, int ya, int yb, char* smem) {
  using T = Tile<PSEUDO, H>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x0 = strip * OUT, c = x0 - HX + 2 * lane;
  const bool mine = lane >= HX / 2 && lane < 32 - HX / 2;
  const bool out1 = mine && c < L.nx;   // (both columns: walk)
  const int ca = wrap_col(c, L.nx), cb = wrap_col(c + 1, L.nx);
  const bool split = (L.nx & 3) != 0 && (x0 - 2 * HX < 0 || x0 + OUT + 2 * HX > L.nx);
  const float* __restrict__ fin = L.f[cur];
  float* __restrict__ fout = L.f[cur ^ 1];
  float* const fin1 = L.f[0];   // (AA: the one lattice)
  const float* __restrict__ rin = PSEUDO ? L.mu : L.rho;
  int* const flags = reinterpret_cast<int*>(smem + T::FLAGS);   // rows ya - 3 ..: 1 some column solid, 2 none fluid
  auto row_of = [&](int r) {
    if (L.walls) return min(max(r, 0), L.ny - 1);
    return r < 0 ? r + L.ny : (r >= L.ny ? r - L.ny : r);
  };
  // rows of the tile's arrays by lattice row
  auto rho_row = [&](int r) { return reinterpret_cast<float2*>(smem + T::RHO) + (r - ya + T::RR) * SP + HX / 2 + lane; };
  auto mu_row = [&](int r) { return reinterpret_cast<float2*>(smem + T::MU) + (r - ya + T::MR) * SP + HX / 2 + lane; };
  auto pop_row = [&](int y) { return reinterpret_cast<float2*>(smem + (y - ya + 1) * ROW_F) + lane; };
  // ---- everything the tile reads
  {
    const int p4 = wrap_col(x0 - HX + 4 * (lane & 15), L.nx), q4 = wrap_col(x0 - 2 * HX + 4 * lane, L.nx);
    int e4[3] = {0, 0, 0};
    if (split) {
#pragma unroll
      for (int j = 0; j < 3; ++j) e4[j] = wrap_col(x0 - 2 * HX + lane + 32 * j, L.nx);
    }
    for (int r = ya - T::RR + warp; r < yb + T::RR; r += W) {
      const int n = row_of(r) * L.pitch;
      char* const d = smem + T::RHO + (r - ya + T::RR) * SP * 8;
      if (!split) {
        if (lane < RHO_CHUNKS) cp16(d + 16 * lane, rin + n + q4);
      } else {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (lane + 32 * j < 4 * RHO_CHUNKS) cp4(d + 4 * (lane + 32 * j), rin + n + e4[j]);
      }
    }
    const int y0 = AA ? ya : ya - 1, y1 = AA ? yb : yb + 1;   // rows collided
    for (int y = y0 + warp; y < y1; y += W) {
      const int n = row_of(y) * L.pitch;
      char* const d = smem + (y - ya + 1) * ROW_F;
      if constexpr (AA == 2) {
        // direction i from plane opp(i), row y - e_y
        const int nm = row_of(y - 1) * L.pitch, np = row_of(y + 1) * L.pitch;
        auto from = [&](int i) { return fin + opp(i) * (long long)L.plane + (ey(i) == 0 ? n : ey(i) > 0 ? nm : np); };
        if (!split) {
#pragma unroll
          for (int k = 0; k < 4; ++k) cp16(d + 512 * k + 16 * lane, (lane & 16 ? from(2 * k + 1) : from(2 * k)) + p4);
          if (lane < 16) cp16(d + 2048 + 16 * lane, from(8) + p4);
        } else {
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            cp4(d + 256 * i + 8 * lane, from(i) + ca);
            cp4(d + 256 * i + 8 * lane + 4, from(i) + cb);
          }
        }
      } else if (!split) {
        const float* base = fin + (lane >> 4) * (long long)L.plane + n + p4;
#pragma unroll
        for (int k = 0; k < 4; ++k) cp16(d + 512 * k + 16 * lane, base + 2ll * k * L.plane);
        if (lane < 16) cp16(d + 2048 + 16 * lane, base + 8ll * L.plane);
      } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          cp4(d + 256 * i + 8 * lane, fin + i * L.plane + n + ca);
          cp4(d + 256 * i + 8 * lane + 4, fin + i * L.plane + n + cb);
        }
      }
    }
    cp_commit();
  }
  // node classes of this warp's chemical-potential rows (psi: of the rows the force flags need), and
  // the walls' chemical potential where they are solid
  constexpr int M0 = 3, NMR = (H + 6 + W - 1) / W;
  unsigned fl[NMR];
  float2 wall[NMR];
#pragma unroll
  for (int k = 0; k < NMR; ++k) {
    const int m = ya - M0 + warp + k * W;
    fl[k] = 0u;
    if (m >= yb + M0) continue;
    const uint8_t* kd = L.kind + row_of(m) * L.pitch;
    fl[k] = (kd[ca] == KIND_FLUID ? 1u : 0u) | (kd[cb] == KIND_FLUID ? 2u : 0u);
  }
#pragma unroll
  for (int k = 0; k < NMR; ++k) {
    const int m = ya - M0 + warp + k * W;
    if (m >= yb + M0) continue;
    const float* w = L.mu + row_of(m) * L.pitch;
    wall[k] = make_float2(0.f, 0.f);
    if (!PSEUDO && !(fl[k] & 1u)) wall[k].x = w[ca];
    if (!PSEUDO && !(fl[k] & 2u)) wall[k].y = w[cb];
    const bool all = __all_sync(0xffffffffu, fl[k] == 3u), any = __any_sync(0xffffffffu, fl[k] != 0u);
    if (lane == 0) flags[m - ya + M0] = (all ? 0 : 1) | (any ? 0 : 2);
  }
  cp_wait<0>();
  __syncthreads();
  // ---- chemical potentials
  if (!PSEUDO) {
#pragma unroll
    for (int k = 0; k < NMR; ++k) {
      const int m = ya - M0 + warp + k * W;
      if (m >= yb + M0) continue;
      const float2* q = rho_row(m);
      const float2 C = q[0], l = q[-1], g = q[1], u1 = q[SP], u2 = q[2 * SP], d1 = q[-SP], d2 = q[-2 * SP];
      const float t = sub_rn(C.y, C.x);
      const float2 x1 = make_float2(add_rn(t, sub_rn(l.y, C.x)), add_rn(sub_rn(g.x, C.y), -t));
      const float2 lap = lap4_diff(x1, add_rn(sub_rn(C, g), sub_rn(C, l)), add_rn(sub_rn(u1, C), sub_rn(d1, C)),
                                   add_rn(sub_rn(C, u2), sub_rn(C, d2)));
      const float2 mu = mu_of(L, psi_prime_shifted(L, C), lap);
      const float2 v = make_float2(fl[k] & 1u ? mu.x : wall[k].x, fl[k] & 2u ? mu.y : wall[k].y);
      *mu_row(m) = v;
      if (L.mu_out && m >= ya && m < yb) {
        float* p = L.mu_out + m * L.pitch + c;
        if (out1) *reinterpret_cast<float2*>(p) = v;
      }
    }
    __syncthreads();
  }
  // ---- collisions and streaming
  for (int y = (AA ? ya : ya - 1) + warp; y < (AA ? yb : yb + 1); y += W) {
    const int* fg = flags + (y - ya + M0);
    if (fg[0] & 2) continue;
    float2 v[9];
    float2* const pr = pop_row(y);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if (AA == 2 && ex(i) != 0) {
        const float* p = reinterpret_cast<const float*>(pr + 32 * i) - ex(i);
        v[i] = make_float2(p[0], p[1]);
      } else {
        v[i] = pr[32 * i];
      }
    }
    float2 drho, jx, jy, Fx, Fy;
    moments(v, drho, jx, jy);
    const float2 rho = add_rn(splat<float2>(L.rho_ref), drho);
    const float2* q = rho_row(y);
    if constexpr (PSEUDO) {
      const float2 C = q[0], U = q[SP], D = q[-SP];
      float2 ax, ay;
      pp_sums(make_float2(C.y, q[1].x), U, make_float2(q[-1].y, C.x), D, make_float2(U.y, q[SP + 1].x),
              make_float2(q[SP - 1].y, U.x), make_float2(q[-SP - 1].y, D.x), make_float2(D.y, q[-SP + 1].x), ax, ay);
      Fx = force_pp(rho, L.gx, C, ax);
      Fy = force_pp(rho, L.gy, C, ay);
    } else {
      const float2* z = mu_row(y);
      auto dx_of = [](const float2* p) {
        const float2 l = p[-1], C = p[0], g = p[1];
        return fma_rn(splat<float2>(8.0f), make_float2(sub_rn(C.y, l.y), sub_rn(g.x, C.x)), sub_rn(l, g));
      };
      Fx = force_cp(rho, L.gx, dx_of(z), dx_of(q));
      Fy = force_cp(rho, L.gy, diff4_of(z[SP], z[-SP], z[2 * SP], z[-2 * SP]), diff4_of(q[SP], q[-SP], q[2 * SP], q[-2 * SP]));
    }
    const bool mid = y >= ya && y < yb, up = y + 1 < yb, dn = y > ya;
    if (mid && ((fg[-1] | fg[0] | fg[1]) & 1)) {
      // next to a solid: the force for the boundary phase (read at boundary nodes only)
      const int nf = y * L.pitch + c;
      if (out1) {
        *reinterpret_cast<float2*>(L.fx + nf) = Fx;
        *reinterpret_cast<float2*>(L.fy + nf) = Fy;
      }
    }
    collide_node(L, v, rho, drho, jx, jy, Fx, Fy);
    auto right = [](float2 a) { return make_float2(__shfl_up_sync(0xffffffffu, a.y, 1), a.x); };
    auto left = [](float2 a) { return make_float2(a.y, __shfl_down_sync(0xffffffffu, a.x, 1)); };
    const float2 r1 = right(v[1]), r5 = right(v[5]), r8 = right(v[8]);
    const float2 l3 = left(v[3]), l6 = left(v[6]), l7 = left(v[7]);
    const int n = y * L.pitch + c;
    if constexpr (AA == 1) {
      // each node's own slot opp(i)
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        float* p = fin1 + opp(i) * (long long)L.plane + n;
        if (out1) *reinterpret_cast<float2*>(p) = v[i];
      }
    } else if constexpr (AA == 2) {
      // slot i of x + e_i: the slots read
      const uint8_t* kd = L.kind + y * L.pitch;
      const bool w0 = out1 && kd[c] == KIND_FLUID, w1 = out1 && c + 1 < L.nx && kd[c + 1] == KIND_FLUID;
      const int nm = row_of(y - 1) * L.pitch, n0 = y * L.pitch, np = row_of(y + 1) * L.pitch;
      const int cm = c == 0 ? L.nx - 1 : c - 1, c1 = c + 1 == L.nx ? 0 : c + 1, c2 = c1 + 1 == L.nx ? 0 : c1 + 1;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        float* p = fin1 + i * (long long)L.plane + (ey(i) == 0 ? n0 : ey(i) > 0 ? np : nm);
        if (w0) p[ex(i) == 0 ? c : ex(i) > 0 ? c1 : cm] = v[i].x;
        if (w1) p[ex(i) == 0 ? c1 : ex(i) > 0 ? c2 : c] = v[i].y;
      }
    } else if (out1) {
      auto put = [&](int i, int at, float2 a) { *reinterpret_cast<float2*>(fout + (long long)i * L.plane + at) = a; };
      if (mid) {
        put(0, n, v[0]);
        put(1, n, r1);
        put(3, n, l3);
      }
      if (up) {
        put(2, n + L.pitch, v[2]);
        put(5, n + L.pitch, r5);
        put(6, n + L.pitch, l6);
      }
      if (dn) {
        put(4, n - L.pitch, v[4]);
        put(7, n - L.pitch, l7);
        put(8, n - L.pitch, r8);
      }
    }
    // what the densities of rows y - 1, y and y + 1 are summed from, in place of the populations
    pr[0] = v[0];
    pr[32] = add_rn(r1, l3);
    pr[64] = v[2];
    pr[96] = r5;
    pr[128] = l6;
    pr[160] = v[4];
    pr[192] = l7;
    pr[224] = r8;
  }
  __syncthreads();
  // ---- densities (psi) of the outputs; rows next to solids hold meaningless values where a source
  // is solid: the boundary phase forms the boundary nodes' densities
  for (int y = ya + (AA ? 1 : 0) + warp; y < yb - (AA ? 1 : 0); y += W) {
    if (flags[y - ya + M0] & 2) continue;
    const float2* o = pop_row(y);
    const float2* d = o - 9 * 32;
    const float2* u = o + 9 * 32;
    const float2 sum = add_rn(o[0], add_rn(add_rn(o[32], add_rn(d[64], u[160])), add_rn(add_rn(d[96], u[192]), add_rn(d[128], u[224]))));
    float2 q = add_rn(splat<float2>(L.rho_ref), sum);
    if (PSEUDO) q = psi_of(L, q);
    float* p = L.rho_next + y * L.pitch + c;
    if constexpr (AA != 0) {
      const bool first = c == x0, last = c + 1 == x0 + OUT - 1 || c + 1 == L.nx - 1;
      if (out1 && !first && !last) *reinterpret_cast<float2*>(p) = q;
      else if (out1 && !first) *p = q.x;
      else if (out1 && !last) p[1] = q.y;
      continue;
    }
    if (out1) *reinterpret_cast<float2*>(p) = q;
  }
}

template <bool PSEUDO, int H, int W, int MINB, int AA = 0>
__global__ void __launch_bounds__(32 * W, MINB) k_tile(const __grid_constant__ Lattice<float> L, int cur, int strips, int rows) {
  extern __shared__ __align__(16) char smem[];
  const int band = blockIdx.x / strips, strip = blockIdx.x - band * strips;
  const int ya = band * rows, yb = min(ya + rows, L.ny);
  grid_wait();
  grid_launch();
  tile<PSEUDO, H, W, AA>(L, cur, strip, ya, yb, smem);
}
template <int H, int W, int MINB>
__global__ void __launch_bounds__(32 * W, MINB) k_tile_batch(const Lattice<float>* lat, const int4* items, int cur) {
  extern __shared__ __align__(16) char smem[];
  __shared__ __align__(16) Lattice<float> L;
  const int4 it = items[blockIdx.x];
  take_lattice(L, lat, it.x);
  __syncthreads();
  grid_wait();
  grid_launch();
  tile<false, H, W>(L, cur, it.y, it.z, it.z + it.w, smem);
}

constexpr int BC_BLOCK = 64;
template <bool PSEUDO, int AA = 0>
__global__ void __launch_bounds__(BC_BLOCK) k_bc_fused(const __grid_constant__ Lattice<float> L, int cur) {
  links<PSEUDO, true, AA>(L, cur, blockIdx.x * BC_BLOCK + threadIdx.x);
}
// item: (instance, first boundary node)
__global__ void __launch_bounds__(BC_BLOCK) k_bc_batch(const Lattice<float>* lat, const int2* items, int cur) {
  __shared__ __align__(16) Lattice<float> L;
  const int2 it = items[blockIdx.x];
  take_lattice(L, lat, it.x);
  __syncthreads();
  links<false, true>(L, cur, it.y + threadIdx.x);
}

constexpr int SOLID_BLOCK = 256;
template <bool PSEUDO>
__global__ void __launch_bounds__(SOLID_BLOCK) k_solids(const __grid_constant__ Lattice<float> L, int blocks2, int blocks1,
                                                        int steps) {
  solids<PSEUDO, SOLID_BLOCK>(L, blockIdx.x, blocks2, blocks1, steps);
}
// The solid layers of an AA lattice and, in blocks of their own, the densities its pass leaves: the
// outermost rows of the bands (edge_rows of them) and columns of the strips, from the populations of
// the state in slot order `cur`, which the links have completed.  A column of a large lattice is a
// memory access of its own for each population (35 us of 2048 x 4096): there (WALK) the walks hand
// those columns' populations on in aa_edge, and only the lattice's own ends are read that way.
template <bool PSEUDO, bool WALK>
__global__ void __launch_bounds__(SOLID_BLOCK) k_layers_aa(const __grid_constant__ Lattice<float> L, int blocks2, int blocks1,
                                                           int cur, int strips, int rows, int edge_rows) {
  const int blk = (int)blockIdx.x - (blocks2 + blocks1 + 1);
  if (blk < 0) {
    solids<PSEUDO, SOLID_BLOCK>(L, blockIdx.x, blocks2, blocks1, 1);
    return;
  }
  unsigned e = (unsigned)blk * SOLID_BLOCK + threadIdx.x;
  const unsigned in_rows = (unsigned)edge_rows * (unsigned)L.nx, ends = WALK ? 2u * L.ny : 0u;
  int x = 0, y = L.ny;
  const float* from = nullptr;
  if (e < in_rows) {
    const int k = (int)(e / (unsigned)L.nx), ya = (k >> 1) * rows;
    x = (int)(e - (unsigned)k * L.nx);
    y = k & 1 ? min(ya + rows, L.ny) - 1 : ya;
  } else if ((e -= in_rows) < ends) {
    y = (int)(e >> 1);
    x = e & 1u ? L.nx - 1 : 0;
  } else if (WALK) {
    // the columns left (x) and right of boundary b between two strips
    e -= ends;
    const unsigned b = e / (unsigned)L.ny;
    if ((int)b < strips - 1) {
      y = (int)(e - b * L.ny);
      x = (int)(b + 1) * OUT - 1;
      from = L.aa_edge + 16ll * e;
    }
  } else {
    y = (int)(e / (2u * strips));
    const int k = (int)(e - (unsigned)y * (2u * strips));
    // (the last column of a strip and the first of the next are neighbours in the list)
    x = k == 2 * strips - 1 ? L.nx - 1 : ((k + 1) >> 1) * OUT - (k & 1);
  }
  const int n = y * L.pitch + x;
  if (WALK && from) {
    // not next to a solid node (a boundary node has its density from the links), nor an end or in an
    // outermost row
    const int ya = y / rows * rows;
    const bool inside = y > ya && y < min(ya + rows, L.ny) - 1;   // (rows y - 1 and y + 1 exist)
    bool all[4];   // all of a column's three nodes fluid: x - 1 .. x + 2
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      all[k] = inside;
      if (inside) {
#pragma unroll
        for (int d = -1; d <= 1; ++d) all[k] &= L.kind[node_at(L, x - 1 + k, y + d)] == KIND_FLUID;
      }
    }
    const bool left = all[0] && all[1] && all[2], right = all[1] && all[2] && all[3] && x + 1 < L.nx - 1;
    grid_wait();
    grid_launch();
    if (!left && !right) return;
    // record of the strip left of the boundary, then of the one right of it
    const float4* p = reinterpret_cast<const float4*>(from);
    const float4 h0 = p[0], h1 = p[1], g0 = p[2], g1 = p[3];
    auto put = [&](int at, float f0, float f1, float f3, float f24, float f5, float f7, float f6, float f8) {
      const float sum = add_rn(f0, add_rn(add_rn(add_rn(f1, f3), f24), add_rn(add_rn(f5, f7), add_rn(f6, f8))));
      const float r = add_rn(L.rho_ref, sum);
      L.rho_next[at] = PSEUDO ? psi_of(L, r) : r;
    };
    if (left) put(n, h0.x, h0.y, g1.y, h0.z, h0.w, g1.w, g1.z, h1.x);
    if (right) put(n + 1, g0.x, h1.y, g0.y, g0.z, h1.z, g1.x, g0.w, h1.w);
    return;
  }
  const bool live = y < L.ny && L.kind[n] == KIND_FLUID;
  grid_wait();
  grid_launch();
  if (!live) return;
  float v[9];
  load_pops(L, cur, x, y, v);
  const float r = density_of(L, v);
  L.rho_next[n] = PSEUDO ? psi_of(L, r) : r;
}
// item: (instance, its block)
__global__ void __launch_bounds__(SOLID_BLOCK) k_solids_batch(const Lattice<float>* lat, const int2* items, int steps) {
  __shared__ __align__(16) Lattice<float> L;
  const int2 it = items[blockIdx.x];
  take_lattice(L, lat, it.x);
  __syncthreads();
  solids<false, SOLID_BLOCK>(L, it.y, (8 * L.n_s2 + SOLID_BLOCK - 1) / SOLID_BLOCK, (L.n_s1 + SOLID_BLOCK - 1) / SOLID_BLOCK, steps);
}

// ---------------------------------------------------------------------------------------
// Read-out of a state whose density (psi) plane is current, in one launch: density and v = u +
// F/(2 rho) into dense nx x ny arrays (k_fields' values).  A block forms the chemical potentials its
// rows' forces need from the staged density rows; the populations go straight to registers.
constexpr int RO_H = 8, RO_W = 4;
template <bool PSEUDO>
__global__ void __launch_bounds__(32 * RO_W) k_fields_fused(const __grid_constant__ Lattice<float> L, int cur, int strips,
                                                            float* __restrict__ rho_out, float* __restrict__ vx_out,
                                                            float* __restrict__ vy_out) {
  constexpr int MR = 2, RR = PSEUDO ? 1 : 4;   // chemical-potential and density rows beyond the outputs
  __shared__ __align__(16) float2 s_rho[(RO_H + 2 * RR) * SP];
  __shared__ __align__(16) float2 s_mu[PSEUDO ? 1 : (RO_H + 2 * MR) * SP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int band = blockIdx.x / strips, strip = blockIdx.x - band * strips;
  const int ya = band * RO_H, yb = min(ya + RO_H, L.ny);
  const int x0 = strip * OUT, c = x0 - HX + 2 * lane;
  const bool mine = lane >= HX / 2 && lane < 32 - HX / 2;
  const int ca = wrap_col(c, L.nx), cb = wrap_col(c + 1, L.nx);
  const float* __restrict__ rin = PSEUDO ? L.mu : L.rho;
  auto row_at = [&](int r) {
    if (L.walls) r = min(max(r, 0), L.ny - 1);
    else r = r < 0 ? r + L.ny : (r >= L.ny ? r - L.ny : r);
    return r * L.pitch;
  };
  int e[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) e[j] = wrap_col(x0 - 2 * HX + lane + 32 * j, L.nx);
  for (int r = ya - RR + warp; r < yb + RR; r += RO_W) {
    float* const d = reinterpret_cast<float*>(s_rho + (r - ya + RR) * SP);
    const float* const q = rin + row_at(r);
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (lane + 32 * j < 2 * SP) d[lane + 32 * j] = q[e[j]];
  }
  __syncthreads();
  if (!PSEUDO) {
    for (int m = ya - MR + warp; m < yb + MR; m += RO_W) {
      const float2* q = s_rho + (m - ya + RR) * SP + HX / 2 + lane;
      const float2 C = q[0], l = q[-1], g = q[1], u1 = q[SP], u2 = q[2 * SP], d1 = q[-SP], d2 = q[-2 * SP];
      const float t = sub_rn(C.y, C.x);
      const float2 x1 = make_float2(add_rn(t, sub_rn(l.y, C.x)), add_rn(sub_rn(g.x, C.y), -t));
      const float2 lap = lap4_diff(x1, add_rn(sub_rn(C, g), sub_rn(C, l)), add_rn(sub_rn(u1, C), sub_rn(d1, C)),
                                   add_rn(sub_rn(C, u2), sub_rn(C, d2)));
      float2 mu = mu_of(L, psi_prime_shifted(L, C), lap);
      const int n = row_at(m);
      if (L.kind[n + ca] != KIND_FLUID) mu.x = L.mu[n + ca];
      if (L.kind[n + cb] != KIND_FLUID) mu.y = L.mu[n + cb];
      s_mu[(m - ya + MR) * SP + HX / 2 + lane] = mu;
    }
    __syncthreads();
  }
  for (int y = ya + warp; y < yb; y += RO_W) {
    const int n = y * L.pitch;
    const bool f0 = L.kind[n + ca] == KIND_FLUID, f1 = L.kind[n + cb] == KIND_FLUID;
    float2 r = make_float2(0.f, 0.f), vx = r, vy = r;
    if (f0 || f1) {
      const float* __restrict__ f = L.f[cur] + n;
      float2 v[9], drho, jx, jy, Fx, Fy;
      if (L.aa && cur == 1) {
        float a[9], b[9];
        load_pops(L, cur, ca, y, a);
        load_pops(L, cur, cb, y, b);
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = make_float2(a[i], b[i]);
      } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = make_float2(f[i * (long long)L.plane + ca], f[i * (long long)L.plane + cb]);
      }
      moments(v, drho, jx, jy);
      const float2 rho = add_rn(splat<float2>(L.rho_ref), drho);
      const float2* q = s_rho + (y - ya + RR) * SP + HX / 2 + lane;
      if constexpr (PSEUDO) {
        const float2 C = q[0], U = q[SP], D = q[-SP];
        float2 ax, ay;
        pp_sums(make_float2(C.y, q[1].x), U, make_float2(q[-1].y, C.x), D, make_float2(U.y, q[SP + 1].x),
                make_float2(q[SP - 1].y, U.x), make_float2(q[-SP - 1].y, D.x), make_float2(D.y, q[-SP + 1].x), ax, ay);
        Fx = force_pp(rho, L.gx, C, ax);
        Fy = force_pp(rho, L.gy, C, ay);
      } else {
        const float2* z = s_mu + (y - ya + MR) * SP + HX / 2 + lane;
        auto dx_of = [](const float2* p) {
          const float2 l = p[-1], C = p[0], g = p[1];
          return fma_rn(splat<float2>(8.0f), make_float2(sub_rn(C.y, l.y), sub_rn(g.x, C.x)), sub_rn(l, g));
        };
        Fx = force_cp(rho, L.gx, dx_of(z), dx_of(q));
        Fy = force_cp(rho, L.gy, diff4_of(z[SP], z[-SP], z[2 * SP], z[-2 * SP]), diff4_of(q[SP], q[-SP], q[2 * SP], q[-2 * SP]));
      }
      if (f0) { r.x = rho.x; vx.x = fmaf(0.5f, Fx.x, jx.x) / rho.x; vy.x = fmaf(0.5f, Fy.x, jy.x) / rho.x; }
      if (f1) { r.y = rho.y; vx.y = fmaf(0.5f, Fx.y, jx.y) / rho.y; vy.y = fmaf(0.5f, Fy.y, jy.y) / rho.y; }
    }
    if (!mine || c >= L.nx) continue;
    const long long d = (long long)y * L.nx + c;
    if (c + 1 < L.nx && (d & 1) == 0) {
      *reinterpret_cast<float2*>(rho_out + d) = r;
      *reinterpret_cast<float2*>(vx_out + d) = vx;
      *reinterpret_cast<float2*>(vy_out + d) = vy;
    } else {
      rho_out[d] = r.x;
      vx_out[d] = vx.x;
      vy_out[d] = vy.x;
      if (c + 1 < L.nx) {
        rho_out[d + 1] = r.y;
        vx_out[d + 1] = vx.y;
        vy_out[d + 1] = vy.y;
      }
    }
  }
}

// A new state (set up, loaded or advanced by the separate passes) in lattice `cur`: the density
// (psi) of its fluid nodes into rho_next, and of its boundary nodes into rho_b, from which k_solids
// forms the solid layers.
template <bool PSEUDO>
__device__ __forceinline__ void density(const Lattice<float>& L, int cur, int x, int y) {
  const int n = y * L.pitch + x;
  if (x >= L.nx || L.kind[n] != KIND_FLUID) return;
  float v[9];
  load_pops(L, cur, x, y, v);
  const float r = density_of(L, v);
  L.rho_next[n] = PSEUDO ? psi_of(L, r) : r;
}
template <bool PSEUDO>
__global__ void __launch_bounds__(128) k_density(const __grid_constant__ Lattice<float> L, int cur, int per_row) {
  const int y = blockIdx.x / per_row;
  density<PSEUDO>(L, cur, (blockIdx.x - y * per_row) * 128 + threadIdx.x, y);
}
// a batch: the pass's items (64 threads cover a strip's columns)
__global__ void __launch_bounds__(64) k_density_batch(const Lattice<float>* lat, const int4* items, int cur) {
  __shared__ __align__(16) Lattice<float> L;
  const int4 it = items[blockIdx.x];
  take_lattice(L, lat, it.x);
  __syncthreads();
  if (threadIdx.x >= OUT) return;
  for (int y = it.z; y < it.z + it.w; ++y) density<false>(L, cur, it.y * OUT + threadIdx.x, y);
}
__device__ __forceinline__ void boundary_density(const Lattice<float>& L, int cur, int b) {
  if (b >= L.n_bnodes) return;
  const int n = L.bnode[b];
  float v[9];
  load_pops(L, cur, n % L.pitch, n / L.pitch, v);
  L.rho_b[b] = density_of(L, v);
  if (L.aa) moments(v, L.bmom[3 * b], L.bmom[3 * b + 1], L.bmom[3 * b + 2]);
}
__global__ void __launch_bounds__(128) k_boundary_density(const __grid_constant__ Lattice<float> L, int cur) {
  boundary_density(L, cur, blockIdx.x * blockDim.x + threadIdx.x);
}
__global__ void __launch_bounds__(BC_BLOCK) k_boundary_density_batch(const Lattice<float>* lat, const int2* items, int cur) {
  __shared__ __align__(16) Lattice<float> L;
  const int2 it = items[blockIdx.x];
  take_lattice(L, lat, it.x);
  __syncthreads();
  boundary_density(L, cur, it.y + threadIdx.x);
}

inline unsigned blocks_for(int n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

static long long fused_tiles(int nx, int ny) { return (long long)((nx + OUT - 1) / OUT) * ((ny + TH_M - 1) / TH_M); }
constexpr int MIN_TILE_ROWS = 2;

// How the pass runs on a lattice of nx x ny, counted in tiles of 14 rows:
//   from 10 tiles an SM on the walk wins, whose rows are formed twice only at the bands' ends and
//   whose loads run through all of its rows (walk / tiles, us a step: 1001 x 1024 (8.8 tiles) 35.8 /
//   32.0, 1024 x 1024 (9.3) 32.6 / 33.2, 1201 x 1300 (13.5) 43.4 / 46.0, 1024 x 1536 (13.8) 37.1 / 45.2,
//   1200 x 2200 (22.7) 57 / 67, 2048 x 4096 148 / 175).  A walk takes as many rows as give every SM the
//   twelve warps that fit at once (one wave / two: 1671 x 2453 87 / 92, 2048 x 2048 84 / 87), but where
//   that is more than 64 rows half as many, so that the walks that take longer (strips at an end with
//   nx % 4 != 0, rows with solids) do not set the pass's time alone (2048 x 4096 151 / 148).
//   below, tiles of at most 14 rows and eight warps, or (from 6 tiles an SM) 10 rows and four warps,
//   of which five fit an SM and so overlap their phases better (800 x 800 21.7 / 22.8).  The bands have
//   equal heights and as many as give every SM the same number of tiles (500 x 300 13.0 -> 11.8, 96 x 96
//   10.3 -> 8.2).
PassPlan fused_plan(int nx, int ny, int sms) {
  const int strips = (nx + OUT - 1) / OUT;
  const long long tiles = fused_tiles(nx, ny);
  PassPlan p;
  if (tiles >= 10LL * sms) {
    p.kind = PassPlan::WALK;
    auto rows = [&](int per_sm) {
      const long long bands = std::max(1LL, (long long)per_sm * sms / strips);
      return std::max(8, (int)((ny + bands - 1) / bands));
    };
    p.rows = rows(12);
    if (p.rows > 64) p.rows = rows(24);
    return p;
  }
  p.kind = tiles >= 6LL * sms ? PassPlan::TILE_L : PassPlan::TILE_M;
  const int most = p.kind == PassPlan::TILE_L ? TH_L : TH_M;
  const long long least = (ny + most - 1) / most, per_sm = (strips * least + sms - 1) / sms;
  const long long bands = std::max(least, per_sm * sms / strips);
  p.rows = std::max((int)((ny + bands - 1) / bands), MIN_TILE_ROWS);
  return p;
}

// the same without the walk (whose kernel keeps no chemical potential)
PassPlan fused_tile_plan(int nx, int ny, int sms) {
  PassPlan p = fused_plan(nx, ny, sms);
  if (p.kind != PassPlan::WALK) return p;
  p.kind = PassPlan::TILE_L;
  p.rows = TH_L;
  return p;
}

// ... of an AA lattice: the same walks; its tiles are of the first shape, whose bands leave fewer
// outermost rows to k_layers_aa.  (separate passes / fused, us a step: 131 x 97 24.6 / 9.3, 512 x 512
// 30 / 15.4, 1024 x 1024 46 / 33, 1600 x 2000 95 / 80, 2048 x 4096 206 / 172.)
PassPlan fused_aa_plan(int nx, int ny, int sms) {
  PassPlan p = fused_plan(nx, ny, sms);
  if (p.kind != PassPlan::TILE_L) return p;
  p.kind = PassPlan::TILE_M;
  p.rows = TH_M;
  return p;
}

bool fused_setup() {
  auto allow = [](const void* k, int bytes) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
  };
  return allow((const void*)k_tile<false, TH_M, TW_M, TB_M>, Tile<false, TH_M>::BYTES) &&
         allow((const void*)k_tile<true, TH_M, TW_M, TB_M>, Tile<true, TH_M>::BYTES) &&
         allow((const void*)k_walk_batch, Reach<false>::BYTES) &&
         allow((const void*)k_tile<false, TH_L, TW_L, TB_L>, Tile<false, TH_L>::BYTES) &&
         allow((const void*)k_tile<true, TH_L, TW_L, TB_L>, Tile<true, TH_L>::BYTES) &&
         allow((const void*)k_tile_batch<TH_L, TW_L, TB_L>, Tile<false, TH_L>::BYTES) &&
         allow((const void*)k_tile<false, TH_M, TW_M, TB_M, 1>, Tile<false, TH_M>::BYTES) &&
         allow((const void*)k_tile<false, TH_M, TW_M, TB_M, 2>, Tile<false, TH_M>::BYTES) &&
         allow((const void*)k_tile<true, TH_M, TW_M, TB_M, 1>, Tile<true, TH_M>::BYTES) &&
         allow((const void*)k_tile<true, TH_M, TW_M, TB_M, 2>, Tile<true, TH_M>::BYTES) &&
         allow((const void*)k_walk<false, 1>, Reach<false>::BYTES) && allow((const void*)k_walk<false, 2>, Reach<false>::BYTES) &&
         allow((const void*)k_walk<true, 1>, Reach<true>::BYTES) && allow((const void*)k_walk<true, 2>, Reach<true>::BYTES) &&
         allow((const void*)k_walk<false>, Reach<false>::BYTES) && allow((const void*)k_walk<true>, Reach<true>::BYTES);
}

static cudaError_t launch_solids(const Lattice<float>& L, int steps, cudaStream_t s) {
  const int b2 = (int)blocks_for(8 * L.n_s2, SOLID_BLOCK), b1 = (int)blocks_for(L.n_s1, SOLID_BLOCK);
  return launch_after(L.pseudo ? k_solids<true> : k_solids<false>, dim3((unsigned)(b2 + b1 + 1)), SOLID_BLOCK, 0, s, L, b2, b1, steps);
}

cudaError_t launch_fused_prepare(const Lattice<float>& L, int cur, cudaStream_t s) {
  const unsigned per_row = blocks_for(L.nx, 128), grid = per_row * (unsigned)L.ny;
  if (L.pseudo) k_density<true><<<grid, 128, 0, s>>>(L, cur, (int)per_row);
  else k_density<false><<<grid, 128, 0, s>>>(L, cur, (int)per_row);
  if (L.n_bnodes > 0) k_boundary_density<<<blocks_for(L.n_bnodes, 128), 128, 0, s>>>(L, cur);
  return launch_solids(L, 0, s);
}

template <int H, int W, int B>
static cudaError_t launch_tiles(const Lattice<float>& L, int cur, int rows, cudaStream_t s) {
  const int strips = (L.nx + OUT - 1) / OUT, bands = (L.ny + rows - 1) / rows;
  return L.pseudo ? launch_after(k_tile<true, H, W, B>, dim3((unsigned)(strips * bands)), 32 * W, Tile<true, H>::BYTES, s, L, cur, strips, rows)
                  : launch_after(k_tile<false, H, W, B>, dim3((unsigned)(strips * bands)), 32 * W, Tile<false, H>::BYTES, s, L, cur, strips, rows);
}
static cudaError_t launch_pass(const Lattice<float>& L, int cur, PassPlan p, cudaStream_t s) {
  if (p.kind == PassPlan::TILE_M) return launch_tiles<TH_M, TW_M, TB_M>(L, cur, p.rows, s);
  if (p.kind == PassPlan::TILE_L) return launch_tiles<TH_L, TW_L, TB_L>(L, cur, p.rows, s);
  const int strips = (L.nx + OUT - 1) / OUT, bands = (L.ny + p.rows - 1) / p.rows;
  return L.pseudo ? launch_after(k_walk<true>, dim3((unsigned)(strips * bands)), 32, Reach<true>::BYTES, s, L, cur, strips, p.rows)
                  : launch_after(k_walk<false>, dim3((unsigned)(strips * bands)), 32, Reach<false>::BYTES, s, L, cur, strips, p.rows);
}

cudaError_t launch_fused_step(const Lattice<float>& L, int cur, PassPlan plan, cudaStream_t s, unsigned parts) {
  cudaError_t e = parts & PART_PASS ? launch_pass(L, cur, plan, s) : cudaSuccess;
  if (e == cudaSuccess && L.n_bnodes > 0 && (parts & PART_LINKS))
    e = launch_after(L.pseudo ? k_bc_fused<true> : k_bc_fused<false>, dim3(blocks_for(L.n_bnodes, BC_BLOCK)), BC_BLOCK, 0, s, L, cur);
  return e == cudaSuccess && (parts & PART_LAYERS) ? launch_solids(L, 1, s) : e;
}

// One lattice in AA order, from slot order cur
cudaError_t launch_fused_step_aa(const Lattice<float>& L, int cur, PassPlan p, cudaStream_t s, unsigned parts) {
  const int strips = (L.nx + OUT - 1) / OUT, bands = (L.ny + p.rows - 1) / p.rows;
  const dim3 grid((unsigned)(strips * bands)), nb(blocks_for(L.n_bnodes, BC_BLOCK));
  const int b2 = (int)blocks_for(8 * L.n_s2, SOLID_BLOCK), b1 = (int)blocks_for(L.n_s1, SOLID_BLOCK);
  const int edge_rows = 2 * bands;
  // (strips <= nx / OUT + 1 and rows >= 2: at most twice the lattice's nodes, 32-bit)
  const unsigned edge = (unsigned)edge_rows * (unsigned)L.nx +
                        (p.kind == PassPlan::WALK ? strips + 1u : 2u * (unsigned)strips) * (unsigned)L.ny;
  const dim3 layers((unsigned)(b2 + b1 + 1) + (edge + SOLID_BLOCK - 1) / SOLID_BLOCK);
  auto tiles = [&](auto* k, int bytes) { return launch_after(k, grid, 32 * TW_M, bytes, s, L, cur, strips, p.rows); };
  auto walks = [&](auto* k, int bytes) { return launch_after(k, grid, 32, bytes, s, L, cur, strips, p.rows); };
  cudaError_t e = cudaSuccess;
  if (!(parts & PART_PASS)) {
  } else if (p.kind == PassPlan::WALK) {
    if (L.pseudo) e = cur ? walks(k_walk<true, 2>, Reach<true>::BYTES) : walks(k_walk<true, 1>, Reach<true>::BYTES);
    else e = cur ? walks(k_walk<false, 2>, Reach<false>::BYTES) : walks(k_walk<false, 1>, Reach<false>::BYTES);
  } else if (L.pseudo) e = cur ? tiles(k_tile<true, TH_M, TW_M, TB_M, 2>, Tile<true, TH_M>::BYTES)
                        : tiles(k_tile<true, TH_M, TW_M, TB_M, 1>, Tile<true, TH_M>::BYTES);
  else e = cur ? tiles(k_tile<false, TH_M, TW_M, TB_M, 2>, Tile<false, TH_M>::BYTES)
               : tiles(k_tile<false, TH_M, TW_M, TB_M, 1>, Tile<false, TH_M>::BYTES);
  if (e == cudaSuccess && L.n_bnodes > 0 && (parts & PART_LINKS)) {
    auto bc = [&](auto* k) { return launch_after(k, nb, BC_BLOCK, 0, s, L, cur); };
    if (L.pseudo) e = cur ? bc(k_bc_fused<true, 2>) : bc(k_bc_fused<true, 1>);
    else e = cur ? bc(k_bc_fused<false, 2>) : bc(k_bc_fused<false, 1>);
  }
  if (e != cudaSuccess || !(parts & PART_LAYERS)) return e;
  auto* k = p.kind == PassPlan::WALK ? (L.pseudo ? k_layers_aa<true, true> : k_layers_aa<false, true>)
                                     : (L.pseudo ? k_layers_aa<true, false> : k_layers_aa<false, false>);
  return launch_after(k, layers, SOLID_BLOCK, 0, s, L, b2, b1, cur ^ 1, strips, p.rows, edge_rows);
}

// ---- batches
void fused_batch_items(int k, int nx, int ny, int n_bnodes, int n_s1, int n_s2, int rows, std::vector<int4>* pass,
                       std::vector<int2>* bc, std::vector<int2>* solid) {
  const int strips = (nx + OUT - 1) / OUT;
  const int most = rows > 0 ? rows : TH_L, bands = (ny + most - 1) / most;
  const int per = (ny + bands - 1) / bands;   // bands of equal height
  for (int b = 0; b * per < ny; ++b)
    for (int st = 0; st < strips; ++st) pass->push_back(make_int4(k, st, b * per, std::min(per, ny - b * per)));
  for (int b = 0; b < n_bnodes; b += BC_BLOCK) bc->push_back(make_int2(k, b));
  const int blocks = (int)(blocks_for(8 * n_s2, SOLID_BLOCK) + blocks_for(n_s1, SOLID_BLOCK)) + 1;
  for (int b = 0; b < blocks; ++b) solid->push_back(make_int2(k, b));
}
// upper bounds of the three lists for one instance
void fused_batch_caps(int nx, int ny, long long bnodes, long long s1, long long s2, long long* pass, long long* bc,
                      long long* solid) {
  *pass += (long long)((nx + OUT - 1) / OUT) * ((ny + TH_L - 1) / TH_L);
  *bc += (bnodes + BC_BLOCK - 1) / BC_BLOCK;
  *solid += (8 * s2 + SOLID_BLOCK - 1) / SOLID_BLOCK + (s1 + SOLID_BLOCK - 1) / SOLID_BLOCK + 1;
}
// Rows a warp of the batch walks, or 0 for tiles: 64 walks an SM, several waves that even out the
// instances' widths and solids (48 / 64 / 96: 367 / 364 / 375 us a step on 64 lattices of 128..768), if
// that leaves them 20 rows (walk / tiles, with its rows: 64 of 128..768 (30 rows) 368 / 401, 60 of
// 200..400 (11) 196 / 180, 12 of 500..768 (11) 152 / 133, 256 of 64..128 (5) 144 / 121).
int fused_batch_rows(long long strip_rows, int sms) {
  const long long rows = strip_rows / (64LL * sms);
  return rows < 20 ? 0 : (int)rows;
}
long long fused_strip_rows(int nx, int ny) { return (long long)((nx + OUT - 1) / OUT) * ny; }

cudaError_t launch_fused_batch_prepare(const FusedBatch& B, int cur, cudaStream_t s) {
  const Lattice<float>* lat = B.lat[cur ^ 1];   // whose next plane is this state's
  k_density_batch<<<B.n_pass, 64, 0, s>>>(lat, B.pass, cur);
  if (B.n_bc > 0) k_boundary_density_batch<<<B.n_bc, BC_BLOCK, 0, s>>>(lat, B.bc, cur);
  k_solids_batch<<<B.n_solid, SOLID_BLOCK, 0, s>>>(lat, B.solid, 0);
  return cudaGetLastError();
}
cudaError_t launch_fused_batch_step(const FusedBatch& B, int cur, cudaStream_t s) {
  const Lattice<float>* lat = B.lat[cur];
  cudaError_t e = B.rows > 0 ? launch_after(k_walk_batch, dim3((unsigned)B.n_pass), 32, Reach<false>::BYTES, s, lat, B.pass, cur)
                             : launch_after(k_tile_batch<TH_L, TW_L, TB_L>, dim3((unsigned)B.n_pass), 32 * TW_L, Tile<false, TH_L>::BYTES, s, lat,
                                            B.pass, cur);
  if (e == cudaSuccess && B.n_bc > 0) e = launch_after(k_bc_batch, B.n_bc, BC_BLOCK, 0, s, lat, B.bc, cur);
  return e == cudaSuccess ? launch_after(k_solids_batch, B.n_solid, SOLID_BLOCK, 0, s, lat, B.solid, 1) : e;
}

cudaError_t launch_fused_fields(const Lattice<float>& L, int cur, float* r, float* vx, float* vy, cudaStream_t s) {
  const int strips = (L.nx + OUT - 1) / OUT, bands = (L.ny + RO_H - 1) / RO_H;
  if (L.pseudo) k_fields_fused<true><<<dim3((unsigned)(strips * bands)), 32 * RO_W, 0, s>>>(L, cur, strips, r, vx, vy);
  else k_fields_fused<false><<<dim3((unsigned)(strips * bands)), 32 * RO_W, 0, s>>>(L, cur, strips, r, vx, vy);
  return cudaGetLastError();
}

int fused_launches(const Lattice<float>& L) { return 2 + (L.n_bnodes > 0 ? 1 : 0); }

}  // namespace lbmgb
