// Device-side building blocks of the multiphase curved-boundary LBM step (sm_103a).
//
// Layout in HBM (one lattice): every per-node quantity is a plane of `pitch * ny` elements,
// node (x, y) at y*pitch + x with pitch = nx rounded up to a 128-byte multiple, so that each
// row starts on a cache-line boundary and a warp touches whole lines.  Populations are 9
// such planes (structure of arrays) per lattice, two lattices A/B swapped every step, stored
// in offset form  f_i - w_i rho_ref.  Padding nodes (x >= nx) carry kind KIND_PAD and are
// never read as data.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace lbmgb {

enum : uint8_t { KIND_FLUID = 0, KIND_SOLID1 = 1, KIND_SOLID2 = 2, KIND_DEEP = 3, KIND_PAD = 255 };
enum { EOS_NONE = 0, EOS_CS = 1, EOS_PR = 2 };
enum { COLL_BGK = 0, COLL_MRT = 1 };
enum { BC_PRESENT = 0, BC_IBC = 1, BC_MIBC = 2, BC_HBB = 3 };
constexpr int DM_RING = 4096;

// D2Q9 velocities in the order of the columns of the transformation matrix M (Eq. 2).
__host__ __device__ constexpr int ex(int i) { return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }
__host__ __device__ constexpr int ey(int i) { return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0); }
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : (i <= 4 ? ((i + 1) & 3) + 1 : ((i - 3) & 3) + 5); }
__host__ __device__ constexpr double wgt(int i) { return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }

// Everything a kernel needs to address one lattice and evaluate its physics.
template <typename real>
struct Lattice {
  int nx, ny, pitch, walls;
  int plane;                    // pitch * ny (9 * plane < 2^31)
  real* f[2];                   // the two population lattices (9 planes each); with aa set both
                                // point at the one lattice, updated in place
  int aa;                       // one lattice (AA order): the state of lattice 0 is in natural
                                // order, that of lattice 1 holds f_i(x) in slot opp(i) of x - e_i
  real* bmom;                   // aa: per boundary node, the pre-collision (delta rho, jx, jy) the
                                // boundary phase needs, saved before the collide overwrites them
  real* rho;                    // density plane (fluid and the two solid layers)
  real* rho_b;                  // if set: the boundary phase leaves the density of each
                                // boundary node's final populations here (one per node)
  real* mu;                     // chemical potential minus k^2 mu_sat (constant at solids)
  real* rho_next;               // fused and FP64 steps: the next state's density (psi) plane
  real* mu_out;                 // ... if set (tiles): this state's chemical potential is kept here
  real* aa_edge;                // ... in AA order, walked: what the strips left and right of a boundary between
                                // two hand on of their outermost columns, 2 x 8 values a row, by boundary
  real* fx;                     // fused step (FP32): the force at nodes next to solids, left by
  real* fy;                     // the pass for the boundary phase
  real* psip;                   // if set: psi'(rho) - mu_sat of every fluid node, left by the
                                // density pass for the chemical-potential pass (single lattices)
  const uint8_t* kind;
  const int* body;              // body of each solid node (cylinders 0.., then bottom, top wall)
  const double* cyl;            // per cylinder: cx, cy, r, wall chemical-potential offset
  // equation of state, Eq. 12: mu~ = k^2 (psi'(rho) - mu_sat) - kappa lap(rho)
  int eos;
  real RT, a, b, aalpha, k2, kappa, mu_sat;
  real rho_split;                // sqrt(rho_g rho_l): below it mu is evaluated against rho_g
  // CS, per reference density rho0 in {rho_g, rho_l} (index 0 gas, 1 liquid), storage-rounded:
  // rho0, 1/rho0, the coefficients of N(h) (psi_prime_cs), psi'(rho0) - mu_sat (FP64 on the host)
  real b4;                       // b / 4
  real cs_r0[2], cs_inv_r0[2], cs_m0[2], cs_m1[2], cs_m2[2], cs_c0[2];
  // PR, besides rho0, 1/rho0 and psi'(rho0) - mu_sat: -K; 2 sqrt 2 b/(c1+x0), x0, RT b/(1-x0),
  // -a alpha/D0 (psi_prime_pr)
  real pr_nk, pr_kb[2], pr_x0[2], pr_rtb[2], pr_naD[2];
  real rho_ref;
  // collision, Eqs. 3-4
  int coll;
  real omega;                   // 1 / tau (BGK)
  real s_e, s_eps, s_q, s_nu;
  real nke36, kp36, kq12, kn4;  // (s_e - 1)/36, (1 - s_eps)/36, (1 - s_q)/12, (1 - s_nu)/4
  real gx, gy;
  int bc;
  // pseudopotential force model (instead of Eqs. 9 and 12): mu holds psi, the solid layers
  // psi(rho_s) (1 + c_w) with c_w = cyl[4 b + 3] of cylinder b, cw_walls of the flat walls
  int pseudo;
  int n_cyl;
  double cw_walls;
  // cut links, CSR over boundary-fluid nodes sorted by node
  int n_bnodes;
  const int* bnode;
  const int* bstart;
  const uint8_t* ldir;
  const real* lq;
  const uint8_t* lx2f;
  // the same by boundary node: node and column; bits 0-7 the directions 1-8 it cuts, bits
  // 8-15 whether x2 is fluid there; q of direction i at bq[(i - 1) bcap + b]
  const int2* bnd;
  const unsigned short* bmask;
  const real* bq;
  int bcap;
  // first and second solid layers for Eq. 15
  int n_s1, n_s2;
  const int* s1node;
  const uint8_t* s1mask;         // bit i-1 set: neighbour e_i (i = 1..8) contributes
  const int* s1nb;              // per first-layer entry, 8 ints: the boundary-node index of each
                                // contributing neighbour (-1 elsewhere)
  const real* s1winv;
  const int* s2nb;              // per second-layer entry, 8 ints: the first-layer index of each
                                // contributing neighbour (-1 elsewhere)
  const int* s2node;
  const uint8_t* s2mask;
  const real* s2winv;
  double* carry;                // per boundary node: Eq. 18 residual below storage precision
  // reductions (FP64)
  double* partials;             // per-block partial sums
  unsigned int* counter;        // last-block-done counter (returns to 0)
  double* dM_ring;              // per-step domain sum of the Eq. 18 compensation
  unsigned long long* step_ctr; // steps taken (device side)
  double* scalars;              // [0] mass, [1] non-finite count
  unsigned int* kerr;           // set by a kernel whose bounded wait gave up (0 otherwise)
  long long spin_limit;         // polls before a pipelined kernel's wait for its loads gives up
                                // (its wait for copies in flight before leaving keeps the full limit)
  int mu_kernel;                // host side: the chemical-potential pass (0 per node, 1 row
                                // vectors, 2 row sweeps, FP32 only; 3: formed with the next
                                // state's density in one tiled pass, then near_list fixed up)
  int n_near;                   // fluid nodes whose chemical-potential stencil reaches a solid or
  const int* near_list;         // a boundary node (their mu waits for the boundary phase)
  const void* tma;              // host side: TMA descriptors of the pipelined collide kernel
                                // (FP32), null for the plain kernel
  int sweep;                    // host side: the step's collide kernel forms the next state's
                                // density by column sweeps (FP32, chemical-potential force)
  // y-slab of a larger lattice: local row y is global row y + y_off (mod ny_glob when ny_glob >
  // 0); the audits sum rows [own_lo, own_hi) and the Eq. 18 sum boundary nodes [b_lo, b_hi)
  // only.  A whole lattice has y_off = ny_glob = 0, own = [0, ny), b = [0, n_bnodes).
  int y_off, ny_glob;
  int own_lo, own_hi;
  int b_lo, b_hi;
};

// global row of local row y (slabs; the identity for a whole lattice)
template <typename real>
__device__ __forceinline__ int global_row(const Lattice<real>& L, int y) {
  int g = y + L.y_off;
  if (L.ny_glob > 0) g = g < 0 ? g + L.ny_glob : (g >= L.ny_glob ? g - L.ny_glob : g);
  return g;
}

template <typename real>
__device__ __forceinline__ int wrap_x(const Lattice<real>& L, int x) {
  return x < 0 ? x + L.nx : (x >= L.nx ? x - L.nx : x);
}
template <typename real>
__device__ __forceinline__ int wrap_y(const Lattice<real>& L, int y) {
  if (L.walls) return y;
  return y < 0 ? y + L.ny : (y >= L.ny ? y - L.ny : y);
}
template <typename real>
__device__ __forceinline__ int node_at(const Lattice<real>& L, int x, int y) {
  return wrap_y(L, y) * L.pitch + wrap_x(L, x);
}

// Index (into L.f[c]) of population i of node (x, y) of the state held as lattice c: slot i of
// the node, or in AA order (aa, c = 1) slot opp(i) of node (x, y) - e_i.  x, y may lie one node
// outside the lattice (wrapped like node_at).
template <typename real>
__device__ __forceinline__ int pop_index(const Lattice<real>& L, int c, int i, int x, int y) {
  if (L.aa && c == 1) return opp(i) * L.plane + node_at(L, x - ex(i), y - ey(i));
  return i * L.plane + node_at(L, x, y);
}
// the nine populations of node (x, y) of the state held as lattice c
template <typename real>
__device__ __forceinline__ void load_pops(const Lattice<real>& L, int c, int x, int y, real (&fl)[9]) {
  const real* f = L.f[c];
#pragma unroll
  for (int i = 0; i < 9; ++i) fl[i] = f[pop_index(L, c, i, x, y)];
}

// Sums of products with a fixed rounding order.  Where an expression adds two products
// the compiler may fuse either into an FMA, and may choose differently in different kernels;
// the EOS terms, the force and mu are assembled through these, so that every kernel that
// evaluates them (density, scatter, chemical potential, collide, boundary, read-out, batched)
// gets the same bits.
// The same functions on float2 take two nodes at once in sm_103a's packed FP32 instructions
// (add / sub / mul / fma .f32x2), each half rounded like the scalar operation: half the issue
// slots, the same bits.
// One difference: ptxas fuses a packed product with a packed sum that follows, rounding spelled
// out or not, so shared code hands a product to fma_rn or another product, never to add_rn or sub_rn.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
#define LBMGB_PACKED(name, op)                                                            \
  __device__ __forceinline__ float2 name(float2 a, float2 b) {                           \
    float2 d;                                                                            \
    asm(op ".rn.f32x2 %0, %1, %2;"                                                       \
        : "=l"(reinterpret_cast<unsigned long long&>(d))                                 \
        : "l"(reinterpret_cast<const unsigned long long&>(a)),                           \
          "l"(reinterpret_cast<const unsigned long long&>(b)));                          \
    return d;                                                                            \
  }
LBMGB_PACKED(add_rn, "add")
LBMGB_PACKED(sub_rn, "sub")
LBMGB_PACKED(mul_rn, "mul")
#undef LBMGB_PACKED
__device__ __forceinline__ float2 fma_rn(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)),
        "l"(reinterpret_cast<const unsigned long long&>(c)));
  return d;
}
// the same value in every half
template <typename V> struct SplatOf;
template <> struct SplatOf<float> { static __device__ __forceinline__ float of(float a) { return a; } };
template <> struct SplatOf<double> { static __device__ __forceinline__ double of(double a) { return a; } };
template <> struct SplatOf<float2> { static __device__ __forceinline__ float2 of(float a) { return make_float2(a, a); } };
template <typename V, typename T>
__device__ __forceinline__ V splat(T a) { return SplatOf<V>::of(a); }
// the scalar type of a value of one or two nodes
template <typename V> struct ScalarOf { using type = V; };
template <> struct ScalarOf<float2> { using type = float; };

// FP32 reciprocal, square root and log1p without branches, so that the instructions around them
// interleave (the compiler's division and log1pf test for special arguments and branch).  The first
// two are the hardware approximation y (relative error e of 2^-23 and 2^-22) and one Newton step whose
// residual a fused multiply-add gives without cancellation (Markstein, IBM J. Res. Dev. 34, 1990): what
// is left of e is e^2, far below the last rounding, so the result is the correctly rounded one but
// for arguments within 1e-3 of a rounding boundary (tests/test_gpu_device_math.py: at most
// 0.501 ulp).  For normal arguments whose reciprocal is normal: zero, infinity and subnormal
// numbers give NaN, where a division gives an infinity or zero -- a density or 1 - b rho of that kind
// leaves no finite value at its node either way.
__device__ __forceinline__ float approx_rcp(float a) { float y; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a)); return y; }
__device__ __forceinline__ float2 approx_rcp(float2 a) { return make_float2(approx_rcp(a.x), approx_rcp(a.y)); }
template <typename V>
__device__ __forceinline__ V recip(V a) {
  const V y = approx_rcp(a);
  return fma_rn(y, fma_rn(mul_rn(splat<V>(-1.0f), a), y, splat<V>(1.0f)), y);
}
template <>
__device__ __forceinline__ double recip<double>(double a) { return 1.0 / a; }
// sqrt of positive values
__device__ __forceinline__ float approx_rsqrt(float a) { float y; asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(a)); return y; }
__device__ __forceinline__ float2 approx_rsqrt(float2 a) { return make_float2(approx_rsqrt(a.x), approx_rsqrt(a.y)); }
template <typename V>
__device__ __forceinline__ V root(V a) {
  const V y = approx_rsqrt(a), q = mul_rn(a, y);
  return fma_rn(fma_rn(mul_rn(splat<V>(-1.0f), q), q, a), mul_rn(splat<V>(0.5f), y), q);
}
template <>
__device__ __forceinline__ double root<double>(double a) { return sqrt(a); }
// log(1 + a b), by the classic reduction (Cody and Waite, Software Manual for the Elementary
// Functions, 1980): 2^e is the power of two that brings 1 + a b into [sqrt(1/2), sqrt(2)), f = (1 + a b)
// 2^-e - 1, log = e ln 2 + f + f^2 Q(f).  a 2^-e and 2^-e - 1 are exact, so f is a b 2^-e + (2^-e - 1)
// rounded once, where log1pf of the rounded product carries that rounding divided by 1 + a b.  Q is
// the minimax polynomial of degree 8, weighted for the relative error, on that range
// (tests/golden/make_log1p_polynomial.py; 5e-9).  Against the logarithm of the exact a b, measured: at
// most 1.52 ulp, near zero, most of it f's rounding (log1pf of the rounded product 1.48 there, 2.4 for a b
// below -0.3, 300 at -0.9999); over the densities of a liquid and a gas 0.33 ulp rms (0.56).  NaN unless
// 1 + a b > 0.
__device__ __forceinline__ int log_exponent(float u) { return (__float_as_int(u) - 0x3f3504f3) & (int)0xff800000; }
__device__ __forceinline__ float log_or_nan(float u, float v) { return u > 0.0f ? v : __int_as_float(0x7fffffff); }
struct LogParts {   // k: e 2^23, s: 2^-e
  static __device__ __forceinline__ void of(float u, float& k, float& s) {
    const int i = log_exponent(u);
    k = (float)i;
    s = __int_as_float(0x3f800000 - i);
  }
  static __device__ __forceinline__ void of(float2 u, float2& k, float2& s) {
    of(u.x, k.x, s.x);
    of(u.y, k.y, s.y);
  }
  static __device__ __forceinline__ float checked(float u, float v) { return log_or_nan(u, v); }
  static __device__ __forceinline__ float2 checked(float2 u, float2 v) {
    return make_float2(log_or_nan(u.x, v.x), log_or_nan(u.y, v.y));
  }
};
template <typename V>
__device__ __forceinline__ V log1p_product(V a, V b) {
  auto K = [](float c) { return splat<V>(c); };
  V k, s;
  const V u = fma_rn(a, b, K(1.0f));
  LogParts::of(u, k, s);
  const V f = fma_rn(mul_rn(a, s), b, sub_rn(s, K(1.0f)));
  V q = fma_rn(K(-0.0762307197f), f, K(0.1290552169f));
  q = fma_rn(q, f, K(-0.1324298531f));
  q = fma_rn(q, f, K(0.1418163329f));
  q = fma_rn(q, f, K(-0.1660905629f));
  q = fma_rn(q, f, K(0.2000198513f));
  q = fma_rn(q, f, K(-0.2500158549f));
  q = fma_rn(q, f, K(0.3333332539f));
  q = fma_rn(q, f, K(-0.4999998808f));
  const V r = fma_rn(mul_rn(f, f), q, f);
  return LogParts::checked(u, fma_rn(k, K(8.26295829e-8f), r));   // ln 2 / 2^23
}
template <>
__device__ __forceinline__ double log1p_product<double>(double a, double b) { return log1p(__dmul_rn(a, b)); }
// hi where r > split, else lo
__device__ __forceinline__ float pick(float r, float split, float lo, float hi) { return r > split ? hi : lo; }
__device__ __forceinline__ double pick(double r, double split, double lo, double hi) { return r > split ? hi : lo; }
__device__ __forceinline__ float2 pick(float2 r, float split, float lo, float hi) {
  return make_float2(r.x > split ? hi : lo, r.y > split ? hi : lo);
}

// ---------------------------------------------------------------------------------------
// Equation of state: bulk chemical potential psi'(rho) minus its coexistence value.
//   CS: psi' = RT [ln rho + (8 eta - 9 eta^2 + 3 eta^3)/(1-eta)^3] - 2 a rho,  eta = b rho/4
//   PR: Eq. 11 without the gradient term.
// ---------------------------------------------------------------------------------------

// CS: psi'(rho) - mu_sat evaluated against the nearer coexistence density rho0 (gas below
// sqrt(rho_g rho_l), liquid above), where psi'(rho0) = mu_sat:
//   RT ln(rho/rho0) + RT [G(eta) - G(eta0)] - 2a (rho - rho0) + c0,
//   G(eta) = P(eta)/(1-eta)^3,  P = 8 eta - 9 eta^2 + 3 eta^3,
// with ln(rho/rho0) = log1p((rho - rho0)/rho0) and the exact factorisation
//   G(eta) - G(eta0) = h N(h) / (1-eta)^3,  h = eta - eta0,  a = 1 - eta0,
//   N = 8 - 9(eta+eta0) + 3(eta^2 + eta eta0 + eta0^2) + (P(eta0)/a^3) (a^2 + a (1-eta) + (1-eta)^2),
// a quadratic m0 + m1 h + m2 h^2 in h whose coefficients belong to rho0, so that every term
// vanishes with rho - rho0 (which is exact near rho0) instead of cancelling between terms of size
// RT ln rho.  c0 = psi'(rho0) - mu_sat of the storage-rounded rho0 and the m's are computed in
// FP64 on the host, so both branches meet the same function.  One reciprocal.
template <typename V, typename real>
__device__ __forceinline__ V psi_prime_cs(const Lattice<real>& L, V r) {
  auto K = [](real c) { return splat<V>(c); };
  auto C = [&](const real (&c)[2]) { return pick(r, L.rho_split, c[0], c[1]); };
  const V dr = sub_rn(r, C(L.cs_r0));
  const V h = mul_rn(K(L.b4), dr);
  const V ib = recip(fma_rn(K(-L.b4), r, K(1)));
  const V ib3 = mul_rn(mul_rn(ib, ib), ib);
  const V N = fma_rn(fma_rn(C(L.cs_m2), h, C(L.cs_m1)), h, C(L.cs_m0));
  const V lg = log1p_product(dr, C(L.cs_inv_r0));
  return fma_rn(K(L.RT), lg, fma_rn(mul_rn(K(L.RT), h), mul_rn(N, ib3), fma_rn(K(real(-2) * L.a), dr, C(L.cs_c0))));
}
// Peng-Robinson, Eq. 11 without the gradient term,
//   RT ln(rho/(1-x)) - K ln((c1+x)/(c2-x)) + RT/(1-x) - a alpha rho/D - mu_sat,
//   x = b rho, c1,2 = sqrt 2 -+ 1, D = 1 + 2x - x^2 = (c1+x)(c2-x), K = a alpha/(2 sqrt 2 b),
// against the nearer coexistence density likewise: the differences from rho0 are, exactly,
//   ln: log1p(dr / (rho0 (1-x))) and log1p(2 sqrt 2 b dr / ((c1+x0)(c2-x))),
//   RT b dr / ((1-x0)(1-x)),  a alpha dr (1 + x x0) / (D0 D).
template <typename V, typename real>
__device__ __forceinline__ V psi_prime_pr(const Lattice<real>& L, V r) {
  auto K = [](real c) { return splat<V>(c); };
  auto C = [&](const real (&c)[2]) { return pick(r, L.rho_split, c[0], c[1]); };
  const V dr = sub_rn(r, C(L.cs_r0)), x = mul_rn(K(L.b), r);
  const V iom = recip(fma_rn(K(-L.b), r, K(1))), ic2 = recip(fma_rn(K(-L.b), r, K(real(2.414213562373095))));
  const V iD = mul_rn(ic2, recip(fma_rn(K(L.b), r, K(real(0.41421356237309503)))));
  const V l1 = log1p_product(dr, mul_rn(C(L.cs_inv_r0), iom)), l2 = log1p_product(dr, mul_rn(C(L.pr_kb), ic2));
  const V t = mul_rn(mul_rn(C(L.pr_naD), fma_rn(x, C(L.pr_x0), K(1))), iD);
  const V S = fma_rn(C(L.pr_rtb), iom, t);
  return fma_rn(K(L.RT), l1, fma_rn(K(L.pr_nk), l2, fma_rn(dr, S, C(L.cs_c0))));
}
template <typename V, typename real>
__device__ __forceinline__ V psi_prime_shifted(const Lattice<real>& L, V r) {
  return L.eos == EOS_CS ? psi_prime_cs(L, r) : psi_prime_pr(L, r);
}

// Fourth-order central first derivatives and Laplacian along the lattice axes.
struct Stencil {
  int xm2, xm1, xp1, xp2, ym2, ym1, yp1, yp2;
};
template <typename real>
__device__ __forceinline__ bool interior(const Lattice<real>& L, int x, int y) {
  // no periodic wrap within two nodes (with walls the rows never wrap: fluid nodes keep two
  // solid rows below and above them)
  return x >= 2 && x < L.nx - 2 && (L.walls || (y >= 2 && y < L.ny - 2));
}

template <typename real>
__device__ __forceinline__ Stencil stencil_at(const Lattice<real>& L, int x, int y) {
  Stencil s;
  if (interior(L, x, y)) {
    const int n = y * L.pitch + x, p = L.pitch;
    s.xm2 = n - 2; s.xm1 = n - 1; s.xp1 = n + 1; s.xp2 = n + 2;
    s.ym2 = n - 2 * p; s.ym1 = n - p; s.yp1 = n + p; s.yp2 = n + 2 * p;
    return s;
  }
  const int row = y * L.pitch;
  s.xm2 = row + wrap_x(L, x - 2);
  s.xm1 = row + wrap_x(L, x - 1);
  s.xp1 = row + wrap_x(L, x + 1);
  s.xp2 = row + wrap_x(L, x + 2);
  s.ym2 = wrap_y(L, y - 2) * L.pitch + x;
  s.ym1 = wrap_y(L, y - 1) * L.pitch + x;
  s.yp1 = wrap_y(L, y + 1) * L.pitch + x;
  s.yp2 = wrap_y(L, y + 2) * L.pitch + x;
  return s;
}

// Undivided fourth-order differences D(p) = 8 (p_1 - p_-1) - (p_2 - p_-2) = 12 dp/dx along
// each axis (8 x exact, so fused or not it rounds the same).
template <typename V>
__device__ __forceinline__ V diff4_of(V p1, V pm1, V p2, V pm2) {
  return fma_rn(splat<V>(typename ScalarOf<V>::type(8)), sub_rn(p1, pm1), sub_rn(pm2, p2));
}
template <typename real>
__device__ __forceinline__ void diff4(const real* __restrict__ p, const Stencil& s, real& dx, real& dy) {
  dx = diff4_of(__ldg(p + s.xp1), __ldg(p + s.xm1), __ldg(p + s.xp2), __ldg(p + s.xm2));
  dy = diff4_of(__ldg(p + s.yp1), __ldg(p + s.ym1), __ldg(p + s.yp2), __ldg(p + s.ym2));
}

template <typename real>
__device__ __forceinline__ void grad4(const real* __restrict__ p, const Stencil& s, real& gx, real& gy) {
  const real c = real(1.0 / 12.0);
  gx = (real(8) * (__ldg(p + s.xp1) - __ldg(p + s.xm1)) - (__ldg(p + s.xp2) - __ldg(p + s.xm2))) * c;
  gy = (real(8) * (__ldg(p + s.yp1) - __ldg(p + s.ym1)) - (__ldg(p + s.yp2) - __ldg(p + s.ym2))) * c;
}

// Written as differences from the centre value, (-p2 + 16 p1 - 30 c + 16 p-1 - p-2)/12 =
// (16 [(p1 - c) + (p-1 - c)] - [(p2 - c) + (p-2 - c)])/12: inside a bulk phase the
// differences are exact (Sterbenz), so FP32 keeps the Laplacian's relative accuracy there
// instead of losing it to cancellation between terms of size 30 rho.
// the Laplacian from the second differences over one node and the negated ones over two, x and y
template <typename V>
__device__ __forceinline__ V lap4_diff(V x1, V nx2, V y1, V ny2) {
  using real = typename ScalarOf<V>::type;
  const V c16 = splat<V>(real(16));
  return mul_rn(add_rn(fma_rn(c16, x1, nx2), fma_rn(c16, y1, ny2)), splat<V>(real(1.0 / 12.0)));
}
template <typename V>
__device__ __forceinline__ V lap4_of(V c, V xp1, V xm1, V xp2, V xm2, V yp1, V ym1, V yp2, V ym2) {
  return lap4_diff(add_rn(sub_rn(xp1, c), sub_rn(xm1, c)), add_rn(sub_rn(c, xp2), sub_rn(c, xm2)),
                   add_rn(sub_rn(yp1, c), sub_rn(ym1, c)), add_rn(sub_rn(c, yp2), sub_rn(c, ym2)));
}
template <typename real>
__device__ __forceinline__ real lap4(const real* __restrict__ p, int n, const Stencil& s) {
  return lap4_of(p[n], p[s.xp1], p[s.xm1], p[s.xp2], p[s.xm2], p[s.yp1], p[s.ym1], p[s.yp2], p[s.ym2]);
}


// Eq. 12 in mesh units, shifted: mu~ = k^2 (psi'(rho) - mu_sat) - kappa^ lap(rho)
template <typename V, typename real>
__device__ __forceinline__ V mu_of(const Lattice<real>& L, V psip, V lap) {
  return fma_rn(splat<V>(L.k2), psip, mul_rn(splat<V>(-L.kappa), lap));
}
// delta rho / 36 to within an ulp: the product with the rounded reciprocal, corrected once
// with its FMA residual
template <typename V>
__device__ __forceinline__ V div36(V d) {
  const V c = splat<V>(1.0f / 36.0f);
  const V q = mul_rn(d, c);
  return fma_rn(fma_rn(splat<V>(-36.0f), q, d), c, q);
}
// (FP64: the same; with the correctly rounded reciprocal that is the rounded quotient, after Markstein
// (1990), in three FP64 instructions where the division takes about ten)
template <>
__device__ __forceinline__ double div36<double>(double d) {
  const double c = 1.0 / 36.0, q = d * c;
  return fma_rn(fma_rn(-36.0, q, d), c, q);
}

// F = rho g - rho grad(mu) + c_s^2 grad(rho) (Eq. 9), one component, from the undivided
// differences D(mu) and D(rho) of diff4 (grad = D/12, c_s^2 = 1/3):
//   F = [D(rho) - 3 rho D(mu)] / 36 + rho g.
// Inside an interface the two terms are large and nearly cancel.  The product rho D(mu) enters
// the difference exactly (with its FMA residual), and the division by 36 is corrected to
// within an ulp: no rounded constant (1/12, 1/3) scales either term, because such a constant
// biases the force the same way at every node and step, and that bias builds up in the flow
// where unbiased rounding errors do not.
template <typename V, typename real>
__device__ __forceinline__ V force_cp(V r, real g, V dmu, V drho) {
  const V pn = mul_rn(mul_rn(splat<V>(real(-1)), r), dmu);   // -r D(mu)
  const V e = fma_rn(r, dmu, pn);
  const V G = fma_rn(splat<V>(real(-3)), e, fma_rn(splat<V>(real(3)), pn, drho));
  return fma_rn(r, splat<V>(g), div36(G));
}
// F = rho g + c a, the pseudopotential force of centre value c and sum a, one component
template <typename V, typename real>
__device__ __forceinline__ V force_pp(V r, real g, V c, V a) {
  return fma_rn(c, a, mul_rn(r, splat<V>(g)));
}

// Pseudopotential of the pseudopotential force model, psi = [2 (rho c_s^2 - k^2 p0(rho))]^(1/2)
// clamped at zero (rho c_s^2 + (G/2) psi^2 = k^2 p0 with G = -1), p0 the CS or PR pressure.
// As 2 rho w with w = 1/3 - k^2 p0 / rho.
template <typename V, typename real>
__device__ __forceinline__ V psi_cs(const Lattice<real>& L, V r) {
  auto K = [](real c) { return splat<V>(c); };
  const V om = fma_rn(K(-L.b4), r, K(1)), eta = mul_rn(K(L.b4), r);
  const V ib = recip(om);
  const V poly = fma_rn(eta, fma_rn(eta, om, K(1)), K(1));   // 1 + eta + eta^2 - eta^3
  const V t = fma_rn(mul_rn(K(L.RT), poly), mul_rn(mul_rn(ib, ib), ib), mul_rn(K(-L.a), r));
  const V w = fma_rn(K(-L.k2), t, K(real(1.0 / 3.0)));
  return mul_rn(mul_rn(K(2), r), w);
}
__device__ __forceinline__ float positive_root(float a, float q) { return a > 0.0f ? q : 0.0f; }
__device__ __forceinline__ double positive_root(double a, double q) { return a > 0.0 ? q : 0.0; }
__device__ __forceinline__ float2 positive_root(float2 a, float2 q) {
  return make_float2(positive_root(a.x, q.x), positive_root(a.y, q.y));
}
template <typename real>
__device__ __forceinline__ real psi_pr(const Lattice<real>& L, real r) {
  const real br = mul_rn(L.b, r);
  const real p0 = mul_rn(r, L.RT) / (real(1) - br) - mul_rn(mul_rn(L.aalpha, r), r) / fma_rn(br, real(2) - br, real(1));
  return mul_rn(real(2), fma_rn(r, real(1.0 / 3.0), -mul_rn(L.k2, p0)));
}
template <typename real>
__device__ __forceinline__ real psi_of(const Lattice<real>& L, real r) {
  const real arg = L.eos == EOS_CS ? psi_cs(L, r) : psi_pr(L, r);
  return positive_root(arg, root(arg));
}
__device__ __forceinline__ float2 psi_of(const Lattice<float>& L, float2 r) {
  const float2 arg = L.eos == EOS_CS ? psi_cs(L, r) : make_float2(psi_pr(L, r.x), psi_pr(L, r.y));
  return positive_root(arg, root(arg));
}

// Adds the pseudopotential force -G psi(x) sum_i w_i psi(x + e_i) e_i (G = -1, w = 1/3 on the
// axes, 1/12 on the diagonals) from the centre value c and the eight neighbours, as
// differences of opposite neighbours (exact inside a bulk phase).
template <typename V>
__device__ __forceinline__ void pp_sums(V e, V n, V w, V s, V ne, V nw, V sw, V se, V& ax, V& ay) {
  using real = typename ScalarOf<V>::type;
  const V d1 = sub_rn(ne, sw), d2 = sub_rn(se, nw);
  const V third = splat<V>(real(1.0 / 3.0)), twelfth = splat<V>(real(1.0 / 12.0));
  ax = fma_rn(sub_rn(e, w), third, mul_rn(add_rn(d1, d2), twelfth));
  ay = fma_rn(sub_rn(n, s), third, mul_rn(sub_rn(d1, d2), twelfth));
}

// Nonideal force of Eq. 9 in mesh units, F = -rho grad(mu^) + c_s^2 grad(rho), plus rho g;
// with PSEUDO the pseudopotential force from the psi plane instead.
template <typename real, bool PSEUDO = false>
__device__ __forceinline__ void force_at(const Lattice<real>& L, int x, int y, real r, real& Fx, real& Fy) {
  Fx = r * L.gx;
  Fy = r * L.gy;
  if (L.eos == EOS_NONE) return;
  if (PSEUDO) {
    const real* __restrict__ p = L.mu;
    auto at = [&](int dx, int dy) { return __ldg(p + node_at(L, x + dx, y + dy)); };
    real ax, ay;
    pp_sums(at(1, 0), at(0, 1), at(-1, 0), at(0, -1), at(1, 1), at(-1, 1), at(-1, -1), at(1, -1), ax, ay);
    const real c = at(0, 0);
    Fx = force_pp(r, L.gx, c, ax);
    Fy = force_pp(r, L.gy, c, ay);
    return;
  }
  {
    Stencil s = stencil_at(L, x, y);
    real dmx, dmy, drx, dry;
    diff4(L.mu, s, dmx, dmy);
    diff4(L.rho, s, drx, dry);
    Fx = force_cp(r, L.gx, dmx, drx);
    Fy = force_cp(r, L.gy, dmy, dry);
  }
}

// Exact-difference forcing term of Eq. 13 for direction i,
//   F_i = f_i^eq(rho, u + du) - f_i^eq(rho, u),  du = F / rho,
// written as a difference so that FP32 keeps its relative accuracy:
//   w_i rho [3 e.du + 4.5 (e.du)(e.(2u+du)) - 1.5 du.(2u+du)].
template <typename real>
__device__ __forceinline__ real edm_term(int i, real r, real ux, real uy, real dux, real duy) {
  // (products rounded explicitly, the arguments' by the caller: every kernel that evaluates a link gets
  // the same bits; products by 2 and by the directions' components are exact)
  const real ax = real(2) * ux + dux, ay = real(2) * uy + duy;
  const real edu = real(ex(i)) * dux + real(ey(i)) * duy;
  const real e2u = real(ex(i)) * ax + real(ey(i)) * ay;
  const real du2u = fma_rn(dux, ax, mul_rn(duy, ay));
  const real t = fma_rn(real(3), edu, fma_rn(mul_rn(real(4.5), edu), e2u, mul_rn(real(-1.5), du2u)));
  return mul_rn(mul_rn(real(wgt(i)), r), t);
}

// Moments of a node's offset populations: delta rho = sum_i (f_i - w_i rho_ref) and
// j = sum_i f_i e_i.  j is summed as differences of opposite populations, which are exact in
// floating point near equilibrium (Sterbenz), so the momentum keeps its relative accuracy
// although it is a small difference of populations of size ~rho/9.
template <typename V>
__device__ __forceinline__ V density_sum(const V (&f)[9]) {
  return add_rn(f[0], add_rn(add_rn(add_rn(f[1], f[3]), add_rn(f[2], f[4])), add_rn(add_rn(f[5], f[7]), add_rn(f[6], f[8]))));
}

template <typename V>
__device__ __forceinline__ void moments(const V (&f)[9], V& drho, V& jx, V& jy) {
  drho = density_sum(f);
  const V d57 = sub_rn(f[5], f[7]), d86 = sub_rn(f[8], f[6]);
  jx = add_rn(sub_rn(f[1], f[3]), add_rn(d57, d86));
  jy = add_rn(sub_rn(f[2], f[4]), sub_rn(d57, d86));
}

// Density as the read-out pass and the sweep store it (the same sum, in the same order).
template <typename V, typename real>
__device__ __forceinline__ V density_of(const Lattice<real>& L, const V (&f)[9]) {
  return add_rn(splat<V>(L.rho_ref), density_sum(f));
}

// Collision (Eq. 4) of offset populations with the exact-difference term (Eq. 13).
//   MRT: f~ = f - M^-1 S (m - m_eq) + F_i,  M of Eq. 2, S of Eq. 3, m_eq listed under Eq. 1
//        (q_y^eq = -j_y), all offset by the moments of w_i rho_ref (= m_eq(rho_ref, 0));
//   BGK: f~ = f - (f - f^eq)/tau + F_i.
// The exact-difference term is f^eq(rho, u') - f^eq(rho, u) with u' = u + F/rho, so the
// post-collision populations are f^eq(rho, u') plus the relaxed non-equilibrium part:
//   f~_i = f^eq_i(rho, u') + [M^-1 (I - S) (m - m_eq)]_i,
// M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4); the conserved moments
// drop out.  FP32: the large part of f^eq, w_i delta rho, is formed as {16, 4, 1} x
// (delta rho / 36) -- exact multiples of one quotient, so the weights sum to one exactly and
// no mass bias arises -- and the small terms are added before the final rounding.  The odd
// part of f^eq, w_i rho 3 e_i.u, is formed from the momentum J = rho u itself (odd_split), not
// from rho/9 and rho/36 times u = J/rho: the rounded constants and 1/rho would scale the
// momentum the collision passes on by a fixed factor every step, and at a steady state such a
// bias builds up where unbiased rounding does not.
template <typename V>
__device__ __forceinline__ void odd_split(V Jx, V Jy, V& px, V& py, V& pd, V& pa) {
  // w_i rho 3 e_i.u for e = (1,1) and (-1,1) is (Jx + Jy)/12 and (Jy - Jx)/12; the axis terms
  // take what is left of J/2, so that the first moment of the odd parts is J up to rounding of
  // the sums, whatever the rounding of 1/12
  using real = typename ScalarOf<V>::type;
  const V c12 = splat<V>(real(1.0 / 12.0)), n12 = splat<V>(real(-1.0 / 12.0)), half = splat<V>(real(0.5));
  const V s = add_rn(Jx, Jy), d = sub_rn(Jy, Jx);
  const V npd = mul_rn(s, n12);
  pd = mul_rn(s, c12);
  pa = mul_rn(d, c12);
  px = fma_rn(half, Jx, fma_rn(d, c12, npd));
  py = fma_rn(half, Jy, fma_rn(d, n12, npd));
}

// collide_node's BGK branch in FP64, whose instructions are what it costs (two lanes an SM and clock):
// f~ = (1 - 1/tau) f + [f^eq(rho, u') - (1 - 1/tau) f^eq(rho, u)], the difference formed in delta rho, j and the three
// second-order products before it is spread over the directions: 45 operations instead of 93 (a node's
// collision with its force: 160 -> 105; 512 x 512: 129 -> 101 us a step).  1/tau enters as
// 1 - (1 - 1/tau) only, so mass and momentum balance whatever the rounding of either.
__device__ __forceinline__ void collide_bgk64(const Lattice<double>& L, double (&f)[9], double r, double drho, double jx,
                                              double jy, double Fx, double Fy) {
  const double keep = 1.0 - L.omega, inv_r = 1.0 / r, nk = -keep;
  const double Jx = add_rn(jx, Fx), Jy = add_rn(jy, Fy);
  const double q = div36(drho), qw = fma(nk, q, q);
  const double vx = Jx * inv_r, vy = Jy * inv_r, ux = (nk * jx) * inv_r, uy = (nk * jy) * inv_r;
  const double X = fma(Jx, vx, jx * ux), Y = fma(Jy, vy, jy * uy), Z = fma(Jx, vy, jx * uy), S = X + Y;
  double px, py, pd, pa;
  odd_split(fma(nk, jx, Jx), fma(nk, jy, Jy), px, py, pd, pa);
  const double q4 = 4.0 * qw;
  const double ex0 = fma(1.0 / 3.0, X, fma(-1.0 / 6.0, Y, q4)), ey0 = fma(1.0 / 3.0, Y, fma(-1.0 / 6.0, X, q4));
  const double ed = fma(1.0 / 12.0, S, qw), e5 = fma(0.25, Z, ed), e6 = fma(-0.25, Z, ed);
  f[0] = fma(keep, f[0], fma(-2.0 / 3.0, S, 16.0 * qw));
  f[1] = fma(keep, f[1], ex0 + px);
  f[3] = fma(keep, f[3], ex0 - px);
  f[2] = fma(keep, f[2], ey0 + py);
  f[4] = fma(keep, f[4], ey0 - py);
  f[5] = fma(keep, f[5], e5 + pd);
  f[7] = fma(keep, f[7], e5 - pd);
  f[6] = fma(keep, f[6], e6 + pa);
  f[8] = fma(keep, f[8], e6 - pa);
}

// The second-order part w_i rho (4.5 (e_i.v)^2 - 1.5 v^2) of f^eq from X = Jx vx, Y = Jy vy,
// Z = Jx vy (J = rho v): X/3 - Y/6 and Y/3 - X/6 on the axes, (X + Y)/12 +- Z/4 on the two
// diagonals, -2 (X + Y)/3 at rest; the rounded constants are exact multiples of one another, so
// the parts sum to zero.
//
// Every operation is rounded explicitly (add_rn ... fma_rn), so that no kernel's compiler fuses
// them differently, and no product enters a plain sum (ptxas fuses mul.rn.f32x2 with a following
// add.rn.f32x2): all kernels that collide a node, or two at once, get the same bits.
// Opposite directions share their even and odd parts, f~_i = w_i delta rho + (even +- odd).
template <typename V, typename real>
__device__ __forceinline__ void collide_node(const Lattice<real>& L, V (&f)[9], V r, V drho, V jx, V jy, V Fx, V Fy) {
  if constexpr (sizeof(real) == 8) {
    if (L.coll != COLL_MRT) {
      collide_bgk64(L, f, r, drho, jx, jy, Fx, Fy);
      return;
    }
  }
  auto K = [](real c) { return splat<V>(c); };
  const real third = real(1.0 / 3.0), sixth = real(1.0 / 6.0), twelfth = real(1.0 / 12.0), twothirds = real(2.0 / 3.0);
  const V inv_r = recip(r);
  const V q36 = div36(drho);
  const V ux = mul_rn(jx, inv_r), uy = mul_rn(jy, inv_r);
  const V Jx = add_rn(jx, Fx), Jy = add_rn(jy, Fy);
  const V vx = mul_rn(Jx, inv_r), vy = mul_rn(Jy, inv_r);
  const V X = mul_rn(Jx, vx), Y = mul_rn(Jy, vy), Z = mul_rn(Jx, vy);
  const V S = fma_rn(Jx, vx, Y);
  V px, py, pd, pa;
  odd_split(Jx, Jy, px, py, pd, pa);
  // even parts of the rest, x, y, diagonal (5, 7) and antidiagonal (6, 8) directions, odd parts
  V n0, nx, ny, nd, na, ox, oy, od, oa;
  if (L.coll == COLL_MRT) {
    const V s13 = add_rn(f[1], f[3]), s24 = add_rn(f[2], f[4]), s57 = add_rn(f[5], f[7]), s68 = add_rn(f[6], f[8]);
    const V sa = add_rn(s13, s24), sd = add_rn(s57, s68);
    const V njx = mul_rn(K(-1), jx);
    const V j2 = fma_rn(jx, ux, mul_rn(jy, uy));   // j.j / rho
    // non-equilibrium moments; the factors (1 - s_k) over the norms of M's rows follow
    const V me = fma_rn(K(-3), j2, fma_rn(K(2), drho, sub_rn(add_rn(sd, sd), fma_rn(K(4), f[0], sa))));
    const V mp = fma_rn(K(3), j2, sub_rn(fma_rn(K(4), f[0], fma_rn(K(-2), sa, sd)), drho));
    const V qx = add_rn(fma_rn(K(-3), sub_rn(f[1], f[3]), jx), jx);
    const V qy = add_rn(fma_rn(K(-3), sub_rn(f[2], f[4]), jy), jy);
    const V pxx = fma_rn(jy, uy, fma_rn(njx, ux, sub_rn(s13, s24)));
    const V pxy = fma_rn(njx, uy, sub_rn(s57, s68));
    const V a14 = fma_rn(K(L.nke36), me, mul_rn(K(real(-2) * L.kp36), mp));
    const V a58 = fma_rn(K(real(-2) * L.nke36), me, mul_rn(K(L.kp36), mp));
    n0 = fma_rn(K(real(4) * L.nke36), me, mul_rn(K(real(4) * L.kp36), mp));
    nx = fma_rn(K(L.kn4), pxx, a14);
    ny = fma_rn(K(-L.kn4), pxx, a14);
    nd = fma_rn(K(L.kn4), pxy, a58);
    na = fma_rn(K(-L.kn4), pxy, a58);
    ox = fma_rn(K(real(-2) * L.kq12), qx, px);
    oy = fma_rn(K(real(-2) * L.kq12), qy, py);
    od = fma_rn(K(L.kq12), add_rn(qx, qy), pd);
    oa = fma_rn(K(L.kq12), sub_rn(qy, qx), pa);
  } else {
    // (1 - 1/tau) (f - f^eq(rho, u)), as half sums and half differences of opposite directions
    const real keep = real(1) - L.omega;
    const real kh = real(0.5) * keep;
    const V x0 = mul_rn(jx, ux), y0 = mul_rn(jy, uy), z0 = mul_rn(jx, uy), s0 = fma_rn(jx, ux, y0);
    V bx, by, bd, ba;
    odd_split(jx, jy, bx, by, bd, ba);
    auto even = [&](V a, V b, V q, V ne) {   // keep ((f_a + f_b)/2 + q + ne), -q the share of delta rho
      return mul_rn(K(keep), fma_rn(K(0.5), add_rn(add_rn(a, q), add_rn(b, q)), ne));
    };
    const V m4q = mul_rn(K(-4), q36), m1q = mul_rn(K(-1), q36);
    n0 = mul_rn(K(keep), fma_rn(K(twothirds), s0, fma_rn(K(-16), q36, f[0])));
    nx = even(f[1], f[3], m4q, fma_rn(K(-third), x0, mul_rn(K(sixth), y0)));
    ny = even(f[2], f[4], m4q, fma_rn(K(-third), y0, mul_rn(K(sixth), x0)));
    nd = even(f[5], f[7], m1q, fma_rn(K(-0.25), z0, mul_rn(K(-twelfth), s0)));
    na = even(f[6], f[8], m1q, fma_rn(K(0.25), z0, mul_rn(K(-twelfth), s0)));
    ox = fma_rn(K(kh), sub_rn(f[1], f[3]), fma_rn(K(-keep), bx, px));
    oy = fma_rn(K(kh), sub_rn(f[2], f[4]), fma_rn(K(-keep), by, py));
    od = fma_rn(K(kh), sub_rn(f[5], f[7]), fma_rn(K(-keep), bd, pd));
    oa = fma_rn(K(kh), sub_rn(f[6], f[8]), fma_rn(K(-keep), ba, pa));
  }
  nx = fma_rn(K(third), X, fma_rn(K(-sixth), Y, nx));
  ny = fma_rn(K(third), Y, fma_rn(K(-sixth), X, ny));
  nd = fma_rn(K(0.25), Z, fma_rn(K(twelfth), S, nd));
  na = fma_rn(K(-0.25), Z, fma_rn(K(twelfth), S, na));
  f[0] = fma_rn(K(16), q36, fma_rn(K(-twothirds), S, n0));
  f[1] = fma_rn(K(4), q36, add_rn(nx, ox));
  f[3] = fma_rn(K(4), q36, sub_rn(nx, ox));
  f[2] = fma_rn(K(4), q36, add_rn(ny, oy));
  f[4] = fma_rn(K(4), q36, sub_rn(ny, oy));
  f[5] = add_rn(q36, add_rn(nd, od));
  f[7] = add_rn(q36, sub_rn(nd, od));
  f[6] = add_rn(q36, add_rn(na, oa));
  f[8] = add_rn(q36, sub_rn(na, oa));
}

// Eqs. 16-17 (present scheme) and their variants for one link.
//   a  = f~_i(x1, t)      (parked in the solid node's slot by the push)
//   b2 = f~_i(x2, t)      (streamed into x1)
//   c  = f~_ibar(x1, t)   (streamed into x2)
//   Fi = F_i(x1, t)       (exact-difference term of direction i at x1)
template <typename real>
__device__ __forceinline__ real link_rule(int bc, real q, int x2_fluid, real a, real b2, real c, real Fi) {
  if (bc == BC_HBB) return a;
  // v = A a + W (b2 or c) [+ W Fi]
  const bool low = q < real(0.5);
  if (low && !x2_fluid) return a;
  const real q2 = mul_rn(real(2), q);
  const real inv = recip(low ? real(1) : q2);
  const real A = low ? q2 : inv;
  const real W = low ? real(1) - q2 : mul_rn(q2 - real(1), inv);
  const real v = fma_rn(A, a, mul_rn(W, low ? b2 : c));
  return bc == BC_PRESENT ? fma_rn(W, Fi, v) : v;
}

// Deterministic block sum of one double per thread (fixed shuffle tree, then warps in order).
__device__ __forceinline__ double block_sum(double v, double* smem /* >= 32 */) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) smem[warp] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  double t = 0.0;
  if (warp == 0) {
    t = lane < nw ? smem[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  __syncthreads();
  return t;   // valid in thread 0
}

// Last-block-done finish of a two-level deterministic reduction: every block stores its
// partial; the block that arrives last sums all partials in index order.  Returns true in
// thread 0 of that block, with the total in *total.
__device__ __forceinline__ bool finish_reduction(double block_total, double* partials, unsigned int* counter,
                                                 double* total, double* smem) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = block_total;
    __threadfence();
    unsigned int prev = atomicAdd(counter, 1u);
    last = prev == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double v = 0.0;
  for (unsigned int k = threadIdx.x; k < gridDim.x; k += blockDim.x) v += ((volatile double*)partials)[k];
  double s = block_sum(v, smem);
  if (threadIdx.x == 0) {
    *total = s;
    *counter = 0u;
  }
  return threadIdx.x == 0;
}

}  // namespace lbmgb
