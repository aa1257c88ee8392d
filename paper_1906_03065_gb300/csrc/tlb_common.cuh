// Shared device definitions of the GB300 ternary LB + IBM library.
//
// Internal geometry: every lattice is stored as nx * ny * nz cells with
// linear index (z*ny + y)*nx + x.  A 2D lattice of the paper (D2Q9, Sec. 3.1)
// is embedded as nx * 1 * ny: its y axis becomes the internal z axis, so the
// same plane-sweep kernels serve both; markers of a 2D ring are stored as
// (x, 0, y).  Walls, when present, bound the internal z axis.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "../../include/tlb.h"

#define TLB_HD __host__ __device__ __forceinline__

// ------------------------------------------------------------ velocity sets
// D2Q9 in the order printed in Sec. 3.1, embedded in the internal (x, z) plane.
struct D2Q9 {
  static constexpr int Q = 9;
  static constexpr int DIM = 2;
  TLB_HD static constexpr int cx(int i) {
    return i == 1 || i == 5 || i == 8 ? 1 : (i == 2 || i == 6 || i == 7 ? -1 : 0);
  }
  TLB_HD static constexpr int cy(int) { return 0; }
  TLB_HD static constexpr int cz(int i) {
    return i == 3 || i == 5 || i == 7 ? 1 : (i == 4 || i == 6 || i == 8 ? -1 : 0);
  }
  TLB_HD static constexpr double w(int i) {
    return i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
  TLB_HD static constexpr int opp(int i) {
    return i == 0 ? 0 : (i == 1 ? 2 : i == 2 ? 1 : i == 3 ? 4 : i == 4 ? 3 : i == 5 ? 6 : i == 6 ? 5 : i == 7 ? 8 : 7);
  }
  static constexpr int NCOL = 3;  // in-plane velocities (c_x, c_y), see col_dir
};

// D3Q19: rest; +x,-x,+y,-y,+z,-z (w = 1/18); then the edge velocities of the
// xy, xz and yz planes with sign pairs (+,+),(+,-),(-,+),(-,-) (w = 1/36).
struct D3Q19 {
  static constexpr int Q = 19;
  static constexpr int DIM = 3;
  TLB_HD static constexpr int comp(int i, int a) {
    // axis velocities
    return i == 0 ? 0
         : i <= 6 ? ((i - 1) / 2 == a ? ((i - 1) % 2 == 0 ? 1 : -1) : 0)
                  : edge(i - 7, a);
  }
  TLB_HD static constexpr int edge(int e, int a) {
    // e = 4*plane + signs; planes (0,1), (0,2), (1,2)
    return (a == pa(e / 4) ? ((e % 4) < 2 ? 1 : -1) : 0) + (a == pb(e / 4) ? ((e % 4) % 2 == 0 ? 1 : -1) : 0);
  }
  TLB_HD static constexpr int pa(int p) { return p == 2 ? 1 : 0; }
  TLB_HD static constexpr int pb(int p) { return p == 0 ? 1 : 2; }
  TLB_HD static constexpr int cx(int i) { return comp(i, 0); }
  TLB_HD static constexpr int cy(int i) { return comp(i, 1); }
  TLB_HD static constexpr int cz(int i) { return comp(i, 2); }
  TLB_HD static constexpr double w(int i) { return i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0); }
  TLB_HD static constexpr int opp(int i) {
    return i == 0 ? 0 : (i <= 6 ? (i % 2 == 1 ? i + 1 : i - 1) : 7 + 4 * ((i - 7) / 4) + (3 - (i - 7) % 4));
  }
  static constexpr int NCOL = 9;
};

// In-plane velocity k of a lattice: rest, +x, -x, then (3D) +y, -y and the
// four diagonals.
TLB_HD constexpr int col_cx(int k) { return k == 1 || k == 5 || k == 6 ? 1 : (k == 2 || k == 7 || k == 8 ? -1 : 0); }
TLB_HD constexpr int col_cy(int k) { return k == 3 || k == 5 || k == 7 ? 1 : (k == 4 || k == 6 || k == 8 ? -1 : 0); }
// Direction with in-plane velocity k and c_z = cz, -1 if the set has none.
template <class L>
TLB_HD constexpr int col_dir(int k, int cz) {
  for (int i = 0; i < L::Q; ++i)
    if (L::cx(i) == col_cx(k) && L::cy(i) == col_cy(k) && L::cz(i) == cz) return i;
  return -1;
}

// c_i . u of an unrolled direction: its one or two signed terms (a product
// with the zero components would not be folded away).
template <class L, class R>
__device__ __forceinline__ R cdot(int i, const R* u) {
  const int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
  const R x = cx > 0 ? u[0] : -u[0], y = cy > 0 ? u[1] : -u[1], z = cz > 0 ? u[2] : -u[2];
  if (cx && cy) return x + y;
  if (cx && cz) return x + z;
  if (cy && cz) return y + z;
  return cx ? x : (cy ? y : (cz ? z : R(0)));
}

// ------------------------------------------------------------ precisions
template <int MODE> struct Prec;
template <> struct Prec<TLB_F64> { using Real = double; using Store = double; using Rest = double; };
template <> struct Prec<TLB_F32> { using Real = float; using Store = float; using Rest = float; };
template <> struct Prec<TLB_F16> { using Real = float; using Store = __half; using Rest = float; };
template <> struct Prec<TLB_BF16> { using Real = float; using Store = __nv_bfloat16; using Rest = float; };

TLB_HD double to_real(double v) { return v; }
TLB_HD float to_real(float v) { return v; }
__device__ __forceinline__ float to_real(__half v) { return __half2float(v); }
__device__ __forceinline__ float to_real(__nv_bfloat16 v) { return __bfloat162float(v); }

template <class S> __device__ __forceinline__ S from_real(double v);
template <class S> __device__ __forceinline__ S from_real(float v);
template <> __device__ __forceinline__ double from_real<double>(double v) { return v; }
template <> __device__ __forceinline__ float from_real<float>(float v) { return v; }
template <> __device__ __forceinline__ __half from_real<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 from_real<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// A value as its storage type holds it: one rounding with 16-bit storage,
// the value itself otherwise.
template <class S, class R>
__device__ __forceinline__ R as_stored(R v) {
  return to_real(from_real<S>(v));
}

// The same of two values: with 16-bit storage one conversion for both.
template <class S, class R>
__device__ __forceinline__ void as_stored2(R& a, R& b) {
  if constexpr (std::is_same<S, __half>::value) {
    const float2 v = __half22float2(__floats2half2_rn(a, b));
    a = v.x;
    b = v.y;
  } else if constexpr (std::is_same<S, __nv_bfloat16>::value) {
    const float2 v = __bfloat1622float2(__floats2bfloat162_rn(a, b));
    a = v.x;
    b = v.y;
  }
}

// Two consecutive Real values (one 8 or 16-byte load).
template <class R> struct R2Of;
template <> struct R2Of<float> { using T = float2; };
template <> struct R2Of<double> { using T = double2; };
template <class R> using R2 = typename R2Of<R>::T;

// ------------------------------------------------------------ geometry
struct Geo {
  int nx, ny, nz;
  int wall;        // walls at both ends of z
  long long N;     // cells
  long long P;     // plane stride of population / field arrays (>= N, padded)
  int P32;         // P as int: every population offset (3Q planes) fits 31 bits
};

// Cell (x, y, z) of linear index n < N (N < 2^31: every population offset
// fits 31 bits), by two 32-bit divisions.
__device__ __forceinline__ void cell_xyz(const Geo& G, long long n, int& x, int& y, int& z) {
  const unsigned un = (unsigned)n, t = un / (unsigned)G.nx, zz = t / (unsigned)G.ny;
  x = (int)(un - t * (unsigned)G.nx);
  y = (int)(t - zz * (unsigned)G.ny);
  z = (int)zz;
}

// Block coordinates of a launch.  Kernel bodies take them as an argument, so
// one body runs either as its own grid (the hardware block index) or as one
// virtual block of a batched persistent launch over many lattices.
struct Blk {
  int x, y, z;     // block index
  int gx, gy, gz;  // grid size in blocks
};
__device__ __forceinline__ Blk hw_blk() {
  return {(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, (int)gridDim.x, (int)gridDim.y, (int)gridDim.z};
}

TLB_HD int wrapc(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// Population layout: `lo` holds 3Q-2 planes of Store -- f_0..f_{Q-1} stored
// as f_i - w_i, then g_1..g_{Q-1}, then h_1..h_{Q-1}; `rest` holds g_0, h_0 in
// the Rest type.  Plane k of `lo` starts at lo + k*P.
template <class L> TLB_HD int plane_f(int i) { return i; }
template <class L> TLB_HD int plane_g(int i) { return L::Q + i - 1; }
template <class L> TLB_HD int plane_h(int i) { return 2 * L::Q - 1 + i - 1; }

template <class Real>
struct CellMoments {
  Real drho;     // rho - 1 (sum of the stored deviations)
  Real j[3];     // sum_i c_i f_i
  Real phi, psi;
};

// Source of the populations arriving at cell (x, y, z): direction i comes
// from x - c_i (periodic wrap), or, across a wall, from the cell itself in
// direction opp(i) (halfway bounce-back).  The wrapped neighbour rows are
// computed once per cell, so each pulled population costs one add.
template <class L>
struct Nbr {
  int self;
  int row[3][3];  // [dz + 1][dy + 1]: (z + dz, y + dy) row start
  int xs[3];      // x - 1, x, x + 1 (wrapped)
  bool wlo, whi;  // cell touches the bottom / top wall

  __device__ __forceinline__ Nbr(const Geo& G, int x, int y, int z) {
    self = (z * G.ny + y) * G.nx + x;
    xs[0] = x == 0 ? G.nx - 1 : x - 1;
    xs[1] = x;
    xs[2] = x == G.nx - 1 ? 0 : x + 1;
    int ys[3] = {y == 0 ? G.ny - 1 : y - 1, y, y == G.ny - 1 ? 0 : y + 1};
    int zs[3] = {z == 0 ? G.nz - 1 : z - 1, z, z == G.nz - 1 ? 0 : z + 1};
    wlo = G.wall && z == 0;
    whi = G.wall && z == G.nz - 1;
#pragma unroll
    for (int dz = 0; dz < 3; ++dz)
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) row[dz][dy] = (zs[dz] * G.ny + ys[dy]) * G.nx;
  }
  // bounce-back applies to direction i at this cell
  __device__ __forceinline__ bool bounce(int i) const {
    return (L::cz(i) > 0 && wlo) || (L::cz(i) < 0 && whi);
  }
  __device__ __forceinline__ int src(int i) const {
    return bounce(i) ? self : row[1 - L::cz(i)][1 - L::cy(i)] + xs[1 - L::cx(i)];
  }
  // offset of the population of direction i arriving here, in a plane array
  // whose plane for direction i (no bounce) or opp(i) (bounce) is given
  __device__ __forceinline__ int off(int i, int plane_i, int plane_opp, int P32) const {
    return (bounce(i) ? plane_opp : plane_i) * P32 + src(i);
  }
};

// Pull of the populations arriving at cell (x, y, z): f_i(x) = f*_i(x - c_i);
// across a wall, halfway bounce-back returns f*_{opp(i)}(x).  Both the moment
// kernel and the collision kernel use this routine so they agree bit for bit.
template <class L, int MODE>
struct Pull {
  using Real = typename Prec<MODE>::Real;
  using Store = typename Prec<MODE>::Store;
  using Rest = typename Prec<MODE>::Rest;
  Real f[L::Q], g[L::Q], h[L::Q];  // f holds f_i - w_i

  __device__ __forceinline__ void load(const Store* __restrict__ lo, const Rest* __restrict__ rest,
                                       const Geo& G, int x, int y, int z) {
    const Nbr<L> nb(G, x, y, z);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      f[i] = to_real(__ldg(lo + nb.off(i, plane_f<L>(i), plane_f<L>(L::opp(i)), G.P32)));
      if (i == 0) {
        g[0] = to_real(__ldg(rest + nb.self));
        h[0] = to_real(__ldg(rest + G.P32 + nb.self));
      } else {
        g[i] = to_real(__ldg(lo + nb.off(i, plane_g<L>(i), plane_g<L>(L::opp(i)), G.P32)));
        h[i] = to_real(__ldg(lo + nb.off(i, plane_h<L>(i), plane_h<L>(L::opp(i)), G.P32)));
      }
    }
  }

  // Sums in the order a sweep along z meets the populations: those with c_z
  // = 1 (they come from the plane below), then c_z = 0, then c_z = -1, each
  // over the in-plane velocities; so the rebuilding sweep of the tau = 1
  // scheme (moments_recon_body) gives the same bits.  The rest populations
  // are added last: g_0 and h_0 carry nearly all of
  // phi and psi, so the small moving populations are summed first at their
  // own scale and the sum is rounded once at the scale of phi (adding them
  // one by one to g_0 rounds each addition there: in FP32 that made the
  // force about 4 times noisier).
  __device__ __forceinline__ CellMoments<Real> moments() const {
    CellMoments<Real> m;
    Real r = 0, jx = 0, jy = 0, jz = 0, p = 0, s = 0;
#pragma unroll
    for (int cz = 1; cz >= -1; --cz)
#pragma unroll
      for (int k = 0; k < L::NCOL; ++k) {
        const int i = col_dir<L>(k, cz);
        if (i <= 0) continue;
        r += f[i];
        if (L::cx(i)) jx += L::cx(i) > 0 ? f[i] : -f[i];
        if (L::cy(i)) jy += L::cy(i) > 0 ? f[i] : -f[i];
        if (L::cz(i)) jz += L::cz(i) > 0 ? f[i] : -f[i];
        p += g[i];
        s += h[i];
      }
    r += f[0];
    p += g[0];
    s += h[0];
    m.drho = r;
    m.j[0] = jx;
    m.j[1] = jy;
    m.j[2] = jz;
    m.phi = p;
    m.psi = s;
    return m;
  }
};

// Cells the membrane work of a step touches: the marker box of the step
// (cur[0..2] = floor(min X), cur[3..5] = -ceil(max X)) widened by `margin`
// cells, unwrapped; walls clamp z; at most one period per axis.
__device__ __forceinline__ void marker_box(const int* cur, int margin, const Geo& G, bool d2, int* lo, int* hi) {
  const int n[3] = {G.nx, G.ny, G.nz};
  for (int d = 0; d < 3; ++d) {
    int bl = cur[d] - margin, bh = -cur[3 + d] + margin;
    if (d == 1 && d2) { bl = 0; bh = 0; }
    if (d == 2 && G.wall) { bl = max(bl, 0); bh = min(bh, n[2] - 1); }
    if (bh - bl + 1 > n[d]) bh = bl + n[d] - 1;
    if (bh < bl) bh = bl;
    lo[d] = bl;
    hi[d] = bh;
  }
}

// Chemical potentials of App. A (eq. AppA) without the ideal-gas part of
// mu_rho; mu_psi' adds kappa_c (psi - I) (Sec. 3.1).  The density enters as
// drho = rho - 1 (and Lr as its Laplacian, which is the Laplacian of rho):
// with A = rho + phi - psi = 1 + a, A (A - 1)(A - 2) = a (a^2 - 1), the same
// polynomial written around the bulk value, so that a working-precision
// drho keeps its low bits (rho = 1 + drho would round them away).
template <class Real>
struct FEParams {
  Real k1, k2, k3, kc, a2;  // kappa_1..3, kappa_c, alpha^2
};
template <class Real>
__device__ __forceinline__ void chem_potentials(const FEParams<Real>& fe, Real drho, Real phi, Real psi,
                                                Real Lr, Real Lp, Real Ls, Real I, Real& mr,
                                                Real& mp, Real& ms) {
  const Real a = drho + phi - psi, b = drho - phi - psi;  // A - 1, B - 1
  Real tA = fe.k1 * Real(0.125) * a * (a * a - Real(1));
  Real tB = fe.k2 * Real(0.125) * b * (b * b - Real(1));
  Real q = Real(0.25) * fe.a2;
  Real kp = fe.k1 + fe.k2, km = fe.k2 - fe.k1;
  mr = tA + tB + q * (kp * (Ls - Lr) + km * Lp);
  mp = tA - tB + q * (km * (Lr - Ls) - kp * Lp);
  ms = -tA - tB + q * (kp * Lr - km * Lp - (kp + Real(4) * fe.k3) * Ls) +
       fe.k3 * psi * (psi - Real(1)) * (Real(2) * psi - Real(1)) + fe.kc * (psi - I);
}

// Explicitly rounded arithmetic (round to nearest, never contracted): the
// same expression then rounds the same way in every kernel it is inlined
// into, whatever the compiler's multiply-add contraction would choose there.
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// ------------------------------------------------ the tau = 1 state
// At tau = tau_phi = tau_psi = 1 with the exact difference method every
// post-collision population is an equilibrium (eq. EDF) of its cell:
// f*_i = f_i^eq(rho, w) with w = u + du, g*_i = g_i^eq(phi, Gamma_phi mu_phi,
// v), h*_i = h_i^eq(psi, Gamma_psi mu_psi', v) (eq. LBE at tau = 1).  These
// 11 values per cell stand for the 3Q populations between steps; the pull of
// the next step rebuilds each population from the cell it streams from, as
// its storage type holds it: with 16-bit storage every rebuilt population is
// rounded, so the state is that of stored populations, bit for bit.
// They are kept as three 16-byte vectors per cell (32 in double precision),
// one plane array each: (rho - 1, q), (phi, 3 Gamma_phi mu_phi, psi,
// 3 Gamma_psi mu_psi'), (v, 1/rho) with q = rho w = j + F.  A cell is then
// moved by three vector copies instead of eleven.  The momentum q, rounded
// once, is the linear part of every f_i; w would be rounded three times on its
// way back to it (in FP32 that made the velocity's error a quarter larger than
// with stored populations).  3 Gamma mu and 1/rho spare the readers their
// products and the division.
enum { M_F = 0, M_ORD = 1, M_V = 2, M_COUNT = 3 };

// Four values of one cell side by side: one 16-byte access (two in double
// precision).
template <class R>
struct alignas(4 * sizeof(R)) R4 {
  R x, y, z, w;
};
// one vector through the read-only path
__device__ __forceinline__ R4<float> ldg4(const R4<float>* p) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ R4<double> ldg4(const R4<double>* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = __ldg(q), b = __ldg(q + 1);
  return {a.x, a.y, b.x, b.y};
}

// The post-collision populations of one cell from its stored state, with the
// explicitly rounded operations (see rmul), so the rebuild in the pull, in
// the interpolation and in the materialised populations gives the same value.
template <class L, int MODE>
struct EqCell {
  using Real = typename Prec<MODE>::Real;
  using Store = typename Prec<MODE>::Store;
  Real ds, k, q[3], ord[2], gm3[2], v[3], v15;
  // rho - 1, q and 1/rho only (what f_i needs)
  __device__ __forceinline__ void set_f(const R4<Real>& A, Real irho) {
    q[0] = A.y;
    q[1] = A.z;
    q[2] = A.w;
    const Real qq = rfma(q[2], q[2], rfma(q[1], q[1], rmul(q[0], q[0])));
    k = rmul(Real(4.5), irho);
    ds = rfma(rmul(Real(-1.5), irho), qq, A.x);
  }
  __device__ __forceinline__ void set(const R4<Real>& A, const R4<Real>& B, const R4<Real>& C) {
    set_f(A, C.w);
    ord[0] = B.x;
    gm3[0] = B.y;
    ord[1] = B.z;
    gm3[1] = B.w;
    v[0] = C.x;
    v[1] = C.y;
    v[2] = C.z;
    v15 = rmul(Real(-1.5), rfma(v[2], v[2], rfma(v[1], v[1], rmul(v[0], v[0]))));
  }
  __device__ __forceinline__ void load(const R4<Real>* M, int P32, int c) {
    set(M[M_F * P32 + c], M[M_ORD * P32 + c], M[M_V * P32 + c]);
  }
  // f_i - w_i = w_i (rho - 1 + 3 c.q + (4.5 (c.q)^2 - 1.5 q^2) / rho)
  __device__ __forceinline__ Real f(int i) const { return f_or_back(i, false); }
  // the same of direction i, or of its opposite where `back` (c.q changes sign)
  __device__ __forceinline__ Real f_or_back(int i, bool back) const {
    if (i == 0) return as_stored<Store>(rmul(Real(L::w(0)), ds));
    const Real c = cdot<L>(i, q), cq = back ? -c : c;
    return as_stored<Store>(rmul(Real(L::w(i)), rfma(cq, rfma(k, cq, Real(3)), ds)));
  }
  // 3 c.u + 4.5 (c.u)^2 - 1.5 u^2
  static __device__ __forceinline__ Real poly(int i, const Real* u, Real u15) {
    const Real cu = cdot<L>(i, u);
    return rfma(cu, rfma(Real(4.5), cu, Real(3)), u15);
  }
  // g_i and h_i for i != 0: w_i (3 Gamma mu + ord p(c.v)); the rest population
  // closes the zeroth moment
  __device__ __forceinline__ void gh(int i, Real* g, Real* h) const {
    const Real p = poly(i, v, v15);
    *g = rmul(Real(L::w(i)), rfma(ord[0], p, gm3[0]));
    *h = rmul(Real(L::w(i)), rfma(ord[1], p, gm3[1]));
    as_stored2<Store>(*g, *h);
  }
  __device__ __forceinline__ Real rest(int s) const {
    return radd(rfma(gm3[s], Real(L::w(0)) - Real(1), ord[s]), rmul(rmul(Real(L::w(0)), ord[s]), v15));
  }
};

// Status flags written by kernels (bitwise OR into a device word).
enum { ST_NAN = 1, ST_MARKER_JUMP = 2, ST_TIMEOUT = 4, ST_OVERFLOW = 8 };
