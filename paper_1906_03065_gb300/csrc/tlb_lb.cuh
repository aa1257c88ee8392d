// Lattice Boltzmann kernels: moments, chemical potentials, the fused
// force + collision + streaming plane sweep, initial equilibria and the
// conversions used by read/write of populations.
#pragma once
#include <type_traits>

#include "tlb_common.cuh"

template <int MODE>
struct LBArgs {
  using Real = typename Prec<MODE>::Real;
  using Store = typename Prec<MODE>::Store;
  using Rest = typename Prec<MODE>::Rest;
  Geo G;
  const Store* lo_src;
  const Rest* rest_src;
  Store* lo_dst;
  Rest* rest_dst;
  Real* rho;        // rho - 1 (the deviation keeps its low bits in FP32)
  Real* phi;
  Real* psi;
  R4<Real>* p4;     // [P] (rho - 1, phi, psi, j_x) of the streamed populations
                    // (NULL with the pressure-tensor force: rho, phi, psi)
  // the tau = 1 scheme (NULL otherwise):
  R2<Real>* j2;     // [P] (j_y, j_z)
  R4<Real>* M;      // [3][P] the stored state (see EqCell)
  int pull;         // the state is in the populations, not in M (set by an
                    // initialisation, a load or a write): pull them this once
  const int* in_M;  // not NULL: this device word decides instead (0: pull)
  const Real* I;
  const Real* fib;  // [3][P] immersed-boundary force density
  Real* ftot;       // [3][P] total force of the step (read by the interpolation)
  const unsigned char* bflag;  // per 4x4x4 brick: markers spread force into it
  int nbx, nby;                // brick grid (x, y)
  FEParams<Real> fe;
  Real om, om_phi, om_psi;  // 1/tau
  Real gphi, gpsi;          // Gamma_phi, Gamma_psi
  int zc;                   // planes per block along z (the collide)
  int zcm;                  // the same of the rebuilding moments sweep
  int forcing;              // TLB_FORCE_EDM or TLB_FORCE_GUO
  unsigned* status;
};

// Asynchronous global -> shared copy of one cell's four values (cp.async, 16
// bytes each): the copy runs while the thread computes; cp_async_wait<N>
// blocks until all but the thread's newest N groups have landed.
template <class R>
__device__ __forceinline__ void cp_async_r4(R4<R>* dst, const R4<R>* src) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll
  for (int k = 0; k < (int)(sizeof(R4<R>) / 16); ++k)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s + 16 * k), "l"((const char*)src + 16 * k)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Periodic wrap of a halo index: within two cells of the range except for
// tiles wider than the lattice, which take the division.
__device__ __forceinline__ int halo_wrap(int v, int n) {
  if (v < 0) v += n;
  if (v >= n) v -= n;
  if (v < 0 || v >= n) {
    v %= n;
    if (v < 0) v += n;
  }
  return v;
}
// Plane p of the sweeps' rings: periodic, or the plane next to a wall for the
// ghosts beyond it.
__device__ __forceinline__ int ring_plane(const Geo& G, int p) {
  return G.wall ? min(max(p, 0), G.nz - 1) : halo_wrap(p, G.nz);
}

// ---------------------------------------------------------------- moments
// rho - 1, phi, psi at every cell from the streamed populations (eq.
// MomentsDFs); with the tau = 1 scheme j too.
template <class L, int MODE>
__device__ __forceinline__ void moments_store(const LBArgs<MODE>& a, int n, const CellMoments<typename Prec<MODE>::Real>& m) {
  using Real = typename Prec<MODE>::Real;
  if (a.p4) {
    a.p4[n] = R4<Real>{m.drho, m.phi, m.psi, m.j[0]};
    if (a.j2) {
      R2<Real> t;
      t.x = m.j[1];
      t.y = m.j[2];
      a.j2[n] = t;
    }
  } else {
    a.rho[n] = m.drho;
    a.phi[n] = m.phi;
    a.psi[n] = m.psi;
  }
}
template <class L, int MODE>
__device__ __forceinline__ void moments_body(const LBArgs<MODE>& a, const Blk& blk) {
  const Geo G = a.G;
  long long n = (long long)blk.x * blockDim.x + threadIdx.x;
  if (n >= G.N) return;
  int x, y, z;
  cell_xyz(G, n, x, y, z);
  Pull<L, MODE> p;
  p.load(a.lo_src, a.rest_src, G, x, y, z);
  moments_store<L, MODE>(a, (int)n, p.moments());
}
template <class L, int MODE>
__global__ void __launch_bounds__(256) k_moments(const __grid_constant__ LBArgs<MODE> a) {
  moments_body<L, MODE>(a, hw_blk());
}

// Moments of the streamed populations of the tau = 1 scheme, each population
// rebuilt from the stored state of the cell it streams from (across a wall:
// this cell's opposite direction, halfway bounce-back).
//
// A TX x TY tile of columns walks a.zc planes; a plane of the state (tile
// plus a halo of 1) is copied into one of two shared-memory slots while the
// plane before it is used.  A thread reads the 9 (2D: 3) columns around its
// own once per plane and adds what each sends to the three planes it feeds:
// c_z = 1 starts the sums of the plane above, c_z = 0 continues this plane's,
// c_z = -1 and the rest populations finish those of the plane below.  So the
// running sums of two planes live in registers and a state vector is read 9
// times from shared memory instead of 19.  The order of the additions is
// that of Pull::moments.
//
// Bound by instruction issue and the shared-memory reads, not by its 72 B per
// cell: 128^3 FP32 48 us (3.1 TB/s), where pulling the populations took 79 us
// at 252 B per cell and the full copy bandwidth.
template <class L, int MODE, int TX, int TY>
__device__ __forceinline__ void moments_recon_body(const LBArgs<MODE>& a, const Blk& blk) {
  using Real = typename Prec<MODE>::Real;
  constexpr bool D3 = L::DIM == 3;
  constexpr int HX = TX + 2, HY = D3 ? TY + 2 : 1, CELLS = HX * HY, NT = TX * TY, NL = (CELLS + NT - 1) / NT;
  __shared__ R4<Real> sA[2][CELLS], sB[2][CELLS], sC[2][CELLS];
  const Geo G = a.G;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int x0 = blk.x * TX, y0 = blk.y * TY, z0 = blk.z * a.zcm, z1 = min(z0 + a.zcm, G.nz);
  const int x = x0 + tx, y = y0 + ty;
  const bool active = x < G.nx && y < G.ny;
  if (a.in_M ? *a.in_M == 0 : a.pull) {  // once after an initialisation or a write of populations
    if (active)
      for (int zz = z0; zz < z1; ++zz) {
        Pull<L, MODE> p;
        p.load(a.lo_src, a.rest_src, G, x, y, zz);
        moments_store<L, MODE>(a, (zz * G.ny + y) * G.nx + x, p.moments());
      }
    return;
  }
  int coff[NL];  // in-plane offsets of the cells this thread copies
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    const int k = tid + j * NT, gx = halo_wrap(x0 - 1 + k % HX, G.nx);
    coff[j] = (D3 ? halo_wrap(y0 - 1 + k / HX, G.ny) * G.nx : 0) + gx;
  }
  const int nxy = G.nx * G.ny;
  auto issue = [&](int p, int slot) {
    const R4<Real>* M = a.M + (long long)ring_plane(G, p) * nxy;
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const int k = tid + j * NT;
      if (k < CELLS) {
        cp_async_r4(&sA[slot][k], M + M_F * G.P32 + coff[j]);
        cp_async_r4(&sB[slot][k], M + M_ORD * G.P32 + coff[j]);
        cp_async_r4(&sC[slot][k], M + M_V * G.P32 + coff[j]);
      }
    }
    cp_async_commit();
  };
  struct Acc {
    Real r, jx, jy, jz, p, s;
  };
  Acc lo = {0, 0, 0, 0, 0, 0}, mid = lo;  // sums of planes q - 1 and q
  Real rest_lo[3] = {0, 0, 0};            // rest populations of plane q - 1
  auto add = [](Acc& t, int i, Real f, Real g, Real h) {
    t.r += f;
    if (L::cx(i)) t.jx += L::cx(i) > 0 ? f : -f;
    if (L::cy(i)) t.jy += L::cy(i) > 0 ? f : -f;
    if (L::cz(i)) t.jz += L::cz(i) > 0 ? f : -f;
    t.p += g;
    t.s += h;
  };
  issue(z0 - 1, 0);
  const int sc = (D3 ? ty + 1 : 0) * HX + tx + 1;
  for (int q = z0 - 1; q <= z1; ++q) {
    const int slot = (q - z0 + 1) & 1;
    cp_async_wait<0>();
    __syncthreads();
    if (q < z1) issue(q + 1, slot ^ 1);  // (every thread has left plane q - 1)
    // walls: nothing comes from the ghost planes; a cell next to the wall
    // takes its own opposite populations where theirs would have come
    const bool ghost = G.wall && (q < 0 || q >= G.nz);
    const bool wlo = G.wall && q == 0, whi = G.wall && q == G.nz - 1 && q < z1;
    Acc up = {0, 0, 0, 0, 0, 0};
    Real rest_mid[3] = {0, 0, 0};
    auto bounce = [&](Acc& t, int cz) {  // own populations opposite to the c_z = cz ones
      EqCell<L, MODE> e;
      e.set(sA[slot][sc], sB[slot][sc], sC[slot][sc]);
#pragma unroll
      for (int k = 0; k < L::NCOL; ++k) {
        const int i = col_dir<L>(k, cz);
        if (i < 0) continue;
        const int o = L::opp(i);
        Real g, h;
        e.gh(o, &g, &h);
        add(t, i, e.f(o), g, h);
      }
    };
    if (!ghost) {
      if (wlo) bounce(mid, 1);
#pragma unroll
      for (int k = 0; k < L::NCOL; ++k) {
        // the column whose populations with in-plane velocity k arrive here
        const int n = sc - col_cy(k) * HX - col_cx(k);
        EqCell<L, MODE> e;
        e.set(sA[slot][n], sB[slot][n], sC[slot][n]);
#pragma unroll
        for (int cz = 1; cz >= -1; --cz) {
          const int i = col_dir<L>(k, cz);
          if (i < 0) continue;
          if (i == 0) {
            rest_mid[0] = e.f(0);
            rest_mid[1] = e.rest(0);
            rest_mid[2] = e.rest(1);
          } else {
            Real g, h;
            e.gh(i, &g, &h);
            add(cz > 0 ? up : (cz == 0 ? mid : lo), i, e.f(i), g, h);
          }
        }
      }
    }
    auto put = [&](const Acc& t, const Real* rest, int z) {
      CellMoments<Real> m;
      m.drho = t.r + rest[0];
      m.j[0] = t.jx;
      m.j[1] = t.jy;
      m.j[2] = t.jz;
      m.phi = t.p + rest[1];
      m.psi = t.s + rest[2];
      moments_store<L, MODE>(a, (z * G.ny + y) * G.nx + x, m);
    };
    if (q > z0 && active) put(lo, rest_lo, q - 1);
    if (whi) {  // the top plane is complete with its own bounce (q == z1 - 1)
      bounce(mid, -1);
      if (active) put(mid, rest_mid, q);
      break;
    }
    lo = mid;
    mid = up;
#pragma unroll
    for (int d = 0; d < 3; ++d) rest_lo[d] = rest_mid[d];
  }
  cp_async_wait<0>();
}
// threads per SM the register budget is set for: 768
template <class L, int MODE, int TX, int TY>
__global__ void __launch_bounds__(TX* TY, 768 / (TX * TY)) k_moments_recon(const __grid_constant__ LBArgs<MODE> a) {
  moments_recon_body<L, MODE, TX, TY>(a, hw_blk());
}

// The populations a cell's stored state stands for, written post-collision
// into the population buffers (for the readers of the population state).
// in_M not NULL: only if the state is in M.
template <class L, int MODE>
__global__ void k_materialize(Geo G, const R4<typename Prec<MODE>::Real>* M, typename Prec<MODE>::Store* lo,
                              typename Prec<MODE>::Rest* rest, const int* in_M) {
  using Real = typename Prec<MODE>::Real;
  using Store = typename Prec<MODE>::Store;
  using Rest = typename Prec<MODE>::Rest;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= G.N || (in_M && *in_M == 0)) return;
  EqCell<L, MODE> e;
  e.load(M, G.P32, (int)n);
  lo[(long long)plane_f<L>(0) * G.P + n] = from_real<Store>(e.f(0));
  rest[n] = from_real<Rest>(e.rest(0));
  rest[G.P + n] = from_real<Rest>(e.rest(1));
#pragma unroll
  for (int i = 1; i < L::Q; ++i) {
    Real g, h;
    e.gh(i, &g, &h);
    lo[(long long)plane_f<L>(i) * G.P + n] = from_real<Store>(e.f(i));
    lo[(long long)plane_g<L>(i) * G.P + n] = from_real<Store>(g);
    lo[(long long)plane_h<L>(i) * G.P + n] = from_real<Store>(h);
  }
}

// Second-order polynomial of the equilibria: 3 c.u + 4.5 (c.u)^2 - 1.5 u^2.
template <class Real>
__device__ __forceinline__ Real eq_poly(Real cu, Real uu) {
  return Real(3) * cu + Real(4.5) * cu * cu - Real(1.5) * uu;
}

// Collision of one cell with its populations (eq. LBE): the three sets are
// pulled, collided and stored one after another, so only one is live in
// registers at a time.  rho, phi, psi are the cell's moments, F its force,
// mup and mus its potentials mu_phi and mu_psi'.
template <class L, int MODE>
__device__ __forceinline__ void collide_pops(const LBArgs<MODE>& a, const Nbr<L>& nb, typename Prec<MODE>::Real phi,
                                             typename Prec<MODE>::Real psi, typename Prec<MODE>::Real rho,
                                             const typename Prec<MODE>::Real* F, typename Prec<MODE>::Real mup,
                                             typename Prec<MODE>::Real mus) {
  using Real = typename Prec<MODE>::Real;
  using Store = typename Prec<MODE>::Store;
  using Rest = typename Prec<MODE>::Rest;
  constexpr int Q = L::Q;
  const Geo& G = a.G;
  const int n = nb.self;
  // pull of the order-parameter set `set` (0: g, 1: h) into v
  auto load_set = [&](int set, Real* v) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (i == 0) {
        v[0] = to_real(__ldg(a.rest_src + (set == 0 ? 0 : G.P32) + n));
      } else {
        const int o = set == 0 ? nb.off(i, plane_g<L>(i), plane_g<L>(L::opp(i)), G.P32)
                               : nb.off(i, plane_h<L>(i), plane_h<L>(L::opp(i)), G.P32);
        v[i] = to_real(__ldg(a.lo_src + o));
      }
    }
  };
  // f: pull, first moment, BGK + exact difference method (eq. LBE) for f_i - w_i
  Real fv[Q];
  Real drho = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    fv[i] = to_real(__ldg(a.lo_src + nb.off(i, plane_f<L>(i), plane_f<L>(L::opp(i)), G.P32)));
  }
#pragma unroll
  for (int cz = 1; cz >= -1; --cz)  // in the order of Pull::moments (rest last)
#pragma unroll
    for (int k = 0; k < L::NCOL; ++k) {
      const int i = col_dir<L>(k, cz);
      if (i <= 0) continue;
      drho += fv[i];
      if (L::cx(i)) jx += L::cx(i) > 0 ? fv[i] : -fv[i];
      if (L::cy(i)) jy += L::cy(i) > 0 ? fv[i] : -fv[i];
      if (L::cz(i)) jz += L::cz(i) > 0 ? fv[i] : -fv[i];
    }
  drho += fv[0];
  const Real irho = Real(1) / rho;
  const Real j[3] = {jx, jy, jz};
  Real u[3], du[3], v[3], us[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    u[d] = j[d] * irho;
    du[d] = F[d] * irho;
    v[d] = u[d] + Real(0.5) * du[d];
    us[d] = u[d] + u[d] + du[d];  // u + (u + du)
  }
  const Real uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const Real vv = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
  const Real dus = du[0] * us[0] + du[1] * us[1] + du[2] * us[2];
  const Real om = a.om;
  if (a.forcing == TLB_FORCE_GUO) {
    // Guo forcing: BGK towards f^eq(rho, v) plus (1 - om/2) w_i [3 (c_i - v) + 9 (c_i.v) c_i] . F
    const Real vF = v[0] * F[0] + v[1] * F[1] + v[2] * F[2];
    const Real sc = Real(1) - Real(0.5) * om;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const Real w = Real(L::w(i));
      const Real cv = cdot<L>(i, v);
      const Real cF = cdot<L>(i, F);
      const Real fn = (Real(1) - om) * fv[i] + om * w * (drho + rho * eq_poly(cv, vv)) +
                      sc * w * (Real(3) * (cF - vF) + Real(9) * cv * cF);
      a.lo_dst[plane_f<L>(i) * G.P32 + n] = from_real<Store>(fn);
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const Real w = Real(L::w(i));
      const Real cu = cdot<L>(i, u);
      const Real cdu = cdot<L>(i, du);
      const Real cus = cdot<L>(i, us);
      const Real dP = Real(3) * cdu + Real(4.5) * cdu * cus - Real(1.5) * dus;
      const Real fn = (Real(1) - om) * fv[i] + om * w * (drho + rho * eq_poly(cu, uu)) + w * rho * dP;
      a.lo_dst[plane_f<L>(i) * G.P32 + n] = from_real<Store>(fn);
    }
  }
  // g and h: BGK towards the order-parameter equilibria at v (eq. EDF); the
  // rest population closes the zeroth moment
  const Real w0 = Real(L::w(0));
#pragma unroll
  for (int set = 0; set < 2; ++set) {
    const Real om_s = set == 0 ? a.om_phi : a.om_psi;
    const Real Gm = set == 0 ? a.gphi * mup : a.gpsi * mus;
    const Real ord = set == 0 ? phi : psi;
    Real gv[Q];
    load_set(set, gv);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const Real w = Real(L::w(i));
      const Real cv = cdot<L>(i, v);
      const Real pv = Real(3) * cv + Real(4.5) * cv * cv - Real(1.5) * vv;
      const Real ge = w * (Real(3) * Gm + ord * pv);
      const int pp = set == 0 ? plane_g<L>(i) : plane_h<L>(i);
      a.lo_dst[pp * G.P32 + n] = from_real<Store>((Real(1) - om_s) * gv[i] + om_s * ge);
    }
    const Real ge0 = ord - Real(3) * Gm * (Real(1) - w0) - Real(1.5) * w0 * ord * vv;
    a.rest_dst[(set == 0 ? 0 : G.P32) + n] = from_real<Rest>((Real(1) - om_s) * gv[0] + om_s * ge0);
  }
}

// ------------------------------------------------- fused collide + stream
// One block owns a TX x TY tile of (x, y) columns and sweeps a chunk of z
// planes.  Shared memory holds a 5-plane ring of the moment fields rho - 1,
// phi, psi (halo 2,
// written by k_moments; halo reads are served by L2) and a 3-plane ring of
// the chemical potentials (halo 1), so each cell's radius-2 dependency (mu
// needs the Laplacian of the moments, the force needs the gradient of mu) is
// served on chip.
// Pressure tensor of App. A without its ideal-gas part rho cs^2 delta (the
// force form grad(rho cs^2) - div p needs only the rest), in the variables
// rho, phi, psi with the mixing coefficients k_rr = k_ff = (k1 + k2)/4,
// k_ss = (k1 + k2 + 4 k3)/4, k_rf = -k_fs = (k1 - k2)/4, k_rs = -(k1 + k2)/4:
//   p'_ab = p'_b delta_ab + alpha^2 sum_mn k_mn [d_a m d_b n - delta_ab
//           ((1/2) grad m . grad n + m lap n)],
// with the bulk pressure of eq. PressureV2 (the ideal part dropped),
// p'_b = rho mu_rho^b + phi mu_phi^b + psi mu_psi^b - f_b and f_b = sum_m
// kappa_m/2 C_m^2 (1 - C_m)^2 = kappa1/32 (1 - a^2)^2 + kappa2/32 (1 - b^2)^2
// + kappa3/2 psi^2 (1 - psi)^2 (a = A - 1, b = B - 1 as in chem_potentials).
// Components xx, yy, zz, xy, xz, yz.  gr: the lattice gradients of rho - 1,
// phi, psi; lap: their Laplacians.
template <class Real>
__device__ __forceinline__ void pressure_tensor(const FEParams<Real>& fe, Real drho, Real phi, Real psi,
                                                const Real* lap, const Real (*gr)[3], Real* out) {
  const Real a = drho + phi - psi, b = drho - phi - psi;
  const Real tA = fe.k1 * Real(0.125) * a * (a * a - Real(1));
  const Real tB = fe.k2 * Real(0.125) * b * (b * b - Real(1));
  const Real ta = Real(1) - a * a, tb = Real(1) - b * b, tp = psi * (Real(1) - psi);
  const Real fb = fe.k1 * Real(1.0 / 32) * ta * ta + fe.k2 * Real(1.0 / 32) * tb * tb + fe.k3 * Real(0.5) * tp * tp;
  const Real rho = Real(1) + drho;
  const Real pb = rho * (tA + tB) + phi * (tA - tB) +
                  psi * (-tA - tB + fe.k3 * psi * (psi - Real(1)) * (Real(2) * psi - Real(1))) - fb;
  const Real kp = Real(0.25) * (fe.k1 + fe.k2), km = Real(0.25) * (fe.k1 - fe.k2);
  const Real K[3][3] = {{kp, km, -kp}, {km, kp, -km}, {-kp, -km, kp + fe.k3}};
  const Real val[3] = {rho, phi, psi};
  Real tr = pb;
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const Real gg = gr[m][0] * gr[n][0] + gr[m][1] * gr[n][1] + gr[m][2] * gr[n][2];
      tr -= fe.a2 * K[m][n] * (Real(0.5) * gg + val[m] * lap[n]);
    }
  const int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    Real t = ia[q] == ib[q] ? tr : Real(0);
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int n = 0; n < 3; ++n) t += fe.a2 * K[m][n] * gr[m][ia[q]] * gr[n][ib[q]];
    out[q] = t;
  }
}

// Forms 5 and 6 are the collide at tau = tau_phi = tau_psi = 1 with the exact
// difference method, form 7 the general one with the pressure-tensor force,
// form 1 the general one.
template <int FORM> constexpr bool form_t1() { return FORM == 5 || FORM == 6; }

template <class L, int MODE, int TX, int TY>
__device__ __forceinline__ void collide_pt_body(const LBArgs<MODE>& a, const Blk& blk) {
  using Real = typename Prec<MODE>::Real;
  constexpr int Q = L::Q;
  constexpr bool D3 = L::DIM == 3;
  constexpr int HY = D3 ? 2 : 0;
  constexpr int MX = TX + 4, MY = TY + 2 * HY;
  constexpr int UX = TX + 2, UY = TY + (D3 ? 2 : 0);
  constexpr int NT = TX * TY;
  // per cell of the potentials' ring: p_xx p_yy p_zz p_xy p_xz p_yz, kappa_c
  // (psi - I), mu_phi, mu_psi'
  constexpr int NMU = 9, MUP = 7, MUS = 8;
  __shared__ Real smom[5][3][MY * MX];
  __shared__ Real smu[3][NMU][UY * UX];

  const Geo G = a.G;
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX, tid = threadIdx.x;
  const int x0 = blk.x * TX, y0 = blk.y * TY;
  const int z0 = blk.z * a.zc;
  const int z1 = min(z0 + a.zc, G.nz);
  const int x = x0 + tx, y = y0 + ty;
  const bool active = x < G.nx && y < G.ny;

  auto load_mom = [&](int p) {
    const int slot = (p + 10) % 5;
    const long long zp = (long long)ring_plane(G, p) * G.ny;
    for (int k = tid; k < MX * MY; k += NT) {
      int hx = k % MX, hy = k / MX;
      int gx = halo_wrap(x0 - 2 + hx, G.nx);
      int gy = D3 ? halo_wrap(y0 - HY + hy, G.ny) : 0;
      long long c = (zp + gy) * G.nx + gx;
      smom[slot][0][k] = a.rho[c];
      smom[slot][1][k] = a.phi[c];
      smom[slot][2][k] = a.psi[c];
    }
  };

  // chemical potentials of plane p on the tile plus a halo of 1
  auto compute_mu = [&](int p) {
    const int slot = (p + 9) % 3;
    if (G.wall && (p < 0 || p >= G.nz)) {  // mirror ghost: mu(-1) = mu(0), mu(nz) = mu(nz-1)
      const int src = (min(max(p, 0), G.nz - 1) + 9) % 3;
      for (int k = tid; k < UX * UY; k += NT)
        for (int q = 0; q < NMU; ++q) smu[slot][q][k] = smu[src][q][k];
      return;
    }
    const long long zp = (long long)halo_wrap(p, G.nz) * G.ny;  // periodic ghost planes wrap
    for (int k = tid; k < UX * UY; k += NT) {
      int ux = k % UX, uy = k / UX;
      int hx = ux + 1, hy = uy + (D3 ? 1 : 0);
      const int sc = (p + 10) % 5;
      const int cidx = hy * MX + hx;
      Real lap[3] = {0, 0, 0};
      Real cen[3] = {smom[sc][0][cidx], smom[sc][1][cidx], smom[sc][2][cidx]};
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const int s = (p + L::cz(i) + 10) % 5;
        const int nb = (hy + L::cy(i)) * MX + hx + L::cx(i);
        const Real w = Real(L::w(i));
#pragma unroll
        for (int q = 0; q < 3; ++q) lap[q] += w * (smom[s][q][nb] - cen[q]);
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) lap[q] *= Real(6);  // 2/cs^2
      int gx = halo_wrap(x0 - 1 + ux, G.nx);
      int gy = D3 ? halo_wrap(y0 - 1 + uy, G.ny) : 0;
      Real Iv = a.I[(zp + gy) * G.nx + gx];
      Real mr, mp, ms;
      chem_potentials<Real>(a.fe, cen[0], cen[1], cen[2], lap[0], lap[1], lap[2], Iv, mr, mp, ms);
      {
        // gradients of rho - 1, phi, psi (radius 1, isotropic stencil)
        Real gr[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          const int s = (p + L::cz(i) + 10) % 5;
          const int nb = (hy + L::cy(i)) * MX + hx + L::cx(i);
          const Real w = Real(L::w(i)) * Real(3);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const Real v = w * smom[s][q][nb];
            if (L::cx(i)) gr[q][0] += L::cx(i) > 0 ? v : -v;
            if (L::cy(i)) gr[q][1] += L::cy(i) > 0 ? v : -v;
            if (L::cz(i)) gr[q][2] += L::cz(i) > 0 ? v : -v;
          }
        }
        Real pt[6];
        pressure_tensor<Real>(a.fe, cen[0], cen[1], cen[2], lap, gr, pt);
#pragma unroll
        for (int q = 0; q < 6; ++q) smu[slot][q][k] = pt[q];
        smu[slot][6][k] = a.fe.kc * (cen[2] - Iv);
        smu[slot][MUP][k] = mp;
        smu[slot][MUS][k] = ms;
      }
    }
  };

  auto collide = [&](int zz) {
    if (!active) return;
    const Nbr<L> nb(G, x, y, zz);
    const int n = nb.self;
    const int sm5 = (zz + 10) % 5;
    const int mc = (ty + HY) * MX + tx + 2;
    const Real drho_c = smom[sm5][0][mc], phi = smom[sm5][1][mc], psi = smom[sm5][2][mc];
    const Real rho = Real(1) + drho_c;
    // gradients of the potentials' ring entries (radius 1, isotropic
    // stencil; the 1/cs^2 is applied below)
    constexpr int NG = 7;
    Real gm[NG][3];
#pragma unroll
    for (int q = 0; q < NG; ++q) gm[q][0] = gm[q][1] = gm[q][2] = Real(0);
    const int ux = tx + 1, uy = ty + (D3 ? 1 : 0);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const int s = (zz + L::cz(i) + 9) % 3;
      const int nbi = (uy + L::cy(i)) * UX + ux + L::cx(i);
      const Real w = Real(L::w(i));
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const Real v = w * smu[s][q][nbi];
        if (L::cx(i)) gm[q][0] += L::cx(i) > 0 ? v : -v;
        if (L::cy(i)) gm[q][1] += L::cy(i) > 0 ? v : -v;
        if (L::cz(i)) gm[q][2] += L::cz(i) > 0 ? v : -v;
      }
    }
    const int sc = (zz + 9) % 3;
    const int cc = uy * UX + ux;
    const Real mup = smu[sc][MUP][cc], mus = smu[sc][MUS][cc];
    // force (+ f_IB inside the bricks the markers spread into):
    //  f_FE = -div p' - psi grad(kappa_c (psi - I)), p' the tensor of App. A
    //  without rho cs^2 (whose divergence cancels grad rho cs^2)
    const bool ib = a.bflag[((zz >> 2) * a.nby + (y >> 2)) * a.nbx + (x >> 2)] != 0;
    Real F[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      // row d of the symmetric tensor: (xx, xy, xz), (xy, yy, yz), (xz, yz, zz)
      const int r0 = d == 0 ? 0 : (d == 1 ? 3 : 4), r1 = d == 0 ? 3 : (d == 1 ? 1 : 5),
                r2 = d == 0 ? 4 : (d == 1 ? 5 : 2);
      F[d] = -Real(3) * (gm[r0][0] + gm[r1][1] + gm[r2][2] + psi * gm[6][d]);
      if (ib) F[d] += a.fib[d * G.P32 + n];
    }
    if (!D3) F[1] = 0;
    collide_pops<L, MODE>(a, nb, phi, psi, rho, F, mup, mus);
    if (ib)
#pragma unroll
      for (int d = 0; d < 3; ++d) a.ftot[d * G.P32 + n] = F[d];
    if (!(rho == rho) || !(phi == phi) || !(psi == psi)) atomicOr(a.status, (unsigned)ST_NAN);
  };

  // prologue: moments z0-2 .. z0+1, potentials z0 then z0-1 (a wall ghost
  // copies its neighbour, so the real plane comes first)
  for (int p = z0 - 2; p <= z0 + 1; ++p) load_mom(p);
  __syncthreads();
  compute_mu(z0);
  __syncthreads();
  compute_mu(z0 - 1);
  __syncthreads();
  for (int zz = z0; zz < z1; ++zz) {
    load_mom(zz + 2);
    __syncthreads();
    compute_mu(zz + 1);
    __syncthreads();
    collide(zz);
    __syncthreads();
  }
}

// The collide with the potential force.  T1 (forms 5 and 6; tau = tau_phi =
// tau_psi = 1, exact difference method): every post-collision population is
// an equilibrium of the cell's moments, so nothing is pulled and what is
// stored is the 12 values those equilibria are made of (see EqCell).
// Otherwise the cell's populations are pulled, collided and stored.
//
// A TX x TY tile of columns walks a.zc planes.  The moments of a plane (one
// vector (rho - 1, phi, psi, j_x) per cell, tile plus a halo of 2) are copied
// asynchronously two planes ahead into a ring of three shared-memory slots.
// Per plane and one barrier:
//  * the potentials: each column of the tile plus a halo of 1 reads the 9
//    (2D: 3) moments around it in plane q, forms the in-plane sums of
//    differences, finishes the Laplacian of plane q - 1 (whose own and lower
//    parts are in registers) and stores that plane's potentials in one of two
//    slots;
//  * the force: each cell's column reads the 9 potentials around it in plane
//    r = q - 2, finishes the force of plane r - 1, goes on with that of plane
//    r and starts that of plane r + 1;
//  * plane r - 1 is collided and stored.
// So a plane of either ring is read 9 times per cell, not 19, and the sums
// of a stencil that lie in one plane are formed once for the three planes
// that use them.  Laplacians are sums of differences from the centre of
// their own plane, so FP32 keeps their low bits.
template <class L, int MODE, int TX, int TY, bool T1>
__device__ __forceinline__ void collide_body_of(const LBArgs<MODE>& a, const Blk& blk) {
  using Real = typename Prec<MODE>::Real;
  constexpr bool D3 = L::DIM == 3;
  constexpr int HY = D3 ? 2 : 0;
  constexpr int MX = TX + 4, MY = TY + 2 * HY, MC = MX * MY;
  constexpr int UX = TX + 2, UY = TY + (D3 ? 2 : 0), UC = UX * UY;
  constexpr int NT = TX * TY, NL = (MC + NT - 1) / NT, NH = UC - NT;
  static_assert(NH <= NT, "one halo column of the potentials per thread");
  // stencil weights: lap = 6 sum w (a_n - a), axis 6/18 (2D 6/9), edge 6/36;
  // F = -3 sum w c (...) with the edge weight 3/36 taken out of the sum
  constexpr double WA6 = D3 ? 1.0 / 3 : 2.0 / 3, WE6 = 1.0 / 6, AE = D3 ? 2 : 4;
  __shared__ R4<Real> sp[3][MC];  // (rho - 1, phi, psi, j_x)
  __shared__ R4<Real> su[2][UC];  // (mu~rho, mu_phi, mu_psi', -)

  const Geo G = a.G;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int x0 = blk.x * TX, y0 = blk.y * TY;
  const int z0 = blk.z * a.zc, z1 = min(z0 + a.zc, G.nz);
  const int x = x0 + tx, y = y0 + ty;
  const bool active = x < G.nx && y < G.ny;
  const int nxy = G.nx * G.ny;

  int coff[NL];  // in-plane offsets of the cells this thread copies
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    const int k = tid + j * NT, gx = halo_wrap(x0 - 2 + k % MX, G.nx);
    coff[j] = (D3 ? halo_wrap(y0 - HY + k / MX, G.ny) * G.nx : 0) + gx;
  }
  auto issue = [&](int p, int slot) {
    const R4<Real>* src = a.p4 + (long long)ring_plane(G, p) * nxy;
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const int k = tid + j * NT;
      if (k < MC) cp_async_r4(&sp[slot][k], src + coff[j]);
    }
  };

  // The columns whose potentials this thread computes: its own cell's and,
  // for the first NH threads, one of the halo (the two rows above and below
  // the tile, then the two columns beside it).
  struct Col {
    int m, u, off;       // its cell in a moments slot and in a potentials slot; in-plane offset
    Real P[3], S[3];     // Laplacian so far of plane q - 1; in-plane sums there
    R4<Real> c;          // centre moments of plane q - 1
    Real I;              // membrane profile of plane q - 1
  };
  auto column = [&](int ux, int uy) {
    Col o;
    o.m = (uy + (D3 ? 1 : 0)) * MX + ux + 1;
    o.u = uy * UX + ux;
    o.off = (D3 ? halo_wrap(y0 - 1 + uy, G.ny) * G.nx : 0) + halo_wrap(x0 - 1 + ux, G.nx);
    o.c = R4<Real>{0, 0, 0, 0};
    o.I = 0;
    for (int k = 0; k < 3; ++k) o.P[k] = o.S[k] = 0;
    return o;
  };
  Col own = column(tx + 1, D3 ? ty + 1 : 0), ext;
  const bool has_ext = tid < NH;
  {
    const int k = tid - 2 * UX;
    if (!D3) ext = column(tid == 0 ? 0 : UX - 1, 0);
    else if (tid < 2 * UX) ext = column(tid % UX, tid < UX ? 0 : UY - 1);
    else ext = column(k & 1 ? UX - 1 : 0, 1 + k / 2);
  }
  // plane q of a column: finishes plane q - 1
  auto potentials = [&](Col& o, const R4<Real>* s, R4<Real>* out, int iplane) {
    const R4<Real> c = s[o.m], xm = s[o.m - 1], xp = s[o.m + 1];
    Real s4[3] = {(xm.x - c.x) + (xp.x - c.x), (xm.y - c.y) + (xp.y - c.y), (xm.z - c.z) + (xp.z - c.z)};
    Real sd[3] = {0, 0, 0};
    if constexpr (D3) {
      const R4<Real> ym = s[o.m - MX], yp = s[o.m + MX];
      s4[0] += (ym.x - c.x) + (yp.x - c.x);
      s4[1] += (ym.y - c.y) + (yp.y - c.y);
      s4[2] += (ym.z - c.z) + (yp.z - c.z);
      const R4<Real> a0 = s[o.m - MX - 1], a1 = s[o.m - MX + 1], a2 = s[o.m + MX - 1], a3 = s[o.m + MX + 1];
      sd[0] = ((a0.x - c.x) + (a1.x - c.x)) + ((a2.x - c.x) + (a3.x - c.x));
      sd[1] = ((a0.y - c.y) + (a1.y - c.y)) + ((a2.y - c.y) + (a3.y - c.y));
      sd[2] = ((a0.z - c.z) + (a1.z - c.z)) + ((a2.z - c.z) + (a3.z - c.z));
    }
    // lap(q - 1) = [own plane and below] + (c - c') + S(q) / 6
    const Real d[3] = {c.x - o.c.x, c.y - o.c.y, c.z - o.c.z};
    Real lap[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lap[k] = rfma(Real(WE6), s4[k], o.P[k]) + d[k];
      o.P[k] = rfma(Real(WA6), s4[k], rfma(Real(WE6), sd[k] + o.S[k], -d[k]));
      o.S[k] = s4[k];
    }
    Real mr, mp, ms;
    chem_potentials<Real>(a.fe, o.c.x, o.c.y, o.c.z, lap[0], lap[1], lap[2], o.I, mr, mp, ms);
    out[o.u] = R4<Real>{mr, mp, ms, Real(0)};
    o.c = c;
    o.I = a.I[iplane + o.off];  // (used one plane on)
  };

  // force sums (times -12) of planes r - 1 and r, and what they need: the
  // centre moments of planes r - 1 and r, the centre potentials of planes
  // r - 1 and r - 2 (their difference from plane r's is taken at the end: the
  // sums along z then hold in-plane differences only, at their own scale)
  Real A[3] = {0, 0, 0}, B[3] = {0, 0, 0};
  R4<Real> c1 = {0, 0, 0, 0}, c2 = {0, 0, 0, 0};
  Real h1[3] = {0, 0, 0}, h2[3] = {0, 0, 0};
  // (j_y, j_z) and the brick flag of the plane collided next
  R2<Real> jn;
  jn.x = jn.y = 0;
  bool ibn = false;
  auto ahead = [&](int p) {
    if (!active) return;
    if (T1) jn = a.j2[(p * G.ny + y) * G.nx + x];
    ibn = a.bflag[((p >> 2) * a.nby + (y >> 2)) * a.nbx + (x >> 2)] != 0;
  };

  auto collide = [&](int zz, const Real* F12, const R4<Real>& c) {
    const int n = (zz * G.ny + y) * G.nx + x;
    const Real drho = c.x, phi = c.y, psi = c.z, rho = Real(1) + drho;
    const Real j[3] = {c.w, jn.x, jn.y};
    Real F[3], v[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      F[d] = rmul(Real(-1.0 / 12), F12[d]);
      if (ibn) F[d] = radd(F[d], a.fib[d * G.P32 + n]);
    }
    if (!D3) F[1] = 0;
    if (ibn)
#pragma unroll
      for (int d = 0; d < 3; ++d) a.ftot[d * G.P32 + n] = F[d];
    if (!(rho == rho) || !(phi == phi) || !(psi == psi)) atomicOr(a.status, (unsigned)ST_NAN);
    if constexpr (!T1) {
      collide_pops<L, MODE>(a, Nbr<L>(G, x, y, zz), phi, psi, rho, F, h1[1], h1[2]);
      return;
    }
    const Real irho = rcp_rn(rho);
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = rmul(rfma(Real(0.5), F[d], j[d]), irho);
    R4<Real>* M = a.M + n;
    M[M_F * G.P32] = R4<Real>{drho, radd(j[0], F[0]), radd(j[1], F[1]), radd(j[2], F[2])};
    M[M_ORD * G.P32] = R4<Real>{phi, rmul(Real(3), rmul(a.gphi, h1[1])), psi, rmul(Real(3), rmul(a.gpsi, h1[2]))};
    M[M_V * G.P32] = R4<Real>{v[0], v[1], v[2], irho};
  };

  issue(z0 - 2, 0);
  cp_async_commit();
  issue(z0 - 1, 1);
  cp_async_commit();
  int slot = 0;  // of plane q
  for (int q = z0 - 2; q <= z1 + 2; ++q) {
    cp_async_wait<1>();
    __syncthreads();
    // plane q + 2 takes the slot of plane q - 1, which every thread has left
    if (q + 2 <= z1 + 1) issue(q + 2, slot == 0 ? 2 : slot - 1);
    cp_async_commit();
    const int r = q - 2;
    // (the potentials beyond a wall mirror those next to it: mu(-1) = mu(0),
    // whose part is added to plane 0 with plane 0's own, and mu(nz) = mu(nz - 1))
    if (r >= z0 - 1 && !(G.wall && r < 0)) {
      const R4<Real>* s = su[(G.wall ? min(r, G.nz - 1) : r) & 1];
      const int o = own.u;
      const R4<Real> c = s[o], xm = s[o - 1], xp = s[o + 1];
      const Real* cv = &c.x;
      const Real gx[3] = {xp.x - xm.x, xp.y - xm.y, xp.z - xm.z};
      Real S[3] = {(xm.x - c.x) + (xp.x - c.x), (xm.y - c.y) + (xp.y - c.y), (xm.z - c.z) + (xp.z - c.z)};
      Real gy[3] = {0, 0, 0}, mx[3], my[3] = {0, 0, 0};
      Real gxd[3] = {0, 0, 0};
      if constexpr (D3) {
        const R4<Real> ym = s[o - UX], yp = s[o + UX];
        const R4<Real> mm = s[o - UX - 1], pm = s[o - UX + 1], mp = s[o + UX - 1], pp = s[o + UX + 1];
        const Real *ymv = &ym.x, *ypv = &yp.x, *mmv = &mm.x, *pmv = &pm.x, *mpv = &mp.x, *ppv = &pp.x;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          gy[k] = ypv[k] - ymv[k];
          S[k] += (ymv[k] - cv[k]) + (ypv[k] - cv[k]);
          const Real d0 = ppv[k] - mmv[k], d1 = pmv[k] - mpv[k];
          gxd[k] = d0 + d1;
          my[k] = rfma(Real(AE), gy[k], d0 - d1);
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) mx[k] = rfma(Real(AE), gx[k], gxd[k]);
      // weights rho, phi, psi of planes r - 1, r and r + 1 (the centre of
      // plane r + 1 = q - 1 is the one the potentials hold)
      const Real w1[3] = {Real(1) + c1.x, c1.y, c1.z}, w2[3] = {Real(1) + c2.x, c2.y, c2.z};
      const Real w3[3] = {Real(1) + own.c.x, own.c.y, own.c.z};
      Real N[3] = {0, 0, 0};
      if (G.wall && r == 0) {  // the ghost plane below
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          B[0] = rfma(w2[k], gx[k], B[0]);
          if (D3) B[1] = rfma(w2[k], gy[k], B[1]);
          B[2] = rfma(-w2[k], S[k], B[2]);
          h1[k] = cv[k];
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        A[0] = rfma(w1[k], gx[k], A[0]);
        if (D3) A[1] = rfma(w1[k], gy[k], A[1]);
        A[2] = rfma(w1[k], rfma(Real(6), cv[k] - h2[k], S[k]), A[2]);
        B[0] = rfma(w2[k], mx[k], B[0]);
        if (D3) B[1] = rfma(w2[k], my[k], B[1]);
        N[0] = rfma(w3[k], gx[k], N[0]);
        if (D3) N[1] = rfma(w3[k], gy[k], N[1]);
        N[2] = rfma(-w3[k], S[k], N[2]);
      }
      if (r > z0 && active) collide(r - 1, A, c1);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        A[d] = B[d];
        B[d] = N[d];
        h2[d] = h1[d];
        h1[d] = cv[d];
      }
    }
    if (r >= z0 && r < z1) ahead(r);  // collided next
    c1 = c2;
    c2 = own.c;
    if (q <= z1 + 1) {
      R4<Real>* out = su[(q - 1) & 1];
      const int ip = ring_plane(G, q) * nxy;
      potentials(own, sp[slot], out, ip);
      if (has_ext) potentials(ext, sp[slot], out, ip);
    }
    slot = slot == 2 ? 0 : slot + 1;
  }
  cp_async_wait<0>();
}

// The collide of a form.
template <class L, int MODE, int TX, int TY, int FORM>
__device__ __forceinline__ void collide_body(const LBArgs<MODE>& a, const Blk& blk) {
  if constexpr (FORM == 7)
    collide_pt_body<L, MODE, TX, TY>(a, blk);
  else
    collide_body_of<L, MODE, TX, TY, form_t1<FORM>()>(a, blk);
}
// Forms of the collide: threads per SM the register budget is set for (1, the
// general collide: 512; the tau = 1 collide at 5: 640 and 6: 768; the
// pressure tensor at 7: 640).  The general collide holds its cell's
// populations, so fewer threads with their values in registers win: step of
// 128^3 FP32 0.360 ms on 32 x 4 tiles, against 0.394 at 640, 0.422 at 768 and
// over 0.48 at 896 and 1024 (spills).  The tau = 1 collide holds about 90
// values per thread: at 768 threads per SM it spilled 52 bytes.
template <int FORM> constexpr int collide_threads() { return FORM == 1 ? 512 : (FORM == 6 ? 768 : 640); }
// threads of a collide block: one per cell of the TX x TY tile
template <int FORM, int TX, int TY> constexpr int collide_block() { return TX * TY; }

// blocks per SM of a collide; double precision takes twice the registers
template <int MODE, int FORM, int TX, int TY> constexpr int collide_minb() {
  constexpr int n = collide_threads<FORM>() / (MODE == TLB_F64 ? 2 : 1) / collide_block<FORM, TX, TY>();
  return n > 0 ? n : 1;
}

template <class L, int MODE, int TX, int TY, int FORM>
__global__ void __launch_bounds__(collide_block<FORM, TX, TY>(), collide_minb<MODE, FORM, TX, TY>())
    k_collide(const __grid_constant__ LBArgs<MODE> a) {
  collide_body<L, MODE, TX, TY, FORM>(a, hw_blk());
}

// Calls fn(tile x, tile y, form) with the variant's compile-time values
// (3D tiles 32x4, 32x8, 64x4; 2D rows of 32, 64, 128): variants 0..12 the
// three tiles of the general collide in turn, all in form 1 (each of the three
// has several numbers; see variant_again); 13..18 the tiles in the tau = 1
// forms 5 and 6; 19..21 in form 7, the general collide with the
// pressure-tensor force.
template <int V> using CIdx = std::integral_constant<int, V>;
template <class L, class Fn>
__host__ tlb_status collide_variant(int v, Fn&& fn) {
  constexpr bool D3 = L::DIM == 3;
  constexpr int X1 = D3 ? 32 : 64, Y1 = D3 ? 8 : 1, X2 = D3 ? 64 : 128, Y0 = D3 ? 4 : 1;
  switch (v) {
    case 1: case 4: case 7: case 10: return fn(CIdx<X1>{}, CIdx<Y1>{}, CIdx<1>{});
    case 2: case 5: case 8: case 11: return fn(CIdx<X2>{}, CIdx<Y0>{}, CIdx<1>{});
    case 13: return fn(CIdx<32>{}, CIdx<Y0>{}, CIdx<5>{});
    case 14: return fn(CIdx<X1>{}, CIdx<Y1>{}, CIdx<5>{});
    case 15: return fn(CIdx<X2>{}, CIdx<Y0>{}, CIdx<5>{});
    case 16: return fn(CIdx<32>{}, CIdx<Y0>{}, CIdx<6>{});
    case 17: return fn(CIdx<X1>{}, CIdx<Y1>{}, CIdx<6>{});
    case 18: return fn(CIdx<X2>{}, CIdx<Y0>{}, CIdx<6>{});
    case 19: return fn(CIdx<32>{}, CIdx<Y0>{}, CIdx<7>{});
    case 20: return fn(CIdx<X1>{}, CIdx<Y1>{}, CIdx<7>{});
    case 21: return fn(CIdx<X2>{}, CIdx<Y0>{}, CIdx<7>{});
    // 22..27 name the three tiles again (they were two-cell forms of the
    // tau = 1 collide), 28..31 the 32 x 16 tiles (3D)
    case 22: return fn(CIdx<32>{}, CIdx<Y0>{}, CIdx<5>{});
    case 23: return fn(CIdx<X1>{}, CIdx<Y1>{}, CIdx<5>{});
    case 24: return fn(CIdx<X2>{}, CIdx<Y0>{}, CIdx<5>{});
    case 25: return fn(CIdx<32>{}, CIdx<Y0>{}, CIdx<6>{});
    case 26: return fn(CIdx<X1>{}, CIdx<Y1>{}, CIdx<6>{});
    case 27: return fn(CIdx<X2>{}, CIdx<Y0>{}, CIdx<6>{});
    case 28:
    case 30: return fn(CIdx<32>{}, CIdx<D3 ? 16 : 1>{}, CIdx<5>{});
    case 29:
    case 31: return fn(CIdx<32>{}, CIdx<D3 ? 16 : 1>{}, CIdx<6>{});
    default: return fn(CIdx<32>{}, CIdx<Y0>{}, CIdx<1>{});  // 0, 3, 6, 9, 12
  }
}

// ------------------------------------------------------------- init & I/O
// Chemical potentials from fields in global memory (used at initialisation);
// rho holds rho - 1.
template <class L, int MODE>
__global__ void k_mu_global(Geo G, FEParams<typename Prec<MODE>::Real> fe, const typename Prec<MODE>::Real* rho,
                            const typename Prec<MODE>::Real* phi, const typename Prec<MODE>::Real* psi,
                            const typename Prec<MODE>::Real* I, typename Prec<MODE>::Real* mu) {
  using Real = typename Prec<MODE>::Real;
  long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= G.N) return;
  int x, y, z;
  cell_xyz(G, n, x, y, z);
  const Real* F[3] = {rho, phi, psi};
  Real lap[3] = {0, 0, 0};
  for (int i = 1; i < L::Q; ++i) {
    int sx = wrapc(x + L::cx(i), G.nx), sy = wrapc(y + L::cy(i), G.ny);
    int sz = z + L::cz(i);
    sz = G.wall ? min(max(sz, 0), G.nz - 1) : wrapc(sz, G.nz);
    long long c = ((long long)sz * G.ny + sy) * G.nx + sx;
    for (int q = 0; q < 3; ++q) lap[q] += Real(L::w(i)) * (F[q][c] - F[q][n]);
  }
  Real mr, mp, ms;
  chem_potentials<Real>(fe, rho[n], phi[n], psi[n], 6 * lap[0], 6 * lap[1], 6 * lap[2], I[n], mr, mp, ms);
  mu[n] = mr;
  mu[G.P + n] = mp;
  mu[2 * G.P + n] = ms;
}

// Equilibrium populations (eq. EDF) of the fields (rho holds rho - 1),
// stored post-collision:
// the value of direction i at cell y is the equilibrium f_i at y + c_i (or,
// across a wall, f_{opp(i)} at y), which the next pull brings back to place.
// p4 not NULL: phi and psi there too, for readers of the moment field.
template <class L, int MODE>
__global__ void k_init_eq(Geo G, const typename Prec<MODE>::Real* rho, const typename Prec<MODE>::Real* phi,
                          const typename Prec<MODE>::Real* psi, const typename Prec<MODE>::Real* u,
                          const typename Prec<MODE>::Real* mu, typename Prec<MODE>::Real gphi,
                          typename Prec<MODE>::Real gpsi, typename Prec<MODE>::Store* lo,
                          typename Prec<MODE>::Rest* rest, R4<typename Prec<MODE>::Real>* p4) {
  using Real = typename Prec<MODE>::Real;
  using Store = typename Prec<MODE>::Store;
  using Rest = typename Prec<MODE>::Rest;
  long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= G.N) return;
  if (p4) p4[n] = R4<Real>{rho[n], phi[n], psi[n], 0};
  int x, y, z;
  cell_xyz(G, n, x, y, z);
  for (int i = 0; i < L::Q; ++i) {
    int tz = z + L::cz(i);
    long long src;
    int ii = i;
    if (G.wall && (tz < 0 || tz >= G.nz)) {
      src = n;
      ii = L::opp(i);
    } else {
      src = ((long long)wrapc(tz, G.nz) * G.ny + wrapc(y + L::cy(i), G.ny)) * G.nx + wrapc(x + L::cx(i), G.nx);
    }
    Real dr = rho[src], p = phi[src], s = psi[src];
    Real r = Real(1) + dr;
    Real uv[3] = {u[src], u[G.P + src], u[2 * G.P + src]};
    Real uu = uv[0] * uv[0] + uv[1] * uv[1] + uv[2] * uv[2];
    Real cu = L::cx(ii) * uv[0] + L::cy(ii) * uv[1] + L::cz(ii) * uv[2];
    Real w = Real(L::w(ii)), w0 = Real(L::w(0));
    Real pv = eq_poly(cu, uu);
    lo[(long long)plane_f<L>(i) * G.P + n] = from_real<Store>(w * (dr + r * pv));
    Real mp = mu[G.P + src], ms = mu[2 * G.P + src];
    if (ii == 0) {
      // rest populations are stored in their own planes (direction 0 maps to itself)
      rest[n] = from_real<Rest>(p - Real(3) * gphi * mp * (Real(1) - w0) - Real(1.5) * w0 * p * uu);
      rest[G.P + n] = from_real<Rest>(s - Real(3) * gpsi * ms * (Real(1) - w0) - Real(1.5) * w0 * s * uu);
    } else {
      lo[(long long)plane_g<L>(i) * G.P + n] = from_real<Store>(w * (Real(3) * gphi * mp + p * pv));
      lo[(long long)plane_h<L>(i) * G.P + n] = from_real<Store>(w * (Real(3) * gpsi * ms + s * pv));
    }
  }
}

// Fields of the streamed populations for read-back: rho, phi, psi, u.
// Working-precision copy of a field as doubles (read-out).
template <class Real>
__global__ void k_to_double(const Real* src, long long n, double* dst) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = (double)src[i];
}

// Initial fields from the caller's compositions C = [3][N] (FP64 sums, then
// the working precision): rho - 1 = C1 + C2 + C3 - 1, phi = C1 - C2, psi =
// C3; or, without C, the default state: rho = 1, psi = I, phi = (1 - I)(2 s - 1)
// with the flat interface s(z) = (1 + tanh((z - z0)/(2 alpha)))/2 (s = 0
// when z0 < 0).  The velocity ([3][N], or the uniform u0) goes to uf, 2D
// fields internally as (x, 0, y).
template <class Real>
__global__ void k_init_fields(Geo G, int dim, const double* C, const double* u, double u0x, double u0y,
                              double u0z, double alpha, double z0, const Real* I, Real* rho, Real* phi,
                              Real* psi, Real* uf) {
  const long long N = G.N, P = G.P;
  long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  if (C) {
    rho[n] = (Real)(C[n] + C[N + n] + C[2 * N + n] - 1.0);
    phi[n] = (Real)(C[n] - C[N + n]);
    psi[n] = (Real)C[2 * N + n];
  } else {
    const long long z = n / ((long long)G.nx * G.ny);  // last axis (2D: y)
    double sv = 0.5 * (1.0 + tanh((z - z0) / (2.0 * alpha)));
    if (z0 < 0) sv = 0.0;
    const double ps = (double)I[n];
    rho[n] = (Real)0.0;
    phi[n] = (Real)((1.0 - ps) * (2.0 * sv - 1.0));
    psi[n] = (Real)ps;
  }
  const double v[3] = {u ? u[n] : u0x, u ? u[N + n] : u0y, u ? u[2 * N + n] : u0z};
  if (dim == 2) {
    uf[n] = (Real)v[0];
    uf[P + n] = 0;
    uf[2 * P + n] = (Real)v[1];
  } else {
    for (int d = 0; d < 3; ++d) uf[d * P + n] = (Real)v[d];
  }
}

template <class L, int MODE>
__global__ void k_fields(Geo G, const typename Prec<MODE>::Store* lo, const typename Prec<MODE>::Rest* rest,
                         int field, double* out /* [N], [3][N] for the velocity */) {
  using Real = typename Prec<MODE>::Real;
  long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= G.N) return;
  int x, y, z;
  cell_xyz(G, n, x, y, z);
  Pull<L, MODE> p;
  p.load(lo, rest, G, x, y, z);
  CellMoments<Real> m = p.moments();
  const double rho = 1.0 + (double)m.drho, phi = (double)m.phi, psi = (double)m.psi;
  switch (field) {
    case TLB_FIELD_RHO: out[n] = rho; break;
    case TLB_FIELD_PHI: out[n] = phi; break;
    case TLB_FIELD_PSI: out[n] = psi; break;
    case TLB_FIELD_C1: out[n] = 0.5 * (rho + phi - psi); break;
    case TLB_FIELD_C2: out[n] = 0.5 * (rho - phi - psi); break;
    case TLB_FIELD_C3: out[n] = psi; break;
    default:  // velocity; 2D fields are internal (x, 0, y)
      if (L::DIM == 2) {
        out[n] = (double)m.j[0] / rho;
        out[G.N + n] = (double)m.j[2] / rho;
        out[2 * G.N + n] = 0.0;
      } else {
        for (int d = 0; d < 3; ++d) out[d * G.N + n] = (double)m.j[d] / rho;
      }
  }
}

// ------------------------------------------------------------ residual
// Reference state of the equilibrium residual and the slots its maxima are
// folded into.
struct ResPtrs {
  double* snap;             // [2][P] phi, psi at the reference step
  double* xsnap;            // [nn][3] marker positions at the reference step
  unsigned long long* res;  // [3] max |change| of phi, psi, X (bit patterns)
};

// Largest change since the reference step of phi and psi (FP64 sums of the
// streamed populations) over the cells, then of the marker positions over
// the markers (virtual blocks past the cells); the reference is replaced by
// the current values.  Maxima of non-negative doubles are order independent:
// they are folded with integer atomicMax on the bit patterns, NaN mapped to
// +inf so that a diverged run never reads as converged.
template <class L, int MODE>
__device__ __forceinline__ void residual_body(const Geo& G, const typename Prec<MODE>::Store* lo,
                                              const typename Prec<MODE>::Rest* rest, const double* X, int nn,
                                              const ResPtrs& r, const Blk& blk) {
  const long long ncb = (G.N + blockDim.x - 1) / blockDim.x;
  double m[3] = {0, 0, 0};
  if (blk.x < ncb) {
    const long long n = (long long)blk.x * blockDim.x + threadIdx.x;
    if (n < G.N) {
      int x, y, z;
      cell_xyz(G, n, x, y, z);
      Pull<L, MODE> p;
      p.load(lo, rest, G, x, y, z);
      double ph = 0, ps = 0;
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        ph += (double)p.g[i];
        ps += (double)p.h[i];
      }
      m[0] = fabs(ph - r.snap[n]);
      m[1] = fabs(ps - r.snap[G.P + n]);
      r.snap[n] = ph;
      r.snap[G.P + n] = ps;
    }
  } else {
    const long long l = (long long)(blk.x - ncb) * blockDim.x + threadIdx.x;
    if (l < nn)
      for (int d = 0; d < 3; ++d) {
        m[2] = fmax(m[2], fabs(X[3 * l + d] - r.xsnap[3 * l + d]));
        if (!(X[3 * l + d] == X[3 * l + d])) m[2] = __longlong_as_double(0x7FF0000000000000ll);
        r.xsnap[3 * l + d] = X[3 * l + d];
      }
  }
  for (int q = 0; q < 3; ++q) {
    double v = m[q];
    if (!(v == v)) v = __longlong_as_double(0x7FF0000000000000ll);
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0 && v > 0) atomicMax(r.res + q, (unsigned long long)__double_as_longlong(v));
  }
}

template <class L, int MODE>
__global__ void k_residual(Geo G, const typename Prec<MODE>::Store* lo, const typename Prec<MODE>::Rest* rest,
                           const double* X, int nn, ResPtrs r) {
  residual_body<L, MODE>(G, lo, rest, X, nn, r, hw_blk());
}

// FP64 totals: per-block partial sums of rho (as 1 + sum of deviations),
// phi and psi over a fixed cell partition, combined in fixed order by
// k_reduce_partials, so the result does not depend on scheduling.
template <class L, int MODE>
__global__ void __launch_bounds__(256) k_mass_partials(Geo G, const typename Prec<MODE>::Store* lo,
                                                       const typename Prec<MODE>::Rest* rest, double* part) {
  __shared__ double sm[3][256];
  double acc[3] = {0, 0, 0};
  for (long long n = (long long)blockIdx.x * 256 + threadIdx.x; n < G.N; n += (long long)gridDim.x * 256) {
    double r = 1.0, p = to_real(rest[n]), s = to_real(rest[G.P + n]);
    for (int i = 0; i < L::Q; ++i) r += (double)to_real(lo[(long long)plane_f<L>(i) * G.P + n]);
    for (int i = 1; i < L::Q; ++i) {
      p += (double)to_real(lo[(long long)plane_g<L>(i) * G.P + n]);
      s += (double)to_real(lo[(long long)plane_h<L>(i) * G.P + n]);
    }
    acc[0] += r;
    acc[1] += p;
    acc[2] += s;
  }
  for (int q = 0; q < 3; ++q) sm[q][threadIdx.x] = acc[q];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int q = 0; q < 3; ++q) sm[q][threadIdx.x] += sm[q][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 3; ++q) part[q * gridDim.x + blockIdx.x] = sm[q][0];
}

__global__ void k_reduce_partials(const double* part, int nb, int nq, double* out);
