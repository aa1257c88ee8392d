// Templated host driver: builds kernel arguments from the context and
// enqueues the step of the method on the context stream.
#pragma once
#include <math.h>

#include <vector>

#include "tlb_ctx.h"
#include "tlb_ibm.cuh"
#include "tlb_lb.cuh"
#include "tlb_measure.cuh"
#include "tlb_diag.cuh"

template <class L, int MODE>
struct Impl : ImplBase {
  using Real = typename Prec<MODE>::Real;
  using Store = typename Prec<MODE>::Store;
  using Rest = typename Prec<MODE>::Rest;

  // tiles of the rebuilding moments sweep
  static constexpr int RECON_X = L::DIM == 3 ? 32 : 64, RECON_Y = L::DIM == 3 ? 4 : 1;

  static Geo geo(const Ctx* c) {
    Geo g;
    g.nx = c->nx;
    g.ny = c->ny;
    g.nz = c->nz;
    g.wall = c->p.wall_last;
    g.N = c->N;
    g.P = c->P;
    g.P32 = (int)c->P;
    return g;
  }

  // the arrays of the tau = 1 scheme, or none of them
  static void use_t1(Ctx* c, LBArgs<MODE>& a, bool t1) {
    a.p4 = c->packed() ? c->ptr<R4<Real>>(c->L.p4) : nullptr;
    a.j2 = t1 ? c->idle<R2<Real>>(c->L.j2) : nullptr;
    a.M = t1 ? c->idle<R4<Real>>(c->L.M) : nullptr;
    a.pull = c->state_in_pops;
    a.in_M = t1 && c->asks() ? c->ptr<int>(c->L.in_M) : nullptr;
  }
  static void use_t1(Ctx* c, IBArgs<Real>& a, bool t1) {
    a.psi = c->packed() ? &c->ptr<R4<Real>>(c->L.p4)->z : c->ptr<Real>(c->L.psi);
    a.psi_step = c->packed() ? 4 : 1;
    a.M = t1 ? c->idle<R4<Real>>(c->L.M) : nullptr;
  }

  static LBArgs<MODE> lbargs(Ctx* c, int src) {
    LBArgs<MODE> a;
    a.G = geo(c);
    a.lo_src = c->ptr<Store>(c->L.lo[src]);
    a.rest_src = c->ptr<Rest>(c->L.rest[src]);
    a.lo_dst = c->ptr<Store>(c->L.lo[1 - src]);
    a.rest_dst = c->ptr<Rest>(c->L.rest[1 - src]);
    a.rho = c->ptr<Real>(c->L.rho);
    a.phi = c->ptr<Real>(c->L.phi);
    a.psi = c->ptr<Real>(c->L.psi);
    use_t1(c, a, variant_t1(c->tile_variant));
    a.I = c->ptr<Real>(c->L.I);
    a.fib = c->ptr<Real>(c->L.fib);
    a.ftot = c->ptr<Real>(c->L.ftot);
    a.bflag = c->ptr<unsigned char>(c->L.bflag);
    a.nbx = c->nbx;
    a.nby = c->nby;
    a.fe.k1 = (Real)c->p.kappa[0];
    a.fe.k2 = (Real)c->p.kappa[1];
    a.fe.k3 = (Real)c->p.kappa[2];
    a.fe.kc = (Real)c->p.kappa_c;
    a.fe.a2 = (Real)(c->p.alpha * c->p.alpha);
    a.om = (Real)(1.0 / c->p.tau);
    a.om_phi = (Real)(1.0 / c->p.tau_phi);
    a.om_psi = (Real)(1.0 / c->p.tau_psi);
    a.gphi = (Real)c->p.gamma_phi;
    a.gpsi = (Real)c->p.gamma_psi;
    a.zc = c->tiles_zc;
    a.zcm = c->recon_zc;
    a.forcing = c->p.forcing;
    a.status = c->ptr<unsigned>(c->L.status);
    return a;
  }

  static IBArgs<Real> ibargs(Ctx* c) {
    IBArgs<Real> a;
    a.G = geo(c);
    a.dim = c->p.dim;
    a.NV = c->NV;
    a.nn = c->nn;
    a.ne = c->ne;
    a.X = c->ptr<double>(c->L.X);
    a.E = c->ptr<int>(c->L.E);
    a.ecap = c->ptr<int>(c->L.ecap);
    a.ncap = c->ptr<int>(c->L.ncap);
    const double* cp = c->ptr<double>(c->L.cap_par);
    a.ks = cp;
    a.kb = cp + c->ncap;
    a.sG = cp + 2 * c->ncap;
    a.sC = cp + 3 * c->ncap;
    a.ds0 = c->ptr<double>(c->L.ds0);
    a.rprev = c->ptr<int>(c->L.rprev);
    a.rnext = c->ptr<int>(c->L.rnext);
    a.A0 = c->ptr<double>(c->L.A0);
    a.G0i = c->ptr<double>(c->L.G0i);
    a.inc_off = c->ptr<int>(c->L.inc_off);
    a.inc = c->ptr<int>(c->L.inc);
    a.adj = c->ptr<int>(c->L.adj);
    a.nedge = c->nedge;
    a.edges = c->ptr<int>(c->L.edges);
    a.en = c->ptr<R4<Real>>(c->L.en);
    a.vn = c->ptr<R4<Real>>(c->L.vn);
    a.nadj = c->ptr<R4<Real>>(c->L.nadj);
    a.wts = c->ptr<Real>(c->L.wts);
    a.erel = c->ptr<R4<Real>>(c->L.erel);
    a.eorg = c->ptr<int4>(c->L.eorg);
    a.ecst = c->ptr<R4<Real>>(c->L.ecst);
    a.xo = c->ptr<int>(c->L.xo);
    a.xr = c->ptr<Real>(c->L.xr);
    a.skc = c->ptr<Real>(c->L.skc);
    a.capr = c->ptr<Real>(c->L.capr);
    a.ncaps = c->ncap;
    a.split = c->scat_split;
    a.ncpl = c->ptr<unsigned long long>(c->L.ncpl);
    a.F = c->ptr<Real>(c->L.F);
    a.box = c->ptr<int>(c->L.box);
    a.boxc = c->ptr<int>(c->L.box) + 6;
    a.key = c->ptr<unsigned long long>(c->L.key);
    a.own = c->ptr<int>(c->L.own);
    a.I = c->ptr<Real>(c->L.I);
    a.dsel = c->ptr<Real>(c->L.dsel);
    use_t1(c, a, variant_t1(c->tile_variant));
    a.fib = c->ptr<Real>(c->L.fib);
    a.ftot = c->ptr<Real>(c->L.ftot);
    a.bflag = c->ptr<unsigned char>(c->L.bflag);
    a.bcnt = c->ptr<int>(c->L.bcnt);
    a.bprev = c->ptr<int>(c->L.bprev);
    a.bcur = c->ptr<int>(c->L.bcur);
    a.boff = c->ptr<int>(c->L.boff);
    a.blist = c->ptr<int>(c->L.blist);
    a.bact = c->ptr<int>(c->L.bact);
    a.ctr = c->ptr<int>(c->L.ctr);
    a.nbx = c->nbx;
    a.nby = c->nby;
    a.nbz = c->nbz;
    a.nbricks = c->nbricks;
    a.alpha = (Real)c->p.alpha;
    a.dc = (Real)c->p.dc;
    a.kc = (Real)c->p.kappa_c;
    a.Iin = (Real)(0.5 * (1.0 + tanh(c->p.dc / (2.0 * c->p.alpha))));
    a.Iout = (Real)(0.5 * (1.0 + tanh(-c->p.dc / (2.0 * c->p.alpha))));
    a.status = c->ptr<unsigned>(c->L.status);
    return a;
  }

  static unsigned blocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

  // Work of a step that depends on the marker positions X(t) only (element
  // and vertex normals and the distance scatter here; elastic forces and the
  // brick binning in ibm_bins).  It runs on the side stream while the
  // moments of the step are computed.
  // With snap the geometry kernel also takes the marker box's snapshot (the
  // advection's accumulator) and resets it; `done` is recorded after it.
  static tlb_status ibm_positions(Ctx* c, IBArgs<Real>& a, cudaStream_t s, bool snap = false,
                                  cudaEvent_t done = nullptr) {
    k_geometry<Real><<<blocks(geometry_threads(c->ne, c->nn), 128), 128, 0, s>>>(a, snap ? 1 : 0);
    TLB_LAUNCHED(c, "k_geometry");
    if (done) TLB_CUDA(cudaEventRecord(done, s));
    constexpr int sw = scatter_warps<Real>();
    const unsigned nvb = (unsigned)a.split * blocks(c->features(), 32 * sw);
    k_dist_scatter<Real><<<std::min(nvb, 4u * (unsigned)c->nsm), 32 * sw, 0, s>>>(a, (int)nvb);
    TLB_LAUNCHED(c, "k_dist_scatter");
    return TLB_OK;
  }

  static unsigned fresh_blocks(const Ctx* c) {
    return std::max(blocks(c->nn, 128), std::min(blocks(c->N, 128), 8u * (unsigned)c->nsm));
  }

  // The step's marker box: recompute the accumulator if the markers were
  // overwritten, copy it to the snapshot every kernel of the step reads, and
  // reset it for the advection of this step.
  static tlb_status snapshot_box(Ctx* c, IBArgs<Real>& a, cudaStream_t s, bool fresh) {
    if (fresh) {
      TLB_CUDA(cudaMemsetAsync(a.box, 0x7F, 6 * sizeof(int), s));
      k_fresh<Real><<<fresh_blocks(c), 128, 0, s>>>(a);
      TLB_LAUNCHED(c, "k_fresh");
    }
    TLB_CUDA(cudaMemcpyAsync((void*)a.boxc, a.box, 6 * sizeof(int), cudaMemcpyDeviceToDevice, s));
    TLB_CUDA(cudaMemsetAsync(a.box, 0x7F, 6 * sizeof(int), s));
    return TLB_OK;
  }

  // The binning of markers into spreading bricks (the bins are consumed and
  // reset by k_spread of the same step) and, once the geometry is done, the
  // elastic forces.
  static tlb_status ibm_bins(Ctx* c, IBArgs<Real>& a, cudaStream_t s, cudaEvent_t geometry) {
    k_brick_count<Real><<<blocks(c->nn, 128), 128, 0, s>>>(a);  // (clears ctr)
    TLB_LAUNCHED(c, "k_brick_count");
    k_brick_compact<Real><<<blocks(c->nbricks, 256), 256, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_brick_compact");
    k_brick_fill<Real><<<blocks(c->nn, 128), 128, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_brick_fill");
    TLB_CUDA(cudaStreamWaitEvent(s, geometry, 0));
    k_node_forces<Real><<<blocks((long long)c->nn * 16, 128), 128, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_node_forces");
    return TLB_OK;
  }

  // Profile I of the band and the coupling sums (needs psi(t)); the rest of
  // the box (column fill).
  static tlb_status launch_band(Ctx* c, IBArgs<Real>& a, cudaStream_t s) {
    // one cell of the marker box per thread, as the markers started
    k_band<Real><<<std::max(1, 2 * c->band_blocks), 128, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_band");
    return TLB_OK;
  }
  static tlb_status launch_fill(Ctx* c, IBArgs<Real>& a, cudaStream_t s) {
    k_fill<Real><<<blocks((long long)c->nx * c->ny * 32, 256), 256, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_fill");
    return TLB_OK;
  }
  static tlb_status ibm_band(Ctx* c, IBArgs<Real>& a, cudaStream_t s) {
    tlb_status st = launch_band(c, a, s);
    return st == TLB_OK ? launch_fill(c, a, s) : st;
  }

  static tlb_status ibm_spread(Ctx* c, IBArgs<Real>& a, cudaStream_t s) {
    constexpr int nt = 64;  // (two bricks at a time)
    k_spread<Real><<<min((int)blocks(c->nbricks, nt / 32), 8 * c->nsm), nt, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_spread");
    return TLB_OK;
  }

  tlb_status init_fields(Ctx* c, const double* C, const double* u) override {
    cudaStream_t s = c->stream;
    const long long N = c->N;
    IBArgs<Real> ia = ibargs(c);
    // membrane profile I(X0) (I_out everywhere when there are no membranes)
    if (c->nn > 0) {
      tlb_status st = snapshot_box(c, ia, s, true);
      if (st == TLB_OK) st = ibm_positions(c, ia, s);
      if (st == TLB_OK) st = ibm_band(c, ia, s);
      if (st != TLB_OK) return st;
      c->box_stale = true;  // the first step recomputes the box of X0
    }
    Real* rho = c->ptr<Real>(c->L.rho);
    Real* phi = c->ptr<Real>(c->L.phi);
    Real* psi = c->ptr<Real>(c->L.psi);
    Real* uf = c->ptr<Real>(c->L.ftot);  // velocity (free before the first step)
    // the caller's arrays go to the other population buffer (free until the
    // first step; at least 48 bytes per cell) and are converted on the device
    double* scratch = c->ptr<double>(c->L.lo[1 - c->cur]);
    const double* Cd = nullptr;
    const double* ud = nullptr;
    if (C) {
      TLB_CUDA(cudaMemcpyAsync(scratch, C, 3 * N * sizeof(double), cudaMemcpyHostToDevice, s));
      Cd = scratch;
    }
    if (u) {
      TLB_CUDA(cudaMemcpyAsync(scratch + 3 * N, u, 3 * N * sizeof(double), cudaMemcpyHostToDevice, s));
      ud = scratch + 3 * N;
    }
    TLB_CUDA(cudaMemsetAsync(c->ptr<char>(c->L.ftot), 0, c->L.ftot.bytes, s));
    k_init_fields<Real><<<blocks(N, 256), 256, 0, s>>>(geo(c), c->p.dim, Cd, ud, c->p.u0[0], c->p.u0[1], c->p.u0[2],
                                                       c->p.alpha, c->p.interface_pos, c->ptr<Real>(c->L.I), rho,
                                                       phi, psi, uf);
    TLB_LAUNCHED(c, "k_init_fields");
    Geo G = geo(c);
    LBArgs<MODE> la = lbargs(c, c->cur);
    Real* mu = c->ptr<Real>(c->L.mu);
    k_mu_global<L, MODE><<<blocks(N, 256), 256, 0, s>>>(G, la.fe, rho, phi, psi, la.I, mu);
    TLB_LAUNCHED(c, "k_mu_global");
    k_init_eq<L, MODE><<<blocks(N, 256), 256, 0, s>>>(G, rho, phi, psi, uf, mu, la.gphi, la.gpsi,
                                                       c->ptr<Store>(c->L.lo[c->cur]),
                                                       c->ptr<Rest>(c->L.rest[c->cur]), la.p4);
    TLB_LAUNCHED(c, "k_init_eq");
    TLB_CUDA(cudaMemsetAsync(c->ptr<char>(c->L.ftot), 0, c->L.ftot.bytes, s));
    // the initial state is the first reference of the equilibrium residual
    // (of these populations: what M held before is not written over them)
    tlb_status rs = pops_written(c);
    if (rs == TLB_OK) rs = residual_launch(c);
    if (rs != TLB_OK) return rs;
    TLB_CUDA(cudaStreamSynchronize(s));
    c->t = 0;
    c->t_snap = 0;
    c->initialised = true;
    return TLB_OK;
  }

  static std::vector<SweepTiles> sweep_tiles(const std::vector<Ctx*>& cs, int tx, int ty) {
    std::vector<SweepTiles> t;
    for (const Ctx* c : cs) t.push_back({(long long)blocks(c->nx, tx) * blocks(c->ny, ty), c->nz});
    return t;
  }
  int collide_chunk(const std::vector<Ctx*>& cs, int variant) override {
    constexpr bool f64 = MODE == TLB_F64;
    int zc = 1;
    collide_variant<L>(variant, [&](auto tx, auto ty, auto fm) {
      constexpr int TX = decltype(tx)::value, TY = decltype(ty)::value, FM = decltype(fm)::value;
      zc = sweep_chunk(sweep_tiles(cs, TX, TY), cs[0]->nsm,
                       collide_cost(collide_minb<MODE, FM, TX, TY>(), TX * TY, f64, form_t1<FM>()));
      return TLB_OK;
    });
    return zc;
  }
  int recon_chunk(const std::vector<Ctx*>& cs, int tx, int ty) override {
    return sweep_chunk(sweep_tiles(cs, tx, ty), cs[0]->nsm, recon_cost(768 / (tx * ty), tx * ty, MODE == TLB_F64));
  }

  tlb_status sync_pops(Ctx* c) override {
    if (!c->asks() && (c->state_in_pops || !c->pops_stale)) return TLB_OK;
    k_materialize<L, MODE><<<blocks(c->N, 256), 256, 0, c->stream>>>(
        geo(c), c->idle<R4<Real>>(c->L.M), c->ptr<Store>(c->L.lo[c->cur]), c->ptr<Rest>(c->L.rest[c->cur]),
        c->asks() ? c->ptr<int>(c->L.in_M) : nullptr);
    TLB_LAUNCHED(c, "k_materialize");
    // (captured, it has not run; the flag of a context that asks is not used)
    if (!caller_captures(c->stream)) c->pops_stale = false;
    return TLB_OK;
  }

  // the state is in the populations / in M from here on
  tlb_status pops_written(Ctx* c) override {
    TLB_CUDA(cudaMemsetAsync(c->ptr<int>(c->L.in_M), 0, sizeof(int), c->stream));
    c->state_in_pops = true;
    c->pops_stale = false;
    return TLB_OK;
  }
  static tlb_status entered_M(Ctx* c, cudaStream_t s) {
    TLB_CUDA(cudaMemsetAsync(c->ptr<int>(c->L.in_M), 1, sizeof(int), s));
    c->state_in_pops = false;
    return TLB_OK;
  }
  // The caller is capturing the stream.  (A query that fails, as on the
  // legacy default stream beside another capture, is left to the launches.)
  static bool caller_captures(cudaStream_t s) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess) return cs != cudaStreamCaptureStatusNone;
    (void)cudaGetLastError();
    return false;
  }

  // the moments of the streamed populations: rebuilt from the state in M, or
  // pulled from the population buffer
  static tlb_status launch_moments(Ctx* c, const LBArgs<MODE>& la, cudaStream_t s) {
    if (la.M && (la.in_M || !la.pull)) {
      const dim3 grid(blocks(c->nx, RECON_X), blocks(c->ny, RECON_Y), blocks(c->nz, la.zcm));
      k_moments_recon<L, MODE, RECON_X, RECON_Y><<<grid, RECON_X * RECON_Y, 0, s>>>(la);
      TLB_LAUNCHED(c, "k_moments_recon");
    } else {
      // 16-bit storage: 128-thread blocks, finer grains around the membrane
      // kernels that run beside this one (measured 0.262 -> 0.255 ms per
      // step on the 128^3 capsule; FP32 steps were slower with them)
      const int bt = sizeof(Store) == 2 ? 128 : 256;
      k_moments<L, MODE><<<blocks(c->N, bt), bt, 0, s>>>(la);
      TLB_LAUNCHED(c, "k_moments");
    }
    return TLB_OK;
  }

  tlb_status profile_now(Ctx* c) override {
    if (c->nn == 0) return TLB_OK;
    cudaStream_t s = c->stream;
    IBArgs<Real> ia = ibargs(c);
    tlb_status st = snapshot_box(c, ia, s, true);
    if (st == TLB_OK) st = ibm_positions(c, ia, s);
    if (st == TLB_OK) st = ibm_band(c, ia, s);
    c->box_stale = true;  // the next step recomputes the box of these markers
    return st;
  }

  tlb_status init_from_moments(Ctx* c) override {
    cudaStream_t s = c->stream;
    tlb_status pst = profile_now(c);
    if (pst != TLB_OK) return pst;
    Real* uf = c->ptr<Real>(c->L.ftot);  // u = 0
    TLB_CUDA(cudaMemsetAsync(c->ptr<char>(c->L.ftot), 0, c->L.ftot.bytes, s));
    Geo G = geo(c);
    LBArgs<MODE> la = lbargs(c, c->cur);
    Real* mu = c->ptr<Real>(c->L.mu);
    Real *rho = c->ptr<Real>(c->L.rho), *phi = c->ptr<Real>(c->L.phi), *psi = c->ptr<Real>(c->L.psi);
    k_mu_global<L, MODE><<<blocks(c->N, 256), 256, 0, s>>>(G, la.fe, rho, phi, psi, la.I, mu);
    TLB_LAUNCHED(c, "k_mu_global");
    k_init_eq<L, MODE><<<blocks(c->N, 256), 256, 0, s>>>(G, rho, phi, psi, uf, mu, la.gphi, la.gpsi,
                                                          c->ptr<Store>(c->L.lo[c->cur]),
                                                          c->ptr<Rest>(c->L.rest[c->cur]), la.p4);
    TLB_LAUNCHED(c, "k_init_eq");
    // (of these populations: what M held before is not written over them)
    tlb_status rs = pops_written(c);
    if (rs == TLB_OK) rs = residual_launch(c);
    if (rs != TLB_OK) return rs;
    TLB_CUDA(cudaStreamSynchronize(s));
    c->t = 0;
    c->t_snap = 0;
    c->initialised = true;
    return TLB_OK;
  }

  static ResPtrs resptrs(Ctx* c, unsigned long long* res) {
    return {c->ptr<double>(c->L.snap), c->ptr<double>(c->L.xsnap), res};
  }

  tlb_status residual_launch(Ctx* c) override {
    cudaStream_t s = c->stream;
    if (tlb_status st = sync_pops(c); st != TLB_OK) return st;
    TLB_CUDA(cudaMemsetAsync(c->ptr<char>(c->L.res), 0, c->L.res.bytes, s));
    const unsigned nb = blocks(c->N, 256) + blocks(c->nn, 256);
    k_residual<L, MODE><<<nb, 256, 0, s>>>(geo(c), c->ptr<Store>(c->L.lo[c->cur]), c->ptr<Rest>(c->L.rest[c->cur]),
                                           c->ptr<double>(c->L.X), c->nn,
                                           resptrs(c, c->ptr<unsigned long long>(c->L.res)));
    TLB_LAUNCHED(c, "k_residual");
    return TLB_OK;
  }

  template <int TXv, int TYv, int FORM>
  static tlb_status collide_tile(Ctx* c, LBArgs<MODE>& la, cudaStream_t s) {
    dim3 grid(blocks(c->nx, TXv), blocks(c->ny, TYv), blocks(c->nz, c->tiles_zc));
    k_collide<L, MODE, TXv, TYv, FORM><<<grid, collide_block<FORM, TXv, TYv>(), 0, s>>>(la);
    TLB_LAUNCHED(c, "k_collide");
    return TLB_OK;
  }

  // the collide in the context's variant (tile shape and form)
  static tlb_status collide(Ctx* c, LBArgs<MODE>& la, cudaStream_t s) {
    return collide_variant<L>(c->tile_variant, [&](auto tx, auto ty, auto fm) {
      return collide_tile<decltype(tx)::value, decltype(ty)::value, decltype(fm)::value>(c, la, s);
    });
  }

  // Choose the collide tile shape and z chunk by timing the kernel on the
  // current state (it only reads the current buffer, so repeats are harmless).
  tlb_status autotune(Ctx* c, int* variant, int* zc) override {
    cudaStream_t s = c->stream;
    // the candidates: the tau = 1 variants where they apply (a general one
    // pulls and stores several times their bytes), else the general ones
    const bool t1 = c->t1_ok();
    // (the timed collides write the idle population buffer)
    if (tlb_status st = enter_pops(c); st != TLB_OK) return st;
    LBArgs<MODE> la = lbargs(c, c->cur);
    use_t1(c, la, t1);
    if (tlb_status st = launch_moments(c, la, s); st != TLB_OK) return st;
    cudaEvent_t e0, e1;
    TLB_CUDA(cudaEventCreate(&e0));
    TLB_CUDA(cudaEventCreate(&e1));
    float best = 1e30f;
    int bv = c->tile_variant, bz = c->tiles_zc;
    const std::vector<int> zcs = z_chunk_candidates(c->nz);
    for (int v = 0; v < COLLIDE_NVAR; ++v)
      for (const int zcv : zcs) {
        if (!c->variant_ok(v) || variant_t1(v) != t1 || variant_again(v)) continue;
        c->tile_variant = v;
        c->tiles_zc = zcv;
        la.zc = c->tiles_zc;
        tlb_status st = collide(c, la, s);  // warm
        float tmin = 1e30f;
        for (int r = 0; r < 2 && st == TLB_OK; ++r) {
          cudaEventRecord(e0, s);
          st = collide(c, la, s);
          cudaEventRecord(e1, s);
          cudaEventSynchronize(e1);
          float ms = 0;
          cudaEventElapsedTime(&ms, e0, e1);
          tmin = fminf(tmin, ms);
        }
        if (st != TLB_OK) { cudaEventDestroy(e0); cudaEventDestroy(e1); return st; }
        if (tmin < best) { best = tmin; bv = v; bz = c->tiles_zc; }
      }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->tile_variant = bv;
    c->tiles_zc = bz;
    if (variant) *variant = bv;
    if (zc) *zc = bz;
    TLB_CUDA(cudaStreamSynchronize(s));
    return TLB_OK;
  }

  static tlb_status mark(Ctx* c, int k) {
    if (c->prof) TLB_CUDA(cudaEventRecord(c->prof->ev[k], c->stream));
    return TLB_OK;
  }

  static tlb_status collect(Ctx* c) {
    if (!c->prof) return TLB_OK;
    TLB_CUDA(cudaEventSynchronize(c->prof->ev[4]));
    for (int k = 0; k < 4; ++k) {
      float ms = 0;
      TLB_CUDA(cudaEventElapsedTime(&ms, c->prof->ev[k], c->prof->ev[k + 1]));
      c->prof_ms[k] += ms;
    }
    return TLB_OK;
  }

  // n steps; runs of GRAPH_STEPS steps replay a captured graph where the
  // steps qualify (see graph_ready)
  tlb_status step(Ctx* c, long n) override {
    if (n > 0 && caller_captures(c->stream)) return step_captured(c, n);
    c->known = false;
    const tlb_status st = step_calls(c, n);
    c->known = false;
    return st;
  }

  // A call inside a capture of the caller's stream.  Nothing runs now, and
  // each replay continues from the state it finds, which other calls may have
  // moved in between: the first tau = 1 step asks the device where the state
  // is, the first step rebuilds the marker box (with the profile, as after
  // markers set from outside), and what the host holds about the state is put
  // back.  The step counter advances once, and an odd number of general steps
  // leaves the state in the other population buffer.
  tlb_status step_captured(Ctx* c, long n) {
    const bool sp0 = c->state_in_pops, ps0 = c->pops_stale, stale0 = c->box_stale;
    c->outside = true;
    c->known = false;
    c->box_stale = c->nn > 0;
    c->capturing = true;
    const tlb_status st = step_direct(c, n);
    c->capturing = false;
    c->known = false;
    c->state_in_pops = sp0;
    c->pops_stale = ps0;
    c->box_stale = stale0;
    return st;
  }

  tlb_status step_calls(Ctx* c, long n) {
    if (!graphs_usable(c, n)) return step_direct(c, n);
    while (n > 0) {
      if (n >= Ctx::GRAPH_STEPS && graph_ready(c) && have_graph(c)) {
        tlb_status st = replay(c);
        if (st != TLB_OK) return st;
        n -= Ctx::GRAPH_STEPS;
        continue;
      }
      // direct launches until a step qualifies, the rest at the end
      const long k = n >= Ctx::GRAPH_STEPS && c->graphs ? 1 : n;
      tlb_status st = step_direct(c, k);
      if (st != TLB_OK) return st;
      n -= k;
    }
    return TLB_OK;
  }

  // Graphs serve this call: not while phases are timed; and unless
  // tlb_set_graphs asked for them, only where a graph exists already or the
  // call is long enough to pay for its capture: 0.32 ms, against 10 to 20 us
  // saved per step (32^3 to 128^3 at tau = 1, all of 2D), so from 32 steps on.
  // Where the general collide hides the launches, 7 us are saved (128^3 and
  // 160^3; 10 at 96^3, which comes out even at 32 steps): from 64 steps on.  A
  // first call of 32 or 50 steps of the 128^3 general collide: 374 us per step
  // direct, 378 and 375 with the capture; 100 steps: 373 against 370.  Without
  // membranes two launches a step hardly wait: only where asked for.
  bool graphs_usable(Ctx* c, long n) const {
    if (!c->graphs || c->prof || n < Ctx::GRAPH_STEPS) return false;
    const bool hidden = !variant_t1(c->tile_variant) && c->N * c->Q >= (1ll << 25);
    if (c->graphs_asked) return true;
    return c->nn > 0 && (graph_current(c) || n >= (hidden ? 8 : 4) * Ctx::GRAPH_STEPS);
  }
  bool graph_current(const Ctx* c) const {
    const int k = c->cur;
    return c->gexec[k] && c->gsig[k][0] == c->tile_variant && c->gsig[k][1] == c->tiles_zc;
  }

  // A step replays from a graph when it launches the same work every time:
  // no phase profile, no markers set from outside since the last step (their
  // box is rebuilt first) and the state where the collide variant keeps it
  // (the first tau = 1 step after populations were written pulls them).
  bool graph_ready(Ctx* c) const {
    return c->graphs && !c->box_stale && !c->asks() && c->state_in_pops == !variant_t1(c->tile_variant);
  }

  // the state into the populations, for a step of a general variant
  static tlb_status enter_pops(Ctx* c) {
    if (c->state_in_pops && !c->asks()) return TLB_OK;
    tlb_status st = c->impl->sync_pops(c);
    if (st == TLB_OK) st = c->impl->pops_written(c);
    return st;
  }

  // The calls around a capture of the library's own (stream creation,
  // synchronisation, instantiation) would invalidate a capture of another
  // stream that the program has under way in the global mode.  They concern
  // this context's streams only, so the thread takes the relaxed mode meanwhile.
  struct OwnCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    OwnCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~OwnCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  };

  // The graph of the current buffer, captured first if missing or captured
  // with another collide variant.  Its kernels keep the priorities of the
  // streams they were captured from (the membrane chain's blocks go first
  // beside the moments).  Where the capture fails, the steps are launched
  // directly from here on.
  bool have_graph(Ctx* c) {
    if (graph_current(c)) return true;
    const OwnCapture own;
    const int k = c->cur;
    if (!c->gstream && cudaStreamCreateWithFlags(&c->gstream, cudaStreamNonBlocking) != cudaSuccess) return no_graphs(c);
    cudaStream_t user = c->stream;
    if (c->gexec[k]) {  // (after its last replay has finished)
      if (cudaStreamSynchronize(user) != cudaSuccess) return no_graphs(c);
      cudaGraphExecDestroy(c->gexec[k]);
      c->gexec[k] = nullptr;
    }
    // capture without executing: the host-side state is put back after
    const int cur0 = c->cur;
    const long t0 = c->t, l0 = c->launches;
    const bool sp0 = c->state_in_pops, ps0 = c->pops_stale;
    if (cudaStreamBeginCapture(c->gstream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return no_graphs(c);
    c->capturing = true;
    c->stream = c->gstream;
    const tlb_status st = step_direct(c, Ctx::GRAPH_STEPS);
    c->stream = user;
    c->capturing = false;
    cudaGraph_t g = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(c->gstream, &g);
    c->glaunch[k] = c->launches - l0;
    c->cur = cur0;
    c->t = t0;
    c->launches = l0;
    c->state_in_pops = sp0;
    c->pops_stale = ps0;
    const bool ok = st == TLB_OK && ce == cudaSuccess &&
                    cudaGraphInstantiate(&c->gexec[k], g, cudaGraphInstantiateFlagUseNodePriority) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    // (the event that a direct step waits on before recording it stood for a
    // node of the capture)
    cudaEventRecord(c->ev_interp, user);
    if (!ok) {
      c->gexec[k] = nullptr;
      return no_graphs(c);
    }
    c->gsig[k][0] = c->tile_variant;
    c->gsig[k][1] = c->tiles_zc;
    return true;
  }
  static bool no_graphs(Ctx* c) {
    (void)cudaGetLastError();
    c->graphs = false;
    return false;
  }

  // One launch of the current buffer's graph.  A replay advances the state by
  // GRAPH_STEPS (an even number: the buffer index comes back).
  tlb_status replay(Ctx* c) {
    const int k = c->cur;
    cudaStream_t user = c->stream;
    TLB_CUDA(cudaGraphLaunch(c->gexec[k], user));
    // the events recorded inside the capture stand for graph nodes: the one
    // a direct step waits on before recording it is recorded again here
    TLB_CUDA(cudaEventRecord(c->ev_interp, user));
    c->launches += c->glaunch[k];
    c->t += Ctx::GRAPH_STEPS;
    c->pops_stale = variant_t1(c->tile_variant);
    return TLB_OK;
  }

  tlb_status step_direct(Ctx* c, long n) {
    cudaStream_t s = c->stream;
    tlb_status st;
    // Pipelined: the interpolation and advection of a step runs on the side
    // stream beside the next step's moments (which read the populations
    // only); the next step's marker work waits for it there.  The phase
    // profile keeps every kernel on the main stream.
    const bool pipe = c->nn > 0 && !c->prof;
    const bool t1 = variant_t1(c->tile_variant);
    if (!t1 && (st = enter_pops(c)) != TLB_OK) return st;
    // (the last record may stand for a node of the caller's capture)
    if (pipe && c->outside && !c->capturing) TLB_CUDA(cudaEventRecord(c->ev_interp, s));
    for (long k = 0; k < n; ++k) {
      LBArgs<MODE> la = lbargs(c, c->cur);
      IBArgs<Real> ia = ibargs(c);
      const bool fresh = c->box_stale;  // markers set from outside since the last step
      c->box_stale = false;
      if ((st = mark(c, 0)) != TLB_OK) return st;
      if (c->nn > 0) {  // fork: position-only membrane work on the two side streams
        // The step's marker box: after markers set from outside it is rebuilt
        // (with the coordinate split the side streams read) before the fork;
        // otherwise it is the previous advection's accumulator, copied on the
        // side stream after that advection.
        const bool box_on_side = pipe && !fresh;
        if (!box_on_side && (st = snapshot_box(c, ia, s, fresh)) != TLB_OK) return st;
        TLB_CUDA(cudaEventRecord(c->ev_fork, s));
        TLB_CUDA(cudaStreamWaitEvent(c->side, c->ev_fork, 0));
        TLB_CUDA(cudaStreamWaitEvent(c->side2, c->ev_fork, 0));
        // the previous advection (a graph's first step follows the whole
        // previous launch on the caller's stream instead)
        if (pipe && !(c->capturing && k == 0)) TLB_CUDA(cudaStreamWaitEvent(c->side2, c->ev_interp, 0));
        if ((st = ibm_positions(c, ia, c->side, box_on_side, c->ev_geom)) != TLB_OK) return st;
        if ((st = ibm_bins(c, ia, c->side2, c->ev_geom)) != TLB_OK) return st;
        TLB_CUDA(cudaEventRecord(c->ev_bins, c->side2));
      }
      if ((st = launch_moments(c, la, s)) != TLB_OK) return st;
      if ((st = mark(c, 1)) != TLB_OK) return st;
      // the profile, coupling sums and spreading need psi(t) and the
      // position work: they follow the moments, then the whole lattice is
      // collided in one launch
      if (c->nn > 0) {
        TLB_CUDA(cudaEventRecord(c->ev_join, c->side));
        TLB_CUDA(cudaStreamWaitEvent(s, c->ev_join, 0));
        TLB_CUDA(cudaStreamWaitEvent(s, c->ev_bins, 0));
        // (in order: running the fill beside the spreading, or splitting the
        // collide to overlap this work, measured slower)
        // (the column fill only after markers were set from outside: between
        // fresh starts the band keeps the cells beyond dc)
        if ((st = launch_band(c, ia, s)) != TLB_OK) return st;
        if (fresh && (st = launch_fill(c, ia, s)) != TLB_OK) return st;
        if ((st = ibm_spread(c, ia, s)) != TLB_OK) return st;
      }
      if ((st = mark(c, 2)) != TLB_OK) return st;
      if ((st = collide(c, la, s)) != TLB_OK) return st;
      if ((st = mark(c, 3)) != TLB_OK) return st;
      if (c->nn > 0) {
        cudaStream_t si = s;
        if (pipe) {
          TLB_CUDA(cudaEventRecord(c->ev_coll, s));
          TLB_CUDA(cudaStreamWaitEvent(c->side, c->ev_coll, 0));
          si = c->side;
        }
        k_interp_advect<L, MODE><<<blocks((long long)c->nn * 32, 128), 128, 0, si>>>(ia, la.lo_dst);
        TLB_LAUNCHED(c, "k_interp_advect");
        if (pipe) TLB_CUDA(cudaEventRecord(c->ev_interp, c->side));
      }
      if ((st = mark(c, 4)) != TLB_OK) return st;
      if ((st = collect(c)) != TLB_OK) return st;
      if (t1) {  // the state is M from here on
        if ((la.pull || la.in_M) && (st = entered_M(c, s)) != TLB_OK) return st;
        c->pops_stale = true;
      } else {
        c->cur = 1 - c->cur;
      }
      c->known = true;
      c->t += 1;
    }
    if (pipe && n > 0) TLB_CUDA(cudaStreamWaitEvent(s, c->ev_interp, 0));  // all of it on the caller's stream
    return TLB_OK;
  }

  tlb_status read_field(Ctx* c, int field, double* dst, size_t nvals) override {
    cudaStream_t s = c->stream;
    const long long N = c->N;
    double* rb = c->ptr<double>(c->L.rb);
    const size_t need = field == TLB_FIELD_U ? 3 * (size_t)N : (size_t)N;
    if (nvals < need) { set_error("read_field: buffer too small"); return TLB_ERR_ARG; }
    if (tlb_status st = sync_pops(c); st != TLB_OK) return st;
    // the field is formed on the device, only its values cross to the host
    if (field == TLB_FIELD_I) {
      k_to_double<Real><<<blocks(N, 256), 256, 0, s>>>(c->ptr<Real>(c->L.I), N, rb);
      TLB_LAUNCHED(c, "k_to_double");
    } else {
      k_fields<L, MODE><<<blocks(N, 256), 256, 0, s>>>(geo(c), c->ptr<Store>(c->L.lo[c->cur]),
                                                        c->ptr<Rest>(c->L.rest[c->cur]), field, rb);
      TLB_LAUNCHED(c, "k_fields");
    }
    TLB_CUDA(cudaMemcpyAsync(dst, rb, need * sizeof(double), cudaMemcpyDeviceToHost, s));
    TLB_CUDA(cudaStreamSynchronize(s));
    return TLB_OK;
  }

  // Populations are stored post-collision; the caller's view is the streamed
  // (pre-collision) state.  The conversion runs on the host: it is I/O, not
  // part of the time step.
  static double h2d(double v) { return v; }
  static double h2d(float v) { return v; }
  static double h2d(__half v) { return (double)__half2float(v); }
  static double h2d(__nv_bfloat16 v) { return (double)__bfloat162float(v); }
  static void d2h(double v, double& o) { o = v; }
  static void d2h(double v, float& o) { o = (float)v; }
  static void d2h(double v, __half& o) { o = __float2half_rn((float)v); }
  static void d2h(double v, __nv_bfloat16& o) { o = __float2bfloat16_rn((float)v); }

  static long long hwrap(long long a, long long n) { return ((a % n) + n) % n; }

  tlb_status read_pops(Ctx* c, double* dst) override {
    cudaStream_t s = c->stream;
    if (tlb_status st = sync_pops(c); st != TLB_OK) return st;
    const long long N = c->N, P = c->P;
    std::vector<Store> lo((size_t)(3 * L::Q - 2) * P);
    std::vector<Rest> rest((size_t)2 * P);
    TLB_CUDA(cudaMemcpyAsync(lo.data(), c->ptr<Store>(c->L.lo[c->cur]), lo.size() * sizeof(Store), cudaMemcpyDeviceToHost, s));
    TLB_CUDA(cudaMemcpyAsync(rest.data(), c->ptr<Rest>(c->L.rest[c->cur]), rest.size() * sizeof(Rest), cudaMemcpyDeviceToHost, s));
    TLB_CUDA(cudaStreamSynchronize(s));
    for (long long n = 0; n < N; ++n) {
      long long x = n % c->nx, y = (n / c->nx) % c->ny, z = n / ((long long)c->nx * c->ny);
      for (int i = 0; i < L::Q; ++i) {
        long long sz = z - L::cz(i), src;
        int ii = i;
        if (c->p.wall_last && (sz < 0 || sz >= c->nz)) { src = n; ii = L::opp(i); }
        else src = (hwrap(sz, c->nz) * c->ny + hwrap(y - L::cy(i), c->ny)) * c->nx + hwrap(x - L::cx(i), c->nx);
        dst[(long long)i * N + n] = h2d(lo[(size_t)plane_f<L>(ii) * P + src]) + L::w(ii);
        dst[(long long)(L::Q + i) * N + n] = ii == 0 ? h2d(rest[src]) : h2d(lo[(size_t)plane_g<L>(ii) * P + src]);
        dst[(long long)(2 * L::Q + i) * N + n] = ii == 0 ? h2d(rest[P + src]) : h2d(lo[(size_t)plane_h<L>(ii) * P + src]);
      }
    }
    return TLB_OK;
  }

  tlb_status write_pops(Ctx* c, const double* src_in) override {
    cudaStream_t s = c->stream;
    const long long N = c->N, P = c->P;
    std::vector<Store> lo((size_t)(3 * L::Q - 2) * P);
    std::vector<Rest> rest((size_t)2 * P);
    for (long long n = 0; n < N; ++n) {
      long long x = n % c->nx, y = (n / c->nx) % c->ny, z = n / ((long long)c->nx * c->ny);
      for (int i = 0; i < L::Q; ++i) {
        long long tz = z + L::cz(i), src;
        int ii = i;
        if (c->p.wall_last && (tz < 0 || tz >= c->nz)) { src = n; ii = L::opp(i); }
        else src = (hwrap(tz, c->nz) * c->ny + hwrap(y + L::cy(i), c->ny)) * c->nx + hwrap(x + L::cx(i), c->nx);
        d2h(src_in[(long long)ii * N + src] - L::w(ii), lo[(size_t)plane_f<L>(i) * P + n]);
        if (ii == 0) {
          d2h(src_in[(long long)L::Q * N + src], rest[n]);
          d2h(src_in[(long long)2 * L::Q * N + src], rest[P + n]);
        } else {
          d2h(src_in[(long long)(L::Q + ii) * N + src], lo[(size_t)plane_g<L>(i) * P + n]);
          d2h(src_in[(long long)(2 * L::Q + ii) * N + src], lo[(size_t)plane_h<L>(i) * P + n]);
        }
      }
    }
    TLB_CUDA(cudaMemcpyAsync(c->ptr<Store>(c->L.lo[c->cur]), lo.data(), lo.size() * sizeof(Store), cudaMemcpyHostToDevice, s));
    TLB_CUDA(cudaMemcpyAsync(c->ptr<Rest>(c->L.rest[c->cur]), rest.data(), rest.size() * sizeof(Rest), cudaMemcpyHostToDevice, s));
    if (tlb_status st = pops_written(c); st != TLB_OK) return st;
    TLB_CUDA(cudaStreamSynchronize(s));
    c->initialised = true;
    return TLB_OK;
  }

  // Contact angles (tlb_measure.cuh).  Scratch: phi in the read-back
  // buffer; marker values, edge angles and the per-capsule results in the
  // idle population buffer, past the tau = 1 state if they fit there (or else
  // the state moves to the other buffer, and the next step pulls it: 30 us at
  // 128^3).
  tlb_status contact_angle(Ctx* c, double* out) override {
    cudaStream_t s = c->stream;
    const long long N = c->N;
    const int nedge = c->NV == 2 ? c->nn : c->nedge;
    const size_t need = (size_t)(4 * c->nn + nedge + 4 * c->ncap) * sizeof(double) + (size_t)nedge * sizeof(int);
    if (c->ncap == 0) return TLB_OK;
    const size_t room = c->L.lo[1 - c->cur].bytes;
    if (need > room) { set_error("contact_angle: scratch too small"); return TLB_ERR_ARG; }
    size_t past = c->L.j2.off + c->L.j2.bytes;
    if (need + past > room) past = 0;
    if (tlb_status st = past ? sync_pops(c) : enter_pops(c); st != TLB_OK) return st;
    double* phi = c->ptr<double>(c->L.rb);
    k_fields<L, MODE><<<blocks(N, 256), 256, 0, s>>>(geo(c), c->ptr<Store>(c->L.lo[c->cur]),
                                                      c->ptr<Rest>(c->L.rest[c->cur]), TLB_FIELD_PHI, phi);
    TLB_LAUNCHED(c, "k_fields");
    double* sc = c->idle<double>({past, need});
    AngleArgs a;
    a.G = geo(c);
    a.dim = c->p.dim;
    a.nn = c->nn;
    a.NV = c->NV;
    a.X = c->ptr<double>(c->L.X);
    a.phi = phi;
    a.E = c->ptr<int>(c->L.E);
    a.inc_off = c->ptr<int>(c->L.inc_off);
    a.inc = c->ptr<int>(c->L.inc);
    a.rnext = c->ptr<int>(c->L.rnext);
    a.rprev = c->ptr<int>(c->L.rprev);
    a.edges = c->ptr<int>(c->L.edges);
    a.ncap = c->ptr<int>(c->L.ncap);
    a.nedge = nedge;
    a.mk = sc;
    a.ang = sc + 4 * c->nn;
    double* res = a.ang + nedge;
    a.ecapo = reinterpret_cast<int*>(res + 4 * c->ncap);
    k_marker_phi<<<blocks(c->nn, 128), 128, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_marker_phi");
    k_contact_edges<L><<<blocks(nedge, 128), 128, 0, s>>>(a);
    TLB_LAUNCHED(c, "k_contact_edges");
    k_contact_reduce<<<c->ncap, 256, 0, s>>>(a.ang, a.ecapo, nedge, res);
    TLB_LAUNCHED(c, "k_contact_reduce");
    TLB_CUDA(cudaMemcpyAsync(out, res, 4 * c->ncap * sizeof(double), cudaMemcpyDeviceToHost, s));
    TLB_CUDA(cudaStreamSynchronize(s));
    return TLB_OK;
  }

  tlb_status diagnostics(Ctx* c, tlb_diag* out) override {
    if (tlb_status st = sync_pops(c); st != TLB_OK) return st;
    return fp64_diagnostics<L, MODE>(c, c->ptr<double>(c->L.part), 1024, c->ptr<double>(c->L.meas), out);
  }
};
