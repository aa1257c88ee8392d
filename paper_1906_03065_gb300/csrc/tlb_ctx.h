// Host-side context of the library: the arena layout and the per-context
// state.  The caller's arena is carved into fixed regions once, at
// tlb_create; no other device memory is ever allocated.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/tlb.h"

// Collide variants: the 3 tile shapes of the general collide (v = 0..12, tile
// v % 3), the 3 tiles in the two forms of the tau = 1 collide (v = 13..18, see
// variant_t1); 22..27 name those again, 28..31 a fourth tile.
constexpr int COLLIDE_NVAR = 32;
constexpr bool variant_t1(int v) { return (v >= 13 && v <= 18) || v >= 22; }
// variants 22..27 and 30, 31 need an even nx (two-cell forms of the tau = 1
// collide; they run the one-cell kernels)
constexpr bool variant_pair(int v) { return (v >= 22 && v <= 27) || v == 30 || v == 31; }
// variants that run the kernel of another one (3..5 for the general collide):
// an autotuner need not time them
constexpr bool variant_again(int v) { return variant_pair(v) || (v <= 12 && (v < 3 || v > 5)); }
// variants 19..21: the general collide with the pressure-tensor force
constexpr bool variant_pt(int v) { return v >= 19 && v <= 21; }

// z-chunk lengths the collide autotuner tries: every distinct ceil(nz / m)
// of at least 4 planes (each gives another grid, so another fill of the
// last wave of blocks).
inline std::vector<int> z_chunk_candidates(int nz) {
  std::vector<int> v;
  for (int m = 1;; ++m) {
    const int zc = (nz + m - 1) / m;
    if (v.empty() || v.back() != zc) v.push_back(zc);
    if (zc <= 4) break;
  }
  return v;
}

// Length of the z chunks of a plane sweep.  A block of the sweep walks its
// chunk plus `ahead` planes that only fill its rings and running sums, and
// `resident` blocks share an SM; a plane of a block takes 1 + load * b in
// units of what it takes alone when b blocks of the SM run beside each other
// (load: 0 if they only hid each other's latency, large if they only queued
// for the SM's arithmetic).  Short chunks repeat the `ahead` planes, long
// ones leave SMs idle on small lattices or end in a nearly empty last wave:
// the chunk taken is the one with the least sum over its waves.  `tiles`:
// column tiles and planes of each lattice swept together.
struct SweepCost {
  int resident;
  double ahead, load;
};
struct SweepTiles {
  long long columns;
  int nz;
};
inline int sweep_chunk(const std::vector<SweepTiles>& tiles, int nsm, const SweepCost& s) {
  int nzmax = 1, best = 1;
  for (const SweepTiles& t : tiles) nzmax = t.nz > nzmax ? t.nz : nzmax;
  double tbest = 0;
  for (int m = 1, last = 0; m <= nzmax; ++m) {
    const int zc = (nzmax + m - 1) / m;
    if (zc == last) continue;
    last = zc;
    long long n = 0;
    for (const SweepTiles& t : tiles) n += t.columns * ((t.nz + zc - 1) / zc);
    const long long cap = (long long)s.resident * nsm, rest = n % cap;
    const double t = (zc + s.ahead) * ((double)(n / cap) * (1 + s.load * s.resident) +
                                       (rest ? 1 + s.load * (double)((rest + nsm - 1) / nsm) : 0));
    if (tbest == 0 || t < tbest) {
      tbest = t;
      best = zc;
    }
  }
  return best;
}
// The collide and the moments rebuild.  The numbers fit timings of every
// chunk length on 64^2 and 240x120 (FP64, FP32) and 41x37x35 to 192x128x128
// lattices; the chunk taken was within 8% of the fastest one on each, where a
// fixed one (32 planes from nz = 64, else 8) lost 15% at 128^3 (71 against 61
// us), a factor 2 at 64^3 (43 against 18) and 7 at 64^2 FP64 (225 against 30).
// On 13 sizes that took no part in the fit (48x48x200 to 224x160x96, 128x96 to
// 1000x30, every storage type, both collides) it was within 4% in 3D but for
// the general collide at 112^3 (11%), and within 16% in 2D.
inline SweepCost collide_cost(int resident, int threads, bool f64, bool t1) {
  return {resident, t1 ? 5.0 : 3.0, (f64 ? 0.47 : (t1 ? 0.15 : 0.5)) * threads / 128};
}
inline SweepCost recon_cost(int resident, int threads, bool f64) { return {resident, 3.0, (f64 ? 0.8 : 0.6) * threads / 128}; }

// Warps that share one group of 32 features in the distance scatter: as many
// as bring its warps to 16 per SM (a batch: four times that, so that the last
// of its waves over the resident blocks costs little), at most one per round
// of slices (4 slices each, 2 dc + 3 per feature or so); for `warps` groups
// swept together.
inline int scatter_split(long long warps, double dc, int nsm, int waves) {
  const long long rounds = ((long long)(2 * dc) + 3 + 3) / 4, want = (16ll * waves * nsm + warps / 2) / (warps > 0 ? warps : 1);
  return (int)(want < 1 ? 1 : (want > rounds ? rounds : want));
}

struct Ctx;

struct ImplBase {
  virtual ~ImplBase() {}
  virtual tlb_status init_fields(Ctx* c, const double* C, const double* u) = 0;
  virtual tlb_status step(Ctx* c, long n) = 0;
  virtual tlb_status read_field(Ctx* c, int field, double* dst, size_t n) = 0;
  virtual tlb_status read_pops(Ctx* c, double* dst) = 0;
  virtual tlb_status write_pops(Ctx* c, const double* src) = 0;
  virtual tlb_status diagnostics(Ctx* c, tlb_diag* out) = 0;
  virtual tlb_status autotune(Ctx* c, int* variant, int* zc) = 0;
  // launches the residual kernel into c->L.res (zeroed first); no sync
  virtual tlb_status residual_launch(Ctx* c) = 0;
  // initial state from the rho, phi, psi moment arrays as they stand and the
  // current marker positions (profile, u = 0, equilibrium populations)
  virtual tlb_status init_from_moments(Ctx* c) = 0;
  // profile I (with owners and distances) of the current marker positions
  virtual tlb_status profile_now(Ctx* c) = 0;
  // contact angle of every capsule with phi = 0: out[cap] = {mean, min,
  // max, contact points}; synchronises
  virtual tlb_status contact_angle(Ctx* c, double* out) = 0;
  // write the populations that the state in M stands for into the current
  // population buffer if it is stale (no-op otherwise)
  virtual tlb_status sync_pops(Ctx* c) = 0;
  // the population buffer holds the state from here on
  virtual tlb_status pops_written(Ctx* c) = 0;
  // chunk lengths of the plane sweeps for lattices swept together (the
  // default collide variant; the moments rebuild in blocks of bt threads)
  virtual int collide_chunk(const std::vector<Ctx*>& cs, int variant) = 0;
  virtual int recon_chunk(const std::vector<Ctx*>& cs, int tx, int ty) = 0;
};

// CUDA events bracketing the phases of a step when profiling.
struct PhaseEvents {
  cudaEvent_t ev[5];
  bool on = false;
};

// Sizes in bytes of the precision-dependent element types.
struct TypeSizes {
  size_t real, store, rest;
};

// One region of the arena.
struct Region {
  size_t off = 0, bytes = 0;
};

struct Layout {
  // lattice
  Region lo[2], rest[2];
  Region rho, phi, psi, p4, j2, M, I, dsel, own, key, fib, ftot, mu, rb;
  // membranes
  Region X, E, ecap, ncap, cap_par, ds0, rprev, rnext, A0, G0i, inc_off, inc, adj, edges;
  Region en, vn, nadj, wts, erel, eorg, ecst, xo, xr, skc, capr, ncpl, F, box;
  Region bcnt, bprev, bcur, boff, blist, bact, ctr, bflag;
  // misc
  Region status, part, meas;
  Region in_M;
  // equilibrium residual: reference phi, psi and marker positions, maxima
  Region snap, xsnap, res;
  size_t total = 0;
};

struct HostMem {
  int kind, nn, ne;
  std::vector<double> X0;  // internal coordinates, unwrapped along edges
  std::vector<int> E;
  double ks, kb, G, C;
};

struct Ctx {
  tlb_params p;
  // the tau = 1 collide applies: tau = tau_phi = tau_psi = 1 and the exact
  // difference method (every post-collision population is an equilibrium)
  bool t1_ok() const {
    return p.tau == 1.0 && p.tau_phi == 1.0 && p.tau_psi == 1.0 && p.forcing == TLB_FORCE_EDM &&
           p.force_form == TLB_FE_POTENTIAL;
  }
  // the moments are kept packed, one vector per cell (the collides with the
  // potential force read them so)
  bool packed() const { return p.force_form == TLB_FE_POTENTIAL; }
  // a collide variant this context can run: the pressure-tensor variants for
  // the pressure-tensor force only, the tau = 1 ones only where they apply,
  // and with TLB_STATE_MOMENTS only the tau = 1 ones
  bool variant_ok(int v) const {
    if (variant_pt(v) != (p.force_form == TLB_FE_PRESSURE_TENSOR)) return false;
    if (variant_pair(v) && nx % 2 != 0) return false;
    if (variant_t1(v)) return t1_ok();
    return p.state != TLB_STATE_MOMENTS;
  }
  // Where the state is.  A step with a tau = 1 collide variant keeps it in
  // the 12 values per cell of M (see EqCell), any other in the population
  // buffer `cur`.  state_in_pops: in the populations (after an
  // initialisation, a load, a write of populations or a general step), which
  // the next tau = 1 step pulls; otherwise in M, and pops_stale says that the
  // population buffer does not show it yet (sync_pops writes it there).
  bool state_in_pops = true;
  bool pops_stale = false;
  // The device word L.in_M says the same (0: in the populations) and is kept
  // beside the flag.  Once the caller has captured steps into a graph of its
  // own (`outside`), replays move the state without the host: kernels then
  // read the word, except within a step call after its first step (`known`).
  bool outside = false;
  bool known = false;
  bool asks() const { return outside && !known; }
  int Q = 0;
  int nx = 0, ny = 0, nz = 0;  // internal sizes (2D: nx, 1, ny)
  long long N = 0, P = 0;
  TypeSizes ts{};
  Layout L;
  char* base = nullptr;
  size_t bytes = 0;
  cudaStream_t stream = nullptr;
  cudaStream_t side = nullptr;   // membrane work that overlaps the moments: geometry
                                 // and the distance scatter
  cudaStream_t side2 = nullptr;  // brick binning and elastic forces, beside `side`
  cudaEvent_t ev_fork = nullptr, ev_geom = nullptr, ev_join = nullptr, ev_bins = nullptr, ev_coll = nullptr, ev_interp = nullptr;
  int nsm = 1;  // streaming multiprocessors of the device
  int cur = 0;  // population buffer holding the current state
  long t = 0;
  long t_snap = 0;  // step of the residual's reference state
  bool initialised = false;
  bool box_stale = false;  // markers were overwritten: recompute the marker box
  long launches = 0;
  // membranes
  std::vector<HostMem> mems;
  int nn = 0, ne = 0, NV = 0, ncap = 0, nedge = 0;
  int nbx = 0, nby = 0, nbz = 0, nbricks = 0;
  int tiles_zc = 16;
  int recon_zc = 16;     // the same of the moments rebuild
  int scat_split = 1;    // see scatter_split
  int band_blocks = 0, spread_blocks = 0;  // see box_estimates
  long long features() const { return (long long)ne + nedge + nn; }  // of the distance scatter
  int tile_variant = 0;  // collide tile shape and form (see collide_variant)
  PhaseEvents* prof = nullptr;  // non-null while tlb_profile_steps runs
  double prof_ms[4] = {0, 0, 0, 0};
  ImplBase* impl = nullptr;
  // Step graphs: GRAPH_STEPS steps captured from the context's streams and
  // replayed as one graph launch, one graph per starting population buffer;
  // a graph holds the collide variant and z chunk it was captured with.
  static constexpr int GRAPH_STEPS = 8;
  bool graphs = true;          // replay captured steps where a step qualifies
  bool graphs_asked = false;   // ... whatever a capture costs (tlb_set_graphs)
  bool capturing = false;      // the steps being issued are captured
  cudaGraphExec_t gexec[2] = {nullptr, nullptr};
  // graphs are captured on a stream of the context's own (the caller's stream
  // may be the legacy default stream, which cannot be captured)
  cudaStream_t gstream = nullptr;
  int gsig[2][2] = {{-1, -1}, {-1, -1}};  // (tile_variant, tiles_zc) of each graph
  long glaunch[2] = {0, 0};    // kernel launches one replay makes
  void drop_graphs() {
    for (int k = 0; k < 2; ++k) {
      if (gexec[k]) cudaGraphExecDestroy(gexec[k]);
      gexec[k] = nullptr;
      gsig[k][0] = gsig[k][1] = -1;
    }
  }

  template <class T> T* ptr(const Region& r) const { return reinterpret_cast<T*>(base + r.off); }
  // The tau = 1 scheme's state and momenta, M and j2, lie in the population
  // buffer that its steps leave idle (they take 14 planes of the arithmetic
  // type, the buffer holds 3Q - 2 of the storage type: at least 1.7 times as
  // much).  A general step writes its populations there and others use it as
  // scratch, all after the state has entered the current buffer.
  template <class T> T* idle(const Region& r) const { return reinterpret_cast<T*>(base + L.lo[1 - cur].off + r.off); }

  ~Ctx() {
    if (gexec[0] || gexec[1]) cudaEventSynchronize(ev_interp);  // (recorded after every replay)
    drop_graphs();
    if (gstream) cudaStreamDestroy(gstream);
    if (side) cudaStreamSynchronize(side);
    if (side2) cudaStreamSynchronize(side2);
    if (ev_fork) cudaEventDestroy(ev_fork);
    if (ev_geom) cudaEventDestroy(ev_geom);
    if (ev_join) cudaEventDestroy(ev_join);
    if (ev_bins) cudaEventDestroy(ev_bins);
    if (ev_coll) cudaEventDestroy(ev_coll);
    if (ev_interp) cudaEventDestroy(ev_interp);
    if (side) cudaStreamDestroy(side);
    if (side2) cudaStreamDestroy(side2);
  }
};

// Blocks of the box-sized operations (profile band, spreading): the
// work scales with the marker box, estimated from the initial markers.
inline void box_estimates(const Ctx* c, int* band_blocks, int* spread_blocks) {
  if (c->nn == 0) { *band_blocks = *spread_blocks = 0; return; }
  double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
  for (const HostMem& m : c->mems)
    for (int l = 0; l < m.nn; ++l)
      for (int d = 0; d < 3; ++d) {
        lo[d] = std::min(lo[d], m.X0[3 * l + d]);
        hi[d] = std::max(hi[d], m.X0[3 * l + d]);
      }
  const int n[3] = {c->nx, c->ny, c->nz};
  const double margin = 2.0 * (ceil(c->p.dc) + 2.0) + 2.0;
  double cells = 1, bricks = 1;
  for (int d = 0; d < 3; ++d) {
    cells *= std::min((double)n[d], hi[d] - lo[d] + margin);
    bricks *= std::min(ceil(n[d] / 4.0), ceil((hi[d] - lo[d] + 4.0) / 4.0) + 1.0);
  }
  // about two box cells per thread of a 128-thread block
  *band_blocks = (int)std::max(1.0, std::min(65536.0, ceil(cells / 256.0)));
  *spread_blocks = (int)std::max(1.0, std::min((double)c->nbricks, bricks));
}

struct Batch;

struct BatchBase {
  virtual ~BatchBase() {}
  virtual tlb_status step(Batch* b, long n) = 0;
  // launches the residual of every active instance into its slot of b->res
  // (zeroed first); no sync
  virtual tlb_status residual(Batch* b) = 0;
  virtual tlb_status autotune(Batch* b, int* variant, int* zc) = 0;
  // n steps with direct launches, device time of each of the six phases
  // summed into ms[0..5]; synchronises
  virtual tlb_status profile(Batch* b, long n, double* ms) = 0;
};

// A batch of independent contexts of one lattice type and storage, stepped
// together (see tlb_batch.cuh).  The instances live in sub-arenas of the
// batch arena, followed by the batch's own tables.
struct Batch {
  // six phases of a step, the residual, and phase 3 of a step after markers
  // were set from outside (with the column fill)
  static constexpr int NPH = 8, PH_FRESH = 7;
  static constexpr int MAXOPS = 4;   // kernel bodies per phase
  static constexpr size_t ARGS_BYTES = 1024;  // bound on one instance's argument record
  std::vector<Ctx*> inst;
  std::vector<int> act;  // active instances, ascending
  int dim = 0, storage = 0;
  cudaStream_t stream = nullptr;
  cudaStream_t cap = nullptr;  // capture stream of the step graph
  char* base = nullptr;
  size_t bytes = 0;
  Region targs[2], vg, res;
  int ph_ent[NPH] = {0}, ph_total[NPH] = {0}, ph_grid[NPH] = {0};
  cudaGraphExec_t graph = nullptr;
  bool graph_dirty = true;
  bool fresh = false;  // the next step follows markers set from outside
  long graph_launches = 0;  // kernels in one launch of the step graph
  int tile_variant = 0, zc = 16, recon_zc = 16, scat_split = 1;
  long launches = 0;
  BatchBase* impl = nullptr;

  template <class T> T* ptr(const Region& r) const { return reinterpret_cast<T*>(base + r.off); }

  ~Batch() {
    if (stream) cudaStreamSynchronize(stream);
    if (graph) cudaGraphExecDestroy(graph);
    if (cap) cudaStreamDestroy(cap);
    for (Ctx* c : inst) delete c;
  }
};

void set_error(const std::string& msg);
tlb_status cuda_check(cudaError_t e, const char* what);
#define TLB_CUDA(call)                                              \
  do {                                                              \
    tlb_status _s = cuda_check((call), #call);                      \
    if (_s != TLB_OK) return _s;                                    \
  } while (0)
#define TLB_LAUNCHED(ctx, what)                                     \
  do {                                                              \
    (ctx)->launches++;                                              \
    tlb_status _s = cuda_check(cudaGetLastError(), what);           \
    if (_s != TLB_OK) return _s;                                    \
  } while (0)

ImplBase* make_impl_d2q9_f64();
ImplBase* make_impl_d2q9_f32();
ImplBase* make_impl_d3q19_f32();
ImplBase* make_impl_d3q19_f16();
ImplBase* make_impl_d3q19_bf16();
BatchBase* make_batch_impl_d2q9_f64();
BatchBase* make_batch_impl_d2q9_f32();
BatchBase* make_batch_impl_d3q19_f32();
BatchBase* make_batch_impl_d3q19_f16();
BatchBase* make_batch_impl_d3q19_bf16();
