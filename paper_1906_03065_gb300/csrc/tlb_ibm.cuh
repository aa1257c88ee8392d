// Immersed-boundary kernels: membrane profile I (eq. Iprofile), coupling
// force (eqs. DiscreteCE, DiscreteCF), elastic forces (2D: eqs. DiscreteSE,
// DiscreteBE; 3D: Skalak shear and Helfrich bending), spreading (eq.
// Spreading with eq. DiscreteDirac), interpolation and advection (eqs.
// Interpolation, UpdatedXl).
#pragma once
#include <type_traits>

#include "tlb_common.cuh"

constexpr unsigned long long KEY_NONE = ~0ull;
constexpr int BRICK = 4;  // spreading bins are 4x4x4 cells (4x1x4 in 2D)

template <class Real>
struct IBArgs {
  Geo G;
  int dim, NV;  // dim 2: segments (NV = 2); dim 3: triangles (NV = 3)
  int nn, ne;
  double* X;             // [nn][3] unwrapped positions
  int* xo;               // [nn][3] floor(X) (kept by the box and advection kernels)
  Real* xr;              // [nn][3] X - xo
  const int* E;          // [ne][NV]
  const int* ecap;       // element -> capsule
  const int* ncap;       // node -> capsule
  const double* ks;      // per capsule
  const double* kb;
  const double* sG;
  const double* sC;
  const double* ds0;     // 2D: rest length of segment e
  const int* rprev;      // 2D: previous node on the ring
  const int* rnext;      // 2D: next node on the ring
  const double* A0;      // 3D: reference area per triangle
  const double* G0i;     // 3D: inverse reference metric per triangle (3)
  const Real* skc;       // 3D: per triangle G0i[0], 2 G0i[1], G0i[2], det G0i, A0 (working precision)
  const Real* capr;      // per capsule ks, kb, G, C (working precision), [4][ncaps]
  int ncaps;
  int split;             // virtual blocks sharing one block of features (distance scatter)
  const int* inc_off;    // node -> incident elements (CSR, ascending)
  const int* inc;
  const int* adj;        // 3D: triangle across edge q (q: vertex q -> q+1)
  int nedge;             // 3D: unique edges
  const int* edges;      // 3D: [nedge][4] vertex a, vertex b, face left, face right
  // per-step work
  R4<Real>* en;          // [ne] unit outward normal; reach of a thin face's border
                         // (see dist_scatter_body), else 0
  R4<Real>* vn;          // [nn] angle-weighted vertex pseudo-normal
  Real* wts;             // [nn][3][4] kernel weights (eq. DiscreteDirac) at the support
                         // cells floor(X) - 1 .. floor(X) + 2 along each axis
  R4<Real>* nadj;        // [nn] 3D: derivatives of the marker's bending energy with
                         // respect to its K (three) and A (see geometry_body)
  // per element, read as whole vectors by the band:
  R4<Real>* erel;        // [ne] first vertex relative to the element's origin
  int4* eorg;            // [ne] element origin: floor of its first vertex
  R4<Real>* ecst;        // [ne][4] edge vectors ab, ac, bc, Gram entries d00 d01 d11 and
                         // the reciprocals of d00, d11, |bc|^2 and the Gram determinant
  unsigned long long* ncpl;  // [nn][3] coupling force per marker, fixed point (CPL_SCALE)
  Real* F;               // [nn][3] node force
  int* box;              // [6] marker box accumulator: floor(min X), -ceil(max X)
  const int* boxc;       // [6] the step's marker box (snapshot of the accumulator)
  unsigned long long* key;
  int* own;
  Real* I;
  Real* dsel;
  const Real* psi;       // psi(t) of cell n at psi[n * psi_step] (moment field)
  int psi_step;
  const R4<Real>* M;     // tau = 1 scheme: the stored state the interpolation
                         // rebuilds the streamed populations from (NULL: the
                         // population buffers are read)
  Real* fib;             // [3][P]
  const Real* ftot;      // [3][P]
  int* bcnt;             // bricks: count, previous count, cursor, offset
  int* bprev;
  int* bcur;
  int* boff;
  int* blist;
  int* bact;             // active bricks (compacted list)
  unsigned char* bflag;  // per brick: markers spread into it this step
  int* ctr;              // [0] active bricks, [1] list slots claimed
  int nbx, nby, nbz, nbricks;
  Real alpha, dc, kc;
  Real Iin, Iout;        // I beyond dc inside / outside: (1 +- tanh(dc/(2 alpha)))/2
  unsigned* status;
};

// ------------------------------------------------------------ small vectors
template <class T> struct V3 { T x, y, z; };
template <class T> TLB_HD V3<T> mk(T a, T b, T c) { return {a, b, c}; }
template <class T> TLB_HD V3<T> operator+(V3<T> a, V3<T> b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
template <class T> TLB_HD V3<T> operator-(V3<T> a, V3<T> b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
template <class T> TLB_HD V3<T> operator*(T s, V3<T> a) { return {s * a.x, s * a.y, s * a.z}; }
template <class T> TLB_HD T dot(V3<T> a, V3<T> b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
template <class T> TLB_HD V3<T> cross(V3<T> a, V3<T> b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// dot(a, b) with explicit roundings (see rmul): the small strains and
// curvatures left over from sums of larger terms then come out the same in
// every kernel the code is inlined into.
template <class T> __device__ __forceinline__ T rdot(V3<T> a, V3<T> b) {
  return rfma(a.z, b.z, rfma(a.y, b.y, rmul(a.x, b.x)));
}

// Correctly rounded reciprocal (the value of 1 / x, without the division).
__device__ __forceinline__ float rcp_rn(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_rn(double x) { return __drcp_rn(x); }

// rcp_rn(x) for x and 1/x well inside the normal range: an approximation
// (2 ulp) and one Newton step in fused arithmetic (Markstein 1990), the same
// bits for every one of the 2^23 significands.
__device__ __forceinline__ float rcp_normal(float x) {
  const float r = __fdividef(1.0f, x);
  return __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
}

// Marker coordinates in the working precision.  FP32 builds them from the
// split X = xo + xr (integer cell, fraction) so that the per-step kernels
// issue no FP64 instructions (a slow pipe on this GPU); FP64 subtracts the
// positions directly.
// X_j - X_k along axis d:
template <class Real>
__device__ __forceinline__ Real node_dx(const IBArgs<Real>& a, int j, int k, int d) {
  if constexpr (std::is_same<Real, float>::value)
    return (float)(a.xo[3 * j + d] - a.xo[3 * k + d]) + (a.xr[3 * j + d] - a.xr[3 * k + d]);
  else
    return a.X[3 * j + d] - a.X[3 * k + d];
}
template <class Real>
__device__ __forceinline__ V3<Real> node_dv(const IBArgs<Real>& a, int j, int k) {
  return mk<Real>(node_dx(a, j, k, 0), node_dx(a, j, k, 1), node_dx(a, j, k, 2));
}
// X_l - o along axis d for an integer o:
template <class Real>
__device__ __forceinline__ Real node_off(const IBArgs<Real>& a, int l, int d, int o) {
  if constexpr (std::is_same<Real, float>::value)
    return (float)(a.xo[3 * l + d] - o) + a.xr[3 * l + d];
  else
    return a.X[3 * l + d] - (double)o;
}
// the split of one coordinate (clamped like the marker box)
template <class Real>
__device__ __forceinline__ void split_coord(double x, int* xo, Real* xr) {
  const double v = fmax(-1e8, fmin(1e8, x));
  const double f = floor(v);
  *xo = (int)f;
  *xr = (Real)(v - f);
}

// Closest point of cell p (unwrapped) on element e, relative to the cell,
// its barycentric weights and feature (0 interior, 1..3 edge starting at
// vertex feat-1, 4..6 vertex feat-4), without branches: the plane projection when it falls inside the face, else the
// nearest of the three clamped edge projections (ties to the first edge).
// The vertices come from the step's element-relative copy (erel, eorg) and
// the edge constants from ecst, so a cell needs no division and no
// double-precision arithmetic.
template <class Real>
__device__ __forceinline__ V3<Real> elem_closest(const IBArgs<Real>& a, int e, const int4& o, const int* p, Real* beta,
                                                 int* feat) {
  const R4<Real> r = ldg4(a.erel + e), k0 = ldg4(a.ecst + 4 * e), k1 = ldg4(a.ecst + 4 * e + 1),
                 k2 = ldg4(a.ecst + 4 * e + 2), k3 = ldg4(a.ecst + 4 * e + 3);
  const Real k[16] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w, k2.x, k2.y, k2.z, k2.w, k3.x, k3.y, k3.z, k3.w};
  const V3<Real> A = mk<Real>(r.x + (Real)(o.x - p[0]), r.y + (Real)(o.y - p[1]), r.z + (Real)(o.z - p[2]));
  const V3<Real> ab = mk<Real>(k[0], k[1], k[2]);
  const V3<Real> ap = mk<Real>(-A.x, -A.y, -A.z);
  const Real d20 = dot(ap, ab);
  const Real t0 = fmin(Real(1), fmax(Real(0), d20 * k[12]));
  const V3<Real> P0 = A + t0 * ab;
  const int f0 = t0 <= Real(0) ? 4 : (t0 >= Real(1) ? 5 : 1);
  if (a.NV == 2) {
    beta[0] = Real(1) - t0;
    beta[1] = t0;
    beta[2] = 0;
    *feat = f0 == 1 ? 0 : f0;  // a segment's interior is its face
    return P0;
  }
  const V3<Real> ac = mk<Real>(k[3], k[4], k[5]), bc = mk<Real>(k[6], k[7], k[8]);
  const Real d00 = k[9], d01 = k[10], d11 = k[11];
  const Real d21 = dot(ap, ac);
  const Real t1 = fmin(Real(1), fmax(Real(0), d21 * k[13]));
  const V3<Real> P1 = A + t1 * ac;
  const V3<Real> Bv = A + ab;
  const Real t2 = fmin(Real(1), fmax(Real(0), -dot(Bv, bc) * k[14]));
  const V3<Real> P2 = Bv + t2 * bc;
  const Real D0 = dot(P0, P0), D1 = dot(P1, P1), D2 = dot(P2, P2);
  const Real v = (d11 * d20 - d01 * d21) * k[15], w = (d00 * d21 - d01 * d20) * k[15];
  const bool inside = k[15] > Real(0) && v >= Real(0) && w >= Real(0) && v + w <= Real(1);
  if (inside) {
    beta[0] = Real(1) - v - w;
    beta[1] = v;
    beta[2] = w;
    *feat = 0;
    return A + v * ab + w * ac;
  }
  const bool e1 = D1 < D0 && D1 <= D2, e2 = !e1 && D2 < D0;
  if (e2) {
    beta[0] = 0;
    beta[1] = Real(1) - t2;
    beta[2] = t2;
    *feat = t2 <= Real(0) ? 5 : (t2 >= Real(1) ? 6 : 2);
    return P2;
  }
  if (e1) {
    beta[0] = Real(1) - t1;
    beta[1] = 0;
    beta[2] = t1;
    *feat = t1 <= Real(0) ? 4 : (t1 >= Real(1) ? 6 : 3);
    return P1;
  }
  beta[0] = Real(1) - t0;
  beta[1] = t0;
  beta[2] = 0;
  *feat = f0;
  return P0;
}

// ------------------------------------------------------------ delta kernel
// eq. DiscreteDirac along one axis.
template <class Real>
__device__ __forceinline__ Real peskin(Real r) {
  Real x = fabs(r);
  if (x <= Real(1)) return (Real(3) - Real(2) * x + sqrt(fmax(Real(0), Real(1) + Real(4) * x - Real(4) * x * x))) * Real(0.125);
  if (x <= Real(2)) return (Real(5) - Real(2) * x - sqrt(fmax(Real(0), Real(-7) + Real(12) * x - Real(4) * x * x))) * Real(0.125);
  return Real(0);
}

// ------------------------------------------------------------ geometry pass
// Face normal of element e, computed from the marker positions.
template <class Real>
__device__ __forceinline__ V3<Real> face_normal(const IBArgs<Real>& a, int e) {
  if (a.NV == 2) {
    int p = a.E[2 * e], q = a.E[2 * e + 1];
    Real tx = node_dx(a, q, p, 0), tz = node_dx(a, q, p, 2);
    Real l = sqrt(tx * tx + tz * tz);
    return mk<Real>(tz / l, Real(0), -tx / l);
  }
  int p = a.E[3 * e], q = a.E[3 * e + 1], r = a.E[3 * e + 2];
  V3<Real> b = node_dv(a, q, p);
  V3<Real> c = node_dv(a, r, p);
  V3<Real> cr = cross(b, c);
  return (Real(1) / sqrt(dot(cr, cr))) * cr;
}

// Half a unit of the last place, relative.
__device__ __forceinline__ float eps_of(float) { return 0x1p-24f; }
__device__ __forceinline__ double eps_of(double) { return 0x1p-53; }

// A face whose first angle (between ab and ac) lies within 3.6 degrees of 0 or
// 180, from the Gram entries and determinant of ab and ac.  The determinant,
// d00 d11 sin^2, carries an error of a few eps d00 d11, so the barycentric
// coordinates that it gives lose eps / sin^2; below sin = 5e-4 in FP32 it may
// come out as zero or less.  Through the cross product of ab and ac they lose
// eps / sin.
constexpr float FLAT_SIN2 = 0x1p-15f;  // sin^2 up to which a face is its edges for the closest
                                       // point: within sin / 2 of its size, where the
                                       // coordinates lose eps / sin^2 (FP32: 2e-3)
template <class Real>
__device__ __forceinline__ bool thin_face(Real d00, Real d11, Real den) {
  return !(den >= rmul(rmul(d00, d11), Real(1.0 / 256)));
}

// The geometry of the step in one launch.  Threads [0, ne) store the unit
// outward face normals and what the band reads of each face.  Then 16 lanes
// per marker, one incident face each, store the vertex pseudo-normal, the
// angle-weighted sum of the incident face normals (Baerentzen and Aanaes
// 2005; in 2D the sum of the two segment normals), and in 3D the marker's
// part of the Helfrich energy: with E_v = kb |K|^2 / (8 A), K = sum_T (cot_k
// (x_v - x_j) + cot_j (x_v - x_k)) and A the mixed Voronoi area (Meyer et al.
// 2003), the derivatives dE_v/dK = kb K / (4 A) and dE_v/dA = -kb |K|^2 /
// (8 A^2), which the force of every marker around it needs (see
// node_forces_body).  Lane sums are combined by a fixed shuffle tree.
// A chain of dependent loads on few threads: 2562 markers 6 us (10 us with
// one thread per marker and no Helfrich part).
template <class Real>
__device__ __forceinline__ Real group_sum(Real v) {  // over the 16 lanes of a marker
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
TLB_HD int geometry_threads(int ne, int nn) { return (ne + 31) / 32 * 32 + 16 * nn; }
template <class Real>
__device__ __forceinline__ void geometry_body(const IBArgs<Real>& a, const Blk& blk) {
  int t = blk.x * blockDim.x + threadIdx.x;
  if (t < a.ne) {
    V3<Real> n = face_normal(a, t);
    const int* Et = a.E + a.NV * t;
    Real rv[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    int org[3];
    for (int d = 0; d < 3; ++d) {
      org[d] = a.xo[3 * Et[0] + d];
      for (int q = 0; q < a.NV; ++q) rv[q][d] = node_off(a, Et[q], d, org[d]);
    }
    a.eorg[t] = make_int4(org[0], org[1], org[2], 0);
    a.erel[t] = R4<Real>{rv[0][0], rv[0][1], rv[0][2], 0};
    // edge constants of the band's closest-point search (a segment keeps
    // ac = bc = 0)
    const V3<Real> A = mk<Real>(rv[0][0], rv[0][1], rv[0][2]), Bv = mk<Real>(rv[1][0], rv[1][1], rv[1][2]);
    const V3<Real> Cv = a.NV == 3 ? mk<Real>(rv[2][0], rv[2][1], rv[2][2]) : A;
    const V3<Real> ab = Bv - A, ac = a.NV == 3 ? Cv - A : mk<Real>(0, 0, 0), bc = a.NV == 3 ? Cv - Bv : mk<Real>(0, 0, 0);
    const Real d00 = dot(ab, ab), d01 = dot(ab, ac), d11 = dot(ac, ac), dbc = dot(bc, bc);
    const Real den = d00 * d11 - d01 * d01;
    Real reach = 0;
    if (a.NV == 3 && thin_face(d00, d11, den)) {
      const V3<Real> N = cross(ab, ac);
      const Real len = a.dc + sqrt(fmax(d00, d11));
      reach = fmin(a.dc, Real(8) * eps_of(Real(0)) * len * sqrt(rmul(d00, d11) / dot(N, N)));
    }
    a.en[t] = R4<Real>{n.x, n.y, n.z, reach};
    R4<Real>* k = a.ecst + 4 * t;
    k[0] = R4<Real>{ab.x, ab.y, ab.z, ac.x};
    k[1] = R4<Real>{ac.y, ac.z, bc.x, bc.y};
    k[2] = R4<Real>{bc.z, d00, d01, d11};
    k[3] = R4<Real>{d00 > Real(0) ? rcp_rn(d00) : Real(0), d11 > Real(0) ? rcp_rn(d11) : Real(0),
                    dbc > Real(0) ? rcp_rn(dbc) : Real(0), den > rmul(rmul(d00, d11), FLAT_SIN2) ? rcp_rn(den) : Real(0)};
    return;
  }
  if (t < (a.ne + 31) / 32 * 32) return;  // (markers start at a whole warp)
  const int g = t - (a.ne + 31) / 32 * 32, lane = g & 15;
  const bool valid = (g >> 4) < a.nn;
  const int k = valid ? g >> 4 : a.nn - 1;  // every lane takes part in the sums
  const int i0 = a.inc_off[k], ninc = valid ? a.inc_off[k + 1] - i0 : 0;
  // the marker's kernel weights at its 4 support cells along each axis, one
  // per lane (read by the spreading and by the interpolation)
  if (valid && lane < 12) {
    const int d = lane >> 2, c = a.xo[3 * k + d] - 1 + (lane & 3);
    a.wts[12 * k + lane] = d == 1 && a.dim == 2 ? Real(0) : peskin(-node_off(a, k, d, c));
  }
  V3<Real> s = mk<Real>(0, 0, 0), K = s;
  Real A = 0;
  for (int j = lane; j < ninc; j += 16) {
    const int e = a.inc[i0 + j];
    if (a.NV == 2) {
      s = s + face_normal(a, e);
      continue;
    }
    const int q0 = a.E[3 * e], q1 = a.E[3 * e + 1], q2 = a.E[3 * e + 2];
    const int u = q0 == k ? q1 : (q1 == k ? q2 : q0);
    const int v = q0 == k ? q2 : (q1 == k ? q0 : q1);
    const V3<Real> eu = node_dv(a, u, k), ev = node_dv(a, v, k), w = node_dv(a, v, u);
    const V3<Real> cr = cross(eu, ev);
    const Real A2 = sqrt(dot(cr, cr)), iA2 = Real(1) / A2;
    const Real duu = rdot(eu, eu), dvv = rdot(ev, ev), dk = rdot(eu, ev), du = -rdot(eu, w), dv = rdot(ev, w);
    const Real c = dk / sqrt(duu * dvv);
    s = s + (acos(fmin(Real(1), fmax(Real(-1), c))) * iA2) * cr;
    const Real cu = rmul(du, iA2), cv = rmul(dv, iA2);
    K = mk<Real>(rfma(-cu, ev.x, rfma(-cv, eu.x, K.x)), rfma(-cu, ev.y, rfma(-cv, eu.y, K.y)),
                 rfma(-cu, ev.z, rfma(-cv, eu.z, K.z)));
    if (dk < 0) A += Real(0.25) * A2;
    else if (du < 0 || dv < 0) A += Real(0.125) * A2;
    else A += Real(0.125) * (duu * cv + dvv * cu);
  }
  s = mk<Real>(group_sum(s.x), group_sum(s.y), group_sum(s.z));
  if (a.NV == 3) {
    K = mk<Real>(group_sum(K.x), group_sum(K.y), group_sum(K.z));
    A = group_sum(A);
  }
  if (!valid || lane != 0) return;
  a.vn[k] = R4<Real>{s.x, s.y, s.z, 0};
  if (a.NV == 3) {
    const Real kA = Real(0.25) * a.capr[a.ncaps + a.ncap[k]] / A;
    a.nadj[k] = R4<Real>{kA * K.x, kA * K.y, kA * K.z, Real(-0.5) * kA * dot(K, K) / A};
  }
}
template <class Real>
__global__ void k_geometry(const __grid_constant__ IBArgs<Real> a, int snap) {
  // start-of-step bookkeeping of the single-lattice path: clear the
  // coupling sums and, with snap, take the snapshot of the marker box and
  // reset its accumulator
  const long long n3 = 3ll * a.nn;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += (long long)gridDim.x * blockDim.x)
    a.ncpl[i] = 0;
  if (snap && blockIdx.x == 0 && threadIdx.x < 6) {
    a.box[6 + threadIdx.x] = a.box[threadIdx.x];
    a.box[threadIdx.x] = 0x7F7F7F7F;
  }
  geometry_body(a, hw_blk());
}

// Marker bounding box.  The advection kernel accumulates floor(min X) and
// -ceil(max X) per axis with integer atomicMin into box[0..5] (reset to a
// large value after use); k_fresh does the same from scratch where markers
// or the state were set from outside, and both store the split X = xo + xr of
// the positions.
template <class Real>
__device__ __forceinline__ void box_body(const IBArgs<Real>& a, const Blk& blk) {
  int k = blk.x * blockDim.x + threadIdx.x;
  if (k >= a.nn) return;
  for (int d = 0; d < 3; ++d) {
    double v = fmax(-1e8, fmin(1e8, a.X[3 * k + d]));
    atomicMin(a.box + d, (int)floor(v));
    atomicMin(a.box + 3 + d, -(int)ceil(v));
    split_coord(a.X[3 * k + d], a.xo + 3 * k + d, a.xr + 3 * k + d);
  }
}
// With the new box, the profile of a lattice without membranes: the band and
// the column fill of the step write the new box only, and cells that were
// band cells somewhere else must not keep that (see band_body).
template <class Real>
__global__ void k_fresh(const __grid_constant__ IBArgs<Real> a) {
  box_body(a, hw_blk());
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < a.G.N; i += (long long)gridDim.x * blockDim.x) {
    a.own[i] = -1;
    a.dsel[i] = -a.dc;
    a.I[i] = a.Iout;
  }
}

// The box of cells the profile visits: the step's marker box widened by
// dc + 2 cells (unwrapped; walls clamp z; at most one period per axis).
template <class Real>
__device__ __forceinline__ void profile_box(const IBArgs<Real>& a, int* lo, int* hi) {
  marker_box(a.boxc, (int)ceil(a.dc) + 2, a.G, a.dim == 2, lo, hi);
}

// Wrap a coordinate into [0, n): a compare and add within one period of the
// range, the division beyond it.
__device__ __forceinline__ int wrap_coord(int v, int n) {
  if (v < 0) v += n;
  else if (v >= n) v -= n;
  if ((unsigned)v >= (unsigned)n) {
    v %= n;
    if (v < 0) v += n;
  }
  return v;
}

template <class Real>
__device__ __forceinline__ long long cell_of(const IBArgs<Real>& a, const int* pc) {
  if (a.G.wall && (pc[2] < 0 || pc[2] >= a.G.nz)) return -1;
  const int x = wrap_coord(pc[0], a.G.nx), y = wrap_coord(pc[1], a.G.ny), z = wrap_coord(pc[2], a.G.nz);
  return ((long long)z * a.G.ny + y) * a.G.nx + x;
}

// Distance part of a scatter key (d >= 0): the distance on a grid of 2^-34;
// in FP32 the bits of d, which order as d does (from d = 2^-10 up every FP32
// value is on that grid).
__device__ __forceinline__ unsigned long long dist_code(float d) { return __float_as_uint(d); }
__device__ __forceinline__ unsigned long long dist_code(double d) {
  return (unsigned long long)(d * 17179869184.0);
}

// ------------------------------------------------------------ distance scatter
// Every cell within dc of the membrane must receive the key (distance,
// element) of its nearest element; keys are combined with atomicMin.  The
// nearest point P of a cell x lies in the interior of a face, in the
// interior of an edge or on a vertex, and x - P lies in the normal cone of
// that feature: the face normal, the wedge of the two face normals of an
// edge, the cone of the face normals around a vertex (in 2D: segment normal,
// and the fan of the two segment normals at a marker).  Each feature sweeps
// the cells x = P + t m, P on the feature, m in its cone (either sign),
// |t| < dc.  The sweep runs slice by slice along an axis k in which all cone
// generators have a component of one sign; on slice x_k = c the region lies
// in the convex hull of the points where the rays from the feature's corners
// along the generators meet the slice, whose bounding box is enumerated.
// Distances are compared on a grid of 2^-34 lattice units, ties going to the
// lowest element index.
//
// A feature offers its lowest-index face at the cell's distance to the
// feature itself: to the face's plane where the cell projects into the face,
// to the edge where it projects between the edge's ends (ends included, with
// the distance clamped to them), to the vertex.  Where P lies on the feature
// that is |x - P|; elsewhere it is a larger distance, or nothing is offered
// and the feature that holds P offers it.  The boxes are widened by 1e-3
// cells and the ends of an edge likewise, above the rounding of either test,
// so a cell on the border of two features is offered by one of them.  The
// error of a face's normal moves a cell t away by some eps (t + size) / sin in
// the face's plane, sin of its first angle: in FP32 at t = 16 by 1e-3 cells
// from half a degree down.  So thin faces take their coordinates from the
// cross product, a face without area offers nothing, and the edges and
// vertices of a thin face widen their boxes to its reach 8 eps (dc + size) /
// sin where that exceeds 1e-3.  (Without, I was off by up to 0.1 on meshes
// with needle faces.)
// So a cell costs three dot products for a face, two for an edge and one for
// a vertex, where the exact distance to the offered face took seven.
constexpr int MAXG = 12;  // generators (and faces) per feature
constexpr int SCAT_W = 4;       // slices per lane per round
constexpr int SCAT_TAB = 1024;  // cells laid out at a time
// warps per block (every lane sweeps one feature): FP64 halves them to keep
// the shared memory under the static limit
template <class Real> constexpr int scatter_warps() { return sizeof(Real) == 4 ? 4 : 2; }

// Shared memory of one warp: lane l's feature in row l.
template <class Real>
struct ScatterWarp {
  Real cb[32][9];               // corners relative to the feature's origin
  Real gk[32][MAXG];            // 1 / generator component along the slice axis
  Real ga[32][MAXG];            // generator components along the two other axes
  Real gb[32][MAXG];
  R4<Real> rec[32][3];          // what the distance needs (see offer below)
  int4 sl[32][SCAT_W];          // the round's slices: a0, b0, width, first cell
  int4 ft[32][2];               // origin cell (wrapped) and packed axes; face, first slice
  unsigned char tab[SCAT_TAB];  // slice (lane * SCAT_W + h) of each cell of the round
};

// One lane per feature, geometry in Real relative to an integer origin (the
// lattice cell below the first corner), so the FP32 build sweeps in single
// precision without losing accuracy.  The warp then shares out the cells:
// per round every lane sizes SCAT_W slices of its feature, a warp prefix sum
// lays all their cells end to end, every lane enters its slices in a table
// over them, and the lanes take the cells round-robin.  `split` virtual
// blocks set up the same features and take turns over the rounds (the set-up
// is short; the rounds are not; see scatter_split).
//
// Bound by the scattered 64-bit min reductions (lanes that walked their own
// slices, with less arithmetic but neighbouring lanes in unrelated cells, took
// 51 us): 15 360 features, dc = 10, 24 us; 35 us with the exact distance to
// the offered face and a binary search per cell.
template <class Real>
__device__ __forceinline__ void dist_scatter_body(const IBArgs<Real>& a, const Blk& blk) {
  constexpr int SW = scatter_warps<Real>();
  __shared__ ScatterWarp<Real> smw[SW];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w >= SW) return;
  ScatterWarp<Real>& sm = smw[w];
  const int nfeat = a.ne + (a.NV == 3 ? a.nedge : 0) + a.nn;
  const int grp = blk.x / a.split, phase = blk.x % a.split;
  const int f = (grp * SW + w) * 32 + lane;
  if (__ballot_sync(0xffffffffu, f < nfeat) == 0) return;
  // ---- the lane's feature: corners, cone generators (the normals of the
  // faces containing it), slice axis and range, offered face
  int kind = 0, nB = 0, nG = 0, i0 = 0, corners[3] = {0, 0, 0};
  int4 ed = make_int4(0, 0, 0, 0);  // an edge: its ends and faces
  if (f < nfeat) {
    if (f < a.ne) {  // face (3D) or segment (2D)
      nB = a.NV;
      nG = 1;
      for (int q = 0; q < a.NV; ++q) corners[q] = a.E[a.NV * f + q];
    } else if (a.NV == 3 && f < a.ne + a.nedge) {  // edge
      kind = 1;
      ed = __ldg(reinterpret_cast<const int4*>(a.edges) + (f - a.ne));
      corners[0] = ed.x;
      corners[1] = ed.y;
      nB = 2;
      nG = 2;
    } else {  // vertex
      kind = 2;
      const int v = f - a.ne - (a.NV == 3 ? a.nedge : 0);
      corners[0] = v;
      nB = 1;
      i0 = a.inc_off[v];
      nG = min(a.inc_off[v + 1] - i0, MAXG);
    }
  }
  bool ok = nG > 0;
  int o[3] = {0, 0, 0}, tmin = 0x7fffffff;
  Real S[3] = {0, 0, 0};
  const Real eps = Real(1e-3);
  Real reach = 0;  // of the faces that contain the feature; > 0: thin ones among them
  if (ok) {
    for (int d = 0; d < 3; ++d) o[d] = a.xo[3 * corners[0] + d];
    if (a.dim == 2) o[1] = 0;
    // the generators, kept as they come (components x, y, z) until the slice
    // axis is known; the read-only loads of an unrolled group are all in flight
#pragma unroll 4
    for (int j = 0; j < nG; ++j) {
      const int t = kind == 0 ? f : (kind == 1 ? (j ? ed.w : ed.z) : __ldg(a.inc + i0 + j));
      const R4<Real> n = ldg4(a.en + t);
      tmin = min(tmin, t);
      S[0] += n.x;
      S[1] += n.y;
      S[2] += n.z;
      reach = fmax(reach, n.w);
      ok &= fabs(n.x) <= Real(1.001) && fabs(n.y) <= Real(1.001) && fabs(n.z) <= Real(1.001);
      sm.gk[lane][j] = n.x;
      sm.ga[lane][j] = n.y;
      sm.gb[lane][j] = n.z;
    }
    for (int q = 0; q < nB; ++q)
      for (int d = 0; d < 3; ++d) {
        const Real b = node_off(a, corners[q], d, o[d]);
        sm.cb[lane][3 * q + d] = b;
        ok &= fabs(b) < Real(1e6);  // rejects NaN/Inf
      }
    if (!ok) atomicOr(a.status, (unsigned)ST_NAN);
  }
  // slice axis: largest component of the generator sum, all generators of one sign
  int k = 0;
  if (a.dim == 3) {
    if (fabs(S[1]) > fabs(S[k])) k = 1;
    if (fabs(S[2]) > fabs(S[k])) k = 2;
  } else {
    k = fabs(S[2]) > fabs(S[0]) ? 2 : 0;
  }
  int oa, ob;
  if (a.dim == 3) { oa = k == 0 ? 1 : 0; ob = k == 2 ? 1 : 2; }
  else { oa = k == 0 ? 2 : 0; ob = 1; }
  const Real dc = a.dc, widen = kind == 0 ? eps : fmax(eps, reach);  // of the slices' boxes
  int c0 = 0, nsl = 0;
  bool wide = false;
  if (ok) {
    Real gmin = Real(1e30f);
    Real n0[3] = {0, 0, 0};  // a face's normal
    for (int j = 0; j < nG; ++j) {
      const Real n[3] = {sm.gk[lane][j], sm.ga[lane][j], sm.gb[lane][j]};
      const Real gkj = k == 0 ? n[0] : (k == 1 ? n[1] : n[2]);
      gmin = fmin(gmin, gkj * (S[k] >= 0 ? Real(1) : Real(-1)));
      // (the rectangles are widened by eps, far above the rounding of a product)
      sm.gk[lane][j] = rcp_rn(gkj);
      sm.ga[lane][j] = oa == 0 ? n[0] : (oa == 1 ? n[1] : n[2]);
      sm.gb[lane][j] = ob == 0 ? n[0] : (ob == 1 ? n[1] : n[2]);
      if (j == 0)
        for (int d = 0; d < 3; ++d) n0[d] = n[d];
    }
    wide = gmin < Real(0.25);  // a generator nearly parallel to the slices
    Real bmin = 1e30f, bmax = -1e30f;
    for (int q = 0; q < nB; ++q) {
      bmin = fmin(bmin, sm.cb[lane][3 * q + k]);
      bmax = fmax(bmax, sm.cb[lane][3 * q + k]);
    }
    c0 = (int)ceil(bmin - dc - widen);
    nsl = (int)floor(bmax + dc + widen) - c0 + 1;
    // first corner A, then by kind: the face's normal and the vectors whose
    // products with x - A are the barycentric coordinates of the projection
    // (a segment: one), or the edge and the vector that gives its parameter
    const Real A[3] = {sm.cb[lane][0], sm.cb[lane][1], sm.cb[lane][2]};
    Real p[3] = {0, 0, 0}, q[3] = {0, 0, 0}, r[3] = {0, 0, 0};
    if (kind == 0) {
      const Real* e = &a.ecst[4 * f].x;
      const Real d00 = e[9], d01 = e[10], d11 = e[11], iden = e[15];
      for (int d = 0; d < 3; ++d) {
        p[d] = n0[d];
        q[d] = a.NV == 2 ? e[d] * e[12] : (d11 * e[d] - d01 * e[3 + d]) * iden;
        r[d] = a.NV == 2 ? Real(0) : (d00 * e[3 + d] - d01 * e[d]) * iden;
      }
      if (reach > Real(0)) {
        const V3<Real> ab = mk<Real>(e[0], e[1], e[2]), ac = mk<Real>(e[3], e[4], e[5]), N = cross(ab, ac);
        const Real inn = Real(1) / dot(N, N);
        const V3<Real> Q = inn * cross(ac, N), T = inn * cross(N, ab);
        q[0] = Q.x;
        q[1] = Q.y;
        q[2] = Q.z;
        r[0] = T.x;
        r[1] = T.y;
        r[2] = T.z;
        if (!(dot(N, N) > Real(0))) nsl = 0;
      }
    } else if (kind == 1) {
      Real l2 = 0;
      for (int d = 0; d < 3; ++d) {
        p[d] = sm.cb[lane][3 + d] - A[d];
        l2 += p[d] * p[d];
      }
      const Real il2 = l2 > Real(0) ? rcp_rn(l2) : Real(0);  // degenerate edge: its first end
      for (int d = 0; d < 3; ++d) q[d] = p[d] * il2;
    }
    sm.rec[lane][0] = R4<Real>{A[0], A[1], A[2], r[0]};
    sm.rec[lane][1] = R4<Real>{p[0], p[1], p[2], r[1]};
    sm.rec[lane][2] = R4<Real>{q[0], q[1], q[2], r[2]};
    const int ow[3] = {wrap_coord(o[0], a.G.nx), wrap_coord(o[1], a.G.ny), a.G.wall ? o[2] : wrap_coord(o[2], a.G.nz)};
    // no cell the feature can offer lies across a periodic side or a wall
    const int mg = (int)ceil(dc) + 2;
    const int n3[3] = {a.G.nx, a.G.ny, a.G.nz};
    bool inner = true;
    for (int d = 0; d < 3; ++d) {
      if (a.dim == 2 && d == 1) continue;
      Real lo = 0, hi = 0;
      for (int j = 0; j < nB; ++j) {
        lo = fmin(lo, sm.cb[lane][3 * j + d]);
        hi = fmax(hi, sm.cb[lane][3 * j + d]);
      }
      inner &= ow[d] + (int)floor(lo) - mg >= 0 && ow[d] + (int)ceil(hi) + mg < n3[d];
    }
    // (a wide or grazing cone's rectangle can reach beyond dc)
    sm.ft[lane][0] = make_int4(ow[0], ow[1], ow[2], k | (oa << 2) | (ob << 4) | (kind << 6) | (inner ? 256 : 0));
    sm.ft[lane][1] = make_int4(tmin, c0, 0, 0);
  }
  // bounding rectangle of the cone's cross-section in slice c: origin (a0,
  // b0), width wa, cnt cells (0 when empty or flagged as too wide)
  auto slice_rect = [&](int c, int& a0, int& b0, int& wa, int& cnt) {
    Real lo0 = 1e30f, hi0 = -1e30f, lo1 = 1e30f, hi1 = -1e30f;
    for (int q = 0; q < nB; ++q) {
      const Real bk = sm.cb[lane][3 * q + k], ba = sm.cb[lane][3 * q + oa], bb = sm.cb[lane][3 * q + ob];
      if (!wide) {
        for (int j = 0; j < nG; ++j) {
          const Real t = ((Real)c - bk) * sm.gk[lane][j];
          const Real pa = ba + t * sm.ga[lane][j], pb = bb + t * sm.gb[lane][j];
          lo0 = fmin(lo0, pa); hi0 = fmax(hi0, pa);
          lo1 = fmin(lo1, pb); hi1 = fmax(hi1, pb);
        }
      } else {  // conservative: the feature's box widened by dc
        lo0 = fmin(lo0, ba - dc); hi0 = fmax(hi0, ba + dc);
        lo1 = fmin(lo1, bb - dc); hi1 = fmax(hi1, bb + dc);
      }
    }
    a0 = (int)ceil(lo0 - widen);
    const int a1 = (int)floor(hi0 + widen);
    int b1 = 0;
    b0 = 0;
    if (a.dim == 3) { b0 = (int)ceil(lo1 - widen); b1 = (int)floor(hi1 + widen); }
    const int wb = b1 - b0 + 1;
    wa = a1 - a0 + 1;
    cnt = 0;
    if (wa > 0 && wb > 0) {
      if (wa > 1024 || wb > 1024) atomicOr(a.status, (unsigned)ST_OVERFLOW);  // bounded work, flagged
      else cnt = wa * wb;
    }
  };
  const int rounds = (int)__reduce_max_sync(0xffffffffu, (unsigned)((nsl + SCAT_W - 1) / SCAT_W));
  for (int r = phase; r < rounds; r += a.split) {
    int cnt[SCAT_W], tot = 0;
#pragma unroll
    for (int h = 0; h < SCAT_W; ++h) {
      const int sidx = r * SCAT_W + h;
      int a0 = 0, b0 = 0, wa = 1;
      cnt[h] = 0;
      if (sidx < nsl) slice_rect(c0 + sidx, a0, b0, wa, cnt[h]);
      sm.sl[lane][h] = make_int4(a0, b0, wa, tot);
      tot += cnt[h];
    }
    int incl = tot;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, sh);
      if (lane >= sh) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31), first = incl - tot;
#pragma unroll
    for (int h = 0; h < SCAT_W; ++h) sm.sl[lane][h].w += first;
    for (int base = 0; base < total; base += SCAT_TAB) {
      __syncwarp();
      int s = first - base;
#pragma unroll
      for (int h = 0; h < SCAT_W; ++h) {
        const int e = s + cnt[h];
        for (int i = max(s, 0); i < min(e, SCAT_TAB); ++i) sm.tab[i] = (unsigned char)(lane * SCAT_W + h);
        s = e;
      }
      __syncwarp();
      const int n = min(total - base, SCAT_TAB);
      // one cell of the round: its index and key; false if nothing is offered
      auto probe = [&](int i, long long& cell, unsigned long long& key) {
        const int id = sm.tab[i], L = id / SCAT_W, h = id % SCAT_W;
        const int4 e = sm.sl[L][h], F0 = sm.ft[L][0], F1 = sm.ft[L][1];
        const int jj = base + i - e.w;
        // jj / wa with an approximate reciprocal (__fdividef: 2 ulp, 2^-22
        // relative; the product adds 2^-24): jj < 2^20, as slice_rect holds both
        // sides to 1024, so the result is within (0.25 + 0.0625) / wa of (jj + 1/2)
        // / wa, which lies at least 1 / (2 wa) from an integer: the truncation is
        // exact
        const int qb = (int)(((float)jj + 0.5f) * __fdividef(1.0f, (float)e.z));
        const int rk = F1.y + r * SCAT_W + h, ra = e.x + (jj - qb * e.z), rb = a.dim == 3 ? e.y + qb : 0;
        // axes (k, a, b): 3D k = 0: (x, y, z); 1: (y, x, z); 2: (z, x, y); 2D the
        // plane (x, z) with b along the empty y
        const int kk = F0.w & 3;
        const bool face = (F0.w & 192) == 0;
        int rx, ry, rz;
        if (a.dim == 3) {
          rx = kk == 0 ? rk : ra;
          ry = kk == 0 ? ra : (kk == 1 ? rk : rb);
          rz = kk == 2 ? rk : rb;
        } else {
          rx = kk == 0 ? rk : ra;
          ry = 0;
          rz = kk == 0 ? ra : rk;
        }
        // one expression for the three kinds (an edge's u and a vertex's v and
        // p are zero), so that two cells are computed side by side
        const R4<Real> A = sm.rec[L][0], p = sm.rec[L][1], q = sm.rec[L][2];
        const Real ax = (Real)rx - A.x, ay = (Real)ry - A.y, az = (Real)rz - A.z;
        const Real v = ax * q.x + ay * q.y + az * q.z, u = ax * A.w + ay * p.w + az * q.w;
        const Real t = fmin(Real(1), fmax(Real(0), v));
        const Real x = ax - t * p.x, y = ay - t * p.y, z = az - t * p.z;
        const Real dist = face ? fabs(ax * p.x + ay * p.y + az * p.z) : sqrt(x * x + y * y + z * z);
        const bool on = face ? (v >= Real(0) && u >= Real(0) && v + u <= Real(1)) : (v >= -eps && v <= Real(1) + eps);
        const int pc[3] = {F0.x + rx, F0.y + ry, F0.z + rz};
        cell = ((long long)pc[2] * a.G.ny + pc[1]) * a.G.nx + pc[0];
        // (inner features: what they offer lies within dc of them, in the lattice)
        if (!(F0.w & 256)) cell = cell_of(a, pc);
        key = (dist_code(dist) << 24) | (unsigned long long)F1.x;
        return on && dist < dc && cell >= 0;
      };
      for (int i = lane; i < n; i += 64) {  // two cells at a time
        long long c0i, c1i;
        unsigned long long k0, k1;
        const bool v0 = probe(i, c0i, k0), v1 = probe(min(i + 32, n - 1), c1i, k1) && i + 32 < n;
        // no return value: fire-and-forget reductions
        if (v0) atomicMin(a.key + c0i, k0);
        if (v1) atomicMin(a.key + c1i, k1);
      }
    }
    __syncwarp();  // the next round rewrites the slice table
  }
}
// Persistent over nvb virtual blocks (grid capped by the caller).
template <class Real>
__global__ void __launch_bounds__(scatter_warps<Real>() * 32) k_dist_scatter(const __grid_constant__ IBArgs<Real> a, int nvb) {
  for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) dist_scatter_body(a, Blk{vb, 0, 0, nvb, 1, 1});
}

// Sign of x - P relative to the membrane at the closest feature (interior:
// element normal; edge: sum of the two adjacent normals; vertex: vertex
// pseudo-normal): +1 inside (d > 0 in eq. Iprofile), -1 outside.
template <class Real>
__device__ __forceinline__ Real feature_sign(const IBArgs<Real>& a, int e, const R4<Real>& n, int feat, V3<Real> xmP) {
  V3<Real> N = mk<Real>(n.x, n.y, n.z);
  if (a.NV == 3 && feat >= 1 && feat <= 3) {
    const R4<Real> m = ldg4(a.en + __ldg(a.adj + 3 * e + (feat - 1)));
    N = mk<Real>(n.x + m.x, n.y + m.y, n.z + m.z);
  } else if (feat > 0) {
    const R4<Real> m = ldg4(a.vn + __ldg(a.E + a.NV * e + feat - 4));
    N = mk<Real>(m.x, m.y, m.z);
  }
  // x - P points outward for a cell outside
  return dot(xmP, N) > Real(0) ? Real(-1) : Real(1);
}

// Fixed-point scale of the coupling sums: integer additions make the
// per-element totals independent of the order of the contributions.
#define CPL_SCALE 1125899906842624.0  // 2^50
// rint(v 2^50) as hi 2^26 + lo with |lo| <= 2^25: hi = rint(v 2^24), lo the
// rest, which is exact (v - hi 2^-24 is a multiple of v's last place below
// 2^-25) but for its own rounding, so no 64-bit conversion is needed (slow
// on this GPU).  The parts of a warp's lanes add up in 32 bits while every
// |v| < CPL_SMALL, and in 64 bits while hi holds it (|v| < CPL_SPLIT).
constexpr float CPL_SMALL = 3.9f, CPL_SPLIT = 120.0f;
__device__ __forceinline__ void cpl_split(float v, int* hi, int* lo) {
  *hi = __float2int_rn(v * 0x1p24f);
  *lo = __float2int_rn(fmaf((float)*hi, -0x1p-24f, v) * 0x1p50f);
}
__device__ __forceinline__ long long cpl_join(int hi, int lo) { return (long long)hi * (1 << 26) + lo; }
// The same of any v with the slow conversion: saturates at +-2^62 (|v| = 4096;
// a NaN too, so that it shows in the markers).
__device__ __forceinline__ long long cpl_whole(float v) {
  return __float2ll_rn(fmaxf(-4096.0f, fminf(4096.0f, v)) * 0x1p50f);
}
__device__ __forceinline__ long long cpl_fixed(double v) { return llrint(v * CPL_SCALE); }

// Band cells of the marker box (one thread per cell, x fastest): signed
// distance from the nearest element, I = (1 + tanh(d/(2 alpha)))/2 (eq.
// Iprofile), owner element, and the coupling force contributions (eq.
// DiscreteCF from eq. DiscreteCE): node k of the owner receives
//   kappa_c (psi - I) sech^2(d/(2 alpha))/(4 alpha) * (-s beta_k (x - P)/|x - P|),
// summed per marker in fixed point (lanes of a warp with the same element
// are combined before one atomic per node; a reduction per lane measured
// slower on the contended addresses).  Cells without a key are marked -1 for
// the column fill; keys are cleared for the next step.  A cell that was a
// band cell in the previous step and is not one now lies beyond dc on the
// side of its last distance (the membrane moves less than half a cell per
// step and cannot cross a cell farther than dc from it): it takes +-dc and
// I_in/I_out here, so that between fresh starts (k_fresh) the column fill,
// which would find the same sides, is not needed.
// Bound by instruction issue with part-filled warps (half the box lies outside
// the band) and the grouped reductions: radius-20 capsule, 28 us (30 us
// with 64-bit conversions and scalar loads).  Warps on compact 8 x 2 x 2 cells
// instead of rows: 23 us there, but 13% slower on coarse meshes, whose lanes
// then share elements; one warp sum per element: slower on every mesh.
template <class Real>
__device__ __forceinline__ void band_body(const IBArgs<Real>& a, const Blk& blk) {
  int blo[3], bhi[3];
  profile_box(a, blo, bhi);
  const int bx0 = blo[0], by0 = blo[1], bz0 = blo[2];
  const int wx = bhi[0] - bx0 + 1, wy = bhi[1] - by0 + 1, wz = bhi[2] - bz0 + 1;
  const long long total = (long long)wx * wy * wz;
  const bool full[3] = {wx == a.G.nx, a.dim == 3 && wy == a.G.ny, !a.G.wall && wz == a.G.nz};
  const Real ial = rcp_rn(a.alpha), Iin = a.Iin, Iout = a.Iout;
  // the box origin wrapped into the lattice: cells are indexed from it, the
  // geometry uses the unwrapped coordinates
  const int ox = wrap_coord(bx0, a.G.nx), oy = wrap_coord(by0, a.G.ny), oz = a.G.wall ? bz0 : wrap_coord(bz0, a.G.nz);
  const bool narrow = total <= 0xFFFFFFFFll;
  const long long stride = (long long)blk.gx * blockDim.x;
  for (long long t0 = (long long)blk.x * blockDim.x; t0 < total; t0 += stride) {
    const long long t = t0 + threadIdx.x;
    int e = -1;
    Real acc[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    if (t < total) {
      int ix, iy, iz;
      if (narrow) {  // 32-bit division
        const unsigned tt = (unsigned)t, row = tt / (unsigned)wx, zz = row / (unsigned)wy;
        ix = (int)(tt - row * (unsigned)wx);
        iy = (int)(row - zz * (unsigned)wy);
        iz = (int)zz;
      } else {
        ix = (int)(t % wx);
        iy = (int)((t / wx) % wy);
        iz = (int)(t / ((long long)wx * wy));
      }
      const int pc[3] = {bx0 + ix, by0 + iy, bz0 + iz};
      const int pw[3] = {ox + ix, oy + iy, oz + iz};
      long long c = cell_of(a, pw);
      if (c >= 0) {
        // psi is requested with the key, so its latency overlaps the key's
        // and the element's (it is needed only for band cells)
        const Real psic = a.psi[c * a.psi_step];
        unsigned long long key = a.key[c];
        if (key == KEY_NONE) {
          if (a.own[c] >= 0) {  // left the band since the previous step
            const bool in = a.dsel[c] > Real(0);
            a.dsel[c] = in ? a.dc : -a.dc;
            a.I[c] = in ? Iin : Iout;
          }
          a.own[c] = -1;
        } else {
          e = (int)(key & 0xFFFFFF);
          a.key[c] = KEY_NONE;
          Real beta[3];
          int feat;
          // Along an axis where the box spans a whole period a band cell may
          // sit one period away from the element that keyed it: measure from
          // the image of the cell nearest to the element (unique, as
          // periodic sides are at least 2 dc + 8).  A box narrower than the
          // period holds every band cell at that image already.
          // (the element origin, floor of its first vertex, is within a cell
          // of it: the nearest image is the same)
          int pi[3] = {pc[0], pc[1], pc[2]};
          const int4 eo = __ldg(a.eorg + e);
          const R4<Real> en = ldg4(a.en + e);
          if (full[0] | full[1] | full[2]) {
            if (full[0]) pi[0] += a.G.nx * __float2int_rn((float)(eo.x - pi[0]) / (float)a.G.nx);
            if (full[1]) pi[1] += a.G.ny * __float2int_rn((float)(eo.y - pi[1]) / (float)a.G.ny);
            if (full[2]) pi[2] += a.G.nz * __float2int_rn((float)(eo.z - pi[2]) / (float)a.G.nz);
          }
          V3<Real> P = elem_closest(a, e, eo, pi, beta, &feat);
          V3<Real> xmP = mk<Real>(-P.x, -P.y, -P.z);
          Real dist = sqrt(dot(xmP, xmP));
          Real s = feature_sign(a, e, en, feat, xmP);
          Real d = s * dist;
          // with E = exp(-|d|/alpha): I = (1 + tanh(d/(2 alpha)))/2 is 1/(1 + E)
          // inside and E/(1 + E) outside, sech^2(d/(2 alpha)) = 4 E/(1 + E)^2
          const Real E = exp(-dist * ial), iE = rcp_rn(Real(1) + E);
          const Real I = d > Real(0) ? iE : E * iE;
          a.dsel[c] = d;
          a.own[c] = e;
          a.I[c] = I;
          const Real coef = a.kc * (psic - I) * (E * iE) * (iE * ial);
          V3<Real> dir;
          if (dist > Real(1e-12)) dir = (-s / dist) * xmP;
          else dir = mk<Real>(en.x, en.y, en.z);
#pragma unroll
          for (int q = 0; q < 3; ++q) {  // beta[2] = 0 for segments
            acc[q][0] = coef * beta[q] * dir.x;
            acc[q][1] = coef * beta[q] * dir.y;
            acc[q][2] = coef * beta[q] * dir.z;
          }
        }
      }
    }
    // combine lanes that share an element, one fixed-point atomic per group
    const unsigned active = __ballot_sync(0xffffffffu, e >= 0);
    if (e >= 0) {
      const unsigned grp = __match_any_sync(active, e);
      const int leader = __ffs(grp) - 1;
      const int lane = threadIdx.x & 31;
      long long sum[9];
      if constexpr (std::is_same<Real, float>::value) {
        bool small = true;
        int hi[9], lo[9], sh[9], sl[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const float v = acc[i / 3][i % 3];
          small &= fabsf(v) < CPL_SMALL;
          cpl_split(v, hi + i, lo + i);
          sh[i] = sl[i] = 0;
          sum[i] = 0;
        }
        if (__all_sync(active, small)) {
          // sum over the group (integers: any order gives the same total)
          for (unsigned m = grp; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              sh[i] += __shfl_sync(grp, hi[i], src);
              sl[i] += __shfl_sync(grp, lo[i], src);
            }
          }
#pragma unroll
          for (int i = 0; i < 9; ++i) sum[i] = cpl_join(sh[i], sl[i]);
        } else {
          // (what hi cannot hold goes straight to the marker; converting all
          // lanes' values whole instead took the band of a 240x120 ring from 9
          // to 12 us, though no value was that large)
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            const float v = acc[i / 3][i % 3];
            if (fabsf(v) < CPL_SPLIT) continue;
            if (i / 3 < a.NV) atomicAdd(a.ncpl + 3 * a.E[a.NV * e + i / 3] + i % 3, (unsigned long long)cpl_whole(v));
            hi[i] = lo[i] = 0;
          }
          for (unsigned m = grp; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
#pragma unroll
            for (int i = 0; i < 9; ++i)
              sum[i] += cpl_join(__shfl_sync(grp, hi[i], src), __shfl_sync(grp, lo[i], src));
          }
        }
      } else {
        long long v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          v[i] = cpl_fixed((double)acc[i / 3][i % 3]);
          sum[i] = 0;
        }
        for (unsigned m = grp; m; m &= m - 1) {
          const int src = __ffs(m) - 1;
#pragma unroll
          for (int i = 0; i < 9; ++i) sum[i] += __shfl_sync(grp, v[i], src);
        }
      }
      if (lane == leader) {  // straight to the element's nodes
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          if (q >= a.NV) break;
          const int node = a.E[a.NV * e + q];
#pragma unroll
          for (int d = 0; d < 3; ++d)
            if (sum[3 * q + d] != 0) atomicAdd(a.ncpl + 3 * node + d, (unsigned long long)sum[3 * q + d]);
        }
      }
    }
  }
}
template <class Real>
__global__ void k_band(const __grid_constant__ IBArgs<Real> a) {
  band_body(a, hw_blk());
}

// Cells of the box farther than dc from the membrane: one warp per column
// along z, 32 cells at a time.  A cell outside the band takes the side of
// the nearest band cell below it (the membrane cannot be crossed between two
// cells that are both farther than dc from it; the bottom of the box is
// outside every capsule): d = +dc inside, -dc outside.
template <class Real>
__device__ __forceinline__ void fill_body(const IBArgs<Real>& a, const Blk& blk) {
  int blo[3], bhi[3];
  profile_box(a, blo, bhi);
  const int bx0 = blo[0], by0 = blo[1], bz0 = blo[2];
  const int wx = bhi[0] - bx0 + 1, wy = bhi[1] - by0 + 1, wz = bhi[2] - bz0 + 1;
  const int col = (blk.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (col >= wx * wy) return;
  const Real dc = a.dc, Iin = a.Iin, Iout = a.Iout;
  const Geo& G = a.G;
  const long long colc = (long long)wrap_coord(by0 + col / wx, G.ny) * G.nx + wrap_coord(bx0 + col % wx, G.nx);
  const long long plane = (long long)G.nx * G.ny;
  bool inside = false;  // status carried from the chunk below
  for (int z0 = 0; z0 < wz; z0 += 128) {
    // the loads of up to four chunks of 32 cells first (dsel is read for
    // every cell, used for band cells only), then the scans
    long long cq[4];
    int ownq[4];
    Real dq[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int z = z0 + 32 * q + lane, pz = bz0 + z;
      cq[q] = -1;
      ownq[q] = -1;
      dq[q] = 0;
      if (z < wz && (!G.wall || (pz >= 0 && pz < G.nz))) {
        cq[q] = (long long)(G.wall ? pz : wrap_coord(pz, G.nz)) * plane + colc;
        ownq[q] = a.own[cq[q]];
        dq[q] = a.dsel[cq[q]];
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (z0 + 32 * q >= wz) break;
      const long long c = cq[q];
      const bool band = c >= 0 && ownq[q] >= 0, sgn = band && dq[q] > Real(0);
      const unsigned bm = __ballot_sync(0xffffffffu, band);
      const unsigned sm = __ballot_sync(0xffffffffu, sgn);
      const unsigned below = bm & ((1u << lane) - 1u);
      const bool my = below ? ((sm >> (31 - __clz(below))) & 1u) : inside;
      if (c >= 0 && !band) {
        a.dsel[c] = my ? dc : -dc;
        a.I[c] = my ? Iin : Iout;
      }
      // carry: the status at the top band cell of the chunk
      inside = bm ? ((sm >> (31 - __clz(bm))) & 1u) : inside;
    }
  }
}
template <class Real>
__global__ void k_fill(const __grid_constant__ IBArgs<Real> a) {
  fill_body(a, hw_blk());
}

// ------------------------------------------------------------ elastic forces
// Elastic node forces, 16 lanes per marker, summed by a fixed shuffle tree.
// They depend on the marker positions only; the coupling force joins them in
// k_spread.
//
// 3D: lane j takes incident face j = (k, u, v), whose energy as a function of
// X_k is its Skalak energy A0 W, W = (G/4)(I1^2 + 2 I1 - 2 I2 + C I2^2) with
// I1 = tr(G0^-1 g) - 2, I2 = det(G0^-1 g) - 1 of the edge metric g, plus its
// share of the three vertices' bending energies.  The bending energies are
// functions of the sums K_v and A_v, whose derivatives (nadj) are known from
// the geometry pass, so face (k, u, v) contributes the derivative of
//   cot_v P_v + cot_u P_u + cot_k P_k,   P_v = (x_k - x_u).(K'_k - K'_u) +
//   |x_k - x_u|^2 (A'_k + A'_u)/8 and cyclically
// (an obtuse face's areas are A2/4 or A2/8 times the A' instead, A2 twice its
// area), with cot_i = d_i / A2.  (Each marker used to differentiate the
// energies of its whole 1-ring, 42 face terms in dual numbers, for 18 that
// depend on it: 17 us for 2562 markers with 32 lanes each, now 5.5.)
// 2D: lanes 0 and 1 the two segments (eq. DiscreteSE), lanes 2..4 the bending
// at the previous marker, this one and the next (eqs. DiscreteBE,
// DiscreteTheta, DiscreteArcLength).
template <class Real>
__device__ __forceinline__ V3<Real> ring_force(const IBArgs<Real>& a, int k, int lane) {
  const int cap = a.ncap[k];
  const Real ks = a.capr[cap], kb = a.capr[a.ncaps + cap];
  if (lane < 2) {
    const int e = a.inc[a.inc_off[k] + lane];
    const int p = a.E[2 * e], q = a.E[2 * e + 1];
    const Real tx = node_dx(a, q, p, 0), tz = node_dx(a, q, p, 2);
    const Real L = sqrt(tx * tx + tz * tz);
    const Real T = ks * (L / (Real)a.ds0[e] - Real(1)) / L;
    const Real sgn = (p == k) ? Real(1) : Real(-1);  // -dE/dX_p = +T t ; -dE/dX_q = -T t
    return mk<Real>(sgn * T * tx, Real(0), sgn * T * tz);
  }
  const int m = lane == 2 ? a.rprev[k] : (lane == 3 ? k : a.rnext[k]);
  const int mp = a.rnext[m], mq = a.rprev[m];
  const Real ax = node_dx(a, mp, m, 0), az = node_dx(a, mp, m, 2);
  const Real bx = node_dx(a, m, mq, 0), bz = node_dx(a, m, mq, 2);
  const Real la = sqrt(ax * ax + az * az), lb = sqrt(bx * bx + bz * bz);
  const Real ab = ax * bx + az * bz;
  const Real cr = ax * bz - az * bx;
  // theta1 = arccos(a.b / |a||b|), evaluated as atan2(|a x b|, a.b)
  const Real th = atan2(fabs(cr), ab);
  const Real sn = fabs(cr) / (la * lb);
  const Real ratio = th < Real(1e-4) ? Real(1) + th * th / Real(6) : th / sn;
  const Real dsp = la + lb;
  const Real k1 = Real(0.25) * kb * (Real(-8) * ratio / dsp);
  const Real dth = Real(2) * th;
  const Real k2 = Real(0.25) * kb * (dth / dsp) * (dth / dsp);
  const Real iab = Real(1) / (la * lb);
  const Real dya_x = bx * iab - ab * ax * iab / (la * la), dya_z = bz * iab - ab * az * iab / (la * la);
  const Real dyb_x = ax * iab - ab * bx * iab / (lb * lb), dyb_z = az * iab - ab * bz * iab / (lb * lb);
  Real gx = 0, gz = 0;
  if (k == mp) { gx += k1 * dya_x - k2 * ax / la; gz += k1 * dya_z - k2 * az / la; }
  if (k == m) {
    gx += k1 * (dyb_x - dya_x) - k2 * (bx / lb - ax / la);
    gz += k1 * (dyb_z - dya_z) - k2 * (bz / lb - az / la);
  }
  if (k == mq) { gx += -k1 * dyb_x + k2 * bx / lb; gz += -k1 * dyb_z + k2 * bz / lb; }
  return mk<Real>(-gx, Real(0), -gz);
}
template <class Real>
__device__ __forceinline__ V3<Real> face_force(const IBArgs<Real>& a, int k, int e) {
  const int q0 = a.E[3 * e], q1 = a.E[3 * e + 1], q2 = a.E[3 * e + 2];
  const int u = q0 == k ? q1 : (q1 == k ? q2 : q0);
  const int v = q0 == k ? q2 : (q1 == k ? q0 : q1);
  const V3<Real> eu = node_dv(a, u, k), ev = node_dv(a, v, k), w = node_dv(a, v, u);
  const R4<Real> Nk = a.nadj[k], Nu = a.nadj[u], Nv = a.nadj[v];
  const Real duu = rdot(eu, eu), dvv = rdot(ev, ev), dk = rdot(eu, ev), dww = rdot(w, w);
  // bending
  const V3<Real> cr = cross(eu, ev);
  const Real A2 = sqrt(dot(cr, cr)), iA2 = Real(1) / A2;
  const Real du = -rdot(eu, w), dv = rdot(ev, w);
  const Real ck = dk * iA2, cu = du * iA2, cv = dv * iA2;
  const V3<Real> Ku = mk<Real>(Nk.x - Nu.x, Nk.y - Nu.y, Nk.z - Nu.z), Kv = mk<Real>(Nk.x - Nv.x, Nk.y - Nv.y, Nk.z - Nv.z);
  const V3<Real> Kw = mk<Real>(Nu.x - Nv.x, Nu.y - Nv.y, Nu.z - Nv.z);
  Real Pv = -dot(eu, Ku), Pu = -dot(ev, Kv), Pk = -dot(w, Kw), S = 0;  // S: factor of A2
  V3<Real> g = cv * Ku + cu * Kv;  // the cotangents times dP
  if (dk < 0 || du < 0 || dv < 0) {
    S = (dk < 0 ? Real(0.25) : Real(0.125)) * Nk.w + (du < 0 ? Real(0.25) : Real(0.125)) * Nu.w +
        (dv < 0 ? Real(0.25) : Real(0.125)) * Nv.w;
  } else {
    const Real au = Real(0.125) * (Nk.w + Nu.w), av = Real(0.125) * (Nk.w + Nv.w);
    Pv += duu * au;
    Pu += dvv * av;
    Pk += dww * Real(0.125) * (Nu.w + Nv.w);
    g = g - (Real(2) * cv * au) * eu - (Real(2) * cu * av) * ev;
  }
  // d(d_k) = -(eu + ev), d(d_u) = w, d(d_v) = -w, dA2 = n x w
  const V3<Real> dA = iA2 * cross(cr, w);
  g = g + (iA2 * (Pu - Pv)) * w - (iA2 * Pk) * (eu + ev) + (S - iA2 * (cv * Pv + cu * Pu + ck * Pk)) * dA;
  // Skalak: with the metric of the edges from the face's first vertex,
  // dE = D1 dI1 + D2 dI2
  const Real* c = a.skc + 5 * e;
  const int cap = a.ecap[e];
  const Real G = a.capr[2 * a.ncaps + cap], C = a.capr[3 * a.ncaps + cap];
  // e1, e2 of the face in terms of (eu, ev): first vertex k: (eu, ev); v: (-ev,
  // -w) (to k and u); u: (w, -eu) (to v and k)
  const V3<Real> e1 = q0 == k ? eu : (q1 == k ? Real(-1) * ev : w);
  const V3<Real> e2 = q0 == k ? ev : (q1 == k ? Real(-1) * w : Real(-1) * eu);
  const Real g11 = q0 == k ? duu : (q1 == k ? dvv : dww), g22 = q0 == k ? dvv : (q1 == k ? dww : duu);
  const Real g12 = rdot(e1, e2);
  const Real I1 = rfma(c[2], g22, rfma(c[1], g12, rfma(c[0], g11, Real(-2))));
  const Real I2 = rfma(c[3], rfma(g11, g22, -rmul(g12, g12)), Real(-1));
  const Real q = c[4] * G * Real(0.5);
  const Real D1 = q * (I1 + Real(1)), D2 = q * (C * I2 - Real(1)) * c[3];
  const Real h11 = Real(2) * (D1 * c[0] + D2 * g22), h22 = Real(2) * (D1 * c[2] + D2 * g11), h12 = D1 * c[1] - Real(2) * D2 * g12;
  const V3<Real> f1 = h11 * e1 + h12 * e2, f2 = h22 * e2 + h12 * e1;  // dE/de1, dE/de2
  const V3<Real> sk = q0 == k ? Real(-1) * (f1 + f2) : (q1 == k ? f1 : f2);
  return Real(-1) * (g + sk);
}
template <class Real>
__device__ __forceinline__ void node_forces_body(const IBArgs<Real>& a, const Blk& blk) {
  const int t = blk.x * blockDim.x + threadIdx.x, lane = t & 15;
  const bool valid = (t >> 4) < a.nn;
  const int k = valid ? t >> 4 : a.nn - 1;
  V3<Real> F = mk<Real>(0, 0, 0);
  if (valid) {
    if (a.NV == 2) {
      if (lane < 5) F = ring_force(a, k, lane);
    } else {
      const int i0 = a.inc_off[k], ninc = a.inc_off[k + 1] - i0;
      for (int j = lane; j < ninc; j += 16) F = F + face_force(a, k, a.inc[i0 + j]);
    }
  }
  F = mk<Real>(group_sum(F.x), group_sum(F.y), group_sum(F.z));
  if (!valid || lane != 0) return;
  a.F[3 * k] = F.x;
  a.F[3 * k + 1] = a.dim == 2 ? Real(0) : F.y;
  a.F[3 * k + 2] = F.z;
}
template <class Real>
__global__ void k_node_forces(const __grid_constant__ IBArgs<Real> a) {
  node_forces_body(a, hw_blk());
}

// Coupling force on marker k from its fixed-point sum (integer totals, so
// the result does not depend on the order of the contributions).
template <class Real>
__device__ __forceinline__ void coupling_of(const IBArgs<Real>& a, int k, Real* out) {
  long long cpl[3];
  for (int d = 0; d < 3; ++d) cpl[d] = (long long)a.ncpl[3 * k + d];
  for (int d = 0; d < 3; ++d) {
    if constexpr (std::is_same<Real, float>::value)  // one rounding either way
      out[d] = __ll2float_rn(cpl[d]) * 0x1p-50f;
    else
      out[d] = (Real)((double)cpl[d] / CPL_SCALE);
  }
  if (a.dim == 2) out[1] = 0;
}

// ------------------------------------------------------------ spreading
// Distinct bricks touched along one axis by the 4 support cells starting at base.
__device__ __forceinline__ int axis_bricks(int base, int n, int* out) {
  int m = 0;
  for (int s = 0; s < 4; ++s) {
    int c = ((base + s) % n + n) % n;
    int b = c / BRICK;
    bool dup = false;
    for (int j = 0; j < m; ++j) dup |= out[j] == b;
    if (!dup) out[m++] = b;
  }
  return m;
}

template <class Real>
__device__ __forceinline__ int node_bricks(const IBArgs<Real>& a, int l, int* out) {
  int bx[4], by[4], bz[4];
  int nxb = axis_bricks(a.xo[3 * l] - 1, a.G.nx, bx);
  int nyb = 1;
  by[0] = 0;
  if (a.dim == 3) nyb = axis_bricks(a.xo[3 * l + 1] - 1, a.G.ny, by);
  int nzb = axis_bricks(a.xo[3 * l + 2] - 1, a.G.nz, bz);
  int m = 0;
  for (int i = 0; i < nxb; ++i)
    for (int j = 0; j < nyb; ++j)
      for (int k = 0; k < nzb; ++k) out[m++] = (bz[k] * a.nby + by[j]) * a.nbx + bx[i];
  return m;
}

template <class Real>
__device__ __forceinline__ void brick_count_body(const IBArgs<Real>& a, const Blk& blk) {
  int l = blk.x * blockDim.x + threadIdx.x;
  if (l >= a.nn) return;
  int b[64];
  int m = node_bricks(a, l, b);
  for (int j = 0; j < m; ++j) atomicAdd(a.bcnt + b[j], 1);
}
template <class Real>
__global__ void k_brick_count(const __grid_constant__ IBArgs<Real> a) {
  if (blockIdx.x == 0 && threadIdx.x < 2) a.ctr[threadIdx.x] = 0;  // the brick compaction's counters
  brick_count_body(a, hw_blk());
}

// Bricks holding markers now or in the previous step join the active list;
// each claims a contiguous slot range for its marker list.
template <class Real>
__device__ __forceinline__ void brick_compact_body(const IBArgs<Real>& a, const Blk& blk) {
  int b = blk.x * blockDim.x + threadIdx.x;
  if (b >= a.nbricks) return;
  int c = a.bcnt[b];
  a.bflag[b] = c > 0;
  if (c == 0 && a.bprev[b] == 0) return;
  int i = atomicAdd(a.ctr, 1);
  a.bact[i] = b;
  a.boff[b] = atomicAdd(a.ctr + 1, c);
}
template <class Real>
__global__ void k_brick_compact(const __grid_constant__ IBArgs<Real> a) {
  brick_compact_body(a, hw_blk());
}

template <class Real>
__device__ __forceinline__ void brick_fill_body(const IBArgs<Real>& a, const Blk& blk) {
  int l = blk.x * blockDim.x + threadIdx.x;
  if (l >= a.nn) return;
  int b[64];
  int m = node_bricks(a, l, b);
  for (int j = 0; j < m; ++j) {
    int s = atomicAdd(a.bcur + b[j], 1);
    if (s >= a.bcnt[b[j]]) {  // count and fill disagree: flag, never write past the range
      atomicOr(a.status, (unsigned)ST_OVERFLOW);
      continue;
    }
    a.blist[a.boff[b[j]] + s] = l;
  }
}
template <class Real>
__global__ void k_brick_fill(const __grid_constant__ IBArgs<Real> a) {
  brick_fill_body(a, hw_blk());
}

// Each cell of an active brick sums F_l delta_h(x - X_l) over the brick's
// markers in ascending marker order (the list is sorted first, so the result
// does not depend on the order of the atomic slot claims).  Bricks that held
// markers in the previous step are visited too, so their cells return to zero.
// One warp per brick: its work is a chain of dependent loads (brick, list,
// markers), so many small chains beside each other beat a block with barriers
// per brick (24 2D lattices of 240x120, batched: 17.9 -> 10.3 us).
constexpr int SPREAD_WARPS = 4;  // per block (at most)
template <class Real>
__device__ __forceinline__ void spread_body(const IBArgs<Real>& a, const Blk& blk) {
  constexpr int CH = 32;  // markers staged at a time, one per lane
  __shared__ int s_list[SPREAD_WARPS][2][512];
  __shared__ Real s_w[SPREAD_WARPS][CH][13];  // delta_h at the brick's 4 cells along x, y, z
  __shared__ Real s_f[SPREAD_WARPS][CH][3];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  int *list = s_list[w][0], *sorted = s_list[w][1];
  const int nact = min(a.ctr[0], a.nbricks);
  // the lane's cells of the brick: 3D (x, y, z) and (x, y, z + 2), 2D one of 16
  const int lx = lane & 3, ly = a.dim == 3 ? (lane >> 2) & 3 : 0, lz = a.dim == 3 ? lane >> 4 : (lane >> 2) & 3;
  const int ncell = a.dim == 3 ? 2 : (lane < 16 ? 1 : 0);
  for (int ib = blk.x * nw + w; ib < nact; ib += blk.gx * nw) {
    const int b = a.bact[ib];
    if (b < 0 || b >= a.nbricks) continue;
    const int cnt = a.bcnt[b], off = a.boff[b], m = min(cnt, 512);
    if (cnt > 512 && lane == 0) atomicOr(a.status, (unsigned)ST_OVERFLOW);
    for (int j = lane; j < m; j += 32) list[j] = a.blist[off + j];
    __syncwarp();
    // rank sort (marker indices are distinct), so the sum runs in marker order
    for (int j = lane; j < m; j += 32) {
      const int v = list[j];
      int r = 0;
      for (int i = 0; i < m; ++i) r += list[i] < v;
      sorted[r] = v;
    }
    __syncwarp();
    const int o[3] = {b % a.nbx * BRICK, a.dim == 3 ? b / a.nbx % a.nby * BRICK : 0, b / (a.nbx * a.nby) * BRICK};
    Real f[2][3] = {{0, 0, 0}, {0, 0, 0}};
    for (int j0 = 0; j0 < m; j0 += CH) {
      const int mc = min(CH, m - j0);
      if (lane < mc) {
        const int l = sorted[j0 + lane];
        // brick cell c along axis d is support cell c + sh (nearest periodic
        // image of the marker); outside the support the kernel is zero
        auto img = [](int k, int n) { return wrap_coord(k + n / 2, n) - n / 2; };
        const int n3[3] = {a.G.nx, a.G.ny, a.G.nz};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int rel = a.xo[3 * l + d] - o[d];
          const int sh = 1 - (d == 2 && a.G.wall ? rel : img(rel, n3[d]));
#pragma unroll
          for (int c = 0; c < BRICK; ++c)
            s_w[w][lane][4 * d + c] = (unsigned)(c + sh) < 4u ? a.wts[12 * l + 4 * d + c + sh] : Real(0);
        }
        Real cp[3];
        coupling_of(a, l, cp);  // F_mem = F_s + F_b + F_c (eq. MembraneForces)
        for (int d = 0; d < 3; ++d) s_f[w][lane][d] = a.F[3 * l + d] + cp[d];
      }
      __syncwarp();
      for (int j = 0; j < mc; ++j) {  // in marker order across the chunks
        const Real* W = s_w[w][j];
        const Real* F = s_f[w][j];
        const Real xy = a.dim == 3 ? W[lx] * W[4 + ly] : W[lx];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const Real wgt = xy * W[8 + ((lz + 2 * h) & 3)];
          for (int d = 0; d < 3; ++d) f[h][d] += wgt * F[d];
        }
      }
      __syncwarp();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int cx = o[0] + lx, cy = o[1] + ly, cz = o[2] + lz + 2 * h;
      if (h < ncell && cx < a.G.nx && cy < a.G.ny && cz < a.G.nz) {
        const long long c = ((long long)cz * a.G.ny + cy) * a.G.nx + cx;
        for (int d = 0; d < 3; ++d) a.fib[d * a.G.P + c] = f[h][d];
      }
    }
    if (lane == 0) {
      a.bprev[b] = cnt;
      a.bcnt[b] = 0;
      a.bcur[b] = 0;
    }
    __syncwarp();
  }
}
template <class Real>
__global__ void k_spread(const __grid_constant__ IBArgs<Real> a) {
  spread_body(a, hw_blk());
}

// ------------------------------------------------------------ interpolation
// One warp per marker: v(t+1) = (j' + F/2)/rho' on the 4^d support cells
// from the streamed populations and the force of the step, weighted by
// delta_h, reduced over the warp; then X += U (explicit Euler).
template <class L, int MODE>
__device__ __forceinline__ void interp_advect_body(const IBArgs<typename Prec<MODE>::Real>& a,
                                                   const typename Prec<MODE>::Store* lo, const Blk& blk) {
  using Real = typename Prec<MODE>::Real;
  int l = (blk.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (l >= a.nn) return;
  const Geo G = a.G;
  const int bb[3] = {a.xo[3 * l] - 1, a.xo[3 * l + 1] - 1, a.xo[3 * l + 2] - 1};
  // delta_h along each axis at the 4 support offsets: lane 4 d + o
  const Real wax = lane < 12 ? a.wts[12 * l + lane] : Real(0);
  const int ncell = a.dim == 3 ? 64 : 16;
  // the lane's two support cells: weights and addresses first, so that all
  // their loads are in flight together (a cell of weight 0 reads cell 0)
  Real w[2];
  int cx[2], cy[2], cz[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int s = lane + 32 * h;
    const int ox = s % 4, oy = a.dim == 3 ? (s / 4) % 4 : 0, oz = a.dim == 3 ? s / 16 : (s / 4) % 4;
    w[h] = __shfl_sync(0xffffffffu, wax, ox) * __shfl_sync(0xffffffffu, wax, 8 + oz);
    if (a.dim == 3) w[h] *= __shfl_sync(0xffffffffu, wax, 4 + oy);
    const int px = bb[0] + ox, py = a.dim == 3 ? bb[1] + oy : 0, pz = bb[2] + oz;
    const bool ok = s < ncell && w[h] != Real(0) && !(G.wall && (pz < 0 || pz >= G.nz));
    if (!ok) w[h] = 0;
    cx[h] = ok ? wrap_coord(px, G.nx) : 0;
    cy[h] = ok ? wrap_coord(py, G.ny) : 0;
    cz[h] = ok ? wrap_coord(pz, G.nz) : 0;
  }
  Real U[3] = {0, 0, 0};
  if (a.M) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const Nbr<L> nb(G, cx[h], cy[h], cz[h]);
      R4<Real> src[L::Q];
#pragma unroll
      for (int i = 0; i < L::Q; ++i) src[i] = ldg4(a.M + M_F * G.P32 + nb.src(i));
      Real ft[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) ft[d] = a.ftot[d * G.P + nb.self];
      Real r = 0, j[3] = {0, 0, 0};
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        EqCell<L, MODE> e;
        // (the 1/rho that the collide stored: in FP32 formed again, as gathering
        // them took the kernel from 11 to 13 us)
        if constexpr (std::is_same<Real, float>::value) e.set_f(src[i], rcp_normal(1.0f + src[i].x));
        else e.set_f(src[i], __ldg(&a.M[M_V * G.P32 + nb.src(i)].w));
        const Real fi = e.f_or_back(i, nb.bounce(i));
        r += fi;
        if (L::cx(i)) j[0] += L::cx(i) > 0 ? fi : -fi;
        if (L::cy(i)) j[1] += L::cy(i) > 0 ? fi : -fi;
        if (L::cz(i)) j[2] += L::cz(i) > 0 ? fi : -fi;
      }
      Real rho = Real(1) + r;
      if (w[h] != Real(0))
        for (int d = 0; d < 3; ++d) U[d] += w[h] * (j[d] + Real(0.5) * ft[d]) / rho;
    }
  } else {
    // the populations of both support cells (and their forces) are all
    // requested before the first sum, so their latencies overlap
    Real fv[2][L::Q], ft[2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const Nbr<L> nb(G, cx[h], cy[h], cz[h]);
#pragma unroll
      for (int i = 0; i < L::Q; ++i) fv[h][i] = to_real(__ldg(lo + nb.off(i, plane_f<L>(i), plane_f<L>(L::opp(i)), G.P32)));
#pragma unroll
      for (int d = 0; d < 3; ++d) ft[h][d] = __ldg(a.ftot + d * G.P + nb.self);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      Real r = 0, j[3] = {0, 0, 0};
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        const Real fi = fv[h][i];
        r += fi;
        if (L::cx(i)) j[0] += L::cx(i) > 0 ? fi : -fi;
        if (L::cy(i)) j[1] += L::cy(i) > 0 ? fi : -fi;
        if (L::cz(i)) j[2] += L::cz(i) > 0 ? fi : -fi;
      }
      Real rho = Real(1) + r;
      if (w[h] != Real(0))
        for (int d = 0; d < 3; ++d) U[d] += w[h] * (j[d] + Real(0.5) * ft[h][d]) / rho;
    }
  }
  for (int d = 0; d < 3; ++d)
    for (int o = 16; o > 0; o >>= 1) U[d] += __shfl_xor_sync(0xffffffffu, U[d], o);
  // lane 0's totals (each lane's butterfly sums in its own order)
  for (int d = 0; d < 3; ++d) U[d] = __shfl_sync(0xffffffffu, U[d], 0);
  if (a.dim == 2) U[1] = 0;
  if (lane == 0 && !(fabs(U[0]) < Real(0.5) && fabs(U[1]) < Real(0.5) && fabs(U[2]) < Real(0.5)))
    atomicOr(a.status, (unsigned)ST_MARKER_JUMP);
  if (lane < 3) {  // lane d advances coordinate d
    const int d = lane;
    const Real Ud = d == 0 ? U[0] : (d == 1 ? U[1] : U[2]);
    const double Xn = a.X[3 * l + d] + (double)Ud;
    a.X[3 * l + d] = Xn;
    double v = fmax(-1e8, fmin(1e8, Xn));
    atomicMin(a.box + d, (int)floor(v));
    atomicMin(a.box + 3 + d, -(int)ceil(v));
    split_coord(Xn, a.xo + 3 * l + d, a.xr + 3 * l + d);
  }
}
template <class L, int MODE>
__global__ void k_interp_advect(const __grid_constant__ IBArgs<typename Prec<MODE>::Real> a,
                                const typename Prec<MODE>::Store* lo) {
  interp_advect_body<L, MODE>(a, lo, hw_blk());
}

// FP64 capsule measures: 2D enclosed area (shoelace in the internal x-z
// plane); 3D surface area and enclosed volume (divergence theorem).
__global__ void k_capsule_measures(const double* X, const int* E, const int* ecap, int ne, int NV, int ncap,
                                   double* out /* [ncap][2] */);
