// quad.cu -- 2-D and axisymmetric variants (arXiv:1708.08434, Sec. 1 and
// 2.1.1: quadtree grids; Sec. 2.1.2 multigrid; Sec. 2.2-2.4 fluid step) on a
// quadtree of 8^2-cell boxes, in Cartesian (x, y) or cylindrical (r, z)
// coordinates.
//
// The initial mesh's tables are built by host C++ (proper nesting, Morton
// order per level) and copied into the arena; a regrid forms the new box set
// and its tables on the device (k_qrg_*) and the host keeps a copy of them
// for its own queries.  Every field operation runs in the kernels below,
// one warp per box: the box and the ghost layer a kernel needs are staged in
// shared memory, with coarse values at refinement boundaries read through
// the parent's 8-neighbour table (proper nesting guarantees every coarse
// cell a ghost or a prolongation needs lies in the parent or one of its
// neighbours).
//
// Discretisation (the paper gives no 2-D or cylindrical formulas; these are
// the finite-volume forms of the 3-D rules):
//   L phi = [w_lo (phi_W - phi) + w_hi (phi_E - phi) + (phi_S - phi) + (phi_N - phi)] / h^2
// with w_lo = r_{i-1/2}/r_i, w_hi = r_{i+1/2}/r_i in cylindrical coordinates
// (r at (index + 1/2) h from the axis, so w_lo = 0 on the axis) and 1 in
// Cartesian; red-black Gauss-Seidel solves the cell's row of that operator;
// restriction is the volume-weighted mean of the four children (weights
// proportional to the centre radius); prolongation (2c + c_x + c_y)/4;
// coarse-fine potential ghost phi_f/3 + 2 phihat/3, phihat = 3/4 c + 1/4 c_t;
// fluxes as in 3-D with the radial divergence weighted like L and the
// coarse flux at a refinement boundary the area-weighted mean of the two
// fine fluxes.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <utility>
#include <vector>

#include "fluid_dev.cuh"
#include "sm_quad.h"
#include "sm_nvtx.h"

using sm::Table;
using sm::dabs;
using sm::dbits;
using sm::face_flux_d;
using sm::half_index;
using sm::halve;
using sm::index_split;
using sm::size_bits;
using sm::sqrt_newton;

namespace {

constexpr int QN = 8;            // cells per box side
constexpr int QC = QN * QN;      // cells per box
constexpr int WPB = 4;           // boxes (warps) per block
constexpr int QT = 32 * WPB;     // threads per block
constexpr int QMAXL = SM_MAX_LEVELS;
constexpr int S1 = QN + 2;       // staged side with one ghost layer
constexpr int S2 = QN + 4;       // staged side with two ghost layers

// fields in the arena: the public sm_var numbering first (V_ZERO is never
// written: the potential of the residuals' denominator)
enum { V_PHI = 0, V_RHS, V_RES, V_NE, V_NI, V_EMAG, V_RHO, V_OLD, V_ZERO, V_NE1, V_NI1, NV };

struct QBc {
  int type[4];      // 0 Neumann zero (and the axis), 1 Dirichlet
  double g2[4];     // 2 g
};

struct QTabs {
  const int *lev, *par, *chl, *nbr8;
  const int *pn;     // [box][9]: the parent's 3x3 neighbourhood, (dx+1) + 3 (dy+1) (-1 outside, -2 none)
  const int *ref;    // [box]: bit f = face neighbour f has children, bit 4 = the box has children
  const int2 *ij;
  const double *w;   // [box][8][3]: w_lo, w_hi, 1/(w_lo + w_hi + 2) of column i
  const double *wv;  // [box][8]: volume (and y-face area) weight of column i
};

__device__ __forceinline__ int dir8(int dx, int dy) {
  const int d = (dx + 1) + 3 * (dy + 1);
  return d < 4 ? d : d - 1;
}
__device__ __forceinline__ int face_dir8(int f) {
  return f < 2 ? dir8(f ? 1 : -1, 0) : dir8(0, f == 3 ? 1 : -1);
}
// cell at depth t from face f (t = 0 inner layer, t < 0 ghost layers), u along the face
__device__ __forceinline__ void face_cell(int f, int t, int u, int &ci, int &cj) {
  const int v = (f & 1) ? QN - 1 - t : t;
  if (f < 2) {
    ci = v;
    cj = u;
  } else {
    ci = u;
    cj = v;
  }
}

// What a warp needs to know about its box, loaded in one round of
// independent loads at kernel start (the tables are built on the host):
// face neighbours, the parent's 3x3 neighbourhood, coordinates, level and
// the refinement bits.  Every coarse or neighbour value a kernel reads is
// then one dependent load away.
struct BoxCtx {
  int nb[4], pn[9];
  int ix, iy, lev, ref;
};

__device__ __forceinline__ void load_ctx(const QTabs &T, int b, BoxCtx &c, int lane) {
  if (lane < 4) c.nb[lane] = T.nbr8[8 * b + face_dir8(lane)];
  else if (lane < 13) c.pn[lane - 4] = T.pn[9 * b + lane - 4];
  else if (lane == 13) {
    const int2 v = T.ij[b];
    c.ix = v.x;
    c.iy = v.y;
  } else if (lane == 14) c.lev = T.lev[b];
  else if (lane == 15) c.ref = T.ref[b];
  __syncwarp();
}

// Box of level l-1 holding coarse cell (cx, cy) (cells per side ncl): -1
// outside the domain; -2 (and the error flag) when it does not exist.
__device__ __forceinline__ int coarse_box(const BoxCtx &C, int cx, int cy, int ncl, unsigned *err) {
  if (cx < 0 || cy < 0 || cx >= ncl || cy >= ncl) return -1;
  const int dx = (cx >> 3) - (C.ix >> 1), dy = (cy >> 3) - (C.iy >> 1);
  int b = -2;
  if (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1) b = C.pn[(dx + 1) + 3 * (dy + 1)];
  if (b < 0) {
    atomicOr(err, 1u);
    b = -2;
  }
  return b;
}

// value of var at coarse cell q, or across the wall from coarse cell `from`
// (inside): Dirichlet (homog ? 0 : 2g) - v, Neumann / axis v; mirror: always v
__device__ __forceinline__ double coarse_val(const double *var, const BoxCtx &C, int qx, int qy, int fx, int fy,
                                             int ncl, const QBc &bc, int homog, bool mirror, unsigned *err) {
  const bool out = qx < 0 || qy < 0 || qx >= ncl || qy >= ncl;
  const int b = coarse_box(C, out ? fx : qx, out ? fy : qy, ncl, err);
  const double v = b >= 0 ? var[(size_t)b * QC + ((out ? fx : qx) & 7) + QN * ((out ? fy : qy) & 7)] : 0.0;
  if (!out || mirror) return v;
  const int f = qx < 0 ? 0 : (qx >= ncl ? 1 : (qy < 0 ? 2 : 3));
  return bc.type[f] ? (homog ? 0.0 : bc.g2[f]) - v : v;
}

// Programmatic dependent launch: a kernel launched with it may start while
// its predecessor drains; it loads only tables (which no kernel writes)
// before this wait, and every field value after it.
__device__ __forceinline__ void q_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The start of a box kernel: the box's context, the wait for the
// predecessor, then the box's own values (cells lane and lane + 32).
__device__ __forceinline__ void begin_box(const double *var, const QTabs &T, int b, BoxCtx &C, int lane, double &v0,
                                          double &v1) {
  load_ctx(T, b, C, lane);
  q_wait();
  v0 = var[(size_t)b * QC + lane];
  v1 = var[(size_t)b * QC + lane + 32];
}

// Stage box b into s (S1 x S1, interior at (i+1, j+1)) with the potential
// ghost rules: same-level copy, wall ghost, refinement boundary
// phi_f/3 + 2 phihat/3.  v0, v1: the box's own values (cells lane and
// lane + 32).  With `alt`, neighbours with children are read from alt
// instead of var (the FAS step's restricted values); with alt_all every
// same-level neighbour is.
__device__ void stage_phi(const double *var, const double *alt, const BoxCtx &C, int b, const QBc &bc, int homog,
                          double *s, int lane, unsigned *err, double v0, double v1, bool alt_all = false) {
  s[(lane / QN + 1) * S1 + lane % QN + 1] = v0;
  s[((lane + 32) / QN + 1) * S1 + lane % QN + 1] = v1;
  __syncwarp();
  const int f = lane >> 3, u = lane & 7;
  int ci, cj, gi, gj;
  face_cell(f, 0, u, ci, cj);
  face_cell(f, -1, u, gi, gj);
  const double inner = s[(cj + 1) * S1 + ci + 1];
  const int nb = C.nb[f];
  double v;
  if (nb >= 0) {
    int si, sj;
    face_cell(f ^ 1, 0, u, si, sj);
    v = ((alt && (alt_all || ((C.ref >> f) & 1))) ? alt : var)[(size_t)nb * QC + si + QN * sj];
  } else if (nb == -1) {
    v = bc.type[f] ? (homog ? 0.0 : bc.g2[f]) - inner : inner;
  } else {
    const int ncl = QN << (C.lev - 1);
    const int Gx = C.ix * QN + gi, Gy = C.iy * QN + gj, cx = Gx >> 1, cy = Gy >> 1;
    int qx = cx, qy = cy;
    if (f < 2) qy += (Gy & 1) ? 1 : -1;
    else qx += (Gx & 1) ? 1 : -1;
    // the cells across a refinement face belong to a leaf: var holds them
    const double c = coarse_val(var, C, cx, cy, cx, cy, ncl, bc, homog, false, err);
    const double ct = coarse_val(var, C, qx, qy, cx, cy, ncl, bc, homog, false, err);
    const double phat = 0.75 * c + 0.25 * ct;
    v = inner * (1.0 / 3.0) + phat * (2.0 / 3.0);
  }
  s[(gj + 1) * S1 + gi + 1] = v;
  __syncwarp();
}

// L phi at staged cell (i, j) of box b
__device__ __forceinline__ double lap_s(const double *s, const QTabs &T, int b, int i, int j, double inv_h2) {
  const double c = s[(j + 1) * S1 + i + 1];
  const double wl = T.w[(size_t)b * 24 + 3 * i], wh = T.w[(size_t)b * 24 + 3 * i + 1];
  return (wl * (s[(j + 1) * S1 + i] - c) + wh * (s[(j + 1) * S1 + i + 2] - c) + (s[j * S1 + i + 1] - c) +
          (s[(j + 2) * S1 + i + 1] - c)) * inv_h2;
}

#define QWARP()                                  \
  __shared__ BoxCtx ctx_[WPB];                   \
  const int wv_ = threadIdx.x >> 5, lane = threadIdx.x & 31; \
  const int k_ = blockIdx.x * WPB + wv_;         \
  BoxCtx &C = ctx_[wv_];

// one colour pass of red-black Gauss-Seidel on the n boxes of level l
__global__ void __launch_bounds__(QT) k_q_rbgs(int off, int n, int l, int colour, double *__restrict__ phi,
                                               const double *__restrict__ rhs, QTabs T, const __grid_constant__ QBc bc, double h2,
                                               unsigned *err) {
  __shared__ double sm[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;  // the whole warp
  const int b = off + k_;
  double *s = sm[wv_];
  const int j = lane >> 2, i = 2 * (lane & 3) + ((j + colour) & 1);
  const double *wc = T.w + (size_t)b * 24 + 3 * i;
  const double w0 = wc[0], w1 = wc[1], w2 = wc[2];
  double v0, v1;
  begin_box(phi, T, b, C, lane, v0, v1);
  const double fr = rhs[(size_t)b * QC + i + QN * j];
  stage_phi(phi, nullptr, C, b, bc, 0, s, lane, err, v0, v1);
  phi[(size_t)b * QC + i + QN * j] =
      (w0 * s[(j + 1) * S1 + i] + w1 * s[(j + 1) * S1 + i + 2] + s[j * S1 + i + 1] + s[(j + 2) * S1 + i + 1] -
       h2 * fr) *
      w2;
}

// Residual of every box of level l restricted to its parent's quadrant:
// the restricted potential into old[parent] (committed by k_q_fas, so that
// coarse values read for ghosts here stay unchanged), the restricted
// residual into rhs[parent].  Volume-weighted mean of the four children.
// Warps [0, n) take the boxes of level l; warps [n, n + nc) the boxes
// coff.. of level l-1, copying those without children into old (so that
// k_q_fas_rbgs0 finds the whole level in old).
__global__ void __launch_bounds__(QT) k_q_resid_restrict(int off, int n, int l, const double *__restrict__ phi,
                                                         double *__restrict__ rhs, double *__restrict__ old,
                                                         QTabs T, const __grid_constant__ QBc bc, double inv_h2, unsigned *err,
                                                         int coff = 0, int nc = 0) {
  __shared__ double sm[WPB][S1 * S1];
  __shared__ double sr[WPB][QC];
  QWARP();
  if (k_ >= n) {
    if (k_ >= n + nc) return;
    const int bc2 = coff + k_ - n;
    const bool leaf = __ldg(T.chl + 4 * bc2) < 0;
    q_wait();
    if (leaf)
      for (int c = lane; c < QC; c += 32) old[(size_t)bc2 * QC + c] = phi[(size_t)bc2 * QC + c];
    return;
  }
  const int b = off + k_;
  double *s = sm[wv_];
  double v0, v1;
  begin_box(phi, T, b, C, lane, v0, v1);
  stage_phi(phi, nullptr, C, b, bc, 0, s, lane, err, v0, v1);
  for (int c = lane; c < QC; c += 32) {
    const int i = c % QN, j = c / QN;
    sr[wv_][c] = rhs[(size_t)b * QC + c] - lap_s(s, T, b, i, j, inv_h2);
  }
  __syncwarp();
  const int p = C.pn[4];
  const int2 B = make_int2(C.ix, C.iy);
  const int m = lane & 15, ii = m & 3, jj = m >> 2;
  double sum = 0.0, wsum = 0.0;
  for (int dj = 0; dj < 2; ++dj)
    for (int di = 0; di < 2; ++di) {
      const int i = 2 * ii + di, j = 2 * jj + dj;
      const double w = T.wv[(size_t)b * QN + i];
      sum += w * (lane < 16 ? s[(j + 1) * S1 + i + 1] : sr[wv_][i + QN * j]);
      wsum += w;
    }
  const int I = 4 * (B.x & 1) + ii, J = 4 * (B.y & 1) + jj;
  (lane < 16 ? old : rhs)[(size_t)p * QC + I + QN * J] = sum / wsum;
}

// Level l (all boxes): refined boxes take their restricted potential from
// old and get the FAS right-hand side f += L phi; every box ends with
// old = phi (the values the coarse correction is measured against).
__global__ void __launch_bounds__(QT) k_q_fas(int off, int n, int l, double *__restrict__ phi,
                                              double *__restrict__ rhs, double *__restrict__ old, QTabs T, const __grid_constant__ QBc bc,
                                              double inv_h2, unsigned *err) {
  __shared__ double sm[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;
  const int b = off + k_;
  const size_t g0 = (size_t)b * QC + lane, g1 = g0 + 32;
  double v0, v1;
  begin_box(phi, T, b, C, lane, v0, v1);
  const double o0 = old[g0], o1 = old[g1], f0 = rhs[g0], f1 = rhs[g1];
  const bool refined = C.ref & 16;
  double *s = sm[wv_];
  if (refined) {
    // the box's restricted values; neighbours with children read old too
    stage_phi(phi, old, C, b, bc, 0, s, lane, err, o0, o1);
    rhs[g0] = f0 + lap_s(s, T, b, lane % QN, lane / QN, inv_h2);
    rhs[g1] = f1 + lap_s(s, T, b, lane % QN, lane / QN + 4, inv_h2);
    phi[g0] = o0;
    phi[g1] = o1;
  } else {
    old[g0] = v0;
    old[g1] = v1;
  }
}

// k_q_fas fused with the first colour pass (colour 0) of the smoothing that
// follows it on level l.  The FAS term of a box reads its neighbours' face
// cells, whose colour-0 values the neighbours' own warps of this launch
// overwrite; so the box and every same-level neighbour value are read from
// old, which the restriction launch before filled with the whole level as
// it is now (k_q_resid_restrict with nc) and which nothing in this launch
// writes.  The staged box serves the FAS step and the colour-0 update (which
// reads colour-1 cells and ghosts only); the warp's rhs and phi writes are
// ordered before the update by __syncwarp.  The same operations as k_q_fas
// followed by k_q_rbgs with colour 0.
__global__ void __launch_bounds__(QT) k_q_fas_rbgs0(int off, int n, int l, double *__restrict__ phi,
                                                    double *__restrict__ rhs, const double *__restrict__ old,
                                                    QTabs T, const __grid_constant__ QBc bc, double inv_h2, double h2,
                                                    unsigned *err) {
  __shared__ double sm[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;
  const int b = off + k_;
  const size_t g0 = (size_t)b * QC + lane, g1 = g0 + 32;
  double o0, o1;
  begin_box(old, T, b, C, lane, o0, o1);
  const double f0 = rhs[g0], f1 = rhs[g1];
  const bool refined = C.ref & 16;
  double *s = sm[wv_];
  const int j = lane >> 2, i = 2 * (lane & 3) + (j & 1);  // this lane's colour-0 cell
  const double *wc = T.w + (size_t)b * 24 + 3 * i;
  const double w0 = wc[0], w1 = wc[1], w2 = wc[2];
  stage_phi(phi, old, C, b, bc, 0, s, lane, err, o0, o1, true);
  if (refined) {
    rhs[g0] = f0 + lap_s(s, T, b, lane % QN, lane / QN, inv_h2);
    rhs[g1] = f1 + lap_s(s, T, b, lane % QN, lane / QN + 4, inv_h2);
    phi[g0] = o0;
    phi[g1] = o1;
  }
  __syncwarp();
  const double fr = rhs[(size_t)b * QC + i + QN * j];
  phi[(size_t)b * QC + i + QN * j] =
      (w0 * s[(j + 1) * S1 + i] + w1 * s[(j + 1) * S1 + i + 2] + s[j * S1 + i + 1] + s[(j + 2) * S1 + i + 1] -
       h2 * fr) *
      w2;
}

// Prolongation to every box of level l: (2c + c_x + c_y)/4 of the parent
// level.  corr: the correction phi - old (homogeneous wall ghosts) added to
// phi; otherwise phi itself (FMG, wall values) replaces phi.
__global__ void __launch_bounds__(QT) k_q_prolong(int off, int n, int l, double *__restrict__ phi,
                                                  const double *__restrict__ old, int corr, QTabs T, const __grid_constant__ QBc bc,
                                                  unsigned *err) {
  QWARP();
  if (k_ >= n) return;
  const int b = off + k_, ncl = QN << (l - 1);
  load_ctx(T, b, C, lane);
  q_wait();
  const int2 B = make_int2(C.ix, C.iy);
  auto cv = [&](int qx, int qy, int fx, int fy) {
    const double a = coarse_val(phi, C, qx, qy, fx, fy, ncl, bc, corr, false, err);
    return corr ? a - coarse_val(old, C, qx, qy, fx, fy, ncl, bc, corr, false, err) : a;
  };
  for (int c = lane; c < QC; c += 32) {
    const int Gx = B.x * QN + c % QN, Gy = B.y * QN + c / QN, cx = Gx >> 1, cy = Gy >> 1;
    const double sum = 2.0 * cv(cx, cy, cx, cy) + cv(cx + ((Gx & 1) ? 1 : -1), cy, cx, cy) +
                       cv(cx, cy + ((Gy & 1) ? 1 : -1), cx, cy);
    const size_t g = (size_t)b * QC + c;
    if (corr) phi[g] += 0.25 * sum;
    else phi[g] = 0.25 * sum;
  }
}

#include "quadleg.cuh"

// Exact level-0 solve (one box): phi = A^-1 (f - L0), A the operator's
// matrix with homogeneous wall ghosts (inverted on the host), L0 the
// operator of phi = 0 with the wall values.
__global__ void k_q_coarse(double *__restrict__ phi, const double *__restrict__ rhs, const double *__restrict__ ainv,
                           QTabs T, const __grid_constant__ QBc bc, double inv_h2, unsigned *xseq) {
  __shared__ double r[QC];
  const int c = threadIdx.x, i = c % QN, j = c / QN;
  const double wl = T.w[3 * i], wh = T.w[3 * i + 1];
  q_wait();
  if (c == 0) ++*xseq;  // the exchange tags move on between the two legs of every level
  double l0 = 0.0;
  if (i == 0 && bc.type[0]) l0 += wl * bc.g2[0];
  if (i == QN - 1 && bc.type[1]) l0 += wh * bc.g2[1];
  if (j == 0 && bc.type[2]) l0 += bc.g2[2];
  if (j == QN - 1 && bc.type[3]) l0 += bc.g2[3];
  r[c] = rhs[c] - l0 * inv_h2;
  __syncthreads();
  double acc = 0.0;
  for (int k = 0; k < QC; ++k) acc += ainv[c * QC + k] * r[k];
  phi[c] = acc;
}

// device slots (unsigned long long each): time-step maxima, then the solve's
// scalars
enum { QS_ADV = 0, QS_NUM = 4, QS_DEN, QS_CYC, QS_REL, QS_TOL, QS_MAXC, QS_N };

// a solve's stopping parameters, before its graph runs
__global__ void k_q_begin(unsigned long long *slots, double tol, int max_cycles) {
  slots[QS_TOL] = (unsigned long long)__double_as_longlong(tol);
  slots[QS_MAXC] = (unsigned long long)max_cycles;
  slots[QS_CYC] = 0ull;
}

// Stopping test of the device-side cycle loop: relative residual, cycle
// count, and whether another cycle runs (not after a device error)
__global__ void k_q_check(cudaGraphConditionalHandle h, unsigned long long *slots, const unsigned *err) {
  const double num = __longlong_as_double((long long)slots[QS_NUM]);
  const double den = __longlong_as_double((long long)slots[QS_DEN]);
  const double rel = den > 0.0 ? num / den : num;
  const unsigned long long c = slots[QS_CYC] + 1ull;
  slots[QS_CYC] = c;
  slots[QS_REL] = (unsigned long long)__double_as_longlong(rel);
  const double tol = __longlong_as_double((long long)slots[QS_TOL]);
  cudaGraphSetConditional(h, rel > tol && c < slots[QS_MAXC] && *err == 0u ? 1u : 0u);
}

__device__ __forceinline__ void max_bits(unsigned long long *slot, double v) {
  unsigned long long x = (unsigned long long)__double_as_longlong(fabs(v));
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
    x = y > x ? y : x;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(slot, x);
}

// max |f - L var| over the leaf cells of all boxes (var = a zero array for
// the denominator); with `keep` every box of src is also copied there (a copy
// of its own costs a solve 3 us)
__global__ void __launch_bounds__(QT) k_q_resmax(int n, const double *__restrict__ var,
                                                 const double *__restrict__ rhs, QTabs T, const __grid_constant__ QBc bc,
                                                 const double *__restrict__ inv_h2, unsigned long long *slot,
                                                 unsigned *err, const double *__restrict__ src,
                                                 double *__restrict__ keep) {
  __shared__ double sm[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;
  const int b = k_;
  double v0, v1;
  begin_box(var, T, b, C, lane, v0, v1);
  if (keep) {
    keep[(size_t)b * QC + lane] = src[(size_t)b * QC + lane];
    keep[(size_t)b * QC + lane + 32] = src[(size_t)b * QC + lane + 32];
  }
  if (C.ref & 16) return;
  double *s = sm[wv_];
  const int l = C.lev;
  stage_phi(var, nullptr, C, b, bc, 0, s, lane, err, v0, v1);
  double m = 0.0;
  for (int c = lane; c < QC; c += 32)
    m = fmax(m, fabs(rhs[(size_t)b * QC + c] - lap_s(s, T, b, c % QN, c / QN, inv_h2[l])));
  max_bits(slot, m);
}

// Eq. 5 on leaf cells
__global__ void k_q_charge(int n, double *__restrict__ rhs, const double *__restrict__ ne,
                           const double *__restrict__ ni, const double *__restrict__ rho, const int *__restrict__ chl,
                           double q, double inv_eps, int use_rho) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= (long long)n * QC) return;
  if (chl[4 * (g / QC)] >= 0) return;
  rhs[g] = use_rho ? -rho[g] * inv_eps : -q * (ni[g] - ne[g]) * inv_eps;
}

// |E| on leaf cells: face fields (phi_i - phi_{i+1})/h, cell components the
// mean of the two faces; zero on refined boxes
__global__ void __launch_bounds__(QT) k_q_field(int n, const double *__restrict__ phi, double *__restrict__ emag,
                                                QTabs T, const __grid_constant__ QBc bc, const double *__restrict__ inv_h,
                                                unsigned *err) {
  __shared__ double sm[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;
  const int b = k_;
  double v0, v1;
  begin_box(phi, T, b, C, lane, v0, v1);
  if (C.ref & 16) {
    for (int c = lane; c < QC; c += 32) emag[(size_t)b * QC + c] = 0.0;
    return;
  }
  double *s = sm[wv_];
  const int l = C.lev;
  stage_phi(phi, nullptr, C, b, bc, 0, s, lane, err, v0, v1);
  const double hih = 0.5 * inv_h[l];
  for (int c = lane; c < QC; c += 32) {
    const int q = (c / QN + 1) * S1 + c % QN + 1;
    // (the mean of a cell's two face fields is the centred difference)
    const double dx = s[q - 1] - s[q + 1], dy = s[q - S1] - s[q + S1];
    emag[(size_t)b * QC + c] = sqrt_newton(fma(dy, dy, dx * dx)) * hih;
  }
}

// Stage the density n with two ghost layers (S2 x S2, interior at (i+2,
// j+2)), the potential (S1) and the half table index of |E| with one layer:
// density ghosts are
// same-level copies, mirrors at walls and the axis, and at refinement
// boundaries the prolongation (2c + c_x + c_y)/4 of the coarse cell
// containing the ghost, limited to 2c; |E| ghosts the inner value at walls
// and the coarse cell's value at refinement boundaries.
__device__ void stage_fluid(const double *nv, const double *phi, const double *emag, const BoxCtx &C, int b,
                            const QBc &bc, double *sn, double *sp, unsigned long long *se, const Table &tb, int lane,
                            unsigned *err) {
  const int l = C.lev;
  stage_phi(phi, nullptr, C, b, bc, 0, sp, lane, err, phi[(size_t)b * QC + lane], phi[(size_t)b * QC + lane + 32]);
  for (int c = lane; c < QC; c += 32) {
    sn[(c / QN + 2) * S2 + c % QN + 2] = nv[(size_t)b * QC + c];
    se[(c / QN + 1) * S1 + c % QN + 1] = half_index(emag[(size_t)b * QC + c], tb);
  }
  __syncwarp();
  const int2 B = make_int2(C.ix, C.iy);
  const int ncl = l > 0 ? (QN << (l - 1)) : 0;
  for (int g = lane; g < 64; g += 32) {  // density: 4 faces x 2 layers x 8
    const int f = g >> 4, t = 1 + ((g >> 3) & 1), u = g & 7;
    int gi, gj;
    face_cell(f, -t, u, gi, gj);
    const int nb = C.nb[f];
    double v;
    if (nb >= 0) {
      int si, sj;
      face_cell(f ^ 1, t - 1, u, si, sj);
      v = nv[(size_t)nb * QC + si + QN * sj];
    } else if (nb == -1) {
      int mi, mj;
      face_cell(f, t - 1, u, mi, mj);
      v = sn[(mj + 2) * S2 + mi + 2];
    } else {
      const int Gx = B.x * QN + gi, Gy = B.y * QN + gj, cx = Gx >> 1, cy = Gy >> 1;
      const double c = coarse_val(nv, C, cx, cy, cx, cy, ncl, bc, 0, true, err);
      const double sum = 2.0 * c + coarse_val(nv, C, cx + ((Gx & 1) ? 1 : -1), cy, cx, cy, ncl, bc, 0, true, err) +
                         coarse_val(nv, C, cx, cy + ((Gy & 1) ? 1 : -1), cx, cy, ncl, bc, 0, true, err);
      v = fmin(0.25 * sum, 2.0 * c);
    }
    sn[(gj + 2) * S2 + gi + 2] = v;
  }
  {  // |E|: 4 faces x 8
    const int f = lane >> 3, u = lane & 7;
    int ci, cj, gi, gj;
    face_cell(f, 0, u, ci, cj);
    face_cell(f, -1, u, gi, gj);
    const int nb = C.nb[f];
    unsigned long long v;
    if (nb >= 0) {
      int si, sj;
      face_cell(f ^ 1, 0, u, si, sj);
      v = half_index(emag[(size_t)nb * QC + si + QN * sj], tb);
    } else if (nb == -1) {
      v = se[(cj + 1) * S1 + ci + 1];
    } else {
      const int cx = (B.x * QN + gi) >> 1, cy = (B.y * QN + gj) >> 1;
      v = half_index(coarse_val(emag, C, cx, cy, cx, cy, ncl, bc, 0, true, err), tb);
    }
    se[(gj + 1) * S1 + gi + 1] = v;
  }
  __syncwarp();
}

// dx times the flux through face m (between cells m-1 and m) along axis a at u
__device__ __forceinline__ double face_flux(const double *sn, const double *sp, const unsigned long long *se, int a,
                                            int m, int u, const Table &tb) {
  const int q = a == 0 ? (u + 2) * S2 + m + 2 : (m + 2) * S2 + u + 2, sq = a == 0 ? 1 : S2;
  const int r = a == 0 ? (u + 1) * S1 + m + 1 : (m + 1) * S1 + u + 1, sr = a == 0 ? 1 : S1;
  const double nL = sn[q - sq], nR = sn[q];
  return face_flux_d(nL, nR, nL - sn[q - 2 * sq], nR - nL, sn[q + sq] - nR, sp[r - sr] - sp[r], se[r - sr], se[r], tb);
}

// Fine-side fluxes of every leaf box face that borders a coarser leaf:
// cflux[box][face][u]
__global__ void __launch_bounds__(QT) k_q_cf_flux(int n, const double *__restrict__ nv, const double *__restrict__ phi,
                                                  const double *__restrict__ emag, double *__restrict__ cflux,
                                                  QTabs T, const __grid_constant__ QBc bc, Table tb, const double *__restrict__ hs,
                                                  unsigned *err) {
  __shared__ double snm[WPB][S2 * S2], spm[WPB][S1 * S1];
  __shared__ unsigned long long sem[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;
  const int b = k_;
  load_ctx(T, b, C, lane);
  q_wait();
  if (C.ref & 16) return;
  bool any = false;
  for (int f = 0; f < 4; ++f) any |= C.nb[f] == -2;
  if (!any) return;
  const int l = C.lev;
  stage_fluid(nv, phi, emag, C, b, bc, snm[wv_], spm[wv_], sem[wv_], tb, lane, err);
  const int f = lane >> 3, u = lane & 7;
  if (C.nb[f] == -2)
    cflux[(size_t)b * 32 + f * 8 + u] =
        face_flux(snm[wv_], spm[wv_], sem[wv_], f >> 1, (f & 1) ? QN : 0, u, tb) * (1.0 / hs[l]);
}

__device__ __forceinline__ void max_word(unsigned long long *slot, long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
  if ((threadIdx.x & 31) == 0) atomicMax(slot, (unsigned long long)max(x, 0ll));
}

// maxima over a box (a warp) of the three time-step quantities (bit patterns),
// the first two times scale, into slots[0..2] (the products' maximum is the
// maximum's product, rounding being monotonic)
__device__ __forceinline__ void max3_to(unsigned long long *slots, const long long (&m)[3], double scale) {
  max_word(slots, dbits(__longlong_as_double(m[0]) * scale));
  max_word(slots + 1, dbits(__longlong_as_double(m[1]) * scale));
  max_word(slots + 2, m[2]);
}

// sum_d |mu E_d| 2 dx of the staged potential at q, that plus 8 D (both to be
// scaled by 1/(2 dx^2)), and mu n_e, as running maxima of bit patterns
// without negative values and NaNs
__device__ __forceinline__ void dt_cell(const double *sp, int q, double mu, double dc, double ne, long long (&m)[3]) {
  const double adv = dabs(mu) * (dabs(sp[q - 1] - sp[q + 1]) + dabs(sp[q - S1] - sp[q + S1]));
  m[0] = max(m[0], size_bits(adv));
  m[1] = max(m[1], size_bits(fma(8.0, dc, adv)));
  m[2] = max(m[2], size_bits(mu * ne));
}

// One forward Euler stage on every leaf box: dst = src - dt div F + dt
// alpha mu |E| n_e (Eq. 2-3); a face next to a refined box takes the
// area-weighted mean of the two fine fluxes from cflux.  HEUN: dst = (n0 +
// that)/2 (dst may be n0: a cell reads only its own), and the time-step
// maxima of src.  With rhs also the Eq. 5 right-hand side of dst.  The box's
// density differences are formed once and shared by the faces; bound by the
// FP64 pipe (see fluid_dev.cuh).
template <bool HEUN>
__global__ void __launch_bounds__(QT) k_q_update(int n, const double *__restrict__ ne, const double *__restrict__ ni,
                                                 const double *ne0, const double *ni0, double *ne_out, double *ni_out,
                                                 double *__restrict__ rhs, const double *__restrict__ phi,
                                                 const double *__restrict__ emag, const double *__restrict__ cflux,
                                                 QTabs T, const __grid_constant__ QBc bc, Table tb,
                                                 const double *__restrict__ hs, double dt, double qie,
                                                 unsigned long long *slots, unsigned *err) {
  constexpr int DL = QN + 3;  // differences of a line: cells -2 .. 9
  __shared__ double snm[WPB][S2 * S2], spm[WPB][S1 * S1], sf[WPB][2][(QN + 1) * QN], sdm[WPB][2][DL * QN];
  __shared__ unsigned long long sem[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;
  const int b = k_;
  load_ctx(T, b, C, lane);
  q_wait();
  if (C.ref & 16) return;
  const int l = C.lev;
  const double h = hs[l], ih2 = hs[QMAXL + l];
  const double *sn = snm[wv_], *sp = spm[wv_];
  const unsigned long long *se = sem[wv_];
  stage_fluid(ne, phi, emag, C, b, bc, snm[wv_], spm[wv_], sem[wv_], tb, lane, err);
  for (int g = lane; g < 2 * DL * QN; g += 32) {
    const int a = g / (DL * QN), r = g % (DL * QN), k = r / QN, u = r % QN;
    const int q = a == 0 ? (u + 2) * S2 + k : k * S2 + u + 2, sq = a == 0 ? 1 : S2;  // cell k - 2 of line u
    sdm[wv_][a][r] = sn[q + sq] - sn[q];
  }
  __syncwarp();
  for (int g = lane; g < 2 * (QN + 1) * QN; g += 32) {
    const int a = g / ((QN + 1) * QN), r = g % ((QN + 1) * QN), m = r / QN, u = r % QN;
    const int f = 2 * a + (m == QN ? 1 : 0);
    double F;
    if ((m == 0 || m == QN) && ((C.ref >> f) & 1)) {  // refined neighbour: mean of its fine fluxes
      const int cx = a == 0 ? ((f & 1) ? 0 : 1) : u >> 2, cy = a == 0 ? u >> 2 : ((f & 1) ? 0 : 1);
      const int ch = T.chl[4 * C.nb[f] + cx + 2 * cy];
      double s = 0.0, ws = 0.0;
      for (int du = 0; du < 2; ++du) {
        const int uf = 2 * (u & 3) + du;
        const double w = a == 0 ? 1.0 : T.wv[(size_t)ch * QN + uf];
        s += w * cflux[(size_t)ch * 32 + (f ^ 1) * 8 + uf];
        ws += w;
      }
      F = s / ws * h;
    } else {
      const int q = a == 0 ? (u + 2) * S2 + m + 2 : (m + 2) * S2 + u + 2, sq = a == 0 ? 1 : S2;
      const int r1 = a == 0 ? (u + 1) * S1 + m + 1 : (m + 1) * S1 + u + 1, sr = a == 0 ? 1 : S1;
      const double *d = sdm[wv_][a] + r;
      F = face_flux_d(sn[q - sq], sn[q], d[0], d[QN], d[2 * QN], sp[r1 - sr] - sp[r1], se[r1 - sr], se[r1], tb);
    }
    sf[wv_][a][r] = F;
  }
  __syncwarp();
  const double dth = -dt * ih2;
  long long m[3] = {0, 0, 0};
#pragma unroll
  for (int s2 = 0; s2 < 2; ++s2) {
    const int c = lane + 32 * s2, i = c % QN, j = c / QN, q = (j + 1) * S1 + i + 1;
    const double wl = T.w[(size_t)b * 24 + 3 * i], wh = T.w[(size_t)b * 24 + 3 * i + 1];
    const double *fx = sf[wv_][0] + i * QN + j, *fy = sf[wv_][1] + j * QN + i;
    const double div = fma(wh, fx[QN], -wl * fx[0]) + (fy[QN] - fy[0]);  // dx^2 times the divergence
    const size_t g = (size_t)b * QC + c;
    const double nes = sn[(j + 2) * S2 + i + 2], e = emag[g];
    double w;
    const int k = index_split(se[q], se[q], tb, w);
    const double2 cm = __ldg(tb.fc + 2 * k), al = __ldg(tb.al + k);
    const double mu = fma(w, cm.y, cm.x);
    const double src = fma(w, al.y, al.x) * mu * e * nes;
    double a = fma(dth, div, fma(dt, src, nes)), bq = fma(dt, src, ni[g]);
    if (HEUN) {
      a = halve(ne0[g] + a);
      bq = halve(ni0[g] + bq);
      const double2 cd = __ldg(tb.fc + 2 * k + 1);
      dt_cell(sp, q, mu, fma(w, cd.y, cd.x), nes, m);
    }
    ne_out[g] = a;
    ni_out[g] = bq;
    if (rhs) rhs[g] = (bq - a) * qie;
  }
  if (HEUN) max3_to(slots, m, 0.5 * ih2);
}

// Volume-weighted means of the four children of one or two variables into
// every refined box, in one launch without waiting: a warp restricts its
// leaf box into its quadrant of the parent (lanes 0-15 the first variable,
// 16-31 the second) and counts itself in there; the warp that completes the
// parent's four goes on with the parent, the others end.  (A launch per level
// and variable took 3 us each, 84 of them a Heun step on 15 levels.)  The
// counters are zero again after the launch.
__global__ void __launch_bounds__(QT) k_q_restrict_tree(int n, double *v, double *v2, QTabs T, int *count) {
  const int lane = threadIdx.x & 31, k = blockIdx.x * WPB + (threadIdx.x >> 5);
  if (k >= n || T.chl[4 * k] >= 0) return;
  int b = k;
  double *const x = lane < 16 ? v : v2;
  const int ii = lane & 3, jj = (lane >> 2) & 3;
  for (bool first = true;; first = false) {
    const int p = T.par[b];
    if (p < 0) return;
    const int2 B = T.ij[b];
    if (x) {
      double sum = 0.0, wsum = 0.0;
      for (int dj = 0; dj < 2; ++dj)
        for (int di = 0; di < 2; ++di) {
          const int i = 2 * ii + di, j = 2 * jj + dj;
          const double w = T.wv[(size_t)b * QN + i], *c = x + (size_t)b * QC + i + QN * j;
          sum += w * (first ? *c : __ldcg(c));  // a parent's cells were written by other warps: read them from L2
          wsum += w;
        }
      x[(size_t)p * QC + 4 * (B.x & 1) + ii + QN * (4 * (B.y & 1) + jj)] = sum / wsum;
    }
    __threadfence();
    __syncwarp();
    int last = 0;
    if (lane == 0) {
      last = atomicAdd(count + p, 1) == 3;
      if (last) count[p] = 0;
      __threadfence();
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    b = p;
  }
}

// time-step limits: max over leaf cells of sum|v_d|/dx, that plus 4D/dx^2,
// and mu n_e (slots 0..2, bit patterns of non-negative doubles)
__global__ void __launch_bounds__(QT) k_q_dt(int n, const double *__restrict__ phi, const double *__restrict__ emag,
                                             const double *__restrict__ ne, QTabs T, const __grid_constant__ QBc bc, Table tb,
                                             const double *__restrict__ hs, unsigned long long *slots,
                                             unsigned *err) {
  __shared__ double sm[WPB][S1 * S1];
  QWARP();
  if (k_ >= n) return;
  const int b = k_;
  double v0, v1;
  begin_box(phi, T, b, C, lane, v0, v1);
  if (C.ref & 16) return;
  double *s = sm[wv_];
  stage_phi(phi, nullptr, C, b, bc, 0, s, lane, err, v0, v1);
  long long m[3] = {0, 0, 0};
#pragma unroll
  for (int s2 = 0; s2 < 2; ++s2) {
    const int c = lane + 32 * s2;
    const size_t g = (size_t)b * QC + c;
    double w;
    const unsigned long long x = half_index(emag[g], tb);
    const int k = index_split(x, x, tb, w);
    const double2 cm = __ldg(tb.fc + 2 * k), cd = __ldg(tb.fc + 2 * k + 1);
    dt_cell(s, (c / QN + 1) * S1 + c % QN + 1, fma(w, cm.y, cm.x), fma(w, cd.y, cd.x), ne[g], m);
  }
  max3_to(slots, m, 0.5 * hs[QMAXL + C.lev]);
}

// alpha(e) from the table with every operation rounded on its own (no fused
// multiply-add), the arithmetic of the refinement test on both sides
__device__ __forceinline__ double alpha_rn(const double *__restrict__ t, int n, double de, double e) {
  const double x = __ddiv_rn(e, de);
  if (x <= 0.0) return t[0];
  if (x >= (double)(n - 1)) return t[n - 1];
  const int i = (int)x;
  const double w = __dsub_rn(x, (double)i);
  return __dadd_rn(t[i], __dmul_rn(w, __dsub_rn(t[i + 1], t[i])));
}

// Eq. 8 on every leaf box (one warp per box, cells lane and lane + 32):
// need[b] bit c where alpha(c1 |E|) dx >= c0 c1; fine[b] = 1 when every cell
// has alpha(c1 |E|) dx < c0_deref c1 and dx < dx_deref
__global__ void __launch_bounds__(QT) k_q_refcrit(int n, const double *__restrict__ emag, QTabs T,
                                                  const double *__restrict__ alpha, int tab_n, double de, double c1,
                                                  double c0c1, double c0dc1, double dxd,
                                                  const double *__restrict__ hs, unsigned long long *__restrict__ need,
                                                  unsigned char *__restrict__ fine) {
  QWARP();
  if (k_ >= n) return;
  const int b = k_;
  load_ctx(T, b, C, lane);
  q_wait();
  if (C.ref & 16) {
    if (lane == 0) {
      need[b] = 0ull;
      fine[b] = 0;
    }
    return;
  }
  const double dx = hs[C.lev];
  bool nd[2], ok = true;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double ad = __dmul_rn(alpha_rn(alpha, tab_n, de, __dmul_rn(c1, emag[(size_t)b * QC + lane + 32 * h])), dx);
    nd[h] = ad >= c0c1;
    ok &= ad < c0dc1;
  }
  const unsigned lo = __ballot_sync(0xffffffffu, nd[0]), hi = __ballot_sync(0xffffffffu, nd[1]);
  const bool all = __all_sync(0xffffffffu, ok);
  if (lane == 0) {
    need[b] = (unsigned long long)lo | ((unsigned long long)hi << 32);
    fine[b] = (unsigned char)(all && dx < dxd);
  }
}

// After a regrid, box b of the new mesh takes the data of old box
// rg[10 b] (>= 0) from the snapshot snap[var][old box][64] (vars: phi,
// n_e, n_i, f, |E|, rho), or, as a new child (rg[10 b] < 0), the
// prolongation (2c + c_x + c_y)/4 of its old parent's cells, rg[10 b + 1 ..
// 9] being the old parent's 3x3 neighbourhood: wall ghosts for the
// potential, mirrors and the 2c limit for the densities; f, |E| and rho of
// new boxes are zero.
__global__ void __launch_bounds__(QT) k_q_regrid_move(int n, const int *__restrict__ rg,
                                                      const double *__restrict__ snap, size_t stride,
                                                      double *__restrict__ phi, double *__restrict__ ne,
                                                      double *__restrict__ ni, double *__restrict__ rhs,
                                                      double *__restrict__ emag, double *__restrict__ rho, QTabs T,
                                                      const __grid_constant__ QBc bc, unsigned *err) {
  QWARP();
  if (k_ >= n) return;
  const int b = k_;
  double *dst[6] = {phi, ne, ni, rhs, emag, rho};
  const int src = rg[10 * (size_t)b];
  if (src >= 0) {
    for (int v = 0; v < 6; ++v)
      for (int c = lane; c < QC; c += 32) dst[v][(size_t)b * QC + c] = snap[v * stride + (size_t)src * QC + c];
    return;
  }
  if (lane < 9) C.pn[lane] = rg[10 * (size_t)b + 1 + lane];
  if (lane == 9) {
    const int2 v = T.ij[b];
    C.ix = v.x;
    C.iy = v.y;
  }
  if (lane == 10) C.lev = T.lev[b];
  __syncwarp();
  const int ncl = QN << (C.lev - 1);
  for (int c = lane; c < QC; c += 32) {
    const int Gx = C.ix * QN + c % QN, Gy = C.iy * QN + c / QN, cx = Gx >> 1, cy = Gy >> 1;
    const int qx = cx + ((Gx & 1) ? 1 : -1), qy = cy + ((Gy & 1) ? 1 : -1);
    for (int v = 0; v < 3; ++v) {
      const double *sv = snap + v * stride;
      const bool mirror = v > 0;
      const double cv = coarse_val(sv, C, cx, cy, cx, cy, ncl, bc, 0, mirror, err);
      double val = 2.0 * cv;
      val += coarse_val(sv, C, qx, cy, cx, cy, ncl, bc, 0, mirror, err);
      val += coarse_val(sv, C, cx, qy, cx, cy, ncl, bc, 0, mirror, err);
      val = 0.25 * val;
      if (mirror && val > 2.0 * cv) val = 2.0 * cv;
      dst[v][(size_t)b * QC + c] = val;
    }
    for (int v = 3; v < 6; ++v) dst[v][(size_t)b * QC + c] = 0.0;
  }
}

// ---- regrid: the new box set on the device ---------------------------------
//
// Old boxes are stored level by level in Morton order.  The new set keeps
// every box but the children of derefined boxes and adds 4 children per
// refined box; each new level is the merge of two Morton-sorted lists (the
// kept boxes of the level and the children of the refined boxes of the level
// below, whose keys are parent key * 4 + child), so a box's new index is its
// rank in its own list plus the count of keys of the other list below its
// own (binary searches).  Parents, children and same-level neighbours follow
// by binary search in the new levels' keys.

// per-level starts of the compacted lists and of the new levels
struct QRgLevels {
  int kept[QMAXL + 2];  // level l in the kept list
  int ref[QMAXL + 2];   // level l in the refined list
  int nw[QMAXL + 2];    // level l in the new numbering
};
struct QOffsets {
  int v[QMAXL + 2];
};

// Morton key of (i, j) within its level: bit b of i to bit 2b, of j to 2b + 1
__device__ __forceinline__ uint64_t qmorton(int i, int j) {
  auto spread = [](unsigned v) {
    uint64_t x = v & 0x7fffffffu;
    x = (x | (x << 16)) & 0x0000ffff0000ffffull;
    x = (x | (x << 8)) & 0x00ff00ff00ff00ffull;
    x = (x | (x << 4)) & 0x0f0f0f0f0f0f0f0full;
    x = (x | (x << 2)) & 0x3333333333333333ull;
    x = (x | (x << 1)) & 0x5555555555555555ull;
    return x;
  };
  return spread((unsigned)i) | (spread((unsigned)j) << 1);
}

// first index in [lo, hi) whose key is >= x
__device__ __forceinline__ int qlower_bound(const uint64_t *__restrict__ a, int lo, int hi, uint64_t x) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// refinement: a flagged leaf below the maximum level whose 8 neighbour
// positions of its level hold a box or lie outside the domain (else the
// request is dropped: cnt[0])
__global__ void k_qrg_refine(int n, const int *__restrict__ lev, const int *__restrict__ chl,
                             const int *__restrict__ nbr8, const int8_t *__restrict__ flags, int lmax,
                             int *__restrict__ refv, int *cnt) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  int r = 0;
  if (chl[4 * b] < 0 && flags[b] > 0 && lev[b] < lmax) {
    bool ok = true;
    for (int d = 0; d < 8; ++d) ok = ok && nbr8[8 * b + d] != -2;
    if (ok) r = 1;
    else atomicAdd(cnt, 1);
  }
  refv[b] = r;
}

// derefinement of box p: its 4 children are leaves flagged < 0 and no
// neighbour of a child outside the siblings has or gets children (cnt[1]
// counts them)
__global__ void k_qrg_derefine(int n, const int *__restrict__ chl, const int *__restrict__ par,
                               const int *__restrict__ nbr8, const int8_t *__restrict__ flags,
                               const int *__restrict__ refv, int *__restrict__ derv, int *cnt) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  bool ok = chl[4 * p] >= 0;
  for (int c = 0; c < 4 && ok; ++c) {
    const int ch = chl[4 * p + c];
    ok = chl[4 * ch] < 0 && flags[ch] < 0;
  }
  for (int c = 0; c < 4 && ok; ++c) {
    const int ch = chl[4 * p + c];
    for (int d = 0; d < 8 && ok; ++d) {
      const int nb = nbr8[8 * ch + d];
      if (nb >= 0 && par[nb] != p && (chl[4 * nb] >= 0 || refv[nb])) ok = false;
    }
  }
  derv[p] = ok ? 1 : 0;
  if (ok) atomicAdd(cnt + 1, 1);
}

// keepv[b] = b is not a child of a derefined box
__global__ void k_qrg_keep(int n, const int *__restrict__ par, const int *__restrict__ derv,
                           int *__restrict__ keepv) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  const int p = par[b];
  keepv[b] = (p >= 0 && derv[p]) ? 0 : 1;
}

// exclusive prefix sums of two int arrays of n entries (block y = 0: in0 ->
// out0, y = 1: in1 -> out1), out[n] = the total: each thread sums a
// contiguous chunk, the chunk sums are scanned in the block, then each
// thread writes its chunk's prefixes
__global__ void __launch_bounds__(1024) k_qrg_scan2(const int *__restrict__ in0, int *__restrict__ out0,
                                                    const int *__restrict__ in1, int *__restrict__ out1, int n) {
  __shared__ int wsum[32];
  const int *in = blockIdx.y ? in1 : in0;
  int *out = blockIdx.y ? out1 : out0;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int chunk = (n + 1023) / 1024, lo = min(n, t * chunk), hi = min(n, lo + chunk);
  int s = 0;
  for (int i = lo; i < hi; ++i) s += in[i];
  int x = s;  // inclusive scan of the chunk sums: warps, then the warp totals
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    int v = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    wsum[lane] = v;
  }
  __syncthreads();
  int run = x - s + (w ? wsum[w - 1] : 0);
  for (int i = lo; i < hi; ++i) {
    const int v = in[i];
    out[i] = run;
    run += v;
  }
  if (t == 1023) out[n] = wsum[31];
}

// the counts the host needs in one array: dropped and derefined requests,
// then the kept and the refined list positions at the old level offsets
__global__ void k_qrg_counts(const int *__restrict__ cnt, const int *__restrict__ keep_pos,
                             const int *__restrict__ ref_pos, QOffsets off, int nl, int *__restrict__ out) {
  const int t = threadIdx.x;
  if (t < 2) out[t] = cnt[t];
  if (t <= nl) {
    out[2 + t] = keep_pos[off.v[t]];
    out[3 + nl + t] = ref_pos[off.v[t]];
  }
}

// the Morton keys of the kept and of the refined boxes, compacted
__global__ void k_qrg_keys(int n, const int2 *__restrict__ ij, const int *__restrict__ keepv,
                           const int *__restrict__ keep_pos, const int *__restrict__ refv,
                           const int *__restrict__ ref_pos, uint64_t *__restrict__ kept_keys,
                           uint64_t *__restrict__ ref_keys) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  const int2 v = ij[b];
  const uint64_t key = qmorton(v.x, v.y);
  if (keepv[b]) kept_keys[keep_pos[b]] = key;
  if (refv[b]) ref_keys[ref_pos[b]] = key;
}

// new index, level, coordinates and key of every kept box and of the 4
// children of every refined box (4 threads per old box: thread 0 places the
// box itself when kept, thread c its child c when refined), with the move
// descriptor of the new box: its old index, or -1 and the old parent's 3x3
// neighbourhood (old numbering) for a new child
__global__ void k_qrg_place(int n, const int *__restrict__ lev, const int2 *__restrict__ ij,
                            const int *__restrict__ nbr8, const int *__restrict__ keepv,
                            const int *__restrict__ keep_pos, const int *__restrict__ refv,
                            const int *__restrict__ ref_pos, const uint64_t *__restrict__ kept_keys,
                            const uint64_t *__restrict__ ref_keys, QRgLevels L, int *__restrict__ nlev,
                            int2 *__restrict__ nij, uint64_t *__restrict__ nkey, int *__restrict__ rg) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = t >> 2, c = t & 3;
  if (b >= n) return;
  const int l = lev[b];
  const int2 v = ij[b];
  const uint64_t key = qmorton(v.x, v.y);
  if (c == 0 && keepv[b]) {
    // children of refined boxes of level l-1 whose parent key is below this box's
    const int below = l > 0 ? qlower_bound(ref_keys, L.ref[l - 1], L.ref[l], key >> 2) - L.ref[l - 1] : 0;
    const int x = L.nw[l] + (keep_pos[b] - L.kept[l]) + 4 * below;
    nlev[x] = l;
    nij[x] = v;
    nkey[x] = key;
    rg[10 * (size_t)x] = b;
  }
  if (refv[b]) {
    const uint64_t ck = (key << 2) | (uint64_t)c;
    const int below = qlower_bound(kept_keys, L.kept[l + 1], L.kept[l + 2], ck) - L.kept[l + 1];
    const int x = L.nw[l + 1] + 4 * (ref_pos[b] - L.ref[l]) + c + below;
    nlev[x] = l + 1;
    nij[x] = make_int2(2 * v.x + (c & 1), 2 * v.y + (c >> 1));
    nkey[x] = ck;
    int *r = rg + 10 * (size_t)x;
    r[0] = -1;
    for (int k = 0; k < 9; ++k) r[1 + k] = k == 4 ? b : nbr8[8 * b + (k < 4 ? k : k - 1)];
  }
}

// parent and children of every new box by binary search in the new keys
__global__ void k_qrg_links(int m, const int *__restrict__ nlev, const uint64_t *__restrict__ nkey, QRgLevels L,
                            int nlevels, int *__restrict__ par, int *__restrict__ chl) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= m) return;
  const int l = nlev[b];
  const uint64_t key = nkey[b];
  int p = -1;
  if (l > 0) {
    const int i = qlower_bound(nkey, L.nw[l - 1], L.nw[l], key >> 2);
    if (i < L.nw[l] && nkey[i] == key >> 2) p = i;
  }
  par[b] = p;
  int c0 = -1;  // the first child; the four siblings are consecutive keys
  if (l + 1 < nlevels) {
    const int i = qlower_bound(nkey, L.nw[l + 1], L.nw[l + 2], key << 2);
    if (i + 3 < L.nw[l + 2] && nkey[i] == key << 2 && nkey[i + 3] == ((key << 2) | 3ull)) c0 = i;
  }
  for (int c = 0; c < 4; ++c) chl[4 * b + c] = c0 >= 0 ? c0 + c : -1;
}

// same-level neighbours (8 threads per new box, direction d): -1 outside
// the domain, -2 where the level holds no box
__global__ void k_qrg_nbr(int m, const int *__restrict__ nlev, const int2 *__restrict__ nij,
                          const uint64_t *__restrict__ nkey, QRgLevels L, int *__restrict__ nbr8) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = t >> 3, d = t & 7;
  if (b >= m) return;
  const int k = d < 4 ? d : d + 1, dx = k % 3 - 1, dy = k / 3 - 1;
  const int l = nlev[b], side = 1 << l;
  const int2 v = nij[b];
  const int i = v.x + dx, j = v.y + dy;
  int r = -1;
  if (i >= 0 && j >= 0 && i < side && j < side) {
    const uint64_t key = qmorton(i, j);
    const int x = qlower_bound(nkey, L.nw[l], L.nw[l + 1], key);
    r = (x < L.nw[l + 1] && nkey[x] == key) ? x : -2;
  }
  nbr8[8 * b + d] = r;
}

// the tables derived from the links: the parent's 3x3 neighbourhood, the
// refinement bits and the column weights (8 threads per new box, column c)
__global__ void k_qrg_derived(int m, int cyl, const int *__restrict__ par, const int *__restrict__ chl,
                              const int *__restrict__ nbr8, const int2 *__restrict__ ij, int *__restrict__ pn,
                              int *__restrict__ ref, double *__restrict__ w, double *__restrict__ wv) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = t >> 3, c = t & 7;
  if (b >= m) return;
  const int p = par[b];
  const int k = c < 4 ? c : c + 1;  // the 3x3 slots other than the centre
  pn[9 * (size_t)b + k] = p >= 0 ? nbr8[8 * p + c] : -1;
  if (c == 0) {
    pn[9 * (size_t)b + 4] = p;
    int r = chl[4 * b] >= 0 ? 16 : 0;
    const int fd[4] = {3, 4, 1, 6};  // faces -x, +x, -y, +y among the 8 directions
    for (int f = 0; f < 4; ++f) {
      const int nb = nbr8[8 * b + fd[f]];
      if (nb >= 0 && chl[4 * nb] >= 0) r |= 1 << f;
    }
    ref[b] = r;
  }
  // column weights, each operation rounded on its own as on the host
  const int gx = ij[b].x * QN + c;
  const double g = (double)gx, gh = __dadd_rn(g, 0.5);
  const double wl = cyl ? __ddiv_rn(g, gh) : 1.0, wh = cyl ? __ddiv_rn(__dadd_rn(g, 1.0), gh) : 1.0;
  w[24 * (size_t)b + 3 * c] = wl;
  w[24 * (size_t)b + 3 * c + 1] = wh;
  w[24 * (size_t)b + 3 * c + 2] = __ddiv_rn(1.0, __dadd_rn(__dadd_rn(wl, wh), 2.0));
  wv[8 * (size_t)b + c] = cyl ? gh : 1.0;
}

int blocks_for(long long boxes) { return (int)std::max<long long>(1, (boxes + WPB - 1) / WPB); }

}  // namespace

// ---------------------------------------------------------------------------
// context
// ---------------------------------------------------------------------------
struct sm_quad {
  sm_quad_domain dom{};
  int max_boxes = 0, nu1 = 2, nu2 = 2, lbase = 0, lmax = 0;
  cudaStream_t stream = nullptr;
  QBc bc{};
  std::string err;
  long long launches = 0;
  // host tables
  std::vector<int> lev, ix, iy, par, chl, nbr8;
  std::vector<uint64_t> mort;
  int nlev = 0;
  int off[QMAXL + 2] = {0};
  // arena
  char *arena = nullptr;
  int *d_lev = nullptr, *d_par = nullptr, *d_chl = nullptr, *d_nbr8 = nullptr, *d_pn = nullptr, *d_ref = nullptr;
  int2 *d_ij = nullptr;
  double *d_w = nullptr, *d_wv = nullptr;
  double *var[NV] = {nullptr};
  double *cflux = nullptr, *ainv = nullptr, *lut = nullptr, *d_h = nullptr;
  unsigned long long *slots = nullptr;
  unsigned *d_err = nullptr;
  unsigned long long *xch = nullptr;      // exchange words of the one-launch legs [max_boxes][4][8][2]
  unsigned *xseq = nullptr;               // their tag counter
  int *rcount = nullptr;                  // [max_boxes] children counted in by k_q_restrict_tree (zero between)
  int leg_few = 0;                        // boxes of the largest level for the form with more registers
  int leg_max = -1;                       // boxes of the largest level with such legs (-1: not looked up)
  bool legs_off = false;                  // a wait ran out on this mesh: every level by separate launches
  unsigned leg_skew = 0;                  // != 0: the legs' waits run out (sm_quad_leg_wait_selftest)
  double *snap = nullptr;                 // snapshot of a regrid [6][max_boxes][64]; of a solve's first potential
  int *d_rg = nullptr;                    // regrid move descriptors [max_boxes][10]
  unsigned long long *d_need = nullptr;   // refinement test: cells that need refinement, per box
  char *rgw = nullptr;                    // scratch of a regrid (QRgScratch)
  unsigned char *d_fine = nullptr;        // refinement test: derefinable, per box
  int lut_n = 0;
  double lut_emax = 0.0;
  double h[QMAXL], inv_h2[QMAXL];
  std::vector<double> h_ainv;
  // V-cycle graphs per top level (captured on first use, dropped when the
  // mesh changes) and the launches each holds
  cudaStream_t cap = nullptr;
  cudaGraphExec_t vgraph[QMAXL] = {nullptr};
  long long vgraph_launches[QMAXL] = {0};
  // whole solves with the cycle loop on the device [fmg]: launches before the
  // loop and per cycle
  cudaStream_t cap2 = nullptr;
  cudaGraphExec_t sgraph[2] = {nullptr, nullptr};
  long long sgraph_launches[2][2] = {{0, 0}, {0, 0}};
  bool graphs = true, pdl = true;
  ~sm_quad() {
    for (auto &g : vgraph)
      if (g) cudaGraphExecDestroy(g);
    for (auto &g : sgraph)
      if (g) cudaGraphExecDestroy(g);
    if (cap) cudaStreamDestroy(cap);
    if (cap2) cudaStreamDestroy(cap2);
  }
};

namespace {

int qfail(sm_quad *q, int code, const std::string &msg) {
  if (q) q->err = msg;
  return code;
}

uint64_t morton2(int i, int j) {
  uint64_t k = 0;
  for (int b = 0; b < 31; ++b) k |= (uint64_t)((i >> b) & 1) << (2 * b) | (uint64_t)((j >> b) & 1) << (2 * b + 1);
  return k;
}

int dir8h(int dx, int dy) {
  const int d = (dx + 1) + 3 * (dy + 1);
  return d < 4 ? d : d - 1;
}

int find_box(const sm_quad *q, int l, int i, int j) {
  const int n = 1 << l;
  if (i < 0 || j < 0 || i >= n || j >= n) return -1;
  if (l >= q->nlev) return -2;
  const uint64_t key = morton2(i, j);
  int lo = q->off[l], hi = q->off[l + 1] - 1;
  while (lo <= hi) {
    const int mid = (lo + hi) / 2;
    if (q->mort[mid] == key) return mid;
    if (q->mort[mid] < key) lo = mid + 1;
    else hi = mid - 1;
  }
  return -2;
}

// weights of the column with global x index gx (at its box's level):
// w_lo, w_hi, 1/(w_lo + w_hi + 2) and the volume weight; the same roundings
// as the device's regrid tables (col_weights_dev)
void col_weights(const sm_quad *q, int gx, double *w3, double *wv) {
  const bool cyl = q->dom.geometry == SM_AXISYMMETRIC;
  const double wl = cyl ? (double)gx / (gx + 0.5) : 1.0, wh = cyl ? (gx + 1.0) / (gx + 0.5) : 1.0;
  w3[0] = wl;
  w3[1] = wh;
  w3[2] = 1.0 / (wl + wh + 2.0);
  *wv = cyl ? gx + 0.5 : 1.0;
}

void add_box(sm_quad *q, int l, int i, int j, int parent) {
  q->lev.push_back(l);
  q->ix.push_back(i);
  q->iy.push_back(j);
  q->par.push_back(parent);
  q->mort.push_back(morton2(i, j));
  for (int c = 0; c < 4; ++c) q->chl.push_back(-1);
  for (int d = 0; d < 8; ++d) q->nbr8.push_back(-2);
}

void set_neighbours(sm_quad *q, int l) {
  for (int b = q->off[l]; b < q->off[l + 1]; ++b)
    for (int dy = -1; dy <= 1; ++dy)
      for (int dx = -1; dx <= 1; ++dx)
        if (dx || dy) q->nbr8[8 * b + dir8h(dx, dy)] = find_box(q, l, q->ix[b] + dx, q->iy[b] + dy);
}

int n_boxes(const sm_quad *q) { return (int)q->lev.size(); }

int upload_tables(sm_quad *q) {
  const int n = n_boxes(q);
  std::vector<int2> ij(n);
  std::vector<int> pn(9 * (size_t)n, -1), ref(n, 0);
  std::vector<double> w(24 * (size_t)n), wv(8 * (size_t)n);
  for (int b = 0; b < n; ++b) {
    ij[b] = make_int2(q->ix[b], q->iy[b]);
    for (int c = 0; c < QN; ++c) col_weights(q, q->ix[b] * QN + c, &w[24 * (size_t)b + 3 * c], &wv[8 * (size_t)b + c]);
    const int p = q->par[b];
    if (p >= 0)
      for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx)
          pn[9 * (size_t)b + (dx + 1) + 3 * (dy + 1)] = (dx || dy) ? q->nbr8[8 * p + dir8h(dx, dy)] : p;
    int r = q->chl[4 * b] >= 0 ? 16 : 0;
    const int fd[4] = {dir8h(-1, 0), dir8h(1, 0), dir8h(0, -1), dir8h(0, 1)};
    for (int f = 0; f < 4; ++f) {
      const int nb = q->nbr8[8 * b + fd[f]];
      if (nb >= 0 && q->chl[4 * nb] >= 0) r |= 1 << f;
    }
    ref[b] = r;
  }
  cudaStream_t s = q->stream;
  if (cudaMemcpyAsync(q->d_lev, q->lev.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_par, q->par.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_chl, q->chl.data(), sizeof(int) * 4 * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_nbr8, q->nbr8.data(), sizeof(int) * 8 * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_ij, ij.data(), sizeof(int2) * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_pn, pn.data(), sizeof(int) * 9 * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_ref, ref.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_w, w.data(), sizeof(double) * 24 * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_wv, wv.data(), sizeof(double) * 8 * n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return qfail(q, SM_ECUDA, "table upload");
  return SM_OK;
}

QTabs tabs(const sm_quad *q) {
  return {q->d_lev, q->d_par, q->d_chl, q->d_nbr8, q->d_pn, q->d_ref, q->d_ij, q->d_w, q->d_wv};
}
Table qtable(const sm_quad *q) {
  Table tb = {};
  sm::table_index_consts(tb, q->lut + 3 * 4096, q->lut_n, q->lut_emax);
  return tb;
}

// the level-0 operator with homogeneous wall ghosts (columns L e_k) and its
// inverse by Gauss-Jordan elimination with partial pivoting (host)
void coarse_inverse(sm_quad *q) {
  const int n = QC;
  std::vector<double> A((size_t)n * n, 0.0), I((size_t)n * n, 0.0);
  const double ih2 = q->inv_h2[0];
  for (int r = 0; r < n; ++r) {
    const int i = r % QN, j = r / QN;
    double w3[3], wvol;
    col_weights(q, i, w3, &wvol);  // level 0: box 0, global column i
    const double wl = w3[0], wh = w3[1];
    const double wf[4] = {wl, wh, 1.0, 1.0};
    const int nbr[4] = {i > 0 ? r - 1 : -1, i < QN - 1 ? r + 1 : -1, j > 0 ? r - QN : -1, j < QN - 1 ? r + QN : -1};
    for (int f = 0; f < 4; ++f) {
      // L phi = sum_f w_f (phi_f - phi): a wall ghost is -phi (Dirichlet) or phi
      A[(size_t)r * n + r] -= wf[f] * ih2;
      if (nbr[f] >= 0) A[(size_t)r * n + nbr[f]] += wf[f] * ih2;
      else A[(size_t)r * n + r] += (q->bc.type[f] ? -1.0 : 1.0) * wf[f] * ih2;
    }
    I[(size_t)r * n + r] = 1.0;
  }
  for (int c = 0; c < n; ++c) {
    int p = c;
    for (int r = c + 1; r < n; ++r)
      if (std::fabs(A[(size_t)r * n + c]) > std::fabs(A[(size_t)p * n + c])) p = r;
    if (p != c)
      for (int k = 0; k < n; ++k) {
        std::swap(A[(size_t)c * n + k], A[(size_t)p * n + k]);
        std::swap(I[(size_t)c * n + k], I[(size_t)p * n + k]);
      }
    const double d = A[(size_t)c * n + c];
    for (int k = 0; k < n; ++k) {
      A[(size_t)c * n + k] /= d;
      I[(size_t)c * n + k] /= d;
    }
    for (int r = 0; r < n; ++r) {
      if (r == c) continue;
      const double m = A[(size_t)r * n + c];
      if (m == 0.0) continue;
      for (int k = 0; k < n; ++k) {
        A[(size_t)r * n + k] -= m * A[(size_t)c * n + k];
        I[(size_t)r * n + k] -= m * I[(size_t)c * n + k];
      }
    }
  }
  q->h_ainv = I;
}

int check(sm_quad *q, const char *what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return qfail(q, SM_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
  return SM_OK;
}

int level_count(const sm_quad *q, int l) { return q->off[l + 1] - q->off[l]; }

// launch with programmatic dependent launch (every kernel of this file
// waits for its predecessor before reading a field)
template <typename... KArgs, typename... Args>
void qlaunch(sm_quad *q, void (*k)(KArgs...), int grid, int block, Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = q->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = q->pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
  ++q->launches;
}

// nu red-black sweeps of level l; with skip_first the first colour pass has
// already run (k_q_fas_rbgs0)
void smooth(sm_quad *q, int l, int nu, bool skip_first = false) {
  const int n = level_count(q, l);
  for (int s = 0; s < nu; ++s)
    for (int c = 0; c < 2; ++c) {
      if (skip_first && s == 0 && c == 0) continue;
      qlaunch(q, k_q_rbgs, blocks_for(n), QT, q->off[l], n, l, c, q->var[V_PHI], (const double *)q->var[V_RHS],
              tabs(q), q->bc, q->h[l] * q->h[l], q->d_err);
    }
}

void coarse_solve(sm_quad *q) {
  qlaunch(q, k_q_coarse, 1, QC, q->var[V_PHI], (const double *)q->var[V_RHS], (const double *)q->ainv, tabs(q),
          q->bc, q->inv_h2[0], q->xseq);
}

// blocks per SM of the two forms of a leg kernel (200 and 72 registers)
constexpr int LEG_FEW = 10, LEG_MANY = 28;

// Boxes of the largest level whose legs run in one launch (a warp per box,
// all resident at once); 0 without cooperative launch.
int leg_limit(sm_quad *q) {
  if (q->leg_max >= 0) return q->leg_max;
  int dev = 0, coop = 0, sms = 0, most = 1 << 30;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto fits = [&](auto *k) {
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 32, 0) != cudaSuccess) per = 0;
    most = std::min(most, per * sms);
  };
  // the forms for levels of few boxes and of many
  fits(k_q_leg<QL_TOP, LEG_FEW>);
  fits(k_q_leg<QL_FAS, LEG_FEW>);
  fits(k_q_leg<QL_PROLONG, LEG_FEW>);
  fits(k_q_leg<QL_FMG, LEG_FEW>);
  q->leg_few = most;
  most = 1 << 30;
  fits(k_q_leg<QL_TOP, LEG_MANY>);
  fits(k_q_leg<QL_FAS, LEG_MANY>);
  fits(k_q_leg<QL_PROLONG, LEG_MANY>);
  fits(k_q_leg<QL_FMG, LEG_MANY>);
  cudaGetLastError();
  return q->leg_max = coop ? most : 0;
}

bool leg_level(sm_quad *q, int l) {
  return !q->legs_off && l >= 1 && level_count(q, l) > 0 && level_count(q, l) <= leg_limit(q);
}

bool any_leg(sm_quad *q) {
  for (int l = 1; l < q->nlev; ++l)
    if (leg_level(q, l)) return true;
  return false;
}

template <int START>
void leg(sm_quad *q, int l) {
  constexpr bool up = START == QL_PROLONG;
  QLeg a = {};
  a.lo = q->off[l];
  a.nu = up ? q->nu2 : q->nu1;
  a.leg = up ? 0u : 64u;
  a.skew = q->leg_skew;
  a.h2 = q->h[l] * q->h[l];
  a.inv_h2 = q->inv_h2[l];
  a.phi = q->var[V_PHI];
  a.rhs = q->var[V_RHS];
  a.old = q->var[V_OLD];
  a.xch = q->xch;
  a.seq = q->xseq;
  a.err = q->d_err;
  a.lev = l;
  a.T = tabs(q);
  a.bc = q->bc;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(level_count(q, l));
  cfg.blockDim = dim3(32);
  cfg.stream = q->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (level_count(q, l) <= q->leg_few) cudaLaunchKernelEx(&cfg, k_q_leg<START, LEG_FEW>, a);
  else cudaLaunchKernelEx(&cfg, k_q_leg<START, LEG_MANY>, a);
  ++q->launches;
}

// One V-cycle with level `top` on top; with fmg that level first takes the
// prolonged solution of the level below.  A level whose boxes are all
// resident at once runs each leg in one launch, a larger one a launch per
// operation (below another such level the FAS completion also runs the first
// colour pass, on a copy of the whole level that the restriction leaves in
// old).
void vcycle(sm_quad *q, int top, bool fmg = false) {
  bool fused = false;  // the first colour pass of level l has run (k_q_fas_rbgs0)
  if (fmg && !leg_level(q, top)) {
    const int n = level_count(q, top);
    qlaunch(q, k_q_prolong, blocks_for(n), QT, q->off[top], n, top, q->var[V_PHI], (const double *)q->var[V_OLD], 0,
            tabs(q), q->bc, q->d_err);
  }
  for (int l = top; l >= 1; --l) {
    const int n = level_count(q, l), nc = level_count(q, l - 1);
    if (leg_level(q, l)) {
      if (l < top) leg<QL_FAS>(q, l);
      else if (fmg) leg<QL_FMG>(q, l);
      else leg<QL_TOP>(q, l);
      fused = false;
    } else {
      smooth(q, l, q->nu1, fused);
      fused = l - 1 >= 1 && !leg_level(q, l - 1);
      const int ncp = fused ? nc : 0;
      qlaunch(q, k_q_resid_restrict, blocks_for(n + ncp), QT, q->off[l], n, l, (const double *)q->var[V_PHI],
              q->var[V_RHS], q->var[V_OLD], tabs(q), q->bc, q->inv_h2[l], q->d_err, q->off[l - 1], ncp);
    }
    if (leg_level(q, l - 1)) continue;  // its leg completes the FAS right-hand side
    if (fused)
      qlaunch(q, k_q_fas_rbgs0, blocks_for(nc), QT, q->off[l - 1], nc, l - 1, q->var[V_PHI], q->var[V_RHS],
              (const double *)q->var[V_OLD], tabs(q), q->bc, q->inv_h2[l - 1], q->h[l - 1] * q->h[l - 1], q->d_err);
    else
      qlaunch(q, k_q_fas, blocks_for(nc), QT, q->off[l - 1], nc, l - 1, q->var[V_PHI], q->var[V_RHS],
              q->var[V_OLD], tabs(q), q->bc, q->inv_h2[l - 1], q->d_err);
  }
  coarse_solve(q);
  for (int l = 1; l <= top; ++l) {
    if (leg_level(q, l)) {
      leg<QL_PROLONG>(q, l);
      continue;
    }
    const int n = level_count(q, l);
    qlaunch(q, k_q_prolong, blocks_for(n), QT, q->off[l], n, l, q->var[V_PHI], (const double *)q->var[V_OLD], 1,
            tabs(q), q->bc, q->d_err);
    smooth(q, l, q->nu2);
  }
}

void drop_graphs(sm_quad *q) {
  auto drop = [](cudaGraphExec_t &g) {
    if (g) cudaGraphExecDestroy(g);
    g = nullptr;
  };
  for (auto &g : q->vgraph) drop(g);
  for (auto &g : q->sgraph) drop(g);
  q->legs_off = false;
}

// One V-cycle with level `top` on top, as a CUDA graph captured on first
// use (the same launches as vcycle; host launch gaps removed)
int vcycle_g(sm_quad *q, int top) {
  leg_limit(q);  // occupancy queries outside the capture
  if (!q->graphs) {
    vcycle(q, top);
    return check(q, "V-cycle");
  }
  if (!q->vgraph[top]) {
    if (!q->cap && cudaStreamCreateWithFlags(&q->cap, cudaStreamNonBlocking) != cudaSuccess)
      return qfail(q, SM_ECUDA, "capture stream");
    cudaStream_t saved = q->stream;
    const long long l0 = q->launches;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(q->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
      return qfail(q, SM_ECUDA, "begin capture");
    q->stream = q->cap;
    vcycle(q, top);
    q->stream = saved;
    const cudaError_t e = cudaStreamEndCapture(q->cap, &g);
    if (e != cudaSuccess || !g) {
      cudaGetLastError();
      return qfail(q, SM_ECUDA, "V-cycle capture");
    }
    const cudaError_t ei = cudaGraphInstantiate(&q->vgraph[top], g, 0);
    cudaGraphDestroy(g);
    q->vgraph_launches[top] = q->launches - l0;
    q->launches = l0;
    if (ei != cudaSuccess) {
      q->vgraph[top] = nullptr;
      return qfail(q, SM_ECUDA, "V-cycle instantiate");
    }
  }
  if (cudaGraphLaunch(q->vgraph[top], q->stream) != cudaSuccess) return qfail(q, SM_ECUDA, "graph launch");
  q->launches += q->vgraph_launches[top];
  return SM_OK;
}

void restrict_all(sm_quad *q, int v, int v2 = -1);

// Status of a wait of a one-launch leg that ran out, from the device's error
// word (the stream is idle): its bit is cleared and the following V-cycles run
// in a launch per operation, until the mesh changes.
int wait_error(sm_quad *q, unsigned e) {
  if (!(e & Q_ERR_WAIT)) return SM_OK;
  const unsigned rest = e & ~Q_ERR_WAIT;
  if (cudaMemcpyAsync(q->d_err, &rest, sizeof(rest), cudaMemcpyHostToDevice, q->stream) != cudaSuccess ||
      cudaStreamSynchronize(q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "error word");
  drop_graphs(q);
  q->leg_skew = 0;
  q->legs_off = true;
  return qfail(q, SM_ETIMEOUT, "a wait between the blocks of a kernel ran out");
}

// status of the device's error word
int device_error(sm_quad *q, unsigned e) {
  if (int st = wait_error(q, e)) return st;
  if (e) return qfail(q, SM_ESTATE, "a coarse box needed at a refinement boundary is missing");
  return SM_OK;
}

// max leaf residual of var (the potential, or the zero array) into a slot;
// with `keep` the potential is copied there
void resmax(sm_quad *q, int v, int slot, double *keep = nullptr) {
  const int n = n_boxes(q);
  cudaMemsetAsync(q->slots + slot, 0, sizeof(unsigned long long), q->stream);
  k_q_resmax<<<blocks_for(n), QT, 0, q->stream>>>(n, q->var[v], q->var[V_RHS], tabs(q), q->bc, q->d_h + QMAXL,
                                                   q->slots + slot, q->d_err, q->var[V_PHI], keep);
  ++q->launches;
}

// the solve's scalars and the error word (synchronises)
int read_solve(sm_quad *q, unsigned long long (&s)[QS_N]) {
  unsigned e = 0;
  if (cudaMemcpyAsync(s, q->slots, sizeof(s), cudaMemcpyDeviceToHost, q->stream) != cudaSuccess ||
      cudaMemcpyAsync(&e, q->d_err, sizeof(e), cudaMemcpyDeviceToHost, q->stream) != cudaSuccess ||
      cudaStreamSynchronize(q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "residual norm");
  return device_error(q, e);
}

double bits_of(unsigned long long b) {
  double d;
  std::memcpy(&d, &b, sizeof(d));
  return d;
}

// work before the cycle loop: the residual of phi = 0 (the denominator), and
// for FMG the restricted right-hand side, the ladder and its residual; with
// one-launch legs the potential the cycles start from is kept, for the case
// that a wait runs out (FMG does not read it)
void solve_prefix(sm_quad *q, bool fmg) {
  resmax(q, V_ZERO, QS_DEN, !fmg && any_leg(q) ? q->snap : nullptr);
  if (!fmg) return;
  restrict_all(q, V_RHS);
  coarse_solve(q);
  for (int l = 1; l < q->nlev; ++l) vcycle(q, l, true);
  resmax(q, V_PHI, QS_NUM);
}

void solve_body(sm_quad *q) {
  vcycle(q, q->nlev - 1);
  resmax(q, V_PHI, QS_NUM);
}

void solve_check(sm_quad *q, cudaGraphConditionalHandle h) {
  k_q_check<<<1, 1, 0, q->stream>>>(h, q->slots, q->d_err);  // not counted: the host loop tests without a launch
}

// Capture prefix + WHILE { cycle; check } into an executable graph (an FMG
// result is checked once before the loop and counts as cycle 1; otherwise
// the body runs at least once).
int capture_solve(sm_quad *q, bool fmg) {
  if ((!q->cap && cudaStreamCreateWithFlags(&q->cap, cudaStreamNonBlocking) != cudaSuccess) ||
      (!q->cap2 && cudaStreamCreateWithFlags(&q->cap2, cudaStreamNonBlocking) != cudaSuccess))
    return qfail(q, SM_ECUDA, "capture stream");
  leg_limit(q);  // occupancy queries outside the capture
  cudaStream_t saved = q->stream;
  const long long l0 = q->launches;
  long long l1 = l0, l2 = l0;
  cudaGraph_t g = nullptr, body = nullptr, whole = nullptr;
  bool ok = cudaStreamBeginCapture(q->cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
  if (ok) {
    q->stream = q->cap;
    cudaStreamCaptureStatus cs;
    cudaGraphConditionalHandle h = 0;
    const cudaGraphNode_t *deps = nullptr;
    size_t nd = 0;
    cudaGraphNode_t node;
    // the node-parameter union has no default constructor: zeroed raw storage
    alignas(cudaGraphNodeParams) unsigned char pbuf[sizeof(cudaGraphNodeParams)];
    std::memset(pbuf, 0, sizeof pbuf);
    cudaGraphNodeParams &p = *reinterpret_cast<cudaGraphNodeParams *>(pbuf);
    ok = cudaStreamGetCaptureInfo(q->cap, &cs, nullptr, &g, nullptr, nullptr, nullptr) == cudaSuccess &&
         cudaGraphConditionalHandleCreate(&h, g, fmg ? 0u : 1u, cudaGraphCondAssignDefault) == cudaSuccess;
    if (ok) {
      solve_prefix(q, fmg);
      if (fmg) solve_check(q, h);
      l1 = q->launches;
      p.type = cudaGraphNodeTypeConditional;
      p.conditional.handle = h;
      p.conditional.type = cudaGraphCondTypeWhile;
      p.conditional.size = 1;
      ok = cudaStreamGetCaptureInfo(q->cap, &cs, nullptr, nullptr, &deps, nullptr, &nd) == cudaSuccess &&
           cudaGraphAddNode(&node, g, deps, nullptr, nd, &p) == cudaSuccess;
    }
    if (ok) {
      body = p.conditional.phGraph_out[0];
      ok = cudaStreamUpdateCaptureDependencies(q->cap, &node, nullptr, 1, cudaStreamSetCaptureDependencies) ==
               cudaSuccess &&
           cudaStreamBeginCaptureToGraph(q->cap2, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) ==
               cudaSuccess;
    }
    if (ok) {
      q->stream = q->cap2;
      solve_body(q);
      solve_check(q, h);
      l2 = q->launches;
      ok = cudaStreamEndCapture(q->cap2, &body) == cudaSuccess;
    }
    q->stream = saved;
    ok = cudaStreamEndCapture(q->cap, &whole) == cudaSuccess && ok;
  }
  q->launches = l0;
  q->sgraph_launches[fmg][0] = l1 - l0;
  q->sgraph_launches[fmg][1] = l2 - l1;
  ok = ok && cudaGraphInstantiate(&q->sgraph[fmg], whole, 0) == cudaSuccess;
  if (whole) cudaGraphDestroy(whole);
  if (!ok) {
    q->sgraph[fmg] = nullptr;
    cudaGetLastError();
    return qfail(q, SM_ECUDA, "solve capture");
  }
  return SM_OK;
}

// FMG, or V-cycles from the current potential, until the relative residual is
// at most tol: one graph with the loop on the device, or the same launches
// with a read after every cycle
int run_solve_once(sm_quad *q, bool fmg, double tol, int max_cycles, int &c, double &r) {
  unsigned long long s[QS_N];
  c = 0;
  r = 0.0;
  if (q->graphs) {
    if (!q->sgraph[fmg])
      if (int st = capture_solve(q, fmg)) return st;
    k_q_begin<<<1, 1, 0, q->stream>>>(q->slots, tol, max_cycles);
    if (cudaGraphLaunch(q->sgraph[fmg], q->stream) != cudaSuccess) return qfail(q, SM_ECUDA, "graph launch");
    if (int st = read_solve(q, s)) return st;
    c = (int)s[QS_CYC];
    r = bits_of(s[QS_REL]);
    q->launches += q->sgraph_launches[fmg][0] + q->sgraph_launches[fmg][1] * (long long)(fmg ? c - 1 : c);
  } else {
    solve_prefix(q, fmg);
    auto residual = [&] {
      const int st = read_solve(q, s);
      const double num = bits_of(s[QS_NUM]), den = bits_of(s[QS_DEN]);
      r = den > 0.0 ? num / den : num;
      return st;
    };
    if (fmg) {
      c = 1;
      if (int st = residual()) return st;
    }
    while (c == 0 || (r > tol && c < max_cycles)) {
      solve_body(q);
      ++c;
      if (int st = residual()) return st;
    }
  }
  return check(q, "solve");
}

// The solve; when a wait of a one-launch leg ran out (its blocks got no turn
// on the GPU for that long) once more from the potential it started with, in
// a launch per operation.
int run_solve(sm_quad *q, bool fmg, double tol, int max_cycles, int *cycles, double *rel) {
  int c, st;
  double r;
  if ((st = run_solve_once(q, fmg, tol, max_cycles, c, r)) == SM_ETIMEOUT) {
    if (!fmg && cudaMemcpyAsync(q->var[V_PHI], q->snap, sizeof(double) * QC * (size_t)n_boxes(q),
                                cudaMemcpyDeviceToDevice, q->stream) != cudaSuccess)
      return qfail(q, SM_ECUDA, "potential");
    st = run_solve_once(q, fmg, tol, max_cycles, c, r);
  }
  if (st) return st;
  if (cycles) *cycles = c;
  if (rel) *rel = r;
  return r <= tol ? SM_OK : qfail(q, SM_ENOCONV, "tolerance not reached");
}

// refined boxes of variable v (and v2) := the mean of their children
void restrict_all(sm_quad *q, int v, int v2) {
  if (q->nlev < 2) return;
  const int n = n_boxes(q);
  k_q_restrict_tree<<<blocks_for(n), QT, 0, q->stream>>>(n, q->var[v], v2 >= 0 ? q->var[v2] : nullptr, tabs(q),
                                                          q->rcount);
  ++q->launches;
}

// one Euler stage of (sne, sni) into (dne, dni); with n0e >= 0 averaged with
// (n0e, n0i), leaving the time-step maxima in slots 0..2; with `charge` the
// right-hand side (n_i - n_e) qie too, zero where qie is
int euler_stage(sm_quad *q, int sne, int sni, int dne, int dni, double dt, bool charge, double qie, int n0e = -1,
                int n0i = -1) {
  const int n = n_boxes(q);
  k_q_cf_flux<<<blocks_for(n), QT, 0, q->stream>>>(n, q->var[sne], q->var[V_PHI], q->var[V_EMAG], q->cflux, tabs(q),
                                                    q->bc, qtable(q), q->d_h, q->d_err);
  auto run = [&](auto kernel) {
    kernel<<<blocks_for(n), QT, 0, q->stream>>>(
        n, q->var[sne], q->var[sni], n0e >= 0 ? q->var[n0e] : nullptr, n0e >= 0 ? q->var[n0i] : nullptr, q->var[dne],
        q->var[dni], charge ? q->var[V_RHS] : nullptr, q->var[V_PHI], q->var[V_EMAG], q->cflux, tabs(q), q->bc,
        qtable(q), q->d_h, dt, qie, q->slots, q->d_err);
  };
  if (n0e >= 0) run(k_q_update<true>);
  else run(k_q_update<false>);
  q->launches += 2;
  restrict_all(q, dne, dni);
  return check(q, "fluid stage");
}

int charge(sm_quad *q, double c, double eps, int use_rho) {
  const long long cells = (long long)n_boxes(q) * QC;
  k_q_charge<<<(int)((cells + 255) / 256), 256, 0, q->stream>>>(n_boxes(q), q->var[V_RHS], q->var[V_NE],
                                                                  q->var[V_NI], q->var[V_RHO], q->d_chl, c, 1.0 / eps,
                                                                  use_rho);
  ++q->launches;
  return check(q, "charge");
}

int field(sm_quad *q) {
  const int n = n_boxes(q);
  k_q_field<<<blocks_for(n), QT, 0, q->stream>>>(n, q->var[V_PHI], q->var[V_EMAG], tabs(q), q->bc,
                                                  q->d_h + 2 * QMAXL, q->d_err);
  ++q->launches;
  return check(q, "field");
}

// the time step from the maxima in slots 0..2 (synchronises)
int dt_read(sm_quad *q, double c, double eps, double *dt) {
  unsigned long long bits[3];
  unsigned e = 0;
  if (cudaMemcpyAsync(bits, q->slots, sizeof(bits), cudaMemcpyDeviceToHost, q->stream) != cudaSuccess ||
      cudaMemcpyAsync(&e, q->d_err, sizeof(e), cudaMemcpyDeviceToHost, q->stream) != cudaSuccess ||
      cudaStreamSynchronize(q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "dt limit");
  if (int st = wait_error(q, e)) return st;
  double m[3];
  std::memcpy(m, bits, sizeof(m));
  double d = 1e300;
  if (m[0] > 0.0 && 0.5 / m[0] < d) d = 0.5 / m[0];
  if (m[1] > 0.0 && 1.0 / m[1] < d) d = 1.0 / m[1];
  if (m[2] > 0.0 && eps / (c * m[2]) < d) d = eps / (c * m[2]);
  *dt = 0.9 * d;
  return SM_OK;
}

int dt_limit(sm_quad *q, double c, double eps, double *dt) {
  const int n = n_boxes(q);
  if (cudaMemsetAsync(q->slots, 0, 3 * sizeof(unsigned long long), q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "memset");
  k_q_dt<<<blocks_for(n), QT, 0, q->stream>>>(n, q->var[V_PHI], q->var[V_EMAG], q->var[V_NE], tabs(q), q->bc,
                                               qtable(q), q->d_h, q->slots, q->d_err);
  ++q->launches;
  return dt_read(q, c, eps, dt);
}

}  // namespace

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" int sm_quad_create(sm_quad **out, const sm_quad_domain *dom, int max_boxes, int nu1, int nu2,
                              void *stream) {
  if (!out || !dom) return SM_EINVAL;
  *out = nullptr;
  int lb = 0;
  while ((1 << lb) < dom->nb) ++lb;
  if (dom->nb < 1 || (1 << lb) != dom->nb || dom->max_level < 0 || lb + dom->max_level >= QMAXL ||
      !(dom->length > 0.0) || nu1 < 1 || nu2 < 1 || nu1 > 16 || nu2 > 16 ||
      (dom->geometry != SM_CARTESIAN && dom->geometry != SM_AXISYMMETRIC))
    return SM_EINVAL;
  if (dom->geometry == SM_AXISYMMETRIC && dom->origin[0] != 0.0) return SM_EINVAL;
  int dir = 0;
  for (int f = 0; f < 4; ++f) {
    if (dom->bc_type[f] != 0 && dom->bc_type[f] != 1) return SM_EINVAL;
    if (f > 0 || dom->geometry == SM_CARTESIAN) dir |= dom->bc_type[f];
  }
  if (!dir) return SM_EINVAL;
  long long uniform = 0;
  for (int l = 0; l <= lb; ++l) uniform += 1ll << (2 * l);
  if (max_boxes < uniform) return SM_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return SM_ECUDA;
  }
  sm_quad *q = new sm_quad();
  q->dom = *dom;
  q->max_boxes = max_boxes;
  q->nu1 = nu1;
  q->nu2 = nu2;
  q->lbase = lb;
  q->lmax = lb + dom->max_level;
  q->stream = (cudaStream_t)stream;
  for (int f = 0; f < 4; ++f) {
    const bool axis = dom->geometry == SM_AXISYMMETRIC && f == 0;
    q->bc.type[f] = axis ? 0 : dom->bc_type[f];
    q->bc.g2[f] = axis ? 0.0 : 2.0 * dom->bc_val[f];
  }
  for (int l = 0; l < QMAXL; ++l) {
    q->h[l] = dom->length / (QN * (double)(1ll << l));
    q->inv_h2[l] = 1.0 / (q->h[l] * q->h[l]);
  }
  // uniform levels, each in Morton order
  for (int l = 0; l <= lb; ++l) {
    q->off[l] = n_boxes(q);
    const uint64_t nk = 1ull << (2 * l);
    for (uint64_t key = 0; key < nk; ++key) {
      int i = 0, j = 0;
      for (int b = 0; b < 31; ++b) {
        i |= (int)((key >> (2 * b)) & 1) << b;
        j |= (int)((key >> (2 * b + 1)) & 1) << b;
      }
      add_box(q, l, i, j, l ? q->off[l - 1] + (int)(key >> 2) : -1);
    }
    q->off[l + 1] = n_boxes(q);
  }
  for (int l = 0; l < lb; ++l)
    for (int b = q->off[l]; b < q->off[l + 1]; ++b)
      for (int c = 0; c < 4; ++c) q->chl[4 * b + c] = q->off[l + 1] + (int)((q->mort[b] << 2) | (uint64_t)c);
  q->nlev = lb + 1;
  for (int l = 0; l <= lb; ++l) set_neighbours(q, l);
  coarse_inverse(q);
  *out = q;
  return SM_OK;
}

extern "C" int sm_quad_destroy(sm_quad *q) {
  delete q;
  return SM_OK;
}

namespace {
struct QLayout {
  size_t lev, par, chl, nbr8, pn, ref, ij, w, wv, var[NV], cflux, ainv, lut, h, slots, err, xch, xseq, rcount, snap, rg, need, fine,
      rgw, total;
};

// hands out 256-byte aligned parts of a range, and counts them when there is
// no range yet
struct Parts {
  char *base = nullptr;
  size_t t = 0;
  size_t take(size_t bytes) {
    const size_t at = t;
    t = (t + bytes + 255) & ~(size_t)255;
    return at;
  }
  template <typename T>
  T *of(size_t n) {
    const size_t at = take(sizeof(T) * n);
    return base ? reinterpret_cast<T *>(base + at) : nullptr;
  }
};

// scratch of a regrid on at most M boxes; at(nullptr, M) gives its size alone
struct QRgScratch {
  int8_t *flags;
  int *refv, *keepv, *derv, *ref_pos, *keep_pos;
  uint64_t *ref_keys, *kept_keys;
  int *nlev;
  int2 *nij;
  uint64_t *nkey;
  int *cnt, *counts;
  size_t bytes;
  static QRgScratch at(char *base, size_t M) {
    QRgScratch S;
    Parts p{base};
    S.flags = p.of<int8_t>(M);
    S.refv = p.of<int>(M);
    S.keepv = p.of<int>(M);
    S.derv = p.of<int>(M);
    S.ref_pos = p.of<int>(M + 1);
    S.keep_pos = p.of<int>(M + 1);
    S.ref_keys = p.of<uint64_t>(M);
    S.kept_keys = p.of<uint64_t>(M);
    S.nlev = p.of<int>(M);
    S.nij = p.of<int2>(M);
    S.nkey = p.of<uint64_t>(M);
    S.cnt = p.of<int>(2);
    S.counts = p.of<int>(2 * QMAXL + 8);
    S.bytes = p.t;
    return S;
  }
};

QLayout qlayout(const sm_quad *q) {
  QLayout L{};
  Parts p;
  auto take = [&](size_t bytes) { return p.take(bytes); };
  const size_t nb = (size_t)q->max_boxes;
  L.lev = take(sizeof(int) * nb);
  L.par = take(sizeof(int) * nb);
  L.chl = take(sizeof(int) * 4 * nb);
  L.nbr8 = take(sizeof(int) * 8 * nb);
  L.pn = take(sizeof(int) * 9 * nb);
  L.ref = take(sizeof(int) * nb);
  L.ij = take(sizeof(int2) * nb);
  L.w = take(sizeof(double) * 24 * nb);
  L.wv = take(sizeof(double) * 8 * nb);
  for (int v = 0; v < NV; ++v) L.var[v] = take(sizeof(double) * QC * nb);
  L.cflux = take(sizeof(double) * 32 * nb);
  L.ainv = take(sizeof(double) * QC * QC);
  L.lut = take(sizeof(double) * 9 * 4096);  // mu, D, alpha; the same packed by entry
  L.h = take(sizeof(double) * 3 * QMAXL);
  L.slots = take(sizeof(unsigned long long) * QS_N);
  L.err = take(sizeof(unsigned));
  L.xch = take(sizeof(unsigned long long) * 64 * nb);
  L.xseq = take(sizeof(unsigned));
  L.rcount = take(sizeof(int) * nb);
  L.snap = take(sizeof(double) * 6 * QC * nb);
  L.rg = take(sizeof(int) * 10 * nb);
  L.need = take(sizeof(unsigned long long) * nb);
  L.fine = take(nb);
  L.rgw = take(QRgScratch::at(nullptr, nb).bytes);
  L.total = p.t;
  return L;
}
}  // namespace

extern "C" int sm_quad_arena_size(const sm_quad *q, size_t *bytes) {
  if (!q || !bytes) return SM_EINVAL;
  *bytes = qlayout(q).total;
  return SM_OK;
}

extern "C" int sm_quad_bind_arena(sm_quad *q, void *dev_ptr, size_t bytes) {
  if (!q || !dev_ptr) return SM_EINVAL;
  const QLayout L = qlayout(q);
  if (bytes < L.total) return qfail(q, SM_ENOMEM, "arena too small");
  if (((uintptr_t)dev_ptr & 255) != 0) return qfail(q, SM_EINVAL, "arena not 256-byte aligned");
  char *a = (char *)dev_ptr;
  drop_graphs(q);
  q->arena = a;
  q->d_lev = (int *)(a + L.lev);
  q->d_par = (int *)(a + L.par);
  q->d_chl = (int *)(a + L.chl);
  q->d_nbr8 = (int *)(a + L.nbr8);
  q->d_pn = (int *)(a + L.pn);
  q->d_ref = (int *)(a + L.ref);
  q->d_ij = (int2 *)(a + L.ij);
  q->d_w = (double *)(a + L.w);
  q->d_wv = (double *)(a + L.wv);
  for (int v = 0; v < NV; ++v) q->var[v] = (double *)(a + L.var[v]);
  q->cflux = (double *)(a + L.cflux);
  q->ainv = (double *)(a + L.ainv);
  q->lut = (double *)(a + L.lut);
  q->d_h = (double *)(a + L.h);
  q->slots = (unsigned long long *)(a + L.slots);
  q->d_err = (unsigned *)(a + L.err);
  q->xch = (unsigned long long *)(a + L.xch);
  q->xseq = (unsigned *)(a + L.xseq);
  q->rcount = (int *)(a + L.rcount);
  q->snap = (double *)(a + L.snap);
  q->d_rg = (int *)(a + L.rg);
  q->d_need = (unsigned long long *)(a + L.need);
  q->d_fine = (unsigned char *)(a + L.fine);
  q->rgw = a + L.rgw;
  std::vector<double> hs(3 * QMAXL);
  for (int l = 0; l < QMAXL; ++l) {
    hs[l] = q->h[l];
    hs[QMAXL + l] = q->inv_h2[l];
    hs[2 * QMAXL + l] = 1.0 / q->h[l];
  }
  if (cudaMemsetAsync(a, 0, L.total, q->stream) != cudaSuccess ||
      cudaMemcpyAsync(q->ainv, q->h_ainv.data(), sizeof(double) * QC * QC, cudaMemcpyHostToDevice, q->stream) !=
          cudaSuccess ||
      cudaMemcpyAsync(q->d_h, hs.data(), sizeof(double) * 3 * QMAXL, cudaMemcpyHostToDevice, q->stream) !=
          cudaSuccess)
    return qfail(q, SM_ECUDA, "arena initialisation");
  return upload_tables(q);
}

extern "C" int sm_quad_refine_level(sm_quad *q, int level, const int8_t *flags, int *n_new, int *n_dropped) {
  SM_RANGE();
  if (!q || !flags) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  if (level != q->nlev - 1 || level >= q->lmax) return qfail(q, SM_ESTATE, "not the finest refinable level");
  std::vector<int> todo;
  int dropped = 0;
  for (int b = q->off[level]; b < q->off[level + 1]; ++b) {
    if (flags[b - q->off[level]] <= 0) continue;
    bool ok = true;
    for (int d = 0; d < 8; ++d) ok &= q->nbr8[8 * b + d] != -2;
    if (ok) todo.push_back(b);
    else ++dropped;
  }
  if ((long long)n_boxes(q) + 4ll * (long long)todo.size() > q->max_boxes)
    return qfail(q, SM_ENOMEM, "box capacity exceeded");
  const int start = n_boxes(q);
  for (int b : todo)
    for (int c = 0; c < 4; ++c) {
      const int nb = n_boxes(q);
      add_box(q, level + 1, 2 * q->ix[b] + (c & 1), 2 * q->iy[b] + (c >> 1), b);
      q->chl[4 * b + c] = nb;
    }
  if (n_new) *n_new = n_boxes(q) - start;
  if (n_dropped) *n_dropped = dropped;
  if (todo.empty()) return SM_OK;
  q->off[level + 2] = n_boxes(q);
  q->nlev = level + 2;
  set_neighbours(q, level + 1);
  drop_graphs(q);
  // the new boxes' fields start at zero
  for (int v = 0; v < NV; ++v)
    if (cudaMemsetAsync(q->var[v] + (size_t)start * QC, 0, sizeof(double) * QC * (size_t)(n_boxes(q) - start),
                        q->stream) != cudaSuccess)
      return qfail(q, SM_ECUDA, "memset");
  return upload_tables(q);
}

extern "C" int sm_quad_get_tables(const sm_quad *q, int *nb, int *nl, int32_t *level_offset, int32_t *level,
                                  int32_t *ij, uint64_t *morton, int32_t *parent, int32_t *child, int32_t *nbr) {
  if (!q) return SM_EINVAL;
  const int n = n_boxes(q);
  if (nb) *nb = n;
  if (nl) *nl = q->nlev;
  if (level_offset)
    for (int l = 0; l <= q->nlev; ++l) level_offset[l] = q->off[l];
  for (int b = 0; b < n; ++b) {
    if (level) level[b] = q->lev[b];
    if (ij) {
      ij[2 * b] = q->ix[b];
      ij[2 * b + 1] = q->iy[b];
    }
    if (morton) morton[b] = q->mort[b];
    if (parent) parent[b] = q->par[b];
    if (child)
      for (int c = 0; c < 4; ++c) child[4 * b + c] = q->chl[4 * b + c];
    if (nbr)
      for (int d = 0; d < 8; ++d) nbr[8 * b + d] = q->nbr8[8 * b + d];
  }
  return SM_OK;
}

extern "C" int sm_quad_var_ptr(sm_quad *q, int v, double **dev) {
  if (!q || !dev || v < 0 || v > V_RHO) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  *dev = q->var[v];
  return SM_OK;
}

extern "C" int sm_quad_upload(sm_quad *q, int v, const double *host) {
  if (!q || !host || v < 0 || v > V_RHO) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  if (cudaMemcpyAsync(q->var[v], host, sizeof(double) * QC * (size_t)n_boxes(q), cudaMemcpyHostToDevice,
                      q->stream) != cudaSuccess ||
      cudaStreamSynchronize(q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "upload");
  return SM_OK;
}

extern "C" int sm_quad_download(sm_quad *q, int v, double *host) {
  if (!q || !host || v < 0 || v > V_RHO) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  unsigned e = 0;
  if (cudaMemcpyAsync(host, q->var[v], sizeof(double) * QC * (size_t)n_boxes(q), cudaMemcpyDeviceToHost,
                      q->stream) != cudaSuccess ||
      cudaMemcpyAsync(&e, q->d_err, sizeof(e), cudaMemcpyDeviceToHost, q->stream) != cudaSuccess ||
      cudaStreamSynchronize(q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "download");
  return wait_error(q, e);
}

extern "C" int sm_quad_set_table(sm_quad *q, int n, double e_max, const double *mu, const double *diff,
                                 const double *alpha) {
  if (!q || !mu || !diff || !alpha || n < 2 || n > 4096 || !(e_max > 0.0)) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  std::vector<double> t(9 * 4096, 0.0);
  std::memcpy(t.data(), mu, sizeof(double) * n);
  std::memcpy(t.data() + n, diff, sizeof(double) * n);
  std::memcpy(t.data() + 2 * n, alpha, sizeof(double) * n);
  sm::table_pack(t.data() + 3 * 4096, n, mu, diff, alpha);
  if (cudaMemcpyAsync(q->lut, t.data(), sizeof(double) * t.size(), cudaMemcpyHostToDevice, q->stream) != cudaSuccess ||
      cudaStreamSynchronize(q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "table upload");
  q->lut_n = n;
  q->lut_emax = e_max;
  return SM_OK;
}

extern "C" int sm_quad_charge_rhs(sm_quad *q, double c, double eps, int use_rho) {
  if (!q || !(eps > 0.0)) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  return charge(q, c, eps, use_rho);
}

extern "C" int sm_quad_fmg(sm_quad *q, double tol, int max_cycles, int *cycles, double *rel) {
  SM_RANGE();
  if (!q || max_cycles < 1 || !(tol >= 0.0)) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  return run_solve(q, true, tol, max_cycles, cycles, rel);
}

extern "C" int sm_quad_solve(sm_quad *q, double tol, int max_cycles, int *cycles, double *rel) {
  SM_RANGE();
  if (!q || max_cycles < 1 || !(tol >= 0.0)) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  return run_solve(q, false, tol, max_cycles, cycles, rel);
}

extern "C" int sm_quad_vcycles(sm_quad *q, int n) {
  SM_RANGE();
  if (!q || n < 0) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  for (int c = 0; c < n; ++c)
    if (int st = vcycle_g(q, q->nlev - 1)) return st;
  return check(q, "V-cycle");
}

extern "C" int sm_quad_leg_wait_selftest(sm_quad *q) {
  if (!q) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  if (!any_leg(q)) return qfail(q, SM_ESTATE, "no level runs in one-launch legs");
  drop_graphs(q);  // captured legs hold their waits' tags
  q->leg_skew = 1u << 30;
  return SM_OK;
}

extern "C" int sm_quad_compute_field(sm_quad *q) {
  SM_RANGE();
  if (!q) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  return field(q);
}

extern "C" int sm_quad_dt_limit(sm_quad *q, double c, double eps, double *dt) {
  SM_RANGE();
  if (!q || !dt || !(eps > 0.0)) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  if (!q->lut_n) return qfail(q, SM_ESTATE, "no coefficient table");
  return dt_limit(q, c, eps, dt);
}

extern "C" int sm_quad_fluid_stage(sm_quad *q, double dt) {
  SM_RANGE();
  if (!q) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  if (!q->lut_n) return qfail(q, SM_ESTATE, "no coefficient table");
  restrict_all(q, V_NE, V_NI);
  if (int st = euler_stage(q, V_NE, V_NI, V_NE1, V_NI1, dt, false, 0.0)) return st;
  const size_t bytes = sizeof(double) * QC * (size_t)n_boxes(q);
  if (cudaMemcpyAsync(q->var[V_NE], q->var[V_NE1], bytes, cudaMemcpyDeviceToDevice, q->stream) != cudaSuccess ||
      cudaMemcpyAsync(q->var[V_NI], q->var[V_NI1], bytes, cudaMemcpyDeviceToDevice, q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "copy");
  return SM_OK;
}

extern "C" int sm_quad_advance(sm_quad *q, double dt, double c, double eps, double tol, int max_cycles,
                               double *dt_next, int *cycles) {
  SM_RANGE();
  if (!q || !(eps > 0.0) || max_cycles < 1) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  if (!q->lut_n) return qfail(q, SM_ESTATE, "no coefficient table");
  const double qie = -c / eps;
  restrict_all(q, V_NE, V_NI);
  // stage 1 into the work densities; stage 2 averages them back in place
  if (int st = euler_stage(q, V_NE, V_NI, V_NE1, V_NI1, dt, true, qie)) return st;
  int c1 = 0, c2 = 0;
  const int st1 = run_solve(q, false, tol, max_cycles, &c1, nullptr);
  if (st1 && st1 != SM_ENOCONV) return st1;
  if (int st = field(q)) return st;
  if (cudaMemsetAsync(q->slots, 0, 3 * sizeof(unsigned long long), q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "memset");
  if (int st = euler_stage(q, V_NE1, V_NI1, V_NE, V_NI, dt, true, qie, V_NE, V_NI)) return st;
  const int st2 = run_solve(q, false, tol, max_cycles, &c2, nullptr);
  if (st2 && st2 != SM_ENOCONV) return st2;
  if (int st = field(q)) return st;
  double dtn = 0.0;
  if (int st = dt_read(q, c, eps, &dtn)) return st;
  if (dt_next) *dt_next = dtn;
  if (cycles) {
    cycles[0] = c1;
    cycles[1] = c2;
  }
  return st1 ? st1 : st2;
}

// Eq. 8 with buffer and derefinement flags (the rules of the 3-D form on
// the quadtree): the per-cell test on the GPU, the buffer (same-level leaf
// neighbours within `buffer` cells, Chebyshev distance) on the host from
// the per-box masks
extern "C" int sm_quad_refine_flags(sm_quad *q, double c0, double c1, double c0_deref, double dx_deref, int buffer,
                                    int8_t *flags) {
  SM_RANGE();
  if (!q || !flags || buffer < 0 || buffer > QN) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  if (!q->lut_n) return qfail(q, SM_ESTATE, "no coefficient table");
  const int n = n_boxes(q);
  const double de = q->lut_emax / (q->lut_n - 1);
  qlaunch(q, k_q_refcrit, blocks_for(n), QT, n, (const double *)q->var[V_EMAG], tabs(q),
          (const double *)(q->lut + 2 * q->lut_n), q->lut_n, de, c1, c0 * c1, c0_deref * c1, dx_deref,
          (const double *)q->d_h, q->d_need, q->d_fine);
  std::vector<unsigned long long> need(n);
  std::vector<unsigned char> fine(n);
  if (cudaMemcpyAsync(need.data(), q->d_need, sizeof(unsigned long long) * n, cudaMemcpyDeviceToHost, q->stream) !=
          cudaSuccess ||
      cudaMemcpyAsync(fine.data(), q->d_fine, n, cudaMemcpyDeviceToHost, q->stream) != cudaSuccess ||
      cudaStreamSynchronize(q->stream) != cudaSuccess)
    return qfail(q, SM_ECUDA, "refinement test");
  // cells of a neighbour in direction (dx, dy) within `buffer` cells of the box
  auto axis_ok = [&](int d, int i) { return d < 0 ? i >= QN - buffer : (d > 0 ? i <= buffer - 1 : true); };
  unsigned long long mask[8];
  for (int dy = -1, k = 0; dy <= 1; ++dy)
    for (int dx = -1; dx <= 1; ++dx) {
      if (!dx && !dy) continue;
      unsigned long long m = 0;
      for (int c = 0; c < QC; ++c)
        if (axis_ok(dx, c % QN) && axis_ok(dy, c / QN)) m |= 1ull << c;
      mask[k++] = m;
    }
  for (int b = 0; b < n; ++b) {
    flags[b] = 0;
    if (q->chl[4 * b] >= 0) continue;
    bool marked = need[b] != 0;
    for (int d = 0; d < 8 && !marked; ++d) {
      const int nb = q->nbr8[8 * b + d];
      if (nb >= 0 && q->chl[4 * nb] < 0 && (need[nb] & mask[d])) marked = true;
    }
    if (marked) {
      if (q->lev[b] < q->lmax) flags[b] = 1;
    } else if (fine[b] && q->lev[b] > q->lbase) {
      flags[b] = -1;
    }
  }
  return SM_OK;
}

// The new box set, its tables and the move descriptors are formed on the
// device (k_qrg_*); the host reads the request counts and per-level list
// sizes once, then the new tables for its own copy of the mesh.
extern "C" int sm_quad_regrid(sm_quad *q, const int8_t *flags, int *n_refined, int *n_derefined, int *n_dropped) {
  SM_RANGE();
  if (!q || !flags) return SM_EINVAL;
  if (!q->arena) return qfail(q, SM_ESTATE, "no arena bound");
  const int n = n_boxes(q), M = q->max_boxes, L0 = q->nlev, T = 256;
  cudaStream_t s = q->stream;
  restrict_all(q, V_NE, V_NI);
  const QRgScratch S = QRgScratch::at(q->rgw, (size_t)M);
  int8_t *const dflags = S.flags;
  int *const refv = S.refv, *const keepv = S.keepv, *const derv = S.derv, *const ref_pos = S.ref_pos;
  int *const keep_pos = S.keep_pos, *const nlev = S.nlev, *const cnt = S.cnt, *const counts = S.counts;
  uint64_t *const ref_keys = S.ref_keys, *const kept_keys = S.kept_keys, *const nkey = S.nkey;
  int2 *const nij = S.nij;
  const int gb = (n + T - 1) / T;
  if (cudaMemcpyAsync(dflags, flags, (size_t)n, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemsetAsync(cnt, 0, 8, s) != cudaSuccess)
    return qfail(q, SM_ECUDA, "regrid flags");
  k_qrg_refine<<<gb, T, 0, s>>>(n, q->d_lev, q->d_chl, q->d_nbr8, dflags, q->lmax, refv, cnt);
  k_qrg_derefine<<<gb, T, 0, s>>>(n, q->d_chl, q->d_par, q->d_nbr8, dflags, refv, derv, cnt);
  k_qrg_keep<<<gb, T, 0, s>>>(n, q->d_par, derv, keepv);
  k_qrg_scan2<<<dim3(1, 2), 1024, 0, s>>>(refv, ref_pos, keepv, keep_pos, n);
  QOffsets off{};
  for (int l = 0; l <= L0; ++l) off.v[l] = q->off[l];
  k_qrg_counts<<<1, 32, 0, s>>>(cnt, keep_pos, ref_pos, off, L0, counts);
  q->launches += 5;
  std::vector<int> hc(3 + 2 * L0 + 1);
  unsigned ev = 0;
  if (int st = check(q, "regrid decisions")) return st;
  if (cudaMemcpyAsync(hc.data(), counts, sizeof(int) * hc.size(), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(&ev, q->d_err, sizeof(ev), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return qfail(q, SM_ECUDA, "regrid counts");
  if (int st = wait_error(q, ev)) return st;  // of V-cycles enqueued before: the mesh is unchanged
  const int *hk = &hc[2], *hr = &hc[3 + L0];
  const int nref = hr[L0], nder = hc[1];
  if (n_refined) *n_refined = nref;
  if (n_derefined) *n_derefined = nder;
  if (n_dropped) *n_dropped = hc[0];
  if (nref == 0 && nder == 0) return SM_OK;
  QRgLevels L{};
  int nlevels = 0, m = 0;
  for (int l = 0; l < QMAXL + 2; ++l) {
    const int kept = l < L0 ? hk[l + 1] - hk[l] : 0;
    const int born = (l >= 1 && l - 1 < L0) ? 4 * (hr[l] - hr[l - 1]) : 0;
    L.kept[l] = l <= L0 ? hk[l] : hk[L0];
    L.ref[l] = l <= L0 ? hr[l] : hr[L0];
    L.nw[l] = m;
    m += kept + born;
    if (kept + born > 0) nlevels = l + 1;
  }
  if (m > M) return qfail(q, SM_ENOMEM, "box capacity exceeded");
  k_qrg_keys<<<gb, T, 0, s>>>(n, q->d_ij, keepv, keep_pos, refv, ref_pos, kept_keys, ref_keys);
  k_qrg_place<<<(4 * n + T - 1) / T, T, 0, s>>>(n, q->d_lev, q->d_ij, q->d_nbr8, keepv, keep_pos, refv, ref_pos,
                                               kept_keys, ref_keys, L, nlev, nij, nkey, q->d_rg);
  q->launches += 2;
  // snapshot of the old fields (the move writes the same arrays)
  const int vars[6] = {V_PHI, V_NE, V_NI, V_RHS, V_EMAG, V_RHO};
  const size_t stride = (size_t)M * QC;
  for (int v = 0; v < 6; ++v)
    if (cudaMemcpyAsync(q->snap + v * stride, q->var[vars[v]], sizeof(double) * QC * (size_t)n,
                        cudaMemcpyDeviceToDevice, s) != cudaSuccess)
      return qfail(q, SM_ECUDA, "regrid snapshot");
  // the new tables in place of the old ones
  if (cudaMemcpyAsync(q->d_lev, nlev, sizeof(int) * m, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(q->d_ij, nij, sizeof(int2) * m, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return qfail(q, SM_ECUDA, "regrid tables");
  const int gm = (m + T - 1) / T, gm8 = (8 * m + T - 1) / T;
  k_qrg_links<<<gm, T, 0, s>>>(m, nlev, nkey, L, nlevels, q->d_par, q->d_chl);
  k_qrg_nbr<<<gm8, T, 0, s>>>(m, nlev, nij, nkey, L, q->d_nbr8);
  k_qrg_derived<<<gm8, T, 0, s>>>(m, q->dom.geometry == SM_AXISYMMETRIC, q->d_par, q->d_chl, q->d_nbr8, q->d_ij,
                                  q->d_pn, q->d_ref, q->d_w, q->d_wv);
  q->launches += 3;
  if (int st = check(q, "regrid tables")) return st;
  drop_graphs(q);
  k_q_regrid_move<<<blocks_for(m), QT, 0, s>>>(m, q->d_rg, q->snap, stride, q->var[V_PHI], q->var[V_NE],
                                               q->var[V_NI], q->var[V_RHS], q->var[V_EMAG], q->var[V_RHO], tabs(q),
                                               q->bc, q->d_err);
  ++q->launches;
  // the host's copy of the new mesh
  std::vector<int2> hij(m);
  q->lev.resize(m);
  q->par.resize(m);
  q->chl.resize(4 * (size_t)m);
  q->nbr8.resize(8 * (size_t)m);
  q->mort.resize(m);
  if (cudaMemcpyAsync(q->lev.data(), q->d_lev, sizeof(int) * m, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(hij.data(), q->d_ij, sizeof(int2) * m, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(q->par.data(), q->d_par, sizeof(int) * m, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(q->chl.data(), q->d_chl, sizeof(int) * 4 * m, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(q->nbr8.data(), q->d_nbr8, sizeof(int) * 8 * m, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(q->mort.data(), nkey, sizeof(uint64_t) * m, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(&ev, q->d_err, sizeof(ev), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return qfail(q, SM_ECUDA, "regrid move");
  q->ix.resize(m);
  q->iy.resize(m);
  for (int b = 0; b < m; ++b) {
    q->ix[b] = hij[b].x;
    q->iy[b] = hij[b].y;
  }
  q->nlev = nlevels;
  for (int l = 0; l <= QMAXL + 1; ++l) q->off[l] = l <= nlevels ? L.nw[l] : m;
  if (ev) return qfail(q, SM_ESTATE, "a coarse box needed by the regrid prolongation is missing");
  return SM_OK;
}

extern "C" int sm_quad_set_graphs(sm_quad *q, int on) {
  if (!q) return SM_EINVAL;
  q->graphs = on != 0;
  return SM_OK;
}

extern "C" int sm_quad_set_pdl(sm_quad *q, int on) {
  if (!q) return SM_EINVAL;
  q->pdl = on != 0;
  drop_graphs(q);
  return SM_OK;
}

extern "C" int sm_quad_launch_count(const sm_quad *q, long long *n) {
  if (!q || !n) return SM_EINVAL;
  *n = q->launches;
  return SM_OK;
}

extern "C" const char *sm_quad_last_error(const sm_quad *q) { return q ? q->err.c_str() : "null context"; }
