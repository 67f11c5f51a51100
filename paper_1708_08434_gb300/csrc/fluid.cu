// fluid.cu -- field and drift-diffusion-reaction step (Sec. 2.2-2.4):
// cell |E| from the potential, Eq. 5 right-hand side, Koren-limited upwind
// advective flux (Eq. 6-7) plus central diffusive flux with coefficients
// from a lookup table, refinement-boundary ghosts and flux averaging,
// forward-Euler stages combined into the explicit trapezoidal (Heun) step,
// and the time-step limits reduced by block/atomic maxima.
#include <math.h>
#include <string.h>

#include "fluid_dev.cuh"
#include "sm_internal.cuh"
#include "sm_nvtx.h"

using namespace sm;

int sm_mg_solve_internal(sm_ctx *ctx, double tol, int max_cycles, int *cycles);

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------

// Density ghost (depth t = 1 or 2) across refinement face f of fine box b
// at face cell (u,w): linear prolongation (c + c_sx + c_sy + c_sz)/4 of the
// coarse cell c that contains the ghost, limited to 2c (Sec. 2.3).
__device__ double density_cf_ghost(const double *__restrict__ n, const int32_t *__restrict__ nbr6,
                                   const int32_t *__restrict__ parent, const int32_t *__restrict__ ijk, int b,
                                   int f, int t, int u, int w, unsigned long long *err) {
  int a = f >> 1, t1 = (a + 1) % 3, t2 = (a + 2) % 3;
  int G[3];
  G[a] = NC * ijk[3 * b + a] + ((f & 1) ? NC - 1 + t : -t);
  G[t1] = NC * ijk[3 * b + t1] + u;
  G[t2] = NC * ijk[3 * b + t2] + w;
  int P = parent[b];
  int Q = nbr6[6 * P + f];
  if (Q < 0) {
    atomicOr(err, 4ull);
    return 0.0;
  }
  int lc[3];
  for (int d = 0; d < 3; ++d) lc[d] = (G[d] >> 1) - NC * ijk[3 * Q + d];
  double c = n[(size_t)Q * CELLS + cidx(lc[0], lc[1], lc[2])];
  double sum = c;
  for (int d = 0; d < 3; ++d) {
    int s = (G[d] & 1) ? 1 : -1;
    int q[3] = {lc[0], lc[1], lc[2]};
    q[d] += s;
    double v;
    if (q[d] >= 0 && q[d] < NC) {
      v = n[(size_t)Q * CELLS + cidx(q[0], q[1], q[2])];
    } else {
      int Qn = nbr6[6 * Q + 2 * d + (s > 0)];
      if (Qn >= 0) {
        q[d] = s > 0 ? 0 : NC - 1;
        v = n[(size_t)Qn * CELLS + cidx(q[0], q[1], q[2])];
      } else {
        if (Qn == -2) atomicOr(err, 8ull);
        v = c;  // Neumann wall: mirror of c
      }
    }
    sum += v;
  }
  double g = 0.25 * sum;
  return g > 2.0 * c ? 2.0 * c : g;
}

// |E| ghost at a refinement face: the coarse cell containing the ghost
__device__ double emag_cf_ghost(const double *__restrict__ em, const int32_t *__restrict__ nbr6,
                                const int32_t *__restrict__ parent, const int32_t *__restrict__ ijk, int b, int f,
                                int u, int w) {
  int a = f >> 1, t1 = (a + 1) % 3, t2 = (a + 2) % 3;
  int G[3];
  G[a] = NC * ijk[3 * b + a] + ((f & 1) ? NC : -1);
  G[t1] = NC * ijk[3 * b + t1] + u;
  G[t2] = NC * ijk[3 * b + t2] + w;
  int Q = nbr6[6 * parent[b] + f];
  if (Q < 0) return 0.0;
  int lc[3];
  for (int d = 0; d < 3; ++d) lc[d] = (G[d] >> 1) - NC * ijk[3 * Q + d];
  return em[(size_t)Q * CELLS + cidx(lc[0], lc[1], lc[2])];
}

// local cell (i,j,k) of face f at depth dep (0 = next to the face)
__device__ __forceinline__ void face_loc(int f, int dep, int u, int w, int c[3]) {
  int a = f >> 1;
  c[a] = (f & 1) ? NC - 1 - dep : dep;
  c[(a + 1) % 3] = u;
  c[(a + 2) % 3] = w;
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------

// |E| on leaf cells: cell component = mean of the two face fields
// (phi_{i-1} - phi_i)/dx and (phi_i - phi_{i+1})/dx
__global__ void __launch_bounds__(512) k_field(const int32_t *__restrict__ leaf, const int32_t *__restrict__ level,
                                               const double *__restrict__ phi, const double *__restrict__ gh,
                                               const int32_t *__restrict__ nbr6, Bc bc, LevelH lh,
                                               double *__restrict__ emag) {
  int b = leaf[blockIdx.x];
  int t = threadIdx.x;
  int c[3] = {t & 7, (t >> 3) & 7, t >> 6};
  double ih = lh.inv_h[level[b]];
  const double *p = phi + (size_t)b * CELLS;
  double pc = p[t];
  const int stride[3] = {1, NC, FACE};
  double d[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double pm = c[a] > 0 ? p[t - stride[a]] : pot_ghost(phi, nbr6, gh, b, 2 * a, c[0], c[1], c[2], pc, bc, 0);
    double pp = c[a] < NC - 1 ? p[t + stride[a]]
                              : pot_ghost(phi, nbr6, gh, b, 2 * a + 1, c[0], c[1], c[2], pc, bc, 0);
    d[a] = pm - pp;
  }
  // |E| = |(p_-d - p_+d)| / (2 dx) summed in quadrature: each component is
  // the mean of (p_-d - p_c)/dx and (p_c - p_+d)/dx
  emag[(size_t)b * CELLS + t] = sqrt_newton(fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0]))) * (0.5 * ih);
}

// Eq. 5 right-hand side on leaf cells
__global__ void __launch_bounds__(512) k_charge(const int32_t *__restrict__ leaf, const double *__restrict__ ne,
                                                const double *__restrict__ ni, const double *__restrict__ rho,
                                                double q, double inv_eps, int use_rho, double *__restrict__ rhs) {
  size_t x = (size_t)leaf[blockIdx.x] * CELLS + threadIdx.x;
  rhs[x] = use_rho ? -rho[x] * inv_eps : -q * (ni[x] - ne[x]) * inv_eps;
}

// Per-cell time-step quantities at the table index of the cell's |E| (x: half
// of it): sum_d |mu E_d| 2 dx with E_d = (p_{-d} - p_{+d})/(2 dx) (the mean of
// the two face fields), that plus 12 D (both to be scaled by 1/(2 dx^2)), and
// mu n_e
__device__ __forceinline__ void dt_terms(const double *__restrict__ phi, const double *__restrict__ gh,
                                         const int32_t *__restrict__ nbr6, const Bc &bc, int b, int t,
                                         unsigned long long x, double ne, const Table &tb, double &adv, double &ad,
                                         double &drt) {
  int c[3] = {t & 7, (t >> 3) & 7, t >> 6};
  const double *p = phi + (size_t)b * CELLS;
  double pc = p[t];
  const int stride[3] = {1, NC, FACE};
  double w;
  const double2 *fc = tb.fc + 2 * index_split(x, x, tb, w);
  const double2 cm = __ldg(fc), cd = __ldg(fc + 1);
  const double mu = fma(w, cm.y, cm.x);
  double d[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double pm = c[a] > 0 ? p[t - stride[a]] : pot_ghost(phi, nbr6, gh, b, 2 * a, c[0], c[1], c[2], pc, bc, 0);
    double pp = c[a] < NC - 1 ? p[t + stride[a]]
                              : pot_ghost(phi, nbr6, gh, b, 2 * a + 1, c[0], c[1], c[2], pc, bc, 0);
    d[a] = dabs(pm - pp);
  }
  adv = dabs(mu) * ((d[0] + d[1]) + d[2]);
  ad = fma(12.0, fma(w, cd.y, cd.x), adv);
  drt = mu * ne;
}

// block maxima of three non-negative quantities (negative values and NaNs
// count as 0) into slots[0..2], compared as bit patterns on the integer pipe, the
// first two times scale (rounding is monotonic: the maximum of the products
// is the product of the maximum); red: 3 * (blockDim.x / 32) words of shared
// memory
__device__ __forceinline__ void block_max3_to(unsigned long long *slots, double a, double b, double c,
                                              long long *red, double scale) {
  long long v[3] = {size_bits(a), size_bits(b), size_bits(c)};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = max(v[i], __shfl_xor_sync(0xffffffffu, v[i], o));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < 3; ++i) red[3 * wid + i] = v[i];
  __syncthreads();
  if (threadIdx.x < 3) {
    long long m = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, red[3 * w + threadIdx.x]);
    if (threadIdx.x < 2) m = max(dbits(__longlong_as_double(m) * scale), 0ll);
    atomicMax(slots + threadIdx.x, (unsigned long long)m);
  }
}

__global__ void __launch_bounds__(512) k_dt(const int32_t *__restrict__ leaf, const int32_t *__restrict__ level,
                                            const double *__restrict__ phi, const double *__restrict__ gh,
                                            const double *__restrict__ emag, const double *__restrict__ ne,
                                            const int32_t *__restrict__ nbr6, Bc bc, LevelH lh, Table tb,
                                            unsigned long long *slots) {
  __shared__ long long red[48];
  int b = leaf[blockIdx.x];
  int t = threadIdx.x;
  size_t x = (size_t)b * CELLS + t;
  double adv, ad, drt;
  dt_terms(phi, gh, nbr6, bc, b, t, half_index(emag[x], tb), ne[x], tb, adv, ad, drt);
  block_max3_to(slots + SC_ADV, adv, ad, drt, red, 0.5 * lh.inv_h2[level[b]]);
}

// Fine-side fluxes through the refinement faces of leaf boxes: 64 threads, a
// face cell each, per box of the list of leaves that have such a face and
// axis (only the face on the octant's side of an axis can be one; a block
// per box that walked its six faces took 26 us on streamer6); read by the
// box itself and averaged by its coarse neighbour, so both sides use the same
// numbers.
__global__ void __launch_bounds__(64) k_cf_flux(const int32_t *__restrict__ leaf, const int32_t *__restrict__ level,
                                                const double *__restrict__ n, const double *__restrict__ phi,
                                                const double *__restrict__ gh, const double *__restrict__ emag,
                                                const int32_t *__restrict__ nbr6,
                                                const int32_t *__restrict__ parent,
                                                const int32_t *__restrict__ ijk, LevelH lh, Table tb,
                                                double *__restrict__ cflux, unsigned long long *err) {
  const int b = leaf[blockIdx.x], a = blockIdx.y, f = 2 * a + (ijk[3 * b + a] & 1);
  if (__ldg(nbr6 + 6 * b + f) != -2) return;
  const int u = threadIdx.x & 7, w = threadIdx.x >> 3;
  const size_t base = (size_t)b * CELLS;
  int c0[3], c1[3];
  face_loc(f, 0, u, w, c0);
  face_loc(f, 1, u, w, c1);
  const double n0 = n[base + cidx(c0[0], c0[1], c0[2])], n1 = n[base + cidx(c1[0], c1[1], c1[2])];
  const double g1 = density_cf_ghost(n, nbr6, parent, ijk, b, f, 1, u, w, err);
  const double g2 = density_cf_ghost(n, nbr6, parent, ijk, b, f, 2, u, w, err);
  const double p0 = phi[base + cidx(c0[0], c0[1], c0[2])];
  const double pg = p0 * (1.0 / 3.0) + (2.0 / 3.0) * gh[(size_t)(6 * b + f) * FACE + fcell(a, c0[0], c0[1], c0[2])];
  const unsigned long long x0 = half_index(emag[base + cidx(c0[0], c0[1], c0[2])], tb),
                           xg = half_index(emag_cf_ghost(emag, nbr6, parent, ijk, b, f, u, w), tb);
  const double F = (f & 1) ? face_flux_d(n0, g1, n0 - n1, g1 - n0, g2 - g1, p0 - pg, x0, xg, tb)
                           : face_flux_d(g1, n0, g1 - g2, n0 - g1, n1 - n0, pg - p0, xg, x0, tb);
  cflux[(size_t)(6 * b + f) * FACE + u + NC * w] = F * lh.inv_h[level[b]];
}

// index in a staged box of pitch P (O ghost layers) of the cell with
// coordinate ca along axis a and u, w along axes (a+1)%3, (a+2)%3 (no
// arrays indexed at run time: those would live in local memory)
template <int P, int O>
__device__ __forceinline__ int lin_axis(int a, int ca, int u, int w) {
  const int x = a == 0 ? ca : (a == 1 ? w : u);
  const int y = a == 0 ? u : (a == 1 ? ca : w);
  const int z = a == 0 ? w : (a == 1 ? u : ca);
  return (x + O) + P * ((y + O) + P * (z + O));
}

// Shared memory of the update kernel.  Row and plane pitches make 16 lanes
// on consecutive y (or x) of two consecutive z hit 16 different 8-byte banks.
constexpr int UT = 192;                  // threads: one line of faces each (3 axes x 64)
constexpr int NY = 13, NZ = 168;         // density with 2 ghost layers on faces
constexpr int PY = 11, PZ = 120;         // potential and half index with 1 ghost layer
constexpr int DY = 9, DZ = 72, DA = 576; // flux differences [axis][cell], over the density
struct UpdSmem {
  double n[12 * NZ];
  double p[10 * PZ];
  unsigned long long x[10 * PZ];
  long long red[3 * (UT / 32)];
};
static_assert(3 * DA <= 12 * NZ, "the flux differences fit the density's place");
__device__ __forceinline__ int iN(int x, int y, int z) { return (x + 2) + NY * (y + 2) + NZ * (z + 2); }
__device__ __forceinline__ int iP(int x, int y, int z) { return (x + 1) + PY * (y + 1) + PZ * (z + 1); }

// One forward-Euler stage on a leaf box: dst = src + dt F(src), with
// F = -div(flux) + alpha mu |E| n_e for electrons and the same source for
// ions.  HEUN: dst = (n0 + src + dt F(src))/2, and the time-step maxima of
// src.  Also writes the Eq. 5 right-hand side from dst.
//
// Bound by the FP64 pipe (2 instructions per clock and SM), so the work is
// laid out to issue few of them: a thread marches one line of 9 faces along
// an axis and forms each density difference once (three faces use it), table
// indices and halvings are integer operations, and dt / dx^2 is one factor.  52.7
// FP64 instructions per cell in stage 1 (the cell-and-face form before: 64).
template <bool HEUN>
__global__ void __launch_bounds__(UT, 5) k_update(
    const int32_t *__restrict__ leaf, const int32_t *__restrict__ level, const double *__restrict__ ne_src,
    const double *__restrict__ ni_src, const double *__restrict__ ne0, const double *__restrict__ ni0,
    double *__restrict__ ne_dst, double *__restrict__ ni_dst, const double *__restrict__ phi,
    const double *__restrict__ gh, const double *__restrict__ emag, const double *__restrict__ cflux,
    const int32_t *__restrict__ nbr6, const int32_t *__restrict__ child, const int32_t *__restrict__ parent,
    const int32_t *__restrict__ ijk, Bc bc, LevelH lh, Table tb, double dt, double qie, double *__restrict__ rhs,
    unsigned long long *slots) {
  extern __shared__ __align__(16) unsigned char smraw[];
  UpdSmem &S = *reinterpret_cast<UpdSmem *>(smraw);
  const int b = leaf[blockIdx.x], t = threadIdx.x, l = level[b];
  const double ih2 = lh.inv_h2[l];
  const size_t base = (size_t)b * CELLS;
  // x pairs of cells: pair t, and t + 192 for the first 64 threads
  double2 nc[2], ec[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int pi = t + UT * s;
    if (pi >= CELLS / 2) continue;
    const int x = 2 * (pi & 3), y = (pi >> 2) & 7, z = pi >> 5;
    nc[s] = reinterpret_cast<const double2 *>(ne_src + base)[pi];
    ec[s] = reinterpret_cast<const double2 *>(emag + base)[pi];
    const double2 pc = reinterpret_cast<const double2 *>(phi + base)[pi];
    const int q = iP(x, y, z);
    S.n[iN(x, y, z)] = nc[s].x;
    S.n[iN(x + 1, y, z)] = nc[s].y;
    S.p[q] = pc.x;
    S.p[q + 1] = pc.y;
    S.x[q] = half_index(ec[s].x, tb);
    S.x[q + 1] = half_index(ec[s].y, tb);
  }
  // fluxes known before the faces are walked: this thread's line meets the
  // box's low and high face, whose flux at a refinement face is the fine
  // side's (k_cf_flux), on the coarse side the mean of the four fine ones
  const int a = t >> 6, c0 = t & 7, c1 = (t >> 3) & 7;
  const int fu = a == 1 ? c1 : c0, fw = a == 1 ? c0 : c1;  // the line's face coordinates
  double Fk[2] = {0.0, 0.0};
  bool known[2] = {false, false};
#pragma unroll
  for (int hi = 0; hi < 2; ++hi) {
    const int f = 2 * a + hi, nb = nbr6[6 * b + f];
    if (nb == -2) {
      Fk[hi] = cflux[(size_t)(6 * b + f) * FACE + fu + NC * fw] * lh.h[l];
      known[hi] = true;
    } else if (nb >= 0 && child[8 * nb] >= 0) {
      const int ch = child[8 * nb + lin_axis<2, 0>(a, hi ? 0 : 1, fu >> 2, fw >> 2)];
      const double *cf = cflux + (size_t)(6 * ch + (f ^ 1)) * FACE;
      const int uf = 2 * (fu & 3), wf = 2 * (fw & 3);
      double s = 0.0;
      s += cf[uf + NC * wf];
      s += cf[uf + 1 + NC * wf];
      s += cf[uf + NC * (wf + 1)];
      s += cf[uf + 1 + NC * (wf + 1)];
      Fk[hi] = (s * 0.25) * lh.h[l];
      known[hi] = true;
    }
  }
  __syncthreads();
  // face halos: 6 x 64 face cells, two per thread
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int it = t + UT * s, f = it >> 6, ha = f >> 1, hi = f & 1;
    const int x8 = it & 7, y8 = (it >> 3) & 7;
    const int u = ha == 1 ? y8 : x8, w = ha == 1 ? x8 : y8;
    const int nb = nbr6[6 * b + f];
    // depths 0, 1 inside the face and the ghosts -1, -2 along the face axis
    const int d0 = hi ? NC - 1 : 0, sg = hi ? 1 : -1;
    const int X = ha == 0 ? d0 : x8, Y = ha == 0 ? x8 : (ha == 1 ? d0 : y8), Z = ha == 2 ? d0 : y8;
    const int qn = iN(X, Y, Z), sn = sg * (ha == 0 ? 1 : (ha == 1 ? NY : NZ));
    const int qp = iP(X, Y, Z), sp = sg * (ha == 0 ? 1 : (ha == 1 ? PY : PZ));
    double vg1, vg2, pg;
    unsigned long long xg;
    if (nb >= 0) {
      // the neighbour's cells at depths 0 and 1 of its opposite face
      const int m0 = lin_axis<8, 0>(ha, hi ? 0 : NC - 1, u, w), m1 = lin_axis<8, 0>(ha, hi ? 1 : NC - 2, u, w);
      const size_t nbase = (size_t)nb * CELLS;
      vg1 = ne_src[nbase + m0];
      vg2 = ne_src[nbase + m1];
      pg = phi[nbase + m0];
      xg = child[8 * nb] < 0 ? half_index(emag[nbase + m0], tb) : 0ull;
    } else if (nb == -1) {
      vg1 = S.n[qn];
      vg2 = S.n[qn - sn];
      pg = bc.type[f] ? 2.0 * bc.val[f] - S.p[qp] : S.p[qp];
      xg = S.x[qp];
    } else {
      vg1 = density_cf_ghost(ne_src, nbr6, parent, ijk, b, f, 1, u, w, slots + SC_ERR);
      vg2 = density_cf_ghost(ne_src, nbr6, parent, ijk, b, f, 2, u, w, slots + SC_ERR);
      pg = S.p[qp] * (1.0 / 3.0) + (2.0 / 3.0) * gh[(size_t)(6 * b + f) * FACE + u + NC * w];
      xg = half_index(emag_cf_ghost(emag, nbr6, parent, ijk, b, f, u, w), tb);
    }
    S.n[qn + sn] = vg1;
    S.n[qn + 2 * sn] = vg2;
    S.p[qp + sp] = pg;
    S.x[qp + sp] = xg;
  }
  __syncthreads();
  // the line's 9 faces: face m between cells m - 1 and m
  double D[NC];
  {
    const int X = a == 0 ? 0 : c0, Y = a == 0 ? c0 : (a == 1 ? 0 : c1), Z = a == 2 ? 0 : c1;
    const int sn = a == 0 ? 1 : (a == 1 ? NY : NZ), sp = a == 0 ? 1 : (a == 1 ? PY : PZ);
    const double *n = S.n + iN(X, Y, Z), *p = S.p + iP(X, Y, Z);
    const unsigned long long *xi = S.x + iP(X, Y, Z);
    double nL = n[-sn], nR = n[0], dm = nL - n[-2 * sn], dn = nR - nL, pL = p[-sp], F0 = 0.0;
    unsigned long long xL = xi[-sp];
#pragma unroll
    for (int m = 0; m <= NC; ++m) {
      const double n2 = n[(m + 1) * sn], dq = n2 - nR, pR = p[m * sp];
      const unsigned long long xR = xi[m * sp];
      double F;
      if (m == 0 && known[0]) F = Fk[0];
      else if (m == NC && known[1]) F = Fk[1];
      else F = face_flux_d(nL, nR, dm, dn, dq, pL - pR, xL, xR, tb);
      if (m > 0) D[m - 1] = F - F0;
      F0 = F;
      nL = nR;
      nR = n2;
      dm = dn;
      dn = dq;
      pL = pR;
      xL = xR;
    }
    __syncthreads();  // the density is no longer read: its place takes the differences
    double *d = S.n + DA * a + X + DY * Y + DZ * Z;
    const int sd = a == 0 ? 1 : (a == 1 ? DY : DZ);
#pragma unroll
    for (int m = 0; m < NC; ++m) d[m * sd] = D[m];
  }
  __syncthreads();
  const double dth = -dt * ih2;
  long long m_adv = 0, m_ad = 0, m_drt = 0;  // maxima of bit patterns, as block_max3_to compares them
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int pi = t + UT * s;
    if (pi >= CELLS / 2) continue;
    const int x0 = 2 * (pi & 3), y = (pi >> 2) & 7, z = pi >> 5;
    const double2 ni = reinterpret_cast<const double2 *>(ni_src + base)[pi];
    double2 e0, i0;
    if (HEUN) {
      e0 = reinterpret_cast<const double2 *>(ne0 + base)[pi];
      i0 = reinterpret_cast<const double2 *>(ni0 + base)[pi];
    }
    double ne_new[2], ni_new[2], f[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const double *d = S.n + (x0 + c) + DY * y + DZ * z;
      const double div = (d[0] + d[DA]) + d[2 * DA];  // dx^2 times the divergence
      const double nes = c ? nc[s].y : nc[s].x, e = c ? ec[s].y : ec[s].x, nis = c ? ni.y : ni.x;
      const int q = iP(x0 + c, y, z);
      double w;
      const int i = index_split(S.x[q], S.x[q], tb, w);
      const double2 cm = __ldg(tb.fc + 2 * i), al = __ldg(tb.al + i);
      const double mu = fma(w, cm.y, cm.x);
      const double src = fma(w, al.y, al.x) * mu * e * nes;
      ne_new[c] = fma(dth, div, fma(dt, src, nes));
      ni_new[c] = fma(dt, src, nis);
      if (HEUN) {
        ne_new[c] = halve((c ? e0.y : e0.x) + ne_new[c]);
        ni_new[c] = halve((c ? i0.y : i0.x) + ni_new[c]);
        // sum_d mu |E_d| 2 dx, that plus 12 D (both times 1/(2 dx^2) below), mu n_e
        const double gx = dabs(S.p[q - 1] - S.p[q + 1]), gy = dabs(S.p[q - PY] - S.p[q + PY]),
                     gz = dabs(S.p[q - PZ] - S.p[q + PZ]);
        const double adv = dabs(mu) * ((gx + gy) + gz);
        const double2 cd = __ldg(tb.fc + 2 * i + 1);
        const double ad = fma(12.0, fma(w, cd.y, cd.x), adv), drt = mu * nes;
        m_adv = max(m_adv, size_bits(adv));
        m_ad = max(m_ad, size_bits(ad));
        m_drt = max(m_drt, size_bits(drt));
      }
      f[c] = (ni_new[c] - ne_new[c]) * qie;
    }
    reinterpret_cast<double2 *>(ne_dst + base)[pi] = make_double2(ne_new[0], ne_new[1]);
    reinterpret_cast<double2 *>(ni_dst + base)[pi] = make_double2(ni_new[0], ni_new[1]);
    reinterpret_cast<double2 *>(rhs + base)[pi] = make_double2(f[0], f[1]);
  }
  if (HEUN)
    block_max3_to(slots + SC_ADV, __longlong_as_double(m_adv), __longlong_as_double(m_ad),
                  __longlong_as_double(m_drt), S.red, 0.5 * ih2);
}

// ---------------------------------------------------------------------------
// host drivers
// ---------------------------------------------------------------------------
static Table table_of(const sm_ctx *ctx) {
  Table tb = {};
  table_index_consts(tb, ctx->tab + 6 * 4096, ctx->tab_n, ctx->tab_emax);
  return tb;
}

static int ready(sm_ctx *ctx) {
  if (!ctx) return SM_EINVAL;
  if (!ctx->arena || ctx->n_levels == 0) return sm_fail(ctx, SM_ESTATE, "octree not built");
  return SM_OK;
}

extern "C" int sm_compute_field(sm_ctx *ctx) {
  SM_RANGE();
  int st = ready(ctx);
  if (st) return st;
  if ((st = sm_fill_all_cf(ctx, ctx->phi))) return st;
  k_field<<<ctx->n_leaves, 512, 0, ctx->stream>>>(ctx->leaf, ctx->level, ctx->phi, ctx->gh, ctx->nbr6, ctx->bc,
                                                  ctx->lh, ctx->emag);
  ++ctx->n_launch;
  SM_CKL("field");
  return SM_OK;
}

extern "C" int sm_charge_rhs(sm_ctx *ctx, double q, double eps, int use_rho) {
  int st = ready(ctx);
  if (st) return st;
  if (!(eps != 0.0)) return SM_EINVAL;
  k_charge<<<ctx->n_leaves, 512, 0, ctx->stream>>>(ctx->leaf, ctx->nbuf[ctx->ncur], ctx->ibuf[ctx->ncur], ctx->rho,
                                                   q, 1.0 / eps, use_rho, ctx->rhs);
  ++ctx->n_launch;
  SM_CKL("charge");
  return SM_OK;
}

extern "C" int sm_restrict_densities(sm_ctx *ctx) {
  int st = ready(ctx);
  if (st) return st;
  return sm_restrict_pair(ctx, ctx->nbuf[ctx->ncur], ctx->ibuf[ctx->ncur]);
}

// dt from time-step maxima already copied to host scalars hs (SC_N words)
static int dt_of(sm_ctx *ctx, const double *hs, double q, double eps, double *dt) {
  unsigned long long e;
  memcpy(&e, &hs[SC_ERR], sizeof e);
  if (e) return sm_fail(ctx, SM_ESTATE, "device consistency check failed (flags 0x%llx)", e);
  double m_adv = hs[SC_ADV], m_ad = hs[SC_AD], m_drt = hs[SC_DRT];
  double d = 1e300;
  if (m_adv > 0.0 && 0.5 / m_adv < d) d = 0.5 / m_adv;
  if (m_ad > 0.0 && 1.0 / m_ad < d) d = 1.0 / m_ad;
  if (m_drt > 0.0 && eps / (q * m_drt) < d) d = eps / (q * m_drt);
  *dt = 0.9 * d;
  return SM_OK;
}

static int dt_from_slots(sm_ctx *ctx, double q, double eps, double *dt) {
  SM_CK(cudaMemcpyAsync(ctx->hscal, ctx->dscal, sizeof(double) * SC_N, cudaMemcpyDeviceToHost, ctx->stream));
  SM_CK(cudaStreamSynchronize(ctx->stream));
  return dt_of(ctx, ctx->hscal, q, eps, dt);
}

extern "C" int sm_dt_limit(sm_ctx *ctx, double q, double eps, double *dt) {
  SM_RANGE();
  int st = ready(ctx);
  if (st) return st;
  if (!dt || ctx->tab_n < 2) return sm_fail(ctx, SM_ESTATE, "no coefficient table");
  if ((st = sm_fill_all_cf(ctx, ctx->phi))) return st;
  SM_CK(cudaMemsetAsync(ctx->dscal + SC_ADV, 0, 3 * sizeof(unsigned long long), ctx->stream));
  k_dt<<<ctx->n_leaves, 512, 0, ctx->stream>>>(ctx->leaf, ctx->level, ctx->phi, ctx->gh, ctx->emag,
                                               ctx->nbuf[ctx->ncur], ctx->nbr6, ctx->bc, ctx->lh, table_of(ctx),
                                               ctx->dscal);
  ++ctx->n_launch;
  SM_CKL("dt");
  return dt_from_slots(ctx, q, eps, dt);
}

// one stage from buffer s into buffer d; with h0 >= 0 averaged with buffer h0
// (second Heun stage), leaving the time-step maxima of s
static int stage(sm_ctx *ctx, int s, int d, int h0, double dt, double q, double eps) {
  int st;
  Table tb = table_of(ctx);
  if ((st = sm_fill_all_cf(ctx, ctx->phi))) return st;
  if (ctx->n_cf_leaves > 0) {
    k_cf_flux<<<dim3(ctx->n_cf_leaves, 3), 64, 0, ctx->stream>>>(ctx->cf_leaf, ctx->level, ctx->nbuf[s], ctx->phi,
                                                         ctx->gh, ctx->emag, ctx->nbr6, ctx->parent, ctx->ijk,
                                                         ctx->lh, tb, ctx->cflux, ctx->dscal + SC_ERR);
    ++ctx->n_launch;
    SM_CKL("cf_flux");
  }
  const size_t smem = sizeof(UpdSmem);
  // rhs = -q (n_i - n_e) / eps of the new densities; with h0 the Heun average
  auto run = [&](auto kernel) {
    kernel<<<ctx->n_leaves, UT, smem, ctx->stream>>>(
        ctx->leaf, ctx->level, ctx->nbuf[s], ctx->ibuf[s], h0 >= 0 ? ctx->nbuf[h0] : nullptr,
        h0 >= 0 ? ctx->ibuf[h0] : nullptr, ctx->nbuf[d], ctx->ibuf[d], ctx->phi, ctx->gh, ctx->emag, ctx->cflux,
        ctx->nbr6, ctx->child, ctx->parent, ctx->ijk, ctx->bc, ctx->lh, tb, dt, -q * (1.0 / eps), ctx->rhs,
        ctx->dscal);
  };
  if (h0 >= 0) run(k_update<true>);
  else run(k_update<false>);
  ++ctx->n_launch;
  SM_CKL("update");
  return sm_restrict_pair(ctx, ctx->nbuf[d], ctx->ibuf[d]);
}

extern "C" int sm_fluid_stage(sm_ctx *ctx, double dt) {
  SM_RANGE();
  int st = ready(ctx);
  if (st) return st;
  if (ctx->tab_n < 2) return sm_fail(ctx, SM_ESTATE, "no coefficient table");
  int a = ctx->ncur, b = (a + 1) % 3;
  if ((st = sm_restrict_pair(ctx, ctx->nbuf[a], ctx->ibuf[a]))) return st;
  // q/eps only feed the right-hand side written alongside; a stage alone
  // uses SI values
  if ((st = stage(ctx, a, b, -1, dt, 1.602176634e-19, 8.8541878128e-12))) return st;
  ctx->ncur = b;
  return SM_OK;
}

extern "C" int sm_advance_fluid_coeffs(sm_ctx *ctx, double dt, const sm_fluid_coeffs *c, double *dt_next,
                                       int *cycles) {
  if (!c) return SM_EINVAL;
  return sm_advance_fluid(ctx, dt, c->q, c->eps, c->tol, c->max_cycles, dt_next, cycles);
}

extern "C" int sm_advance_fluid(sm_ctx *ctx, double dt, double q, double eps, double tol, int max_cycles,
                                double *dt_next, int *cycles) {
  SM_RANGE();
  int st = ready(ctx);
  if (st) return st;
  if (ctx->tab_n < 2) return sm_fail(ctx, SM_ESTATE, "no coefficient table");
  if (!(eps != 0.0) || max_cycles < 1) return SM_EINVAL;
  int A = ctx->ncur, B = (A + 1) % 3, C = (A + 2) % 3;
  if ((st = sm_restrict_pair(ctx, ctx->nbuf[A], ctx->ibuf[A]))) return st;
  // stage 1: n1 = n0 + dt F(n0); new field
  if ((st = stage(ctx, A, B, -1, dt, q, eps))) return st;
  int c1 = 0, c2 = 0, st1, st2;
  if (ctx->pre_solve && (st = ctx->pre_solve(ctx->hook_obj, ctx))) return st;
  st1 = sm_mg_solve(ctx, tol, max_cycles, &c1, nullptr);
  if (st1 && st1 != SM_ENOCONV) return st1;
  if (ctx->post_solve && (st = ctx->post_solve(ctx->hook_obj, ctx))) return st;
  if ((st = sm_compute_field(ctx))) return st;
  // stage 2: n = (n0 + n1 + dt F(n1))/2 with the time-step limits at n1
  SM_CK(cudaMemsetAsync(ctx->dscal + SC_ADV, 0, 3 * sizeof(unsigned long long), ctx->stream));
  if ((st = stage(ctx, B, C, A, dt, q, eps))) return st;
  ctx->ncur = C;
  // the maxima go to the staged host copy without a wait: the solve below
  // synchronises before they are read
  double *staged = ctx->hscal + SC_N;
  SM_CK(cudaMemcpyAsync(staged, ctx->dscal, sizeof(double) * SC_N, cudaMemcpyDeviceToHost, ctx->stream));
  if (ctx->pre_solve && (st = ctx->pre_solve(ctx->hook_obj, ctx))) return st;
  st2 = sm_mg_solve(ctx, tol, max_cycles, &c2, nullptr);
  if (st2 && st2 != SM_ENOCONV) return st2;
  if (ctx->post_solve && (st = ctx->post_solve(ctx->hook_obj, ctx))) return st;
  if ((st = sm_compute_field(ctx))) return st;
  SM_CK(cudaStreamSynchronize(ctx->stream));
  double dtn = 0.0;
  if ((st = dt_of(ctx, staged, q, eps, &dtn))) return st;
  if (dt_next) *dt_next = dtn;
  if (cycles) {
    cycles[0] = c1;
    cycles[1] = c2;
  }
  if (st1 || st2) return sm_fail(ctx, SM_ENOCONV, "a Poisson solve did not reach tol %.3e", tol);
  return SM_OK;
}
