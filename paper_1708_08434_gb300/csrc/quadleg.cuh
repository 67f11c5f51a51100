// quadleg.cuh -- one leg of a quadtree level's V-cycle visit in one launch
// (Sec. 2.1.2; included by quad.cu inside its namespace).
//
// A quadtree level holds some hundred 8^2 boxes, so each of its kernels is
// launch and load latency: a V-cycle of 15 levels took 142 launches of 3.2
// us.  Here a leg -- the FAS completion or the prolongation, 2 nu colour
// passes, the residual with restriction -- is one cooperative launch with a
// warp per box: lane (i2, j) keeps the x pair of columns 2 i2, 2 i2 + 1 of
// row j in registers, neighbours inside the box come by shuffles, and face
// cells go to the face neighbours' warps through memory after every pass.
//
// Exchange.  A face cell is two 64-bit words, each half of the value beside
// the 32-bit tag of its publication (one relaxed 16-byte store; each word
// proves itself, so nothing rests on the pair arriving together).  The
// reader polls until both tags are the expected one.  Tags grow with time:
// 128 per V-cycle (one counter, advanced by the level-0 solve between the
// two legs of every level), 64 for the down leg, one per publication.  A
// word is overwritten two publications later by the lane whose own halo came
// from that word's reader, so it cannot be overwritten unread.  All blocks
// of the cooperative launch are resident; a poll gives up after Q_SPIN tries
// (err bit 2, the solve returns SM_ETIMEOUT).
//
// What a warp reads of its neighbours' cells in memory, at the start of a
// down leg, they store only after awaiting words that depend on what was
// read: phi is stored at the very end.  Restricted values go to old and rhs
// of the level below, which the leg of that level starts from (a leaf box
// there starts from phi); nothing in a leg writes the phi of another level.
// The arithmetic is that of the separate kernels, in their order.
//
// Bound: latency of the exchange (700 to 1050 cycles a word) and of the
// FP64 chain of a cell.

enum { QL_TOP = 0, QL_FAS = 1, QL_PROLONG = 2, QL_FMG = 3 };  // how a leg starts

constexpr unsigned Q_ERR_WAIT = 2u;
constexpr int Q_SPIN = 1 << 18;  // polls of one wait (a few tenths of a second)

struct QLeg {
  int lo, nu;
  unsigned leg, skew;  // tag offset of the leg; skew only for testing the bounded wait
  double h2, inv_h2;
  double *phi, *rhs, *old;
  unsigned long long *xch;  // [box][face][8][2]
  const unsigned *seq;
  unsigned *err;
  int lev;
  QTabs T;
  QBc bc;
};

__device__ __forceinline__ void qx_put(unsigned long long *p, double v, unsigned tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"((b & 0xffffffff00000000ull) | tag),
               "l"((b << 32) | tag)
               : "memory");
}
// true when both halves carry the tag
__device__ __forceinline__ bool qx_get(const unsigned long long *p, unsigned tag, double &v) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  v = __longlong_as_double((long long)((a & 0xffffffff00000000ull) | (b >> 32)));
  return (unsigned)a == tag && (unsigned)b == tag;
}

template <int START>
__global__ void __launch_bounds__(32, 28) k_q_leg(const __grid_constant__ QLeg a) {
  constexpr bool UP = START == QL_PROLONG, PRO = START == QL_PROLONG || START == QL_FMG;
  constexpr unsigned ALL = 0xffffffffu;
  __shared__ double sph[32];  // phihat of the refinement faces' cells [face][8]
  const int lane = threadIdx.x, i2 = lane & 3, j = lane >> 2, b = a.lo + blockIdx.x;
  const QTabs &T = a.T;
  const size_t g = (size_t)b * QC + QN * j + 2 * i2;  // the lane's pair

  // one round of loads: tables, the box's own cells, the tag counter
  const int fx = i2 == 0 ? 0 : 1, fy = j == 0 ? 2 : 3;
  const bool atx = i2 == 0 || i2 == 3, aty = j == 0 || j == QN - 1;
  const int nx = atx ? T.nbr8[8 * b + face_dir8(fx)] : -3, ny = aty ? T.nbr8[8 * b + face_dir8(fy)] : -3;
  const int pnl = lane < 9 ? T.pn[9 * b + lane] : 0;  // the parent's neighbourhood, an entry a lane
  const int2 ij = T.ij[b];
  const int ref = T.ref[b];
  const unsigned tag0 = (*a.seq << 7) + a.leg;
  const unsigned stop = *a.err & Q_ERR_WAIT;
  const double *wc = T.w + (size_t)b * 24 + 6 * i2;
  const double wl[2] = {wc[0], wc[3]}, wh[2] = {wc[1], wc[4]}, wi[2] = {wc[2], wc[5]};
  double2 f2 = *reinterpret_cast<const double2 *>(a.rhs + g);
  double2 u2 = make_double2(0.0, 0.0);
  if (START != QL_FMG) u2 = *reinterpret_cast<const double2 *>(a.phi + g);
  const bool refined = START == QL_FAS && (ref & 16);
  if (START == QL_FAS) {
    const double2 o2 = *reinterpret_cast<const double2 *>(a.old + g);
    if (refined) u2 = o2;
    else *reinterpret_cast<double2 *>(a.old + g) = u2;
  }
  if (stop) return;  // a wait of an earlier launch ran out
  double u[2] = {u2.x, u2.y}, f[2] = {f2.x, f2.y};  // by column parity
  const int ncl = QN << (a.lev - 1);
  // entry of the parent's neighbourhood that holds coarse cell (cx, cy)
  auto cbox = [&](int cx, int cy) { return ((cx >> 3) - (ij.x >> 1) + 1) + 3 * ((cy >> 3) - (ij.y >> 1) + 1); };
  // value of the level below at coarse cell (qx, qy), or across the wall from
  // (cx, cy) inside; every lane calls it (the neighbourhood sits across lanes)
  auto coarse = [&](auto val, int qx, int qy, int cx, int cy, bool homog) {
    const bool out = qx < 0 || qy < 0 || qx >= ncl || qy >= ncl;
    const int x = out ? cx : qx, y = out ? cy : qy;
    const int q = __shfl_sync(ALL, pnl, cbox(x, y));
    const bool ok = q >= 0;
    if (!ok) atomicOr(a.err, 1u);  // a coarse box needed here is missing
    const double v = ok ? val((size_t)q * QC + (x & 7) + QN * (y & 7)) : 0.0;
    if (!out) return v;
    const int w = qx < 0 ? 0 : (qx >= ncl ? 1 : (qy < 0 ? 2 : 3));
    return a.bc.type[w] ? (homog ? 0.0 : a.bc.g2[w]) - v : v;
  };

  const bool bx = nx >= 0, by = ny >= 0;
  auto own = [&](int c) { return ((j + c) & 1) ? u[1] : u[0]; };
  // the x face belongs to the cell of colour c: column 0 (p = 0) at -x, column 7 (p = 1) at +x
  auto xact = [&](int c) { return atx && ((j + c) & 1) == fx; };
  unsigned long long *const mx = a.xch + 2 * ((size_t)b * 32 + fx * 8 + j);
  unsigned long long *const my = a.xch + 2 * ((size_t)b * 32 + fy * 8 + 2 * i2);
  const unsigned long long *const qx_ = a.xch + 2 * ((size_t)(bx ? nx : b) * 32 + (fx ^ 1) * 8 + j);
  const unsigned long long *const qy_ = a.xch + 2 * ((size_t)(by ? ny : b) * 32 + (fy ^ 1) * 8 + 2 * i2);
  auto publish = [&](int c, unsigned ev) {
    const double v = own(c);
    if (bx && xact(c)) qx_put(mx, v, tag0 + ev);
    if (by) qx_put(my + 2 * ((j + c) & 1), v, tag0 + ev);
  };
  // halo of the lane's colour-c cell across its x and y faces
  double hx = 0.0, hy = 0.0;
  auto await = [&](int c, unsigned ev) {
    const unsigned tag = tag0 + ev + a.skew;
    const bool x = bx && xact(c);
    if (x || by) {
      for (int it = 0;; ++it) {
        bool ok = true;
        if (x) ok = qx_get(qx_, tag, hx);
        if (by) ok = qx_get(qy_ + 2 * ((j + c) & 1), tag, hy) && ok;
        if (ok) break;
        if (it > Q_SPIN) {
          atomicOr(a.err, Q_ERR_WAIT);
          break;
        }
      }
    }
  };
  // the four neighbours of the lane's colour-c cell: shuffles inside the box,
  // halos x and y from other boxes, ghosts at walls and refinement faces
  auto around = [&](int c, double x, double y, double &L, double &R, double &S, double &N) {
    const int p = (j + c) & 1;
    const double me = own(c), oth = own(c ^ 1);
    double xs = __shfl_sync(ALL, oth, p ? lane + 1 : lane - 1);
    S = __shfl_sync(ALL, oth, lane - 4);
    N = __shfl_sync(ALL, oth, lane + 4);
    auto ghost = [&](int nb, int face, int at) {
      if (nb == -1) return a.bc.type[face] ? a.bc.g2[face] - me : me;
      return me * (1.0 / 3.0) + sph[8 * face + at] * (2.0 / 3.0);
    };
    if (xact(c)) xs = bx ? x : ghost(nx, fx, j);
    if (aty) {
      const double v = by ? y : ghost(ny, fy, 2 * i2 + p);
      if (j == 0) S = v;
      else N = v;
    }
    L = p ? oth : xs;
    R = p ? xs : oth;
  };
  auto lap = [&](int c, double L, double R, double S, double N) {
    const int p = (j + c) & 1;
    const double v = own(c);
    return ((p ? wl[1] : wl[0]) * (L - v) + (p ? wh[1] : wh[0]) * (R - v) + (S - v) + (N - v)) * a.inv_h2;
  };
  auto set = [&](double (&d)[2], int c, double v) {
    if ((j + c) & 1) d[1] = v;
    else d[0] = v;
  };

  if (PRO) {
    // (2c + c_x + c_y)/4: one coarse cell under the pair, its x neighbour for
    // each column, the y neighbour for both
    const int cx = 4 * ij.x + i2, cy = (QN * ij.y + j) >> 1, qy = cy + ((j & 1) ? 1 : -1);
    auto cv = [&](int x, int y) {
      const double p = coarse([&](size_t k) { return a.phi[k]; }, x, y, cx, cy, UP);
      return UP ? p - coarse([&](size_t k) { return a.old[k]; }, x, y, cx, cy, true) : p;
    };
    const double c0 = 2.0 * cv(cx, cy), cl = cv(cx - 1, cy), cr = cv(cx + 1, cy), cq = cv(cx, qy);
    const double s0 = c0 + cl + cq, s1 = c0 + cr + cq;
    u[0] = UP ? u[0] + 0.25 * s0 : 0.25 * s0;
    u[1] = UP ? u[1] + 0.25 * s1 : 0.25 * s1;
    publish(1, 0);
  }
  {
    // phihat of the refinement faces: lane -> (face, cell)
    const int face = lane >> 3, at = lane & 7;
    const int nb = T.nbr8[8 * b + face_dir8(face)];
    if (__any_sync(ALL, nb == -2)) {
      int gi, gj;
      face_cell(face, -1, at, gi, gj);
      const int Gx = ij.x * QN + gi, Gy = ij.y * QN + gj;
      // lanes of other faces read the cell under the box (any existing one)
      const bool cf = nb == -2;
      const int cx = cf ? Gx >> 1 : 4 * ij.x, cy = cf ? Gy >> 1 : 4 * ij.y;
      int qx = cx, qy = cy;
      if (cf && face < 2) qy += (Gy & 1) ? 1 : -1;
      else if (cf) qx += (Gx & 1) ? 1 : -1;
      auto val = [&](size_t k) { return a.phi[k]; };
      const double c = coarse(val, cx, cy, cx, cy, false);
      const double ct = coarse(val, qx, qy, cx, cy, false);
      sph[lane] = 0.75 * c + 0.25 * ct;
      __syncwarp();
    }
  }
  unsigned ev = 0;
  if (!PRO) {
    // halos from the neighbours' cells (FAS start: restricted values of a
    // refined neighbour are in old, a leaf's in phi)
    auto of = [&](int face) { return START == QL_FAS && ((ref >> face) & 1) ? a.old : a.phi; };
    double x = 0.0, y[2] = {0.0, 0.0};
    if (bx) x = of(fx)[(size_t)nx * QC + QN * j + (fx ? 0 : QN - 1)];
    if (by) {
      const double2 v = *reinterpret_cast<const double2 *>(of(fy) + (size_t)ny * QC + QN * (fy == 2 ? QN - 1 : 0) + 2 * i2);
      y[0] = v.x;
      y[1] = v.y;
    }
    double L, R, S, N;
    around(0, x, (j & 1) ? y[1] : y[0], L, R, S, N);
    if (refined) {
      double L1, R1, S1_, N1;
      around(1, x, (j & 1) ? y[0] : y[1], L1, R1, S1_, N1);
      const double l0 = lap(0, L, R, S, N), l1 = lap(1, L1, R1, S1_, N1);
      const bool odd = j & 1;  // colour 0 is the odd column
      f[0] += odd ? l1 : l0;
      f[1] += odd ? l0 : l1;
      *reinterpret_cast<double2 *>(a.rhs + g) = make_double2(f[0], f[1]);
    }
    const int p = j & 1;
    set(u, 0, ((p ? wl[1] : wl[0]) * L + (p ? wh[1] : wh[0]) * R + S + N - a.h2 * (p ? f[1] : f[0])) * (p ? wi[1] : wi[0]));
    publish(0, ++ev);
  }
  double x1 = 0.0, y1 = 0.0;  // colour 1's halo in the last pass
  for (int sweep = 0; sweep < a.nu; ++sweep) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (!PRO && c == 0 && sweep == 0) continue;
      await(c, ev);
      if (!UP && c == 1) {
        x1 = hx;
        y1 = hy;
      }
      double L, R, S, N;
      around(c, hx, hy, L, R, S, N);
      const int p = (j + c) & 1;
      set(u, c, ((p ? wl[1] : wl[0]) * L + (p ? wh[1] : wh[0]) * R + S + N - a.h2 * (p ? f[1] : f[0])) * (p ? wi[1] : wi[0]));
      ++ev;
      if (!UP || c == 0 || sweep + 1 < a.nu) publish(c, ev);
    }
  }
  if (!UP) {
    await(0, ev);  // the neighbours' last colour-1 cells
    double L, R, S, N;
    around(0, hx, hy, L, R, S, N);
    const double l0 = lap(0, L, R, S, N);
    around(1, x1, y1, L, R, S, N);
    const double l1 = lap(1, L, R, S, N);
    const bool odd = j & 1;
    const double r[2] = {f[0] - (odd ? l1 : l0), f[1] - (odd ? l0 : l1)};
    // volume-weighted means over the 2 x 2 children: the even row's lane sums
    // the potential, the odd row's the residual
    const double w0 = T.wv[(size_t)b * QN + 2 * i2], w1 = T.wv[(size_t)b * QN + 2 * i2 + 1];
    const double t0 = __shfl_xor_sync(ALL, odd ? u[0] : r[0], 4), t1 = __shfl_xor_sync(ALL, odd ? u[1] : r[1], 4);
    const double a0 = odd ? t0 : u[0], a1 = odd ? t1 : u[1], b0 = odd ? r[0] : t0, b1 = odd ? r[1] : t1;
    double sum = 0.0, ws = 0.0;
    sum += w0 * a0;
    ws += w0;
    sum += w1 * a1;
    ws += w1;
    sum += w0 * b0;
    ws += w0;
    sum += w1 * b1;
    ws += w1;
    const int P = __shfl_sync(ALL, pnl, 4);
    (odd ? a.rhs : a.old)[(size_t)P * QC + 4 * (ij.x & 1) + i2 + QN * (4 * (ij.y & 1) + (j >> 1))] = sum / ws;
  }
  *reinterpret_cast<double2 *>(a.phi + g) = make_double2(u[0], u[1]);
}
