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
// (Q_ERR_WAIT): later legs return at once, and the solve runs again with a
// launch per operation.
//
// What a warp reads of its neighbours' cells in memory, at the start of a
// down leg, they store only after awaiting words that depend on what was
// read: phi is stored at the very end.  Restricted values go to old and rhs
// of the level below, which the leg of that level starts from (a leaf box
// there starts from phi); nothing in a leg writes the phi of another level.
//
// Bound: the exchange (700 to 1050 cycles a word) and the FP64 pipe, which
// takes 16 cycles for a warp's instruction: with four warps on an SM each
// waits some 64 cycles per FP64 instruction.  So instructions are counted.
// w_lo + w_hi is 2 in both geometries, so the Gauss-Seidel division is a
// quarter, done on the exponent; an update is four FP64 instructions before
// the halo is awaited and two after it.

enum { QL_TOP = 0, QL_FAS = 1, QL_PROLONG = 2, QL_FMG = 3 };  // how a leg starts

constexpr unsigned Q_ERR_WAIT = 2u;
constexpr int Q_SPIN = 1 << 18;  // pairs of polls of one wait (0.11 s)

struct QLeg {
  int lo, nu;
  unsigned leg, skew;  // tag offset of the leg; skew != 0 only in the self-test
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
struct QWord {
  unsigned long long a, b;
  __device__ __forceinline__ void load(const unsigned long long *p) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  }
  // 0 when both halves carry the tag
  __device__ __forceinline__ unsigned off(unsigned tag) const { return ((unsigned)a ^ tag) | ((unsigned)b ^ tag); }
  __device__ __forceinline__ double value() const {
    return __longlong_as_double((long long)((a & 0xffffffff00000000ull) | (b >> 32)));
  }
};

// OCC: blocks an SM has to hold (more registers for a level of few boxes)
template <int START, int OCC>
__global__ void __launch_bounds__(32, OCC) k_q_leg(const __grid_constant__ QLeg a) {
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
  const int nbl = T.nbr8[8 * b + face_dir8(lane >> 3)];  // neighbour across the face of lane / 8
  const int2 ij = T.ij[b];
  const int ref = T.ref[b];
  double wv[2] = {1.0, 1.0};
  if (!UP) {
    wv[0] = T.wv[(size_t)b * QN + 2 * i2];
    wv[1] = T.wv[(size_t)b * QN + 2 * i2 + 1];
  }
  const unsigned tag0 = (*a.seq << 7) + a.leg;
  const unsigned stop = *a.err & Q_ERR_WAIT;
  const double *wc = T.w + (size_t)b * 24 + 6 * i2;
  const double wl[2] = {wc[0], wc[3]}, wh[2] = {wc[1], wc[4]};
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
  // Halo of the lane's colour-c cell across its x and y faces (0 where there
  // is none).  Two polls are kept in flight: the first is issued before the
  // arithmetic that needs no halo, so that its trip to memory is not added to
  // it.
  double hx = 0.0, hy = 0.0;
  struct Poll {
    QWord x, y;
  };
  auto poll = [&](int c, Poll &q) {
    if (bx && xact(c)) q.x.load(qx_);
    if (by) q.y.load(qy_ + 2 * ((j + c) & 1));
  };
  auto await = [&](int c, unsigned ev, Poll &q) {
    const unsigned tag = tag0 + ev + a.skew;
    const bool x = bx && xact(c);
    auto off = [&](const Poll &w) { return (x ? w.x.off(tag) : 0u) | (by ? w.y.off(tag) : 0u); };
    if (x || by) {
      Poll w = q;
      for (int it = 0;; ++it) {
        poll(c, w);
        if (off(q) == 0u) break;
        poll(c, q);
        if (off(w) == 0u) {
          q = w;
          break;
        }
        if (it > Q_SPIN) {
          atomicOr(a.err, Q_ERR_WAIT);
          break;
        }
      }
    }
    hx = x ? q.x.value() : 0.0;
    hy = by ? q.y.value() : 0.0;
  };
  // The four neighbours of the lane's colour-c cell: the pair's other column,
  // the next column beyond the pair, and the rows below and above, by
  // shuffles; 0 where that leaves the box.
  struct Around {
    double me, oth, xs, S, N;
  };
  auto around = [&](int c) {
    Around r;
    r.me = own(c);
    r.oth = own(c ^ 1);
    r.xs = __shfl_sync(ALL, r.oth, ((j + c) & 1) ? lane + 1 : lane - 1);
    r.S = __shfl_sync(ALL, r.oth, lane - 4);
    r.N = __shfl_sync(ALL, r.oth, lane + 4);
    if (xact(c)) r.xs = 0.0;
    if (j == 0) r.S = 0.0;
    if (j == QN - 1) r.N = 0.0;
    return r;
  };
  // A ghost at a wall or refinement face is A + B own (Dirichlet 2g - own,
  // Neumann own, 2/3 phihat + own / 3): of the x face's cell and of the y
  // face's two (by column); no ghost: zeros
  double gxA = 0.0, gxB = 0.0, gyA[2] = {0.0, 0.0}, gyB = 0.0;
  const bool anyg = __any_sync(ALL, nx == -1 || nx == -2 || ny == -1 || ny == -2);
  auto ghosts = [&] {
    if (nx == -1) {
      gxA = a.bc.type[fx] ? a.bc.g2[fx] : 0.0;
      gxB = a.bc.type[fx] ? -1.0 : 1.0;
    } else if (nx == -2) {
      gxA = sph[8 * fx + j];
      gxB = 1.0 / 3.0;
    }
    if (ny == -1) {
      gyA[0] = gyA[1] = a.bc.type[fy] ? a.bc.g2[fy] : 0.0;
      gyB = a.bc.type[fy] ? -1.0 : 1.0;
    } else if (ny == -2) {
      gyA[0] = sph[8 * fy + 2 * i2];
      gyA[1] = sph[8 * fy + 2 * i2 + 1];
      gyB = 1.0 / 3.0;
    }
  };
  // four times the red-black update of colour c: uA - uB own + w oth + w' xs
  // + S + N + w' hx + hy, ghosts folded into uA and uB
  double uA[2], uB[2] = {0.0, 0.0};
  auto w_in = [&](int c) { return ((j + c) & 1) ? wl[1] : wh[0]; };  // the pair's other column
  auto w_out = [&](int c) { return ((j + c) & 1) ? wh[1] : wl[0]; };  // the column beyond
  auto update_form = [&](int c) {
    const int p = (j + c) & 1;
    uA[c] = -a.h2 * (p ? f[1] : f[0]);
    if (anyg) {
      const double w = xact(c) ? w_out(c) : 0.0;
      uA[c] += fma(w, gxA, p ? gyA[1] : gyA[0]);
      uB[c] = fma(w, gxB, gyB);
    }
  };
  auto update0 = [&](int c, const Around &r) {
    double t = fma(w_in(c), r.oth, uA[c]);
    if (anyg) t = fma(uB[c], r.me, t);
    return fma(w_out(c), r.xs, t) + (r.S + r.N);
  };
  auto update1 = [&](int c, double base) {
    const double t = fma(w_out(c), hx, base + hy);  // hx, hy are 0 where there is no halo
    // a quarter on the exponent (zeros, small and non-finite values multiply)
    const long long b = __double_as_longlong(t);
    const int ex = (int)((unsigned long long)b >> 52) & 0x7ff;
    return ex > 2 && ex < 0x7ff ? __longlong_as_double(b - (2ll << 52)) : 0.25 * t;
  };
  // h^2 L phi at the lane's colour-c cell from its neighbours with the halo x,
  // y; differences first, which keeps the rounding at that of the differences
  auto lap = [&](int c, const Around &r, double x, double y) {
    const int p = (j + c) & 1;
    double X = bx ? x : 0.0, Y = by ? y : 0.0;
    if (anyg) {
      X = bx ? X : fma(gxB, r.me, gxA);
      Y = by ? Y : fma(gyB, r.me, p ? gyA[1] : gyA[0]);
    }
    const double xs = xact(c) ? X : r.xs, S = j == 0 ? Y : r.S, N = j == QN - 1 ? Y : r.N;
    return fma(w_in(c), r.oth - r.me, fma(w_out(c), xs - r.me, (S - r.me) + (N - r.me)));
  };
  auto set = [&](double (&d)[2], int c, double v) {
    if ((j + c) & 1) d[1] = v;
    else d[0] = v;
  };

  if (PRO) {
    // (2c + c_x + c_y)/4: one coarse cell under the pair, its x neighbour for
    // each column, the y neighbour for both
    const int cx = 4 * ij.x + i2, cy = (QN * ij.y + j) >> 1, qy = cy + ((j & 1) ? 1 : -1);
    const int px[4] = {cx, cx - 1, cx + 1, cx}, py[4] = {cy, cy, cy, qy};
    double cv[4], ov[4] = {0.0, 0.0, 0.0, 0.0};
    bool out[4], missing = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // every load before any use
      out[k] = px[k] < 0 || py[k] < 0 || px[k] >= ncl || py[k] >= ncl;
      const int x = out[k] ? cx : px[k], y = out[k] ? cy : py[k];
      const int q = __shfl_sync(ALL, pnl, cbox(x, y));
      missing |= q < 0;
      const size_t at = (size_t)(q < 0 ? 0 : q) * QC + (x & 7) + QN * (y & 7);
      cv[k] = a.phi[at];
      if (UP) ov[k] = a.old[at];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (UP) cv[k] -= ov[k];
      if (out[k]) {
        const int w = px[k] < 0 ? 0 : (px[k] >= ncl ? 1 : (py[k] < 0 ? 2 : 3));
        cv[k] = a.bc.type[w] ? (UP ? 0.0 : a.bc.g2[w]) - cv[k] : cv[k];
      }
    }
    if (missing) atomicOr(a.err, 1u);  // a coarse box needed here is missing
    const double t = fma(2.0, cv[0], cv[3]);
    u[0] = UP ? fma(0.25, t + cv[1], u[0]) : 0.25 * (t + cv[1]);
    u[1] = UP ? fma(0.25, t + cv[2], u[1]) : 0.25 * (t + cv[2]);
    publish(1, 0);
  }
  {
    // 2/3 phihat of the refinement faces: lane -> (face, cell)
    const int face = lane >> 3, at = lane & 7;
    const bool cf = nbl == -2;
    if (__any_sync(ALL, cf)) {
      int gi, gj;
      face_cell(face, -1, at, gi, gj);
      const int Gx = ij.x * QN + gi, Gy = ij.y * QN + gj;
      // lanes of other faces read a cell under the box
      const int cx = cf ? Gx >> 1 : 4 * ij.x, cy = cf ? Gy >> 1 : 4 * ij.y;
      int qx = cx, qy = cy;
      if (cf && face < 2) qy += (Gy & 1) ? 1 : -1;
      else if (cf) qx += (Gx & 1) ? 1 : -1;
      const bool out = qx < 0 || qy < 0 || qx >= ncl || qy >= ncl;
      const int x = out ? cx : qx, y = out ? cy : qy;
      const int b0 = __shfl_sync(ALL, pnl, cbox(cx, cy)), b1 = __shfl_sync(ALL, pnl, cbox(x, y));
      if (b0 < 0 || b1 < 0) atomicOr(a.err, 1u);
      const double c = a.phi[(size_t)(b0 < 0 ? 0 : b0) * QC + (cx & 7) + QN * (cy & 7)];
      double ct = a.phi[(size_t)(b1 < 0 ? 0 : b1) * QC + (x & 7) + QN * (y & 7)];
      if (out) {
        const int w = qx < 0 ? 0 : (qx >= ncl ? 1 : (qy < 0 ? 2 : 3));
        ct = a.bc.type[w] ? a.bc.g2[w] - ct : ct;
      }
      sph[lane] = fma(1.0 / 6.0, ct, 0.5 * c);
      __syncwarp();
    }
  }
  ghosts();
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
    const bool odd = j & 1;  // colour 0 is the odd column of odd rows
    const Around r0 = around(0);
    if (refined) {  // the FAS right-hand side f += L phi
      const Around r1 = around(1);
      const double t0 = lap(0, r0, x, odd ? y[1] : y[0]), t1 = lap(1, r1, x, odd ? y[0] : y[1]);
      f[0] = fma(odd ? t1 : t0, a.inv_h2, f[0]);
      f[1] = fma(odd ? t0 : t1, a.inv_h2, f[1]);
    }
    hx = xact(0) ? x : 0.0;
    hy = odd ? y[1] : y[0];
    update_form(0);
    set(u, 0, update1(0, update0(0, r0)));
    publish(0, ++ev);
    update_form(1);
    if (refined) *reinterpret_cast<double2 *>(a.rhs + g) = make_double2(f[0], f[1]);
  } else {
    update_form(0);
    update_form(1);
  }
  // weights of the restriction's means
  double w0 = 0.0, w1 = 0.0;
  if (!UP) {
    const double r = 0.5 * sm::recip(wv[0] + wv[1]);
    w0 = wv[0] * r;
    w1 = wv[1] * r;
  }
  double x1 = 0.0, y1 = 0.0;  // colour 1's halo in the last pass
  for (int sweep = 0; sweep < a.nu; ++sweep) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (!PRO && c == 0 && sweep == 0) continue;
      Poll q = {};
      const Around r = around(c);
      poll(c, q);
      const double base = update0(c, r);
      await(c, ev, q);
      if (!UP && c == 1) {
        x1 = hx;
        y1 = hy;
      }
      set(u, c, update1(c, base));
      ++ev;
      if (!UP || c == 0 || sweep + 1 < a.nu) publish(c, ev);
    }
  }
  if (!UP) {
    Poll q = {};
    poll(0, q);
    const Around n1 = around(1), n0 = around(0);
    const bool odd = j & 1;
    const double r1 = fma(-lap(1, n1, x1, y1), a.inv_h2, odd ? f[0] : f[1]);  // colour 1: the even column of odd rows
    const int P = __shfl_sync(ALL, pnl, 4);
    await(0, ev, q);  // the neighbours' last colour-1 cells
    const double r0 = fma(-lap(0, n0, hx, hy), a.inv_h2, odd ? f[1] : f[0]);
    const double r[2] = {odd ? r1 : r0, odd ? r0 : r1};
    // volume-weighted means over the 2 x 2 children: the even row's lane forms
    // the potential's, the odd row's the residual's
    const double t0 = __shfl_xor_sync(ALL, odd ? u[0] : r[0], 4), t2 = __shfl_xor_sync(ALL, odd ? u[1] : r[1], 4);
    const double m = fma(w0, t0 + (odd ? r[0] : u[0]), w1 * (t2 + (odd ? r[1] : u[1])));
    (odd ? a.rhs : a.old)[(size_t)P * QC + 4 * (ij.x & 1) + i2 + QN * (4 * (ij.y & 1) + (j >> 1))] = m;
  }
  *reinterpret_cast<double2 *>(a.phi + g) = make_double2(u[0], u[1]);
}
