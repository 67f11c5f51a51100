// mglevel.cuh -- one leg of a small level's V-cycle visit in one launch
// (Sec. 2.1.2; fixed point, included by multigrid.cu after mgfix.cuh).
//
// On a level whose boxes all fit on the GPU at once (one block per box) the
// separate kernels of a leg -- 2 nu colour passes, the FAS completion or
// the prolongation before them, the residual with restriction after them --
// each cost a launch, a chain of table and cell loads and a write-back of
// values the next launch reads again: 2.5 us a colour pass at 900 boxes,
// ten launches a level and V-cycle.  Here a block keeps its box in registers
// (thread (r, h): the four cells i = 4h .. 4h + 3 of x row r) and in shared
// memory (both colours, for the y and z neighbours) from the start of the
// leg to its end, and after every pass hands only the face cells it changed
// to the face neighbours' blocks.  V(2,2) on streamer6 (9 levels of 8 to 928
// boxes): 276 -> 173 us; on a uniform 64^3 grid 75 -> 50 us.
//
// What bounds it: latency.  A word stored by one SM is seen by a polling SM
// 700 cycles later (1050 across the two dies; measured ping-pong); a pass
// takes 1100 (8 boxes) to 1500 cycles (6 boxes an SM), the rest being the
// dependent integer chain of a cell.  64 threads a box (a whole row each)
// measured 193 us, ghosts formed by their own rows' threads 185 us.
//
// Exchange.  A box owns one 64-bit word per face cell (6 faces x 2 colours
// x 32).  A word is value * 256 + tag: stored values are below 2^55 quanta,
// so the low byte is free, and one relaxed 64-bit store carries the value
// together with the proof that it is the awaited one -- no fence, no flag,
// no second trip to L2.  The reader polls the word until its tag is the
// expected one.  The tag counts: 32 per down/up pair of legs of the level
// (xseq[l], advanced by the level-0 solve, which runs between the two legs
// of every level), 16 for the down leg, one per publication (at most 15).
// Every word with a reader is rewritten at every second publication of
// every leg, so what it holds before is always a neighbouring tag, never
// the same byte one round of 256 ago.  A word is overwritten two
// publications later by a thread whose own halo came from the reader of
// that very word, so it cannot be overwritten unread.
//
// The launch is cooperative: all blocks are resident, so every awaited
// block runs.  A poll gives up after WAIT_SPIN tries (ERR_WAIT); the launch's
// other waits run to their own limits, later launches of the solve return at
// once, and the solve runs again with a launch per operation.
//
// What a block reads of its neighbours' cells in memory, at the start of a
// down leg, they overwrite only after awaiting words whose values depend on
// what was read: phx is stored at the very end, after the last wait.  A
// lower level's down leg starts from the restricted values, which are in
// oldx for refined boxes; a leaf box starts from phx and leaves the copy the
// correction is measured against in its own oldx, which nobody reads in
// this launch.  An up leg reads only the level below.  A leg that starts
// with the prolonged FMG solution reads phx of the level below and restricts
// into oldx alone (set_phx 0): a refinement face may read coarse cells that
// the children of a box across an edge restrict into.  The integer sums
// are those of the separate kernels: the same bits.
#pragma once

namespace fx {

enum { FS_TOP = 0, FS_FAS = 1, FS_PROLONG = 2, FS_FMG = 3 };  // how a leg starts

constexpr int WAIT_SPIN = 1 << 18;             // polls of one wait (0.06 s)
constexpr int LEG_MAX_NU = 7;                  // 2 nu + 1 publications fit the tag's 16

struct LevArgs {
  int lo, nu;            // first box, sweeps
  int set_phx;           // down leg: restricted values also go to phx (else to oldx alone)
  unsigned leg, skew;    // tag offset of the leg; skew != 0 only in the self-tests
  long long *phx, *gx, *oldx, *ghx, *xch;  // xch: words of box lo
  const int32_t *rows;  // k_leg_rows
  const unsigned *seq;  // xseq of the level
  unsigned long long *sc;
  Bc bc;
};

__device__ __forceinline__ void xst(long long *p, long long v, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"((v << 8) | (long long)tag) : "memory");
}
__device__ __forceinline__ void xst2(long long *p, long long v0, long long v1, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"((v0 << 8) | (long long)tag),
               "l"((v1 << 8) | (long long)tag)
               : "memory");
}
__device__ __forceinline__ long long xld(const long long *p) {
  long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void xld2(const long long *p, long long &v0, long long &v1) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v0), "=l"(v1) : "l"(p) : "memory");
}

// Ghat = 2c + c_t1 + c_t2 of ghost cell (u, w) of the refinement face of
// axis A of a box in octant oct of its parent (as fx_cf_value).  Only the
// three faces on the octant's side can be refinement faces; the coarse cells
// are in the parent's neighbour Q across the face, and where a tangential
// step leaves Q, in the parent's edge neighbour.
template <int A>
__device__ __forceinline__ long long leg_ghat(const long long *phx, const Bc &bc, const int (&pn)[3],
                                              const int (&pe)[3], int oct, int u, int w, const long long *swall,
                                              unsigned long long *err) {
  constexpr int T1 = (A + 1) % 3, T2 = (A + 2) % 3;
  const int e = ((oct >> A) & 1) ? 0 : NC - 1;
  const int o1 = (oct >> T1) & 1, o2 = (oct >> T2) & 1, l1 = 4 * o1 + (u >> 1), l2 = 4 * o2 + (w >> 1);
  auto cell = [&](int c1, int c2) {  // coordinates along T1 and T2
    return A == 0 ? xpos(e, c1, c2) : (A == 1 ? xpos(c2, e, c1) : xpos(c1, c2, e));
  };
  const int n1 = l1 + ((u & 1) ? 1 : -1), n2 = l2 + ((w & 1) ? 1 : -1);
  const int Q = pn[A], Q1 = (n1 & ~7) ? pe[T2] : Q, Q2 = (n2 & ~7) ? pe[T1] : Q;
  if (Q < 0 || Q1 == -2 || Q2 == -2) {  // nesting violated: no coarse box where one must be
    atomicOr(err, 2ull);
    return 0;
  }
  const long long c = phx[(size_t)Q * CELLS + cell(l1, l2)];
  const long long c1 = phx[(size_t)(Q1 >= 0 ? Q1 : Q) * CELLS + cell(Q1 >= 0 ? n1 & 7 : l1, l2)];
  const long long c2 = phx[(size_t)(Q2 >= 0 ? Q2 : Q) * CELLS + cell(l1, Q2 >= 0 ? n2 & 7 : l2)];
  const long long w1 = Q1 == -1 && bc.type[2 * T1 + o1] ? swall[2 * T1 + o1] - c1 : c1;
  const long long w2 = Q2 == -1 && bc.type[2 * T2 + o2] ? swall[2 * T2 + o2] - c2 : c2;
  return 2 * c + w1 + w2;
}

template <int START>
__global__ void __launch_bounds__(128, 8) k_flevel(const __grid_constant__ LevArgs a) {
  constexpr int CFS = 0x3f << 16, GHOSTS = 0x3f << 10 | CFS;  // any refinement face; any wall or refinement face
  constexpr bool UP = START == FS_PROLONG, PRO = START == FS_PROLONG || START == FS_FMG;
  __shared__ longlong2 sv[2][65][2];       // [colour][row][half]; row 64 stays 0
  __shared__ long long sg[3][FACE];        // Ghat of the outward faces that are refinement faces
  __shared__ longlong2 sgh[2][3][16];      // [colour][axis] ghosts of the outward face, in word order
  __shared__ long long sp[PRO ? 216 : 1];  // coarse values under the box
  __shared__ long long swall[6];           // 2g of a Dirichlet face
  const int t = threadIdx.x, r = t >> 1, h = t & 1, j = r & 7, k = r >> 3, par = (j + k) & 1;
  const int b = a.lo + blockIdx.x;
  unsigned long long *sc = a.sc;
  const size_t base = (size_t)b * CELLS + 4 * r + 2 * h;  // the half row's entries in colour 0 (+ 256: colour 1)

  // one round of loads: the box's row, its own cells, the scale, the tags
  const int32_t *row = a.rows + (size_t)LROW * b;
  // the faces the half row touches: x face h, a y and a z face on the box's
  // sides (neighbour -3: not at such a face)
  const int fy = j == 0 ? 2 : 3, fz = k == 0 ? 4 : 5;
  const int nx = __ldg(row + LR_NB + h);
  const int ny = (j == 0 || j == NC - 1) ? __ldg(row + LR_NB + fy) : -3;
  const int nz = (k == 0 || k == NC - 1) ? __ldg(row + LR_NB + fz) : -3;
  const int P = __ldg(row + LR_P), flags = __ldg(row + LR_FLAGS);
  const bool refined = START == FS_FAS && (flags & 8);
  const unsigned long long stop = sc[SC_ERR] & ERR_WAIT;  // a wait of an earlier launch ran out
  const unsigned tag0 = (*a.seq << 5) + a.leg;
  int pn[3] = {0, 0, 0}, pe[3] = {0, 0, 0};
  if (PRO) {
#pragma unroll
    for (int A = 0; A < 3; ++A) {
      pn[A] = __ldg(row + LR_PN + A);
      pe[A] = __ldg(row + LR_PE + A);
    }
  }
  long long v[2][2], G[2][2];  // [colour][e]: cells i = 2 (2h + e) + ((colour + j + k) & 1); G holds 6 G later
  half_ld(a.gx + base, G[0]);
  half_ld(a.gx + base + 256, G[1]);
  if (START != FS_FMG) {
    half_ld(a.phx + base, v[0]);
    half_ld(a.phx + base + 256, v[1]);
  }
  if (START == FS_FAS) {
    long long w0[2], w1[2];
    half_ld(a.oldx + base, w0);
    half_ld(a.oldx + base + 256, w1);
    if (refined) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        v[0][e] = w0[e];
        v[1][e] = w1[e];
      }
    }
  }
  if (t < 6) swall[t] = a.bc.type[t] ? fx_2g(sc, t) : 0;
  if (t < 4) sv[t >> 1][64][t & 1] = make_longlong2(0, 0);
  // (another block of this launch may set the bit between the reads of two
  // warps: the part of a block that stays then works on what the other part
  // has not staged.  Barriers count the warps that are left, waits end by
  // themselves, and the launch's results are void)
  if (stop) return;

  const int cf = (h + par) & 1, oct = flags & 7;  // cf: colour of the row's cell at x face h
  const bool bx = nx >= 0, by = ny >= 0, bz = nz >= 0;  // a box across the face
  // halo of colour c's cells: hx across the x face (when cf == c), hy, hz
  // across the y and z faces; 0 where no box is
  long long hx = 0, hy[2] = {0, 0}, hz[2] = {0, 0};
  // from the neighbours' cells in memory (FAS start: of a refined box in
  // oldx, of a leaf in phx)
  auto load_halo = [&](int c, long long &x, long long (&y)[2], long long (&z)[2]) {
    const int o = (c ^ 1) << 8;
    auto of = [&](int f) { return START == FS_FAS && ((flags >> (4 + f)) & 1) ? a.oldx : a.phx; };
    if (bx && cf == c) x = of(h)[(size_t)nx * CELLS + o + 4 * r + (h ? 0 : 3)];
    if (by) half_ld(of(fy) + (size_t)ny * CELLS + o + 4 * (fy == 2 ? NC - 1 : 0) + 32 * k + 2 * h, y);
    if (bz) half_ld(of(fz) + (size_t)nz * CELLS + o + 4 * j + 32 * (fz == 4 ? NC - 1 : 0) + 2 * h, z);
  };
  // exchange words (offsets in xch; + 32 for colour 1) of this thread's face
  // cells, and of the cells across: x faces by (j / 2, k), y faces by (q, k),
  // z faces by (q, j)
  const int me = blockIdx.x * XWORDS, ax = (j >> 1) + 4 * k, ay = 4 * k + 2 * h, az = 4 * j + 2 * h;
  const int wx = me + 64 * h + ax + 32 * cf, wy = me + 64 * fy + ay, wz = me + 64 * fz + az;
  const int qx = (nx - a.lo) * XWORDS + 64 * (h ^ 1) + ax + 32 * (cf ^ 1), qy = (ny - a.lo) * XWORDS + 64 * (fy ^ 1) + ay,
            qz = (nz - a.lo) * XWORDS + 64 * (fz ^ 1) + az;
  auto publish = [&](int c, unsigned ev) {  // this thread's face cells of colour c
    const unsigned tag = (tag0 + ev) & 0xffu;
    if (bx && cf == c) xst(a.xch + wx, h ? v[c][1] : v[c][0], tag);
    if (by) xst2(a.xch + wy + 32 * c, v[c][0], v[c][1], tag);
    if (bz) xst2(a.xch + wz + 32 * c, v[c][0], v[c][1], tag);
  };
  auto await = [&](int c, unsigned ev) {  // the halo of colour c's cells: the neighbours' other colour
    const unsigned tag = (tag0 + ev + a.skew) & 0xffu;
    const bool x = bx && cf == c;
    hx = 0;
    if (x || by || bz) {
      for (int it = 0;; ++it) {
        if (x) hx = xld(a.xch + qx);
        if (by) xld2(a.xch + qy + 32 * (c ^ 1), hy[0], hy[1]);
        if (bz) xld2(a.xch + qz + 32 * (c ^ 1), hz[0], hz[1]);
        unsigned d = 0;
        if (x) d |= (unsigned)hx ^ tag;
        if (by) d |= ((unsigned)hy[0] ^ tag) | ((unsigned)hy[1] ^ tag);
        if (bz) d |= ((unsigned)hz[0] ^ tag) | ((unsigned)hz[1] ^ tag);
        if ((d & 0xffu) == 0) break;
        if (it > WAIT_SPIN) {
          atomicOr(sc + SC_ERR, ERR_WAIT);
          break;
        }
      }
    }
    hx >>= 8;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      hy[e] >>= 8;
      hz[e] >>= 8;
    }
  };
  auto stage = [&](int c) { sv[c][r][h] = make_longlong2(v[c][0], v[c][1]); };
  // Sums of the six neighbours of this thread's cells of colour c in three
  // parts: inside the box, ghosts at walls and refinement faces (from the
  // cells' own values), halo.  The first two are formed before the halo is
  // awaited, so that only a few additions and the division by 6 lie between
  // its arrival and the next publication.  Rows outside the box are the zero
  // row.
  //
  // A box of level >= 1 has a sibling across three of its faces; only the
  // three outward ones (on the side of its octant) can be walls or refinement
  // faces.  Their ghosts depend on the colour's own values alone, so they are
  // formed one pass ahead, while the block waits for a halo: 32 cells a face,
  // a warp a face, from the staged values (a half row's own thread would form
  // up to five of them one after another with most of its warp idle).
  const int rym = j > 0 ? r - 1 : 64, ryp = j < NC - 1 ? r + 1 : 64, rzm = k > 0 ? r - 8 : 64,
            rzp = k < NC - 1 ? r + 8 : 64;
  auto inside = [&](int c, long long (&s)[2]) {
    const int oc = c ^ 1, p = (c + par) & 1;
    const longlong2 w0 = sv[oc][rym][h], w1 = sv[oc][ryp][h], w2 = sv[oc][rzm][h], w3 = sv[oc][rzp][h];
    const long long R0 = v[oc][0], R1 = v[oc][1];
    long long nb = __shfl_xor_sync(0xffffffffu, p ? R0 : R1, 1);  // one beyond the half
    nb = cf == c ? 0 : nb;
    s[0] = (R0 + (p ? R1 : nb)) + ((w0.x + w1.x) + (w2.x + w3.x));
    s[1] = (R1 + (p ? nb : R0)) + ((w0.y + w1.y) + (w2.y + w3.y));
  };
  auto make_ghosts = [&](int c) {
    const int A = t >> 5, at = t & 31;
    if (A == 3) return;
    const int hi = (oct >> A) & 1, f = 2 * A + hi, e = hi ? NC - 1 : 0;
    if (!((flags >> (10 + f)) & 65)) return;  // a box
    const int w = at >> 2;
    // cell (i, jj, kk) of the face, entry q of its row in colour c
    const int kk = A == 2 ? e : w, jj = A == 0 ? 2 * (at & 3) + ((c + e + w) & 1) : (A == 1 ? e : w);
    const int q = A == 0 ? e >> 1 : at & 3, i = 2 * q + ((c + jj + kk) & 1);
    const long long own = reinterpret_cast<const long long *>(sv[c][jj + NC * kk])[q];
    long long g;
    if ((flags >> (16 + f)) & 1) g = fx_div6(2 * own + sg[A][A == 0 ? jj + NC * kk : (A == 1 ? kk + NC * i : i + NC * jj)]);
    else g = a.bc.type[f] ? swall[f] - own : own;  // Dirichlet 2g - own, Neumann own
    reinterpret_cast<long long *>(sgh[c][A])[at] = g;
  };
  auto ghost_sum = [&](int c, long long (&s)[2]) {
    if (!(flags & GHOSTS)) return;  // the same for the whole block
    if (nx < 0 && cf == c) {
      const long long g = reinterpret_cast<const long long *>(sgh[c][0])[ax];
      s[0] += h ? 0 : g;
      s[1] += h ? g : 0;
    }
    auto add2 = [&](const longlong2 &w) {
      s[0] += w.x;
      s[1] += w.y;
    };
    if (ny == -1 || ny == -2) add2(sgh[c][1][ay >> 1]);
    if (nz == -1 || nz == -2) add2(sgh[c][2][az >> 1]);
  };
  auto halo_sum = [&](long long (&s)[2], long long x, const long long (&y)[2], const long long (&z)[2]) {
    s[0] += (h ? 0 : x) + (y[0] + z[0]);  // x is 0 unless cf is the colour
    s[1] += (h ? x : 0) + (y[1] + z[1]);
  };
  auto any_bad = [&](const long long (&x)[2]) { return fx_bad(x[0]) || fx_bad(x[1]); };
  auto put = [&](long long *p, const long long (&x)[2]) {
    *reinterpret_cast<longlong2 *>(p) = make_longlong2(x[0], x[1]);
  };
  bool bad = false;
  long long hx1 = 0, hy1[2] = {0, 0}, hz1[2] = {0, 0};  // colour 1's halo at a FAS start

  if (PRO) {
    // prolongation (as k_fprolong_half): coarse values of the parent region,
    // the 4^3 cells under the box and their 96 face neighbours
    auto val = [&](int Q, int c) {
      const size_t x = (size_t)Q * CELLS + c;
      return START == FS_FMG ? a.phx[x] : a.phx[x] - a.oldx[x];
    };
    auto reg = [](int x, int y, int z) { return x + 6 * y + 36 * z; };
    const int o0 = 4 * (flags & 1), o1 = 4 * ((flags >> 1) & 1), o2 = 4 * ((flags >> 2) & 1);
    if (t < 64) {
      const int x = t & 3, y = (t >> 2) & 3, z = t >> 4;
      sp[reg(x + 1, y + 1, z + 1)] = val(P, xpos(o0 + x, o1 + y, o2 + z));
    }
    const int e = t >= 64 ? t - 64 : t + 64;
    if (e < 96) {
      const int F = e >> 4, E = F >> 1, S = (F & 1) ? 1 : -1;
      const int u = e & 3, w = (e >> 2) & 3, ce = S > 0 ? 5 : 0;
      const int rx = E == 0 ? ce : (E == 1 ? w + 1 : u + 1);
      const int ry = E == 0 ? u + 1 : (E == 1 ? ce : w + 1);
      const int rz = E == 0 ? w + 1 : (E == 1 ? u + 1 : ce);
      const int lx = o0 - 1 + rx, ly = o1 - 1 + ry, lz = o2 - 1 + rz;
      const int le = E == 0 ? lx : (E == 1 ? ly : lz);
      const int Qn = le >= 0 && le < NC ? P : (E == 0 ? pn[0] : (E == 1 ? pn[1] : pn[2]));
      // the cell itself, the neighbour's across the face (the coordinate
      // wraps), or, without one, the cell inside next to the face
      const int d = Qn >= 0 ? 0 : S;
      long long w0 = val(Qn >= 0 ? Qn : P, xpos((lx - (E == 0 ? d : 0)) & 7, (ly - (E == 1 ? d : 0)) & 7,
                                                (lz - (E == 2 ? d : 0)) & 7));
      if (Qn < 0) {
        if (Qn == -1) w0 = a.bc.type[F] ? (START == FS_FMG ? fx_2g(sc, F) : 0) - w0 : w0;
        else atomicOr(sc + SC_ERR, 1ull);
      }
      sp[reg(rx, ry, rz)] = w0;
    }
    __syncthreads();
    {
      const int y = (j >> 1) + 1, z = (k >> 1) + 1, sy = (j & 1) ? 6 : -6, sz = (k & 1) ? 36 : -36;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int at = reg(2 * h + q + 1, y, z);
        const long long yz = sp[at] + sp[at + sy] + sp[at + sz];
        // the even cell of the pair has colour par, the odd one the other
        const long long ce = fx_rdiv<4>(yz + sp[at - 1]), co = fx_rdiv<4>(yz + sp[at + 1]);
        const long long d0 = par ? co : ce, d1 = par ? ce : co;
        v[0][q] = START == FS_FMG ? d0 : v[0][q] + d0;
        v[1][q] = START == FS_FMG ? d1 : v[1][q] + d1;
      }
    }
    publish(1, 0);
    bad = any_bad(v[0]) || any_bad(v[1]);
    if (flags & CFS) {  // Ghat of the refinement faces: axes 0 and 2 by warps 0-1, axis 1 by warps 2-3
      const int u = t & 7, w = (t >> 3) & 7;
      auto cfa = [&](int A) { return (flags >> (16 + 2 * A + ((oct >> A) & 1))) & 1; };
      auto keep = [&](int A, long long g) {
        sg[A][t & 63] = g;
        a.ghx[(size_t)(6 * b + 2 * A + ((oct >> A) & 1)) * FACE + (t & 63)] = g;
      };
      if (t < 64) {
        if (cfa(0)) keep(0, leg_ghat<0>(a.phx, a.bc, pn, pe, oct, u, w, swall, sc + SC_ERR));
        if (cfa(2)) keep(2, leg_ghat<2>(a.phx, a.bc, pn, pe, oct, u, w, swall, sc + SC_ERR));
      } else {
        if (cfa(1)) keep(1, leg_ghat<1>(a.phx, a.bc, pn, pe, oct, u, w, swall, sc + SC_ERR));
      }
    }
  } else {
    load_halo(0, hx, hy, hz);
    if (refined) load_halo(1, hx1, hy1, hz1);
    if (flags & CFS) {
      for (int n = t; n < 3 * FACE; n += 128) {
        const int A = n >> 6, f = 2 * A + ((oct >> A) & 1);
        if ((flags >> (16 + f)) & 1) sg[A][n & 63] = a.ghx[(size_t)(6 * b + f) * FACE + (n & 63)];
      }
    }
    if (START == FS_FAS && !refined) {
      put(a.oldx + base, v[0]);
      put(a.oldx + base + 256, v[1]);
    }
  }
  stage(0);
  stage(1);
  __syncthreads();
  if (flags & GHOSTS) {
    make_ghosts(0);
    if (!PRO) make_ghosts(1);
    __syncthreads();
  }
  unsigned ev = 0;  // the last publication made
  long long s[2], s1[2];
  if (!PRO) {
    // first pass (colour 0), after the FAS right-hand side of a refined box,
    // G = (children's sum - 2 T) / 12, T = h^2 L phi, from the same sums
    inside(0, s);
    ghost_sum(0, s);
    halo_sum(s, hx, hy, hz);
    if (refined) {
      inside(1, s1);
      ghost_sum(1, s1);
      halo_sum(s1, hx1, hy1, hz1);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        G[0][e] = fx_rdiv<12>(G[0][e] - 2 * (s[e] - 6 * v[0][e]));
        G[1][e] -= 2 * (s1[e] - 6 * v[1][e]);
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) v[0][e] = fx_div6(s[e] + 6 * G[0][e]);
    publish(0, ++ev);
    if (refined) {
#pragma unroll
      for (int e = 0; e < 2; ++e) G[1][e] = fx_rdiv<12>(G[1][e]);
      bad = any_bad(G[0]) || any_bad(G[1]);
      put(a.gx + base, G[0]);
      put(a.gx + base + 256, G[1]);
      __syncthreads();  // colour 0 of sv has been read for colour 1's sums
    }
    bad |= any_bad(v[0]);
    stage(0);
    __syncthreads();
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    G[0][e] *= 6;
    G[1][e] *= 6;
  }
  for (int sweep = 0; sweep < a.nu; ++sweep) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (!PRO && c == 0 && sweep == 0) continue;
      long long g[2] = {G[c][0], G[c][1]};
      inside(c, s);
      ghost_sum(c, g);
      if (flags & GHOSTS) make_ghosts(c ^ 1);  // for the next pass
      await(c, ev);
      halo_sum(s, hx, hy, hz);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (!UP && c == 1) s1[e] = s[e];  // colour 1's sums without its ghosts
        v[c][e] = fx_div6(s[e] + g[e]);
      }
      ++ev;
      if (!UP || c == 0 || sweep + 1 < a.nu) {
        publish(c, ev);
        stage(c);
        __syncthreads();
      }
      bad |= any_bad(v[c]);
    }
  }
  if (!UP) {
    // residual 6 G + T of every cell and both 8-child sums (the x pair of
    // coarse cell 2h + e is entry e of the two colours; rows j ^ 1 and k ^ 1
    // are lanes ^ 2 and ^ 16)
    inside(0, s);
    ghost_sum(0, s);
    if (flags & GHOSTS) {  // colour 1's of its last values
      make_ghosts(1);
      __syncthreads();
      ghost_sum(1, s1);
    }
    long long ap[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      ap[e] = v[0][e] + v[1][e];
      s[e] += (G[0][e] + G[1][e]) - 6 * ap[e] + s1[e];
      ap[e] += __shfl_xor_sync(0xffffffffu, ap[e], 2);
      ap[e] += __shfl_xor_sync(0xffffffffu, ap[e], 16);
      ap[e] = fx_rdiv<8>(ap[e]);
    }
    await(0, ev);  // the neighbours' last colour-1 cells
    halo_sum(s, hx, hy, hz);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      s[e] += __shfl_xor_sync(0xffffffffu, s[e], 2);
      s[e] += __shfl_xor_sync(0xffffffffu, s[e], 16);
    }
    if (((j | k) & 1) == 0) {
      const size_t pb = (size_t)P * CELLS;
      const int cx = 4 * (flags & 1) + 2 * h, cy = 4 * ((flags >> 1) & 1) + (j >> 1),
                cz = 4 * ((flags >> 2) & 1) + (k >> 1);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const size_t cc = pb + xpos(cx + e, cy, cz);
        if (a.set_phx) a.phx[cc] = ap[e];
        a.oldx[cc] = ap[e];
        a.gx[cc] = s[e];
      }
    }
  }
  put(a.phx + base, v[0]);
  put(a.phx + base + 256, v[1]);
  fx_flag(bad, sc);
}

}  // namespace fx
