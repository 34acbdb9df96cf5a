// rbsolve.cuh -- the persistent solve on colour-split levels.
//
// Multigrid (arXiv:1809.03745, Sec. 3.3.2) with every level stored split by
// the red-black colouring: the red cells of an x row lie next to each other,
// then, in a second half, the black ones.  What that buys on a GB300:
//   * a colour pass reads only the other colour's values and its own
//     right-hand side and writes only its own values, four cells of the colour
//     per 16-byte access, where the plain layout moves both colours' lines for
//     each pass (256^3 FP32: 100 MB per pass instead of 218 MB);
//   * a pass writes a third buffer, which then takes the place of the colour's
//     old one.  The sparse rows of the colour's cut cells, whose stencils may
//     reach cells of their own colour, therefore read the values of before the
//     pass, in the same phase as the regular cells: one grid barrier per
//     colour instead of two, with the same values;
//   * the four (2D: two) red cells under four neighbouring coarse cells lie at
//     the same four positions as those, so restriction and prolongation are
//     vector passes too.  After a black pass the residual of a regular black
//     cell is zero (its equation was just solved), so restriction forms the
//     red ones only.
// The correction of each V-cycle joins a Krylov space (rb_kry_coeff): a few
// modes that the coarse grids represent badly (a pin thinner than a coarse
// cell, a rough interface) no longer set the rate, so three sweeps per leg do
// in 3D what six did.  Measured on a GB300, solves to 1e-13 of max|b|, against
// the plain layout without any of this: pin-plane 256^3 134 -> 34 ms (24
// V-cycles of 6+6 sweeps -> 16 of 3+3), 384^3 334 -> 89 ms; rod-plane 128^2
// 3.5 -> 2.7 ms, 1024^2 10.3 -> 7.0 ms; 632 x 488, whose 79 x 61 bottom was
// BiCGStab over the grid and is now algebraic levels, 62.6 -> 6.3 ms; 512^2 in
// FP64 20.7 -> 9.3 ms.
// The phases are functions out of line: inlined into one kernel, ptxas spilled
// 4.8 KB of them and took minutes.  The grid barrier, the bounded waits and the
// trace are those of persistent.cuh.
#pragma once

#include "persistent.cuh"

namespace ebp {

constexpr int RMAX = 28;  // levels, the algebraic ones included
constexpr int KH = 4;     // Krylov slots: the new direction and the three before it
constexpr int KDOT = 2 * KH;  // sums per pass: (r, q), (q, q), then (q, q_i) and (r, q_i)
struct KryState;

// split flags: the cell flags of eb_common.cuh and, per cell,
constexpr unsigned R_SPC = 8;       // a child has a sparse row (its right-hand side comes from the special list)
constexpr unsigned R_LIN0 = 16;     // phase p: every coarse cell of the linear interpolation has an unknown (R_LIN0 << p)
constexpr unsigned R_NOHOME0 = 64;  // phase p: the coarse cell above has no unknown (R_NOHOME0 << p)
constexpr unsigned R_BASE = 0x07070707u;

template <class T>
struct RLev {
  FastDiv dq, dn1;  // nq, n[1]
  int D, n[3];
  int hx;   // cells of one colour per x row, rounded up to 4 (entries past the row have flags 0)
  int nq;   // groups of four of them
  int nqt;  // groups per colour
  int H;    // entries per colour
  int two;  // both phases
  int dense;  // the level has regular cells
  int full;   // x rows fill their groups (n[0] a multiple of 8)
  int wide;   // at least two cells along every axis
  T dge[2];   // diagonal count of a cell at the low / high x wall and nowhere else
  T ide[2][2];  // and its reciprocal with the shift, [side][phase]
  int p1o, p1n;  // the entries of a dielectric half that are stored (the slabs that hold the phase)
  T wr[6], w3[6], lh[2], idg[2], ceps[2], h2e[2];
  // per phase three halves: after s sweeps red is x[p][2s % 3], black
  // x[p][(2s + 1) % 3], and the third is written next
  T* x[2][3];
  T* b[2][2];  // [phase][colour]
  const uint8_t* f[2];
  // groups per colour that a pass does not find on the common path (group | phase << 31), see rb_dense
  const unsigned* gl[2];
  int ngl[2];
  // sparse rows of cells and phases with an unknown, red first
  int nr, nr0;
  int staged;            // entries in T in this CTA's shared memory
  const int2* re;        // first and last entry
  const unsigned* rs;    // the row's own cell: phase << 31 | colour * H + position
  const unsigned* col;   // entries' cells, encoded alike
  const void *val, *dinv;  // double, or T when staged; dinv = 1 / diagonal
  // restriction rows: per unknown of the next level whose cell has a child
  // with a sparse row, the mean of its children's residuals as one row over
  // this level (first entry; entries | children mask << 16 | phase << 24;
  // position of child 0; the unknown as colour * H + position)
  int nsp;
  int sstaged;
  const int4* sd;
  const unsigned* scol;
  const void* sval;  // double, or T when staged
};

template <class T>
struct RHier {
  int nlev, lc;     // levels; the first one inside CTA 0
  int nu1[RMAX], nu2[RMAX], bsweeps;  // sweeps per level, and on the last one
  int bot;          // 0 relaxation, 1 inverse (in CTA 0 when local, else over the grid)
  int bm;           // order of the inverse
  const T* binv;    // [bm][bm] row-major, slots as bslot
  const unsigned* bslot;  // slot -> phase << 31 | colour * H + position; ~0u: no unknown
  int smem;         // levels lc.. in CTA 0's shared memory
  RLev<T> L[RMAX + 1];  // L[RMAX]: level lc as the whole group sees it
  // byte offsets into shared memory of levels lc..
  int off_x[RMAX][2][3], off_b[RMAX][2][2], off_f[RMAX][2], off_re[RMAX], off_rs[RMAX], off_col[RMAX], off_val[RMAX],
      off_di[RMAX], off_sd[RMAX], off_sc[RMAX], off_sv[RMAX], nnz[RMAX], snnz[RMAX];
  int srows[RMAX];  // 1: rows staged too, 2: restriction rows
  // finest level in FP64: natural cell of every sparse row, entries' natural
  // columns and values, the rows' diagonals
  const int *rnat, *ncol;
  const double *rval, *rdiag;
  // Krylov directions of the finest level, [slot][phase][colour]: z and q = A z
  T *kz[KH][2][2], *kq[KH][2][2];
  double* kpart;       // [chunk][KDOT] partial sums
  int kcs, kch, krows;  // groups per chunk, chunks, sparse rows per chunk
  KryState* kst;
};

// What a phase runs on: the whole group of CTAs, or CTA 0 alone.  Kept in
// shared memory; what differs between threads is worked out where it is used.
struct RCtx {
  int st, gst;  // strides over items and over groups of 8 lanes
  bool local;
  int gcta, gsize;
  Barrier B;
  unsigned* epoch;
  unsigned long long* tr;
  unsigned* tn;
  __device__ __forceinline__ int wi() const { return (int)(threadIdx.x >> 5) * gsize + gcta; }  // warps interleaved over the CTAs
  __device__ __forceinline__ int i0() const { return local ? (int)threadIdx.x : wi() * 32 + (int)(threadIdx.x & 31); }
  // groups of 8 lanes are counted from the other end
  __device__ __forceinline__ int g0() const {
    return local ? (int)(threadIdx.x >> 3) : gst - 1 - (wi() * 4 + (int)((threadIdx.x >> 3) & 3));
  }
  __device__ __forceinline__ bool sync(int code) const {
    bool ok = true;
    if (local) __syncthreads();
    else ok = grid_sync(B, epoch, gsize);
    if (tr && gcta == 0 && threadIdx.x == 0 && *tn < TRMAX) {
      tr[1 + *tn] = ((unsigned long long)code << 48) | (now_ns() & 0xffffffffffffULL);
      *tn += 1;
    }
    return ok;
  }
};

// The directions kept: in shared memory, and in global memory between the
// launches of a resumed solve.
struct KryState {
  int count, next;   // directions kept, slot of the next one
  int es;            // the solve's unit is 2^es (see unit_of)
  double g[KH][KH];  // (q_i, q_j) by slot
  double rn[KH];     // 1 / |q_i|
};
// The state of a launch.  The phases are functions out of line that find it
// here and take a few integers: ptxas gives a function the registers that its
// callers leave, and with descriptions, contexts and loop state held in the
// callers' registers the phases spilled in their loops (a tenth of all
// instructions; a solve of 1024^2 took 7.5 ms instead of 6.9, one of 256^3 35.7 instead of 33.7).
template <class T>
struct RShared {
  RHier<T> H;
  RCtx c[2];  // the group, CTA 0 alone
  Op<double> F;
  unsigned epoch, tn;
  int cur;  // phi and b are in units of 2^cur
  T red[PT / 32][KDOT];
  double dots[KDOT], coef[KH];
  KryState K;
};
template <class T>
__device__ __forceinline__ RShared<T>& rsh() {
  __shared__ RShared<T> s;
  return s;
}

template <class T>
__device__ __forceinline__ void st4(T* p, const T v[4]) {
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
  }
}
template <class T>
__device__ __forceinline__ void ld2(const T* p, T& a, T& b) {
  if constexpr (sizeof(T) == 4) {
    const float2 q = *reinterpret_cast<const float2*>(p);
    a = q.x;
    b = q.y;
  } else {
    const double2 q = *reinterpret_cast<const double2*>(p);
    a = q.x;
    b = q.y;
  }
}

// a group of four cells of one colour: x row (j, k), positions q0 .. q0 + 3,
// cells i = 2 q + s
struct QPos {
  int t, j, k, q0, s;
};
template <class T>
__device__ __forceinline__ QPos quad_pos(const RLev<T>& L, int t, int colour) {
  QPos g;
  const unsigned row = fdiv((unsigned)t, L.dq);
  const unsigned kq = fdiv(row, L.dn1);
  g.t = t;
  g.j = (int)(row - kq * (unsigned)L.n[1]);
  g.k = (int)kq;
  g.q0 = 4 * (t - (int)row * L.nq);
  g.s = (g.j + g.k + colour) & 1;
  return g;
}
// bytes 0xff where the cell is regular and of phase p
__device__ __forceinline__ unsigned regular_mask(unsigned w, int p) {
  return __vcmpeq4(w & R_BASE, p ? 0x02020202u : 0x01010101u);
}

// the other colour's values around a group: row centre, y and z neighbours,
// and the one x neighbour outside the group
template <class T>
struct QNb {
  T c[4], ym[4], yp[4], zm[4], zp[4], xs;
};
template <class T>
__device__ __forceinline__ void quad_load(const RLev<T>& L, const QPos& g, const T* xn, QNb<T>& v) {
  const T* c = xn + 4 * (long long)g.t;
  const int sy = L.hx, sz = L.hx * L.n[1];
  ld4(c, v.c);
  v.xs = T(0);
  if (g.s == 0) {
    if (g.q0 > 0) v.xs = c[-1];
  } else if (2 * g.q0 + 8 < L.n[0]) {
    v.xs = c[4];
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) v.ym[e] = v.yp[e] = v.zm[e] = v.zp[e] = T(0);
  if (g.j > 0) ld4(c - sy, v.ym);
  if (g.j < L.n[1] - 1) ld4(c + sy, v.yp);
  if (L.D == 3) {
    if (g.k > 0) ld4(c - sz, v.zm);
    if (g.k < L.n[2] - 1) ld4(c + sz, v.zp);
  }
}
// per lane the neighbour sum and the diagonal count (open faces, 3 w per wall
// face of weight w) of the implicit stencil; walls as in mg_kernels.cuh
template <class T>
__device__ __forceinline__ void quad_sums(const RLev<T>& L, const QPos& g, QNb<T>& v, T sum[4], T dg[4]) {
  T d0 = T(2 * L.D);
  if (g.j == 0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v.ym[e] = L.w3[2] * v.yp[e];
    d0 += T(3) * L.wr[2] - T(1);
  }
  if (g.j == L.n[1] - 1) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v.yp[e] = L.w3[3] * v.ym[e];
    d0 += T(3) * L.wr[3] - T(1);
  }
  if (L.D == 3) {
    if (g.k == 0) {
#pragma unroll
      for (int e = 0; e < 4; ++e) v.zm[e] = L.w3[4] * v.zp[e];
      d0 += T(3) * L.wr[4] - T(1);
    }
    if (g.k == L.n[2] - 1) {
#pragma unroll
      for (int e = 0; e < 4; ++e) v.zp[e] = L.w3[5] * v.zm[e];
      d0 += T(3) * L.wr[5] - T(1);
    }
  }
  const int last = L.n[0] - 1 - 2 * g.q0 - g.s;  // twice the lane of the row's last cell, if even
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    T l = g.s ? v.c[e] : (e ? v.c[e ? e - 1 : 0] : v.xs);
    T r = g.s ? (e < 3 ? v.c[e < 3 ? e + 1 : 3] : v.xs) : v.c[e];
    T d = d0;
    if (e == 0 && g.s == 0 && g.q0 == 0) {
      l = L.w3[0] * r;
      d += T(3) * L.wr[0] - T(1);
    }
    if (last == 2 * e) {
      r = L.w3[1] * l;
      d += T(3) * L.wr[1] - T(1);
    }
    sum[e] = ((l + r) + (v.ym[e] + v.yp[e])) + (v.zm[e] + v.zp[e]);
    dg[e] = d;
  }
}
// The same in a third of the instructions on levels of two cells or more along
// each axis: every load goes out at once, what lies outside a y or z wall from
// the opposite side (which is what the wall's stencil takes, scaled), and the
// cells at the x walls, lane 0 of a row's first group and lane `hi` of its last
// one, are put right afterwards.
struct QEnd {
  bool lo;
  int hi;  // 4 or more: none
};
template <class T>
__device__ __forceinline__ QEnd quad_end(const RLev<T>& L, const QPos& g) {
  const int last = L.n[0] - 1 - 2 * g.q0 - g.s;  // of both colours' cells, the row's last one lies `last` cells on
  return QEnd{g.s == 0 && g.q0 == 0, (last & 1) ? 4 : last >> 1};
}
template <class T>
__device__ __forceinline__ void quad_load_in(const RLev<T>& L, const QPos& g, const T* xn, QNb<T>& v) {
  const T* c = xn + 4 * g.t;
  ld4(c, v.c);
  v.xs = c[g.s ? (g.q0 + 4 < L.hx ? 4 : 0) : (g.q0 ? -1 : 0)];
  ld4(c + (g.j > 0 ? -L.hx : L.hx), v.ym);
  ld4(c + (g.j < L.n[1] - 1 ? L.hx : -L.hx), v.yp);
  if (L.D == 3) {
    const int sz = L.hx * L.n[1];
    ld4(c + (g.k > 0 ? -sz : sz), v.zm);
    ld4(c + (g.k < L.n[2] - 1 ? sz : -sz), v.zp);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) v.zm[e] = v.zp[e] = T(0);
  }
}
// scales what was loaded across y and z walls; the diagonal count they add
template <class T>
__device__ __forceinline__ T quad_walls(const RLev<T>& L, const QPos& g, QNb<T>& v) {
  T d = T(0);
  if (g.j == 0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v.ym[e] *= L.w3[2];
    d += T(3) * L.wr[2] - T(1);
  }
  if (g.j == L.n[1] - 1) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v.yp[e] *= L.w3[3];
    d += T(3) * L.wr[3] - T(1);
  }
  if (L.D == 3) {
    if (g.k == 0) {
#pragma unroll
      for (int e = 0; e < 4; ++e) v.zm[e] *= L.w3[4];
      d += T(3) * L.wr[4] - T(1);
    }
    if (g.k == L.n[2] - 1) {
#pragma unroll
      for (int e = 0; e < 4; ++e) v.zp[e] *= L.w3[5];
      d += T(3) * L.wr[5] - T(1);
    }
  }
  return d;
}
template <class T>
__device__ __forceinline__ void quad_sums_in(const RLev<T>& L, const QPos& g, const QEnd& x, const QNb<T>& v, T sum[4]) {
  const T o = v.xs + (g.s ? v.c[3] : v.c[0]), a = v.c[0] + v.c[1], b = v.c[1] + v.c[2], d = v.c[2] + v.c[3];
  T h[4] = {g.s ? a : o, g.s ? b : a, g.s ? d : b, g.s ? o : d};
  if (x.lo) h[0] = v.c[0] + L.w3[0] * v.c[0];
  if ((unsigned)x.hi < 4u) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const T l = g.s ? v.c[e] : (e ? v.c[e ? e - 1 : 0] : v.xs);
      if (e == x.hi) h[e] = l + L.w3[1] * l;
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) sum[e] = (h[e] + (v.ym[e] + v.yp[e])) + (v.zm[e] + v.zp[e]);
}
// A group away from the y and z walls whose row goes on behind it or ends with
// its last lane: only lane 0 (s = 0) or lane 3 (s = 1) may lie at an x wall,
// and nothing has to be scaled.  Nearly every group is one, and takes two
// thirds of the instructions.
__host__ __device__ __forceinline__ bool inner_group(int D, int n0, int n1, int n2, const QPos& g) {
  return (n0 % 8 == 0 || 2 * g.q0 + 8 < n0) && g.j > 0 && g.j < n1 - 1 && (D == 2 || (g.k > 0 && g.k < n2 - 1));
}
template <class T>
__device__ __forceinline__ bool quad_inner(const RLev<T>& L, const QPos& g) {
  return (L.full || 2 * g.q0 + 8 < L.n[0]) && (unsigned)(g.j - 1) < (unsigned)(L.n[1] - 2) &&
         (L.D == 2 || (unsigned)(g.k - 1) < (unsigned)(L.n[2] - 2));
}
template <class T>
__device__ __forceinline__ bool quad_edge(const RLev<T>& L, const QPos& g) {
  return g.s ? g.q0 + 4 == L.hx : g.q0 == 0;
}
template <class T>
__device__ __forceinline__ void quad_sums_inner(const RLev<T>& L, const QPos& g, bool edge, const QNb<T>& v, T sum[4]) {
  const T ce = g.s ? v.c[3] : v.c[0];
  const T xs = edge ? L.w3[g.s] * ce : v.xs;
  const T o = xs + ce, a = v.c[0] + v.c[1], b = v.c[1] + v.c[2], d = v.c[2] + v.c[3];
  const T h[4] = {g.s ? a : o, g.s ? b : a, g.s ? d : b, g.s ? o : d};
#pragma unroll
  for (int e = 0; e < 4; ++e) sum[e] = (h[e] + (v.ym[e] + v.yp[e])) + (v.zm[e] + v.zp[e]);
}
// operator values of such a group from its own values xo
template <class T>
__device__ __forceinline__ void quad_apply_in(const RLev<T>& L, const QPos& g, int p, QNb<T>& v, const T xo[4], T q[4]) {
  T sum[4];
  const T ce = L.ceps[p];
  if (quad_inner(L, g)) {
    const bool edge = quad_edge(L, g);
    quad_sums_inner(L, g, edge, v, sum);
    const T d = T(2 * L.D) + L.lh[p], de = edge ? L.dge[g.s] + L.lh[p] : d;
    q[0] = ce * ((g.s ? d : de) * xo[0] - sum[0]);
    q[1] = ce * (d * xo[1] - sum[1]);
    q[2] = ce * (d * xo[2] - sum[2]);
    q[3] = ce * ((g.s ? de : d) * xo[3] - sum[3]);
    return;
  }
  const QEnd x = quad_end(L, g);
  const T dw = quad_walls(L, g, v);
  quad_sums_in(L, g, x, v, sum);
  const T d = T(2 * L.D) + dw + L.lh[p], d0 = x.lo ? L.dge[0] + dw + L.lh[p] : d, d1 = L.dge[1] + dw + L.lh[p];
#pragma unroll
  for (int e = 0; e < 4; ++e) q[e] = ce * ((e == x.hi ? d1 : (e ? d : d0)) * xo[e] - sum[e]);
}
template <class T>
__device__ __forceinline__ T quad_inv(const RLev<T>& L, int p, T dg) {
  return dg == T(2 * L.D) ? L.idg[p] : rcp_rn(dg + L.lh[p]);
}

// writes the lanes of `m` (byte masks) of a group
template <class T>
__device__ __forceinline__ void quad_store(T* dst, unsigned m, const T v[4]) {
  if (m == 0xffffffffu) {
    st4(dst, v);
    return;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if ((m >> (8 * e)) & 1u) dst[e] = v[e];
}

// The residual (bb) or the operator value (no bb) of any group, out of line:
// for levels one cell thick and the residual of both colours.  A persistent
// kernel runs a different phase every few microseconds, and the instructions
// it has to fetch for one cost more than a small level's arithmetic.
template <class T>
__device__ __noinline__ void quad_slow(const RLev<T>& __restrict__ L, int t, int colour, int p, const T* xn, const T* xo,
                                       const T* bb, T* o) {
  const QPos g = quad_pos(L, t, colour);
  QNb<T> v;
  T sum[4], dg[4];
  quad_load(L, g, xn, v);
  quad_sums(L, g, v, sum, dg);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const T r = L.ceps[p] * ((dg[e] + L.lh[p]) * xo[4 * (long long)t + e] - sum[e]);
    o[e] = bb ? bb[4 * (long long)t + e] - r : r;
  }
}

// buffers of a level after s sweeps
__device__ __forceinline__ int rb_red(int s) { return (2 * s) % 3; }
__device__ __forceinline__ int rb_black(int s) { return (2 * s + 1) % 3; }

// the diagonals' reciprocals of a group: inside, at lane 0, at lane x.hi
template <class T>
__device__ __forceinline__ void quad_inverse(const RLev<T>& L, const QEnd& x, int p, T dw, T& in, T& v0, T& v1) {
  in = L.idg[p];
  v0 = x.lo ? L.ide[0][p] : in;
  v1 = L.ide[1][p];
  if (dw != T(0)) {
    in = rcp_rn(T(2 * L.D) + dw + L.lh[p]);
    v0 = x.lo ? rcp_rn(L.dge[0] + dw + L.lh[p]) : in;
    v1 = rcp_rn(L.dge[1] + dw + L.lh[p]);
  }
}

// The regular cells of one colour in sweep s: the inner groups, the phase of
// each that rb_dense_list does not have.
template <class T>
__device__ __noinline__ void rb_dense(int lv, int colour, int s, int cx) {
  const RLev<T>& L = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const int in = colour ? rb_red(s + 1) : rb_black(s);
  const int out = colour ? rb_black(s + 1) : rb_red(s + 1);
  const unsigned* fw = reinterpret_cast<const unsigned*>(L.f[colour]);
  const int st = c.st, nqt = L.nqt;
  // U groups per thread with all their loads issued first; the flags of the
  // next ones are loaded one iteration ahead
  constexpr int U = sizeof(T) == 4 ? 2 : 1;
  unsigned wn[U];
#pragma unroll
  for (int u = 0; u < U; ++u) wn[u] = c.i0() + u * st < nqt ? fw[c.i0() + u * st] : 0u;
#pragma unroll 1
  for (int t0 = c.i0(); t0 < nqt; t0 += U * st) {
    unsigned w[U], m[U];
    int pp[U];
    QPos g[U];
    QNb<T> v[U];
    T bb[U][4];
    bool ed[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      w[u] = wn[u];
      const int tn = t0 + (U + u) * st;
      wn[u] = tn < nqt ? fw[tn] : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      m[u] = regular_mask(w[u], 0);
      pp[u] = m[u] ? 0 : 1;
      if (!m[u]) m[u] = regular_mask(w[u], 1);
      if (!m[u]) continue;
      g[u] = quad_pos(L, t0 + u * st, colour);
      if (!quad_inner(L, g[u])) {
        m[u] = 0u;
        continue;
      }
      const T* x = L.x[pp[u]][in] + 4 * g[u].t;
      ed[u] = quad_edge(L, g[u]);
      ld4(x, v[u].c);
      v[u].xs = x[ed[u] ? 0 : (g[u].s ? 4 : -1)];
      ld4(x - L.hx, v[u].ym);
      ld4(x + L.hx, v[u].yp);
      if (L.D == 3) {
        const int sz = L.hx * L.n[1];
        ld4(x - sz, v[u].zm);
        ld4(x + sz, v[u].zp);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[u].zm[e] = v[u].zp[e] = T(0);
      }
      ld4(L.b[pp[u]][colour] + 4 * g[u].t, bb[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!m[u]) continue;
      T o[4], sum[4];
      const int p = pp[u];
      const T h = L.h2e[p], iv = L.idg[p], ve = ed[u] ? L.ide[g[u].s][p] : iv;
      quad_sums_inner(L, g[u], ed[u], v[u], sum);
      o[0] = (h * bb[u][0] + sum[0]) * (g[u].s ? iv : ve);
      o[1] = (h * bb[u][1] + sum[1]) * iv;
      o[2] = (h * bb[u][2] + sum[2]) * iv;
      o[3] = (h * bb[u][3] + sum[3]) * (g[u].s ? ve : iv);
      quad_store(L.x[p][out] + 4 * g[u].t, m[u], o);
    }
  }
}
// The other groups, from a list made at set-up: those at a y or z wall or in
// the last group of a padded row, and the dielectric's cells of a group that
// holds both phases.  Handled where rb_dense meets them they cost a 1024^2
// level 1.1 us of a pass and a 256^3 level 6: the general arithmetic is
// branches and code in the way of every group.  Spread from the middle of the
// grid on, so that small levels have them on warps of their own.
template <class T>
__device__ __noinline__ void rb_dense_list(int lv, int colour, int s, int cx) {
  const RLev<T>& L = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const int in = colour ? rb_red(s + 1) : rb_black(s);
  const int out = colour ? rb_black(s + 1) : rb_red(s + 1);
  const int n = L.ngl[colour], half = c.st / 2;
  const unsigned* gl = L.gl[colour];
  const uint8_t* f = L.f[colour];
  for (int i = c.i0() < half ? c.i0() + half : c.i0() - half; i < n; i += c.st) {
    const unsigned en = gl[i];
    const int p = (int)(en >> 31), t = (int)(en & 0x7fffffffu);
    const unsigned m = regular_mask(reinterpret_cast<const unsigned*>(f)[t], p);
    const QPos g = quad_pos(L, t, colour);
    QNb<T> v;
    T bb[4], sum[4], o[4];
    ld4(L.b[p][colour] + 4 * t, bb);
    if (L.wide) {
      T iv, v0, v1;
      const QEnd x = quad_end(L, g);
      quad_load_in(L, g, L.x[p][in], v);
      const T dw = quad_walls(L, g, v);
      quad_sums_in(L, g, x, v, sum);
      quad_inverse(L, x, p, dw, iv, v0, v1);
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = (L.h2e[p] * bb[e] + sum[e]) * (e == x.hi ? v1 : (e ? iv : v0));
    } else {
      T dg[4];
      quad_load(L, g, L.x[p][in], v);
      quad_sums(L, g, v, sum, dg);
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = (L.h2e[p] * bb[e] + sum[e]) * quad_inv(L, p, dg[e]);
    }
    quad_store(L.x[p][out] + 4 * t, m, o);
  }
}
// all of them in the first red pass over a zero iterate, which is not read
template <class T>
__device__ __noinline__ void rb_dense_zero(int lv, int s, int cx) {
  const RLev<T>& L = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const int out = rb_red(s + 1);
  const unsigned* fw = reinterpret_cast<const unsigned*>(L.f[0]);
  for (int t = c.i0(); t < L.nqt; t += c.st) {
    const unsigned w = fw[t];
#pragma unroll 1
    for (int p = 0; p <= L.two; ++p) {
      const unsigned m = regular_mask(w, p);
      if (!m) continue;
      T o[4], bb[4];
      const QPos g = quad_pos(L, t, 0);
      QNb<T> v;
      ld4(L.b[p][0] + 4 * t, bb);
      if (L.wide) {
        const QEnd x = quad_end(L, g);
        T iv, v0, v1;
        quad_inverse(L, x, p, quad_walls(L, g, v), iv, v0, v1);
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = L.h2e[p] * bb[e] * (e == x.hi ? v1 : (e ? iv : v0));
      } else {
        T sum[4], dg[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v.c[e] = v.ym[e] = v.yp[e] = v.zm[e] = v.zp[e] = T(0);
        v.xs = T(0);
        quad_sums(L, g, v, sum, dg);
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = L.h2e[p] * bb[e] * quad_inv(L, p, dg[e]);
      }
      quad_store(L.x[p][out] + 4 * t, m, o);
    }
  }
}

// a value by its encoded cell (phase << 31 | colour * H + position)
template <class T>
struct Gather {
  const T *r0, *b0, *r1, *b1;
  unsigned H;
  __device__ __forceinline__ T operator()(unsigned cl) const {
    const unsigned s = cl & 0x7fffffffu;
    const bool blk = s >= H;
    const T* p = (cl >> 31) ? (blk ? b1 : r1) : (blk ? b0 : r0);
    return p[blk ? s - H : s];
  }
};
template <class T>
__device__ __forceinline__ Gather<T> rb_gather(const RLev<T>& L, int red, int black) {
  return Gather<T>{L.x[0][red], L.x[0][black], L.x[1][red], L.x[1][black], (unsigned)L.H};
}
template <class T>
__device__ __forceinline__ T* rb_rhs(const RLev<T>& L, unsigned cl, unsigned& pos) {
  const unsigned s = cl & 0x7fffffffu;
  const int colour = s >= (unsigned)L.H;
  pos = colour ? s - (unsigned)L.H : s;
  return L.b[cl >> 31][colour];
}

// off-diagonal sum of a row by one thread, entries eight at a time
template <class T, class V>
__device__ __forceinline__ V row_sum1(const RLev<T>& L, int2 re, const Gather<T>& x, unsigned lim) {
  V s = V(0);
  const V* val = (const V*)L.val;
  for (int e = re.x; e < re.y; e += 8) {
    unsigned cl[8];
    V a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      cl[k] = 0xffffffffu;
      a[k] = V(0);
      if (e + k < re.y) {
        cl[k] = L.col[e + k];
        a[k] = val[e + k];
      }
    }
    T xv[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) xv[k] = (e + k < re.y && (cl[k] & 0x7fffffffu) < lim) ? x(cl[k]) : T(0);
#pragma unroll
    for (int k = 0; k < 8; ++k) s += a[k] * (V)xv[k];
  }
  return s;
}

// a lane's part (entries g, g + GL, ...) of the sum by a group of GL lanes, the
// loads of up to six entries per lane in flight at once
template <class T, class V, int GL>
__device__ __forceinline__ V row_sumg(const unsigned* __restrict__ col, const V* __restrict__ val, int2 re, int g,
                                      const Gather<T>& x, unsigned lim) {
  constexpr int RU = 6;
  V s = V(0);
  for (int e = re.x + g; e < re.y; e += GL * RU) {
    unsigned cl[RU];
    V a[RU];
    T xv[RU];
#pragma unroll
    for (int k = 0; k < RU; ++k) {
      cl[k] = 0x7fffffffu;
      a[k] = V(0);
      if (e + GL * k < re.y) {
        cl[k] = col[e + GL * k];
        a[k] = val[e + GL * k];
      }
    }
#pragma unroll
    for (int k = 0; k < RU; ++k) xv[k] = e + GL * k < re.y && (cl[k] & 0x7fffffffu) < lim ? x(cl[k]) : T(0);
#pragma unroll
    for (int k = 0; k < RU; ++k) s += a[k] * (V)xv[k];
  }
  return s;
}

// The sparse rows of one colour in sweep s: the new values from the current
// iterate, into the buffer the colour's regular cells are written to.  On
// grid levels a group of 8 lanes takes a row (a row is a chain of dependent
// loads, so rows in flight matter, not lanes per row), counted from the other
// end of the grid than the regular cells so that small levels use different
// warps for the two; the sum is in a fixed lane order.  Inside CTA 0 a thread
// takes a row.
template <class T, class V>
__device__ __noinline__ void rb_rows_v(int lv, int colour, int s, bool zero, int cx) {
  const RLev<T>& L = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const int r0 = colour ? L.nr0 : 0, r1 = colour ? L.nr : L.nr0;
  const int ired = colour ? rb_red(s + 1) : rb_red(s), iblk = rb_black(s);
  const int out = colour ? rb_black(s + 1) : rb_red(s + 1);
  const Gather<T> x = rb_gather(L, ired, iblk);
  // zero: entries whose cells are still zero (all of them in the red pass, the black ones in the black pass)
  const unsigned lim = zero ? (colour ? (unsigned)L.H : 0u) : 0x80000000u;
  const V* dgp = (const V*)L.dinv;
  if (c.local) {
    for (int r = r0 + (int)threadIdx.x; r < r1; r += blockDim.x) {
      const unsigned cl = L.rs[r];
      unsigned pos;
      const T* b = rb_rhs(L, cl, pos);
      const V v = (V)b[pos] - (lim ? row_sum1<T, V>(L, L.re[r], x, lim) : V(0));
      L.x[cl >> 31][out][pos] = (T)(v * dgp[r]);
    }
    return;
  }
  const int g = threadIdx.x & 7;
  const unsigned gmask = 0xffu << (threadIdx.x & 24);
  const V* val = (const V*)L.val;
  const int rend = r0 + ((r1 - r0 + c.gst - 1) / c.gst) * c.gst;  // every lane of a warp runs the same trips
  for (int r = r0 + c.g0(); r < rend; r += c.gst) {
    const bool live = r < r1;
    const int2 re = live ? L.re[r] : make_int2(0, 0);
    const unsigned cl = live ? L.rs[r] : 0u;
    const V d = live ? dgp[r] : V(0);
    unsigned pos = 0;
    V bc = V(0), sum = V(0);
    if (live) {
      const T* b = rb_rhs(L, cl, pos);
      bc = (V)b[pos];
      if (lim) sum = row_sumg<T, V, 8>(L.col, val, re, g, x, lim);
    }
    for (int off = 4; off > 0; off >>= 1) sum += __shfl_xor_sync(gmask, sum, off);
    if (live && g == 0) L.x[cl >> 31][out][pos] = (T)((bc - sum) * d);
  }
}

// one colour of sweep s
template <class T>
__device__ __forceinline__ void rb_pass(int lv, int colour, int s, bool zero, int cx) {
  const RLev<T>& L = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const bool rows = colour ? L.nr > L.nr0 : L.nr0 > 0;
  // rows and regular cells are independent: every other warp takes the rows
  // last, so that their chains of dependent loads and the regular cells'
  // streams share the pass
  const bool late = L.dense && !c.local && ((threadIdx.x >> 5) & 1), none = zero && colour == 0;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    if ((h != 0) == late) {
      if (L.ngl[colour] && !none) rb_dense_list<T>(lv, colour, s, cx);
      if (!rows) continue;
      if (L.staged) rb_rows_v<T, T>(lv, colour, s, zero, cx);
      else rb_rows_v<T, double>(lv, colour, s, zero, cx);
    } else if (L.dense) {
      if (none) rb_dense_zero<T>(lv, s, cx);
      else rb_dense<T>(lv, colour, s, cx);
    }
  }
}

// sweeps s0 .. s1 - 1 of level l; zero: the first one starts from a zero
// iterate, which is not read
template <class T>
__device__ __forceinline__ bool rb_smooth(int lv, int s0, int s1, bool zero, int cx, int l) {
  for (int s = s0; s < s1; ++s)
    for (int colour = 0; colour < 2; ++colour) {
      rb_pass<T>(lv, colour, s, zero && s == s0, cx);
      if (!rsh<T>().c[cx].sync((l << 4) | (colour ? 3 : 1))) return false;
    }
  return true;
}

// zero iterate (V-cycles without pre-smoothing)
template <class T>
__device__ __noinline__ bool rb_zero(int lv, int cx, int l) {
  const RLev<T>& L = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const T z[4] = {T(0), T(0), T(0), T(0)};
  for (int t = c.i0(); t < L.nqt; t += c.st) {
    const unsigned w = reinterpret_cast<const unsigned*>(L.f[0])[t] | reinterpret_cast<const unsigned*>(L.f[1])[t];
    for (int p = 0; p < 2; ++p)
      if (w & (p ? 0x02020202u : 0x01010101u)) {
        st4(L.x[p][rb_red(0)] + 4 * (long long)t, z);
        st4(L.x[p][rb_black(0)] + 4 * (long long)t, z);
      }
  }
  return c.sync((l << 4) | 12);
}

// The restriction rows, a group of 8 lanes each (2D) or a warp (3D, where a
// row joins up to eight children's rows): everything a row needs is three
// dependent loads away (descriptor, entries and the children's right-hand
// sides, values), where walking the children's rows was seven or more; at
// about 0.7 us per load that reaches L2 this is what a small level's
// restriction costs (128^2 to 512^2 levels: 14.5 us before, 8.3 us now).
template <class T, class V, int GL>
__device__ __noinline__ void rb_restrict_special(int lf, int lv, int cx, int red, int black) {
  const RLev<T>& F = rsh<T>().H.L[lf];
  const RLev<T>& C = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const Gather<T> x = rb_gather(F, red, black);
  const int lane = threadIdx.x & (GL - 1), nch = 1 << F.D;
  const unsigned gmask = GL == 32 ? 0xffffffffu : 0xffu << (threadIdx.x & 24);
  const V scale = V(1) / V(nch);
  const V* val = (const V*)F.sval;
  const int g0 = GL == 32 ? c.g0() >> 2 : c.g0(), gst = GL == 32 ? c.gst >> 2 : c.gst;
  const int nend = ((F.nsp + gst - 1) / gst) * gst;
  const int s1 = F.hx, s2 = F.hx * F.n[1];
  for (int q = g0; q < nend; q += gst) {
    const bool live = q < F.nsp;
    const int4 d = live ? F.sd[q] : make_int4(0, 0, 0, 0);
    const int p = d.y >> 24;
    V acc = V(0);
    if (lane < nch && ((d.y >> (16 + lane)) & 1))
      acc = scale * (V)F.b[p][(lane ^ (lane >> 1) ^ (lane >> 2)) & 1][d.z + s1 * ((lane >> 1) & 1) + s2 * (lane >> 2)];
    acc -= row_sumg<T, V, GL>(F.scol, val, make_int2(d.x, d.x + (d.y & 0xffff)), lane, x, 0x80000000u);
    for (int off = GL / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(gmask, acc, off);
    if (live && lane == 0) {
      const int colour = d.w >= C.H;
      C.b[p][colour][colour ? d.w - C.H : d.w] = (T)acc;
    }
  }
}

// Residual of F after s sweeps, averaged over the children into C's
// right-hand side: four coarse cells per item, whose children of one colour
// are the groups at the same position of the fine rows.  full: black
// residuals too (no sweep has solved them).
template <class T>
__device__ __noinline__ void rb_restrict(int lf, int lv, int s, bool full, int cx) {
  const RLev<T>& F = rsh<T>().H.L[lf];
  const RLev<T>& C = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  if (F.nsp) {
    const int rd = rb_red(s), bk = rb_black(s);
    if (F.D == 3) {
      if (F.sstaged) rb_restrict_special<T, T, 32>(lf, lv, cx, rd, bk);
      else rb_restrict_special<T, double, 32>(lf, lv, cx, rd, bk);
    } else {
      if (F.sstaged) rb_restrict_special<T, T, 8>(lf, lv, cx, rd, bk);
      else rb_restrict_special<T, double, 8>(lf, lv, cx, rd, bk);
    }
  }
  if (!F.dense) return;
  const int rows = C.n[1] * C.n[2], items = rows * F.nq;
  const T scale = T(1) / T(1 << F.D);
  const unsigned* fr = reinterpret_cast<const unsigned*>(F.f[0]);
  const int ir = rb_red(s), ib = rb_black(s);
  for (int it = c.i0(); it < items; it += c.st) {
    const unsigned rc = fdiv((unsigned)it, F.dq);
    const int g = it - (int)rc * F.nq;
    const unsigned K = fdiv(rc, C.dn1);
    const int J = (int)(rc - K * (unsigned)C.n[1]);
    // coarse flags: cells 4g, 4g + 2 of one colour, 4g + 1, 4g + 3 of the other
    const int ce = (J + (int)K) & 1;
    const long long cp = (long long)rc * C.hx + 2 * g;
    const unsigned short fe = *reinterpret_cast<const unsigned short*>(C.f[ce] + cp);
    const unsigned short fo = *reinterpret_cast<const unsigned short*>(C.f[ce ^ 1] + cp);
    if (!((fe | fo) & 0x0303u)) continue;
    const int t00 = (2 * J + (F.D == 3 ? F.n[1] * 2 * (int)K : 0)) * F.nq + g;
    const bool whole = !full && F.wide;
#pragma unroll 1
    for (int p = 0; p <= F.two; ++p) {
      const unsigned pm = 0x0101u << p;
      if (!((fe | fo) & pm)) continue;
      T acc[4] = {T(0), T(0), T(0), T(0)};
      if (whole) {
        // two rows' loads at a time
#pragma unroll 1
        for (int hh = 0; hh < F.D - 1; ++hh) {
          QNb<T> v[2];
          T bb[2][4], xo[2][4];
          QPos q[2];
          unsigned m[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int t = t00 + u * F.nq + hh * F.nq * F.n[1];
            q[u] = QPos{t, 2 * J + u, F.D == 3 ? 2 * (int)K + hh : 0, 4 * g, (u + hh) & 1};
            m[u] = q[u].j < F.n[1] && q[u].k < F.n[2] ? regular_mask(fr[t], p) : 0u;
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (!m[u]) continue;
            quad_load_in(F, q[u], F.x[p][ib], v[u]);
            ld4(F.x[p][ir] + 4 * q[u].t, xo[u]);
            ld4(F.b[p][0] + 4 * q[u].t, bb[u]);
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (!m[u]) continue;
            T o[4];
            quad_apply_in(F, q[u], p, v[u], xo[u], o);
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] += (m[u] >> (8 * e)) & 1u ? bb[u][e] - o[e] : T(0);
          }
        }
      } else {
#pragma unroll 1
        for (int h = 0; h < (F.D == 3 ? 8 : 4); ++h) {
          const int j = 2 * J + (h & 1), k = F.D == 3 ? 2 * (int)K + ((h >> 1) & 1) : 0, colour = h >> (F.D - 1);
          if (j >= F.n[1] || k >= F.n[2] || (colour && !full)) continue;
          const int t = (j + F.n[1] * k) * F.nq + g;
          const unsigned m = regular_mask(reinterpret_cast<const unsigned*>(F.f[colour])[t], p);
          if (!m) continue;
          T o[4];
          quad_slow(F, t, colour, p, F.x[p][colour ? rb_red(s) : rb_black(s)],
                    F.x[p][colour ? rb_black(s) : rb_red(s)], F.b[p][colour], o);
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if ((m >> (8 * e)) & 1u) acc[e] += o[e];
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned f = ((e & 1) ? fo : fe) >> (8 * (e >> 1));
        if (((f >> p) & 1u) && !(f & R_SPC)) C.b[p][(e & 1) ? ce ^ 1 : ce][cp + (e >> 1)] = acc[e] * scale;
      }
    }
  }
}

// x += P e: (bi/tri)linear where every coarse cell of the interpolation has an
// unknown of the phase, the value of the cell above elsewhere (0 where that
// one has none).  An item is the eight cells of one position of a fine row,
// both colours; sF, sC: the sweeps done on the two levels.
template <class T>
__device__ __noinline__ void rb_prolong(int lf, int lv, int sF, int sC, int cx) {
  const RLev<T>& F = rsh<T>().H.L[lf];
  const RLev<T>& C = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const int cr = rb_red(sC), cb = rb_black(sC);
  const unsigned *f0 = reinterpret_cast<const unsigned*>(F.f[0]), *f1 = reinterpret_cast<const unsigned*>(F.f[1]);
  const int i0 = c.i0();
  unsigned n0 = i0 < F.nqt ? f0[i0] : 0u, n1 = i0 < F.nqt ? f1[i0] : 0u;  // flags one item ahead
  for (int t = i0; t < F.nqt; t += c.st) {
    const unsigned w0 = n0, w1 = n1;
    if (t + c.st < F.nqt) {
      n0 = f0[t + c.st];
      n1 = f1[t + c.st];
    }
    if (!((w0 | w1) & 0x03030303u)) continue;
    const QPos g = quad_pos(F, t, 0);  // red cells at i = 2 q + s
    const unsigned we = g.s ? w1 : w0, wo = g.s ? w0 : w1;  // flags of the even and the odd cells
    const int J = g.j >> 1, K = g.k >> 1;
    const int J2 = min(max(J + ((g.j & 1) ? 1 : -1), 0), C.n[1] - 1);
    const int K2 = min(max(K + ((g.k & 1) ? 1 : -1), 0), C.n[2] - 1);
#pragma unroll 1
    for (int p = 0; p <= F.two; ++p) {
      const unsigned pm = 0x01010101u << p;
      if (!((w0 | w1) & pm)) continue;
      T cs[6] = {T(0), T(0), T(0), T(0), T(0), T(0)}, home[4] = {T(0), T(0), T(0), T(0)};
      T *xe = F.x[p][g.s ? rb_black(sF) : rb_red(sF)] + 4 * (long long)t;
      T *xo = F.x[p][g.s ? rb_red(sF) : rb_black(sF)] + 4 * (long long)t;
      T ve[4], vo[4], a[4][6];
      ld4(xe, ve);
      ld4(xo, vo);
      // a neighbour outside the grid is replaced by the cell itself: no lane
      // that is interpolated linearly uses it, and every load goes out at once
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (h >= 2 && F.D == 2) continue;
        const int j = (h & 1) ? J2 : J, k = (h & 2) ? K2 : K;
        const int par = (j + k) & 1;  // colour of the coarse cells at even I
        const T* ae = C.x[p][par ? cb : cr];
        const T* ao = C.x[p][par ? cr : cb];
        const int cp = C.hx * (j + C.n[1] * k) + (g.q0 >> 1);
        ld2(ae + cp, a[h][1], a[h][3]);
        ld2(ao + cp, a[h][2], a[h][4]);
        a[h][0] = ao[g.q0 > 0 ? cp - 1 : cp];
        a[h][5] = ae[g.q0 + 4 < C.n[0] ? cp + 2 : cp];
      }
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (h >= 2 && F.D == 2) continue;
        const T wgt = ((h & 1) ? T(0.25) : T(0.75)) * (F.D == 3 ? ((h & 2) ? T(0.25) : T(0.75)) : T(1));
#pragma unroll
        for (int e = 0; e < 6; ++e) cs[e] += wgt * a[h][e];
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) home[e] = a[0][e + 1];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned a = we >> (8 * e), b = wo >> (8 * e);
        const T le = T(0.75) * cs[e + 1] + T(0.25) * cs[e], lo = T(0.75) * cs[e + 1] + T(0.25) * cs[e + 2];
        const T he = (a & (R_NOHOME0 << p)) ? T(0) : home[e], ho = (b & (R_NOHOME0 << p)) ? T(0) : home[e];
        if ((a >> p) & 1u) ve[e] += (a & (R_LIN0 << p)) ? le : he;
        if ((b >> p) & 1u) vo[e] += (b & (R_LIN0 << p)) ? lo : ho;
      }
      st4(xe, ve);
      st4(xo, vo);
    }
  }
}

// x = binv b on the bottom level: a warp per row, lanes over the columns
template <class T>
__device__ __noinline__ void rb_inverse(int lv, int cx) {
  const RHier<T>& H = rsh<T>().H;
  const RLev<T>& L = rsh<T>().H.L[lv];
  const RCtx& c = rsh<T>().c[cx];
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int w0 = c.local ? (int)(threadIdx.x >> 5) : (int)(threadIdx.x >> 5) * c.gsize + c.gcta;
  const int ws = c.local ? nw : nw * c.gsize;
  for (int i = w0; i < H.bm; i += ws) {
    const unsigned si = H.bslot[i];
    if (si == 0xffffffffu) continue;
    const T* row = H.binv + (long long)i * H.bm;
    T acc = T(0);
    for (int j = lane; j < H.bm; j += 32) {
      const unsigned sj = H.bslot[j];
      if (sj == 0xffffffffu) continue;
      unsigned pos;
      const T* b = rb_rhs(L, sj, pos);
      acc += row[j] * b[pos];
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) {
      const unsigned s = si & 0x7fffffffu;
      const int colour = s >= (unsigned)L.H;
      L.x[si >> 31][colour ? rb_black(0) : rb_red(0)][colour ? s - (unsigned)L.H : s] = acc;
    }
  }
}

// BiCGStab on a bottom level of at most 32 rows by one warp, a lane per row,
// from zero until |r| <= 1e-4 |b| (2-norms) or 16 iterations; vectors in
// registers, matrix-vector products through the level's own arrays.
template <class T, class V>
__device__ __noinline__ void rb_bicgstab_v(int lv) {
  const RLev<T>& L = rsh<T>().H.L[lv];
  const int lane = threadIdx.x & 31;
  const bool live = lane < L.nr;
  const unsigned cl = live ? L.rs[lane] : 0u;
  const int2 re = live ? L.re[lane] : make_int2(0, 0);
  const T di = live ? (T)((const V*)L.dinv)[lane] : T(1), d = rcp_rn(di);
  unsigned pos;
  const T* bp = rb_rhs(L, cl, pos);
  const bool blk = (cl & 0x7fffffffu) >= (unsigned)L.H;
  T* slot = L.x[cl >> 31][blk ? rb_black(0) : rb_red(0)] + pos;
  const Gather<T> x = rb_gather(L, rb_red(0), rb_black(0));
  auto dot = [](T a, T b) {
    T v = a * b;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  auto mul = [&](T y) {
    __syncwarp();
    if (live) *slot = y;
    __syncwarp();
    return live ? (T)(d * y + (T)row_sum1<T, V>(L, re, x, 0x80000000u)) : T(0);
  };
  const T b = live ? *bp : T(0);
  T r = b, pv = T(0), v = T(0), sol = T(0);
  const T r0 = b, bb = dot(b, b);
  T rho = T(1), alpha = T(1), omega = T(1);
#pragma unroll 1
  for (int it = 0; it < 16 && bb > T(0); ++it) {
    const T rho1 = dot(r0, r);
    if (rho1 == T(0) || omega == T(0)) break;
    pv = r + (rho1 / rho) * (alpha / omega) * (pv - omega * v);
    rho = rho1;
    // diagonal scaling: the cells' coefficients differ by the permittivities and cut fractions
    const T ph = pv * di;
    v = mul(ph);
    const T rv = dot(r0, v);
    if (rv == T(0)) break;
    alpha = rho / rv;
    const T sv = r - alpha * v;
    const T sh = sv * di;
    const T t = mul(sh);
    const T tt = dot(t, t);
    omega = tt > T(0) ? dot(t, sv) / tt : T(0);
    sol += alpha * ph + omega * sh;
    r = sv - omega * t;
    if (dot(r, r) <= T(1e-8) * bb) break;
  }
  __syncwarp();
  if (live) *slot = sol;
}

// sweeps done on a level when its correction is taken up by the finer one
template <class T>
__device__ __forceinline__ int rb_done(const RHier<T>& H, int l) {
  return l < H.nlev - 1 ? H.nu1[l] + H.nu2[l] : (H.bot ? 0 : H.bsweeps);
}

// level L (index l) down to N, the next one, and back up
template <class T>
__device__ __forceinline__ bool rb_down(int lv, int ln, int l, int cx) {
  const int nu = rsh<T>().H.nu1[l];
  if (nu == 0) {
    if (!rb_zero<T>(lv, cx, l)) return false;
  } else if (!rb_smooth<T>(lv, 0, nu, true, cx, l)) {
    return false;
  }
  rb_restrict<T>(lv, ln, nu, nu == 0, cx);
  return rsh<T>().c[cx].sync((l << 4) | 6);
}
template <class T>
__device__ __forceinline__ bool rb_up(int lv, int ln, int l, int cx) {
  const RHier<T>& H = rsh<T>().H;
  const int nu = H.nu1[l];
  rb_prolong<T>(lv, ln, nu, rb_done(H, l + 1), cx);
  if (!rsh<T>().c[cx].sync((l << 4) | 7)) return false;
  return rb_smooth<T>(lv, nu, nu + H.nu2[l], false, cx, l);
}

__device__ __forceinline__ void copy_words(void* dst, const void* src, long long bytes) {
  const int* s = (const int*)src;
  int* d = (int*)dst;
  for (long long i = threadIdx.x; i < bytes / 4; i += blockDim.x) d[i] = s[i];
}

// levels lc.. inside CTA 0; g: level lc as the grid sees it
template <class T>
__device__ __noinline__ void rb_coarse() {
  const RHier<T>& H = rsh<T>().H;
  const RLev<T>&s = H.L[H.lc], &g = H.L[RMAX];
  if (H.smem) {
    for (int p = 0; p <= s.two; ++p) {
      const int o = p ? s.p1o : 0, n = p ? s.p1n : s.H;
      for (int q = 0; q < 2; ++q) copy_words(s.b[p][q] + o, g.b[p][q] + o, (long long)n * sizeof(T));
    }
    __syncthreads();
  }
#pragma unroll 1
  for (int l = H.lc; l < H.nlev - 1; ++l) rb_down<T>(l, l + 1, l, 1);
  const int lb = H.nlev - 1;
  if (H.bot == 0) {
    rb_smooth<T>(lb, 0, H.bsweeps, true, 1, lb);
  } else {
    if (H.bot == 1) rb_inverse<T>(lb, 1);
    else if (threadIdx.x < 32) {
      if (H.L[lb].staged) rb_bicgstab_v<T, T>(lb);
      else rb_bicgstab_v<T, double>(lb);
    }
    rsh<T>().c[1].sync((lb << 4) | 9);
  }
#pragma unroll 1
  for (int l = H.nlev - 2; l >= H.lc; --l) rb_up<T>(l, l + 1, l, 1);
  if (H.smem) {
    const int d = rb_done(H, H.lc);
    for (int p = 0; p <= s.two; ++p) {
      const int o = p ? s.p1o : 0, n = p ? s.p1n : s.H;
      copy_words(g.x[p][rb_red(d)] + o, s.x[p][rb_red(d)] + o, (long long)n * sizeof(T));
      copy_words(g.x[p][rb_black(d)] + o, s.x[p][rb_black(d)] + o, (long long)n * sizeof(T));
    }
  }
}

// one V-cycle from zero: level 0's right-hand side in its b, the result in
// its x after rb_done(H, 0) sweeps
template <class T>
__device__ __noinline__ bool rb_vcycle() {
  const RHier<T>& H = rsh<T>().H;
#pragma unroll 1
  for (int l = 0; l < H.lc; ++l)
    if (!rb_down<T>(l, l + 1 == H.lc ? RMAX : l + 1, l, 0)) return false;
  if (H.bot == 1 && !H.smem) {  // the inverse applied by the whole grid
    rb_inverse<T>(RMAX, 0);
    if (!rsh<T>().c[0].sync(((H.nlev - 1) << 4) | 9)) return false;
  } else {
    if (rsh<T>().c[0].gcta == 0) rb_coarse<T>();
    if (!rsh<T>().c[0].sync((15 << 4) | 8)) return false;
  }
#pragma unroll 1
  for (int l = H.lc - 1; l >= 0; --l)
    if (!rb_up<T>(l, l + 1 == H.lc ? RMAX : l + 1, l, 0)) return false;
  return true;
}


// ------------------------------------------------------------ the FP64 outer loop

// max over non-negative doubles by their bit patterns (NaN passed over, as fmax does)
__device__ __forceinline__ void bits_max(unsigned long long& m, double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  if (b > m && b <= 0x7ff0000000000000ull) m = b;
}

// The unit of a mixed solve.  The Krylov sums multiply FP32 residuals: below about
// 1e-20 these products vanish, above 1e17 they overflow, and data in SI units
// reach both.  Where max|b| is outside 2^-10 .. 2^50, phi and b are therefore
// divided by 2^es, the power of two under max|b|, for the solve; that is exact, so
// it takes the same steps in every unit.  Inside that range, where a residual 13
// digits under max|b| still has its square in FP32's range, es is 0.  Where max|r|
// leaves 2^-56 .. 2^50 units (a guess far from the solution), es is chosen anew
// from it; the directions kept stay in the unit they were formed in, since z and A
// z scale alike.  FP64 V-cycles have the range as they are.  (A unit in the phases
// themselves, a factor on every residual and correction, cost every solve 0.5 to 2%,
// and as builds of their own the phases beside them 1% at 384^3.)
constexpr int ES_LO = -56, ES_MIN = -10, ES_HI = 50;
__device__ __forceinline__ int exponent_of(double v) {
  const int e = ((__double2hiint(v) >> 20) & 0x7ff) - 1023;
  return max(-900, min(900, e));
}
__device__ __forceinline__ int unit_of(double v) {
  const int e = exponent_of(v);
  return e >= ES_MIN && e <= ES_HI ? 0 : e;
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// phi and b times 2^e
template <class T>
__device__ __noinline__ bool rb_rescale(int e) {
  const Op<double>& F = rsh<T>().F;
  const RCtx& G = rsh<T>().c[0];
  const double u = pow2(e / 2), v = pow2(e - e / 2);  // e may be twice what an exponent holds
  for (int p = 0; p < 2; ++p) {
    if (!F.x[p]) continue;
    for (long long c = G.i0(); c < F.ncell; c += G.st) {
      F.x[p][c] = F.x[p][c] * u * v;
      F.b[p][c] = F.b[p][c] * u * v;
    }
  }
  return G.sync((14 << 4) | 10);
}

// FP64 residual of the finest level into level 0's right-hand side (rounded
// to T) and its max norm (in the caller's unit); eight cells of an x row per item,
// seven FP64 operations each (GB300 issues about two FP64 operations per clock and
// SM, which bounds the pass from 256^2 cells up).
template <class T>
__device__ __noinline__ bool rb_resid64(unsigned long long* norm) {
  const RHier<T>& H = rsh<T>().H;
  const RLev<T>& L = H.L[H.lc == 0 ? RMAX : 0];
  const Op<double>& F = rsh<T>().F;
  const RCtx& G = rsh<T>().c[0];
  unsigned long long mx = 0ull;
  {
    const int g = threadIdx.x & 7;
    const unsigned gmask = 0xffu << (threadIdx.x & 24);
    const int rend = ((L.nr + G.gst - 1) / G.gst) * G.gst;
    for (int r = G.g0(); r < rend; r += G.gst) {
      const bool live = r < L.nr;
      const int2 re = live ? L.re[r] : make_int2(0, 0);
      const unsigned cl = live ? L.rs[r] : 0u;
      const int p = (int)(cl >> 31);
      double s = 0.0, bc = 0.0, xc = 0.0, d = 0.0;
      if (live) {
        const int c = H.rnat[r];
        d = H.rdiag[r];
        bc = F.b[p][c];
        xc = F.x[p][c];
        for (int e = re.x + g; e < re.y; e += 32) {
          unsigned ce[4];
          double a[4], xv[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            ce[k] = 0u;
            a[k] = 0.0;
            if (e + 8 * k < re.y) {
              ce[k] = (unsigned)H.ncol[e + 8 * k];
              a[k] = H.rval[e + 8 * k];
            }
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) xv[k] = e + 8 * k < re.y ? F.x[ce[k] >> 30][ce[k] & 0x3fffffffu] : 0.0;
#pragma unroll
          for (int k = 0; k < 4; ++k) s += a[k] * xv[k];
        }
      }
      for (int off = 4; off > 0; off >>= 1) s += __shfl_xor_sync(gmask, s, off);
      if (live && g == 0) {
        const double v = (bc - s) - d * xc;
        unsigned pos;
        T* b = rb_rhs(L, cl, pos);
        b[pos] = (T)v;
        bits_max(mx, v);
      }
    }
  }
  const int n0 = F.n[0], n1 = F.n[1], n2 = F.D == 3 ? F.n[2] : 1;
  const long long sy = n0, sz = (long long)n0 * n1;
  for (int t = G.i0(); t < L.nqt; t += G.st) {
    const unsigned w0 = reinterpret_cast<const unsigned*>(L.f[0])[t], w1 = reinterpret_cast<const unsigned*>(L.f[1])[t];
    if (!((w0 | w1) & 0x03030303u)) continue;
    const QPos g = quad_pos(L, t, 0);
    const unsigned we = g.s ? w1 : w0, wo = g.s ? w0 : w1;
    const long long nb = ((long long)g.j + (long long)n1 * g.k) * n0 + 2 * g.q0;
#pragma unroll 1
    for (int p = 0; p <= L.two; ++p) {
      const unsigned me = regular_mask(we, p), mo = regular_mask(wo, p);
      if (!(me | mo)) continue;
      const double* x = F.x[p] + nb;
      double c[8], s[8];
      ld4(x, c);
      ld4(x + 4, c + 4);
      const double xl = g.q0 > 0 ? x[-1] : F.w3[0] * c[1];
      const double xr = 2 * g.q0 + 8 < n0 ? x[8] : F.w3[1] * c[6];
      double d0 = (double)(2 * F.D) + F.lh[p];
      double dl = d0, dr = d0;
#pragma unroll
      for (int e = 0; e < 8; ++e) s[e] = (e ? c[e ? e - 1 : 0] : xl) + (e < 7 ? c[e < 7 ? e + 1 : 7] : xr);
      double wd = 0.0;
#pragma unroll 1
      for (int a = 1; a < F.D; ++a) {
        const long long st = a == 1 ? sy : sz;
        const int i = a == 1 ? g.j : g.k, n = a == 1 ? n1 : n2;
        double u[8], v[8];
        if (i > 0) {
          ld4(x - st, u);
          ld4(x - st + 4, u + 4);
        }
        if (i < n - 1) {
          ld4(x + st, v);
          ld4(x + st + 4, v + 4);
        }
        if (i == 0) {
          wd += 3.0 * F.wr[2 * a] - 1.0;
#pragma unroll
          for (int e = 0; e < 8; ++e) u[e] = F.w3[2 * a] * v[e];
        }
        if (i == n - 1) {
          wd += 3.0 * F.wr[2 * a + 1] - 1.0;
#pragma unroll
          for (int e = 0; e < 8; ++e) v[e] = F.w3[2 * a + 1] * u[e];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] += u[e] + v[e];
      }
      if (wd != 0.0) d0 += wd;
      dl = g.q0 > 0 ? d0 : d0 + 3.0 * F.wr[0] - 1.0;
      dr = 2 * g.q0 + 8 < n0 ? d0 : d0 + 3.0 * F.wr[1] - 1.0;
      double bb[8];
      ld4(F.b[p] + nb, bb);
      ld4(F.b[p] + nb + 4, bb + 4);
      T oe[4], oo[4];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const double dg = e == 0 ? dl : (e == 7 ? dr : d0);
        const double r = bb[e] - F.ceps[p] * (dg * c[e] - s[e]);
        if (e & 1) oo[e >> 1] = (T)r;
        else oe[e >> 1] = (T)r;
        if (((e & 1) ? mo : me) >> (8 * (e >> 1)) & 1u) bits_max(mx, r);
      }
      quad_store(L.b[p][g.s] + 4 * (long long)t, me, oe);
      quad_store(L.b[p][g.s ^ 1] + 4 * (long long)t, mo, oo);
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
    mx = o > mx ? o : mx;
  }
  if ((threadIdx.x & 31) == 0 && mx) {
    if (rsh<T>().cur) mx = (unsigned long long)__double_as_longlong(__longlong_as_double((long long)mx) * pow2(rsh<T>().cur));
    atomicMax(norm, mx);
  }
  return G.sync((14 << 4) | 11);
}

// Krylov pass 1: q = A z of the V-cycle's result z (level 0 after sZ sweeps)
// into slot `slot`, and the partial sums of (r, q), (q, q) and, for the m
// directions before it, (q, q_i) and (r, q_i).  The sums' chunks depend on the level alone, not
// on the CTAs that take them, so a solve's results do not depend on its group.
template <class T>
__device__ __noinline__ void rb_kry1() {
  const RHier<T>& H = rsh<T>().H;
  const RLev<T>& L = H.L[H.lc == 0 ? RMAX : 0];
  const RCtx& G = rsh<T>().c[0];
  const int sZ = rb_done(H, 0), slot = rsh<T>().K.next, m = rsh<T>().K.count;
  T(*red)[KDOT] = rsh<T>().red;
  const int ir = rb_red(sZ), ib = rb_black(sZ);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int os[KH];
#pragma unroll
  for (int i = 0; i < KH - 1; ++i) os[i] = (slot + KH - 1 - i) % KH;
  const Gather<T> x = rb_gather(L, ir, ib);
  for (int ch = G.gcta; ch < H.kch; ch += G.gsize) {
    T acc[KDOT];
#pragma unroll
    for (int d = 0; d < KDOT; ++d) acc[d] = T(0);
    // the chunk's share of the sparse rows, a group of 8 lanes each
    {
      const int g = threadIdx.x & 7;
      const unsigned gmask = 0xffu << (threadIdx.x & 24);
      const int r1 = min((ch + 1) * H.krows, L.nr), ng = (int)(blockDim.x >> 3);
      for (int r0 = ch * H.krows; r0 < r1; r0 += ng) {
        const int r = r0 + (int)(threadIdx.x >> 3);
        const bool live = r < r1;
        const int2 re = live ? L.re[r] : make_int2(0, 0);
        const unsigned cl = live ? L.rs[r] : 0u;
        double s = row_sumg<T, double, 8>(L.col, H.rval, re, g, x, 0x80000000u);
        for (int off = 4; off > 0; off >>= 1) s += __shfl_xor_sync(gmask, s, off);
        if (live && g == 0) {
          unsigned pos;
          const T* b = rb_rhs(L, cl, pos);
          const int colour = (cl & 0x7fffffffu) >= (unsigned)L.H, p = (int)(cl >> 31);
          const T q = (T)(s + H.rdiag[r] * (double)x(cl));
          H.kq[slot][p][colour][pos] = q;
          const T rv = b[pos];
          acc[0] += rv * q;
          acc[1] += q * q;
#pragma unroll
          for (int i = 0; i < KH - 1; ++i)
            if (i < m) {
              const T qi = H.kq[os[i]][p][colour][pos];
              acc[2 + i] += q * qi;
              acc[KH + 1 + i] += rv * qi;
            }
        }
      }
    }
    const int t1 = min((ch + 1) * H.kcs, L.nqt);
    for (int t = ch * H.kcs + (int)threadIdx.x; t < t1; t += (int)blockDim.x) {
      const unsigned w[2] = {reinterpret_cast<const unsigned*>(L.f[0])[t], reinterpret_cast<const unsigned*>(L.f[1])[t]};
#pragma unroll 1
      for (int pc = 0; pc < 2 * (L.two + 1); ++pc) {
        const int p = pc >> 1, colour = pc & 1;
        const unsigned mk = regular_mask(colour ? w[1] : w[0], p);
        if (!mk) continue;
        const QPos g = quad_pos(L, t, colour);
        const T *xn = L.x[p][colour ? ir : ib], *xw = L.x[p][colour ? ib : ir];
        T q[4], rr[4], qi[KH - 1][4];
        ld4(L.b[p][colour] + 4 * t, rr);
#pragma unroll
        for (int i = 0; i < KH - 1; ++i)
          if (i < m) ld4(H.kq[os[i]][p][colour] + 4 * t, qi[i]);
        if (L.wide) {
          QNb<T> v;
          T xo[4];
          quad_load_in(L, g, xn, v);
          ld4(xw + 4 * t, xo);
          quad_apply_in(L, g, p, v, xo, q);
        } else {
          T os[4];
          quad_slow(L, t, colour, p, xn, xw, (const T*)nullptr, os);
#pragma unroll
          for (int e = 0; e < 4; ++e) q[e] = os[e];
        }
        quad_store(H.kq[slot][p][colour] + 4 * t, mk, q);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!((mk >> (8 * e)) & 1u)) q[e] = T(0);
          const T re = (mk >> (8 * e)) & 1u ? rr[e] : T(0);
          acc[0] += re * q[e];
          acc[1] += q[e] * q[e];
#pragma unroll
          for (int i = 0; i < KH - 1; ++i)
            if (i < m) {
              const T v = (mk >> (8 * e)) & 1u ? qi[i][e] : T(0);
              acc[2 + i] += q[e] * v;
              acc[KH + 1 + i] += re * v;
            }
        }
      }
    }
#pragma unroll
    for (int d = 0; d < KDOT; ++d) {
      T a = acc[d];
      for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
      if (lane == 0) red[wid][d] = a;
    }
    __syncthreads();
    if (threadIdx.x < KDOT) {
      double t = 0.0;
      for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += (double)red[k][threadIdx.x];
      H.kpart[(long long)ch * KDOT + threadIdx.x] = t;
    }
    __syncthreads();
  }
}

// The sums of pass 1 in a fixed order, then the step: the combination of the
// new and the kept directions that minimises |r - sum c q| (2-norm), by the
// normal equations.  The directions stay as they were formed, q = A z each:
// made orthogonal one after the other (as in GCR), their FP32 rounding errors
// pass from one to the next and grow, since successive corrections are nearly
// parallel, until the step no longer belongs to the residual (seen from
// 1e-10 of max|b| on).  c[i]: direction i before the new one, c[KH - 1]: the new one.
__device__ __forceinline__ void rb_kry_coeff(const double* part, int nch, int m, KryState& K, double* dots, double* c) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (wid < KDOT) {
    double s = 0.0;
    for (int k = lane; k < nch; k += 32) s += __ldcg(part + (long long)k * KDOT + wid);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) dots[wid] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = K.next;
    int sl[KH];
    K.g[nw][nw] = dots[1];
    sl[0] = nw;
    for (int i = 0; i < m; ++i) {
      sl[1 + i] = (nw + KH - 1 - i) % KH;
      K.g[nw][sl[1 + i]] = K.g[sl[1 + i]][nw] = dots[2 + i];
    }
    // scaled to a unit diagonal and factored in FP32, newest first: one
    // thread's FP64 chain would cost microseconds, and the step needs no more
    // digits than the sums have; a direction that depends on the ones before it
    // is left out
    float A[KH][KH], y[KH];
    int use[KH], nu = 0;
#pragma unroll
    for (int i = 0; i < KH; ++i) c[i] = 0.0;
    const double s0 = dots[1] > 0.0 ? rsqrt(dots[1]) : 0.0;
    K.rn[nw] = s0;
    for (int i = 0; i <= m; ++i) {
      const double si = K.rn[sl[i]];
      if (!(si > 0.0)) continue;
      float t[KH], p = 1.0f;
      for (int k = 0; k < nu; ++k) {
        float v = (float)(K.g[sl[i]][sl[use[k]]] * si * K.rn[sl[use[k]]]);
        for (int q = 0; q < k; ++q) v -= t[q] * A[k][q];
        t[k] = v / A[k][k];
        p -= t[k] * t[k];
      }
      if (!(p > 1e-5f)) continue;
      for (int k = 0; k < nu; ++k) A[nu][k] = t[k];
      A[nu][nu] = sqrtf(p);
      // right-hand side in units of |r|-like scale: divided by this direction's norm and the newest one's
      float v = (float)((i == 0 ? dots[0] : dots[KH + i]) * si * s0);
      for (int q = 0; q < nu; ++q) v -= A[nu][q] * y[q];
      y[nu] = v / A[nu][nu];
      use[nu++] = i;
    }
    bool fin = nu > 0 && use[0] == 0;
    for (int k = nu - 1; k >= 0; --k) {
      float v = y[k];
      for (int q = k + 1; q < nu; ++q) v -= A[q][k] * y[q];
      y[k] = v / A[k][k];
    }
    for (int k = 0; k < nu; ++k) {
      // back to the directions' own units: times |q_new| / |q_k|
      const double x = (double)y[k] * (dots[1] * s0) * K.rn[sl[use[k]]];
      fin = fin && fabs(x) < 1e3;
      c[use[k] ? use[k] - 1 : KH - 1] = x;
    }
    if (!fin) {
      for (int i = 0; i < KH; ++i) c[i] = 0.0;
      c[KH - 1] = 1.0;  // the plain correction
    }
    K.count = min(m + 1, KH - 1);
    K.next = (nw + 1) % KH;
  }
  __syncthreads();
}

// Krylov pass 2: phi += sum c z in FP64, z kept in slot `slot`, and r -= sum
// c q where another V-cycle follows before the next FP64 residual.  slot < 0:
// the plain correction, phi += z.
template <class T>
__device__ __noinline__ void rb_kry2(int slot, int m, bool upd_r) {
  const RHier<T>& H = rsh<T>().H;
  const RLev<T>& L = H.L[H.lc == 0 ? RMAX : 0];
  const Op<double>& F = rsh<T>().F;
  const RCtx& G = rsh<T>().c[0];
  const int sZ = rb_done(H, 0);
  const double* c = rsh<T>().coef;
  const int ir = rb_red(sZ), ib = rb_black(sZ);
  const int n0 = F.n[0], n1 = F.n[1];
  double cc[KH - 1];
  int os[KH - 1];
#pragma unroll
  for (int i = 0; i < KH - 1; ++i) {
    cc[i] = i < m ? c[i] : 0.0;
    os[i] = (slot + KH - 1 - i) % KH;
  }
  const double cn = slot < 0 ? 1.0 : c[KH - 1];
  for (int t = G.i0(); t < L.nqt; t += G.st) {
    const unsigned w[2] = {reinterpret_cast<const unsigned*>(L.f[0])[t], reinterpret_cast<const unsigned*>(L.f[1])[t]};
    if (!((w[0] | w[1]) & 0x03030303u)) continue;
    const QPos g = quad_pos(L, t, 0);
    const long long o4 = 4 * (long long)t;
#pragma unroll 1
    for (int p = 0; p <= L.two; ++p) {
      if (!((w[0] | w[1]) & (0x01010101u << p))) continue;
      double* ph = F.x[p] + ((long long)g.j + (long long)n1 * g.k) * n0 + 2 * g.q0;
      double f[8];
      ld4(ph, f);
      ld4(ph + 4, f + 4);
#pragma unroll
      for (int colour = 0; colour < 2; ++colour) {
        T z[4], s[4];
        ld4(L.x[p][colour ? ib : ir] + o4, z);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!((w[colour] >> (8 * e + p)) & 1u)) z[e] = T(0);
          s[e] = (T)cn * z[e];
        }
        if (slot >= 0) {
          st4(H.kz[slot][p][colour] + o4, z);
#pragma unroll
          for (int i = 0; i < KH - 1; ++i) {
            if (i >= m) continue;
            T zi[4];
            ld4(H.kz[os[i]][p][colour] + o4, zi);
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] += (T)cc[i] * zi[e];
          }
          if (upd_r) {
            T r[4], q[4];
            ld4(L.b[p][colour] + o4, r);
            ld4(H.kq[slot][p][colour] + o4, q);
#pragma unroll
            for (int e = 0; e < 4; ++e) r[e] -= (T)cn * q[e];
#pragma unroll
            for (int i = 0; i < KH - 1; ++i) {
              if (i >= m) continue;
              ld4(H.kq[os[i]][p][colour] + o4, q);
#pragma unroll
              for (int e = 0; e < 4; ++e) r[e] -= (T)cc[i] * q[e];
            }
            st4(L.b[p][colour] + o4, r);
          }
        }
        const int odd = g.s ^ colour;  // red cells are the even ones where s = 0
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (odd) f[2 * e + 1] += (double)s[e];
          else f[2 * e] += (double)s[e];
        }
      }
      st4(ph, f);
      st4(ph + 4, f + 4);
    }
  }
}

// The start of a launch: the hierarchy's description and the contexts into
// shared memory, and in CTA 0 the levels it keeps there (their flags, rows with
// entries in T and restriction rows, constant over the launch).
template <class T>
__device__ __noinline__ void rb_begin(const RHier<T>* __restrict__ Hg, const Barrier& B, int gcta, int gsize) {
  extern __shared__ __align__(128) unsigned char dyn[];
  RHier<T>& H = rsh<T>().H;
  copy_words(&H, Hg, sizeof(RHier<T>));
  if (threadIdx.x < 2) {
    RCtx& c = rsh<T>().c[threadIdx.x];
    c.local = threadIdx.x == 1;
    c.gcta = gcta;
    c.gsize = gsize;
    c.st = c.local ? (int)blockDim.x : gsize * (int)blockDim.x;
    c.gst = c.st >> 3;
    c.B = B;
    c.epoch = &rsh<T>().epoch;
    c.tn = &rsh<T>().tn;
    c.tr = nullptr;
    if (threadIdx.x == 0) rsh<T>().epoch = rsh<T>().tn = 0u;
  }
  __syncthreads();
  if (gcta == 0 && H.smem) {
    for (int l = H.lc; l < H.nlev; ++l) {
      const RLev<T>& g = Hg->L[l];
      for (int q = 0; q < 2; ++q) copy_words(dyn + H.off_f[l][q], g.f[q], g.H);
      // zeros, as the vectors in global memory start with
      for (int p = 0; p <= g.two; ++p)
        for (int k = 0; k < 5; ++k) {
          T* v = (T*)(dyn + (k < 3 ? H.off_x[l][p][k] : H.off_b[l][p][k - 3]));
          for (int i = threadIdx.x; i < g.H; i += blockDim.x) v[i] = T(0);
        }
      if (H.srows[l] & 1) {
        copy_words(dyn + H.off_re[l], g.re, 8ll * g.nr);
        copy_words(dyn + H.off_rs[l], g.rs, 4ll * g.nr);
        copy_words(dyn + H.off_col[l], g.col, 4ll * H.nnz[l]);
        T* v = (T*)(dyn + H.off_val[l]);
        for (int i = threadIdx.x; i < H.nnz[l]; i += blockDim.x) v[i] = (T)((const double*)g.val)[i];
        T* di = (T*)(dyn + H.off_di[l]);
        for (int i = threadIdx.x; i < g.nr; i += blockDim.x) di[i] = (T)((const double*)g.dinv)[i];
      }
      if (H.srows[l] & 2) {
        copy_words(dyn + H.off_sd[l], g.sd, 16ll * g.nsp);
        copy_words(dyn + H.off_sc[l], g.scol, 4ll * H.snnz[l]);
        T* sv = (T*)(dyn + H.off_sv[l]);
        for (int i = threadIdx.x; i < H.snnz[l]; i += blockDim.x) sv[i] = (T)((const double*)g.sval)[i];
      }
    }
    if ((int)threadIdx.x >= H.lc && (int)threadIdx.x < H.nlev) {
      const int l = threadIdx.x;
      RLev<T>& v = H.L[l];
      for (int p = 0; p <= v.two; ++p) {
        for (int k = 0; k < 3; ++k) v.x[p][k] = (T*)(dyn + H.off_x[l][p][k]);
        for (int k = 0; k < 2; ++k) v.b[p][k] = (T*)(dyn + H.off_b[l][p][k]);
      }
      for (int k = 0; k < 2; ++k) v.f[k] = dyn + H.off_f[l][k];
      if (H.srows[l] & 1) {
        v.re = (const int2*)(dyn + H.off_re[l]);
        v.rs = (const unsigned*)(dyn + H.off_rs[l]);
        v.col = (const unsigned*)(dyn + H.off_col[l]);
        v.val = dyn + H.off_val[l];
        v.dinv = dyn + H.off_di[l];
        v.staged = 1;
      }
      if (H.srows[l] & 2) {
        v.sd = (const int4*)(dyn + H.off_sd[l]);
        v.scol = (const unsigned*)(dyn + H.off_sc[l]);
        v.sval = dyn + H.off_sv[l];
        v.sstaged = 1;
      }
    }
  }
  __syncthreads();
}
template <class T>
__device__ __forceinline__ void rb_solve_group(const RHier<T>* __restrict__ Hg, const Op<double>* __restrict__ Fg,
                                               const SolveCtl& ctl, const Barrier& B, int gcta, int gsize) {
  RShared<T>& S = rsh<T>();
  const Op<double>& F = S.F;
  copy_words(&S.F, Fg, sizeof(Op<double>));
  copy_words(&S.K, Hg->kst, sizeof(KryState));
  rb_begin<T>(Hg, B, gcta, gsize);
  if (threadIdx.x == 0) {
    S.cur = 0;
    if (ctl.fresh) {
      S.K.count = S.K.next = 0;
      S.K.es = sizeof(T) == 4 ? unit_of(*ctl.bnorm) : 0;
    }
  }
  __syncthreads();
  const RCtx& G = S.c[0];
  const double bn = *ctl.bnorm;
  int it = 0, cycles = 0, status = 0;
  if (bn == 0.0) {  // b = 0: the solution is 0
    for (long long cc = G.i0(); cc < F.ncell; cc += G.st) {
      F.x[0][cc] = 0.0;
      if (F.x[1]) F.x[1][cc] = 0.0;
    }
  }
  // norms are read again where they are needed: little stays in registers across the phases
#pragma unroll 1
  for (; *ctl.bnorm != 0.0;) {
    if (!rb_resid64<T>(ctl.norms + it)) {
      status = 5;
      break;
    }
    const double r = load_norm(ctl.norms + it);
    if (r <= ctl.tol * *ctl.bnorm) break;
    if (cycles + ctl.inner > ctl.max_cycles || !(r == r) || r > 1e6 * load_norm(ctl.norms)) {
      status = 3;
      break;
    }
    if (ctl.max_iters && it >= ctl.max_iters) {  // resumable: stop at a V-cycle boundary
      status = 7;
      break;
    }
    bool ok = true;
    if (sizeof(T) == 4) {
      int want = S.K.es;  // the same in every CTA
      const int off = exponent_of(r) - want;
      if (off < ES_LO || off > ES_HI) want = unit_of(r);
      if (want != S.cur) {
        if (!rb_rescale<T>(S.cur - want)) {
          status = 5;
          break;
        }
        __syncthreads();
        if (threadIdx.x == 0) S.cur = S.K.es = want;
        __syncthreads();
        continue;  // the residual in the new unit
      }
    }
#pragma unroll 1
    for (int k = 0; k < ctl.inner && ok; ++k) {
      if (ctl.trace && threadIdx.x == 0 && G.gcta == 0) {  // trace the first V-cycle; this thread alone reads tr
        const bool on = it == 0 && k == 0;
        S.c[0].tr = S.c[1].tr = on ? ctl.trace : nullptr;
        if (on) ctl.trace[1 + S.tn++] = ((unsigned long long)0xfff << 48) | (now_ns() & 0xffffffffffffULL);
      }
      ok = rb_vcycle<T>();
      if (!ok) break;
      int slot = -1, m = 0;
      if (ctl.kry) {
        slot = S.K.next;
        m = S.K.count;
        rb_kry1<T>();
        ok = G.sync((14 << 4) | 14);
        if (!ok) break;
        rb_kry_coeff(S.H.kpart, S.H.kch, m, S.K, S.dots, S.coef);
      }
      rb_kry2<T>(slot, m, ctl.kry && k + 1 < ctl.inner);
      ok = G.sync((14 << 4) | 12);
    }
    if (threadIdx.x == 0) S.c[0].tr = S.c[1].tr = nullptr;
    if (!ok) {
      status = 5;
      break;
    }
    cycles += ctl.inner;
    ++it;
  }
  if (sizeof(T) == 4 && S.cur && status != 5) rb_rescale<T>(S.cur);
  if (gcta == 0 && threadIdx.x == 0) {
    if (ctl.trace) ctl.trace[0] = S.tn;
    const double r = bn == 0.0 ? 0.0 : load_norm(ctl.norms + it);
    ctl.norms[ctl.max_cycles + 1] = (unsigned long long)__double_as_longlong(r);  // final residual max
    ctl.out[0] = status;
    ctl.out[1] = it;
    ctl.out[2] = cycles;
    ctl.out[3] = it;
    *S.H.kst = S.K;
  }
}

template <class T>
__global__ void __launch_bounds__(PT, 1) k_rb_solve(const RHier<T>* __restrict__ Hg, const Op<double>* __restrict__ Fg,
                                                    SolveCtl ctl, Barrier B) {
  rb_solve_group<T>(Hg, Fg, ctl, B, (int)blockIdx.x, (int)gridDim.x);
}

// One V-cycle as a preconditioner: x = M b, or x += M b, on FP64 vectors in
// the plain layout (entries without an unknown are left alone).
template <class T>
__global__ void __launch_bounds__(PT, 1) k_rb_vcycle(const RHier<T>* __restrict__ Hg, long long ncell,
                                                     const double* __restrict__ b, double* __restrict__ x, int add,
                                                     Barrier B) {
  rb_begin<T>(Hg, B, (int)blockIdx.x, (int)gridDim.x);
  const RHier<T>& H = rsh<T>().H;
  const RCtx& G = rsh<T>().c[0];
  const RLev<T>& L = H.L[H.lc == 0 ? RMAX : 0];
  for (int t = G.i0(); t < L.nqt; t += G.st) {
    const unsigned w0 = reinterpret_cast<const unsigned*>(L.f[0])[t], w1 = reinterpret_cast<const unsigned*>(L.f[1])[t];
    const QPos g = quad_pos(L, t, 0);
    for (int p = 0; p <= L.two; ++p) {
      if (!((w0 | w1) & (0x01010101u << p))) continue;
      const double* src = b + p * ncell + ((long long)g.j + (long long)L.n[1] * g.k) * L.n[0] + 2 * g.q0;
      double v[8];
      ld4(src, v);
      ld4(src + 4, v + 4);
      const T e[4] = {(T)v[0], (T)v[2], (T)v[4], (T)v[6]}, o[4] = {(T)v[1], (T)v[3], (T)v[5], (T)v[7]};
      st4(L.b[p][g.s] + 4 * (long long)t, e);
      st4(L.b[p][g.s ^ 1] + 4 * (long long)t, o);
    }
  }
  if (!G.sync(0) || !rb_vcycle<T>()) return;
  const int d = rb_done(H, 0), ir = rb_red(d), ib = rb_black(d);
  for (int t = G.i0(); t < L.nqt; t += G.st) {
    const unsigned w[2] = {reinterpret_cast<const unsigned*>(L.f[0])[t], reinterpret_cast<const unsigned*>(L.f[1])[t]};
    const QPos g = quad_pos(L, t, 0);
    for (int p = 0; p <= L.two; ++p) {
      if (!((w[0] | w[1]) & (0x01010101u << p))) continue;
      double* dst = x + p * ncell + ((long long)g.j + (long long)L.n[1] * g.k) * L.n[0] + 2 * g.q0;
      double v[8];
      ld4(dst, v);
      ld4(dst + 4, v + 4);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        T z[4];
        ld4(L.x[p][c ? ib : ir] + 4 * (long long)t, z);
        const int odd = g.s ^ c;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!((w[c] >> (8 * e + p)) & 1u)) continue;
          double& q = odd ? v[2 * e + 1] : v[2 * e];
          q = (add ? q : 0.0) + (double)z[e];
        }
      }
      st4(dst, v);
      st4(dst + 4, v + 4);
    }
  }
}

// many independent solves in one cooperative launch (see BatchItem)
template <class T>
struct RBatchItem {
  const RHier<T>* H;
  const Op<double>* F;
  SolveCtl ctl;
  Barrier B;
  int start, size;
};
template <class T>
__global__ void __launch_bounds__(PT, 1) k_rb_batch(const RBatchItem<T>* __restrict__ items,
                                                    const int* __restrict__ cta_item) {
  const RBatchItem<T>& it = items[cta_item[blockIdx.x]];
  rb_solve_group<T>(it.H, it.F, it.ctl, it.B, (int)blockIdx.x - it.start, it.size);
}

// single phases of the finest level in the persistent kernel's grid shape, to
// time them: 0 a colour pass (its regular cells, listed groups and sparse rows),
// 1 the residual + restriction, 6 the prolongation
template <class T>
__global__ void __launch_bounds__(PT, 1) k_rb_phase(const RHier<T>* __restrict__ Hg, int kernel, int colour) {
  RHier<T>& H = rsh<T>().H;
  copy_words(&H.L[0], &Hg->L[0], sizeof(RLev<T>));
  copy_words(&H.L[1], &Hg->L[Hg->nlev > 1 ? 1 : 0], sizeof(RLev<T>));
  if (threadIdx.x == 0) {
    RCtx& c = rsh<T>().c[0];
    c.local = false;
    c.gcta = (int)blockIdx.x;
    c.gsize = (int)gridDim.x;
    c.st = (int)(gridDim.x * blockDim.x);
    c.gst = c.st >> 3;
  }
  __syncthreads();
  if (kernel == 0) rb_pass<T>(0, colour, 1, false, 0);
  else if (kernel == 1) rb_restrict<T>(0, 1, 1, false, 0);
  else rb_prolong<T>(0, 1, 1, rb_done(*Hg, 1), 0);
}
}  // namespace ebp
