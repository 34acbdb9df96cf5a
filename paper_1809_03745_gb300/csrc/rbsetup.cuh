// rbsetup.cuh -- set-up of the colour-split hierarchy of rbsolve.cuh: the
// algebraic levels below a coarsest grid that no dense inverse covers, and
// the split form of every level (flags, sparse rows, restriction lists).
#pragma once

#include "eb_internal.h"
#include "rbsolve.cuh"

namespace ebp {

// ------------------------------------------------------------ algebraic levels
//
// The geometric coarsening stops where a size is odd, where a coarse cell
// would hold two kinds of boundary, or at 8 cells.  Below that, cells are
// joined two by two per axis (an odd last one stays alone) and the operator is
// the Galerkin product with piecewise-constant transfer,
//   A_c = 2^-D P^T A P,  times 1/2 except for the Helmholtz shift.
// The factor is what rediscretisation has over that product away from
// boundaries (the flux between joined cells spans twice the distance), so a
// V-cycle with linear interpolation treats these levels like geometric ones.
// Every cell of such a level has a sparse row.

struct AlgView {
  int D, n[3];
  const uint8_t* flags;
  const int *irr_of_cell, *row_ptr, *col;
  const double *val, *diag;
  const double* sdiag;  // shift part of diag per row (algebraic levels), or null:
  const int* cut_of_cell;  // then kappa lam, kappa from the cut records
  const double* kappa;
  long long ncut;
  double ce[2], lam[2], w[6];
};

constexpr int ALG_MAXE = 64;  // entries of a row while it is summed; further ones join the diagonal

__global__ void k_alg_flags(AlgView f, int n0, int n1, int n2, uint8_t* flags) {
  const int c = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (c >= n0 * n1 * n2) return;
  const int I[3] = {c % n0, c / n0 % n1, c / (n0 * n1)};
  unsigned m = 0;
  for (int ch = 0; ch < (1 << f.D); ++ch) {
    const int i = 2 * I[0] + (ch & 1), j = 2 * I[1] + ((ch >> 1) & 1), k = f.D == 3 ? 2 * I[2] + (ch >> 2) : 0;
    if (i < f.n[0] && j < f.n[1] && k < f.n[2]) m |= f.flags[(long long)i + (long long)f.n[0] * (j + (long long)f.n[1] * k)] & 3u;
  }
  flags[c] = m ? (uint8_t)(m | F_IRR) : 0;
}

// one CTA: position of every true entry among the true ones of a run of
// blockDim entries (ascending), and their number
__device__ __forceinline__ int block_rank(bool v, int* total) {
  __shared__ int wsum[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  const unsigned b = __ballot_sync(0xffffffffu, v);
  __syncthreads();
  if (lane == 0) wsum[wid] = __popc(b);
  __syncthreads();
  int before = 0, all = 0;
  for (int k = 0; k < nw; ++k) {
    if (k < wid) before += wsum[k];
    all += wsum[k];
  }
  *total = all;
  return before + __popc(b & ((1u << lane) - 1u));
}

// cells with a row, red ones first; counts[0] of them, counts[1] red
__global__ void k_alg_order(const uint8_t* flags, int n0, int n1, int n, int* irr_cell, int* irr_of_cell, int* counts) {
  int at = 0;
  for (int colour = 0; colour < 2; ++colour) {
    for (int base = 0; base < n; base += (int)blockDim.x) {
      const int c = base + (int)threadIdx.x;
      const bool v = c < n && flags[c] && ((c % n0 + c / n0 % n1 + c / (n0 * n1)) & 1) == colour;
      int tot;
      const int r = block_rank(v, &tot);
      if (v) {
        irr_cell[at + r] = c;
        irr_of_cell[c] = at + r;
      }
      at += tot;
    }
    if (threadIdx.x == 0) counts[colour ? 0 : 1] = at;
  }
}

struct AlgRow {
  unsigned col[ALG_MAXE];
  double v[ALG_MAXE];
  int n;
  double dg, sd;
};
__device__ __forceinline__ void alg_add(AlgRow& R, unsigned self, unsigned col, double v) {
  if (col == self) {
    R.dg += v;
    return;
  }
  for (int k = 0; k < R.n; ++k)
    if (R.col[k] == col) {
      R.v[k] += v;
      return;
    }
  if (R.n < ALG_MAXE) {
    R.col[R.n] = col;
    R.v[R.n] = v;
    ++R.n;
  } else {
    R.dg += v;  // keeps the row sum
  }
}
// the Galerkin row of coarse cell C, phase p (columns phase << 30 | cell)
__device__ void alg_row(const AlgView& f, const int nc[3], int C, int p, AlgRow& R) {
  const int I[3] = {C % nc[0], C / nc[0] % nc[1], C / (nc[0] * nc[1])};
  auto up = [&](unsigned c) {  // coarse cell of a fine one
    const int i = (int)(c % (unsigned)f.n[0]) >> 1, r = (int)(c / (unsigned)f.n[0]);
    const int j = (r % f.n[1]) >> 1, k = f.D == 3 ? (r / f.n[1]) >> 1 : 0;
    return (unsigned)(i + nc[0] * (j + nc[1] * k));
  };
  const unsigned self = ((unsigned)p << 30) | (unsigned)C;
  R.n = 0;
  R.dg = R.sd = 0.0;
  for (int ch = 0; ch < (1 << f.D); ++ch) {
    const int c[3] = {2 * I[0] + (ch & 1), 2 * I[1] + ((ch >> 1) & 1), f.D == 3 ? 2 * I[2] + (ch >> 2) : 0};
    if (c[0] >= f.n[0] || c[1] >= f.n[1] || c[2] >= f.n[2]) continue;
    const long long cc = (long long)c[0] + (long long)f.n[0] * (c[1] + (long long)f.n[1] * c[2]);
    const unsigned fl = f.flags[cc];
    if (!((fl >> p) & 1u)) continue;
    if (fl & F_IRR) {
      const long long r = 2ll * f.irr_of_cell[cc] + p;
      double sd = 0.0;
      if (f.sdiag) sd = f.sdiag[r];
      else if (f.lam[p] != 0.0) {
        const int q = f.cut_of_cell[cc];
        sd = f.lam[p] * (q >= 0 ? f.kappa[p * f.ncut + q] : 1.0);
      }
      R.sd += sd;
      R.dg += f.diag[r] - sd;
      for (int e = f.row_ptr[r]; e < f.row_ptr[r + 1]; ++e) {
        const unsigned cl = (unsigned)f.col[e];
        alg_add(R, self, (cl & 0xc0000000u) | up(cl & 0x3fffffffu), f.val[e]);
      }
    } else {
      const double ce = f.ce[p];
      R.sd += f.lam[p];
      long long st = 1;
      for (int a = 0; a < f.D; ++a) {
        const unsigned lo = (unsigned)(cc - st), hi = (unsigned)(cc + st);
        for (int s = 0; s < 2; ++s) {
          const bool open = s ? c[a] < f.n[a] - 1 : c[a] > 0;
          if (open) {
            R.dg += ce;
            alg_add(R, self, ((unsigned)p << 30) | up(s ? hi : lo), -ce);
          } else if (f.w[2 * a + s] != 0.0) {
            R.dg += 3.0 * f.w[2 * a + s] * ce;
            alg_add(R, self, ((unsigned)p << 30) | up(s ? lo : hi), -f.w[2 * a + s] * ce / 3.0);
          }
        }
        st *= f.n[a];
      }
    }
  }
}
__global__ void k_alg_count(AlgView f, int n0, int n1, int n2, const int* irr_cell, const uint8_t* flags, int nirr,
                            int* counts) {
  const int r = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (r >= 2 * nirr) return;
  const int C = irr_cell[r >> 1], p = r & 1;
  const int nc[3] = {n0, n1, n2};
  int n = 0;
  if ((flags[C] >> p) & 1) {
    AlgRow R;
    alg_row(f, nc, C, p, R);
    n = R.n;
  }
  counts[r] = n;
}
// one CTA: row_ptr from the counts, in place (row_ptr[n] = total, also in *total)
__global__ void k_alg_scan(int* c, int n, int* total) {
  __shared__ int sh[1024];
  int run = 0;
  for (int base = 0; base < n; base += 1024) {
    const int i = base + (int)threadIdx.x;
    const int v = i < n ? c[i] : 0;
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      const int y = (int)threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
      __syncthreads();
      sh[threadIdx.x] += y;
      __syncthreads();
    }
    if (i < n) c[i] = run + sh[threadIdx.x] - v;
    run += sh[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    c[n] = run;
    *total = run;
  }
}
__global__ void k_alg_fill(AlgView f, int n0, int n1, int n2, const int* irr_cell, const uint8_t* flags, int nirr,
                           const int* row_ptr, int* col, double* val, double* diag, double* sdiag) {
  const int r = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (r >= 2 * nirr) return;
  const int C = irr_cell[r >> 1], p = r & 1;
  const int nc[3] = {n0, n1, n2};
  diag[r] = sdiag[r] = 0.0;
  if (!((flags[C] >> p) & 1)) return;
  AlgRow R;
  alg_row(f, nc, C, p, R);
  const double sc = 1.0 / (double)(1 << f.D);
  double off = 0.0;
  for (int k = 0; k < R.n; ++k) {
    col[row_ptr[r] + k] = (int)R.col[k];
    val[row_ptr[r] + k] = 0.5 * sc * R.v[k];
    off += fabs(0.5 * sc * R.v[k]);
  }
  double d = 0.5 * sc * R.dg + sc * R.sd;
  if (!(d > 0.0)) d = off > 0.0 ? off : 1.0;
  diag[r] = d;
  sdiag[r] = sc * R.sd;
}

static AlgView alg_view(const DevLevel& L) {
  AlgView f{};
  f.D = L.g.D;
  for (int k = 0; k < 3; ++k) f.n[k] = L.g.n[k];
  f.flags = L.flags;
  f.irr_of_cell = L.irr_of_cell;
  f.row_ptr = L.row_ptr;
  f.col = L.col;
  f.val = L.val;
  f.diag = L.diag;
  f.sdiag = L.sdiag;
  f.cut_of_cell = L.cut_of_cell;
  f.kappa = L.R.kappa;
  f.ncut = L.R.ncut;
  for (int p = 0; p < 2; ++p) {
    f.ce[p] = L.g.eps[p] / (L.g.h * L.g.h);
    f.lam[p] = L.g.lam[p];
  }
  for (int k = 0; k < 2 * L.g.D; ++k) {
    if (L.g.bc[k] == 1) f.w[k] = 1.0;
    else if (L.g.bc[k] == 2) f.w[k] = L.g.rob[k][0] / (L.g.rob[k][0] + L.g.rob[k][1] * 8.0 / (3.0 * L.g.h));
  }
  return f;
}

// the algebraic level below F
static eb_status build_alg_level(const DevLevel& F, DevLevel& C, long long* bytes, cudaStream_t s) {
  C.g = F.g;
  C.coarse = 1;
  for (int k = 0; k < 3; ++k) C.g.n[k] = k < F.g.D ? (F.g.n[k] + 1) / 2 : 1;
  C.g.h = 2.0 * F.g.h;
  C.g.ncell = (long long)C.g.n[0] * C.g.n[1] * C.g.n[2];
  const int n = (int)C.g.ncell, *nc = C.g.n;
  const AlgView f = alg_view(F);
  eb_status st = EB_OK;
  std::vector<void*> tmp;
  C.flags = (uint8_t*)dev_alloc(C.allocs, n, bytes, &st);
  C.irr_cell = (int*)dev_alloc(C.allocs, sizeof(int) * n, bytes, &st);
  C.irr_of_cell = (int*)dev_alloc(C.allocs, sizeof(int) * n, bytes, &st);
  C.row_ptr = (int*)dev_alloc(C.allocs, sizeof(int) * (2 * (size_t)n + 1), bytes, &st);
  C.diag = (double*)dev_alloc(C.allocs, sizeof(double) * 2 * n, bytes, &st);
  C.sdiag = (double*)dev_alloc(C.allocs, sizeof(double) * 2 * n, bytes, &st);
  int* cnt = (int*)dev_alloc(tmp, 4 * sizeof(int), nullptr, &st);
  int h[3] = {0, 0, 0};
  cudaError_t e = cudaSuccess;
  if (st == EB_OK) {
    k_alg_flags<<<(n + 255) / 256, 256, 0, s>>>(f, nc[0], nc[1], nc[2], C.flags);
    cudaMemsetAsync(C.irr_of_cell, 0xff, sizeof(int) * n, s);
    k_alg_order<<<1, 1024, 0, s>>>(C.flags, nc[0], nc[1], n, C.irr_cell, C.irr_of_cell, cnt);
    e = cudaMemcpyAsync(h, cnt, 2 * sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  if (st == EB_OK && e == cudaSuccess) {
    C.nirr = h[0];
    C.nirr_red = h[1];
    const int rows = 2 * h[0];
    if (rows) k_alg_count<<<(rows + 63) / 64, 64, 0, s>>>(f, nc[0], nc[1], nc[2], C.irr_cell, C.flags, h[0], C.row_ptr);
    k_alg_scan<<<1, 1024, 0, s>>>(C.row_ptr, rows, cnt + 2);
    e = cudaMemcpyAsync(h + 2, cnt + 2, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    C.nnz = h[2];
    C.col = (int*)dev_alloc(C.allocs, sizeof(int) * std::max<size_t>(C.nnz, 1), bytes, &st);
    C.val = (double*)dev_alloc(C.allocs, sizeof(double) * std::max<size_t>(C.nnz, 1), bytes, &st);
    if (st == EB_OK && e == cudaSuccess && rows)
      k_alg_fill<<<(rows + 63) / 64, 64, 0, s>>>(f, nc[0], nc[1], nc[2], C.irr_cell, C.flags, h[0], C.row_ptr, C.col,
                                                 C.val, C.diag, C.sdiag);
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  if (e == cudaSuccess && st == EB_OK) e = cudaStreamSynchronize(s);
  for (void* p : tmp) cudaFree(p);
  if (e != cudaSuccess) return cuda_fail(e, "algebraic level");
  return st;
}

// ------------------------------------------------------------ split form

struct SplitDim {
  int n0, n1, n2, hx, H;
};
__device__ __forceinline__ unsigned split_index(const SplitDim& d, unsigned c) {
  const int i = (int)(c % (unsigned)d.n0), r = (int)(c / (unsigned)d.n0);
  const int j = r % d.n1, k = r / d.n1;
  return (unsigned)(((i + j + k) & 1) * d.H + (i >> 1) + d.hx * r);
}

// split flags of a level from its cell flags, its children's (fl, may be
// null) and its parents' (cf, may be null); sets *hasreg where a cell is regular
__global__ void k_split_flags(int D, SplitDim d, const uint8_t* flags, const uint8_t* fl, int f0, int f1, int f2,
                              const uint8_t* cf, int c0, int c1, int c2, uint8_t* out, int* hasreg) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= (long long)d.n0 * d.n1 * d.n2) return;
  const int i = (int)(c % d.n0), r = (int)(c / d.n0), j = r % d.n1, k = r / d.n1;
  unsigned f = flags[c] & 7u;
  if ((f & 3u) && !(f & F_IRR) && *hasreg == 0) *hasreg = 1;
  if (fl) {
    for (int ch = 0; ch < (1 << D); ++ch) {
      const int a = 2 * i + (ch & 1), b = 2 * j + ((ch >> 1) & 1), e = D == 3 ? 2 * k + (ch >> 2) : 0;
      if (a < f0 && b < f1 && e < f2 && (fl[(long long)a + (long long)f0 * (b + (long long)f1 * e)] & F_IRR)) f |= R_SPC;
    }
  }
  if (cf) {
    const int I[3] = {i >> 1, j >> 1, D == 3 ? k >> 1 : 0};
    const int J[3] = {I[0] + ((i & 1) ? 1 : -1), I[1] + ((j & 1) ? 1 : -1), D == 3 ? I[2] + ((k & 1) ? 1 : -1) : 0};
    unsigned all = 3u, home = 0u;
    for (int q = 0; q < (1 << D); ++q) {
      const int a = (q & 1) ? J[0] : I[0], b = (q & 2) ? J[1] : I[1], e = (q & 4) ? J[2] : I[2];
      unsigned v = 0;
      if (a >= 0 && a < c0 && b >= 0 && b < c1 && e >= 0 && e < c2) v = cf[(long long)a + (long long)c0 * (b + (long long)c1 * e)] & 3u;
      all &= v;
      if (q == 0) home = v;
    }
    f |= all * R_LIN0;
    f |= ((~home) & 3u) * R_NOHOME0;
  }
  out[split_index(d, (unsigned)c)] = (uint8_t)f;
}

// one CTA: the rows of cells and phases with an unknown, in order (red first)
__global__ void k_split_rows(SplitDim d, const uint8_t* flags, const int* irr_cell, int nirr, int nirr_red,
                             const int* row_ptr, const double* diag, int2* re, unsigned* rs, double* dg, double* di, int* rnat,
                             int* counts) {
  int at = 0, red = 0;
  for (int base = 0; base < 2 * nirr; base += (int)blockDim.x) {
    const int r = base + (int)threadIdx.x;
    int c = 0;
    bool v = false;
    if (r < 2 * nirr) {
      c = irr_cell[r >> 1];
      v = ((flags[c] >> (r & 1)) & 1) && diag[r] != 0.0;
    }
    int tot, totr;
    const int k = block_rank(v, &tot);
    block_rank(v && (r >> 1) < nirr_red, &totr);
    if (v) {
      re[at + k] = make_int2(row_ptr[r], row_ptr[r + 1]);
      rs[at + k] = ((unsigned)(r & 1) << 31) | split_index(d, (unsigned)c);
      dg[at + k] = diag[r];
      di[at + k] = 1.0 / diag[r];
      rnat[at + k] = c;
    }
    at += tot;
    red += totr;
  }
  if (threadIdx.x == 0) {
    counts[0] = at;
    counts[1] = red;
  }
}
__global__ void k_split_cols(SplitDim d, const int* col, long long nnz, unsigned* out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nnz) return;
  const unsigned cl = (unsigned)col[e];
  out[e] = ((cl >> 30) << 31) | split_index(d, cl & 0x3fffffffu);
}
// The groups that a pass takes from a list (rb_dense_list): counted into
// n[colour], and written to out[colour] where that is given.
__global__ void k_split_list(int D, SplitDim d, const uint8_t* f, int* n, unsigned* out0, unsigned* out1) {
  const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x), colour = blockIdx.y, nq = d.hx / 4;
  if (t >= d.H / 4) return;
  const unsigned w = reinterpret_cast<const unsigned*>(f + (long long)colour * d.H)[t];
  const unsigned m0 = regular_mask(w, 0), m1 = regular_mask(w, 1);
  if (!(m0 | m1)) return;
  QPos g;
  const int row = t / nq;
  g.t = t;
  g.j = row % d.n1;
  g.k = row / d.n1;
  g.q0 = 4 * (t - row * nq);
  const bool inner = inner_group(D, d.n0, d.n1, d.n2, g);
  unsigned* out = colour ? out1 : out0;
  for (unsigned p = 0; p < 2; ++p) {
    if (!(p ? m1 : m0) || (inner && !(p && m0))) continue;
    const int i = atomicAdd(n + colour, 1);
    if (out) out[i] = (unsigned)t | p << 31;
  }
}
// Restriction rows: for every unknown of the coarse grid whose cell has a
// child with a sparse row, the mean of its children's residuals as one row
// over the fine level, the children's rows one after the other.  all: black
// regular children too (without a sweep their residuals are not zero).  The
// order of the rows does not matter (each writes its own unknown).
struct RestrictView {
  AlgView f;
  SplitDim fd, cd;
  const uint8_t* cf;
  int c0, c1, c2, all;
};
__device__ __forceinline__ bool child_cell(const RestrictView& v, int C, int ch, int c[3], long long& cell) {
  const int i = C % v.c0, j = C / v.c0 % v.c1, k = C / (v.c0 * v.c1);
  c[0] = 2 * i + (ch & 1);
  c[1] = 2 * j + ((ch >> 1) & 1);
  c[2] = v.f.D == 3 ? 2 * k + (ch >> 2) : 0;
  cell = (long long)c[0] + (long long)v.f.n[0] * (c[1] + (long long)v.f.n[1] * c[2]);
  return c[0] < v.f.n[0] && c[1] < v.f.n[1] && c[2] < v.f.n[2];
}
__global__ void k_restrict_count(RestrictView v, int2* list, int* len, int* counts) {
  const int C = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (C >= v.c0 * v.c1 * v.c2) return;
  bool any = false;
  int c[3];
  long long cell;
  for (int ch = 0; ch < (1 << v.f.D); ++ch)
    if (child_cell(v, C, ch, c, cell) && (v.f.flags[cell] & F_IRR)) any = true;
  if (!any) return;
  for (int p = 0; p < 2; ++p) {
    if (!((v.cf[C] >> p) & 1)) continue;
    int n = 0;
    for (int ch = 0; ch < (1 << v.f.D); ++ch) {
      if (!child_cell(v, C, ch, c, cell) || !((v.f.flags[cell] >> p) & 1)) continue;
      if (v.f.flags[cell] & F_IRR) {
        const long long r = 2ll * v.f.irr_of_cell[cell] + p;
        if (v.f.diag[r] != 0.0) n += v.f.row_ptr[r + 1] - v.f.row_ptr[r] + 1;
      } else if (v.all || !((c[0] + c[1] + c[2]) & 1)) {
        n += 1 + 2 * v.f.D;
      }
    }
    const int q = atomicAdd(counts + 2, 1);
    list[q] = make_int2(C, p);
    len[q] = n;
  }
}
// one CTA: exclusive sums of len[0..*n) in place, the total to *total
__global__ void k_restrict_scan(int* len, const int* n, int* total) {
  __shared__ int sh[1024];
  int run = 0;
  for (int base = 0; base < *n; base += 1024) {
    const int i = base + (int)threadIdx.x;
    const int v = i < *n ? len[i] : 0;
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      const int y = (int)threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
      __syncthreads();
      sh[threadIdx.x] += y;
      __syncthreads();
    }
    if (i < *n) len[i] = run + sh[threadIdx.x] - v;
    run += sh[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = run;
}
__global__ void k_restrict_fill(RestrictView v, const int2* list, const int* start, const int* n, int4* sd,
                                unsigned* scol, double* sval) {
  const int q = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (q >= *n) return;
  const int C = list[q].x, p = list[q].y;
  const double sc = 1.0 / (double)(1 << v.f.D);
  int at = start[q];
  unsigned mask = 0u;
  for (int ch = 0; ch < (1 << v.f.D); ++ch) {
    int c[3];
    long long cell;
    if (!child_cell(v, C, ch, c, cell) || !((v.f.flags[cell] >> p) & 1)) continue;
    const unsigned self = ((unsigned)p << 31) | split_index(v.fd, (unsigned)cell);
    if (v.f.flags[cell] & F_IRR) {
      const long long r = 2ll * v.f.irr_of_cell[cell] + p;
      if (v.f.diag[r] == 0.0) continue;
      mask |= 1u << ch;
      scol[at] = self;
      sval[at++] = sc * v.f.diag[r];
      for (int e = v.f.row_ptr[r]; e < v.f.row_ptr[r + 1]; ++e) {
        const unsigned cl = (unsigned)v.f.col[e];
        scol[at] = ((cl >> 30) << 31) | split_index(v.fd, cl & 0x3fffffffu);
        sval[at++] = sc * v.f.val[e];
      }
    } else if (v.all || !((c[0] + c[1] + c[2]) & 1)) {
      mask |= 1u << ch;
      const int me = at++;
      double dg = v.f.lam[p] / v.f.ce[p];
      long long st = 1;
      for (int a = 0; a < v.f.D; ++a) {
        for (int s = 0; s < 2; ++s) {
          const bool open = s ? c[a] < v.f.n[a] - 1 : c[a] > 0;
          const double w = v.f.w[2 * a + s];
          const long long nb = cell + ((s == 1) == open ? st : -st);
          scol[at] = ((unsigned)p << 31) | split_index(v.fd, (unsigned)nb);
          sval[at++] = -sc * v.f.ce[p] * (open ? 1.0 : w / 3.0);
          dg += open ? 1.0 : 3.0 * w;
        }
        st *= v.f.n[a];
      }
      scol[me] = self;
      sval[me] = sc * v.f.ce[p] * dg;
    }
  }
  const int i = C % v.c0, j = C / v.c0 % v.c1, k = C / (v.c0 * v.c1);
  const int base = i + v.fd.hx * (2 * j + v.f.n[1] * 2 * k);
  sd[q] = make_int4(start[q], (at - start[q]) | (int)(mask << 16) | (p << 24), base, (int)split_index(v.cd, (unsigned)C));
}
// first and last x row that holds a dielectric unknown
__global__ void k_phase1_rows(const uint8_t* flags, long long ncell, int n0, int* lohi) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool v = c < ncell && (flags[c] & 2);
  int lo = v ? (int)(c / n0) : 0x7fffffff, hi = v ? (int)(c / n0) : -1;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0 && hi >= 0) {
    atomicMin(lohi, lo);
    atomicMax(lohi + 1, hi);
  }
}
// inverse slots (phase * ncell + cell) in the split encoding
__global__ void k_split_slots(SplitDim d, const uint8_t* flags, int m, int ncell, unsigned* out) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= m) return;
  const int p = i / ncell, c = i - p * ncell;
  out[i] = ((flags[c] >> p) & 1) ? (((unsigned)p << 31) | split_index(d, (unsigned)c)) : 0xffffffffu;
}
}  // namespace ebp
