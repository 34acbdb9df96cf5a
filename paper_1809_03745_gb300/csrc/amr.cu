// amr.cu -- composite multi-level solve: nested ratio-2 refined boxes, one
// per level (Sec. 3.3.2 runs its multigrid over refined levels; the
// coarse-fine coupling of each pair of levels follows the refluxing of
// Sec. 3.3).
//
// Composite operator (the same reading as the oracle's):
//   * every box is a grid of its own whose coarse-fine (CF) sides are
//     homogeneous Neumann walls; the CF flux eps0 (ghost - phi_F)/h_f times the
//     fine aperture is added to each fine cell next to a CF side, the ghost by
//     quadratic tangential then quadratic normal Lagrange steps (fallbacks to
//     linear, then constant) precomputed per face at set-up;
//   * a coarse cell outside the box next to a CF side loses the coarse
//     operator's own flux through that face and gains minus the mean of the
//     fine fluxes through it (refluxing: exact conservation);
//   * cells under the next finer box carry no equation; where a stencil
//     reaches one, its value is the kappa-weighted mean of its children, which
//     are such means themselves under a still finer box;
//   * each box keeps one parent cell away from its parent's CF sides (proper
//     nesting), so every coarse cell across a CF face carries an equation.
// Solve: restarted FGMRES in FP64 on the composite system, right-
// preconditioned by one multiplicative FAC sweep from level 0 up: a level-0
// correction over the whole domain (the finer parts of the vector restricted
// under the boxes), added constant per parent on level 1, then on every finer
// level a correction of what remains there with zero Dirichlet data on its CF
// sides.  Every correction runs one V-cycle of the persistent multigrid
// kernel; dot products are summed in a fixed order (deterministic).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "eb_internal.h"

using namespace ebp;

namespace {

constexpr int TBA = 256;
int nb(long long n) { return (int)std::max<long long>(1, (n + TBA - 1) / TBA); }

struct BoxIdx {
  int D;
  int nc[3], nf[3], lo[3], hi[3];
};
// coarse cells under the box: the launch size of the passes that touch only them
long long box_cells(const BoxIdx& B) {
  return (long long)(B.hi[0] - B.lo[0]) * (B.hi[1] - B.lo[1]) * (B.hi[2] - B.lo[2]);
}

// cell indices of linear index c (grids of fewer than 2^32 cells: 32-bit
// divisions, several times cheaper than 64-bit ones in these memory-bound
// passes over every coarse cell)
__device__ __forceinline__ void ijk3(const int n[3], long long c, int I[3]) {
  const unsigned cu = (unsigned)c, n0 = (unsigned)n[0], n1 = (unsigned)n[1];
  const unsigned r = cu / n0;
  I[0] = (int)(cu - r * n0);
  const unsigned k = r / n1;
  I[1] = (int)(r - k * n1);
  I[2] = (int)k;
}
__device__ __forceinline__ long long lin3(const int n[3], const int I[3]) {
  return (long long)I[0] + (long long)n[0] * ((long long)I[1] + (long long)n[1] * I[2]);
}
__device__ __forceinline__ bool under_box(const BoxIdx& B, const int I[3]) {
  for (int k = 0; k < B.D; ++k)
    if (I[k] < B.lo[k] || I[k] >= B.hi[k]) return false;
  return true;
}
// the t-th coarse cell under the box (x fastest); false past the last one.
// Passes that only touch the cells under the box launch over these alone.
__device__ __forceinline__ bool box_cell(const BoxIdx& B, long long t, int I[3]) {
  const unsigned e0 = (unsigned)(B.hi[0] - B.lo[0]), e1 = (unsigned)(B.hi[1] - B.lo[1]);
  const unsigned e2 = (unsigned)(B.hi[2] - B.lo[2]);
  if (t >= (long long)e0 * e1 * e2) return false;
  const unsigned tu = (unsigned)t, r = tu / e0;
  I[0] = B.lo[0] + (int)(tu - r * e0);
  I[1] = B.lo[1] + (int)(r % e1);
  I[2] = B.lo[2] + (int)(r / e1);
  return true;
}

// coarse values under the box: kappa-weighted mean of the children with the phase
__global__ void k_avg_down(BoxIdx B, const uint8_t* cflags, const uint8_t* fflags, const double* kf, const double* pf,
                           double* pc, long long ncc, long long nff) {
  int I[3];
  if (!box_cell(B, (long long)blockIdx.x * blockDim.x + threadIdx.x, I)) return;
  const long long c = lin3(B.nc, I);
  for (int p = 0; p < 2; ++p) {
    if (!((cflags[c] >> p) & 1)) {
      pc[p * ncc + c] = 0.0;
      continue;
    }
    double num = 0.0, den = 0.0;
    for (int k = 0; k < (1 << B.D); ++k) {
      int F[3] = {0, 0, 0};
      for (int a = 0; a < B.D; ++a) F[a] = 2 * (I[a] - B.lo[a]) + ((k >> a) & 1);
      long long f = lin3(B.nf, F);
      if ((fflags[f] >> p) & 1) {
        double w = kf[p * nff + f];
        num += w * pf[p * nff + f];
        den += w;
      }
    }
    pc[p * ncc + c] = den > 0.0 ? num / den : 0.0;
  }
}

// alpha_f times the CF flux out of the fine cell, per fine CF face
__global__ void k_cf_flux(const CFFace* faces, long long nface, const double* pc, const double* pf, double eps0,
                          double hf, double* fl) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nface) return;
  const CFFace f = faces[t];
  double v = 0.0;
  if (f.al > 0.0) {
    double tv = 0.0;
    for (int k = 0; k < f.nc; ++k) tv += f.cw[k] * pc[f.cc[k]];
    double ghost = f.wf * pf[f.fcell] + f.wc * tv;
    if (f.f2 >= 0) ghost += f.wf2 * pf[f.f2];
    v = f.al * eps0 * (ghost - pf[f.fcell]) / hf;
  }
  fl[t] = v;
}

// fine rows of one CF side (one face per fine cell within a side)
__global__ void k_cf_fine_apply(const CFFace* faces, long long t0, long long t1, const double* fl, double hf,
                                double* rf) {  // hf < 0: the fluxes' share of A phi instead of b - A phi
  long long t = t0 + (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= t1) return;
  const CFFace& f = faces[t];
  if (f.al > 0.0) rf[f.fcell] += fl[t] / hf;
}

// coarse rows next to the box: take the coarse face flux out, put minus the
// mean fine flux in
__global__ void k_cf_coarse_apply(const CFCoarse* cf, long long n, const double* fl, const double* pc, long long ncc,
                                  double hc, int D, double sgn, double* rc) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const CFCoarse& c = cf[t];
  if (c.ccell < 0) return;
  double own = 0.0;
  for (int k = 0; k < c.n; ++k) {
    unsigned cl = (unsigned)c.col[k];
    own += c.w[k] * pc[(long long)(cl >> 30) * ncc + (cl & 0x3fffffffu)];
  }
  double fsum = 0.0;
  for (int k = 0; k < c.nfine; ++k) fsum += fl[c.fine[k]];
  rc[c.ccell] += sgn * (-own - fsum / (hc * (double)(1 << (D - 1))));
}

__global__ void k_zero_under(BoxIdx B, double* rc, long long ncc) {
  int I[3];
  if (!box_cell(B, (long long)blockIdx.x * blockDim.x + threadIdx.x, I)) return;
  const long long c = lin3(B.nc, I);
  rc[c] = rc[ncc + c] = 0.0;
}

// coarse correction right-hand side under the box: mean fine residual of the
// children carrying the phase
__global__ void k_restrict_under(BoxIdx B, const uint8_t* fflags, const double* rf, double* rc, long long ncc,
                                 long long nff) {
  int I[3];
  if (!box_cell(B, (long long)blockIdx.x * blockDim.x + threadIdx.x, I)) return;
  const long long c = lin3(B.nc, I);
  for (int p = 0; p < 2; ++p) {
    double s = 0.0;
    int m = 0;
    for (int k = 0; k < (1 << B.D); ++k) {
      int F[3] = {0, 0, 0};
      for (int a = 0; a < B.D; ++a) F[a] = 2 * (I[a] - B.lo[a]) + ((k >> a) & 1);
      long long f = lin3(B.nf, F);
      if ((fflags[f] >> p) & 1) {
        s += rf[p * nff + f];
        ++m;
      }
    }
    rc[p * ncc + c] = m ? s / m : 0.0;
  }
}

// pf = e_c of the parent where the fine cell has the phase
__global__ void k_prolong_const(BoxIdx B, const uint8_t* fflags, const double* ec, double* pf, long long ncc,
                                long long nff) {
  long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nff) return;
  const unsigned fl = fflags[f];
  if (!(fl & 3u)) return;
  int F[3];
  ijk3(B.nf, f, F);
  int I[3] = {0, 0, 0};
  for (int a = 0; a < B.D; ++a) I[a] = B.lo[a] + F[a] / 2;
  long long c = lin3(B.nc, I);
  for (int p = 0; p < 2; ++p)
    if ((fl >> p) & 1) pf[p * nff + f] = ec[p * ncc + c];
}
__global__ void k_absmax2(const uint8_t* flags, long long n, const double* v, unsigned long long* out) {
  long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double m = 0.0;
  if (c < n)
    for (int p = 0; p < 2; ++p)
      if ((flags[c] >> p) & 1) m = fmax(m, fabs(v[p * n + c]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0 && m > 0.0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// Composite vectors: one [2][n] array per level.  The entries that count are
// those of a level's own unknowns: `own` holds its flags with the cells under
// the next finer box cleared.  Entries without them (and all of the second
// phase's, where a group of four cells has none of it) are neither read nor
// written.  Sums go block by block into `part`, and one block adds those in a
// fixed order, so every dot product is deterministic.
constexpr int DOT_BLOCKS = 608;
constexpr int CV_MAXV = 14;
struct CVPtrs {
  const double* v[CV_MAXV];
  double a[CV_MAXV];
};
__global__ void k_own_flags(BoxIdx B, const uint8_t* flags, long long n, int coarse, uint8_t* own) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  unsigned f = flags[c] & 3u;
  if (f && coarse) {
    int I[3];
    ijk3(B.nc, c, I);
    if (under_box(B, I)) f = 0;
  }
  own[c] = (uint8_t)f;
}
__device__ __forceinline__ void ldq(const double* p, double v[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}
__device__ __forceinline__ void stq(double* p, const double v[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}
// the lanes of a group of four cells that carry phase p, as bits
__device__ __forceinline__ unsigned lanes4(unsigned w, int p) {
  const unsigned b = (w >> p) & 0x01010101u;
  return (b & 1u) | ((b >> 7) & 2u) | ((b >> 14) & 4u) | ((b >> 21) & 8u);
}
template <int NS>
__device__ __forceinline__ void block_sums(double (&acc)[NS], int m, double* part) {
  __shared__ double sh[NS][TBA / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    if (i >= m) continue;
    double a = acc[i];
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) sh[i][wid] = a;
  }
  __syncthreads();
  if ((int)threadIdx.x < m) {
    double t = 0.0;
    for (int k = 0; k < TBA / 32; ++k) t += sh[threadIdx.x][k];
    part[threadIdx.x * gridDim.x + blockIdx.x] = t;
  }
}
// (v_i, w) for i < m; *go = 0 skips the pass
template <int MAXM>
__global__ void __launch_bounds__(TBA) k_cv_mdot(const uint8_t* __restrict__ own, long long n, int m, CVPtrs V,
                                                 const double* __restrict__ w, const int* go, double* part) {
  if (go && !*go) return;
  double acc[MAXM];
#pragma unroll
  for (int i = 0; i < MAXM; ++i) acc[i] = 0.0;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; 4 * q < n; q += (long long)gridDim.x * blockDim.x) {
    const unsigned f = reinterpret_cast<const unsigned*>(own)[q];
    for (int p = 0; p < 2; ++p) {
      const unsigned ln = lanes4(f, p);
      if (!ln) continue;
      const long long c = p * n + 4 * q;
      double wv[4];
      ldq(w + c, wv);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (!((ln >> e) & 1u)) wv[e] = 0.0;
#pragma unroll
      for (int i = 0; i < MAXM; ++i) {
        if (i >= m) continue;
        double v[4];
        ldq(V.v[i] + c, v);
        if (ln != 15u) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (!((ln >> e) & 1u)) v[e] = 0.0;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i] += v[e] * wv[e];
      }
    }
  }
  block_sums<MAXM>(acc, m, part);
}
// w -= sum_i h_i v_i, and the block sums of the new (w, w); *go = 0 skips the pass
__global__ void __launch_bounds__(TBA) k_cv_maxpy_norm(const uint8_t* __restrict__ own, long long n, int m, CVPtrs V,
                                                       const double* __restrict__ h, double* __restrict__ w,
                                                       const int* go, double* part) {
  if (go && !*go) return;
  double acc[1] = {0.0};
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; 4 * q < n; q += (long long)gridDim.x * blockDim.x) {
    const unsigned f = reinterpret_cast<const unsigned*>(own)[q];
    for (int p = 0; p < 2; ++p) {
      const unsigned ln = lanes4(f, p);
      if (!ln) continue;
      const long long c = p * n + 4 * q;
      double t[4], t0[4];
      ldq(w + c, t);
#pragma unroll
      for (int e = 0; e < 4; ++e) t0[e] = t[e];
      for (int i = 0; i < m; ++i) {
        double v[4];
        ldq(V.v[i] + c, v);
        const double a = h[i];
#pragma unroll
        for (int e = 0; e < 4; ++e) t[e] -= a * v[e];
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (!((ln >> e) & 1u)) t[e] = t0[e];
        else acc[0] += t[e] * t[e];
      }
      stq(w + c, t);
    }
  }
  block_sums<1>(acc, 1, part);
}
// one block: the m sums over nlev levels' blocks, a warp each, in a fixed
// order; what follows from them (the Gram-Schmidt step's numbers) on thread 0:
//   0  out[0..m) = the sums (3: if *go)
//   1  out[0] = the new norm after the first pass; *go = the second one is
//      needed (the norm fell below 1/sqrt(2) of the old one, sqrt(in[m0]),
//      the criterion of Daniel, Gragg, Kaufman and Stewart)
//   2  out[0] = the norm after the second pass, if it ran (4: the norm)
__global__ void k_cv_finish(const double* part, int nlev, long long lstride, int m, int what, const double* in, int m0,
                            int* go, double* out) {
  if ((what == 2 || what == 3) && !*go) return;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wid >= m) return;
  double s = 0.0;
  for (int l = 0; l < nlev; ++l)
    for (int k = lane; k < DOT_BLOCKS; k += 32) s += part[l * lstride + (long long)wid * DOT_BLOCKS + k];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane) return;
  if (what == 0 || what == 3) {
    out[wid] = s;
    return;
  }
  const double w1 = sqrt(fmax(s, 0.0));
  out[0] = w1;
  if (what == 1) *go = w1 < sqrt(fmax(in[m0], 0.0)) * 0.70710678118654752440 ? 1 : 0;
}
// w *= 1 / *norm (left alone when it is not positive)
__global__ void k_cv_scale(const uint8_t* __restrict__ own, long long n, const double* norm, double* __restrict__ w) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (4 * q >= n) return;
  const double a = *norm;
  if (!(a > 0.0)) return;
  const double s = 1.0 / a;
  const unsigned f = reinterpret_cast<const unsigned*>(own)[q];
  for (int p = 0; p < 2; ++p) {
    if (!lanes4(f, p)) continue;
    double t[4];
    ldq(w + p * n + 4 * q, t);
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] *= s;
    stq(w + p * n + 4 * q, t);
  }
}
// x += sum_i a_i z_i on a level's unknowns (x: the caller's array)
__global__ void k_cv_update(const uint8_t* __restrict__ flags, long long n, int m, CVPtrs Z, double* __restrict__ x) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const unsigned f = flags[c];
  for (int p = 0; p < 2; ++p) {
    if (!((f >> p) & 1u)) continue;
    double t = x[p * n + c];
    for (int i = 0; i < m; ++i) t += Z.a[i] * Z.v[i][p * n + c];
    x[p * n + c] = t;
  }
}

// entries without an unknown of the caller's array = 0
__global__ void k_zero_absent(const uint8_t* __restrict__ flags, long long n, double* __restrict__ x) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const unsigned f = flags[c];
  if (!(f & 1u)) x[c] = 0.0;
  if (!(f & 2u)) x[n + c] = 0.0;
}

}  // namespace

constexpr int AMR_MAXL = EB_AMR_MAX_LEVELS;

// A composite vector: one [2][n_l] array per level (entries under the next
// finer box and without an unknown ignored)
struct CVec {
  double* v[AMR_MAXL] = {};
};

// One level: its grid as an operator (CF sides homogeneous Neumann) and, from
// level 1 on, as a correction grid (CF sides zero Dirichlet)
struct AmrLevel {
  eb_geom_desc d{}, d0{};
  eb_geom *G = nullptr, *G0 = nullptr;
  eb_poisson *P = nullptr, *P0 = nullptr;  // level 0: P0 == P
  long long n = 0;
  double h = 0.0;
  const uint8_t* flags = nullptr;  // finest-level flags of G (owned by G)
  uint8_t* own = nullptr;          // the same without the cells under the next box
  double *pc = nullptr;            // phi with the cells under the next box replaced by the finer means
  double *r = nullptr, *b0 = nullptr, *kap = nullptr;
};

// The coupling of levels l-1 (coarse) and l (fine), stored at index l
struct AmrPair {
  BoxIdx B{};
  CFBox cfb{};
  long long nface = 0, ncface = 0;
  CFFace* faces = nullptr;
  CFCoarse* cfaces = nullptr;
  double* fl = nullptr;
};

struct eb_amr {
  int D = 2, L = 2;
  AmrLevel lv[AMR_MAXL];
  AmrPair pr[AMR_MAXL];
  std::vector<eb_prim> prims;
  std::vector<eb_csg> nodes;
  eb_solver_opts o{};
  double eps0 = 1.0;
  int* d_status = nullptr;
  unsigned long long* d_norm = nullptr;
  // FGMRES work space (allocated at the first solve)
  std::vector<CVec> V, Z;
  double* d_part = nullptr;  // block sums
  double* d_h = nullptr;     // Gram-Schmidt numbers of the current step
  int* d_go = nullptr;
  double* h_h = nullptr;     // their copy (pinned)
  std::vector<cudaEvent_t> ev;  // pairs around the V-cycles of a solve
  std::vector<void*> allocs;
  long long bytes = 0;
  // persistent solve launches of the last composite solve, coarse [0] and
  // finer levels' [1] correction solvers: launches, kernel ms, V-cycles, FP64 outer iterations
  double kstat[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
};

static void amr_count(eb_amr* A, int which, int cyc, int outer, double ms) {
  A->kstat[which][0] += 1.0;
  A->kstat[which][1] += ms;
  A->kstat[which][2] += cyc;
  A->kstat[which][3] += outer;
}

static eb_status amr_fail(eb_amr* A, eb_status st) {
  eb_amr_destroy(A);
  return st;
}

extern "C" void eb_amr_destroy(eb_amr* A) {
  if (!A) return;
  cudaDeviceSynchronize();
  for (int l = 0; l < AMR_MAXL; ++l) {
    AmrLevel& v = A->lv[l];
    if (v.P0 != v.P) eb_poisson_destroy(v.P0);
    eb_poisson_destroy(v.P);
    eb_geom_destroy(v.G0);
    eb_geom_destroy(v.G);
  }
  for (void* p : A->allocs) cudaFree(p);
  for (cudaEvent_t e : A->ev) cudaEventDestroy(e);
  if (A->h_h) cudaFreeHost(A->h_h);
  delete A;
}

// is side s2 of axis k of the box of pair B a CF side (inside its parent grid)?
static bool cf_side(const BoxIdx& B, int k, int s2) { return s2 == 0 ? B.lo[k] > 0 : B.hi[k] < B.nc[k]; }

extern "C" eb_status eb_amr_setup_levels(const eb_geom_desc* desc, int n_levels, const int* box_lo,
                                         const int* box_hi, const eb_solver_opts* opts, void* stream,
                                         eb_amr** out) {
  if (!desc || !box_lo || !box_hi || !out) {
    set_error("null argument");
    return EB_ERR_INVALID;
  }
  *out = nullptr;
  if (n_levels < 2 || n_levels > AMR_MAXL) {
    set_error("a composite grid has 2 to " + std::to_string(AMR_MAXL) + " levels");
    return EB_ERR_INVALID;
  }
  if (desc->n_prims < 0 || desc->n_prims > EB_MAX_PRIMS || desc->n_nodes < 0 || desc->n_nodes > EB_MAX_NODES ||
      (desc->n_prims && !desc->prims) || (desc->n_nodes && !desc->nodes)) {
    set_error("invalid primitive or CSG node list");
    return EB_ERR_INVALID;
  }
  if (desc->dim < 2 || desc->dim > 3) {
    set_error("dimension must be 2 or 3");
    return EB_ERR_INVALID;
  }
  cudaStream_t s = (cudaStream_t)stream;
  eb_amr* A = new eb_amr();
  A->D = desc->dim;
  A->L = n_levels;
  const int D = A->D, L = A->L;
  if (opts) A->o = *opts;
  else eb_solver_opts_default(&A->o);
  A->o.launch_mode = 0;
  A->prims.assign(desc->prims, desc->prims + desc->n_prims);
  A->nodes.assign(desc->nodes, desc->nodes + desc->n_nodes);
  A->lv[0].d = *desc;
  A->lv[0].d.prims = A->prims.data();
  A->lv[0].d.nodes = A->nodes.data();
  // level descriptions: each box over cells [lo, hi) of its parent's grid
  for (int l = 1; l < L; ++l) {
    const eb_geom_desc& pd = A->lv[l - 1].d;
    BoxIdx& B = A->pr[l].B;
    const int* lo = box_lo + 3 * (l - 1);
    const int* hi = box_hi + 3 * (l - 1);
    B.D = D;
    for (int k = 0; k < 3; ++k) {
      B.nc[k] = k < D ? pd.n[k] : 1;
      B.lo[k] = k < D ? lo[k] : 0;
      B.hi[k] = k < D ? hi[k] : 1;
      B.nf[k] = k < D ? 2 * (B.hi[k] - B.lo[k]) : 1;
      if (k < D && (B.lo[k] < 0 || B.hi[k] > B.nc[k] || B.hi[k] - B.lo[k] < 4 || (B.hi[k] - B.lo[k]) % 4)) {
        delete A;
        set_error("the box of level " + std::to_string(l) +
                  " must lie in its parent grid with sides a positive multiple of 4 parent cells");
        return EB_ERR_INVALID;
      }
    }
    // proper nesting: one parent cell between the box and each CF side of the parent
    if (l >= 2)
      for (int k = 0; k < D; ++k) {
        const BoxIdx& PB = A->pr[l - 1].B;
        if ((cf_side(PB, k, 0) && B.lo[k] < 1) || (cf_side(PB, k, 1) && B.hi[k] > B.nc[k] - 1)) {
          delete A;
          set_error("the box of level " + std::to_string(l) +
                    " must keep one parent cell away from every coarse-fine side of its parent");
          return EB_ERR_INVALID;
        }
      }
    eb_geom_desc& d = A->lv[l].d;
    d = pd;
    for (int k = 0; k < D; ++k) {
      d.n[k] = B.nf[k];
      d.lo[k] = pd.lo[k] + B.lo[k] * pd.h;
    }
    d.h = pd.h / 2.0;
    // sides on the domain boundary keep the parent's (domain) conditions
    eb_geom_desc& d0 = A->lv[l].d0;
    d0 = d;
    for (int k = 0; k < D; ++k)
      for (int s2 = 0; s2 < 2; ++s2) {
        if (!cf_side(B, k, s2)) continue;
        d.bc_type[2 * k + s2] = EB_BC_NEUMANN;
        d.bc_value[2 * k + s2] = 0.0;
        d0.bc_type[2 * k + s2] = EB_BC_DIRICHLET;
        d0.bc_value[2 * k + s2] = 0.0;
      }
    d0.n_electrodes = pd.n_electrodes;
    for (int e = 0; e < pd.n_electrodes; ++e) d0.electrode_phi[e] = 0.0;
  }
  eb_status st = EB_OK;
  for (int l = 0; l < L && st == EB_OK; ++l) {
    st = eb_geom_build(&A->lv[l].d, stream, &A->lv[l].G);
    if (st == EB_OK && l > 0) st = eb_geom_build(&A->lv[l].d0, stream, &A->lv[l].G0);
  }
  if (st != EB_OK) return amr_fail(A, st);
  for (int l = 0; l < L; ++l) {
    AmrLevel& v = A->lv[l];
    v.n = v.G->L[0].g.ncell;
    v.h = v.d.h;
    v.flags = v.G->L[0].flags;
    if (v.n >= (1LL << 32)) {  // the composite kernels index cells in 32 bits
      set_error("composite grids are limited to 2^32 cells per level");
      return amr_fail(A, EB_ERR_INVALID);
    }
  }
  A->eps0 = desc->eps_gas;
  auto alloc = [&](size_t bytes) { return dev_alloc(A->allocs, std::max<size_t>(bytes, 16), &A->bytes, &st); };
  // CF sides and face counts of every pair
  for (int l = 1; l < L; ++l) {
    AmrPair& P = A->pr[l];
    const BoxIdx& B = P.B;
    CFBox& cb = P.cfb;
    std::memset(&cb, 0, sizeof(cb));
    for (int k = 0; k < 3; ++k) {
      cb.lo[k] = B.lo[k];
      cb.hi[k] = B.hi[k];
    }
    long long off = 0, coff = 0;
    for (int a = 0; a < D; ++a)
      for (int s2 = 0; s2 < 2; ++s2) {
        if (!cf_side(B, a, s2)) continue;
        long long nfa = 1, nca = 1;
        for (int k = 0; k < D; ++k)
          if (k != a) {
            nfa *= B.nf[k];
            nca *= B.hi[k] - B.lo[k];
          }
        cb.side_a[cb.nside] = a;
        cb.side_s[cb.nside] = s2;
        cb.off[cb.nside] = off;
        cb.coff[cb.nside] = coff;
        ++cb.nside;
        off += nfa;
        coff += nca;
      }
    cb.off[cb.nside] = off;
    cb.coff[cb.nside] = coff;
    P.nface = off;
    P.ncface = coff;
    P.faces = (CFFace*)alloc(sizeof(CFFace) * off);
    P.cfaces = (CFCoarse*)alloc(sizeof(CFCoarse) * coff);
    P.fl = (double*)alloc(sizeof(double) * off);
  }
  for (int l = 0; l < L; ++l) {
    AmrLevel& v = A->lv[l];
    const size_t b2 = sizeof(double) * 2 * v.n;
    if (l < L - 1) v.pc = (double*)alloc(b2);
    if (l > 0) v.kap = (double*)alloc(b2);
    v.r = (double*)alloc(b2);
    v.b0 = (double*)alloc(b2);
    v.own = (uint8_t*)alloc(v.n);
  }
  A->d_status = (int*)alloc(sizeof(int));
  A->d_norm = (unsigned long long*)alloc(sizeof(unsigned long long) * 2);
  if (st != EB_OK) return amr_fail(A, st);
  for (int l = 0; l < L; ++l) {
    AmrLevel& v = A->lv[l];
    k_own_flags<<<nb(v.n), TBA, 0, s>>>(A->pr[l + 1 < L ? l + 1 : l].B, v.flags, v.n, l < L - 1, v.own);
    if (v.pc) cudaMemsetAsync(v.pc, 0, sizeof(double) * 2 * v.n, s);
  }
  for (int l = 1; l < L && st == EB_OK; ++l) {
    AmrPair& P = A->pr[l];
    st = build_cf(A->lv[l].G, A->lv[l - 1].G, P.cfb, P.faces, P.cfaces, A->d_status, s);
    if (st != EB_OK) break;
    eb_geom_arrays ga;
    std::memset(&ga, 0, sizeof(ga));
    ga.kappa = A->lv[l].kap;
    st = eb_geom_export(A->lv[l].G, &ga, stream);
  }
  if (st != EB_OK) return amr_fail(A, st);
  // a correction inside the preconditioner is one V-cycle of 3+3 sweeps (on the
  // 256^3 + 128^3 pin-plane grid, before the levels were split by colour: 21
  // FGMRES iterations and 285 ms, against 19 and 447 ms with two 6+6 V-cycles to
  // 1e-2; 2+2 sweeps needed 23 iterations; now 84 ms).  A relaxed bottom grid
  // takes at most 32 sweeps (then 243 ms against 252 ms with 64; 16 sweeps needed
  // 23 iterations).
  eb_solver_opts oc = A->o;
  oc.inner_cycles = 1;
  oc.nu1 = oc.nu2 = 3;
  oc.bottom_sweeps = std::min(oc.bottom_sweeps, 32);
  st = poisson_setup(A->lv[0].G, &oc, PS_PLAIN, &A->lv[0].P);
  A->lv[0].P0 = A->lv[0].P;
  for (int l = 1; l < L && st == EB_OK; ++l) {
    st = poisson_setup(A->lv[l].G, &A->o, PS_OPERATOR, &A->lv[l].P);
    if (st == EB_OK) st = poisson_setup(A->lv[l].G0, &oc, PS_PLAIN, &A->lv[l].P0);
  }
  if (st != EB_OK) return amr_fail(A, st);
  if (cudaStreamSynchronize(s) != cudaSuccess) return amr_fail(A, cuda_fail(cudaGetLastError(), "amr setup"));
  *out = A;
  return EB_OK;
}

extern "C" eb_status eb_amr_setup(const eb_geom_desc* desc, const int box_lo[3], const int box_hi[3],
                                  const eb_solver_opts* opts, void* stream, eb_amr** out) {
  return eb_amr_setup_levels(desc, 2, box_lo, box_hi, opts, stream, out);
}

extern "C" eb_status eb_amr_query(const eb_amr* A, long long* n_coarse, long long* n_fine, int fine_n[3],
                                  long long* cf_faces) {
  if (!A) {
    set_error("null argument");
    return EB_ERR_INVALID;
  }
  if (n_coarse) *n_coarse = A->lv[0].n;
  if (n_fine) *n_fine = A->lv[1].n;
  if (fine_n)
    for (int k = 0; k < 3; ++k) fine_n[k] = A->pr[1].B.nf[k];
  if (cf_faces) *cf_faces = A->pr[1].nface;
  return EB_OK;
}

extern "C" eb_status eb_amr_level_query(const eb_amr* A, int level, int* n_levels, long long* n_cells, int n[3],
                                        double lo[3], double* h, long long* cf_faces) {
  if (!A || level < 0 || level >= A->L) {
    set_error(A ? "level out of range" : "null argument");
    return EB_ERR_INVALID;
  }
  const AmrLevel& v = A->lv[level];
  if (n_levels) *n_levels = A->L;
  if (n_cells) *n_cells = v.n;
  for (int k = 0; k < 3; ++k) {
    if (n) n[k] = k < A->D ? v.d.n[k] : 1;
    if (lo) lo[k] = k < A->D ? v.d.lo[k] : 0.0;
  }
  if (h) *h = v.h;
  if (cf_faces) *cf_faces = level > 0 ? A->pr[level].nface : 0;
  return EB_OK;
}

extern "C" eb_status eb_amr_level_geom(const eb_amr* A, int level, const eb_geom** out) {
  if (!A || !out || level < 0 || level >= A->L) {
    set_error(A && out ? "level out of range" : "null argument");
    return EB_ERR_INVALID;
  }
  *out = A->lv[level].G;
  return EB_OK;
}

// b of every level's operator for the given data, into lv[l].b0
static eb_status amr_rhs(eb_amr* A, const double* const* rhs, const double* const* sig, cudaStream_t s) {
  eb_status st = EB_OK;
  for (int l = 0; l < A->L && st == EB_OK; ++l)
    st = poisson_rhs(A->lv[l].P, rhs[l], sig ? sig[l] : nullptr, A->lv[l].b0, s);
  return st;
}

// The composite operator on levels >= lmin.  phi's values under a finer box
// are first replaced by the finer level's means, finest first: in place
// (copy = false), or in lv[l].pc.  out[l] = b[l] - A phi, or A phi where b is
// null (entries without an unknown left alone).  Rows under a box come out
// 0, except on a level whose out is the remainder of a correction (zero =
// false), where restrict_down sets them.
static eb_status amr_apply(eb_amr* A, const double* const* b, double* const* phi, double* const* out, int lmin,
                           bool copy, bool zero, cudaStream_t s) {
  const int L = A->L;
  const double sgn = b ? 1.0 : -1.0;
  const double* val[AMR_MAXL];
  val[L - 1] = phi[L - 1];
  for (int l = L - 2; l >= 0; --l) {
    AmrLevel &c = A->lv[l], &f = A->lv[l + 1];
    val[l] = phi[l];
    if (l < lmin) continue;  // read outside its box alone
    double* pc = phi[l];
    if (copy) {
      pc = c.pc;
      cudaMemcpyAsync(pc, phi[l], 2 * c.n * sizeof(double), cudaMemcpyDeviceToDevice, s);
    }
    k_avg_down<<<nb(box_cells(A->pr[l + 1].B)), TBA, 0, s>>>(A->pr[l + 1].B, c.flags, f.flags, f.kap, val[l + 1], pc,
                                                            c.n, f.n);
    note_launch();
    val[l] = pc;
  }
  eb_status st = EB_OK;
  for (int l = lmin; l < L && st == EB_OK; ++l) st = poisson_apply(A->lv[l].P, b ? b[l] : nullptr, val[l], sgn, out[l], s);
  if (st != EB_OK) return st;
  for (int l = std::max(1, lmin); l < L; ++l) {
    const AmrPair& P = A->pr[l];
    AmrLevel &c = A->lv[l - 1], &f = A->lv[l];
    if (!P.nface) continue;
    k_cf_flux<<<nb(P.nface), TBA, 0, s>>>(P.faces, P.nface, val[l - 1], val[l], A->eps0, f.h, P.fl);
    note_launch();
    for (int sd = 0; sd < P.cfb.nside; ++sd) {
      long long t0 = P.cfb.off[sd], t1 = P.cfb.off[sd + 1];
      k_cf_fine_apply<<<nb(t1 - t0), TBA, 0, s>>>(P.faces, t0, t1, P.fl, sgn * f.h, out[l]);
      note_launch();
    }
    if (l - 1 < lmin) continue;
    k_cf_coarse_apply<<<nb(P.ncface), TBA, 0, s>>>(P.cfaces, P.ncface, P.fl, val[l - 1], c.n, c.h, A->D, sgn, out[l - 1]);
    note_launch();
  }
  for (int l = std::max(1, lmin + 1); l < L && zero; ++l) {
    k_zero_under<<<nb(box_cells(A->pr[l].B)), TBA, 0, s>>>(A->pr[l].B, out[l - 1], A->lv[l - 1].n);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? EB_OK : cuda_fail(e, "composite residual");
}

// composite residual of the data in lv[l].b0 into lv[l].r
static eb_status amr_resid(eb_amr* A, double* const* phi, bool copy, cudaStream_t s) {
  const double* b[AMR_MAXL];
  double* r[AMR_MAXL];
  for (int l = 0; l < A->L; ++l) {
    b[l] = A->lv[l].b0;
    r[l] = A->lv[l].r;
  }
  return amr_apply(A, b, phi, r, 0, copy, true, s);
}

static eb_status amr_norm(eb_amr* A, cudaStream_t s, double* out) {
  cudaMemsetAsync(A->d_norm, 0, sizeof(unsigned long long), s);
  for (int l = 0; l < A->L; ++l) {
    k_absmax2<<<nb(A->lv[l].n), TBA, 0, s>>>(A->lv[l].flags, A->lv[l].n, A->lv[l].r, A->d_norm);
    note_launch();
  }
  unsigned long long v = 0;
  cudaError_t e = cudaMemcpyAsync(&v, A->d_norm, sizeof(v), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "composite norm");
  std::memcpy(out, &v, sizeof(double));
  return EB_OK;
}

static bool all_set(const double* const* p, int n) {
  if (!p) return false;
  for (int l = 0; l < n; ++l)
    if (!p[l]) return false;
  return true;
}

extern "C" eb_status eb_amr_residual_levels(eb_amr* A, const double* const* d_rhs, const double* const* d_sig,
                                            const double* const* d_phi, double* const* d_r, void* stream) {
  if (!A || !all_set(d_rhs, A->L) || !all_set(d_phi, A->L) || !d_r || !all_set(d_r, A->L)) {
    set_error("null argument");
    return EB_ERR_INVALID;
  }
  cudaStream_t s = (cudaStream_t)stream;
  eb_status st = amr_rhs(A, d_rhs, d_sig, s);
  for (int l = 0; l < A->L; ++l) cudaMemsetAsync(A->lv[l].r, 0, 2 * A->lv[l].n * sizeof(double), s);
  if (st == EB_OK) st = amr_resid(A, const_cast<double* const*>(d_phi), true, s);  // copies: d_phi is only read
  if (st != EB_OK) return st;
  for (int l = 0; l < A->L; ++l)
    cudaMemcpyAsync(d_r[l], A->lv[l].r, 2 * A->lv[l].n * sizeof(double), cudaMemcpyDeviceToDevice, s);
  cudaError_t e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? EB_OK : cuda_fail(e, "composite residual");
}

extern "C" eb_status eb_amr_residual(eb_amr* A, const double* d_rhs_c, const double* d_sig_c, const double* d_rhs_f,
                                     const double* d_sig_f, const double* d_phi_c, const double* d_phi_f,
                                     double* d_r_c, double* d_r_f, void* stream) {
  if (A && A->L != 2) {
    set_error("eb_amr_residual serves two-level grids; use eb_amr_residual_levels");
    return EB_ERR_INVALID;
  }
  const double* rhs[2] = {d_rhs_c, d_rhs_f};
  const double* sig[2] = {d_sig_c, d_sig_f};
  const double* phi[2] = {d_phi_c, d_phi_f};
  double* r[2] = {d_r_c, d_r_f};
  return eb_amr_residual_levels(A, rhs, sig, phi, r, stream);
}

static CVPtrs cv_ptrs(const std::vector<CVec>& V, int l, int m) {
  CVPtrs p{};
  for (int i = 0; i < m; ++i) p.v[i] = V[i].v[l];
  return p;
}
static constexpr long long CV_PART = (long long)CV_MAXV * DOT_BLOCKS;  // block sums per level

// the sums of m vectors V[0..m) (and w itself when self) with w into d_h[0..)
static void cv_mdot(eb_amr* A, int m, const CVec& w, bool self, const int* go, double* out, cudaStream_t s) {
  const int k = m + (self ? 1 : 0);
  for (int l = 0; l < A->L; ++l) {
    const AmrLevel& v = A->lv[l];
    CVPtrs p = cv_ptrs(A->V, l, m);
    if (self) p.v[m] = w.v[l];
    double* part = A->d_part + l * CV_PART;
    // fewer accumulators leave registers for more loads in flight
    if (k <= 4) k_cv_mdot<4><<<DOT_BLOCKS, TBA, 0, s>>>(v.own, v.n, k, p, w.v[l], go, part);
    else if (k <= 8) k_cv_mdot<8><<<DOT_BLOCKS, TBA, 0, s>>>(v.own, v.n, k, p, w.v[l], go, part);
    else k_cv_mdot<CV_MAXV><<<DOT_BLOCKS, TBA, 0, s>>>(v.own, v.n, k, p, w.v[l], go, part);
    note_launch();
  }
  k_cv_finish<<<1, 32 * CV_MAXV, 0, s>>>(A->d_part, A->L, CV_PART, k, go ? 3 : 0, nullptr, 0, A->d_go, out);
  note_launch();
}
static void cv_maxpy_norm(eb_amr* A, int m, const double* h, const CVec& w, const int* go, int what, const double* in,
                          double* out, cudaStream_t s) {
  for (int l = 0; l < A->L; ++l) {
    const AmrLevel& v = A->lv[l];
    k_cv_maxpy_norm<<<DOT_BLOCKS, TBA, 0, s>>>(v.own, v.n, m, cv_ptrs(A->V, l, m), h, w.v[l], go, A->d_part + l * CV_PART);
    note_launch();
  }
  k_cv_finish<<<1, 32, 0, s>>>(A->d_part, A->L, CV_PART, 1, what, in, m, A->d_go, out);
  note_launch();
}
static void cv_scale(eb_amr* A, const double* norm, const CVec& w, cudaStream_t s) {
  for (int l = 0; l < A->L; ++l) {
    const AmrLevel& v = A->lv[l];
    k_cv_scale<<<nb((v.n + 3) / 4), TBA, 0, s>>>(v.own, v.n, norm, w.v[l]);
    note_launch();
  }
}

// w[l] for l = L-2 .. lmin: cells under the next finer box take the mean of
// that level's children (finest first, so every level sees the whole remainder)
static void restrict_down(eb_amr* A, double* const* w, int lmin, cudaStream_t s) {
  for (int l = A->L - 2; l >= lmin; --l) {
    const AmrLevel &c = A->lv[l], &f = A->lv[l + 1];
    k_restrict_under<<<nb(box_cells(A->pr[l + 1].B)), TBA, 0, s>>>(A->pr[l + 1].B, f.flags, w[l + 1], w[l], c.n, f.n);
    note_launch();
  }
}

// events around the next V-cycle of a solve
static cudaEvent_t* next_events(eb_amr* A, size_t* used) {
  while (A->ev.size() < *used + 2) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    A->ev.push_back(e);
  }
  *used += 2;
  return A->ev.data() + *used - 2;
}

// z = M^-1 v: one multiplicative FAC sweep from zero, coarse to fine: a
// V-cycle on level 0 over the domain (the finer parts of v restricted under
// the boxes, into v's entries there, which nothing else reads), constant per
// parent on level 1; then on every finer level a V-cycle on what remains there,
// v - A z (zero Dirichlet CF sides; the remainder of the still finer levels,
// where z is still zero, restricted under its box), added to the level and
// constant per parent on the next.  (Passing the whole of z on instead of the
// level's own correction stalls with four levels.)  Only the levels that a
// correction needs are applied, and A z is subtracted from v in the same
// pass.  Uses lv[].r for the remainders and lv[].pc for inner corrections.
static eb_status fac_apply(eb_amr* A, const CVec& v, const CVec& z, int* cycles, size_t* used, cudaStream_t s) {
  const int L = A->L;
  double* rem[AMR_MAXL];
  for (int l = 0; l < L; ++l) rem[l] = A->lv[l].r;
  restrict_down(A, v.v, 0, s);
  for (int l = 2; l < L; ++l) cudaMemsetAsync(z.v[l], 0, 2 * A->lv[l].n * sizeof(double), s);
  eb_status st = poisson_vcycle(A->lv[0].P, v.v[0], z.v[0], false, next_events(A, used), s);
  const double* e = z.v[0];
  for (int l = 1; l < L && st == EB_OK; ++l) {
    const AmrLevel& f = A->lv[l];
    k_prolong_const<<<nb(f.n), TBA, 0, s>>>(A->pr[l].B, f.flags, e, z.v[l], A->lv[l - 1].n, f.n);
    note_launch();
    st = amr_apply(A, v.v, z.v, rem, l, false, false, s);
    if (st != EB_OK) break;
    restrict_down(A, rem, l, s);
    if (l == L - 1) {
      st = poisson_vcycle(f.P0, rem[l], z.v[l], true, next_events(A, used), s);
    } else {
      st = poisson_vcycle(f.P0, rem[l], f.pc, false, next_events(A, used), s);
      CVPtrs p{};
      p.v[0] = f.pc;
      p.a[0] = 1.0;
      k_cv_update<<<nb(f.n), TBA, 0, s>>>(f.own, f.n, 1, p, z.v[l]);
      note_launch();
      e = f.pc;
    }
  }
  *cycles += L;
  return st;
}

static constexpr int GM = 12;  // FGMRES restart length
// d_h: the first pass's sums, the second one's, the new norm, and the flag
static constexpr int H2 = CV_MAXV, HN = 2 * CV_MAXV, HGO = HN + 2, HLEN = HGO + 2;

static eb_status amr_workspace(eb_amr* A) {
  if (!A->V.empty()) return EB_OK;
  eb_status st = EB_OK;
  auto vec = [&]() {
    CVec v;
    for (int l = 0; l < A->L; ++l) {
      v.v[l] = (double*)dev_alloc(A->allocs, 2 * A->lv[l].n * sizeof(double), &A->bytes, &st);
      if (v.v[l]) cudaMemset(v.v[l], 0, 2 * A->lv[l].n * sizeof(double));
    }
    return v;
  };
  for (int i = 0; i <= GM; ++i) A->V.push_back(vec());
  for (int i = 0; i < GM; ++i) A->Z.push_back(vec());
  A->d_part = (double*)dev_alloc(A->allocs, A->L * CV_PART * sizeof(double), &A->bytes, &st);
  A->d_h = (double*)dev_alloc(A->allocs, HLEN * sizeof(double), &A->bytes, &st);
  A->d_go = (int*)(A->d_h + HGO);
  if (st == EB_OK && !A->h_h) {
    cudaError_t e = cudaMallocHost(&A->h_h, HLEN * sizeof(double));
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) st = cuda_fail(e, "composite work space");
  }
  if (st != EB_OK) {
    A->V.clear();
    A->Z.clear();
  }
  return st;
}

extern "C" eb_status eb_amr_solve_levels(eb_amr* A, const double* const* d_rhs, const double* const* d_sig,
                                         double* const* d_phi, eb_solve_info* info, void* stream) {
  if (!A || !all_set(d_rhs, A->L) || !d_phi || !all_set(d_phi, A->L)) {
    set_error("null argument");
    return EB_ERR_INVALID;
  }
  const int L = A->L;
  cudaStream_t s = (cudaStream_t)stream;
  eb_solve_info inf;
  std::memset(&inf, 0, sizeof(inf));
  std::memset(A->kstat, 0, sizeof(A->kstat));
  const long long launches0 = launch_total();
  eb_status st = amr_workspace(A);
  if (st != EB_OK) return st;
  for (int l = 0; l < L; ++l) poisson_vcycle_begin(A->lv[l].P0, s);
  // b: the composite residual at phi = 0
  for (int l = 0; l < L; ++l) cudaMemsetAsync(A->Z[0].v[l], 0, 2 * A->lv[l].n * sizeof(double), s);
  st = amr_rhs(A, d_rhs, d_sig, s);
  if (st == EB_OK) st = amr_resid(A, A->Z[0].v, false, s);
  double bn = 0.0, r = 0.0;
  if (st == EB_OK) st = amr_norm(A, s, &bn);
  if (st != EB_OK) return st;
  int it = 0, cycles = 0;
  size_t used = 0;  // events
  const int max_it = std::max(1, A->o.max_cycles);
  // restarted FGMRES, right-preconditioned by one FAC sweep (Sec. 3.3.2's
  // multigrid as the inner solver of every correction)
  st = EB_ERR_NOT_CONVERGED;
  while (it < max_it) {
    eb_status s2 = amr_resid(A, d_phi, false, s);
    if (s2 == EB_OK) s2 = amr_norm(A, s, &r);
    for (int l = 0; l < L && s2 == EB_OK && it > 0; ++l) s2 = poisson_vcycle_error(A->lv[l].P0, s);
    if (s2 != EB_OK) {
      st = s2;
      break;
    }
    if (bn == 0.0 || r <= A->o.tol * bn) {
      st = EB_OK;
      break;
    }
    if (!(r == r) || r > 1e6 * bn) break;
    // v0 = r / |r|_2
    for (int l = 0; l < L; ++l)
      cudaMemcpyAsync(A->V[0].v[l], A->lv[l].r, 2 * A->lv[l].n * sizeof(double), cudaMemcpyDeviceToDevice, s);
    cv_maxpy_norm(A, 0, nullptr, A->V[0], nullptr, 4, nullptr, A->d_h + HN, s);
    cv_scale(A, A->d_h + HN, A->V[0], s);
    cudaMemcpyAsync(A->h_h, A->d_h, HLEN * sizeof(double), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    const double beta = A->h_h[HN];
    if (!(beta > 0.0)) {
      st = EB_OK;
      break;
    }
    // this cycle's target in the 2-norm estimate: the reduction the max norm
    // still needs, with a factor 1/2 of margin
    const double target = 0.5 * (A->o.tol * bn / r) * beta;
    double H[GM + 1][GM], cs[GM], sn[GM], g[GM + 1];
    std::memset(H, 0, sizeof(H));
    std::memset(g, 0, sizeof(g));
    g[0] = beta;
    int k = 0;
    for (; k < GM && it < max_it; ++k, ++it) {
      const CVec& w = A->V[k + 1];
      s2 = fac_apply(A, A->V[k], A->Z[k], &cycles, &used, s);
      if (s2 == EB_OK) s2 = amr_apply(A, nullptr, A->Z[k].v, w.v, 0, false, true, s);
      if (s2 != EB_OK) break;
      // classical Gram-Schmidt, all k + 1 projections in one pass, repeated
      // only when the pass removed most of w (cancellation may then have left
      // it short of orthogonal).  The sums, the decision and the norm stay on
      // the device; the host reads the step's column of H once.
      cv_mdot(A, k + 1, w, true, nullptr, A->d_h, s);
      cv_maxpy_norm(A, k + 1, A->d_h, w, nullptr, 1, A->d_h, A->d_h + HN, s);
      cv_mdot(A, k + 1, w, false, A->d_go, A->d_h + H2, s);
      cv_maxpy_norm(A, k + 1, A->d_h + H2, w, A->d_go, 2, nullptr, A->d_h + HN, s);
      cv_scale(A, A->d_h + HN, w, s);
      cudaError_t e = cudaMemcpyAsync(A->h_h, A->d_h, HLEN * sizeof(double), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) {
        s2 = cuda_fail(e, "composite step");
        break;
      }
      int go = 0;
      std::memcpy(&go, A->h_h + HGO, sizeof(go));
      for (int i = 0; i <= k; ++i) H[i][k] = A->h_h[i] + (go ? A->h_h[H2 + i] : 0.0);
      H[k + 1][k] = A->h_h[HN];
      for (int i = 0; i < k; ++i) {  // earlier rotations
        double t = cs[i] * H[i][k] + sn[i] * H[i + 1][k];
        H[i + 1][k] = -sn[i] * H[i][k] + cs[i] * H[i + 1][k];
        H[i][k] = t;
      }
      double den = std::hypot(H[k][k], H[k + 1][k]);
      cs[k] = den > 0.0 ? H[k][k] / den : 1.0;
      sn[k] = den > 0.0 ? H[k + 1][k] / den : 0.0;
      H[k][k] = den;
      H[k + 1][k] = 0.0;
      g[k + 1] = -sn[k] * g[k];
      g[k] = cs[k] * g[k];
      // the 2-norm estimate far below the target: stop the cycle and check the true max norm
      if (std::fabs(g[k + 1]) <= target) {
        ++k;
        ++it;
        break;
      }
    }
    if (s2 != EB_OK) {
      st = s2;
      break;
    }
    // x += Z y with H y = g (upper triangular)
    double y[GM];
    for (int i = k - 1; i >= 0; --i) {
      double t = g[i];
      for (int j = i + 1; j < k; ++j) t -= H[i][j] * y[j];
      y[i] = H[i][i] != 0.0 ? t / H[i][i] : 0.0;
    }
    for (int l = 0; l < L; ++l) {
      CVPtrs p = cv_ptrs(A->Z, l, k);
      for (int i = 0; i < k; ++i) p.a[i] = y[i];
      k_cv_update<<<nb(A->lv[l].n), TBA, 0, s>>>(A->lv[l].flags, A->lv[l].n, k, p, d_phi[l]);
      note_launch();
    }
  }
  // report every level's phi under the next finer box as the finer means
  // (finest first), and 0 where there is no unknown: what the guess held in those
  // entries was neither read nor written so far
  if (st == EB_OK || st == EB_ERR_NOT_CONVERGED) {
    for (int l = 0; l < L; ++l) {
      k_zero_absent<<<nb(A->lv[l].n), TBA, 0, s>>>(A->lv[l].flags, A->lv[l].n, d_phi[l]);
      note_launch();
    }
    for (int l = L - 2; l >= 0; --l) {
      const AmrLevel &c = A->lv[l], &f = A->lv[l + 1];
      k_avg_down<<<nb(box_cells(A->pr[l + 1].B)), TBA, 0, s>>>(A->pr[l + 1].B, c.flags, f.flags, f.kap,
                                                              d_phi[l + 1], d_phi[l], c.n, f.n);
      note_launch();
    }
    if (st == EB_ERR_NOT_CONVERGED) set_error("composite iteration cap reached");
  }
  for (int l = 0; l < L && it > 0 && (st == EB_OK || st == EB_ERR_NOT_CONVERGED); ++l) {
    const eb_status s2 = poisson_vcycle_error(A->lv[l].P0, s);
    if (s2 != EB_OK) st = s2;
  }
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess && (st == EB_OK || st == EB_ERR_NOT_CONVERGED)) st = cuda_fail(e, "composite solve");
  for (size_t i = 0; i + 1 < used; i += 2) {  // a sweep's V-cycles in order of level
    float ms = 0.0f;
    if (cudaEventElapsedTime(&ms, A->ev[i], A->ev[i + 1]) == cudaSuccess) amr_count(A, (i / 2) % L ? 1 : 0, 1, 1, ms);
  }
  cudaGetLastError();
  inf.status = st;
  inf.outer_iters = it;
  inf.vcycles = cycles;
  inf.bnorm = bn;
  inf.rel_res = bn > 0.0 ? r / bn : 0.0;
  inf.kernel_ms = A->kstat[0][1] + A->kstat[1][1];
  inf.kernel_launches = launch_total() - launches0;
  if (info) *info = inf;
  return st;
}

extern "C" eb_status eb_amr_solve(eb_amr* A, const double* d_rhs_c, const double* d_sig_c, const double* d_rhs_f,
                                  const double* d_sig_f, double* d_phi_c, double* d_phi_f, eb_solve_info* info,
                                  void* stream) {
  if (A && A->L != 2) {
    set_error("eb_amr_solve serves two-level grids; use eb_amr_solve_levels");
    return EB_ERR_INVALID;
  }
  const double* rhs[2] = {d_rhs_c, d_rhs_f};
  const double* sig[2] = {d_sig_c, d_sig_f};
  double* phi[2] = {d_phi_c, d_phi_f};
  return eb_amr_solve_levels(A, rhs, sig, phi, info, stream);
}

extern "C" eb_status eb_amr_field_eval(eb_amr* A, int level, const double* d_phi, const double* d_sigma,
                                       double* d_E, double* d_En, void* stream) {
  if (!A || level < 0 || level >= A->L) {
    set_error(A ? "level out of range" : "null argument");
    return EB_ERR_INVALID;
  }
  return eb_field_eval(A->lv[level].P, d_phi, d_sigma, d_E, d_En, stream);
}

extern "C" eb_status eb_amr_kernel_stats(const eb_amr* A, double out[8]) {
  if (!A || !out) {
    set_error("null argument");
    return EB_ERR_INVALID;
  }
  for (int w = 0; w < 2; ++w)
    for (int k = 0; k < 4; ++k) out[4 * w + k] = A->kstat[w][k];
  return EB_OK;
}
