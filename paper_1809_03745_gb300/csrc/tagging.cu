// tagging.cu -- refinement tags of Sec. 6 and the box a regrid step takes
// from them.
//
// The tracer is T = |E| / max |E|; a cell is tagged for refinement when
// |grad T| dx / T > eps1 or T > eps2 and for coarsening when
// |grad T| dx / T < eps3 and T < eps4, with centred or one-sided differences
// in index units (dx cancels).  The tags are a function of E alone: every
// product and sum is written with round-to-nearest intrinsics (this unit is
// also compiled without FMA contraction), sqrt and division are correctly
// rounded, and they match a plain FP64 evaluation in the same order.
//
// FP64 is slow on this part (two operations per clock and SM), and a tag is
// four comparisons, so almost no cell needs it.  The first pass writes |E| in
// FP32 and takes max |E|^2 in FP64 (order-free atomicMax on the bit pattern;
// the square root is monotone, so its root is max |E|).  The second evaluates
// the tests in FP32 with a bound on their error, and where a threshold lies
// within it, or a value outside FP32's range, in FP64 from E as above.
// 256^3 on a random field: 0.30 + 0.41 ms, against 0.55 + 0.25 + 1.23 ms for
// three passes in FP64.
#include <cuda_runtime.h>

#include <climits>
#include <cmath>
#include <cstring>
#include <string>

#include "eb_internal.h"

using namespace ebp;

namespace {

constexpr int TBT = 256;
int nbt(long long n) { return (int)std::max<long long>(1, std::min<long long>((n + TBT - 1) / TBT, 152LL * 16)); }

struct TagOut {
  unsigned long long emax;  // bit pattern of max |E|^2
  unsigned long long count;
  int lo[3], hi[3];  // hi inclusive while reducing
};

struct TagView {
  int D;
  int n[3];
  long long ncell;
  const uint8_t* flags;
  const double* E;  // [D][2][ncell]
};

// largest squared field magnitude over the phases with an unknown (0 where covered)
__device__ __forceinline__ double cell_mag2(const TagView& v, unsigned f, long long c) {
  double m = 0.0;
  for (int p = 0; p < 2; ++p) {
    if (!((f >> p) & 1u)) continue;  // a phase without an unknown is never selected: skip its reads
    const double e0 = v.E[(long long)p * v.ncell + c];
    double m2 = __dmul_rn(e0, e0);
    for (int a = 1; a < v.D; ++a) {
      const double e = v.E[((long long)a * 2 + p) * v.ncell + c];
      m2 = __dadd_rn(m2, __dmul_rn(e, e));
    }
    if (m2 > m) m = m2;
  }
  return m;
}

__global__ void __launch_bounds__(TBT) k_emag(TagView v, float* __restrict__ M, TagOut* out) {
  unsigned long long m = 0ull;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < v.ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const double m2 = cell_mag2(v, v.flags[c], c);
    M[c] = sqrtf((float)m2);
    const unsigned long long b = (unsigned long long)__double_as_longlong(m2);
    m = b > m ? b : m;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, m, o);
    m = b > m ? b : m;
  }
  if ((threadIdx.x & 31) == 0 && m) atomicMax(&out->emax, m);
}

// T of a cell in FP64
__device__ __forceinline__ double tracer(const TagView& v, long long c, double emax) {
  return emax > 0.0 ? sqrt(cell_mag2(v, v.flags[c], c)) / emax : 0.0;
}
// the tag of a cell in FP64 (bit 0 refine, bit 1 coarsen)
template <int D>
__device__ __noinline__ unsigned tag_exact(const TagView& v, long long c, const int I[3], double emax, double eps1,
                                           double eps2, double eps3, double eps4) {
  const long long stride[3] = {1, v.n[0], (long long)v.n[0] * v.n[1]};
  const double T = tracer(v, c, emax);
  double s2 = 0.0;
  for (int a = 0; a < D; ++a) {
    const bool hp = I[a] + 1 < v.n[a] && (v.flags[c + stride[a]] & 3u);
    const bool hm = I[a] > 0 && (v.flags[c - stride[a]] & 3u);
    const double Tp = hp ? tracer(v, c + stride[a], emax) : 0.0;
    const double Tm = hm ? tracer(v, c - stride[a], emax) : 0.0;
    const double d = hp && hm ? __dmul_rn(__dsub_rn(Tp, Tm), 0.5) : hp ? __dsub_rn(Tp, T)
                                                                  : hm ? __dsub_rn(T, Tm) : 0.0;
    s2 = __dadd_rn(s2, __dmul_rn(d, d));
  }
  const double g = sqrt(s2);
  const double ratio = T > 0.0 ? g / T : (g > 0.0 ? INFINITY : 0.0);
  return (ratio > eps1 || T > eps2 ? 1u : 0u) | (ratio < eps3 && T < eps4 ? 2u : 0u);
}

template <int D>
__global__ void __launch_bounds__(TBT) k_tag(TagView v, const float* __restrict__ M, double eps1, double eps2,
                                             double eps3, double eps4, int keep, int klo0, int klo1, int klo2,
                                             int khi0, int khi1, int khi2, uint8_t* tags, TagOut* out) {
  const int klo[3] = {klo0, klo1, klo2}, khi[3] = {khi0, khi1, khi2};
  int mlo[3] = {INT_MAX, INT_MAX, INT_MAX}, mhi[3] = {-1, -1, -1};
  unsigned cnt = 0;
  const double emax = sqrt(__longlong_as_double((long long)out->emax));
  const float inv = (float)(1.0 / emax);
  // FP32 decides where the magnitudes are far from its ends
  const bool fast = emax > 1e-12 && emax < 1e12;
  const float e1 = (float)eps1, e2 = (float)eps2, e3 = (float)eps3, e4 = (float)eps4;
  const int stride[3] = {1, v.n[0], v.n[0] * v.n[1]};
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < v.ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const unsigned cu = (unsigned)c, r = cu / (unsigned)v.n[0];
    const int I[3] = {(int)(cu - r * (unsigned)v.n[0]), (int)(r % (unsigned)v.n[1]), (int)(r / (unsigned)v.n[1])};
    unsigned t = 0;
    if (v.flags[c] & 3u) {
      const float m = M[c];
      float s2 = 0.0f, sum = 0.0f;
      bool small = !(m > 1e-15f);
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const bool hp = I[a] + 1 < v.n[a] && (v.flags[c + stride[a]] & 3u);
        const bool hm = I[a] > 0 && (v.flags[c - stride[a]] & 3u);
        const float mp = hp ? M[c + stride[a]] : 0.0f, mm = hm ? M[c - stride[a]] : 0.0f;
        const float d = hp && hm ? 0.5f * (mp - mm) : hp ? mp - m : hm ? m - mm : 0.0f;
        s2 += d * d;
        sum += mp + mm + m;
        small = small || (hp && !(mp > 1e-15f)) || (hm && !(mm > 1e-15f));
      }
      const float T = m * inv, ratio = sqrtf(s2) / m;
      // a magnitude is off by less than 2^-22 of itself, a difference by 2^-22
      // of the sum of its two, so the ratio by 2^-22 (sum / m + ratio) with
      // room for the rounding of the tests themselves
      const float er = 1e-6f * (sum / m + ratio), et = 1e-6f * T;
      const bool sure = fast && !small && sum < 1e18f && fabsf(ratio - e1) > er + 1e-6f * fabsf(e1) &&
                        fabsf(ratio - e3) > er + 1e-6f * fabsf(e3) && fabsf(T - e2) > et + 1e-6f * fabsf(e2) &&
                        fabsf(T - e4) > et + 1e-6f * fabsf(e4);
      if (sure) t = (ratio > e1 || T > e2 ? 1u : 0u) | (ratio < e3 && T < e4 ? 2u : 0u);
      else t = tag_exact<D>(v, c, I, emax, eps1, eps2, eps3, eps4);
      bool marked = t & 1u;
      if (!marked && keep && !(t & 2u)) {
        marked = true;
#pragma unroll
        for (int a = 0; a < D; ++a) marked = marked && I[a] >= klo[a] && I[a] < khi[a];
      }
      if (marked) {
        ++cnt;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          mlo[a] = min(mlo[a], I[a]);
          mhi[a] = max(mhi[a], I[a]);
        }
      }
    }
    if (tags) tags[c] = (uint8_t)t;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mlo[a] = __reduce_min_sync(0xffffffffu, mlo[a]);
    mhi[a] = __reduce_max_sync(0xffffffffu, mhi[a]);
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if ((threadIdx.x & 31) == 0 && cnt) {
    atomicAdd(&out->count, (unsigned long long)cnt);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      atomicMin(&out->lo[a], mlo[a]);
      atomicMax(&out->hi[a], mhi[a]);
    }
  }
}

}  // namespace

extern "C" eb_status eb_tag_cells(const eb_geom* G, const double* d_E, const double eps[4], const int* keep_lo,
                                  const int* keep_hi, unsigned char* d_tags, int bbox_lo[3], int bbox_hi[3],
                                  long long* n_marked, double* e_max, void* stream) {
  if (!G || !d_E || !eps || !bbox_lo || !bbox_hi || !n_marked || (!keep_lo) != (!keep_hi)) {
    set_error("null argument (keep_lo and keep_hi go together)");
    return EB_ERR_INVALID;
  }
  for (int k = 0; k < 4; ++k)
    if (!std::isfinite(eps[k])) {
      set_error("tagging thresholds must be finite");
      return EB_ERR_INVALID;
    }
  // the geometry's arrays live on the device it was built on: the kernels
  // must run there
  int dev = -1;
  cudaError_t ed = cudaGetDevice(&dev);
  if (ed != cudaSuccess) return cuda_fail(ed, "device query");
  if (dev != G->device) {
    set_error("the current device (" + std::to_string(dev) + ") is not the geometry's device (" +
              std::to_string(G->device) + ")");
    return EB_ERR_INVALID;
  }
  const DevLevel& F = G->L[0];
  TagView v;
  v.D = F.g.D;
  for (int k = 0; k < 3; ++k) v.n[k] = k < v.D ? F.g.n[k] : 1;
  v.ncell = F.g.ncell;
  v.flags = F.flags;
  v.E = d_E;
  cudaStream_t s = (cudaStream_t)stream;
  TagOut init;
  std::memset(&init, 0, sizeof(init));
  for (int a = 0; a < 3; ++a) {
    init.lo[a] = INT_MAX;
    init.hi[a] = -1;
  }
  // one block: the result words, then |E| in FP32.  The geometry keeps it for
  // the next call; a call that finds it in use by another thread takes its own.
  const size_t head = (sizeof(TagOut) + 255) / 256 * 256;
  std::unique_lock<std::mutex> lock(G->scratch_lock, std::try_to_lock);
  const bool kept = lock.owns_lock();
  char* d_buf = kept ? (char*)G->scratch : nullptr;
  cudaError_t e = cudaSuccess;
  const size_t size = head + sizeof(float) * (size_t)v.ncell;
  if (!d_buf) e = cudaMalloc(&d_buf, size);
  if (e != cudaSuccess) return cuda_fail(e, "tag scratch");
  if (kept) {
    G->scratch = d_buf;
    G->scratch_bytes = (long long)size;
  }
  TagOut* d_out = (TagOut*)d_buf;
  float* d_M = (float*)(d_buf + head);
  e = cudaMemcpyAsync(d_out, &init, sizeof(init), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    k_emag<<<nbt(v.ncell), TBT, 0, s>>>(v, d_M, d_out);
    note_launch();
    const int keep = keep_lo ? 1 : 0;
    int klo[3] = {0, 0, 0}, khi[3] = {0, 0, 0};
    if (keep)
      for (int a = 0; a < 3; ++a) {
        klo[a] = keep_lo[a];
        khi[a] = keep_hi[a];
      }
    if (v.D == 2)
      k_tag<2><<<nbt(v.ncell), TBT, 0, s>>>(v, d_M, eps[0], eps[1], eps[2], eps[3], keep, klo[0], klo[1], klo[2],
                                            khi[0], khi[1], khi[2], d_tags, d_out);
    else
      k_tag<3><<<nbt(v.ncell), TBT, 0, s>>>(v, d_M, eps[0], eps[1], eps[2], eps[3], keep, klo[0], klo[1], klo[2],
                                            khi[0], khi[1], khi[2], d_tags, d_out);
    note_launch();
    e = cudaGetLastError();
  }
  TagOut res;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&res, d_out, sizeof(res), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (!kept) cudaFree(d_buf);
  if (e != cudaSuccess) return cuda_fail(e, "refinement tags");
  *n_marked = (long long)res.count;
  for (int a = 0; a < 3; ++a) {
    bbox_lo[a] = res.count ? res.lo[a] : 0;
    bbox_hi[a] = res.count ? res.hi[a] + 1 : 0;
  }
  if (e_max) {
    double m2 = 0.0;
    std::memcpy(&m2, &res.emax, sizeof(double));
    *e_max = std::sqrt(m2);
  }
  return EB_OK;
}

extern "C" eb_status eb_regrid_box(int dim, const int n[3], const int cf_lo[3], const int cf_hi[3],
                                   const int bbox_lo[3], const int bbox_hi[3], long long n_marked, int buf, int block,
                                   int box_lo[3], int box_hi[3], int* has_box) {
  if (!n || !cf_lo || !cf_hi || !bbox_lo || !bbox_hi || !box_lo || !box_hi || !has_box || dim < 2 || dim > 3 ||
      buf < 0 || block < 1) {
    set_error("invalid argument");
    return EB_ERR_INVALID;
  }
  *has_box = 0;
  for (int a = 0; a < 3; ++a) {
    box_lo[a] = 0;
    box_hi[a] = a < dim ? 0 : 1;
  }
  if (n_marked <= 0) return EB_OK;
  auto floor_to = [block](long long x) { return (x >= 0 ? x / block : -((-x + block - 1) / block)) * block; };
  auto ceil_to = [block](long long x) { return (x >= 0 ? (x + block - 1) / block : -((-x) / block)) * block; };
  int lo[3], hi[3];
  for (int a = 0; a < dim; ++a) {
    long long l = floor_to((long long)bbox_lo[a] - buf), h = ceil_to((long long)bbox_hi[a] + buf);
    const long long lmin = cf_lo[a] ? block : 0, hmax = cf_hi[a] ? (long long)n[a] - block : n[a];
    l = std::max(l, lmin);
    h = std::min(h, hmax);
    if (h - l < block) {  // widened away from the clipped side to one block
      if (l == lmin) h = l + block;
      else l = h - block;
      if (l < lmin || h > hmax) return EB_OK;
    }
    lo[a] = (int)l;
    hi[a] = (int)h;
  }
  for (int a = 0; a < dim; ++a) {
    box_lo[a] = lo[a];
    box_hi[a] = hi[a];
  }
  *has_box = 1;
  return EB_OK;
}
