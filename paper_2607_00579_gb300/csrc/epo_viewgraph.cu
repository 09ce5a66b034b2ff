// Viewgraph estimation (Section 3, Viewgraph Estimation, Eq. 2; Algorithm 1 BuildViewgraph),
// run once before the optimisation.  For every ordered pair (i, j) of a scene, every source
// pixel of a regular grid of view i with a valid depth is projected into view j with Z_i
// (Eq. 2's pi), lifted there with Z_j at the nearest pixel and projected back into view i;
// the pair's fraction is the share of those pixels whose round trip stays in front of both
// cameras, inside view j, and returns within tau pixels.  A pair is kept when the fraction
// is at least min_frac in both directions (the paper's 12.5 % at tau = 3 px).
//
// The counts are those of an FP64 evaluation in which every product, sum, quotient and root is
// rounded on its own in a fixed order (trip_exact), whatever the compiler would fuse.  On this GPU
// that evaluation is ~200 instructions of the 1/64-rate FP64 pipe per grid pixel (24 views of
// 518x392 at stride 4: 2.5 ms), so every grid pixel first runs in FP32 beside a bound on its error,
// and only those with a decision inside the bound (well under 1 % of them) are kept in shared
// memory and evaluated in FP64, 32 to a warp (the same 24 views: 2544 -> 131 us for the whole call).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "../../include/epo.h"
#include "epo_internal.cuh"

namespace {

struct VgView {
  int32_t W, H;
  int64_t off;   // first depth element of the view
  double K[4];   // fx, fy, cx, cy
  double T[12];  // world -> camera [R|t], row-major
};

__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }

// camera v pixel (x, y) at depth z -> camera w pixel; false when not in front of w.
__device__ bool reproject(const VgView& v, const VgView& w, double x, double y, double z, double& xo, double& yo) {
  const double Xc0 = mul(__ddiv_rn(sub(x, v.K[2]), v.K[0]), z);
  const double Xc1 = mul(__ddiv_rn(sub(y, v.K[3]), v.K[1]), z);
  const double q0 = sub(Xc0, v.T[3]), q1 = sub(Xc1, v.T[7]), q2 = sub(z, v.T[11]);
  double Xw[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) Xw[c] = add(add(mul(v.T[c], q0), mul(v.T[4 + c], q1)), mul(v.T[8 + c], q2));
  double Y[3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
    Y[r] = add(add(add(mul(w.T[4 * r], Xw[0]), mul(w.T[4 * r + 1], Xw[1])), mul(w.T[4 * r + 2], Xw[2])), w.T[4 * r + 3]);
  if (!(Y[2] > 0.0)) return false;
  xo = add(__ddiv_rn(mul(w.K[0], Y[0]), Y[2]), w.K[2]);
  yo = add(__ddiv_rn(mul(w.K[1], Y[1]), Y[2]), w.K[3]);
  return true;
}

// One round trip of pixel (x, y) of view i at depth z, in FP64.
__device__ __noinline__ bool trip_exact(const VgView& vi, const VgView& vj, const float* depth, int x, int y, float zf,
                                        double tau) {
  const double z = (double)zf;
  double xj, yj;
  if (!reproject(vi, vj, (double)x, (double)y, z, xj, yj)) return false;
  if (!(xj >= 0.0 && xj <= (double)(vj.W - 1) && yj >= 0.0 && yj <= (double)(vj.H - 1))) return false;
  const int xn = (int)floor(add(xj, 0.5)), yn = (int)floor(add(yj, 0.5));  // nearest pixel
  if (xn < 0 || xn >= vj.W || yn < 0 || yn >= vj.H) return false;
  const double zj = (double)depth[vj.off + (int64_t)yn * vj.W + xn];
  if (!(zj > 0.0) || !isfinite(zj)) return false;
  double xb, yb;
  if (!reproject(vj, vi, xj, yj, zj, xb, yb)) return false;
  const double dx = sub(xb, (double)x), dy = sub(yb, (double)y);
  return __dsqrt_rn(add(mul(dx, dx), mul(dy, dy))) < tau;
}

constexpr int kVgThreads = 256;
constexpr int kVgRound = 1024;           // grid pixels between two looks at the kept ones
constexpr int kVgExact = 2 * kVgRound;   // room for the kept ones: evaluated once half full
constexpr int kVgBlocks = 4 * 152;  // one wave of resident blocks: fewer pairs are split over several
constexpr int64_t kVgMaxCount = 1 << 30;  // grid pixels of a block: its loop counts in int

// One direction of a pair in FP32: Y = M X + t, and the constants of the bound
//   |Y_r - Y_r(FP64)| <= E = z Ca + Cb.
// With u = 2^-24 and G >= 1, |X0| / z, |X1| / z anywhere in the image: X0 = ((x - cx) / fx) z carries
// 5u G z (the rounded cx, 1 / fx, and three operations), M's and t's entries u, the FMA chain at
// most 3u of each term, so |dY_r| <= 9u sum_c |M_rc| G z + 4u |t_r|: Ca = 10u m G, Cb = 10u max |t|
// with m the largest row sum.  The FP64 evaluation goes through world coordinates, at most ~40
// roundings of terms that |R_w| |R_v|^T (|X| + |t_v|) + |t_w| bounds: 1e-14 of that is added.
struct VgDir {
  float M[9], t[3];
  float Ca, Cb, m;
};

// Projects (X0, X1, z) with |Y_r| errors below E: q = Y_0,1 / Y_2 and the bound eq on its error.
// front: in front for certain and q, eq valid; behind: behind for certain; neither: not decided (near
// the camera plane, not a number, where E could underflow, or from 1e30 on: the reciprocal is flushed
// to zero above 2^126 and a sum that overflowed has lost its sign).  For e = E / Y2 <= 1/64,
// |q - q*| <= e (1 + |q|) / (1 - e) plus 4u |q| for the reciprocal and the product.  No branches: the
// callers keep what the flags allow.
__device__ __forceinline__ void project(const VgDir& d, float X0, float X1, float z, float E, float& qu, float& qv,
                                        float& eu, float& ev, bool& front, bool& behind) {
  constexpr float u = epo::kU32;
  const float Y0 = fmaf(d.M[2], z, fmaf(d.M[1], X1, fmaf(d.M[0], X0, d.t[0])));
  const float Y1 = fmaf(d.M[5], z, fmaf(d.M[4], X1, fmaf(d.M[3], X0, d.t[1])));
  const float Y2 = fmaf(d.M[8], z, fmaf(d.M[7], X1, fmaf(d.M[6], X0, d.t[2])));
  float iz;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(iz) : "f"(Y2));
  const float e = E * iz;
  front = Y2 > 1e-20f && Y2 < 1e30f && e <= 1.f / 64.f;
  behind = Y2 < -1e-20f && Y2 > -1e30f && Y2 < -E;
  qu = Y0 * iz;
  qv = Y1 * iz;
  const float e1 = 1.05f * e;
  eu = fmaf(e1 + 4.f * u, fabsf(qu), e1);
  ev = fmaf(e1 + 4.f * u, fabsf(qv), e1);
}

// Pixel coordinate f q + c and its error bound (the rounded f and c, the FMA, the comparisons).
__device__ __forceinline__ float pixel(float f, float c, float q, float eq, float& t) {
  const float p = fmaf(f, q, c);
  t = fmaf(f, eq, 6.f * epo::kU32 * (fabsf(p) + 2.f * fabsf(c)));
  return p;
}

// Four blocks per SM (64 registers): 131 us for the call on 24 views; five 145. The trips run without
// branches; with an early exit at every decision 146.
__global__ void __launch_bounds__(kVgThreads, 4) k_viewgraph(const VgView* views, const float* depth, int n, int stride,
                                                          double tau, int per_block, uint2* counts) {
  constexpr float u = epo::kU32;
  __shared__ VgView vi, vj;
  __shared__ VgDir fwd, bwd;
  __shared__ double s_M[9];
  __shared__ float s_n[2][8];  // per view: largest row and column sum of |R|, |t|, G
  __shared__ int s_list[kVgExact];
  __shared__ int s_count;
  const int i = blockIdx.x / (n - 1), j0 = blockIdx.x % (n - 1), j = j0 + (j0 >= i);
  {
    constexpr int words = sizeof(VgView) / 8;
    const double* a = reinterpret_cast<const double*>(views + i);
    const double* b = reinterpret_cast<const double*>(views + j);
    if (threadIdx.x < words) reinterpret_cast<double*>(&vi)[threadIdx.x] = a[threadIdx.x];
    else if (threadIdx.x < 2 * words) reinterpret_cast<double*>(&vj)[threadIdx.x - words] = b[threadIdx.x - words];
    if (threadIdx.x == 0) s_count = 0;
  }
  __syncthreads();
  if (threadIdx.x < 9) {  // M = R_j R_i^T
    const int r = threadIdx.x / 3, c = threadIdx.x % 3;
    const double m = vj.T[4 * r] * vi.T[4 * c] + vj.T[4 * r + 1] * vi.T[4 * c + 1] + vj.T[4 * r + 2] * vi.T[4 * c + 2];
    s_M[threadIdx.x] = m;
    fwd.M[threadIdx.x] = (float)m;
    bwd.M[3 * c + r] = (float)m;
  } else if (threadIdx.x == 32 || threadIdx.x == 64) {
    const int w = threadIdx.x / 32 - 1;
    const VgView& v = w ? vj : vi;
    float row = 0.f, col = 0.f, tm = 0.f;
    for (int r = 0; r < 3; ++r) {
      row = fmaxf(row, fabsf((float)v.T[4 * r]) + fabsf((float)v.T[4 * r + 1]) + fabsf((float)v.T[4 * r + 2]));
      col = fmaxf(col, fabsf((float)v.T[r]) + fabsf((float)v.T[4 + r]) + fabsf((float)v.T[8 + r]));
      tm = fmaxf(tm, fabsf((float)v.T[4 * r + 3]));
    }
    const float gx = ((float)v.W + fabsf((float)v.K[2])) / (float)v.K[0];
    const float gy = ((float)v.H + fabsf((float)v.K[3])) / (float)v.K[1];
    s_n[w][0] = row;
    s_n[w][1] = col;
    s_n[w][2] = tm;
    // images whose pixel coordinates are not exact in FP32, or whose pixels an int does not number,
    // take no decision there
    s_n[w][3] = v.W <= (1 << 22) && v.H <= (1 << 22) && (int64_t)v.W * v.H <= INT32_MAX ? fmaxf(1.f, fmaxf(gx, gy)) : INFINITY;
  }
  __syncthreads();
  if (threadIdx.x < 2) {  // t_ji = t_j - M t_i, and back t_ij = t_i - M^T t_j
    const int w = threadIdx.x;
    VgDir& d = w ? bwd : fwd;
    const VgView& from = w ? vj : vi;
    const VgView& to = w ? vi : vj;
    const float* nf = s_n[w];
    const float* nt = s_n[1 - w];
    float m = 0.f, tm = 0.f;
    for (int r = 0; r < 3; ++r) {
      double t = to.T[4 * r + 3];
      for (int c = 0; c < 3; ++c) t -= (w ? s_M[3 * c + r] : s_M[3 * r + c]) * from.T[4 * c + 3];
      d.t[r] = (float)t;
      tm = fmaxf(tm, fabsf((float)t));
      m = fmaxf(m, fabsf(d.M[3 * r]) + fabsf(d.M[3 * r + 1]) + fabsf(d.M[3 * r + 2]));
    }
    const float mm = 1e-14f * nt[0] * nf[1];  // rows of |R_to| times columns of |R_from|
    // the limits of either image hold for both directions: a trip indexes the depths of the other view
    const float G = nt[3] < INFINITY ? nf[3] : INFINITY;
    d.m = 1.01f * m;
    d.Ca = 1.01f * G * (10.f * u * m + mm);
    d.Cb = 1.01f * (10.f * u * tm + mm * nf[2] + 1e-14f * nt[2]);
  }
  __syncthreads();
  // the block's grid pixels are first .. first + count - 1 of the view's, which an int may not number,
  // and have numbers of their own from 0
  const unsigned gw = (unsigned)((vi.W - 1) / stride + 1), gh = (unsigned)((vi.H - 1) / stride + 1);
  const int64_t first = (int64_t)blockIdx.y * per_block;
  const int count = (int)max((int64_t)0, min((int64_t)per_block, (int64_t)gw * gh - first));  // 0: a smaller view's grid
  const float fxi = (float)vi.K[0], fyi = (float)vi.K[1], cxi = (float)vi.K[2], cyi = (float)vi.K[3];
  const float fxj = (float)vj.K[0], fyj = (float)vj.K[1], cxj = (float)vj.K[2], cyj = (float)vj.K[3];
  const float rfx = (float)(1.0 / vi.K[0]), rfy = (float)(1.0 / vi.K[1]);
  const float Wm1 = (float)(vj.W - 1), Hm1 = (float)(vj.H - 1), tf = (float)tau;
  const float* di = depth + vi.off;
  const float* dj = depth + vj.off;
  unsigned valid = 0u, good = 0u;
  // two grid pixels per thread in flight: each trip is two dependent loads, and the kernel waits
  // for them rather than for its arithmetic (one in flight: 205 us for the call on 24 views of
  // 518x392, two: 166)
  constexpr int ILP = 2;
  constexpr int kStep = ILP * kVgThreads;
  const unsigned dr = kStep / gw, dc = kStep % gw;
  const unsigned row0 = (unsigned)(first / gw), col0 = (unsigned)(first % gw);
  unsigned row[ILP], col[ILP];
#pragma unroll
  for (int k = 0; k < ILP; ++k) {
    const unsigned g = col0 + k * kVgThreads + threadIdx.x;
    row[k] = row0 + g / gw;
    col[k] = g % gw;
  }
  for (int round = 0; round < count; round += kVgRound) {
    const int end = min(count, round + kVgRound);
    for (int base = round; base < end; base += kStep) {
      float z[ILP], qu[ILP], qv[ILP], eu[ILP], ev[ILP], zj[ILP], xf[ILP], yf[ILP];
      bool doubt[ILP], on[ILP];  // an FP32 decision is in doubt; so far the trip holds
      int at[ILP];
#pragma unroll
      for (int k = 0; k < ILP; ++k) {
        const int x = (int)col[k] * stride, y = (int)row[k] * stride;
        const bool in = base + k * kVgThreads + (int)threadIdx.x < end;
        z[k] = in ? di[(int64_t)y * vi.W + x] : 0.f;
        xf[k] = (float)x;
        yf[k] = (float)y;
        row[k] += dr;
        col[k] += dc;
        if (col[k] >= gw) {
          col[k] -= gw;
          ++row[k];
        }
      }
#pragma unroll
      for (int k = 0; k < ILP; ++k) {
        const bool live = z[k] > 0.f && z[k] < INFINITY;
        valid += live;
        bool front, behind;
        project(fwd, (xf[k] - cxi) * rfx * z[k], (yf[k] - cyi) * rfy * z[k], z[k], fmaf(z[k], fwd.Ca, fwd.Cb), qu[k], qv[k],
                eu[k], ev[k], front, behind);
        float tu, tv;
        const float up = pixel(fxj, cxj, qu[k], eu[k], tu), vp = pixel(fyj, cyj, qv[k], ev[k], tv);
        const float ou = up - Wm1, ov = vp - Hm1;
        const bool outside = up < -tu || ou > tu || vp < -tv || ov > tv;
        const float fu = floorf(up), fv = floorf(vp), ru = up - fu - 0.5f, rv = vp - fv - 0.5f;
        on[k] = live && front && up >= tu && -ou >= tu && vp >= tv && -ov >= tv && fabsf(ru) > tu && fabsf(rv) > tv;
        doubt[k] = live && !on[k] && !behind && !(front && outside);
        at[k] = on[k] ? ((int)fv + (rv > 0.f)) * vj.W + (int)fu + (ru > 0.f) : 0;
      }
#pragma unroll
      for (int k = 0; k < ILP; ++k) zj[k] = on[k] ? dj[at[k]] : 0.f;
#pragma unroll
      for (int k = 0; k < ILP; ++k) {
        on[k] = zj[k] > 0.f && zj[k] < INFINITY;  // only trips that hold so far have read a depth
        const float E = fmaf(zj[k], fmaf(bwd.m, fmaxf(eu[k], ev[k]), bwd.Ca), bwd.Cb);
        float bu, bv;
        bool front, behind;
        project(bwd, qu[k] * zj[k], qv[k] * zj[k], zj[k], E, bu, bv, eu[k], ev[k], front, behind);
        float tu, tv;
        const float dx = pixel(fxi, cxi, bu, eu[k], tu) - xf[k], dy = pixel(fyi, cyi, bv, ev[k], tv) - yf[k];
        float d;
        asm("sqrt.approx.f32 %0, %1;" : "=f"(d) : "f"(fmaf(dx, dx, dy * dy)));  // relative error below 2^-22
        const float td = tu + tv + 10.f * u * (d + tf);
        const bool near = front && d + td < tf, far = front && d - td > tf;
        good += on[k] && near;
        doubt[k] = doubt[k] || (on[k] && !near && !far && !behind);
        if (doubt[k]) s_list[atomicAdd(&s_count, 1)] = base + k * kVgThreads + (int)threadIdx.x;
      }
    }
    __syncthreads();
    const int kept = s_count;
    __syncthreads();  // every thread has read it before the next round appends
    if (kept > kVgExact - kVgRound || end == count) {
      for (int k = threadIdx.x; k < kept; k += kVgThreads) {
        const int64_t g = first + s_list[k];
        const int x = (int)(g % gw) * stride, y = (int)(g / gw) * stride;
        good += trip_exact(vi, vj, depth, x, y, di[(int64_t)y * vi.W + x], tau);
      }
      __syncthreads();
      if (threadIdx.x == 0) s_count = 0;
      __syncthreads();
    }
  }
  valid = __reduce_add_sync(0xffffffffu, valid);
  good = __reduce_add_sync(0xffffffffu, good);
  if ((threadIdx.x & 31) == 0) {
    uint2* c = counts + (size_t)i * n + j;
    if (valid) atomicAdd(&c->x, valid);
    if (good) atomicAdd(&c->y, good);
  }
}

}  // namespace

extern "C" epo_status epo_build_viewgraph(int32_t n_views, const int32_t* W, const int32_t* H, const double* K,
                                          const double* T, const float* depth_dev, int32_t stride, double tau,
                                          double min_frac, double* frac, int32_t* pairs, int32_t* n_pairs,
                                          void* cuda_stream) {
  EPO_RANGE("epo_build_viewgraph");
  if (n_views < 1 || n_views > 46340 || !W || !H || !K || !T || !depth_dev || stride < 1 || !(tau > 0) ||
      !(min_frac >= 0) || !n_pairs)
    return EPO_ERR_INVALID_ARG;
  const int n = n_views;
  std::vector<VgView> hv(n);
  int64_t off = 0, grid = 1;  // grid: the most grid pixels of a view
  for (int v = 0; v < n; ++v) {
    if (W[v] < 1 || H[v] < 1) return EPO_ERR_INVALID_ARG;
    hv[v].W = W[v];
    hv[v].H = H[v];
    hv[v].off = off;
    off += (int64_t)W[v] * H[v];
    for (int k = 0; k < 4; ++k) hv[v].K[k] = K[4 * v + k];
    for (int k = 0; k < 12; ++k) hv[v].T[k] = T[12 * v + k];
    if (!(hv[v].K[0] > 0) || !(hv[v].K[1] > 0)) return EPO_ERR_INVALID_ARG;
    grid = std::max(grid, (int64_t)((W[v] - 1) / stride + 1) * ((H[v] - 1) / stride + 1));
  }
  if (grid > (int64_t)UINT32_MAX) return EPO_ERR_TOO_LARGE;  // the counts are 32-bit
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // the view table and the pairs' counts in one allocation
  const size_t view_bytes = sizeof(VgView) * n, count_bytes = sizeof(uint2) * (size_t)n * n;
  static_assert(sizeof(VgView) % 8 == 0, "the counts follow the view table");
  char* d_buf = nullptr;
  std::vector<uint2> counts((size_t)n * n);
  epo_status rc = EPO_OK;
  if (cudaMalloc(&d_buf, view_bytes + count_bytes) != cudaSuccess) {
    rc = EPO_ERR_OOM;
  } else {
    const VgView* d_views = reinterpret_cast<const VgView*>(d_buf);
    uint2* d_counts = reinterpret_cast<uint2*>(d_buf + view_bytes);
    // one block per ordered pair; with few pairs each pair's grid is split over several blocks
    // (at least 512 pixels each) so that they fill the GPU, in one wave: each block forms its pair's
    // constants in FP64 first (24 views, with branches: 146 us unsplit, 156 in halves, 168 in quarters)
    const int64_t pairs_n = (int64_t)n * (n - 1);
    int64_t split = std::min<int64_t>(std::max<int64_t>(1, kVgBlocks / std::max<int64_t>(pairs_n, 1)), (grid + 511) / 512);
    split = std::max(split, (grid + kVgMaxCount - 1) / kVgMaxCount);
    const int per_block = (int)((grid + split - 1) / split);
    if (cudaMemcpyAsync(d_buf, hv.data(), view_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemsetAsync(d_counts, 0, count_bytes, st) != cudaSuccess)
      rc = EPO_ERR_CUDA;
    if (rc == EPO_OK && pairs_n > 0) {
      k_viewgraph<<<dim3((unsigned)pairs_n, (unsigned)split), kVgThreads, 0, st>>>(d_views, depth_dev, n, stride, tau,
                                                                                  per_block, d_counts);
      if (cudaGetLastError() != cudaSuccess) rc = EPO_ERR_CUDA;
    }
    if (rc == EPO_OK &&
        (cudaMemcpyAsync(counts.data(), d_counts, count_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
         cudaStreamSynchronize(st) != cudaSuccess))
      rc = EPO_ERR_CUDA;
  }
  if (d_buf) cudaFree(d_buf);
  if (rc != EPO_OK) return rc;
  std::vector<double> f((size_t)n * n);
  for (size_t k = 0; k < f.size(); ++k) f[k] = counts[k].x ? (double)counts[k].y / (double)counts[k].x : 0.0;
  // pairs kept in both directions, row-major
  int32_t m = 0;
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) {
      if (i == j || std::min(f[(size_t)i * n + j], f[(size_t)j * n + i]) < min_frac) continue;
      if (pairs) {
        pairs[2 * m] = i;
        pairs[2 * m + 1] = j;
      }
      ++m;
    }
  *n_pairs = m;
  if (frac) std::copy(f.begin(), f.end(), frac);
  return EPO_OK;
}
