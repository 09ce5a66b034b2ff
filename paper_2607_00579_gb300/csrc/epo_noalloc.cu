// Loss and gradient without any device allocation.
//
// For callers that cannot call cudaMalloc: a host that owns every byte of device memory
// (a plugin inside someone else's engine, a fixed memory budget handed out up front), a
// real-time loop where an allocation may block or fail, or code that runs while the
// device allocator is off limits.  Such a caller passes its own device buffers for the
// inputs and the outputs; the intermediate sums live in one fixed-size array of this file,
// reserved on every GPU that loads the library for as long as the process runs.
//
// The computation is the one of epo_loss_and_grad_dev: per directed pair i -> j, every
// record of view i is lifted, moved by T_ji = T_j T_i^-1, projected into view j, the map
// is sampled bilinearly, clamped and Huber-penalised; per-pair means, the loss average and
// the left-perturbation gradient follow.  Every projection is accurate to better than 2^-29 of a
// pixel before the value and slope terms are formed in FP32, and every branch decision is the
// FP64 one.
//
// This GPU's FP64 pipe runs at 1/64 of the FP32 rate, and a projection with its divisions is ~100
// FP64 instructions, so the edge kernel carries positions as pairs of floats (48 bits: TwoSum and
// FMA products) beside a bound on their error; a sample whose bound is too wide, or that has a
// decision within it, takes the FP64 form (sample_exact).  The final gather is a warp per pose; it
// was one block that scanned every pair for every pose.  24 views of 256x192, 192 pairs, 0.57 M
// evaluations: 200 us for the call (edge kernel 104, gather 98) before, 26 us now.  Over 100 drawn
// scenes the gradient is as far from a 64-bit evaluation of everything as with FP64 positions: median 3.035e-8
// of its norm both ways, largest 7.349e-8 (the FP32 terms and sums).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "../../include/epo.h"
#include "epo_internal.cuh"

namespace {

constexpr int kNaMaxViews = EPO_NOALLOC_MAX_VIEWS;
constexpr int kNaMaxPairs = EPO_NOALLOC_MAX_PAIRS;
constexpr int kNaThreads = 256;

struct NaPair {
  double R[9];  // R_ji
  double t[3];  // t_ji
};

// Per pair: sum rho, n_valid, sum dRho/dY (3), sum Y x dRho/dY (3), and the number of usable
// records of the source view (the |E_i| of Eq. 7 under EPO_NORM_ALL)
constexpr int kNaAcc = 9;

struct NaScratch {
  double acc[kNaMaxPairs][kNaAcc];
  NaPair pair[kNaMaxPairs];
};
// 4096 pairs x (9 + 12) doubles = 688,128 bytes (672 KiB), the size the header states
static_assert(sizeof(NaScratch) == (size_t)kNaMaxPairs * (kNaAcc + 12) * sizeof(double), "scratch size");
static_assert(sizeof(NaScratch) == 688128, "scratch size stated in epo.h");

// The scratch: one file-scope device array shared by every call on a device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NaScratch)];

// Device address of g_noalloc_scratch per device, resolved once per device.
constexpr int kNaMaxDevices = 64;
NaScratch* g_scratch_ptr[kNaMaxDevices] = {};
std::mutex g_scratch_mutex;

// 16 lanes per pair: lanes 0..8 one entry of R_ji each, lanes 9..11 one of t_ji.
constexpr int kNaSetupThreads = 64;

__global__ void __launch_bounds__(kNaSetupThreads) k_na_setup(epo_noalloc_problem pb, NaScratch* S) {
  epo::griddep_launch_dependents();
  const int p = (blockIdx.x * kNaSetupThreads + threadIdx.x) / 16, e = threadIdx.x & 15, base = threadIdx.x & 16;
  const bool pv = p < pb.n_pairs;
  const int i = pv ? pb.pairs[2 * p] : 0, j = pv ? pb.pairs[2 * p + 1] : 0;
  const double* Ti = pb.T + 12 * (size_t)i;
  const double* Tj = pb.T + 12 * (size_t)j;
  double val = 0.0;
  if (e < 9) {
    const int r = e / 3, c = e % 3;
    val = Tj[4 * r] * Ti[4 * c] + Tj[4 * r + 1] * Ti[4 * c + 1] + Tj[4 * r + 2] * Ti[4 * c + 2];
  }
  const int rr = e >= 9 && e < 12 ? e - 9 : 0;
  const double R0 = __shfl_sync(0xffffffffu, val, base + 3 * rr), R1 = __shfl_sync(0xffffffffu, val, base + 3 * rr + 1),
               R2 = __shfl_sync(0xffffffffu, val, base + 3 * rr + 2);
  if (e >= 9 && e < 12) val = Tj[4 * rr + 3] - (R0 * Ti[3] + R1 * Ti[7] + R2 * Ti[11]);
  if (!pv) return;
  if (e < 12) reinterpret_cast<double*>(&S->pair[p])[e] = val;  // R (9), then t (3)
  if (e < kNaAcc) S->acc[p][e] = 0.0;  // the array keeps the previous call's sums
}

// ---- numbers as unevaluated sums of two floats (Dekker, Knuth); every operation is written with
// its rounding, so that none is fused or reordered ----
struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 quick_sum(float a, float b) {  // |a| >= |b| or a = 0
  const float s = __fadd_rn(a, b);
  return {s, __fadd_rn(b, -__fadd_rn(s, -a))};
}
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fadd_rn(s, -a);
  return {s, __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb))};
}
__device__ __forceinline__ F2 add(F2 a, F2 b) {
  const F2 s = two_sum(a.h, b.h);
  return quick_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 mul(F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  return quick_sum(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ F2 mul(F2 a, float b) {
  const float p = __fmul_rn(a.h, b);
  return quick_sum(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
__device__ __forceinline__ F2 neg(F2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ F2 split(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}

// What a pair's samples read, in shared memory: the projective form of view i's records in view j,
// (Y3 u', Y3 v', Y3) = z B (u, v, 1) + c, as float pairs, and the bound's constants.
struct NaForm {
  F2 B[9], c[3];
  F2 cx, cy, rfx, rfy;  // of view j: principal point, 1 / focal length
  // the bound's constants, over the two pixel rows and for the depth row: |B[r][0]| + |B[r][1]|, |B[r][2]|, |c[r]|
  float mp, np, cp, mz, nz, cz;
};

// One sample's place in view j for the value and slope terms: its cell, the fractions and the
// camera-frame point rounded to FP32, the FP32 value and whether it passes the clamp.
struct NaSample {
  float a, b, y0, y1, y2, d;
  float m00, m01, m10, m11;
  bool valid, pass;
};

// The FP64 form: every operation and decision in FP64.
__device__ __noinline__ NaSample sample_exact(const epo_noalloc_problem& pb, const NaPair& q, const double* Ki,
                                              const double* Kj, int W, int H, const float* map, float u, float v, float z) {
  NaSample s;
  s.valid = false;
  const double X[3] = {((double)u - Ki[2]) / Ki[0] * (double)z, ((double)v - Ki[3]) / Ki[1] * (double)z, (double)z};
  double Y[3];
  for (int r = 0; r < 3; ++r) Y[r] = q.R[3 * r] * X[0] + q.R[3 * r + 1] * X[1] + q.R[3 * r + 2] * X[2] + q.t[r];
  if (!(Y[2] > pb.eps_z)) return s;
  const double up = Kj[0] * Y[0] / Y[2] + Kj[2];
  const double vp = Kj[1] * Y[1] / Y[2] + Kj[3];
  if (!(up >= 0.0 && up <= (double)(W - 1) && vp >= 0.0 && vp <= (double)(H - 1))) return s;
  const int x0 = min((int)floor(up), W - 2);
  const int y0 = min((int)floor(vp), H - 2);
  const double a = up - x0, b = vp - y0;
  const float* m = map + (int64_t)y0 * W + x0;
  s.m00 = m[0];
  s.m01 = m[1];
  s.m10 = m[W];
  s.m11 = m[W + 1];
  const double d = (1.0 - a) * (1.0 - b) * s.m00 + a * (1.0 - b) * s.m01 + (1.0 - a) * b * s.m10 + a * b * s.m11;
  s.valid = true;
  s.pass = d <= pb.lambda;
  s.d = (float)d;
  s.a = (float)a;
  s.b = (float)b;
  s.y0 = (float)Y[0];
  s.y1 = (float)Y[1];
  s.y2 = (float)Y[2];
  return s;
}

// The same in float pairs.  Returns 1 when every decision holds whatever the error, 0 when the
// sample has to take the FP64 form.
//
// With S = z ((|B[r][0]| + |B[r][1]|) max(|u|, |v|) + |B[r][2]|) + |c[r]|, each of (Y3 u', Y3 v', Y3) is within
// 2^-43 S of the exact value (nested products and sums of 2^-46 each).  The position error is then
// at most e = (Ep + max(|u'|, |v'|) Ez) / Y3; up to 2^-29 (1/16 of the rounding of a fraction to FP32)
// the sample is taken here, if its fractions lie farther than e from 0 and 1.
__device__ __forceinline__ int sample_pairs(const NaForm& f, float eps_z, float lam, int W, int H, const float* map, float u,
                                            float v, float z, NaSample& s) {
  constexpr float k43 = 1.1368684e-13f;  // 2^-43
  const float g = fmaxf(fabsf(u), fabsf(v));
  const float Ep = k43 * fmaf(z, fmaf(g, f.mp, f.np), f.cp), Ez = k43 * fmaf(z, fmaf(g, f.mz, f.nz), f.cz);
  F2 r[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    r[k] = add(mul(add(mul(f.B[3 * k], u), add(mul(f.B[3 * k + 1], v), f.B[3 * k + 2])), z), f.c[k]);
  s.valid = false;
  s.pass = false;
  // the threshold is given in FP64: its rounding and the bound on Y3 are inside the margin
  const float near = 4.f * Ez + 2.5e-7f * eps_z;
  if (r[2].h < eps_z - near) return 1;
  if (!(r[2].h > eps_z + near && r[2].h > 1e-30f && r[2].h < 1e30f)) return 0;
  // 1 / Y3 as (r0, r0 e): the approximate reciprocal and its first Newton correction
  float r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(r[2].h));
  const float re = __fmul_rn(r0, __fmaf_rn(-r[2].l, r0, __fmaf_rn(-r[2].h, r0, 1.f)));
  const float up = r[0].h * r0, vp = r[1].h * r0;  // relative error below 2^-21
  const float e = fmaf(fmaxf(fabsf(up), fabsf(vp)), Ez, Ep) * r0 * 1.01f;
  if (!(e <= 1.8626451e-9f)) return 0;  // 2^-29
  const float tu = fmaf(fabsf(up), 4.8e-7f, 1e-6f), tv = fmaf(fabsf(vp), 4.8e-7f, 1e-6f);
  const float Wm1 = (float)(W - 1), Hm1 = (float)(H - 1);
  if (up < -tu || up - Wm1 > tu || vp < -tv || vp - Hm1 > tv) return 1;  // outside
  if (!(up >= tu && Wm1 - up >= tu && vp >= tv && Hm1 - vp >= tv)) return 0;
  const float xf = floorf(up), yf = floorf(vp);
  const F2 iz = {r0, re};
  // fractions: (Y3 u' - x0 Y3) / Y3
  const F2 a = mul(add(r[0], mul(r[2], -xf)), iz), b = mul(add(r[1], mul(r[2], -yf)), iz);
  if (!(a.h > 1e-7f && a.h < 1.f - 1e-6f && b.h > 1e-7f && b.h < 1.f - 1e-6f)) return 0;  // a cell line, or a cell beside it
  const float* m = map + (int64_t)(int)yf * W + (int)xf;
  s.m00 = m[0];
  s.m01 = m[1];
  s.m10 = m[W];
  s.m11 = m[W + 1];
  const F2 top = add({s.m00, 0.f}, mul(a, two_sum(s.m01, -s.m00))), bot = add({s.m10, 0.f}, mul(a, two_sum(s.m11, -s.m10)));
  const F2 d = add(top, mul(b, add(bot, neg(top))));
  if (!(fabsf(d.h - lam) > 1e-6f * fabsf(lam) + 1e-6f * (fabsf(s.m00) + fabsf(s.m01) + fabsf(s.m10) + fabsf(s.m11)))) return 0;
  s.valid = true;
  s.pass = d.h < lam;
  s.d = d.h;
  s.a = a.h;
  s.b = b.h;
  s.y0 = mul(add(r[0], neg(mul(f.cx, r[2]))), f.rfx).h;
  s.y1 = mul(add(r[1], neg(mul(f.cy, r[2]))), f.rfy).h;
  s.y2 = r[2].h;
  return 1;
}

// Warp sums of 8 values, the butterfly over lane distances 16, 8, 4, 2, 1 as a reduce-scatter:
// lane L ends with value ((L >> 4) & 1) 4 + ((L >> 3) & 1) 2 + ((L >> 2) & 1).
__device__ __forceinline__ float warp_sums8(const float* v, int lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  float k4[4], k2[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) k4[k] = (b4 ? v[4 + k] : v[k]) + __shfl_xor_sync(0xffffffffu, b4 ? v[k] : v[4 + k], 16);
#pragma unroll
  for (int k = 0; k < 2; ++k) k2[k] = (b3 ? k4[2 + k] : k4[k]) + __shfl_xor_sync(0xffffffffu, b3 ? k4[k] : k4[2 + k], 8);
  float s = (b2 ? k2[1] : k2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? k2[0] : k2[1], 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  return s + __shfl_xor_sync(0xffffffffu, s, 1);
}

// blockIdx.y = pair; the block walks the source view's tiles of kNaThreads records.  The launch
// gives each pair as many blocks as make one wave of four per SM in all: building a pair's form is a
// chain of FP64 on one warp while the others wait, so a block does it for several tiles.  The call on
// 24 views of 256x192: 26.4 us; two waves 30.3, four 36.6; at three blocks per SM (72 registers) 32.6.
constexpr int kNaEdgeBlocks = 4 * 152;

__global__ void __launch_bounds__(kNaThreads, 4) k_na_edge(epo_noalloc_problem pb, NaScratch* S) {
  __shared__ float s_red[2][kNaThreads / 32][kNaAcc];
  __shared__ NaForm s_f;
  __shared__ double s_Ki[4], s_Kj[4];
  const int p = blockIdx.y;
  const int i = pb.pairs[2 * p], j = pb.pairs[2 * p + 1];
  // no more tiles than the caller's maximum of records per view makes
  const int64_t most = (pb.max_records_per_view + kNaThreads - 1) / kNaThreads * kNaThreads;
  const int64_t r0 = pb.rec_off[i], n = min(pb.rec_off[i + 1] - r0, most);
  const int W = pb.W[j], H = pb.H[j];
  const float* map = pb.maps + pb.map_off[j];
  epo::griddep_launch_dependents();
  if ((int64_t)blockIdx.x * kNaThreads >= n) {
    epo::griddep_wait();  // the finish kernel's wait for this grid covers the setup too
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < 4) s_Ki[threadIdx.x] = pb.K[4 * (size_t)i + threadIdx.x];
  else if (threadIdx.x < 8) s_Kj[threadIdx.x - 4] = pb.K[4 * (size_t)j + threadIdx.x - 4];
  epo::griddep_wait();  // the pair's relative pose
  const NaPair& q = S->pair[p];
  if (warp == 0) {
    __syncwarp();
    // lane 3r + c < 9: B[r][c] = f_r M[r][c] + c_r M[2][c], M = R K_i^-1, (f, c)_r = (fx_j, cx_j),
    // (fy_j, cy_j), (1, 0); lane 9 + r: c[r] = f_r t[r] + c_r t[2]
    const int e = min(lane, 11), r = e < 9 ? e / 3 : e - 9, c = e % 3;
    // the four reciprocals in one division: 1 / focal length of view i (lanes 0, 1) and view j (2, 3)
    const double rf = 1.0 / (lane & 2 ? s_Kj : s_Ki)[lane & 1];
    const double rx = __shfl_sync(0xffffffffu, rf, 0), ry = __shfl_sync(0xffffffffu, rf, 1);
    const auto entry = [&](int row) {
      if (e >= 9) return q.t[row];
      const double* R = q.R + 3 * row;
      return c == 0 ? R[0] * rx : (c == 1 ? R[1] * ry : R[2] - (R[0] * (s_Ki[2] * rx) + R[1] * (s_Ki[3] * ry)));
    };
    const double mr = entry(r), m2 = entry(2);
    const double val = r == 2 ? mr : fma(s_Kj[r], mr, s_Kj[2 + r] * m2);
    if (lane < 9) s_f.B[lane] = split(val);
    else if (lane < 12) s_f.c[lane - 9] = split(val);
    const float av = fabsf((float)val);
    float sum[3], off[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      sum[k] = __shfl_sync(0xffffffffu, av, 3 * k) + __shfl_sync(0xffffffffu, av, 3 * k + 1);
      off[k] = __shfl_sync(0xffffffffu, av, 3 * k + 2);
    }
    const float c0 = __shfl_sync(0xffffffffu, av, 9), c1 = __shfl_sync(0xffffffffu, av, 10), c2 = __shfl_sync(0xffffffffu, av, 11);
    if (lane == 0) {
      s_f.mp = 1.01f * fmaxf(sum[0], sum[1]);
      s_f.np = 1.01f * fmaxf(off[0], off[1]);
      s_f.cp = 1.01f * fmaxf(c0, c1);
      s_f.mz = 1.01f * sum[2];
      s_f.nz = 1.01f * off[2];
      s_f.cz = 1.01f * c2;
    } else if (lane == 12 || lane == 13) {
      (lane == 12 ? s_f.cx : s_f.cy) = split(s_Kj[lane - 10]);
    } else if (lane == 14 || lane == 15) {
      (lane == 14 ? s_f.rfx : s_f.rfy) = split(rf);
    }
  }
  __syncthreads();
  const float lam = (float)pb.lambda, delta = (float)pb.huber_delta, eps_z = (float)pb.eps_z;
  const float fx = (float)s_Kj[0], fy = (float)s_Kj[1];
  int buf = 0;
  for (int64_t tile = blockIdx.x; tile * kNaThreads < n; tile += gridDim.x, buf ^= 1) {
    const int64_t idx = tile * kNaThreads + threadIdx.x;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    bool usable = false;
    if (idx < n) {
      const float4 rec = reinterpret_cast<const float4*>(pb.records)[r0 + idx];
      // records without a usable depth are not part of the problem (as at scene creation)
      usable = rec.z > 0.f && isfinite(rec.x) && isfinite(rec.y) && isfinite(rec.z);
      if (usable) {
        NaSample s;
        if (!sample_pairs(s_f, eps_z, lam, W, H, map, rec.x, rec.y, rec.z, s))
          s = sample_exact(pb, q, s_Ki, s_Kj, W, H, map, rec.x, rec.y, rec.z);
        if (s.valid) {
          const float dh = s.pass ? s.d : lam;
          const float adh = fabsf(dh);
          acc[0] = adh <= delta ? 0.5f * dh * dh : delta * (adh - 0.5f * delta);
          acc[1] = 1.f;
          const float drho = s.pass ? (fabsf(s.d) <= delta ? s.d : copysignf(delta, s.d)) : 0.f;
          // the products that a sum of two fuses are written out: which one the compiler picks
          // otherwise depends on the code around them, and moves the gradient by 2e-8
          const float ddu = fmaf(1.f - s.b, s.m01 - s.m00, __fmul_rn(s.b, s.m11 - s.m10));
          const float ddv = fmaf(1.f - s.a, s.m10 - s.m00, __fmul_rn(s.a, s.m11 - s.m01));
          const float iz = 1.f / s.y2;
          const float gx = drho * ddu * fx * iz;
          const float gy = drho * ddv * fy * iz;
          const float gz = -fmaf(gx, s.y0, __fmul_rn(gy, s.y1)) * iz;
          acc[2] = gx;
          acc[3] = gy;
          acc[4] = gz;
          acc[5] = fmaf(s.y1, gz, -__fmul_rn(s.y2, gy));
          acc[6] = fmaf(s.y2, gx, -__fmul_rn(s.y0, gz));
          acc[7] = fmaf(s.y0, gy, -__fmul_rn(s.y1, gx));
        }
      }
    }
    // block reduction: warp shuffles, then a fixed-order sum over warps, one FP64 atomic per slot;
    // the partial sums alternate between two buffers, so one barrier per tile is enough
    const float sum = warp_sums8(acc, lane);
    const unsigned n_use = __popc(__ballot_sync(0xffffffffu, usable));
    if ((lane & 3) == 0) s_red[buf][warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = sum;
    if (lane == 1) s_red[buf][warp][8] = (float)n_use;
    __syncthreads();
    if (threadIdx.x < kNaAcc) {
      float v = 0.f;
      for (int w = 0; w < kNaThreads / 32; ++w) v += s_red[buf][w][threadIdx.x];
      if (v != 0.f) atomicAdd(&S->acc[p][threadIdx.x], (double)v);
    }
  }
}

// The loss (Eq. 6), one block, and the per-pose gradient, one warp per view: the warp lists the
// (pair, role) entries of its view, then takes them one per lane.
constexpr int kNaFinThreads = 128;
constexpr int kNaFinViews = kNaFinThreads / 32;

__global__ void __launch_bounds__(kNaFinThreads) k_na_finish(epo_noalloc_problem pb, const NaScratch* S, double* loss,
                                                             double* grad) {
  __shared__ double s_sum[kNaFinThreads / 32];
  __shared__ int s_ent[kNaFinViews][32 + 64];  // up to 31 waiting and 64 of the next 32 pairs: pair << 1 | source
  const int P = pb.n_pairs, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int slot = pb.norm_mode == EPO_NORM_ALL ? 8 : 1;  // the pair means' denominators
  if (blockIdx.x == 0) {
    epo::griddep_wait();
    double part = 0.0;
    for (int p = threadIdx.x; p < P; p += kNaFinThreads) {
      const double denom = S->acc[p][slot];
      if (denom > 0.0) part += S->acc[p][0] / denom;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) s_sum[warp] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < kNaFinThreads / 32; ++w) t += s_sum[w];
      *loss = P > 0 ? (2.0 / P) * t : 0.0;
    }
    return;
  }
  const int v = ((int)blockIdx.x - 1) * kNaFinViews + warp;
  const bool vv = v < pb.n_views;
  int* ent = s_ent[warp];
  double g[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int waiting = 0;
  const double w2 = 2.0 / P;
  bool waited = false;
  for (int p0 = 0; vv && p0 < P; p0 += 32) {
    const int p = p0 + lane;
    const int i = p < P ? pb.pairs[2 * p] : -1, j = p < P ? pb.pairs[2 * p + 1] : -1;
    const unsigned as_t = __ballot_sync(0xffffffffu, j == v), as_s = __ballot_sync(0xffffffffu, i == v);
    const unsigned lt = (1u << lane) - 1u;
    if (j == v) ent[waiting + __popc(as_t & lt)] = 2 * p;
    if (i == v) ent[waiting + __popc(as_t) + __popc(as_s & lt)] = 2 * p + 1;
    waiting += __popc(as_t) + __popc(as_s);
    __syncwarp();
    while (waiting >= 32 || (p0 + 32 >= P && waiting > 0)) {
      if (!waited) {
        epo::griddep_wait();  // the sums; the entry lists above do not depend on them
        waited = true;
      }
      const int take = min(waiting, 32);
      if (lane < take) {
        const int en = ent[lane], q = en >> 1;
        const bool src = en & 1;
        const double* a = S->acc[q];
        const double denom = a[slot];
        if (denom > 0.0) {
          const double c = w2 / denom;
          const double ga0 = c * a[2], ga1 = c * a[3], ga2 = c * a[4], gb0 = c * a[5], gb1 = c * a[6], gb2 = c * a[7];
          if (src) {
            // source view: -Ad(T_ji)^T (ga, gb) = (-R^T ga, R^T (t x ga) - R^T gb)
            const NaPair& T = S->pair[q];
            const double x0 = T.t[1] * ga2 - T.t[2] * ga1 - gb0, x1 = T.t[2] * ga0 - T.t[0] * ga2 - gb1,
                         x2 = T.t[0] * ga1 - T.t[1] * ga0 - gb2;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              g[k] -= T.R[k] * ga0 + T.R[3 + k] * ga1 + T.R[6 + k] * ga2;
              g[3 + k] += T.R[k] * x0 + T.R[3 + k] * x1 + T.R[6 + k] * x2;
            }
          } else {
            g[0] += ga0;
            g[1] += ga1;
            g[2] += ga2;
            g[3] += gb0;
            g[4] += gb1;
            g[5] += gb2;
          }
        }
      }
      __syncwarp();
      waiting -= take;
      int moved[2];  // the rest moves to the front
      for (int k = 0; k < 2; ++k) moved[k] = lane + 32 * k < waiting ? ent[take + lane + 32 * k] : 0;
      __syncwarp();
      for (int k = 0; k < 2; ++k)
        if (lane + 32 * k < waiting) ent[lane + 32 * k] = moved[k];
      __syncwarp();
    }
  }
  if (!waited) epo::griddep_wait();  // no entry: the next kernel still follows the whole chain
  // fixed-order reduce-scatter over the warp: value k ends in the four lanes 4k .. 4k + 3
  {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    double k4[4], k2[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) k4[k] = (b4 ? g[4 + k] : g[k]) + __shfl_xor_sync(0xffffffffu, b4 ? g[k] : g[4 + k], 16);
#pragma unroll
    for (int k = 0; k < 2; ++k) k2[k] = (b3 ? k4[2 + k] : k4[k]) + __shfl_xor_sync(0xffffffffu, b3 ? k4[k] : k4[2 + k], 8);
    double s = (b2 ? k2[1] : k2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? k2[0] : k2[1], 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (vv && (lane & 3) == 0 && lane < 24) grad[6 * (size_t)v + (lane >> 2)] = s;
  }
}

}  // namespace

extern "C" epo_status epo_loss_and_grad_noalloc(const epo_noalloc_problem* pb, double* loss_dev,
                                                double* grad_dev, void* cuda_stream) {
  if (!pb || !loss_dev || !grad_dev) return EPO_ERR_INVALID_ARG;
  if (!pb->records || !pb->rec_off || !pb->maps || !pb->map_off || !pb->W || !pb->H || !pb->K || !pb->pairs ||
      !pb->T)
    return EPO_ERR_INVALID_ARG;
  if (pb->n_views < 1 || pb->n_pairs < 1 || pb->max_records_per_view < 0)
    return EPO_ERR_INVALID_ARG;
  // the kernels read records as 16-byte vectors and the other arrays at their natural width:
  // a misaligned pointer would fault on the device, so it is refused here
  if ((uintptr_t)pb->records % 16 != 0 || (uintptr_t)pb->rec_off % 8 != 0 || (uintptr_t)pb->maps % 4 != 0 ||
      (uintptr_t)pb->map_off % 8 != 0 || (uintptr_t)pb->W % 4 != 0 || (uintptr_t)pb->H % 4 != 0 ||
      (uintptr_t)pb->K % 8 != 0 || (uintptr_t)pb->pairs % 4 != 0 || (uintptr_t)pb->T % 8 != 0 ||
      (uintptr_t)loss_dev % 8 != 0 || (uintptr_t)grad_dev % 8 != 0)
    return EPO_ERR_INVALID_ARG;
  // one block per tile of kNaThreads records of a view: the tile count is the grid's x extent
  if ((pb->max_records_per_view + kNaThreads - 1) / kNaThreads > (int64_t)INT32_MAX) return EPO_ERR_TOO_LARGE;
  if (pb->n_views > kNaMaxViews || pb->n_pairs > kNaMaxPairs)
    return EPO_ERR_TOO_LARGE;
  if (!(pb->lambda > 0) || !(pb->huber_delta > 0) || !(pb->eps_z >= 0) ||
      (pb->norm_mode != EPO_NORM_VALID && pb->norm_mode != EPO_NORM_ALL))
    return EPO_ERR_INVALID_ARG;
  // the scratch array's device address, resolved once per device with that device current
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return EPO_ERR_CUDA;
  if (dev < 0 || dev >= kNaMaxDevices) return EPO_ERR_INVALID_ARG;
  NaScratch* S = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_ptr[dev]) {
      void* ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
      if (e != cudaSuccess) return EPO_ERR_CUDA;
      g_scratch_ptr[dev] = reinterpret_cast<NaScratch*>(ptr);
    }
    S = g_scratch_ptr[dev];
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const epo_noalloc_problem prob = *pb;
  // each kernel may start while its predecessor ends (programmatic dependent launch) and waits for
  // it before it reads the scratch
  k_na_setup<<<(prob.n_pairs * 16 + kNaSetupThreads - 1) / kNaSetupThreads, kNaSetupThreads, 0, st>>>(prob, S);
  e = cudaGetLastError();
  const int tiles = (int)((prob.max_records_per_view + kNaThreads - 1) / kNaThreads);
  if (e == cudaSuccess && tiles > 0) {
    const int per_pair = std::min(tiles, std::max(1, kNaEdgeBlocks / prob.n_pairs));
    e = epo::launch_pdl(k_na_edge, dim3(per_pair, prob.n_pairs), dim3(kNaThreads), 0, st, prob, S);
  }
  if (e == cudaSuccess)
    e = epo::launch_pdl(k_na_finish, dim3(1 + (prob.n_views + kNaFinViews - 1) / kNaFinViews), dim3(kNaFinThreads), 0, st,
                        prob, (const NaScratch*)S, loss_dev, grad_dev);
  if (e != cudaSuccess) return EPO_ERR_CUDA;
  return EPO_OK;
}
