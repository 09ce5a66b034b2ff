// The paper's pose parameterisation (Section 3, Pose Refinement, Eq. 3) on the device:
//
//     P_i^s = phi(P_i^0 + MLP(P_i^0)) + [0 | delta_i]
//
// with a six-layer MLP of hidden width 128 (ReLU after the first five layers, the first
// layer's output added to the third's), phi = Gram-Schmidt on the 6D representation (the first
// two columns of the 3x3 block), one MLP per scene and one translation offset delta_i per view,
// trained by AdamW with a linear warm-up and cosine decay of the learning rate (Implementation
// Details).  The parameterisation acts on the scene at unit scale: with s the RMS spread of the
// P^0 camera centres, the MLP sees the translations divided by s, and its translation output and
// delta are multiplied by s (the paper's inputs are normalised foundation-model outputs).  A step in this mode is: the fused pass and the pose kernel's gradient G_i (the
// left-perturbation gradient of the objective at P^s), then
//   k_mlp_backward  one block per view: G_i -> derivatives of the pose entries (FP64), through
//                   phi (FP64, one thread) and the MLP's layers (FP32, one column per thread);
//   k_mlp_update    one block per four outputs of a layer: the gradient summed over the scene's views
//                   in a fixed order, AdamW; the last block advances the step counter;
//   k_mlp_forward   one block per view: the next poses P^{s+1} (MLP in FP32, phi and the pose
//                   in FP64) and the activations the next backward needs.
// The MLP is tiny (69 k parameters, one 128-wide mat-vec per layer and view): these are latency
// kernels, not contractions worth the tensor cores.  The two per-view kernels copy the weights into
// shared memory with cp.async, all but one of the hidden layers at once, so that the layers wait for
// one trip to L2 and not for one each; backward starts them while the pose kernel still runs
// (programmatic launch) and forms the FP64 part meanwhile.  32 views, one scene, warm caches:
// forward 29-32 -> 12.6 us, backward 19.6 -> 14.6 (its roots run before the wait, beside the pose kernel),
// update 17 -> 8; a step with its read-backs 172 -> 131.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "epo_internal.cuh"

namespace epo {

namespace {

constexpr int H = kMlpHid;
// offsets of W_l and b_l (l = 0..5) in a scene's parameter vector
__host__ __device__ constexpr int mlp_in(int l) { return l == 0 ? 12 : H; }
__host__ __device__ constexpr int mlp_out(int l) { return l == 5 ? 12 : H; }
__host__ __device__ constexpr int mlp_w(int l) {
  int o = 0;
  for (int k = 0; k < l; ++k) o += mlp_out(k) * mlp_in(k) + mlp_out(k);
  return o;
}
__host__ __device__ constexpr int mlp_b(int l) { return mlp_w(l) + mlp_out(l) * mlp_in(l); }
static_assert(mlp_w(6) == kMlpParams, "pose MLP layout");
__device__ __forceinline__ int mlp_b_at(int l) {  // mlp_b for a layer known at run time
  return l == 0 ? mlp_b(0) : (l == 5 ? mlp_b(5) : mlp_b(1) + (l - 1) * (H * H + H));
}

// ---- staging of the weights in shared memory ----
// A layer's W and b are contiguous; every offset is a multiple of 16 bytes.
constexpr int kLayerFloats = H * H + H;              // a hidden layer
constexpr int kInFloats = 12 * H + H, kOutFloats = 12 * H + 12;
static_assert(kMlpParams % 4 == 0 && kLayerFloats % 4 == 0 && kInFloats % 4 == 0 && kOutFloats % 4 == 0, "16-byte copies");
constexpr int kMlpThreads = 512;
struct MlpStage {
  float hid[3][kLayerFloats];  // three of the four hidden layers; the fourth follows the first one used
  float in[kInFloats], out[kOutFloats];
};

__device__ __forceinline__ void stage(float* dst, const float* src, int floats) {
  for (int k = threadIdx.x; k < floats / 4; k += blockDim.x) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst + 4 * k);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + 4 * k) : "memory");
  }
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>  // until at most the N youngest groups are in flight
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// x / d of a warp-uniform vector x: one division for the three (an FP64 instruction costs a warp the
// same for one lane as for 32).  Every lane calls it.
__device__ __forceinline__ void div3(const double* x, double d, double* q, int lane) {
  const double y = (lane == 0 ? x[0] : (lane == 1 ? x[1] : x[2])) / d;
#pragma unroll
  for (int r = 0; r < 3; ++r) q[r] = __shfl_sync(0xffffffffu, y, r);
}

// Sums of 8 values over a warp, the butterfly over lane distances 16, 8, 4, 2, 1 as a reduce-scatter:
// lane L ends with value L >> 2.
__device__ __forceinline__ float warp_sums8(const float* v, int lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  float k4[4], k2[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) k4[k] = (b4 ? v[4 + k] : v[k]) + __shfl_xor_sync(0xffffffffu, b4 ? v[k] : v[4 + k], 16);
#pragma unroll
  for (int k = 0; k < 2; ++k) k2[k] = (b3 ? k4[2 + k] : k4[k]) + __shfl_xor_sync(0xffffffffu, b3 ? k4[k] : k4[2 + k], 8);
  float r = (b2 ? k2[1] : k2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? k2[0] : k2[1], 4);
  r += __shfl_xor_sync(0xffffffffu, r, 2);
  return r + __shfl_xor_sync(0xffffffffu, r, 1);
}

__device__ __forceinline__ double dot3(const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
__device__ __forceinline__ void cross3(const double* a, const double* b, double* c) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}

// phi: Gram-Schmidt on the first two columns a1, a2 of a 3x4 matrix P, b1 = a1 / n1, b2 = u2 / n2 with
// u2 = a2 - c b1, c = b1 . a2.  Warp-uniform; every lane calls it.
struct Phi {
  double a2[3], b1[3], b2[3], n1, n2, c;
};
__device__ __forceinline__ void gram_schmidt(const double* P, Phi& f, int lane) {
  const double a1[3] = {P[0], P[4], P[8]};
  f.n1 = sqrt(dot3(a1, a1));
  div3(a1, f.n1, f.b1, lane);
  double u2[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) f.a2[r] = P[4 * r + 1];
  f.c = dot3(f.b1, f.a2);
#pragma unroll
  for (int r = 0; r < 3; ++r) u2[r] = f.a2[r] - f.c * f.b1[r];
  f.n2 = sqrt(dot3(u2, u2));
  div3(u2, f.n2, f.b2, lane);
}

}  // namespace

// ------------------------------------------------------------------------------------------
// forward: P^s from the current parameters
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kMlpThreads) k_mlp_forward(StepArgs a, int change) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  MlpStage& st = *reinterpret_cast<MlpStage*>(s_raw);
  __shared__ float s_x[12], s_a[2][H], s_a1[H], s_y[12];
  __shared__ double s_Pp[12], s_T[12];
  __shared__ int s_ok;
  const int v = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sc = a.views[v].scene;
  const float* th = a.mlp_theta + (size_t)sc * kMlpParams;
  griddep_launch_dependents();
  griddep_wait();  // the weights
  stage(st.in, th + mlp_w(0), kInFloats);
  stage(st.out, th + mlp_w(5), kOutFloats);
  stage_commit();
  for (int l = 1; l <= 3; ++l) {
    stage(st.hid[l - 1], th + mlp_w(l), kLayerFloats);
    stage_commit();
  }
  const double sc_s = a.mlp_scale[sc];
  if (tid < 12) {
    const float xv = (float)(a.mlp_P0[12 * (size_t)v + tid] / ((tid & 3) == 3 ? sc_s : 1.0));
    s_x[tid] = xv;
    a.mlp_x[12 * (size_t)v + tid] = xv;
  }
  stage_wait<3>();
  __syncthreads();
  float* zs = a.mlp_z + (size_t)v * 5 * H;
  if (tid < H) {
    float z = st.in[12 * H + tid];
#pragma unroll
    for (int k = 0; k < 12; ++k) z = fmaf(st.in[tid * 12 + k], s_x[k], z);
    zs[tid] = z;
    s_a[0][tid] = s_a1[tid] = fmaxf(z, 0.f);
  }
  // hidden layers: each of the 16 warps forms eight outputs, lane l summing the columns l, l + 32,
  // l + 64, l + 96 and the lanes by shuffles
#pragma unroll
  for (int l = 1; l <= 4; ++l) {
    // in flight behind this layer: 2, 3 at the first; 3 at the second; the fourth at the third
    if (l == 1) stage_wait<2>();
    else if (l <= 3) stage_wait<1>();
    else stage_wait<0>();
    __syncthreads();
    if (l == 2) {  // every warp is past layer 1: its buffer takes the fourth
      stage(st.hid[0], th + mlp_w(4), kLayerFloats);
      stage_commit();
    }
    const float* W = st.hid[(l - 1) % 3];
    const float* x = s_a[(l - 1) & 1];
    const float a0 = x[lane], a1 = x[lane + 32], a2 = x[lane + 64], a3 = x[lane + 96];
    float acc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float* Wr = W + (8 * warp + u) * H;
      acc[u] = fmaf(Wr[lane], a0, fmaf(Wr[lane + 32], a1, fmaf(Wr[lane + 64], a2, Wr[lane + 96] * a3)));
    }
    const float sum = warp_sums8(acc, lane);
    if ((lane & 3) == 0) {
      const int o = 8 * warp + (lane >> 2);
      const float z = W[H * H + o] + sum;
      zs[l * H + o] = z;
      float h = fmaxf(z, 0.f);
      if (l == 2) h += s_a1[o];  // the skip connection after the third layer
      s_a[l & 1][o] = h;
    }
  }
  __syncthreads();
  if (warp < 12) {  // output layer: one output per warp
    const float* Wr = st.out + warp * H;
    const float* x = s_a[0];
    float acc = fmaf(Wr[lane], x[lane], fmaf(Wr[lane + 32], x[lane + 32], fmaf(Wr[lane + 64], x[lane + 64], Wr[lane + 96] * x[lane + 96])));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) s_y[warp] = st.out[12 * H + warp] + acc;
  }
  __syncthreads();
  if (warp != 0) return;
  // P' = P^0 + MLP(P^0), one entry per lane
  if (lane < 12) {
    const double Pp = a.mlp_P0[12 * (size_t)v + lane] + ((lane & 3) == 3 ? sc_s : 1.0) * (double)s_y[lane];
    s_Pp[lane] = Pp;
    a.mlp_Pp[12 * (size_t)v + lane] = Pp;
  }
  __syncwarp();
  double* Ts = a.T_store + 12 * (size_t)v;
  Phi f;
  gram_schmidt(s_Pp, f, lane);
  if (lane == 0) {
    // the pose: phi's columns and the offset delta (FP64)
    const double* Pp = s_Pp;
    double b3[3];
    cross3(f.b1, f.b2, b3);
    bool finite = true;
    for (int r = 0; r < 3; ++r) {
      s_T[4 * r] = f.b1[r];
      s_T[4 * r + 1] = f.b2[r];
      s_T[4 * r + 2] = b3[r];
      s_T[4 * r + 3] = Pp[4 * r + 3] + sc_s * (double)a.mlp_delta[3 * (size_t)v + r];
    }
    for (int k = 0; k < 12; ++k) finite = finite && isfinite(s_T[k]);
    s_ok = finite;
    if (!finite) atomicOr(a.flag, 1);  // the poses stay; the host reports the step as refused
  }
  __syncwarp();
  if (!s_ok) return;
  if (change && a.schedule && lane == 0) {
    // the step's pose change (Section 3, Optimization Schedule), as the pose kernel forms it
    const double* T = s_T;
    double tr = 0.0, dot = 0.0, nn = 0.0, no = 0.0;
    for (int r = 0; r < 3; ++r) {
      for (int cc = 0; cc < 3; ++cc) tr += T[4 * r + cc] * Ts[4 * r + cc];
      dot += T[4 * r + 3] * Ts[4 * r + 3];
      nn += T[4 * r + 3] * T[4 * r + 3];
      no += Ts[4 * r + 3] * Ts[4 * r + 3];
    }
    const double deg = 180.0 / 3.14159265358979323846;
    a.pose_dR[v] = deg * acos(fmin(1.0, fmax(-1.0, (tr - 1.0) * 0.5)));
    const double nm = sqrt(nn) * sqrt(no);
    a.pose_dt[v] = nm > 0.0 ? deg * acos(fmin(1.0, fmax(-1.0, dot / nm))) : 0.0;
  }
  __syncwarp();  // the old pose has been read
  if (lane < 12) Ts[lane] = s_T[lane];
}

// ------------------------------------------------------------------------------------------
// backward: dL/dz of every layer and dL/ddelta of every view
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kMlpThreads) k_mlp_backward(StepArgs a) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  MlpStage& st = *reinterpret_cast<MlpStage*>(s_raw);
  __shared__ float s_dy[12];
  __shared__ __align__(16) float s_dz[2][H];
  const int v = blockIdx.x, j = threadIdx.x;
  const int sc = a.views[v].scene;
  const float* th = a.mlp_theta + (size_t)sc * kMlpParams;
  griddep_launch_dependents();
  // the weights and activations are the last step's: their loads overlap the pose kernel
  stage(st.out, th + mlp_w(5), kOutFloats);
  stage_commit();
  for (int l = 4; l >= 2; --l) {
    stage(st.hid[4 - l], th + mlp_w(l), kLayerFloats);
    stage_commit();
  }
  float z[5] = {};
  if (j < H) {
    const float* zs = a.mlp_z + (size_t)v * 5 * H;
#pragma unroll
    for (int l = 0; l < 5; ++l) z[l] = zs[l * H + j];
  }
  Phi f;
  if (j < 32) gram_schmidt(a.mlp_Pp + 12 * (size_t)v, f, j);
  griddep_wait();  // the poses' gradient
  if (j < 32) {
    // G = (g_v, g_w) at T = P^s: dL/dt = g_v, and (for the tangent dR = [w]x R that phi
    // produces) dL/dR = 1/2 [g_w + g_v x t]x R; then back through Gram-Schmidt (FP64)
    const double* G = a.grad + 6 * (size_t)v;
    const double* T = a.T_store + 12 * (size_t)v;
    const double gv[3] = {G[0], G[1], G[2]}, t[3] = {T[3], T[7], T[11]};
    double w[3];
    cross3(gv, t, w);
    for (int r = 0; r < 3; ++r) w[r] = 0.5 * (w[r] + G[3 + r]);
    const double r1[3] = {T[0], T[4], T[8]}, r2[3] = {T[1], T[5], T[9]}, r3[3] = {T[2], T[6], T[10]};
    // columns of dL/dR = [w]x R
    double g1[3], g2[3], g3[3];
    cross3(w, r1, g1);
    cross3(w, r2, g2);
    cross3(w, r3, g3);
    double x[3];
    cross3(f.b2, g3, x);  // b3 = b1 x b2
    for (int r = 0; r < 3; ++r) g1[r] += x[r];
    cross3(g3, f.b1, x);
    for (int r = 0; r < 3; ++r) g2[r] += x[r];
    const double p2 = dot3(g2, f.b2);  // b2 = u2 / n2
    double gu2[3], ga1[3], ga2[3];
    for (int r = 0; r < 3; ++r) x[r] = g2[r] - p2 * f.b2[r];
    div3(x, f.n2, gu2, j);
    const double q = dot3(gu2, f.b1);  // u2 = a2 - (b1 . a2) b1
    for (int r = 0; r < 3; ++r) {
      ga2[r] = gu2[r] - q * f.b1[r];
      g1[r] -= q * f.a2[r] + f.c * gu2[r];
    }
    const double p1 = dot3(g1, f.b1);  // b1 = a1 / n1
    for (int r = 0; r < 3; ++r) x[r] = g1[r] - p1 * f.b1[r];
    div3(x, f.n1, ga1, j);
    if (j == 0) {
      for (int r = 0; r < 3; ++r) {
        s_dy[4 * r] = (float)ga1[r];
        s_dy[4 * r + 1] = (float)ga2[r];
        s_dy[4 * r + 2] = 0.f;  // the third column does not reach phi
        s_dy[4 * r + 3] = (float)(a.mlp_scale[sc] * gv[r]);  // the translation output is scaled by s
        a.mlp_gdelta[3 * (size_t)v + r] = s_dy[4 * r + 3];
      }
    }
  }
  stage_wait<3>();
  __syncthreads();
  float* dz = a.mlp_dz + (size_t)v * kMlpDz;
  if (j < 12) dz[5 * H + j] = s_dy[j];
  if (j < H) {
    // dL/da_5 = W6^T dy, then through the ReLU of layer 5
    float da = 0.f;
#pragma unroll
    for (int o = 0; o < 12; ++o) da = fmaf(st.out[o * H + j], s_dy[o], da);
    const float d = z[4] > 0.f ? da : 0.f;
    dz[4 * H + j] = d;
    s_dz[0][j] = d;
  }
  float dskip = 0.f;
#pragma unroll
  for (int l = 4; l >= 1; --l) {
    // in flight behind this layer: 3, 2 at the fourth; 2 at the third; the first at the second
    if (l == 4) stage_wait<2>();
    else if (l >= 2) stage_wait<1>();
    else stage_wait<0>();
    __syncthreads();
    if (l == 3) {  // every thread is past layer 4: its buffer takes the first hidden layer
      stage(st.hid[0], th + mlp_w(1), kLayerFloats);
      stage_commit();
    }
    if (j < H) {
      const float* W = st.hid[(4 - l) % 3];
      const float4* d4 = reinterpret_cast<const float4*>(s_dz[(4 - l) & 1]);
      float da = 0.f;
#pragma unroll 8
      for (int i = 0; i < H / 4; ++i) {  // (W_l^T dz_l)_j
        const float4 d = d4[i];
        da = fmaf(W[(4 * i) * H + j], d.x, da);
        da = fmaf(W[(4 * i + 1) * H + j], d.y, da);
        da = fmaf(W[(4 * i + 2) * H + j], d.z, da);
        da = fmaf(W[(4 * i + 3) * H + j], d.w, da);
      }
      if (l == 3) dskip = da;  // a_3 = relu(z_2) + a_1
      if (l == 1) da += dskip;
      const float d = z[l - 1] > 0.f ? da : 0.f;
      dz[(l - 1) * H + j] = d;
      s_dz[(5 - l) & 1][j] = d;
    }
  }
}

// ------------------------------------------------------------------------------------------
// AdamW on theta and delta (a scene whose schedule has converged keeps them); the last block
// advances the step counter
// ------------------------------------------------------------------------------------------
constexpr int kMlpUpdThreads = 256;

__device__ __forceinline__ float adamw_delta(float p, float g, float& m, float& v, float b1, float b2, float c1, float c2,
                                             float lr, float wd, float eps) {
  m = b1 * m + (1.f - b1) * g;
  v = b2 * v + (1.f - b2) * g * g;
  return p * (1.f - lr * wd) - lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// Blocks of one scene: kMlpTiles tiles of kMlpTileOut outputs x 128 inputs (the hidden layers and the
// output layer), whose views' derivatives and inputs go through shared memory, then kMlpRest blocks
// with one parameter per thread (the first layer's weights and every bias); after all scenes, the
// offsets delta.
constexpr int kMlpTileOut = 4;
constexpr int kMlpTiles = (4 * H + 12) / kMlpTileOut;
constexpr int kMlpRestParams = 12 * H + 5 * H + 12;
constexpr int kMlpRest = (kMlpRestParams + kMlpUpdThreads - 1) / kMlpUpdThreads;
constexpr int kMlpUpdViews = 32;  // views staged at a time
static_assert(kMlpUpdThreads == 2 * H && kMlpTileOut == 4, "two outputs per thread");

__global__ void __launch_bounds__(kMlpUpdThreads) k_mlp_update(StepArgs a) {
  __shared__ float s_in[kMlpUpdViews][H];
  __shared__ float4 s_d[kMlpUpdViews];  // the tile's four outputs
  griddep_launch_dependents();
  const int64_t step = *a.step;
  // learning rate of the step: linear warm-up to mlp_lr, then cosine decay to 0
  float lr;
  if (step < a.mlp_warmup) {
    lr = a.mlp_lr * (float)(step + 1) / (float)a.mlp_warmup;
  } else {
    const int64_t span = max(a.mlp_steps - a.mlp_warmup, 1);
    const float t = (float)min(step - a.mlp_warmup + 1, span) / (float)span;
    lr = a.mlp_lr * 0.5f * (1.f + cospif(t));
  }
  const float fs = (float)(step + 1);
  const float c1 = -expm1f(fs * a.log_beta1), c2 = -expm1f(fs * a.log_beta2);
  const float b1 = (float)a.beta1, b2 = (float)a.beta2;
  const auto converged = [&](int sc) { return a.schedule && a.sched_state[2 * sc] == 3; };
  const int sc = blockIdx.x / (kMlpTiles + kMlpRest), item = blockIdx.x % (kMlpTiles + kMlpRest);
  bool refused = false;
  if (sc < a.n_scenes) {
    const int v0 = a.scene_view_off[sc], v1 = a.scene_view_off[sc + 1];
    const size_t base = (size_t)sc * kMlpParams;
    if (item < kMlpTiles) {
      const int o_all = item * kMlpTileOut;  // outputs of layers 1 .. 5 in a row
      const int l = min(1 + o_all / H, 5), o0 = o_all - (l - 1) * H;
      const int i = threadIdx.x % H, half = threadIdx.x / H;
      const size_t k0 = base + mlp_w(1) + (size_t)(l - 1) * kLayerFloats + (size_t)(o0 + 2 * half) * H + i;  // and the next output's, H further
      float p[2], m[2], vv[2], g[2] = {0.f, 0.f};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        p[u] = a.mlp_theta[k0 + u * H];
        m[u] = a.mlp_m[k0 + u * H];
        vv[u] = a.mlp_v[k0 + u * H];
      }
      griddep_wait();  // the derivatives
      refused = (*a.flag & 1) != 0;
      const bool skip = refused || converged(sc);
      for (int vb = v0; vb < v1 && !skip; vb += kMlpUpdViews) {
        const int nv = min(kMlpUpdViews, v1 - vb);
        if (vb > v0) __syncthreads();
#pragma unroll 8
        for (int e = threadIdx.x; e < nv * H; e += kMlpUpdThreads) {
          const int v = e / H, k = e % H;
          const float* zs = a.mlp_z + (size_t)(vb + v) * 5 * H;
          float in = fmaxf(zs[(l - 1) * H + k], 0.f);
          if (l == 3) in += fmaxf(zs[k], 0.f);  // the skip
          s_in[v][k] = in;
        }
        if (threadIdx.x < nv * kMlpTileOut)
          reinterpret_cast<float*>(s_d)[threadIdx.x] =
              a.mlp_dz[(size_t)(vb + threadIdx.x / kMlpTileOut) * kMlpDz + l * H + o0 + threadIdx.x % kMlpTileOut];
        __syncthreads();
#pragma unroll 8
        for (int v = 0; v < nv; ++v) {
          const float in = s_in[v][i];
          const float4 d = s_d[v];
          g[0] = fmaf(half ? d.z : d.x, in, g[0]);
          g[1] = fmaf(half ? d.w : d.y, in, g[1]);
        }
      }
      if (!skip) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          a.mlp_theta[k0 + u * H] = adamw_delta(p[u], g[u], m[u], vv[u], b1, b2, c1, c2, lr, a.mlp_wd, a.mlp_eps);
          a.mlp_m[k0 + u * H] = m[u];
          a.mlp_v[k0 + u * H] = vv[u];
        }
      }
    } else {
      // first layer's weights, then the biases of layers 0 .. 5
      const int r = (item - kMlpTiles) * kMlpUpdThreads + threadIdx.x;
      const bool bias = r >= 12 * H;
      const int l = bias ? min((r - 12 * H) / H, 5) : 0;
      const int o = bias ? r - 12 * H - l * H : r / 12, i = bias ? 0 : r % 12;
      griddep_wait();
      refused = (*a.flag & 1) != 0;
      if (r < kMlpRestParams && !refused && !converged(sc)) {
        float grad = 0.f;
#pragma unroll 16
        for (int v = v0; v < v1; ++v) {
          const float d = a.mlp_dz[(size_t)v * kMlpDz + l * H + o];
          grad = fmaf(d, bias ? 1.f : a.mlp_x[12 * (size_t)v + i], grad);
        }
        const size_t k = base + (bias ? mlp_b_at(l) + o : mlp_w(0) + r);
        a.mlp_theta[k] = adamw_delta(a.mlp_theta[k], grad, a.mlp_m[k], a.mlp_v[k], b1, b2, c1, c2, lr, a.mlp_wd, a.mlp_eps);
      }
    }
  } else {
    griddep_wait();
    refused = (*a.flag & 1) != 0;
    const int64_t k = (int64_t)(blockIdx.x - (unsigned)a.n_scenes * (kMlpTiles + kMlpRest)) * kMlpUpdThreads + threadIdx.x;
    if (k < 3 * (int64_t)a.n_views && !refused && !converged(a.views[k / 3].scene))
      a.mlp_delta[k] = adamw_delta(a.mlp_delta[k], a.mlp_gdelta[k], a.mlp_dm[k], a.mlp_dv[k], b1, b2, c1, c2, lr,
                                   a.mlp_wd_delta, a.mlp_eps);
  }
  // the last block to finish advances the step counter and the beta powers (read by the
  // focal Adam of refine scenes).  The decision rests on the flag every block read, and every
  // block has used its step count before it reports, so the count needs no fence
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int prev = atomicAdd(a.mlp_done, 1u);
    if (prev == gridDim.x - 1) {
      if (!refused) {
        *a.step = step + 1;
        a.bpow[0] *= a.beta1;
        a.bpow[1] *= a.beta2;
      }
      *a.mlp_done = 0u;
    }
  }
}

template <typename K, typename... Args>
static cudaError_t launch_staged(K kernel, int blocks, cudaStream_t s, Args... args) {
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpStage));
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(blocks), dim3(kMlpThreads), sizeof(MlpStage), s, args...);
}

cudaError_t launch_mlp_forward(const StepArgs& a, int change, cudaStream_t s) {
  if (a.n_views <= 0) return cudaSuccess;
  return launch_staged(k_mlp_forward, a.n_views, s, a, change);
}

cudaError_t launch_mlp_backward(const StepArgs& a, cudaStream_t s) {
  if (a.n_views <= 0) return cudaSuccess;
  return launch_staged(k_mlp_backward, a.n_views, s, a);
}

cudaError_t launch_mlp_update(const StepArgs& a, cudaStream_t s) {
  const int64_t n = (int64_t)a.n_scenes * (kMlpTiles + kMlpRest) + (3 * (int64_t)a.n_views + kMlpUpdThreads - 1) / kMlpUpdThreads;
  return launch_pdl(k_mlp_update, dim3((unsigned)n), dim3(kMlpUpdThreads), 0, s, a);
}

}  // namespace epo
