// Learned control variate: per-node features, a 14-64-64-1 GELU MLP with
// BF16 weights and FP32 accumulation (forward, backward, Adam) and the
// qsel_cv object of the C ABI.
//
// The network predicts log(c_i / v_i), the relative Rao-Blackwell correction
// of node i (Algorithm 4: v_i = Sigma*_ii + c_i).  A planner (qsel_cv_plan in
// api.cu) uses it to choose the overlap and the number of samples; the
// estimate itself stays plain RBMC.
//
// Parameter vector (FP32 master copy): W1 (64 x 14), b1 (64), W2 (64 x 64),
// b2 (64), W3 (64), b3 (1) = 5185 values, then the input mean (14) and scale
// (14).  The forward pass reads BF16 copies of W1, W2, W3.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "qsel.h"
#include "kernels.cuh"

namespace qsel {
namespace mlp {

constexpr int NF = QSEL_CV_FEATURES;   // 14
constexpr int H = 64;
constexpr int OFF_W1 = 0, OFF_B1 = H * NF, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H, OFF_W3 = OFF_B2 + H,
              OFF_B3 = OFF_W3 + H, N_TRAIN = OFF_B3 + 1, OFF_MU = N_TRAIN, OFF_SC = OFF_MU + NF,
              N_ALL = OFF_SC + NF;
static_assert(N_TRAIN == QSEL_CV_PARAMS, "parameter count");
constexpr int TILE = 64;   // samples per backward CTA

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }

// {a.x b.x + c.x, a.y b.y + c.y}, each rounded once: one issue slot for two FMAs.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<uint64_t &>(d))
      : "l"(reinterpret_cast<uint64_t &>(a)), "l"(reinterpret_cast<uint64_t &>(b)),
        "l"(reinterpret_cast<uint64_t &>(c)));
  return d;
}

struct Weights {
  const __nv_bfloat16 *w1, *w2, *w3;
  const float *p;   // master parameters: biases, mean, scale
};

// Weights (input unit first), biases, mean and scale staged in shared memory as
// float.
struct __align__(16) SmemW {
  float w1[NF][H], w2[H][H], b1[H], b2[H], w3[H], b3, mu[NF], sc[NF];
};

__device__ void stage_weights(const Weights &W, SmemW &s) {
  for (int i = threadIdx.x; i < H * NF; i += blockDim.x) s.w1[i / H][i % H] = __bfloat162float(W.w1[(i % H) * NF + i / H]);
  for (int i = threadIdx.x; i < H * H; i += blockDim.x) s.w2[i / H][i % H] = __bfloat162float(W.w2[(i % H) * H + i / H]);
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    s.w3[i] = __bfloat162float(W.w3[i]);
    s.b1[i] = W.p[OFF_B1 + i];
    s.b2[i] = W.p[OFF_B2 + i];
  }
  for (int i = threadIdx.x; i < NF; i += blockDim.x) {
    s.mu[i] = W.p[OFF_MU + i];
    s.sc[i] = W.p[OFF_SC + i];
  }
  if (threadIdx.x == 0) s.b3 = W.p[OFF_B3];
  __syncthreads();
}

// S samples per thread.  With act set, a1 and a2 are stored (training).
//
// What bounds it: issue slots -- FMAs, the shared-memory reads that feed them and the
// two error functions per unit.  The first layer's output goes through shared memory
// (h1[unit][sample]; a thread reads what it wrote), so that both layers run as loops
// over 16 units: kept in registers, the 64 units had to be unrolled, and every weight
// was read once per sample and FMA.  A 16-byte read now serves 4 S FMAs, issued in
// pairs; every sum keeps its order.  Measured, 524288 samples: 311 -> 178 us
// (8 or 32 units: 191, 179; one sample per thread: 200); 65000 with act: 74 -> 36 us.
template <int S>
__host__ __device__ constexpr int forward_smem() {
  return (int)sizeof(SmemW) + H * 256 * S * 4;
}

template <int S>
__global__ void __launch_bounds__(256) k_mlp_forward(Weights W, const float *__restrict__ X, int n,
                                                     float *__restrict__ y, float *__restrict__ act) {
  extern __shared__ __align__(16) unsigned char smem_f[];
  SmemW &s = *reinterpret_cast<SmemW *>(smem_f);
  float *h1s = reinterpret_cast<float *>(smem_f + sizeof(SmemW));   // [H][256 S]
  stage_weights(W, s);
  const bool pairs = (reinterpret_cast<uintptr_t>(X) & 7) == 0;   // a caller's rows may start on 4 bytes
  constexpr int B = 16;   // units at a time
  for (int64_t s0 = (int64_t)blockIdx.x * 256 * S; s0 < n; s0 += (int64_t)gridDim.x * 256 * S) {
    float xn[S][NF];
    float out[S];
#pragma unroll
    for (int q = 0; q < S; ++q) {
      const int64_t smp = min(s0 + q * 256 + threadIdx.x, (int64_t)n - 1);
#pragma unroll
      for (int k = 0; k < NF; k += 2) {
        const float *x = X + smp * NF + k;
        const float2 v = pairs ? *reinterpret_cast<const float2 *>(x) : make_float2(x[0], x[1]);
        xn[q][k] = (v.x - s.mu[k]) / s.sc[k];
        xn[q][k + 1] = (v.y - s.mu[k + 1]) / s.sc[k + 1];
      }
      out[q] = s.b3;
    }
#pragma unroll 1
    for (int j = 0; j < H; j += B) {
      float2 a[S][B / 2];
#pragma unroll
      for (int q = 0; q < S; ++q)
#pragma unroll
        for (int u = 0; u < B / 2; ++u) a[q][u] = make_float2(s.b1[j + 2 * u], s.b1[j + 2 * u + 1]);
#pragma unroll
      for (int k = 0; k < NF; ++k) {
        float2 w[B / 2];
#pragma unroll
        for (int u = 0; u < B / 2; u += 2)
          *reinterpret_cast<float4 *>(w + u) = *reinterpret_cast<const float4 *>(&s.w1[k][j + 2 * u]);
#pragma unroll
        for (int q = 0; q < S; ++q)
#pragma unroll
          for (int u = 0; u < B / 2; ++u) a[q][u] = fma2(w[u], make_float2(xn[q][k], xn[q][k]), a[q][u]);
      }
#pragma unroll
      for (int q = 0; q < S; ++q) {
        const int64_t smp = s0 + q * 256 + threadIdx.x;
        if (act && smp < n) {
#pragma unroll
          for (int u = 0; u < B / 2; u += 2)
            *reinterpret_cast<float4 *>(act + smp * 2 * H + j + 2 * u) =
                make_float4(a[q][u].x, a[q][u].y, a[q][u + 1].x, a[q][u + 1].y);
        }
#pragma unroll
        for (int u = 0; u < B / 2; ++u) {
          h1s[(j + 2 * u) * 256 * S + q * 256 + threadIdx.x] = gelu(a[q][u].x);
          h1s[(j + 2 * u + 1) * 256 * S + q * 256 + threadIdx.x] = gelu(a[q][u].y);
        }
      }
    }
    // a thread reads its own samples' units only
#pragma unroll 1
    for (int j = 0; j < H; j += B) {
      float2 a[S][B / 2];
#pragma unroll
      for (int q = 0; q < S; ++q)
#pragma unroll
        for (int u = 0; u < B / 2; ++u) a[q][u] = make_float2(s.b2[j + 2 * u], s.b2[j + 2 * u + 1]);
#pragma unroll 8
      for (int k = 0; k < H; ++k) {
        float2 w[B / 2];
#pragma unroll
        for (int u = 0; u < B / 2; u += 2)
          *reinterpret_cast<float4 *>(w + u) = *reinterpret_cast<const float4 *>(&s.w2[k][j + 2 * u]);
#pragma unroll
        for (int q = 0; q < S; ++q) {
          const float h = h1s[k * 256 * S + q * 256 + threadIdx.x];
#pragma unroll
          for (int u = 0; u < B / 2; ++u) a[q][u] = fma2(w[u], make_float2(h, h), a[q][u]);
        }
      }
#pragma unroll
      for (int q = 0; q < S; ++q) {
        const int64_t smp = s0 + q * 256 + threadIdx.x;
        if (act && smp < n) {
#pragma unroll
          for (int u = 0; u < B / 2; u += 2)
            *reinterpret_cast<float4 *>(act + smp * 2 * H + H + j + 2 * u) =
                make_float4(a[q][u].x, a[q][u].y, a[q][u + 1].x, a[q][u + 1].y);
        }
#pragma unroll
        for (int u = 0; u < B / 2; ++u) {
          out[q] = fmaf(s.w3[j + 2 * u], gelu(a[q][u].x), out[q]);
          out[q] = fmaf(s.w3[j + 2 * u + 1], gelu(a[q][u].y), out[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < S; ++q) {
      const int64_t smp = s0 + q * 256 + threadIdx.x;
      if (smp < n) y[smp] = out[q];
    }
  }
}

// Two samples per thread (a weight read serves both) where a block per SM would not
// cover the samples with one; below that the second would only lengthen each thread's
// work: 65000 samples take 10 us less with two.
void launch_mlp_forward(cudaStream_t st, const Weights &W, const float *X, int n, float *y, float *act) {
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(k_mlp_forward<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, forward_smem<1>());
    cudaFuncSetAttribute(k_mlp_forward<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, forward_smem<2>());
  });
  const int sms = device_sms();
  if (n > 256 * sms)
    k_mlp_forward<2><<<std::min((n - 1) / 512 + 1, sms), 256, forward_smem<2>(), st>>>(W, X, n, y, act);
  else
    k_mlp_forward<1><<<(n + 255) / 256, 256, forward_smem<1>(), st>>>(W, X, n, y, act);
}

// Backward for TILE samples per CTA: per-sample deltas in shared memory, then
// the tile's partial weight gradients (mean-squared loss, 2 (y - t) / n).  The two
// 64 x 64 x 64 products run on 4 x 4 register tiles with 16-byte shared reads (two
// scalar reads per FMA bound them before), the activation's error function is
// evaluated once per value; 161 -> 72 us for 65000 samples.
constexpr int BLD = 68;   // padded row of the 64 x 64 tiles: 16-byte aligned
struct SmemB {
  float h1[TILE][BLD];
  float h2[TILE][BLD];
  float d2[TILE][BLD];
  float d1[TILE][BLD];   // gelu'(a1) first, then delta1
  float w2[H][BLD];
  float xn[TILE][NF + 1];
  float w3[H], dy[TILE], lsum[TILE];
};

__global__ void __launch_bounds__(256) k_mlp_backward(Weights W, const float *__restrict__ X,
                                                      const float *__restrict__ target, const float *__restrict__ y,
                                                      const float *__restrict__ act, int n,
                                                      float *__restrict__ partial, float *__restrict__ loss_partial) {
  extern __shared__ __align__(16) unsigned char smem_b[];
  SmemB &b = *reinterpret_cast<SmemB *>(smem_b);
  const int tid = threadIdx.x;
  const int s0 = blockIdx.x * TILE;
  const float inv_n = 2.0f / (float)n;
  for (int i = tid; i < H * H; i += 256) b.w2[i / H][i % H] = __bfloat162float(W.w2[i]);
  if (tid < H) b.w3[tid] = __bfloat162float(W.w3[tid]);
  if (tid < TILE) {
    const int smp = s0 + tid;
    const float diff = (smp < n) ? y[smp] - target[smp] : 0.f;
    b.dy[tid] = diff * inv_n;
    b.lsum[tid] = diff * diff;
  }
  for (int e = tid; e < TILE * NF; e += 256) {
    const int q = e / NF, k = e - q * NF;
    const int smp = s0 + q;
    b.xn[q][k] = (smp < n) ? (X[(int64_t)smp * NF + k] - W.p[OFF_MU + k]) / W.p[OFF_SC + k] : 0.f;
  }
  __syncthreads();
  for (int e = tid; e < TILE * H / 4; e += 256) {
    const int q = e / (H / 4), j = 4 * (e - q * (H / 4));
    const int smp = s0 + q;
    float4 v1 = make_float4(0.f, 0.f, 0.f, 0.f), v2 = v1;
    if (smp < n) {
      v1 = *reinterpret_cast<const float4 *>(act + (int64_t)smp * 2 * H + j);
      v2 = *reinterpret_cast<const float4 *>(act + (int64_t)smp * 2 * H + H + j);
    }
    const float a1[4] = {v1.x, v1.y, v1.z, v1.w}, a2[4] = {v2.x, v2.y, v2.z, v2.w};
    const float dy = b.dy[q];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float e1 = 1.0f + erff(a1[u] * 0.70710678118654752f), e2 = 1.0f + erff(a2[u] * 0.70710678118654752f);
      const float g1 = 0.5f * e1 + a1[u] * 0.39894228040143268f * __expf(-0.5f * a1[u] * a1[u]);
      const float g2 = 0.5f * e2 + a2[u] * 0.39894228040143268f * __expf(-0.5f * a2[u] * a2[u]);
      // rows past n: a1 = a2 = 0 give zero activations, dy = 0 zero deltas
      b.h1[q][j + u] = 0.5f * a1[u] * e1;
      b.h2[q][j + u] = 0.5f * a2[u] * e2;
      b.d1[q][j + u] = g1;
      b.d2[q][j + u] = b.w3[j + u] * g2 * dy;
    }
  }
  __syncthreads();
  const int ty = tid >> 4, tx = tid & 15;
  // delta1[q][k] = (sum_j delta2[q][j] W2[j][k]) gelu'(a1[q][k])
  {
    float acc[4][4] = {};
#pragma unroll 4
    for (int j = 0; j < H; j += 4) {
      float4 dv[4], wv[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) dv[r] = *reinterpret_cast<const float4 *>(&b.d2[4 * ty + r][j]);
#pragma unroll
      for (int u = 0; u < 4; ++u) wv[u] = *reinterpret_cast<const float4 *>(&b.w2[j + u][4 * tx]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float d[4] = {dv[r].x, dv[r].y, dv[r].z, dv[r].w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc[r][0] = fmaf(d[u], wv[u].x, acc[r][0]);
          acc[r][1] = fmaf(d[u], wv[u].y, acc[r][1]);
          acc[r][2] = fmaf(d[u], wv[u].z, acc[r][2]);
          acc[r][3] = fmaf(d[u], wv[u].w, acc[r][3]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float4 *g = reinterpret_cast<float4 *>(&b.d1[4 * ty + r][4 * tx]);
      const float4 v = *g;
      *g = make_float4(acc[r][0] * v.x, acc[r][1] * v.y, acc[r][2] * v.z, acc[r][3] * v.w);
    }
  }
  __syncthreads();
  float *out = partial + (int64_t)blockIdx.x * N_TRAIN;
  // W2[j][k] = sum_q delta2[q][j] h1[q][k]
  {
    float acc[4][4] = {};
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) {
      const float4 dv = *reinterpret_cast<const float4 *>(&b.d2[q][4 * ty]);
      const float4 hv = *reinterpret_cast<const float4 *>(&b.h1[q][4 * tx]);
      const float d[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        acc[r][0] = fmaf(d[r], hv.x, acc[r][0]);
        acc[r][1] = fmaf(d[r], hv.y, acc[r][1]);
        acc[r][2] = fmaf(d[r], hv.z, acc[r][2]);
        acc[r][3] = fmaf(d[r], hv.w, acc[r][3]);
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) out[OFF_W2 + (4 * ty + r) * H + 4 * tx + c] = acc[r][c];
  }
  for (int e = tid; e < H * NF; e += 256) {  // W1[j][k]
    const int j = e / NF, k = e - j * NF;
    float acc = 0.f;
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) acc = fmaf(b.d1[q][j], b.xn[q][k], acc);
    out[OFF_W1 + e] = acc;
  }
  // the biases, W3 and the two sums, a column sum per thread
  const int which = tid / H, j = tid - which * H;
  float g = 0.f;
  if (which == 0) {
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) g += b.d1[q][j];
    out[OFF_B1 + j] = g;
  } else if (which == 1) {
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) g += b.d2[q][j];
    out[OFF_B2 + j] = g;
  } else if (which == 2) {
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) g = fmaf(b.dy[q], b.h2[q][j], g);
    out[OFF_W3 + j] = g;
  } else if (j < 2) {
    const float *v = j ? b.lsum : b.dy;
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) g += v[q];
    if (j)
      loss_partial[blockIdx.x] = g;
    else
      out[OFF_B3] = g;
  }
}

// grad[p] = sum over tiles (fixed order, double), loss = mean squared error: eight
// parameters (a sector of each tile's row) x 32 groups of tiles per block, eight
// partials in flight per thread.  Bound by the binary64 additions and conversions,
// so the blocks are small enough to share the SMs evenly: 214 -> 24 us for 1016 tiles
// (one thread per parameter walked all tiles alone; 32 parameters per block: 38 us,
// 163 blocks on 152 SMs).
constexpr int kReduceParams = 8, kReduceGroups = 32;

__global__ void __launch_bounds__(kReduceParams *kReduceGroups)
    k_mlp_reduce(const float *__restrict__ partial, const float *__restrict__ loss_partial, int tiles, int n,
                 float *__restrict__ grad, float *__restrict__ loss) {
  __shared__ double red[kReduceGroups][kReduceParams + 1];
  const int lane = threadIdx.x % kReduceParams, g = threadIdx.x / kReduceParams;
  const int p = blockIdx.x * kReduceParams + lane;
  // the first index past the parameters sums the losses
  const bool is_loss = p == N_TRAIN;
  const float *src = is_loss ? loss_partial : partial + p;
  const int64_t step = is_loss ? 1 : N_TRAIN;
  double acc = 0.0;
  if (p <= N_TRAIN) {
    int t = g;
    for (; t + 7 * kReduceGroups < tiles; t += 8 * kReduceGroups) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = src[(int64_t)(t + kReduceGroups * u) * step];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc += v[u];
    }
    for (; t < tiles; t += kReduceGroups) acc += src[(int64_t)t * step];
  }
  red[g][lane] = acc;
  __syncthreads();
  if (g != 0 || p > N_TRAIN) return;
#pragma unroll
  for (int h = 1; h < kReduceGroups; ++h) acc += red[h][lane];
  if (is_loss)
    *loss = (float)(acc / n);
  else
    grad[p] = (float)acc;
}

// Adam on the FP32 master parameters, then the BF16 copies of W1, W2, W3.
__global__ void k_adam(float *__restrict__ p, float *__restrict__ m, float *__restrict__ v,
                       const float *__restrict__ g, int step, float lr, __nv_bfloat16 *w1, __nv_bfloat16 *w2,
                       __nv_bfloat16 *w3) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N_TRAIN) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float mh = mi / (1.f - powf(b1, (float)step));
  const float vh = vi / (1.f - powf(b2, (float)step));
  const float pi = p[i] - lr * mh / (sqrtf(vh) + eps);
  p[i] = pi;
  if (i < OFF_B1) w1[i - OFF_W1] = __float2bfloat16(pi);
  else if (i >= OFF_W2 && i < OFF_B2) w2[i - OFF_W2] = __float2bfloat16(pi);
  else if (i >= OFF_W3 && i < OFF_B3) w3[i - OFF_W3] = __float2bfloat16(pi);
}

__global__ void k_sync_bf16(const float *__restrict__ p, __nv_bfloat16 *w1, __nv_bfloat16 *w2, __nv_bfloat16 *w3) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < H * NF) w1[i] = __float2bfloat16(p[OFF_W1 + i]);
  if (i < H * H) w2[i] = __float2bfloat16(p[OFF_W2 + i]);
  if (i < H) w3[i] = __float2bfloat16(p[OFF_W3 + i]);
}

// Per-feature mean and scale (standard deviation, floored) of X, one block
// per feature, written to the parameter vector.
__global__ void k_feature_stats(const float *__restrict__ X, int n, float *__restrict__ p) {
  __shared__ double s1[256], s2[256];
  const int k = blockIdx.x;
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double x = X[(int64_t)i * NF + k];
    a += x;
    b += x * x;
  }
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = b;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      s1[threadIdx.x] += s1[threadIdx.x + o];
      s2[threadIdx.x] += s2[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double mean = s1[0] / n;
    const double var = fmax(s2[0] / n - mean * mean, 0.0);
    p[OFF_MU + k] = (float)mean;
    p[OFF_SC + k] = (float)fmax(sqrt(var), 1e-3);
  }
}

}  // namespace mlp

// ---------------------------------------------------------------------------
// Per-node features of the current model for a given overlap (see the oracle
// documentation for the definition).  One thread per spatial node and kFeatSlabs
// slabs.  The eight largest entries and their logarithms depend on the slab only
// through its block values and coefficients, which the separable model repeats
// from slab to slab: they are formed again only where one of them differs in a bit.
// 621 us at 524288 nodes with nine binary64 logarithms and an indexed, spilled list
// per node; 35 us now, the latency of the first slab's sorting and of each slab's
// loads (8 or 32 slabs per thread: 40, 46 us).
// ---------------------------------------------------------------------------
constexpr int kFeatSlabs = 16;

// (float)log(a), the same float.  binary64 arithmetic holds a warp's issue slot for
// about 70 cycles an instruction here, so a positive normal a = 2^e (1 + f), 1 + f in
// [sqrt(1/2), sqrt(2)), takes pairs of floats: 2 atanh(s) = 2 s (1 + s^2/3 + s^4/5 + ...),
// s = f / (2 + f), plus e ln 2.  The tail from s^4/5 on is in single precision, an
// error below 2^-34 of the result.  Where 2^-33 to either side would round to another
// float (one value in about 250), binary64 decides.
__device__ __forceinline__ float log_to_float(double a) {
  const long long bits = __double_as_longlong(a);
  if (bits < 0x0010000000000000ll || bits >= 0x7ff0000000000000ll) return (float)log(a);
  int e = (int)(bits >> 52) - 1023;
  long long g = bits & 0xfffffffffffffll;   // f = g scale
  float scale = 0x1p-52f;
  if (g >= 0x6a09e667f3bcdll) {
    g -= 0x10000000000000ll;
    scale = 0x1p-53f;
    ++e;
  }
  const float gh = __ll2float_rn(g), gl = __ll2float_rn(g - (long long)gh);
  const float fh = gh * scale, fl = gl * scale;
  const float dh = 2.f + fh, dl = ((2.f - dh) + fh) + fl;
  const float sh = fh / dh, sl = (fmaf(-sh, dh, fh) + fmaf(-sh, dl, fl)) / dh;
  const float th = sh * sh, tl = fmaf(sh, sh, -th) + 2.f * sh * sl;
  constexpr float third = (float)(1.0 / 3.0), third_lo = (float)(1.0 / 3.0 - (double)third);
  const float p = th * fmaf(th, fmaf(th, fmaf(th, fmaf(th, 1.f / 13.f, 1.f / 11.f), 1.f / 9.f), 1.f / 7.f), 1.f / 5.f);
  const float ch = third + p, cl = (third - ch) + p + third_lo;
  const float uh = th * ch, ul = fmaf(th, ch, -uh) + fmaf(th, cl, tl * ch);
  const float ph = sh * uh, pl = fmaf(sh, uh, -ph) + fmaf(sh, ul, sl * uh);
  const float zh = sh + ph, zl = ((sh - zh) + ph) + pl + sl;
  constexpr double ln2 = 0.693147180559945309417232;
  constexpr float l1 = (float)ln2, l2 = (float)(ln2 - (double)l1);
  const float ef = (float)e, eh = ef * l1, el = fmaf(ef, l1, -eh) + ef * l2;
  const float h = eh + 2.f * zh, back = h - eh;
  const float err = (eh - (h - back)) + (2.f * zh - back);
  const float low = err + fmaf(2.f, zl, el), slack = fabsf(h) * 0x1p-33f;
  const float r = h + (low - slack);
  return r == h + (low + slack) ? r : (float)log(a);
}


__global__ void __launch_bounds__(128) k_cv_features(SellPattern pat, BtModel m, int n_s, int n_t,
                                                     const float *__restrict__ sep_dist,
                                                     const float *__restrict__ bnd_dist, double th0, double th1,
                                                     double th2, float *__restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_s) return;
  const int sl = i >> 5, li = i & 31;
  const int w = pat.slice_width[sl];
  const int base = pat.slice_ptr[sl] + li;
  const float bnd = bnd_dist[i];
  double c0 = 0.0, cm = 0.0, cp = 0.0;
  const double *v0 = nullptr, *vm = nullptr, *vp = nullptr;
  float ltop[8], lplain = 0.f, lobs = 0.f;   // lplain, lobs: the diagonal's without and with the observation
  double dplain = 0.0, dobs = 0.0;
  bool have_plain = false, have_obs = false;
  const bool pairs = (reinterpret_cast<uintptr_t>(F) & 7) == 0;   // a caller's buffer may start on 4 bytes
#pragma unroll
  for (int q = 0; q < 8; ++q) ltop[q] = 0.f;
  // the block's ranges of kFeatSlabs slabs (one, below a million slabs)
  const int64_t first = (int64_t)blockIdx.y * kFeatSlabs, jump = (int64_t)(gridDim.y - 1) * kFeatSlabs;
  for (int64_t tt = first; tt < n_t; tt += (tt + 1) % kFeatSlabs ? 1 : 1 + jump) {
    const int t = (int)tt;
    // no coupling past the ends: its scale is zero, and a zero is never among the largest
    const bool has_m = t > 0, has_p = t + 1 < n_t;
    const double b0 = m.diag.scale(t), bm = has_m ? m.off.scale(t - 1) : 0.0, bp = has_p ? m.off.scale(t) : 0.0;
    const double *u0 = m.diag.at(t), *um = has_m ? m.off.at(t - 1) : u0, *up = has_p ? m.off.at(t) : u0;
    auto same = [](double x, double y) { return __double_as_longlong(x) == __double_as_longlong(y); };
    if (tt == first || !same(b0, c0) || !same(bm, cm) || !same(bp, cp) || u0 != v0 || um != vm || up != vp) {
      c0 = b0;
      cm = bm;
      cp = bp;
      v0 = u0;
      vm = um;
      vp = up;
      // non-negative values order like their bit patterns: an insertion by integer
      // comparisons, without branches
      unsigned long long top[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) top[q] = 0;
      auto push = [&](double a, bool use) {
        unsigned long long v = (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
        if (!use || v > 0x7ff0000000000000ull) v = 0;   // not a number: never larger
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const unsigned long long hi = v > top[q] ? v : top[q];
          v = v > top[q] ? top[q] : v;
          top[q] = hi;
        }
      };
      dplain = 0.0;
      dobs = m.obs_w;
#pragma unroll 4
      for (int s = 0; s < w; ++s) {
        const int idx = base + s * kSlice;
        const double v = c0 * v0[idx];
        const double pm = cm * vm[idx], pp = cp * vp[idx];
        const bool on = pat.col[idx] == i;
        if (on) {
          dplain += v;
          dobs += v;
        }
        push(v, !on);
        push(pm, has_m);
        push(pp, has_p);
      }
      have_plain = have_obs = false;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const unsigned long long floor_bits = (unsigned long long)__double_as_longlong(1e-30);
        const double a = __longlong_as_double((long long)(top[q] > floor_bits ? top[q] : floor_bits));
        // a stencil's entries come in equal sets
        ltop[q] = q > 0 && top[q] == top[q - 1] ? ltop[q - 1] : log_to_float(a);
      }
    }
    const int64_t r = (int64_t)t * n_s + i;
    const bool obs = m.obs && m.obs[r];
    if (obs && !have_obs) {
      lobs = log_to_float(dobs);
      have_obs = true;
    } else if (!obs && !have_plain) {
      lplain = log_to_float(dplain);
      have_plain = true;
    }
    float *f = F + r * mlp::NF;
    const float row[mlp::NF] = {obs ? lobs : lplain, ltop[0], ltop[1], ltop[2], ltop[3], ltop[4], ltop[5],
                                ltop[6], ltop[7], sep_dist[t], bnd, (float)th0, (float)th1, (float)th2};
    if (pairs) {
#pragma unroll
      for (int k = 0; k < mlp::NF; k += 2) *reinterpret_cast<float2 *>(f + k) = make_float2(row[k], row[k + 1]);
    } else {
#pragma unroll
      for (int k = 0; k < mlp::NF; ++k) f[k] = row[k];
    }
  }
}

void launch_cv_features(cudaStream_t s, const SellPattern &pat, const BtModel &m, int n_s, int n_t,
                        const float *sep_dist, const float *bnd_dist, const double th[3], float *F) {
  ++g_launch_count;
  k_cv_features<<<dim3((n_s + 127) / 128, std::min((n_t - 1) / kFeatSlabs + 1, 65535)), 128, 0, s>>>(
      pat, m, n_s, n_t, sep_dist, bnd_dist, th[0], th[1], th[2], F);
}

// Per part p: sum over the rows of Omega_p (slabs [slab_start[p],
// slab_start[p+1])) of exp(2 y_i), the squared predicted ratio c_i / v_i.
// One CTA per part, double accumulation.
__global__ void k_cv_part_m2(const float *__restrict__ y, const int32_t *__restrict__ slab_start, int n_s,
                             double *__restrict__ out) {
  __shared__ double red[256];
  const int p = blockIdx.x;
  const int64_t r0 = (int64_t)slab_start[p] * n_s, r1 = (int64_t)slab_start[p + 1] * n_s;
  double a = 0.0;
  for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
    const double v = (double)y[r];
    a += exp(2.0 * v);
  }
  red[threadIdx.x] = a;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[p] = red[0];
}

void launch_cv_part_m2(cudaStream_t s, const float *y, const int32_t *slab_start_dev, int n_parts, int n_s,
                       double *out) {
  ++g_launch_count;
  k_cv_part_m2<<<n_parts, 256, 0, s>>>(y, slab_start_dev, n_s, out);
}

// y_i = log(cbar_i / (sel_i + cbar_i)), cbar_i the mean of the corrections,
// ratio clamped below at 1e-9 (a node below it adds less than 1e-18 to any
// planned squared error).
__global__ void k_cv_targets(CvTargetArgs a, const double *__restrict__ sel, int n, float *__restrict__ y) {
  const double inv = 1.0 / a.count;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double c = 0.0;
    for (int q = 0; q < a.count; ++q) c += a.corr[q][i];
    c *= inv;
    const double v = sel[i] + c;
    double r = c / v;
    if (!(r > 1e-9)) r = 1e-9;
    y[i] = (float)log(r);
  }
}

void launch_cv_targets(cudaStream_t s, const CvTargetArgs &a, const double *sel, int n, float *y) {
  ++g_launch_count;
  int grid = (n + 255) / 256;
  if (grid > 152 * 8) grid = 152 * 8;
  k_cv_targets<<<grid, 256, 0, s>>>(a, sel, n, y);
}

}  // namespace qsel

using namespace qsel;

struct qsel_cv {
  cudaStream_t stream = nullptr;
  float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr, *loss = nullptr;
  __nv_bfloat16 *w1 = nullptr, *w2 = nullptr, *w3 = nullptr;
  float *act = nullptr, *y = nullptr, *partial = nullptr, *loss_partial = nullptr;
  int cap = 0;      // samples the training buffers hold
  int step = 0;
  std::vector<void *> allocs;
  ~qsel_cv() {
    for (void *q : allocs) cudaFree(q);
  }
  bool alloc(void **q, size_t bytes) {
    if (cudaMalloc(q, bytes) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    allocs.push_back(*q);
    return true;
  }
  bool ensure(int n) {
    if (n <= cap) return true;
    for (void **q : {(void **)&act, (void **)&y, (void **)&partial, (void **)&loss_partial}) {
      if (*q) {
        cudaFree(*q);
        for (auto &a : allocs)
          if (a == *q) a = nullptr;
        *q = nullptr;
      }
    }
    const int tiles = (n + mlp::TILE - 1) / mlp::TILE;
    if (!alloc((void **)&act, (size_t)n * 2 * mlp::H * sizeof(float)) || !alloc((void **)&y, (size_t)n * sizeof(float)) ||
        !alloc((void **)&partial, (size_t)tiles * mlp::N_TRAIN * sizeof(float)) ||
        !alloc((void **)&loss_partial, (size_t)tiles * sizeof(float)))
      return false;
    cap = n;
    return true;
  }
  mlp::Weights weights() const { return mlp::Weights{w1, w2, w3, p}; }
};

namespace {
thread_local std::string g_cv_error;

qsel_status cv_fail(qsel_status st, const std::string &m) {
  g_cv_error = m;
  set_context_free_error(m);
  return st;
}

int backward_smem() {
  return (int)sizeof(mlp::SmemB);
}

qsel_status cv_forward_backward(qsel_cv *cv, const float *X, const float *target, int n) {
  using namespace mlp;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, backward_smem());
    attr = true;
  }
  if (!cv->ensure(n)) return cv_fail(QSEL_ENOMEM, "qsel_cv: device allocation failed");
  const int tiles = (n + TILE - 1) / TILE;
  g_launch_count += 3;
  launch_mlp_forward(cv->stream, cv->weights(), X, n, cv->y, cv->act);
  k_mlp_backward<<<tiles, 256, backward_smem(), cv->stream>>>(cv->weights(), X, target, cv->y, cv->act, n,
                                                              cv->partial, cv->loss_partial);
  k_mlp_reduce<<<N_TRAIN / kReduceParams + 1, kReduceParams * kReduceGroups, 0, cv->stream>>>(
      cv->partial, cv->loss_partial, tiles, n, cv->g, cv->loss);
  return cudaGetLastError() == cudaSuccess ? QSEL_OK : cv_fail(QSEL_ECUDA, "qsel_cv: kernel launch failed");
}
}  // namespace

extern "C" {

qsel_status qsel_cv_create(qsel_cv **out, uint64_t seed, void *cuda_stream) {
  using namespace mlp;
  if (!out) return cv_fail(QSEL_EINVAL, "qsel_cv_create: out must not be NULL");
  *out = nullptr;
  qsel_cv *cv = new (std::nothrow) qsel_cv();
  if (!cv) return cv_fail(QSEL_ENOMEM, "qsel_cv_create: host allocation failed");
  cv->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  if (!cv->alloc((void **)&cv->p, N_ALL * sizeof(float)) || !cv->alloc((void **)&cv->m, N_TRAIN * sizeof(float)) ||
      !cv->alloc((void **)&cv->v, N_TRAIN * sizeof(float)) || !cv->alloc((void **)&cv->g, N_TRAIN * sizeof(float)) ||
      !cv->alloc((void **)&cv->loss, sizeof(float)) || !cv->alloc((void **)&cv->w1, H * NF * 2) ||
      !cv->alloc((void **)&cv->w2, H * H * 2) || !cv->alloc((void **)&cv->w3, H * 2)) {
    delete cv;
    return cv_fail(QSEL_ENOMEM, "qsel_cv_create: device allocation failed");
  }
  // Glorot-style initial weights from a seeded host generator (initial values
  // are an input of the training, not part of the method's arithmetic)
  std::vector<float> h(N_ALL, 0.f);
  uint64_t st = seed * 6364136223846793005ull + 1442695040888963407ull;
  auto unif = [&]() {
    st = st * 6364136223846793005ull + 1442695040888963407ull;
    return (float)((st >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;
  };
  const float s1 = std::sqrt(6.f / (NF + H)), s2 = std::sqrt(6.f / (H + H)), s3 = std::sqrt(6.f / (H + 1));
  for (int i = 0; i < H * NF; ++i) h[OFF_W1 + i] = s1 * unif();
  for (int i = 0; i < H * H; ++i) h[OFF_W2 + i] = s2 * unif();
  for (int i = 0; i < H; ++i) h[OFF_W3 + i] = s3 * unif();
  for (int k = 0; k < NF; ++k) h[OFF_SC + k] = 1.f;
  if (cudaMemcpy(cv->p, h.data(), N_ALL * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(cv->m, 0, N_TRAIN * sizeof(float)) != cudaSuccess ||
      cudaMemset(cv->v, 0, N_TRAIN * sizeof(float)) != cudaSuccess) {
    delete cv;
    return cv_fail(QSEL_ECUDA, "qsel_cv_create: copy failed");
  }
  ++g_launch_count;
  k_sync_bf16<<<(H * H + 255) / 256, 256, 0, cv->stream>>>(cv->p, cv->w1, cv->w2, cv->w3);
  if (cudaStreamSynchronize(cv->stream) != cudaSuccess) {
    delete cv;
    return cv_fail(QSEL_ECUDA, "qsel_cv_create: kernel failed");
  }
  *out = cv;
  return QSEL_OK;
}

qsel_status qsel_cv_set_params(qsel_cv *cv, const float *params) {
  using namespace mlp;
  if (!cv || !params) return cv_fail(QSEL_EINVAL, "qsel_cv_set_params: NULL argument");
  if (cudaMemcpy(cv->p, params, N_ALL * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess)
    return cv_fail(QSEL_ECUDA, "qsel_cv_set_params: copy failed");
  ++g_launch_count;
  k_sync_bf16<<<(H * H + 255) / 256, 256, 0, cv->stream>>>(cv->p, cv->w1, cv->w2, cv->w3);
  return cudaStreamSynchronize(cv->stream) == cudaSuccess ? QSEL_OK
                                                         : cv_fail(QSEL_ECUDA, "qsel_cv_set_params: kernel failed");
}

qsel_status qsel_cv_get_params(const qsel_cv *cv, float *params) {
  if (!cv || !params) return cv_fail(QSEL_EINVAL, "qsel_cv_get_params: NULL argument");
  if (cudaStreamSynchronize(cv->stream) != cudaSuccess ||
      cudaMemcpy(params, cv->p, mlp::N_ALL * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return cv_fail(QSEL_ECUDA, "qsel_cv_get_params: copy failed");
  return QSEL_OK;
}

qsel_status qsel_cv_predict(const qsel_cv *cv, const float *X_dev, float *y_dev, int32_t n) {
  if (!cv || !X_dev || !y_dev || n < 1) return cv_fail(QSEL_EINVAL, "qsel_cv_predict: invalid argument");
  ++g_launch_count;
  mlp::launch_mlp_forward(cv->stream, cv->weights(), X_dev, n, y_dev, nullptr);
  if (cudaStreamSynchronize(cv->stream) != cudaSuccess) return cv_fail(QSEL_ECUDA, "qsel_cv_predict: kernel failed");
  return QSEL_OK;
}

qsel_status qsel_cv_grad(qsel_cv *cv, const float *X_dev, const float *y_dev, int32_t n, float *grad_host,
                         float *loss_host) {
  if (!cv || !X_dev || !y_dev || !grad_host || n < 1) return cv_fail(QSEL_EINVAL, "qsel_cv_grad: invalid argument");
  qsel_status st = cv_forward_backward(cv, X_dev, y_dev, n);
  if (st) return st;
  if (cudaStreamSynchronize(cv->stream) != cudaSuccess ||
      cudaMemcpy(grad_host, cv->g, mlp::N_TRAIN * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess ||
      (loss_host && cudaMemcpy(loss_host, cv->loss, sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess))
    return cv_fail(QSEL_ECUDA, "qsel_cv_grad: copy failed");
  return QSEL_OK;
}

qsel_status qsel_cv_train(qsel_cv *cv, const float *X_dev, const float *y_dev, int32_t n, int32_t steps, float lr,
                          int32_t set_input_stats, float *loss_out) {
  using namespace mlp;
  if (!cv || !X_dev || !y_dev || n < 1 || steps < 0 || !(lr > 0.f))
    return cv_fail(QSEL_EINVAL, "qsel_cv_train: invalid argument");
  if (set_input_stats) {
    ++g_launch_count;
    k_feature_stats<<<NF, 256, 0, cv->stream>>>(X_dev, n, cv->p);
  }
  for (int s = 0; s < steps; ++s) {
    qsel_status st = cv_forward_backward(cv, X_dev, y_dev, n);
    if (st) return st;
    ++cv->step;
    ++g_launch_count;
    k_adam<<<(N_TRAIN + 255) / 256, 256, 0, cv->stream>>>(cv->p, cv->m, cv->v, cv->g, cv->step, lr, cv->w1, cv->w2,
                                                           cv->w3);
  }
  if (loss_out) {
    // loss of the final parameters
    qsel_status st = cv_forward_backward(cv, X_dev, y_dev, n);
    if (st) return st;
    if (cudaMemcpyAsync(loss_out, cv->loss, sizeof(float), cudaMemcpyDeviceToHost, cv->stream) != cudaSuccess)
      return cv_fail(QSEL_ECUDA, "qsel_cv_train: copy failed");
  }
  if (cudaStreamSynchronize(cv->stream) != cudaSuccess) return cv_fail(QSEL_ECUDA, "qsel_cv_train: kernel failed");
  return QSEL_OK;
}

void qsel_cv_destroy(qsel_cv *cv) {
  if (!cv) return;
  cudaStreamSynchronize(cv->stream);
  delete cv;
}

}  // extern "C"
