// Learned row-capacity predictor: row features, capacity labels, and the
// training kernels (forward, backward, Adam) and inference of the MLP
// declared in kk_learned.h.  Everything runs on the GPU in float32.
#include <cooperative_groups.h>

#include <cmath>
#include <cstdio>
#include <vector>

#include "kk_internal.h"
#include "kk_learned.h"
#include "kk_mlp.cuh"
#include "kk_walk.h"

namespace kk {
namespace {

constexpr int kFeatTeam = 8;

// Per B row: smallest and largest column (empty rows: INT_MAX, -1).
__global__ void k_brow_minmax(CsrView B, int2* __restrict__ mm) {
  const int tl = threadIdx.x % kFeatTeam;
  const unsigned mask = team_mask<kFeatTeam>();
  const long long team0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kFeatTeam;
  const long long nteams = (long long)gridDim.x * blockDim.x / kFeatTeam;
  const long long iters = (B.m + nteams - 1) / nteams;
  for (long long it = 0; it < iters; ++it) {
    const long long r = team0 + it * nteams;
    int lo = 0x7fffffff, hi = -1;
    if (r < B.m) {
      for (int q = B.rowptr[r] + tl; q < B.rowptr[r + 1]; q += kFeatTeam) {
        const int c = B.colind[q];
        lo = min(lo, c);
        hi = max(hi, c);
      }
    }
#pragma unroll
    for (int o = kFeatTeam / 2; o > 0; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(mask, lo, o, kFeatTeam));
      hi = max(hi, __shfl_xor_sync(mask, hi, o, kFeatTeam));
    }
    if (r < B.m && tl == 0) mm[r] = make_int2(lo, hi);
  }
}

__global__ void k_row_features(CsrView A, CsrView B, const int2* __restrict__ mm,
                               float* __restrict__ feat) {
  const int tl = threadIdx.x % kFeatTeam;
  const unsigned mask = team_mask<kFeatTeam>();
  const long long team0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kFeatTeam;
  const long long nteams = (long long)gridDim.x * blockDim.x / kFeatTeam;
  const long long iters = (A.m + nteams - 1) / nteams;
  for (long long it = 0; it < iters; ++it) {
    const long long r = team0 + it * nteams;
    long long f = 0;
    int mx = 0, mn = 0x7fffffff, lo = 0x7fffffff, hi = -1, nza = 0;
    if (r < A.m) {
      const int pa = A.rowptr[r], pe = A.rowptr[r + 1];
      nza = pe - pa;
      for (int p = pa + tl; p < pe; p += kFeatTeam) {
        const int j = A.colind[p];
        const int len = B.rowptr[j + 1] - B.rowptr[j];
        f += len;
        mx = max(mx, len);
        mn = min(mn, len);
        if (len > 0) {
          const int2 v = mm[j];
          lo = min(lo, v.x);
          hi = max(hi, v.y);
        }
      }
    }
#pragma unroll
    for (int o = kFeatTeam / 2; o > 0; o >>= 1) {
      f += __shfl_xor_sync(mask, f, o, kFeatTeam);
      mx = max(mx, __shfl_xor_sync(mask, mx, o, kFeatTeam));
      mn = min(mn, __shfl_xor_sync(mask, mn, o, kFeatTeam));
      lo = min(lo, __shfl_xor_sync(mask, lo, o, kFeatTeam));
      hi = max(hi, __shfl_xor_sync(mask, hi, o, kFeatTeam));
    }
    if (r < A.m && tl == 0) {
      if (nza == 0) mn = 0;
      const double span = hi >= lo ? (double)hi - (double)lo + 1.0 : 0.0;
      const double mean = nza ? (double)f / nza : 0.0;
      const double v[kMlpF] = {(double)nza, (double)f, (double)mx, mean, (double)(mx - mn),
                               span, fmin((double)f, span), fmin(fmin((double)f, span), (double)B.n)};
      float* out = feat + r * kMlpF;
#pragma unroll
      for (int t = 0; t < kMlpF; ++t) out[t] = log2f(1.0f + (float)v[t]);
    }
  }
}

__global__ void k_capacity_classes(int32_t m, const int64_t* __restrict__ rp, int32_t* __restrict__ cls) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (long long)gridDim.x * blockDim.x)
    cls[i] = capacity_class_of(rp[i + 1] - rp[i]);
}

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void k_mlp_init(float* __restrict__ P, unsigned long long seed) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kMlpParams) return;
  int fan_in = 0;
  if (i < kOffB1) fan_in = kMlpF;
  else if (i >= kOffW2 && i < kOffB2) fan_in = kMlpH;
  else if (i >= kOffW3 && i < kOffB3) fan_in = kMlpH;
  if (fan_in == 0) {
    P[i] = 0.0f;
    return;
  }
  const unsigned long long r = splitmix64(seed * 0x9E3779B97F4A7C15ull + (unsigned long long)i);
  const float u = (float)((r >> 40) * (1.0 / 16777216.0));  // [0, 1)
  P[i] = (2.0f * u - 1.0f) * sqrtf(6.0f / (float)fan_in);
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

constexpr int kMlpBlock = 128;

// Gradient of the mean loss over `count` samples; sample t of the batch is
// index (pa * (start + t) + pb) mod n of X / y.
//
// A CTA of 8 warps takes tiles of 32 samples, lane = sample; a warp computes a
// fixed eighth of every layer's units for the tile, forward and backward, through
// [unit][sample] tiles in shared memory (rows padded to kGradLd floats, so that
// 16-byte reads along the samples are aligned and spread over the banks; a
// layer's weights are broadcasts).  The gradient of a weight is then the inner
// product of two rows, and every thread owns the same weights for all of the
// CTA's tiles: 4 of W2, 2 of W3, 1 of W1 and one bias, in registers.  At the end a
// cluster of 8 CTAs adds its sums as a tree through distributed shared memory, then
// to grad: a chain of 128 to 608 float32 additions, one per CTA, cost 2.2 us less at
// 4,096 samples but was 1.8 times further from the float64 gradient than a warp sum
// per weight (relative error at 4,096 and 20,001 samples, mean of 12 seeds: warp sums
// 9.5e-8 and 2.0e-7, the chain 1.7e-7 and 3.4e-7, this 8.0e-8 and 1.4e-7).
// What bounds it: latency; the 8 warps of a CTA execute 1,640 instructions each for a
// tile and its share of the sums, with a barrier after each layer.  A thread per sample with a warp sum per weight (1,872 of
// five shuffles, then atomics) took 252 us for 4,096 samples; this takes 14.8.
constexpr int kGradThreads = 256;
constexpr int kGradLd = 36;
constexpr int kGradMaxCtas = 608;
constexpr int kGradCluster = 8;
struct GradSmem {
  float P[kMlpParams];
  float x[kMlpF][kGradLd];
  float h1[kMlpH][kGradLd], h2[kMlpH][kGradLd];
  float z[kMlpC][kGradLd];
  float dz[kMlpC][kGradLd];
  float dh2[kMlpH][kGradLd], dh1[kMlpH][kGradLd];
  float loss;
};

__device__ __forceinline__ float row_dot(const float* a, const float* b) {
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int t = 0; t < 32; t += 4) {
    const float4 u = *reinterpret_cast<const float4*>(a + t), v = *reinterpret_cast<const float4*>(b + t);
    s.x = fmaf(u.x, v.x, s.x);
    s.y = fmaf(u.y, v.y, s.y);
    s.z = fmaf(u.z, v.z, s.z);
    s.w = fmaf(u.w, v.w, s.w);
  }
  return (s.x + s.y) + (s.z + s.w);
}

__global__ void __cluster_dims__(kGradCluster) __launch_bounds__(kGradThreads)
k_mlp_loss_grad(int32_t n, int32_t start, int32_t count, long long pa, long long pb,
                const float* __restrict__ X, const int32_t* __restrict__ y,
                const float* __restrict__ Pg, float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ __align__(16) GradSmem sm;
  const float* P = sm.P;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int i = tid; i < kMlpParams; i += kGradThreads) sm.P[i] = Pg[i];
  float g2[4] = {0.f, 0.f, 0.f, 0.f}, g3[2] = {0.f, 0.f}, g1 = 0.f, gb = 0.f, lsum = 0.f;
  const int j2 = (w * 2 + (lane >> 4)) * 2, k2 = (lane & 15) * 2;  // W2 block of this thread
  const int k3 = tid >> 3, c3 = (tid & 7) * 2;                      // W3 pair
  const float inv_count = 1.0f / (float)count;
  for (int t0 = blockIdx.x * 32; t0 < count; t0 = walk_next_tile(t0, gridDim.x * 32, count)) {
    const bool active = t0 + lane < count;
    const float inv = active ? inv_count : 0.0f;
    int label = 0;
    float xf = 0.0f;
    if (active) {
      const long long s = (pa * (long long)(start + t0 + lane) + pb) % n;
      xf = X[s * kMlpF + w];
      label = y[s];
    }
    sm.x[w][lane] = xf;
    __syncthreads();
    {  // layer 1, units 4 w .. 4 w + 3
      float4 a = *reinterpret_cast<const float4*>(P + kOffB1 + 4 * w);
#pragma unroll
      for (int f = 0; f < kMlpF; ++f) {
        const float v = sm.x[f][lane];
        const float4 q = *reinterpret_cast<const float4*>(P + kOffW1 + f * kMlpH + 4 * w);
        a.x = fmaf(v, q.x, a.x);
        a.y = fmaf(v, q.y, a.y);
        a.z = fmaf(v, q.z, a.z);
        a.w = fmaf(v, q.w, a.w);
      }
      sm.h1[4 * w][lane] = fmaxf(a.x, 0.0f);
      sm.h1[4 * w + 1][lane] = fmaxf(a.y, 0.0f);
      sm.h1[4 * w + 2][lane] = fmaxf(a.z, 0.0f);
      sm.h1[4 * w + 3][lane] = fmaxf(a.w, 0.0f);
    }
    __syncthreads();
    float h2v[4];
    {  // layer 2
      float4 a = *reinterpret_cast<const float4*>(P + kOffB2 + 4 * w);
#pragma unroll 8
      for (int j = 0; j < kMlpH; ++j) {
        const float v = sm.h1[j][lane];
        const float4 q = *reinterpret_cast<const float4*>(P + kOffW2 + j * kMlpH + 4 * w);
        a.x = fmaf(v, q.x, a.x);
        a.y = fmaf(v, q.y, a.y);
        a.z = fmaf(v, q.z, a.z);
        a.w = fmaf(v, q.w, a.w);
      }
      h2v[0] = fmaxf(a.x, 0.0f);
      h2v[1] = fmaxf(a.y, 0.0f);
      h2v[2] = fmaxf(a.z, 0.0f);
      h2v[3] = fmaxf(a.w, 0.0f);
#pragma unroll
      for (int u = 0; u < 4; ++u) sm.h2[4 * w + u][lane] = h2v[u];
    }
    __syncthreads();
    {  // layer 3, classes 2 w and 2 w + 1
      float2 a = *reinterpret_cast<const float2*>(P + kOffB3 + 2 * w);
#pragma unroll 8
      for (int k = 0; k < kMlpH; ++k) {
        const float v = sm.h2[k][lane];
        const float2 q = *reinterpret_cast<const float2*>(P + kOffW3 + k * kMlpC + 2 * w);
        a.x = fmaf(v, q.x, a.x);
        a.y = fmaf(v, q.y, a.y);
      }
      sm.z[2 * w][lane] = a.x;
      sm.z[2 * w + 1][lane] = a.y;
    }
    __syncthreads();
    {  // softmax of the sample (every warp for its two classes)
      float zv[kMlpC], mx, se = 0.0f;
#pragma unroll
      for (int c = 0; c < kMlpC; ++c) zv[c] = sm.z[c][lane];
      mx = zv[0];
#pragma unroll
      for (int c = 1; c < kMlpC; ++c) mx = fmaxf(mx, zv[c]);
#pragma unroll
      for (int c = 0; c < kMlpC; ++c) se += __expf(zv[c] - mx);
      const float lse = mx + __logf(se);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int c = 2 * w + u;
        sm.dz[c][lane] = (__expf(sm.z[c][lane] - lse) - (c == label ? 1.0f : 0.0f)) * inv;
      }
      // a label that is no class has no unit of z to read: its loss is lse
      if (w == 0) lsum += (lse - ((unsigned)label < (unsigned)kMlpC ? sm.z[label][lane] : 0.0f)) * inv;
    }
    __syncthreads();
    {  // dh2, units 4 w .. 4 w + 3
      float dzv[kMlpC];
#pragma unroll
      for (int c = 0; c < kMlpC; ++c) dzv[c] = sm.dz[c][lane];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float a = 0.0f;
#pragma unroll
        for (int c = 0; c < kMlpC; c += 4) {
          const float4 q = *reinterpret_cast<const float4*>(P + kOffW3 + (4 * w + u) * kMlpC + c);
          a = fmaf(q.x, dzv[c], a);
          a = fmaf(q.y, dzv[c + 1], a);
          a = fmaf(q.z, dzv[c + 2], a);
          a = fmaf(q.w, dzv[c + 3], a);
        }
        sm.dh2[4 * w + u][lane] = h2v[u] > 0.0f ? a : 0.0f;
      }
    }
    __syncthreads();
    {  // dh1
      float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
      for (int k = 0; k < kMlpH; k += 4) {
        const float v0 = sm.dh2[k][lane], v1 = sm.dh2[k + 1][lane], v2 = sm.dh2[k + 2][lane],
                    v3 = sm.dh2[k + 3][lane];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 q = *reinterpret_cast<const float4*>(P + kOffW2 + (4 * w + u) * kMlpH + k);
          a[u] = fmaf(q.x, v0, a[u]);
          a[u] = fmaf(q.y, v1, a[u]);
          a[u] = fmaf(q.z, v2, a[u]);
          a[u] = fmaf(q.w, v3, a[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) sm.dh1[4 * w + u][lane] = sm.h1[4 * w + u][lane] > 0.0f ? a[u] : 0.0f;
    }
    __syncthreads();
    // gradients: inner products of rows over the tile's samples
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) g2[2 * u + v] += row_dot(sm.h1[j2 + u], sm.dh2[k2 + v]);
#pragma unroll
    for (int v = 0; v < 2; ++v) g3[v] += row_dot(sm.h2[k3], sm.dz[c3 + v]);
    g1 += row_dot(sm.x[w], sm.dh1[lane]);
    if (tid < 2 * kMlpH + kMlpC) {
      const float* row = tid < kMlpH ? sm.dh1[tid] : tid < 2 * kMlpH ? sm.dh2[tid - kMlpH] : sm.dz[tid - 2 * kMlpH];
      float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int t = 0; t < 32; ++t) a[t & 3] += row[t];
      gb += (a[0] + a[1]) + (a[2] + a[3]);
    }
    __syncthreads();
  }
  __syncthreads();
  // this CTA's sums in the place of the weights, then the cluster's as a tree
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) sm.P[kOffW2 + (j2 + u) * kMlpH + k2 + v] = g2[2 * u + v];
#pragma unroll
  for (int v = 0; v < 2; ++v) sm.P[kOffW3 + k3 * kMlpC + c3 + v] = g3[v];
  sm.P[kOffW1 + w * kMlpH + lane] = g1;
  if (tid < kMlpH) sm.P[kOffB1 + tid] = gb;
  else if (tid < 2 * kMlpH) sm.P[kOffB2 + tid - kMlpH] = gb;
  else if (tid < 2 * kMlpH + kMlpC) sm.P[kOffB3 + tid - 2 * kMlpH] = gb;
  if (w == 0) {
    lsum = warp_sum_f(lsum);
    if (lane == 0) sm.loss = lsum;
  }
  auto cluster = cooperative_groups::this_cluster();
  cluster.sync();
  auto sum = [&](float* at) {
    float v[kGradCluster];
#pragma unroll
    for (int c = 0; c < kGradCluster; ++c) v[c] = *cluster.map_shared_rank(at, c);
#pragma unroll
    for (int o = kGradCluster / 2; o > 0; o >>= 1)
#pragma unroll
      for (int c = 0; c < o; ++c) v[c] += v[c + o];
    return v[0];
  };
  const int rank = (int)cluster.block_rank();
  for (int i = rank * kGradThreads + tid; i < kMlpParams; i += kGradCluster * kGradThreads)
    atomicAdd(&grad[i], sum(&sm.P[i]));
  if (rank == kGradCluster - 1 && tid == kGradThreads - 1) atomicAdd(loss, sum(&sm.loss));
  cluster.sync();  // the peers' shared memory is read until here
}

// CTAs of k_mlp_loss_grad: one per tile up to four per SM, in whole clusters.
int grad_ctas(int count) {
  const int tiles = count / 32 + (count % 32 != 0);
  const int ctas = (tiles + kGradCluster - 1) / kGradCluster * kGradCluster;
  return ctas < kGradMaxCtas ? ctas : kGradMaxCtas;
}

// grad and loss to zero, in one launch.
__global__ void k_mlp_zero(float* __restrict__ grad, float* __restrict__ loss) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kMlpParams) grad[i] = 0.0f;
  if (i == kMlpParams) *loss = 0.0f;
}

__global__ void k_mlp_adam(const float* __restrict__ g, float* __restrict__ P, float* __restrict__ m1,
                           float* __restrict__ m2, float lr_t, float b1, float b2, float eps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kMlpParams) return;
  const float gi = g[i];
  const float a = b1 * m1[i] + (1.0f - b1) * gi;
  const float b = b2 * m2[i] + (1.0f - b2) * gi * gi;
  m1[i] = a;
  m2[i] = b;
  P[i] -= lr_t * a / (sqrtf(b) + eps);
}

__global__ void __launch_bounds__(kMlpBlock)
k_mlp_predict(int32_t n, const float* __restrict__ X, const float* __restrict__ Pg, float q,
              int32_t* __restrict__ cls) {
  __shared__ float P[kMlpParams];
  for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) P[i] = Pg[i];
  __syncthreads();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  float x[kMlpF];
#pragma unroll
  for (int f = 0; f < kMlpF; ++f) x[f] = X[t * kMlpF + f];
  float h1[kMlpH], h2[kMlpH], z[kMlpC];
  mlp_forward(P, x, h1, h2, z);
  cls[t] = mlp_class(z, q);
}

long long gcd_ll(long long a, long long b) {
  while (b) {
    const long long t = a % b;
    a = b;
    b = t;
  }
  return a;
}

}  // namespace

cudaError_t launch_row_features(cudaStream_t s, const CsrView& A, const CsrView& B, int2* mm,
                                float* feat, int num_sms) {
  if (B.m > 0) {
    long long g = ((long long)B.m * kFeatTeam + 255) / 256;
    if (g > num_sms * 8) g = num_sms * 8;
    k_brow_minmax<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(B, mm);
  }
  if (A.m > 0) {
    long long g = ((long long)A.m * kFeatTeam + 255) / 256;
    if (g > num_sms * 8) g = num_sms * 8;
    k_row_features<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(A, B, mm, feat);
  }
  return cudaGetLastError();
}

}  // namespace kk

using namespace kk;

extern "C" {

kk_status kk_capacity_classes(void* stream, int32_t m, const int64_t* c_rowptr, int32_t* cls) {
  if (m < 0 || (m > 0 && (!c_rowptr || !cls))) return KK_ERR_INVALID_ARG;
  if (m == 0) return KK_OK;
  int g = (m + 255) / 256;
  if (g > 4096) g = 4096;
  k_capacity_classes<<<g, 256, 0, static_cast<cudaStream_t>(stream)>>>(m, c_rowptr, cls);
  return cudaGetLastError() == cudaSuccess ? KK_OK : KK_ERR_CUDA;
}

kk_status kk_mlp_init(void* stream, float* params, uint64_t seed) {
  if (!params) return KK_ERR_INVALID_ARG;
  k_mlp_init<<<(kMlpParams + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(params, seed);
  return cudaGetLastError() == cudaSuccess ? KK_OK : KK_ERR_CUDA;
}

kk_status kk_mlp_loss_grad(void* stream, int32_t n, const float* X, const int32_t* y,
                           const float* params, float* grad, float* loss) {
  if (n <= 0 || !X || !y || !params || !grad || !loss) return KK_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  k_mlp_zero<<<kMlpParams / 256 + 1, 256, 0, s>>>(grad, loss);
  k_mlp_loss_grad<<<grad_ctas(n), kGradThreads, 0, s>>>(n, 0, n, 1, 0, X, y, params, grad, loss);
  return cudaGetLastError() == cudaSuccess ? KK_OK : KK_ERR_CUDA;
}

kk_status kk_mlp_adam(void* stream, const float* grad, float* params, float* m1, float* m2,
                      int32_t step, float lr, float beta1, float beta2, float eps) {
  if (!grad || !params || !m1 || !m2 || step < 1) return KK_ERR_INVALID_ARG;
  const float lr_t = lr * sqrtf(1.0f - powf(beta2, (float)step)) / (1.0f - powf(beta1, (float)step));
  k_mlp_adam<<<(kMlpParams + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      grad, params, m1, m2, lr_t, beta1, beta2, eps);
  return cudaGetLastError() == cudaSuccess ? KK_OK : KK_ERR_CUDA;
}

kk_status kk_mlp_train(void* stream, int32_t n, const float* X, const int32_t* y, float* params,
                       int32_t epochs, int32_t batch, float lr, uint64_t seed, float* final_loss) {
  if (n <= 0 || !X || !y || !params || epochs < 0 || batch <= 0) return KK_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* buf = nullptr;  // grad | m1 | m2 | loss
  if (cudaMalloc(&buf, sizeof(float) * (3 * kMlpParams + 4)) != cudaSuccess) return KK_ERR_OOM;
  float* grad = buf;
  float* m1 = buf + kMlpParams;
  float* m2 = buf + 2 * kMlpParams;
  float* loss = buf + 3 * kMlpParams;
  kk_status st = KK_OK;
  if (cudaMemsetAsync(buf, 0, sizeof(float) * (3 * kMlpParams + 4), s) != cudaSuccess) st = KK_ERR_CUDA;
  unsigned long long rng = seed * 0x9E3779B97F4A7C15ull + 1;
  auto next = [&rng]() {
    rng += 0x9E3779B97F4A7C15ull;
    unsigned long long z = rng;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  };
  int step = 0;
  for (int e = 0; e < epochs && st == KK_OK; ++e) {
    // seeded order: sample (a*t + b) mod n with gcd(a, n) = 1
    long long a = (long long)(next() % (unsigned long long)n) | 1;
    while (gcd_ll(a, n) != 1) a = (a + 2) % n == 0 ? 1 : (a + 2) % n;
    const long long b = (long long)(next() % (unsigned long long)n);
    for (int start = 0; start < n && st == KK_OK; start += batch) {
      const int count = n - start < batch ? n - start : batch;
      if (cudaMemsetAsync(grad, 0, sizeof(float) * kMlpParams, s) != cudaSuccess) st = KK_ERR_CUDA;
      k_mlp_loss_grad<<<grad_ctas(count), kGradThreads, 0, s>>>(n, start, count, a, b, X, y, params, grad, loss);
      ++step;
      const float lr_t = lr * sqrtf(1.0f - powf(0.999f, (float)step)) / (1.0f - powf(0.9f, (float)step));
      k_mlp_adam<<<(kMlpParams + 255) / 256, 256, 0, s>>>(grad, params, m1, m2, lr_t, 0.9f, 0.999f, 1e-8f);
      if (cudaGetLastError() != cudaSuccess) st = KK_ERR_CUDA;
    }
  }
  if (st == KK_OK && final_loss) {
    cudaMemsetAsync(grad, 0, sizeof(float) * kMlpParams, s);
    cudaMemsetAsync(loss, 0, sizeof(float), s);
    k_mlp_loss_grad<<<grad_ctas(n), kGradThreads, 0, s>>>(n, 0, n, 1, 0, X, y, params, grad, loss);
    if (cudaMemcpyAsync(final_loss, loss, sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess)
      st = KK_ERR_CUDA;
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) st = KK_ERR_CUDA;
  cudaFree(buf);
  return st;
}

kk_status kk_mlp_predict(void* stream, int32_t n, const float* X, const float* params, float quantile,
                         int32_t* cls) {
  if (n < 0 || (n > 0 && (!X || !params || !cls))) return KK_ERR_INVALID_ARG;
  if (n == 0) return KK_OK;
  k_mlp_predict<<<(n + kMlpBlock - 1) / kMlpBlock, kMlpBlock, 0, static_cast<cudaStream_t>(stream)>>>(
      n, X, params, quantile, cls);
  return cudaGetLastError() == cudaSuccess ? KK_OK : KK_ERR_CUDA;
}

}  // extern "C"
