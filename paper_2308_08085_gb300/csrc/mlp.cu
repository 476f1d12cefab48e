// Learned refinement proposal: a per-block MLP 27 -> 64 -> 64 -> 1 (ReLU,
// sigmoid) with hand-written training and inference kernels.  FP32 master
// weights are trained with Adam on a class-weighted binary cross-entropy; an
// FP16 copy of the weights is what inference reads.  The MLP is small enough
// that every layer runs on CUDA cores (one or two samples per thread for
// inference, one hidden unit per thread for the gradient).
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "../../include/amr.h"

namespace amr {
void set_error(const std::string& msg);

namespace mlp {

constexpr int IN = AMR_MLP_INPUTS;   // 27
constexpr int H = AMR_MLP_HIDDEN;    // 64
// parameter layout: W1[H][IN], b1[H], W2[H][H], b2[H], w3[H], b3
constexpr int OW1 = 0, OB1 = OW1 + H * IN, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H,
              OB3 = OW3 + H, NP = OB3 + 1;

// SplitMix64 (Steele, Lea, Flood 2014) as a counter-based generator
__host__ __device__ inline uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ inline float uniform_pm1(uint64_t seed, uint64_t i) {
  return (float)((splitmix64(seed ^ splitmix64(i)) >> 40) * (1.0 / 16777216.0)) * 2.f - 1.f;
}

// Glorot-uniform weights, zero biases
__global__ void k_init(float* __restrict__ P, uint64_t seed) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NP) return;
  float v = 0.f;
  if (i < OB1) v = uniform_pm1(seed, i) * sqrtf(6.f / (IN + H));
  else if (i >= OW2 && i < OB2) v = uniform_pm1(seed, i) * sqrtf(6.f / (H + H));
  else if (i >= OW3 && i < OB3) v = uniform_pm1(seed, i) * sqrtf(6.f / (H + 1));
  P[i] = v;
}

__device__ inline float softplus(float t) { return t > 0.f ? t + log1pf(expf(-t)) : log1pf(expf(t)); }

// Summed gradient and loss over the samples of one minibatch.  A CTA of 256
// threads takes tiles of S samples: the four groups of 64 threads compute
// hidden unit t % 64 of S / 4 samples each, then every thread owns 16 entries
// of dW2 and up to 7 of dW1 in registers, summed over its CTA's tiles.  A
// minibatch of 1024 is latency-bound: 32 CTAs of 64 threads with 32 samples in a
// row took 88 us, 128 to 256 CTAs with one tile each spread the serial chain of
// a sample over the chip (21 us).  Rows of W2 have a stride of 65 words in shared
// memory (W1: 27), so that both W x and W^T x read without bank conflicts.
// Gradient and loss lose digits with every addition to `grad` and *loss (256
// additions of 4 samples each: relative error of the gradient 2.3e-7, 32 of 32:
// 1.0e-7), so a cluster of eight CTAs is summed first, each CTA an eighth of the
// entries out of the others' shared memory: 1.0e-7, 9e-8 at 8,192 samples, and
// an eighth of the atomic additions (an epoch of 32 minibatches and its check
// 755 -> 691 us).  Sample position pos maps to index (pos * mul + off) mod n,
// a bijection when gcd(mul, n) = 1.
constexpr int GT = 256, GC = 8;   // threads of a CTA, CTAs of a cluster
template <int S>
__global__ void __cluster_dims__(GC, 1, 1) __launch_bounds__(GT)
    k_grad(const float* __restrict__ P, const float* __restrict__ x, const float* __restrict__ y,
           int64_t n, int64_t b0, int64_t bn, int64_t mul, int64_t off,
           float pos_weight, float* __restrict__ grad, float* __restrict__ loss) {
  constexpr int SPG = S / 4;                       // samples of a group
  constexpr int NW = H * IN + H * (H + 1);
  __shared__ float sP[NW > NP ? NW : NP];          // weights, then the CTA's gradient
  float *sW1 = sP, *sW2 = sP + H * IN;
  __shared__ float sx[S][IN + 1], sy[S], sdz[S];
  __shared__ __align__(16) float sh1[S][H], sh2[S][H], sd1[S][H], sd2[S][H];
  __shared__ float sred[S][2];
  __shared__ int64_t sidx[S];
  const int t = threadIdx.x, k = t & (H - 1), grp = t >> 6;
  const bool busy = (int64_t)blockIdx.x * S < bn;   // (a cluster may have CTAs without a tile)
  for (int i = t; busy && i < H * IN; i += GT) sW1[i] = P[OW1 + i];
  for (int i = t; busy && i < H * H; i += GT) sW2[(i >> 6) * (H + 1) + (i & 63)] = P[OW2 + i];
  const float b1 = P[OB1 + k], b2 = P[OB2 + k], w3 = P[OW3 + k], b3 = P[OB3];
  const int row = t >> 2, c1 = (t & 3) * 7, c2 = (t & 3) * 16;   // owned dW1 / dW2 entries
  float gW1[7] = {}, gW2[16] = {}, gb1 = 0.f, gb2 = 0.f, gw3 = 0.f, gb3 = 0.f, lsum = 0.f;
  for (int64_t first = (int64_t)blockIdx.x * S; first < bn; first += (int64_t)gridDim.x * S) {
    __syncthreads();                               // the previous tile is done with
    if (t < S) sidx[t] = first + t < bn ? ((b0 + first + t) * mul + off) % n : -1;
    __syncthreads();
    for (int i = t; i < S * IN; i += GT) {
      const int s = i / IN;
      const int64_t at = sidx[s];
      sx[s][i - s * IN] = at >= 0 ? x[at * IN + (i - s * IN)] : 0.f;
    }
    if (t < S) sy[t] = sidx[t] >= 0 ? y[sidx[t]] : 0.f;
    __syncthreads();
    float h2[SPG];
    {
      float a[SPG];
#pragma unroll
      for (int s = 0; s < SPG; ++s) a[s] = b1;
#pragma unroll
      for (int i = 0; i < IN; ++i) {
        const float w = sW1[k * IN + i];
#pragma unroll
        for (int s = 0; s < SPG; ++s) a[s] += w * sx[grp * SPG + s][i];
      }
#pragma unroll
      for (int s = 0; s < SPG; ++s) sh1[grp * SPG + s][k] = fmaxf(a[s], 0.f);
    }
    __syncthreads();
    {
      float a[SPG];
#pragma unroll
      for (int s = 0; s < SPG; ++s) a[s] = b2;
#pragma unroll 16
      for (int j = 0; j < H; ++j) {
        const float w = sW2[k * (H + 1) + j];
#pragma unroll
        for (int s = 0; s < SPG; ++s) a[s] += w * sh1[grp * SPG + s][j];
      }
#pragma unroll
      for (int s = 0; s < SPG; ++s) {
        h2[s] = fmaxf(a[s], 0.f);
        sh2[grp * SPG + s][k] = h2[s];
        float z = w3 * h2[s];
        for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        if ((t & 31) == 0) sred[grp * SPG + s][(t >> 5) & 1] = z;
      }
    }
    __syncthreads();
    if (t < S) {
      const float z = b3 + sred[t][0] + sred[t][1];
      const float p = 1.f / (1.f + expf(-z));
      const float yy = sy[t];
      const bool there = sidx[t] >= 0;
      const float dz = there ? pos_weight * yy * (p - 1.f) + (1.f - yy) * p : 0.f;
      sdz[t] = dz;
      gb3 += dz;
      if (there) lsum += pos_weight * yy * softplus(-z) + (1.f - yy) * softplus(z);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < SPG; ++s) sd2[grp * SPG + s][k] = h2[s] > 0.f ? sdz[grp * SPG + s] * w3 : 0.f;
    __syncthreads();
    {
      float a[SPG] = {};
#pragma unroll 16
      for (int m = 0; m < H; ++m) {
        const float w = sW2[m * (H + 1) + k];
#pragma unroll
        for (int s = 0; s < SPG; ++s) a[s] += w * sd2[grp * SPG + s][m];
      }
#pragma unroll
      for (int s = 0; s < SPG; ++s)
        sd1[grp * SPG + s][k] = sh1[grp * SPG + s][k] > 0.f ? a[s] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const float d2 = sd2[s][row], d1 = sd1[s][row];
#pragma unroll
      for (int j = 0; j < 16; j += 4) {
        const float4 h = *reinterpret_cast<const float4*>(&sh1[s][c2 + j]);
        gW2[j] += d2 * h.x;
        gW2[j + 1] += d2 * h.y;
        gW2[j + 2] += d2 * h.z;
        gW2[j + 3] += d2 * h.w;
      }
#pragma unroll
      for (int i = 0; i < 7; ++i)
        if (c1 + i < IN) gW1[i] += d1 * sx[s][c1 + i];
      if (t < H) {
        gb1 += sd1[s][t];
        gb2 += sd2[s][t];
        gw3 += sdz[s] * sh2[s][t];
      }
    }
  }
  if (t < 32) {                                    // S <= 32: warp 0 holds every sample's terms
    for (int o = 16; o > 0; o >>= 1) {
      gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
      lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
  }
  __shared__ float s_loss;
  if (t == 0) s_loss = lsum;
  if (busy) {                                      // (the weights are done with)
#pragma unroll
    for (int j = 0; j < 16; ++j) sP[OW2 + row * H + c2 + j] = gW2[j];
#pragma unroll
    for (int i = 0; i < 7; ++i)
      if (c1 + i < IN) sP[OW1 + row * IN + c1 + i] = gW1[i];
    if (t < H) {
      sP[OB1 + t] = gb1;
      sP[OB2 + t] = gb2;
      sP[OW3 + t] = gw3;
    }
    if (t == 0) sP[OB3] = gb3;
  }
  auto cluster = cooperative_groups::this_cluster();
  cluster.sync();
  const int rank = (int)cluster.block_rank();
  // CTAs of this cluster that had a tile (the first always)
  const int64_t rest = (bn + S - 1) / S - (int64_t)(blockIdx.x - rank);
  const int live = rest < GC ? (int)rest : GC;
  for (int i = rank * GT + t; i < NP; i += GC * GT) {
    float v = 0.f;
    for (int r = 0; r < live; ++r) v += *cluster.map_shared_rank(&sP[i], r);
    atomicAdd(grad + i, v);
  }
  if (rank == 0 && t == 0) {
    float v = 0.f;
    for (int r = 0; r < live; ++r) v += *cluster.map_shared_rank(&s_loss, r);
    atomicAdd(loss, v);
  }
  cluster.sync();                                  // shared memory outlives its readers
}

// `clear`: leave the gradient zeroed for the next minibatch.
__global__ void k_adam(float* __restrict__ P, float* __restrict__ m, float* __restrict__ v,
                       __half* __restrict__ Ph, float* __restrict__ grad, float inv_batch,
                       float lr, float b1, float b2, float eps, float bc1, float bc2, bool clear) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NP) return;
  const float g = grad[i] * inv_batch;
  if (clear) grad[i] = 0.f;
  const float mi = b1 * m[i] + (1.f - b1) * g;
  const float vi = b2 * v[i] + (1.f - b2) * g * g;
  m[i] = mi;
  v[i] = vi;
  const float w = P[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  P[i] = w;
  Ph[i] = __float2half_rn(w);
}

__global__ void k_to_half(const float* __restrict__ P, __half* __restrict__ Ph) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < NP) Ph[i] = __float2half_rn(P[i]);
}

// N samples per thread; FP16 weights staged as FP32 in shared memory (rows of
// W1 padded to 28: four weights per load).  Every weight is a broadcast read,
// so two samples per thread halve the loads per multiply-add; with few
// samples one per thread and small CTAs fill more SMs (69,000 samples: 36 us
// with one per thread in CTAs of 256).
// `list` (optional) maps position i to sample list[i]; output prob[sample].
template <int N>
__global__ void __launch_bounds__(64)
    k_infer(const __half* __restrict__ Ph, const float* __restrict__ x,
            const int32_t* __restrict__ list, int64_t n, float* __restrict__ prob) {
  __shared__ __align__(16) float sW1[H][28];
  __shared__ __align__(16) float sW2[H][H];
  __shared__ float sb1[H], sb2[H], sw3[H];
  const int t = threadIdx.x;
  // (many weights in flight: a CTA of 64 threads waits for each round of loads)
#pragma unroll 14
  for (int i = t; i < H * 28; i += 64) {
    const int r = i / 28, c = i - r * 28;
    sW1[r][c] = c < IN ? __half2float(Ph[OW1 + r * IN + c]) : 0.f;
  }
#pragma unroll 16
  for (int i = t; i < H * H; i += 64) sW2[i >> 6][i & 63] = __half2float(Ph[OW2 + i]);
  sb1[t] = __half2float(Ph[OB1 + t]);
  sb2[t] = __half2float(Ph[OB2 + t]);
  sw3[t] = __half2float(Ph[OW3 + t]);
  const float b3 = __half2float(Ph[OB3]);
  __syncthreads();
  int64_t at[N];
  float z[N], h[N][H];
  {
    float xi[N][28];
#pragma unroll
    for (int s = 0; s < N; ++s) {
      const int64_t i = ((int64_t)blockIdx.x * N + s) * 64 + t;
      at[s] = i < n ? (list ? list[i] : i) : -1;
#pragma unroll
      for (int q = 0; q < IN; ++q) xi[s][q] = at[s] >= 0 ? x[at[s] * IN + q] : 0.f;
      xi[s][27] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < H; ++j) {
      float a[N];
#pragma unroll
      for (int s = 0; s < N; ++s) a[s] = sb1[j];
#pragma unroll
      for (int q = 0; q < 28; q += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&sW1[j][q]);
#pragma unroll
        for (int s = 0; s < N; ++s) {
          a[s] += w.x * xi[s][q];
          a[s] += w.y * xi[s][q + 1];
          a[s] += w.z * xi[s][q + 2];
          if (q + 3 < IN) a[s] += w.w * xi[s][q + 3];
        }
      }
#pragma unroll
      for (int s = 0; s < N; ++s) h[s][j] = fmaxf(a[s], 0.f);
    }
  }
#pragma unroll
  for (int s = 0; s < N; ++s) z[s] = b3;
  for (int kk = 0; kk < H; ++kk) {
    float a[N];
#pragma unroll
    for (int s = 0; s < N; ++s) a[s] = sb2[kk];
#pragma unroll
    for (int j = 0; j < H; j += 4) {
      const float4 w = *reinterpret_cast<const float4*>(&sW2[kk][j]);
#pragma unroll
      for (int s = 0; s < N; ++s) {
        a[s] += w.x * h[s][j];
        a[s] += w.y * h[s][j + 1];
        a[s] += w.z * h[s][j + 2];
        a[s] += w.w * h[s][j + 3];
      }
    }
#pragma unroll
    for (int s = 0; s < N; ++s) z[s] += sw3[kk] * fmaxf(a[s], 0.f);
  }
#pragma unroll
  for (int s = 0; s < N; ++s)
    if (at[s] >= 0) prob[at[s]] = 1.f / (1.f + expf(-z[s]));
}

}  // namespace mlp

// used by api.cu (propose marks)
void mlp_infer_list(cudaStream_t s, const void* params_half, const float* x, const int32_t* list,
                    int64_t n, float* prob) {
  if (n <= 0) return;
  // one sample per thread until its CTAs (64 samples) would pass four per SM
  if (n <= 64 * 152 * 4)
    mlp::k_infer<1><<<(int)((n + 63) / 64), 64, 0, s>>>((const __half*)params_half, x, list, n, prob);
  else
    mlp::k_infer<2><<<(int)((n + 127) / 128), 64, 0, s>>>((const __half*)params_half, x, list, n,
                                                          prob);
}

}  // namespace amr

using namespace amr;

extern "C" {

int amr_mlp_param_count(void) { return mlp::NP; }

int amr_mlp_init(float* params, void* params_half, uint64_t seed, void* stream) {
  if (!params) return AMR_E_INVAL;
  cudaStream_t s = (cudaStream_t)stream;
  mlp::k_init<<<(mlp::NP + 255) / 256, 256, 0, s>>>(params, seed);
  if (params_half) mlp::k_to_half<<<(mlp::NP + 255) / 256, 256, 0, s>>>(params, (__half*)params_half);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error(std::string("amr_mlp_init: ") + cudaGetErrorString(e));
    return AMR_E_CUDA;
  }
  return AMR_OK;
}

static int launch_grad(const float* params, const float* x, const float* y, int64_t n, int64_t b0,
                       int64_t bn, int64_t mul, int64_t off, float pos_weight, float* grad,
                       float* loss, cudaStream_t s) {
  // tiles of 4 samples until they would pass two CTAs per SM, then of 8; more
  // tiles than that are taken in turn by the same CTAs
  const int64_t most = 2 * 152;
  auto ctas = [](int64_t n_tiles) {                // whole clusters
    return (unsigned)((n_tiles + mlp::GC - 1) / mlp::GC * mlp::GC);
  };
  const int64_t tiles = (bn + 3) / 4;
  if (tiles <= most)
    mlp::k_grad<4><<<ctas(tiles), mlp::GT, 0, s>>>(params, x, y, n, b0, bn, mul, off, pos_weight,
                                                   grad, loss);
  else
    mlp::k_grad<8><<<ctas(std::min<int64_t>((bn + 7) / 8, most)), mlp::GT, 0, s>>>(
        params, x, y, n, b0, bn, mul, off, pos_weight, grad, loss);
  return cudaGetLastError() == cudaSuccess ? AMR_OK : AMR_E_CUDA;
}

int amr_mlp_grad(const float* params, const float* x, const float* y, int64_t n, float pos_weight,
                 float* grad, float* loss, void* stream) {
  if (!params || !x || !y || !grad || !loss || n <= 0) return AMR_E_INVAL;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(grad, 0, sizeof(float) * mlp::NP, s) != cudaSuccess ||
      cudaMemsetAsync(loss, 0, sizeof(float), s) != cudaSuccess)
    return AMR_E_CUDA;
  return launch_grad(params, x, y, n, 0, n, 1, 0, pos_weight, grad, loss, s);
}

static int64_t gcd64(int64_t a, int64_t b) {
  while (b) {
    const int64_t t = a % b;
    a = b;
    b = t;
  }
  return a;
}

int amr_mlp_train_epoch(const amr_mlp_state* st, const float* x, const float* y, int64_t n,
                        int batch, float lr, float pos_weight, uint64_t epoch_seed,
                        double* mean_loss, void* stream) {
  if (!st || !st->params || !st->adam_m || !st->adam_v || !st->params_half || !st->grad ||
      !st->loss || !x || !y || n <= 0 || batch <= 0)
    return AMR_E_INVAL;
  cudaStream_t s = (cudaStream_t)stream;
  // an arithmetic progression mod n visits every sample once per epoch
  int64_t mul = (int64_t)(mlp::splitmix64(epoch_seed) % (uint64_t)n) | 1;
  while (gcd64(mul, n) != 1) mul += 2;
  const int64_t off = (int64_t)(mlp::splitmix64(epoch_seed + 1) % (uint64_t)n);
  if (cudaMemsetAsync(st->loss, 0, sizeof(float), s) != cudaSuccess ||
      cudaMemsetAsync(st->grad, 0, sizeof(float) * mlp::NP, s) != cudaSuccess)
    return AMR_E_CUDA;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  amr_mlp_state* mst = const_cast<amr_mlp_state*>(st);
  for (int64_t b0 = 0; b0 < n; b0 += batch) {
    const int64_t bn = std::min<int64_t>(batch, n - b0);
    int rc = launch_grad(st->params, x, y, n, b0, bn, mul, off, pos_weight, st->grad, st->loss, s);
    if (rc != AMR_OK) return rc;
    mst->step += 1;
    const float bc1 = 1.f - powf(b1, (float)mst->step);
    const float bc2 = 1.f - powf(b2, (float)mst->step);
    mlp::k_adam<<<(mlp::NP + 255) / 256, 256, 0, s>>>(st->params, st->adam_m, st->adam_v,
                                                      (__half*)st->params_half, st->grad,
                                                      1.f / (float)bn, lr, b1, b2, eps, bc1, bc2,
                                                      b0 + bn < n);
  }
  if (cudaGetLastError() != cudaSuccess) return AMR_E_CUDA;
  if (mean_loss) {
    float l = 0.f;
    if (cudaMemcpyAsync(&l, st->loss, sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return AMR_E_CUDA;
    *mean_loss = (double)l / (double)n;
  }
  return AMR_OK;
}

int amr_mlp_infer(const void* params_half, const float* x, int64_t n, float* prob, void* stream) {
  if (!params_half || !x || !prob || n <= 0) return AMR_E_INVAL;
  mlp_infer_list((cudaStream_t)stream, params_half, x, nullptr, n, prob);
  return cudaGetLastError() == cudaSuccess ? AMR_OK : AMR_E_CUDA;
}

}  // extern "C"
