// Learned cost model for pass selection: a 2 x 64 ReLU MLP that predicts the
// natural log of a fused block's device time (ms) from its features.
//
// The paper leaves the mapping from profile data to optimisation flags open
// and points at learned selection of compiler optimisations as the next step
// (Sec. III-A, "PGO design considerations"). Trained on block profiles the
// simulator records itself (QS_PROFILE), the network stands in for repeated
// profiling runs: candidate plans are scored by the sum of predicted block
// times without running them.
//
// Network: h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2), y = w3 . h2 + b3,
// x standardised with the training set's mean / std, loss = mean squared
// error of y against standardised log-times. Training runs on the GPU with
// the kernels below (layer forward, input / weight gradients, Adam), FP32,
// no atomics (every reduction has a fixed order).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "qs_internal.h"

namespace qs {
std::string &last_error_ref();
}

namespace {

constexpr int kF = QS_MLP_FEATURES;
constexpr int kH = QS_MLP_HIDDEN;

// parameter layout inside one flat array
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kH * kF;
constexpr int kOffW2 = kOffB1 + kH;
constexpr int kOffB2 = kOffW2 + kH * kH;
constexpr int kOffW3 = kOffB2 + kH;
constexpr int kOffB3 = kOffW3 + kH;
constexpr int kParams = kOffB3 + 1;
static_assert(kParams == QS_MLP_PARAMS, "parameter count");

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------
// One thread-block cluster runs a whole epoch (k_fit): the network is so
// small (5,825 parameters) that with a kernel per layer a 256-sample update
// was twelve launches of a few microseconds each around 10 MFLOP of work.
// Every CTA keeps a copy of the parameters in shared memory and takes its
// share of the batch, 16 samples at a time; the CTAs' gradients meet through
// distributed shared memory, each CTA summing (in CTA order), updating (Adam
// moments in registers) and handing round its share of the parameters. Two
// cluster barriers per update are the only synchronisation.

constexpr int kT = 256;         // threads per CTA
constexpr int kS = 16;          // samples per tile
constexpr int kWp1 = kF + 1;    // padded rows: lanes reading different rows hit different banks
constexpr int kWp2 = kH + 1;
constexpr int kMaxCluster = 16;

struct Weights {  // one CTA's copy, rows padded
  float w1[kH * kWp1], b1[kH], w2[kH * kWp2], b2[kH], w3[kH], b3[4];
};

struct Tile {  // one tile of samples and its activations
  float x[kS * kF], t[kS];
  float h1[kS * kH], h2[kS * kH], d1[kS * kH], d2[kS * kH], y[kS], dy[kS];
};

// Where parameter p of the flat vector lives in a Weights struct (float index).
__device__ __forceinline__ int weight_slot(int p) {
  if (p < kOffB1) return p / kF * kWp1 + p % kF;
  if (p < kOffW2) return kH * kWp1 + p - kOffB1;
  if (p < kOffB2) return kH * kWp1 + kH + (p - kOffW2) / kH * kWp2 + (p - kOffW2) % kH;
  return kH * kWp1 + kH + kH * kWp2 + p - kOffB2;  // b2, w3, b3
}

// h[s][o] = relu(b[o] + sum_i w[o][i] in[s][i]), one thread per output o and
// four samples (warps share an o range, so the samples' rows are broadcast).
template <int IN, int WP>
__device__ __forceinline__ void layer_forward(const float *in, const float *w, const float *b, float *h) {
  const int o = threadIdx.x % kH, s0 = threadIdx.x / kH * 4;
  float acc[4];
#pragma unroll
  for (int j = 0; j < 4; j++) acc[j] = b[o];
#pragma unroll 4
  for (int i = 0; i < IN; i += 4) {
    float wv[4];
#pragma unroll
    for (int u = 0; u < 4; u++) wv[u] = w[o * WP + i + u];
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const float4 v = *reinterpret_cast<const float4 *>(in + (s0 + j) * IN + i);
      acc[j] = fmaf(wv[0], v.x, fmaf(wv[1], v.y, fmaf(wv[2], v.z, fmaf(wv[3], v.w, acc[j]))));
    }
  }
#pragma unroll
  for (int j = 0; j < 4; j++) h[(s0 + j) * kH + o] = fmaxf(acc[j], 0.f);
}

// The tile's outputs y[s]; threads of warp w do samples 2w and 2w + 1.
__device__ __forceinline__ void tile_forward(const Weights &W, Tile &T) {
  layer_forward<kF, kWp1>(T.x, W.w1, W.b1, T.h1);
  __syncthreads();
  layer_forward<kH, kWp2>(T.h1, W.w2, W.b2, T.h2);
  __syncthreads();
  const int lane = threadIdx.x & 31, s = threadIdx.x / 32 * 2;
  float a = 0.f, b = 0.f;
#pragma unroll
  for (int u = 0; u < kH; u += 32) {
    a = fmaf(T.h2[s * kH + u + lane], W.w3[u + lane], a);
    b = fmaf(T.h2[(s + 1) * kH + u + lane], W.w3[u + lane], b);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane < 2) T.y[s + lane] = (lane ? b : a) + W.b3[0];
}

struct FitParam {
  const float *x, *t;  // rows of kF features, targets
  const int *idx;      // row of each sample in order; null: row = position
  float *p, *g, *m, *v, *loss;
  int batch, steps;    // samples per update, updates
  int step0;           // updates made before (Adam's bias correction)
  int update;          // 1: Adam updates of p; 0: one batch, its gradient into g
  float lr;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void *p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ float ld_peer(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_peer(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// Adam (Kingma and Ba 2015) with bias correction; step is 1-based.
__device__ __forceinline__ float adam(float p, float g, float &m, float &v, float lr, float c1, float c2) {
  constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  m = b1 * m + (1.f - b1) * g;
  v = b2 * v + (1.f - b2) * g * g;
  return p - lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__global__ void __launch_bounds__(kT) k_fit(const __grid_constant__ FitParam P) {
  extern __shared__ __align__(16) unsigned char smem[];
  Weights &W = *reinterpret_cast<Weights *>(smem);
  Tile &T = *reinterpret_cast<Tile *>(smem + sizeof(Weights));
  float *grad = reinterpret_cast<float *>(smem + sizeof(Weights) + sizeof(Tile));  // this CTA's, flat order
  const int tid = threadIdx.x;
  const uint32_t rank = cluster_rank(), ncta = cluster_size();
  for (int i = tid; i < kParams; i += kT) reinterpret_cast<float *>(&W)[weight_slot(i)] = P.p[i];
  // this CTA's share of the parameters: own0 + tid, own0 + tid + kT, ...
  constexpr int kOwn = 3;  // 3 * 256 >= 5825 / 8: clusters of 8 CTAs or more
  const int share = (kParams + (int)ncta - 1) / (int)ncta;
  const int own0 = (int)rank * share, own1 = min(own0 + share, kParams);
  float m[kOwn], v[kOwn];
#pragma unroll
  for (int j = 0; j < kOwn; j++) {
    const int i = own0 + tid + j * kT;
    m[j] = P.update && i < own1 ? P.m[i] : 0.f;
    v[j] = P.update && i < own1 ? P.v[i] : 0.f;
  }
  // this CTA's samples of every batch
  const int per = (P.batch + (int)ncta - 1) / (int)ncta;
  const int first = min((int)rank * per, P.batch), count = min(per, P.batch - first);
  const int tiles = (count + kS - 1) / kS;
  // the next tile's rows travel in registers while the current one is worked on
  constexpr int kXl = (kS * kF + kT - 1) / kT;
  float nx[kXl], nt = 0.f;
  auto fetch = [&](int step, int tile) {
    const long long at = (long long)step * P.batch + first + tile * kS;
    const int have = step < P.steps ? count - tile * kS : 0;
#pragma unroll
    for (int j = 0; j < kXl; j++) {
      const int e = tid + j * kT, s = e / kF;
      nx[j] = 0.f;
      if (e < kS * kF && s < have) {
        const long long row = P.idx ? P.idx[at + s] : at + s;
        nx[j] = P.x[row * kF + e % kF];
      }
    }
    if (tid < kS) nt = tid < have ? P.t[P.idx ? P.idx[at + tid] : at + tid] : 0.f;
  };
  fetch(0, 0);
  const float scale = 2.f / (float)P.batch;
  const int o4 = tid / 16 * 4, i4 = tid % 16 * 4;      // this thread's 4 x 4 block of dW2
  const int o1 = tid / 4, i1 = tid % 4 * (kF / 4);      // and 1 x 6 of dW1
  const int oc = tid % kH, sc = tid / kH * 4;           // layer outputs: one unit, four samples
  __syncthreads();
  for (int step = 0; step < P.steps; step++) {
    float dw2[16], dw1[kF / 4], db = 0.f;
#pragma unroll
    for (int j = 0; j < 16; j++) dw2[j] = 0.f;
#pragma unroll
    for (int j = 0; j < kF / 4; j++) dw1[j] = 0.f;
    for (int tile = 0; tile < tiles; tile++) {
#pragma unroll
      for (int j = 0; j < kXl; j++)
        if (tid + j * kT < kS * kF) T.x[tid + j * kT] = nx[j];
      if (tid < kS) T.t[tid] = nt;
      __syncthreads();
      if (tile + 1 < tiles) fetch(step, tile + 1);
      else fetch(step + 1, 0);
      tile_forward(W, T);
      __syncthreads();
      if (tid < kS) {
        const bool in = tile * kS + tid < count;
        const float d = in ? T.y[tid] - T.t[tid] : 0.f;
        T.dy[tid] = scale * d;
        if (in && step == P.steps - 1) P.loss[first + tile * kS + tid] = d * d;
      }
      __syncthreads();
      // through the last layer
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int e = (sc + j) * kH + oc;
        T.d2[e] = T.h2[e] > 0.f ? T.dy[sc + j] * W.w3[oc] : 0.f;
      }
      __syncthreads();
      // d1[s][i] = (sum_o d2[s][o] w2[o][i]) where h1 > 0
      {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int o = 0; o < kH; o += 4) {
          float wv[4];
#pragma unroll
          for (int u = 0; u < 4; u++) wv[u] = W.w2[(o + u) * kWp2 + oc];
#pragma unroll
          for (int j = 0; j < 4; j++) {
            const float4 d = *reinterpret_cast<const float4 *>(T.d2 + (sc + j) * kH + o);
            acc[j] = fmaf(d.x, wv[0], fmaf(d.y, wv[1], fmaf(d.z, wv[2], fmaf(d.w, wv[3], acc[j]))));
          }
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const int e = (sc + j) * kH + oc;
          T.d1[e] = T.h1[e] > 0.f ? acc[j] : 0.f;
        }
      }
      // dW2[o][i] += sum_s d2[s][o] h1[s][i]
#pragma unroll 4
      for (int s = 0; s < kS; s++) {
        const float4 d = *reinterpret_cast<const float4 *>(T.d2 + s * kH + o4);
        const float4 h = *reinterpret_cast<const float4 *>(T.h1 + s * kH + i4);
        const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
          for (int b = 0; b < 4; b++) dw2[4 * a + b] = fmaf(dv[a], hv[b], dw2[4 * a + b]);
      }
      __syncthreads();
      // dW1[o][i] += sum_s d1[s][o] x[s][i]; the biases and w3
#pragma unroll 4
      for (int s = 0; s < kS; s++) {
        const float d = T.d1[s * kH + o1];
#pragma unroll
        for (int j = 0; j < kF / 4; j++) dw1[j] = fmaf(d, T.x[s * kF + i1 + j], dw1[j]);
      }
      if (tid < kH) {
        for (int s = 0; s < kS; s++) db += T.d1[s * kH + oc];
      } else if (tid < 2 * kH) {
        for (int s = 0; s < kS; s++) db += T.d2[s * kH + oc];
      } else if (tid < 3 * kH) {
        for (int s = 0; s < kS; s++) db = fmaf(T.dy[s], T.h2[s * kH + oc], db);
      } else if (oc == 0) {
        for (int s = 0; s < kS; s++) db += T.dy[s];
      }
      __syncthreads();
    }
    if (tiles == 0) fetch(step + 1, 0);
#pragma unroll
    for (int a = 0; a < 4; a++)
      *reinterpret_cast<float4 *>(grad + kOffW2 + (o4 + a) * kH + i4) =
          make_float4(dw2[4 * a], dw2[4 * a + 1], dw2[4 * a + 2], dw2[4 * a + 3]);
#pragma unroll
    for (int j = 0; j < kF / 4; j++) grad[kOffW1 + o1 * kF + i1 + j] = dw1[j];
    if (tid < kH) grad[kOffB1 + oc] = db;
    else if (tid < 2 * kH) grad[kOffB2 + oc] = db;
    else if (tid < 3 * kH) grad[kOffW3 + oc] = db;
    else if (oc == 0) grad[kOffB3] = db;
    cluster_sync();
    const float c1 = 1.f - powf(0.9f, (float)(P.step0 + step + 1));
    const float c2 = 1.f - powf(0.999f, (float)(P.step0 + step + 1));
#pragma unroll
    for (int j = 0; j < kOwn; j++) {
      const int i = own0 + tid + j * kT;
      if (i < own1) {
        float s = 0.f;
        for (uint32_t c = 0; c < ncta; c++) s += ld_peer(peer_addr(grad + i, c));
        if (P.update) {
          float *w = reinterpret_cast<float *>(&W) + weight_slot(i);
          const float np = adam(*w, s, m[j], v[j], P.lr, c1, c2);
          for (uint32_t c = 0; c < ncta; c++) st_peer(peer_addr(w, c), np);
        } else {
          P.g[i] = s;
        }
      }
    }
    cluster_sync();  // the new parameters are in place, every peer has read this CTA's gradient
  }
  if (P.update) {
#pragma unroll
    for (int j = 0; j < kOwn; j++) {
      const int i = own0 + tid + j * kT;
      if (i < own1) {
        P.p[i] = reinterpret_cast<float *>(&W)[weight_slot(i)];
        P.m[i] = m[j];
        P.v[i] = v[j];
      }
    }
  }
}

// Means and standard deviations of the features, then of the targets.
struct Scaling {
  float mean[kF + 1], std[kF + 1];
};

// FP64 mean and deviation of column blockIdx.x of n rows of kF features, or of
// the targets (the last block). The FP64 rate (three operations a value, two
// per clock) bounds it: 10 us for 10,000 rows, which the host took 250 us for.
__global__ void __launch_bounds__(kT) k_scaling(const float *__restrict__ x, const float *__restrict__ t, int n,
                                                float *__restrict__ out) {
  __shared__ double part[kT];
  const int f = blockIdx.x, tid = threadIdx.x;
  const float *col = f < kF ? x + f : t;
  const int step = f < kF ? kF : 1;
  auto total = [&](double v) {
    part[tid] = v;
    __syncthreads();
    for (int o = kT / 2; o > 0; o >>= 1) {
      if (tid < o) part[tid] += part[tid + o];
      __syncthreads();
    }
    const double s = part[0];
    __syncthreads();
    return s;
  };
  double s = 0;
  for (int r = tid; r < n; r += kT) s += (double)col[(size_t)r * step];
  const double mean = total(s) / n;
  s = 0;
  for (int r = tid; r < n; r += kT) {
    const double d = (double)col[(size_t)r * step] - mean;
    s = fma(d, d, s);
  }
  const double var = total(s) / n;
  if (tid == 0) {
    out[f] = (float)mean;
    // a feature counts as constant below 1e-6, the targets below a variance of 1e-12
    out[kF + 1 + f] = (f < kF ? sqrt(var) > 1e-6 : var > 1e-12) ? (float)sqrt(var) : 1.f;
  }
}

// Standardises n rows and their targets in place.
__global__ void __launch_bounds__(kT) k_standardise(float *__restrict__ x, float *__restrict__ t, int n,
                                                    const __grid_constant__ Scaling sc) {
  const long long all = (long long)n * kF;
  for (long long e = (long long)blockIdx.x * kT + threadIdx.x; e < all + n; e += (long long)gridDim.x * kT) {
    if (e < all) {
      const int f = (int)(e % kF);
      x[e] = (x[e] - sc.mean[f]) / sc.std[f];
    } else {
      t[e - all] = (t[e - all] - sc.mean[kF]) / sc.std[kF];
    }
  }
}

// y[r] of n feature rows, 16 rows per tile.
__global__ void __launch_bounds__(kT) k_predict(const float *__restrict__ x, const float *__restrict__ p,
                                                float *__restrict__ y, int n, const __grid_constant__ Scaling sc) {
  extern __shared__ __align__(16) unsigned char smem[];
  Weights &W = *reinterpret_cast<Weights *>(smem);
  Tile &T = *reinterpret_cast<Tile *>(smem + sizeof(Weights));
  const int tid = threadIdx.x;
  for (int i = tid; i < kParams; i += kT) reinterpret_cast<float *>(&W)[weight_slot(i)] = p[i];
  for (long long r0 = (long long)blockIdx.x * kS; r0 < n; r0 += (long long)gridDim.x * kS) {
    const int have = (int)min((long long)kS, n - r0);
    for (int e = tid; e < kS * kF; e += kT) T.x[e] = e / kF < have ? (x[r0 * kF + e] - sc.mean[e % kF]) / sc.std[e % kF] : 0.f;
    __syncthreads();
    tile_forward(W, T);
    __syncthreads();
    if (tid < have) y[r0 + tid] = T.y[tid] * sc.std[kF] + sc.mean[kF];
  }
}

}  // namespace

struct qs_mlp {
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // params, grads, Adam moments (one allocation)
  float *x = nullptr, *y = nullptr, *loss = nullptr;  // rows, targets or outputs, squared errors
  int *idx = nullptr;    // sample order
  int cap = 0;           // rows x, y, loss and idx hold
  int step = 0;
  Scaling scaling;
  cudaStream_t stream = nullptr;
};

namespace {

qs_status mfail(qs_status s, const std::string &m) {
  qs::last_error_ref() = m;
  return s;
}

template <typename T> cudaError_t dalloc(T *&p, size_t n) {
  qs::dev_free(p);
  p = nullptr;
  return qs::dev_malloc((void **)&p, sizeof(T) * (n ? n : 1));
}

cudaError_t ensure_rows(qs_mlp *mm, int n) {
  if (n <= mm->cap) return cudaSuccess;
  mm->cap = 0;
  cudaError_t e = dalloc(mm->x, (size_t)n * kF);
  if (e == cudaSuccess) e = dalloc(mm->y, (size_t)n);
  if (e == cudaSuccess) e = dalloc(mm->loss, (size_t)n);
  if (e == cudaSuccess) e = dalloc(mm->idx, (size_t)n);
  if (e == cudaSuccess) mm->cap = n;
  return e;
}

// All of a model's work is ordered on its stream, which need not wait for the
// legacy stream; the host buffer is free again on return.
cudaError_t copy(qs_mlp *mm, void *dst, const void *src, size_t bytes, cudaMemcpyKind kind) {
  cudaError_t e = cudaMemcpyAsync(dst, src, bytes, kind, mm->stream);
  return e == cudaSuccess ? cudaStreamSynchronize(mm->stream) : e;
}

constexpr size_t kFitSmem = sizeof(Weights) + sizeof(Tile) + sizeof(float) * kParams;
constexpr size_t kPredictSmem = sizeof(Weights) + sizeof(Tile);

// One cluster of 16 CTAs (8 where the device does not take 16).
cudaError_t launch_fit(const FitParam &P, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = kFitSmem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static thread_local int configured = -1;
  static thread_local int ncta = 8;
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured != dev) {
    cudaError_t e = cudaFuncSetAttribute(k_fit, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFitSmem);
    if (e != cudaSuccess) return e;
    ncta = 8;
    if (cudaFuncSetAttribute(k_fit, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      int fits = 0;
      cfg.gridDim = dim3(kMaxCluster);
      attr[0].val.clusterDim.x = kMaxCluster;
      if (cudaOccupancyMaxActiveClusters(&fits, k_fit, &cfg) == cudaSuccess && fits > 0) ncta = kMaxCluster;
    }
    cudaGetLastError();  // 16 refused is not an error
    configured = dev;
  }
  cfg.gridDim = dim3(ncta);
  attr[0].val.clusterDim.x = ncta;
  return cudaLaunchKernelEx(&cfg, k_fit, P);
}

cudaError_t launch_predict(qs_mlp *mm, int n) {
  const int tiles = (n + kS - 1) / kS;
  k_predict<<<std::min(tiles, 4 * qs::dev_info().sms), kT, kPredictSmem, mm->stream>>>(mm->x, mm->p, mm->y, n,
                                                                                       mm->scaling);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

qs_status qs_mlp_create(uint64_t seed, void *cuda_stream, qs_mlp **out) {
  if (!out) return mfail(QS_EINVAL, "qs_mlp_create: null output");
  *out = nullptr;
  qs_mlp *mm = new (std::nothrow) qs_mlp();
  if (!mm) return mfail(QS_ENOMEM, "qs_mlp_create: host allocation failed");
  mm->stream = (cudaStream_t)cuda_stream;
  for (int f = 0; f <= kF; f++) {
    mm->scaling.mean[f] = 0.f;
    mm->scaling.std[f] = 1.f;
  }
  // He-uniform initial weights, zero biases, from a seeded generator
  std::vector<float> p(kParams, 0.f);
  std::mt19937_64 rng(seed);
  auto fill = [&](int off, int fan_out, int fan_in) {
    const float lim = std::sqrt(6.f / (float)fan_in);
    std::uniform_real_distribution<float> u(-lim, lim);
    for (int i = 0; i < fan_out * fan_in; i++) p[off + i] = u(rng);
  };
  fill(kOffW1, kH, kF);
  fill(kOffW2, kH, kH);
  fill(kOffW3, 1, kH);
  cudaError_t e = dalloc(mm->p, 4 * kParams);
  if (e == cudaSuccess) {
    mm->g = mm->p + kParams;
    mm->m = mm->g + kParams;
    mm->v = mm->m + kParams;
    e = cudaMemsetAsync(mm->m, 0, 2 * sizeof(float) * kParams, mm->stream);
  }
  if (e == cudaSuccess) e = copy(mm, mm->p, p.data(), sizeof(float) * kParams, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    qs_mlp_free(mm);
    return mfail(QS_ENOMEM, std::string("qs_mlp_create: ") + cudaGetErrorString(e));
  }
  *out = mm;
  return QS_OK;
}

void qs_mlp_free(qs_mlp *mm) {
  if (!mm) return;
  cudaDeviceSynchronize();
  qs::dev_free(mm->p);
  qs::dev_free(mm->x);
  qs::dev_free(mm->y);
  qs::dev_free(mm->loss);
  qs::dev_free(mm->idx);
  delete mm;
}

qs_status qs_mlp_params(qs_mlp *mm, float *host_out, const float *host_in) {
  if (!mm) return mfail(QS_EINVAL, "qs_mlp_params: null model");
  cudaError_t e = cudaSuccess;
  if (host_in) e = copy(mm, mm->p, host_in, sizeof(float) * kParams, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && host_out) e = copy(mm, host_out, mm->p, sizeof(float) * kParams, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return mfail(QS_ECUDA, std::string("qs_mlp_params: ") + cudaGetErrorString(e));
  return QS_OK;
}

qs_status qs_mlp_gradient(qs_mlp *mm, const float *x, const float *y, int n, float *grad_out, float *loss_out) {
  if (!mm || !x || !y || n <= 0 || !grad_out) return mfail(QS_EINVAL, "qs_mlp_gradient: bad arguments");
  cudaError_t e = ensure_rows(mm, n);
  if (e == cudaSuccess) e = cudaMemcpyAsync(mm->x, x, sizeof(float) * (size_t)n * kF, cudaMemcpyHostToDevice, mm->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(mm->y, y, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, mm->stream);
  if (e == cudaSuccess) {
    FitParam P = {mm->x, mm->y, nullptr, mm->p, mm->g, mm->m, mm->v, mm->loss, n, 1, 0, 0, 0.f};
    e = launch_fit(P, mm->stream);
  }
  if (e == cudaSuccess) e = copy(mm, grad_out, mm->g, sizeof(float) * kParams, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && loss_out) {
    std::vector<float> l(n);
    e = copy(mm, l.data(), mm->loss, sizeof(float) * n, cudaMemcpyDeviceToHost);
    double s = 0;
    for (float v : l) s += v;
    *loss_out = (float)(s / n);
  }
  if (e != cudaSuccess) return mfail(QS_ECUDA, std::string("qs_mlp_gradient: ") + cudaGetErrorString(e));
  return QS_OK;
}

qs_status qs_mlp_train(qs_mlp *mm, const float *x, const float *y, int n, int epochs, int batch, float lr,
                       uint64_t seed, float *loss_out) {
  if (!mm || !x || !y || n <= 0 || epochs <= 0 || batch <= 0) return mfail(QS_EINVAL, "qs_mlp_train: bad arguments");
  // standardisation from this training set (features and targets), while the host draws the first order
  static_assert(sizeof(Scaling) <= sizeof(float) * kParams, "the gradient's space holds it meanwhile");
  const int B = std::min(batch, n), steps = n / B;
  cudaError_t e = ensure_rows(mm, n);
  if (e == cudaSuccess) e = cudaMemcpyAsync(mm->x, x, sizeof(float) * (size_t)n * kF, cudaMemcpyHostToDevice, mm->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(mm->y, y, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, mm->stream);
  if (e == cudaSuccess) {
    k_scaling<<<kF + 1, kT, 0, mm->stream>>>(mm->x, mm->y, n, mm->g);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return mfail(QS_ECUDA, std::string("qs_mlp_train: ") + cudaGetErrorString(e));
  std::vector<int> order(n);
  for (int i = 0; i < n; i++) order[i] = i;
  std::mt19937_64 rng(seed);
  std::shuffle(order.begin(), order.end(), rng);
  Scaling sc;
  e = cudaMemcpyAsync(&sc, mm->g, sizeof(sc), cudaMemcpyDeviceToHost, mm->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(mm->stream);
  if (e == cudaSuccess) {
    mm->scaling = sc;
    const long long all = (long long)n * (kF + 1);
    k_standardise<<<(int)std::min<long long>((all + kT - 1) / kT, 8ll * qs::dev_info().sms), kT, 0, mm->stream>>>(
        mm->x, mm->y, n, sc);
    e = cudaGetLastError();
  }
  std::vector<float> lpart(B);
  double last = 0;
  for (int ep = 0; ep < epochs && e == cudaSuccess; ep++) {
    if (ep > 0) std::shuffle(order.begin(), order.end(), rng);  // while the epoch before runs
    // one upload of the epoch's sample order, after the epoch before has read its own; the host buffer is
    // only reused after the stream has consumed it
    e = cudaMemcpyAsync(mm->idx, order.data(), sizeof(int) * n, cudaMemcpyHostToDevice, mm->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(mm->stream);
    if (e != cudaSuccess) break;
    FitParam P = {mm->x, mm->y, mm->idx, mm->p, mm->g, mm->m, mm->v, mm->loss, B, steps, mm->step, 1, lr};
    e = launch_fit(P, mm->stream);
    mm->step += steps;
  }
  // loss of the last batch of the last epoch (standardised units)
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(lpart.data(), mm->loss, sizeof(float) * B, cudaMemcpyDeviceToHost, mm->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(mm->stream);
  if (e == cudaSuccess) {
    double esum = 0;
    for (float v : lpart) esum += v;
    last = esum / B;
  }
  if (e != cudaSuccess) return mfail(QS_ECUDA, std::string("qs_mlp_train: ") + cudaGetErrorString(e));
  if (loss_out) *loss_out = (float)last;
  return QS_OK;
}

qs_status qs_mlp_predict(qs_mlp *mm, const float *x, int n, float *y_out) {
  if (!mm || !x || !y_out || n < 0) return mfail(QS_EINVAL, "qs_mlp_predict: bad arguments");
  if (n == 0) return QS_OK;
  cudaError_t e = ensure_rows(mm, n);
  if (e == cudaSuccess) e = cudaMemcpyAsync(mm->x, x, sizeof(float) * (size_t)n * kF, cudaMemcpyHostToDevice, mm->stream);
  if (e == cudaSuccess) e = launch_predict(mm, n);
  if (e == cudaSuccess) e = cudaMemcpyAsync(y_out, mm->y, sizeof(float) * n, cudaMemcpyDeviceToHost, mm->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(mm->stream);
  if (e != cudaSuccess) return mfail(QS_ECUDA, std::string("qs_mlp_predict: ") + cudaGetErrorString(e));
  return QS_OK;
}

}  // extern "C"
