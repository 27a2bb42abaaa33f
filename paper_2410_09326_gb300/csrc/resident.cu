// Narrow states: all blocks of a plan in one launch.
//
// A state of up to 13 qubits (64 KiB) fits the shared memory of one CTA. Run
// block by block, its kernels take 3 to 10 us each, nearly all of it launch
// and start-up; here one CTA loads the state, applies every block in shared
// memory with a barrier between two blocks, and stores it. The records travel
// in the kernel's parameters (up to 32,764 bytes a launch), so the call
// needs no upload and no device scratch.
#include <cmath>
#include <cstring>

#include "resident.cuh"

namespace qs {
namespace kern {

namespace {

constexpr int kProgWords = 2040;  // 32,640 bytes of records per launch

struct ResidentProg {
  uint4 w[kProgWords];
  float2 *a;
  int n, n_recs, words;
};
static_assert(sizeof(ResidentProg) <= 32764, "kernel parameter space");

template <int MAXT> __global__ void __launch_bounds__(MAXT, 1) k_resident(const __grid_constant__ ResidentProg p) {
  extern __shared__ __align__(16) unsigned char smem[];
  float4 *st = reinterpret_cast<float4 *>(smem);
  uint4 *prog = reinterpret_cast<uint4 *>(smem + (sizeof(float2) << p.n));
  float4 *g = reinterpret_cast<float4 *>(p.a);
  const int n4 = 1 << (p.n - 1);
  for (int i = threadIdx.x; i < n4; i += blockDim.x) st[i] = g[i];
  for (int i = threadIdx.x; i < p.words; i += blockDim.x) prog[i] = p.w[i];
  __syncthreads();
  const uint4 *rec = prog;
  for (int i = 0; i < p.n_recs; i++) {
    rec_apply<MAXT>(reinterpret_cast<float2 *>(st), p.n, rec);
    rec += reinterpret_cast<const RecHead *>(rec)->words;
  }
  for (int i = threadIdx.x; i < n4; i += blockDim.x) g[i] = st[i];
}

uint32_t turn_fraction(double angle) {
  const double t = angle / (2 * M_PI);
  return (uint32_t)(int64_t)std::llrint((t - std::floor(t)) * 4294967296.0);
}

}  // namespace

bool record_encodable(const Block &b, int n, int max_k) {
  switch (b.kind) {
    case BK_DENSE: return !b.tc && b.k >= 1 && b.k <= max_k && b.k + b.nctrl <= kMaxFixed;
    case BK_DIAG: return b.nctrl <= kMaxFixed;
    case BK_PERMUTE: return true;
    case BK_PHASE: return n <= kResidentPhaseBits;
    default: return false;
  }
}

size_t record_words(const Block &b, int n, const int *tile_q) {
  size_t bytes = sizeof(RecHead);
  if (b.kind == BK_PHASE) bytes += tile_q ? sizeof(uint32_t) * (4 + wide_phase_row(n) * (n + 1)) : sizeof(RecPhase);
  else bytes += b.mat.size() * sizeof(float2);
  return (bytes + 15) / 16;
}

void record_encode(const Block &b, uint4 *out, int n, const int *tile_q, int m) {
  const size_t words = record_words(b, n, tile_q);
  std::memset(out, 0, words * sizeof(uint4));
  RecHead h;
  std::memset(&h, 0, sizeof(h));
  h.words = (uint32_t)words;
  h.kind = (uint8_t)b.kind;
  h.k = (uint8_t)b.k;
  // position of a state's bit in the array the record runs on, -1 outside
  auto local = [&](int q) {
    if (!tile_q) return q;
    for (int j = 0; j < m; j++)
      if (tile_q[j] == q) return j;
    return -1;
  };
  uint32_t fixed = 0;
  if (b.kind != BK_PHASE) {
    for (int q = 0; q < 32; q++) {
      if (!((b.cmask >> q) & 1)) continue;
      if (local(q) < 0) h.gmask |= 1u << q;
      else h.cmask |= 1u << local(q);
    }
    for (int j = 0; j < b.k; j++) h.tq[j] = (uint8_t)local(b.q[j]);  // inside: the planner's tiles hold them
    fixed = h.cmask;
    if (b.kind != BK_DIAG)
      for (int j = 0; j < b.k; j++) fixed |= 1u << h.tq[j];
  }
  for (int q = 0; q < 32; q++)
    if ((fixed >> q) & 1) h.fixed[h.nf++] = (uint8_t)q;
  unsigned char *body = (unsigned char *)out + sizeof(h);
  if (b.kind == BK_PHASE) {
    RecPhase p;
    std::memset(&p, 0, sizeof(p));
    std::vector<uint32_t> w;
    const uint32_t row = wide_phase_row(n);
    if (tile_q) {
      h.wide = (uint8_t)n;
      w.assign(4 + row * (n + 1), 0);
    }
    (tile_q ? w[0] : p.c) = turn_fraction(b.ph_c);
    for (int j = 0; j < b.k; j++) {
      const int qj = b.ph_q[j];
      (tile_q ? w[4 + qj] : p.a[qj]) = turn_fraction(b.ph_a[j]);
      for (int l = j + 1; l < b.k; l++) {
        const int ql = b.ph_q[l];
        const uint32_t x = turn_fraction(b.ph_b[tri_index(j, l, b.k)]);
        if (tile_q) w[4 + row * (1 + qj) + ql] = w[4 + row * (1 + ql) + qj] = x;
        else p.b[qj][ql] = p.b[ql][qj] = x;
      }
    }
    if (tile_q) std::memcpy(body, w.data(), w.size() * sizeof(uint32_t));
    else std::memcpy(body, &p, sizeof(p));
  } else {
    for (size_t i = 0; i < b.mat.size(); i++) {
      const float2 z = to_dev<float2>(b.mat[i]);
      std::memcpy(body + i * sizeof(z), &z, sizeof(z));
    }
  }
  std::memcpy(out, &h, sizeof(h));
}

}  // namespace kern

using namespace kern;

bool resident_applies(const std::vector<Block> &plan, int n) {
  if (n > kResidentBits || plan.size() < 2) return false;
  for (const Block &b : plan)
    if (!record_encodable(b, n, 4) || record_words(b) > (size_t)kProgWords) return false;
  return true;
}

cudaError_t run_resident(void *amps, int n, const std::vector<Block> &plan, cudaStream_t s, size_t *sent) {
  // a thread per group of eight amplitudes, no fewer than two warps
  const int threads = n >= 13 ? 1024 : (n <= 9 ? 64 : 1 << (n - 3));
  const size_t smem_max = (sizeof(float2) << kResidentBits) + sizeof(uint4) * kProgWords;
  static thread_local int configured = -1;
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured != dev) {
    cudaError_t e = cudaFuncSetAttribute(k_resident<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_resident<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    if (e != cudaSuccess) return e;
    configured = dev;
  }
  static thread_local ResidentProg p;  // large: kept off the stack; the launch copies it
  p.a = (float2 *)amps;
  p.n = n;
  for (size_t i = 0; i < plan.size();) {
    p.n_recs = p.words = 0;
    for (; i < plan.size(); i++) {
      const size_t w = record_words(plan[i]);
      if (p.words + w > (size_t)kProgWords) break;
      record_encode(plan[i], p.w + p.words);
      p.words += (int)w;
      p.n_recs++;
    }
    const size_t smem = (sizeof(float2) << n) + sizeof(uint4) * (size_t)p.words;
    if (threads == 1024) k_resident<1024><<<1, threads, smem, s>>>(p);
    else k_resident<512><<<1, threads, smem, s>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    *sent += sizeof(p);
  }
  return cudaSuccess;
}

}  // namespace qs
