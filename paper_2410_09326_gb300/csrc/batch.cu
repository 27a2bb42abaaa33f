// Batched simulation: many circuits of uneven width, captured as one CUDA
// graph (the paper's repeated-run use case, Sec. IV-E: a QAOA circuit
// simulated again and again).
//
// Every circuit is planned on the host and its blocks are uploaded once as
// records (resident.cuh). Each run starts every circuit from |0...0>.
//  - Circuits of up to 14 qubits (k_batch): one CTA per circuit, taken from a
//    work queue ordered by decreasing cost (2^n x blocks), so CTAs never wait
//    on one another. The state lives in shared memory for the whole run and
//    is written once at the end.
//  - Wider circuits (k_batch_tile): planned as cache-blocked passes (the tile
//    passes of passes.cpp, diagonal runs as phase polynomials). Launch s
//    applies pass s of every wide circuit that has one, all their tiles
//    spread over the GPU: a tile of 2^13 amplitudes is loaded into shared
//    memory (pass 0 makes |0...0> there), the pass's members are applied, and
//    it is stored. Kernel boundaries order the passes. One CTA per circuit,
//    as above but on a buffer in L2, left a batch waiting for its widest
//    circuits: 20 ms for 192 circuits of 10 to 20 qubits.
// The two kinds run side by side on two streams.
//
// The autotuner times candidate (fusion width, threads per narrow CTA) pairs
// on the batch itself and keeps the fastest; the chosen launches are captured
// once as a CUDA graph, and qs_batch_run replays it.
#include <algorithm>
#include <cstring>
#include <numeric>
#include <string>
#include <vector>

#include "resident.cuh"

namespace qs {
std::string &last_error_ref();
}

namespace qs {
namespace kern {
namespace {

constexpr int kSmemBits = 14;  // 2^14 c64 amplitudes = 128 KiB
// records are staged in shared memory this many words at a time (a 6-target
// record takes 2052)
constexpr int kStageWords = 2064;
constexpr int kMaxBatchN = 26;
constexpr int kTileBits = 13;     // 64 KiB of amplitudes
constexpr int kTileThreads = 256;
constexpr int kWideSmemMax = 112 * 1024;  // tile and records: two CTAs per SM at least

struct BCircuit {
  float2 *amps;
  int n;
  int first_chunk, n_chunks;  // narrow: its records, in chunks of at most kStageWords
};

struct BChunk {  // a run of records: a narrow circuit's share, or a wide one's pass
  long long off;  // first word in the pool
  int words, n_recs;
  int tile_q[16];  // pass: the tile's bits, ascending
};

struct BStep {  // a wide circuit's tiles in one launch
  int first;    // its first tile among the launch's
  int circuit, chunk;
};

template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
    k_batch(const BCircuit *__restrict__ circs, const int *__restrict__ order, int count,
            const BChunk *__restrict__ chunks, const uint4 *__restrict__ pool, int *__restrict__ queue) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint4 *prog = reinterpret_cast<uint4 *>(smem);
  float2 *st = reinterpret_cast<float2 *>(smem + sizeof(uint4) * kStageWords);
  __shared__ int next;
  for (;;) {
    if (threadIdx.x == 0) next = atomicAdd(queue, 1);
    __syncthreads();
    const int c = next;
    __syncthreads();
    if (c >= count) break;
    const BCircuit C = circs[order[c]];
    const int N = 1 << C.n;
    for (int i = threadIdx.x; i < N; i += blockDim.x) st[i] = make_float2(i == 0 ? 1.f : 0.f, 0.f);
    for (int k = 0; k < C.n_chunks; k++) {
      const BChunk &ch = chunks[C.first_chunk + k];
      const uint4 *src = pool + ch.off;
      const int words = ch.words, n_recs = ch.n_recs;
      for (int i = threadIdx.x; i < words; i += blockDim.x) prog[i] = src[i];
      __syncthreads();
      const uint4 *rec = prog;
      for (int r = 0; r < n_recs; r++) {
        rec_apply<MAXT>(st, C.n, rec);
        rec += reinterpret_cast<const RecHead *>(rec)->words;
      }
    }
    __syncthreads();
    float4 *dst = reinterpret_cast<float4 *>(C.amps);
    const float4 *src = reinterpret_cast<const float4 *>(st);
    for (int i = threadIdx.x; i < N / 2; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
  }
}

// One pass of every wide circuit that has it: `steps` lists them with their
// first tiles, n_items tiles in all; a CTA takes a run of consecutive ones, so
// that it stages a circuit's records once. Bound by shared-memory traffic and
// FP32 issue (a 3-target member costs 32 multiply-adds an amplitude); three
// CTAs per SM overlap one's loads with the others' arithmetic.
__global__ void __launch_bounds__(kTileThreads, 3)
    k_batch_tile(const BCircuit *__restrict__ circs, const BStep *__restrict__ steps, int n_steps, long long n_items,
                 const BChunk *__restrict__ chunks, const uint4 *__restrict__ pool, int fresh) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2 *tile = reinterpret_cast<float2 *>(smem);
  uint4 *prog = reinterpret_cast<uint4 *>(smem + (sizeof(float2) << kTileBits));
  __shared__ int tq[16];
  __shared__ uint32_t dep[1 << (kTileBits - kTileLowBits)];  // offset of each run of 2^kTileLowBits amplitudes
  __shared__ RecPhase scratch;
  const long long i0 = n_items * blockIdx.x / gridDim.x, i1 = n_items * (blockIdx.x + 1) / gridDim.x;
  int s = -1, n_recs = 0;
  BCircuit C;
  for (long long item = i0; item < i1; item++) {
    if (s < 0 || (s + 1 < n_steps && item >= steps[s + 1].first)) {
      int lo = 0, hi = n_steps - 1;  // the last entry whose first tile is not past this one
      while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (steps[mid].first <= item) lo = mid;
        else hi = mid - 1;
      }
      s = lo;
      C = circs[steps[s].circuit];
      const BChunk &ch = chunks[steps[s].chunk];
      n_recs = ch.n_recs;
      const int words = ch.words;
      const uint4 *src = pool + ch.off;
      if (threadIdx.x < kTileBits) tq[threadIdx.x] = ch.tile_q[threadIdx.x];
      for (int i = threadIdx.x; i < words; i += kTileThreads) prog[i] = src[i];
      __syncthreads();
      for (int h = threadIdx.x; h < (1 << (kTileBits - kTileLowBits)); h += kTileThreads) {
        uint32_t off = 0;
        for (int j = 0; j < kTileBits - kTileLowBits; j++) off |= ((h >> j) & 1u) << tq[kTileLowBits + j];
        dep[h] = off;
      }
      __syncthreads();
    }
    const uint32_t base = (uint32_t)insert_zeros((uint64_t)(item - steps[s].first), tq, kTileBits);
    constexpr uint32_t kLow = (1u << kTileLowBits) - 1;
    float4 *t4 = reinterpret_cast<float4 *>(tile);
    if (fresh) {
      for (int i = threadIdx.x; i < (1 << (kTileBits - 1)); i += kTileThreads)
        t4[i] = make_float4(base == 0 && i == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);
    } else {
#pragma unroll 8
      for (int i = threadIdx.x; i < (1 << (kTileBits - 1)); i += kTileThreads) {
        const uint32_t e = 2u * i;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(t4 + i);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst),
                     "l"(C.amps + (base + dep[e >> kTileLowBits] + (e & kLow)))
                     : "memory");
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    __syncthreads();
    const uint4 *rec = prog;
    for (int r = 0; r < n_recs; r++) {
      rec_apply<kTileThreads, true>(tile, kTileBits, rec, base, tq, &scratch);
      rec += reinterpret_cast<const RecHead *>(rec)->words;
    }
#pragma unroll 8
    for (int i = threadIdx.x; i < (1 << (kTileBits - 1)); i += kTileThreads) {
      const uint32_t e = 2u * i;
      *reinterpret_cast<float4 *>(C.amps + (base + dep[e >> kTileLowBits] + (e & kLow))) = t4[i];
    }
    __syncthreads();
  }
}

}  // namespace
}  // namespace kern
}  // namespace qs

using namespace qs;
using namespace qs::kern;

struct qs_state;
namespace qs {
// accessors into the opaque state (api.cpp)
void *state_amps(qs_state *st);
int state_n(const qs_state *st);
bool state_c64(const qs_state *st);
int8_t *state_perm(qs_state *st);
cudaStream_t state_stream(const qs_state *st);
}  // namespace qs

struct qs_batch {
  std::vector<qs_state *> states;
  std::vector<std::vector<qs_gate>> gates;
  uint64_t flags = 0;
  qs_opts opts;
  cudaStream_t stream = nullptr;
  int device = 0;
  // device data of the chosen plan
  BCircuit *d_circs = nullptr;
  int *d_order = nullptr;      // narrow circuits, the costliest first
  BChunk *d_chunks = nullptr;
  uint4 *d_pool = nullptr;
  BStep *d_steps = nullptr;    // the wide launches' lists, one after the other
  int *d_queue = nullptr;
  struct Launch {              // one pass of the wide circuits
    int first, count;          // its entries of d_steps
    long long items;
    int words;                 // longest program
  };
  std::vector<Launch> launches;
  int n_narrow = 0;
  cudaStream_t side = nullptr; // the wide circuits' stream
  cudaEvent_t fork = nullptr, join = nullptr;
  std::vector<std::vector<int8_t>> final_perm;
  int k_chosen = 0, threads = 0, grid = 0, total_blocks = 0;
  size_t smem = 0;
  double tune_ms[16] = {0};
  int tune_k[16] = {0}, tune_threads[16] = {0}, n_tune = 0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaStream_t own_stream = nullptr;
};

namespace {

qs_status bfail(qs_status s, const std::string &m) {
  qs::last_error_ref() = m;
  return s;
}

void free_plan(qs_batch *b) {
  qs::dev_free(b->d_circs);
  qs::dev_free(b->d_order);
  qs::dev_free(b->d_chunks);
  qs::dev_free(b->d_pool);
  qs::dev_free(b->d_steps);
  b->d_circs = nullptr;
  b->d_order = nullptr;
  b->d_chunks = nullptr;
  b->d_pool = nullptr;
  b->d_steps = nullptr;
  b->launches.clear();
}

template <typename T> cudaError_t upload(T *&d, std::vector<T> &h) {
  if (h.empty()) h.resize(1);
  cudaError_t e = qs::dev_malloc((void **)&d, sizeof(T) * h.size());
  if (e == cudaSuccess) e = cudaMemcpy(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice);
  return e;
}

// Plans every circuit with the given flags and uploads the records.
qs_status upload_plan(qs_batch *bt, uint64_t flags) {
  free_plan(bt);
  const size_t count = bt->states.size();
  std::vector<BCircuit> circs(count);
  std::vector<BChunk> chunks;
  std::vector<uint4> pool;
  std::vector<int> order;
  std::vector<double> cost(count);
  std::vector<std::vector<int>> passes(count);  // wide circuits: chunk of each pass
  bt->final_perm.assign(count, {});
  bt->total_blocks = 0;
  const int k = QS_FUSE_K_OF(flags);
  qs_opts wide_opts = bt->opts;
  wide_opts.tile_bits = kTileBits;
  wide_opts.tile_k = std::min(k, 4);
  auto append = [&](const Block &b, int n, const int *tile_q) {
    const size_t at = pool.size(), w = record_words(b, n, tile_q);
    pool.resize(at + w);
    record_encode(b, pool.data() + at, n, tile_q, kTileBits);
    chunks.back().words += (int)w;
    chunks.back().n_recs++;
    bt->total_blocks++;
  };
  auto open_chunk = [&] {
    BChunk ch;
    std::memset(&ch, 0, sizeof(ch));
    ch.off = (long long)pool.size();
    chunks.push_back(ch);
  };
  for (size_t c = 0; c < count; c++) {
    const int n = state_n(bt->states[c]);
    const bool wide = n > kSmemBits;
    std::vector<Block> plan;
    PlanStats stats;
    std::string err;
    int8_t perm[QS_MAX_QUBITS];
    for (int q = 0; q < n; q++) perm[q] = (int8_t)q;
    const uint64_t f = wide ? (flags & QS_VSWAP) | QS_TILE : flags & ~(uint64_t)(QS_TC | QS_TILE);
    qs_status s = build_plan(n, bt->gates[c].data(), bt->gates[c].size(), f, wide ? wide_opts : bt->opts, perm, plan,
                             stats, err, false, /*allow_phase=*/!wide, /*repeated=*/true);
    if (s != QS_OK) return bfail(s, "qs_batch: circuit " + std::to_string(c) + ": " + err);
    bt->final_perm[c].assign(perm, perm + n);
    circs[c].amps = (float2 *)state_amps(bt->states[c]);
    circs[c].n = n;
    circs[c].first_chunk = (int)chunks.size();
    circs[c].n_chunks = 0;
    if (wide) {
      if (plan.empty()) {  // no gate: one pass that only writes |0...0>
        plan.emplace_back();
        plan[0].kind = BK_TILE;
        for (int j = 0; j < kTileBits; j++) plan[0].tile_q[j] = j;
      }
      for (const Block &t : plan) {
        if (t.kind != BK_TILE) return bfail(QS_EUNSUPPORTED, "qs_batch: unexpected block in a wide circuit's plan");
        passes[c].push_back((int)chunks.size());
        open_chunk();
        for (int j = 0; j < kTileBits; j++) chunks.back().tile_q[j] = t.tile_q[j];
        for (const Block &b : t.sub) append(b, n, t.tile_q);
      }
      continue;
    }
    order.push_back((int)c);
    cost[c] = std::ldexp(1.0, n) * (double)(plan.size() + 1);
    for (const Block &b : plan) {
      if (!record_encodable(b, n, QS_MAX_FUSE)) return bfail(QS_EUNSUPPORTED, "qs_batch: unexpected block in a plan");
      if (circs[c].n_chunks == 0 || chunks.back().words + record_words(b) > (size_t)kStageWords) {
        open_chunk();
        circs[c].n_chunks++;
      }
      append(b, 0, nullptr);
    }
  }
  bt->n_narrow = (int)order.size();
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
  // launch s: pass s of every wide circuit that has one
  std::vector<BStep> steps;
  for (size_t s = 0;; s++) {
    qs_batch::Launch l = {(int)steps.size(), 0, 0, 0};
    for (size_t c = 0; c < count; c++) {
      if (s >= passes[c].size()) continue;
      steps.push_back({(int)l.items, (int)c, passes[c][s]});
      l.items += 1ll << (circs[c].n - kTileBits);
      l.words = std::max(l.words, chunks[passes[c][s]].words);
      l.count++;
    }
    if (!l.count) break;
    bt->launches.push_back(l);
  }
  cudaError_t e = upload(bt->d_circs, circs);
  if (e == cudaSuccess) e = upload(bt->d_order, order);
  if (e == cudaSuccess) e = upload(bt->d_chunks, chunks);
  if (e == cudaSuccess) e = upload(bt->d_pool, pool);
  if (e == cudaSuccess) e = upload(bt->d_steps, steps);
  if (e == cudaErrorMemoryAllocation) return bfail(QS_ENOMEM, "qs_batch: descriptor allocation failed");
  if (e != cudaSuccess) return bfail(QS_ECUDA, std::string("qs_batch: upload failed: ") + cudaGetErrorString(e));
  return QS_OK;
}

cudaError_t launch_narrow(qs_batch *bt, int threads) {
  cudaError_t e = cudaMemsetAsync(bt->d_queue, 0, sizeof(int), bt->stream);
  if (e != cudaSuccess) return e;
  const int count = bt->n_narrow;
  const int grid = std::min(dev_info().sms, count);  // one CTA per SM: 161 KB of shared memory each
  bt->grid = grid;
  auto go = [&](auto kernel, int t) {
    kernel<<<grid, t, bt->smem, bt->stream>>>(bt->d_circs, bt->d_order, count, bt->d_chunks, bt->d_pool, bt->d_queue);
  };
  if (threads == 256) go(k_batch<256>, 256);
  else if (threads == 1024) go(k_batch<1024>, 1024);
  else go(k_batch<512>, 512);
  return cudaGetLastError();
}

cudaError_t launch_wide(qs_batch *bt, cudaStream_t s) {
  for (size_t i = 0; i < bt->launches.size(); i++) {
    const qs_batch::Launch &l = bt->launches[i];
    const size_t smem = (sizeof(float2) << kTileBits) + sizeof(uint4) * (size_t)l.words;
    const long long wave = (long long)dev_info().sms *
                           std::min(3, resident_ctas((const void *)k_batch_tile, kTileThreads, smem));
    const int grid = (int)std::min(wave, l.items);
    if (bt->n_narrow == 0) bt->grid = std::max(bt->grid, grid);
    k_batch_tile<<<grid, kTileThreads, smem, s>>>(bt->d_circs, bt->d_steps + l.first, l.count, l.items, bt->d_chunks,
                                                  bt->d_pool, i == 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The wide circuits on the side stream where there are narrow ones too.
cudaError_t launch_batch(qs_batch *bt, int threads) {
  if (bt->launches.empty()) return launch_narrow(bt, threads);
  if (bt->n_narrow == 0) return launch_wide(bt, bt->stream);
  cudaError_t e = cudaEventRecord(bt->fork, bt->stream);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(bt->side, bt->fork, 0);
  if (e == cudaSuccess) e = launch_wide(bt, bt->side);
  if (e == cudaSuccess) e = launch_narrow(bt, threads);
  if (e == cudaSuccess) e = cudaEventRecord(bt->join, bt->side);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(bt->stream, bt->join, 0);
  return e;
}

}  // namespace

extern "C" {

qs_status qs_batch_create(qs_state *const *states, const qs_gate *const *gates, const size_t *n_gates, int count,
                          uint64_t flags, const qs_opts *opts, void *cuda_stream, qs_batch **out) {
  if (!out || !states || !gates || !n_gates || count <= 0) return bfail(QS_EINVAL, "qs_batch_create: bad arguments");
  *out = nullptr;
  if (opts && opts->n_global != 0)
    return bfail(QS_EUNSUPPORTED, "qs_batch_create: global bits (opts.n_global) are for qs_plan only");
  qs_batch *bt = new (std::nothrow) qs_batch();
  if (!bt) return bfail(QS_ENOMEM, "qs_batch_create: host allocation failed");
  if (opts) bt->opts = *opts;
  else qs_default_opts(&bt->opts);
  bt->stream = (cudaStream_t)cuda_stream;
  cudaGetDevice(&bt->device);
  for (int c = 0; c < count; c++) {
    if (!states[c] || (n_gates[c] && !gates[c])) {
      delete bt;
      return bfail(QS_EINVAL, "qs_batch_create: null state or gate list");
    }
    if (!state_c64(states[c]) || state_n(states[c]) > kMaxBatchN) {
      delete bt;
      return bfail(QS_EUNSUPPORTED, "qs_batch_create: batches take complex64 states of at most 26 qubits");
    }
    for (int d = 0; d < c; d++)
      if (state_amps(states[d]) == state_amps(states[c])) {
        delete bt;
        return bfail(QS_EINVAL, "qs_batch_create: two entries share one state");
      }
    bt->states.push_back(states[c]);
    bt->gates.emplace_back(gates[c], gates[c] + n_gates[c]);
  }
  bt->smem = sizeof(uint4) * kStageWords + (sizeof(float2) << kSmemBits);
  cudaError_t e = cudaFuncSetAttribute(k_batch<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bt->smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_batch<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bt->smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_batch<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bt->smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_batch_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideSmemMax);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&bt->side, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&bt->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&bt->join, cudaEventDisableTiming);
  if (!bt->stream && e == cudaSuccess) {
    // the legacy stream cannot be captured: the batch runs on its own stream
    e = cudaStreamCreateWithFlags(&bt->own_stream, cudaStreamDefault);  // ordered with the legacy stream
    bt->stream = bt->own_stream;
  }
  if (e == cudaSuccess) e = qs::dev_malloc((void **)&bt->d_queue, sizeof(int));
  if (e != cudaSuccess) {
    qs_batch_free(bt);
    return bfail(QS_ECUDA, std::string("qs_batch_create: ") + cudaGetErrorString(e));
  }
  // fixed width, or autotune (fusion width x threads) on the batch itself
  std::vector<int> ks, ths = {256, 512, 1024};
  const int kfix = (flags & QS_FUSE) ? QS_FUSE_K_OF(flags) : 0;
  if (kfix) ks = {kfix};
  else ks = {2, 3, 4};
  if (bt->opts.threads > 0) ths = {bt->opts.threads};
  if (kfix >= 5) ths = {256};  // the wide mat-vecs need the 256-thread register budget
  const uint64_t base = (flags & (QS_VSWAP | QS_DIAG)) | QS_FUSE;
  double best = 1e300;
  int best_k = ks[0], best_t = ths[0];
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  for (int k : ks) {
    qs_status s = upload_plan(bt, base | QS_FUSE_K(k));
    if (s != QS_OK) {
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      qs_batch_free(bt);
      return s;
    }
    for (int t : ths) {
      float ms = 0;
      if (ks.size() * ths.size() > 1) {
        e = launch_batch(bt, t);  // warm-up
        if (e == cudaSuccess) e = cudaEventRecord(e0, bt->stream);
        if (e == cudaSuccess) e = launch_batch(bt, t);
        if (e == cudaSuccess) e = cudaEventRecord(e1, bt->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e != cudaSuccess) {
          cudaEventDestroy(e0);
          cudaEventDestroy(e1);
          qs_batch_free(bt);
          return bfail(QS_ECUDA, std::string("qs_batch_create: tuning launch failed: ") + cudaGetErrorString(e));
        }
        if (bt->n_tune < 16) {
          bt->tune_ms[bt->n_tune] = ms;
          bt->tune_k[bt->n_tune] = k;
          bt->tune_threads[bt->n_tune] = t;
          bt->n_tune++;
        }
      }
      if (ms < best) {
        best = ms;
        best_k = k;
        best_t = t;
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  qs_status s = upload_plan(bt, base | QS_FUSE_K(best_k));
  if (s != QS_OK) {
    qs_batch_free(bt);
    return s;
  }
  bt->k_chosen = best_k;
  bt->threads = best_t;
  bt->flags = base | QS_FUSE_K(best_k);
  // capture queue reset + kernel once; runs replay the graph
  e = cudaStreamBeginCapture(bt->stream, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    cudaError_t le = launch_batch(bt, bt->threads);
    e = cudaStreamEndCapture(bt->stream, &bt->graph);
    if (le != cudaSuccess) e = le;
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&bt->exec, bt->graph, 0);
  if (e != cudaSuccess) {
    cudaGetLastError();
    if (bt->graph) cudaGraphDestroy(bt->graph);
    bt->graph = nullptr;
    bt->exec = nullptr;  // direct launches instead (still one kernel per run)
  }
  *out = bt;
  return QS_OK;
}

qs_status qs_batch_run(qs_batch *bt) {
  if (!bt) return bfail(QS_EINVAL, "qs_batch_run: null batch");
  cudaError_t e = bt->exec ? cudaGraphLaunch(bt->exec, bt->stream) : launch_batch(bt, bt->threads);
  if (e != cudaSuccess) return bfail(QS_ECUDA, std::string("qs_batch_run: ") + cudaGetErrorString(e));
  for (size_t c = 0; c < bt->states.size(); c++)
    std::memcpy(state_perm(bt->states[c]), bt->final_perm[c].data(), bt->final_perm[c].size());
  return QS_OK;
}

qs_status qs_batch_sync(qs_batch *bt) {
  if (!bt) return bfail(QS_EINVAL, "qs_batch_sync: null batch");
  cudaError_t e = cudaStreamSynchronize(bt->stream);
  if (e != cudaSuccess) return bfail(QS_ECUDA, std::string("qs_batch_sync: ") + cudaGetErrorString(e));
  return QS_OK;
}

qs_status qs_batch_info(const qs_batch *bt, qs_batch_info_t *out) {
  if (!bt || !out) return bfail(QS_EINVAL, "qs_batch_info: null argument");
  std::memset(out, 0, sizeof(*out));
  out->count = (int)bt->states.size();
  out->fuse_k = bt->k_chosen;
  out->threads = bt->threads;
  out->grid = bt->grid;
  out->total_blocks = bt->total_blocks;
  out->graph = bt->exec != nullptr;
  out->n_tuned = bt->n_tune;
  for (int i = 0; i < bt->n_tune; i++) {
    out->tuned_k[i] = bt->tune_k[i];
    out->tuned_threads[i] = bt->tune_threads[i];
    out->tuned_ms[i] = bt->tune_ms[i];
  }
  return QS_OK;
}

void qs_batch_free(qs_batch *bt) {
  if (!bt) return;
  if (bt->stream) cudaStreamSynchronize(bt->stream);
  else cudaDeviceSynchronize();
  if (bt->exec) cudaGraphExecDestroy(bt->exec);
  if (bt->graph) cudaGraphDestroy(bt->graph);
  free_plan(bt);
  qs::dev_free(bt->d_queue);
  if (bt->side) cudaStreamDestroy(bt->side);
  if (bt->fork) cudaEventDestroy(bt->fork);
  if (bt->join) cudaEventDestroy(bt->join);
  if (bt->own_stream) cudaStreamDestroy(bt->own_stream);
  delete bt;
}

qs_status qs_apply_batch(qs_state *const *states, const qs_gate *const *gates, const size_t *n_gates, int count,
                         uint64_t flags, const qs_opts *opts) {
  qs_batch *bt = nullptr;
  qs_status s = qs_batch_create(states, gates, n_gates, count, flags, opts, nullptr, &bt);
  if (s != QS_OK) return s;
  s = qs_batch_run(bt);
  if (s == QS_OK) s = qs_batch_sync(bt);
  const std::string err = s == QS_OK ? std::string() : qs::last_error_ref();
  qs_batch_free(bt);
  if (s != QS_OK) qs::last_error_ref() = err;
  return s;
}

}  // extern "C"
