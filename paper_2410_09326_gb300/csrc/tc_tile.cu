// Tile passes on the tensor cores: several fused blocks in one HBM pass
// (complex64).
//
// A pass's tile spans 12 physical bits (0..3 and eight that the planner
// chose); one tile exists for every value of the other bits. A CTA of four
// warps loads a tile (32 KB) into shared memory, applies the pass's blocks there
// one after another and stores it. Every block has exactly five targets inside
// the tile (narrower ones are widened by an identity), so a tile is 128 groups
// of 32 amplitudes: one group per thread, the 128 rows of a tcgen05.mma. Bits
// outside the tile on which a block acts diagonally (controls, phases) are
// constant for the tile: they pick one of up to four matrices.
//
// Per block, a thread reads its group from shared memory, scales and splits it
// into FP16 halves as tc16.cu does, writes them to its lane of tensor memory
// (the MMA takes A from there: nothing but the tile and B is in shared
// memory), and after the MMAs brings its row of the product back to the
// group's norm (norm_fix) and writes it in place. The three products share one accumulator,
// the small ones first, so that the accumulation's truncation costs no more
// than with an accumulator of their own. B of the next block (16 KB, hi and
// lo) is copied in as soon as this block's MMAs have read theirs.
//
// At 26 qubits a pass of four blocks takes 321 us, three 274 us, one block by
// itself 172 us (one HBM pass: 160 us); the 30-qubit 30-layer random circuit
// 339 ms as single blocks, 165 to 169 on tile passes. Bound by the serial chain
// of a block, the issue slots at 47% and the shared-memory pipe at 52%. 13-bit tiles in two CTAs of 256 threads were 8% slower at 27 qubits,
// two accumulations of the large products 10% (their error 5% less).
//
// Shared memory holds amplitude i at byte address i * 8 with its 16-byte
// chunk's three lowest bits XORed by the chunk bits above them, three at a
// time; the host assigns free bits to lanes so that the eight (16-byte
// accesses) or sixteen (8-byte) lanes of a phase differ in distinct classes
// of those bits: no bank conflicts unless the targets take a whole class.
#include <cstddef>
#include <cstdint>
#include <cstring>

#include "tc16_common.cuh"

namespace qs {
namespace kern {

namespace {

constexpr int M = kTcTileBits;
constexpr int kTtGroups = M - 5;     // free bits of a block: log2 of the groups in a tile
constexpr int kTtThreads = 1 << kTtGroups;
static_assert(kTtThreads == 128, "one group per thread, 128 rows");
constexpr int kTtPerSm = 4;          // CTAs per SM: 48 KB of shared memory and 128 TMEM columns each
constexpr uint32_t kTtTileBytes = 8u << M;
constexpr uint32_t kTtMatBytes = kTcTileBBytes;  // B: 64 x 64, hi then lo
constexpr int kTtCols = 128;         // TMEM: 64 columns of D, 32 of A hi, 32 of A lo

struct alignas(16) TtBlock {
  uint32_t dt[5];          // XOR of the shared-memory address for each target
  uint32_t df[kTtGroups];  // and for each bit of the thread index
  uint32_t mat;            // its first matrix
  uint32_t skip;           // bit v: variant v is the identity
  uint8_t nsel;
  uint8_t sel[3];          // state bits that pick the variant
  uint32_t pad;
};
static_assert(sizeof(TtBlock) == 64 && kTcTileSel <= 3, "read as four 16-byte words");

struct TtParam {
  float2 *a;
  const uint4 *b;
  int *err;
  long long n_tiles;
  int tq[16];      // tile bits, ascending
  int n_blocks;
  int withhold_commit;
  int pad[2];
  TtBlock blk[kTcTileMaxBlocks];
};
static_assert(offsetof(TtParam, blk) % 16 == 0, "16-byte words");

// Shared-memory address of one bit of the tile index; addresses of whole
// indexes are XORs of these.
__host__ __device__ constexpr uint32_t tt_addr(int bit) {
  return (8u << bit) ^ (bit >= 4 ? 16u << ((bit - 1) % 3) : 0u);
}

// Two FP32 values in 64 bits, one operation on both (half the issue slots).
__device__ __forceinline__ uint64_t pack2(uint32_t x, uint32_t y) { return (uint64_t)y << 32 | x; }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float sum4(const uint64_t (&s)[2]) {
  return (__uint_as_float((uint32_t)s[0]) + __uint_as_float((uint32_t)(s[0] >> 32))) +
         (__uint_as_float((uint32_t)s[1]) + __uint_as_float((uint32_t)(s[1] >> 32)));
}

// The power of two (its bits) that brings a row of squared norm nin to a norm in
// [2^13, 2^14]: its components then fit FP16, and its low halves stay clear
// of the subnormals.
__device__ __forceinline__ uint32_t norm_scale(float nin) {
  const int e = (int)(__float_as_uint(nin) >> 23) - 126;  // nin in [2^(e - 1), 2^e)
  return (uint32_t)(127 + kOperandBits - ((e + 1) >> 1)) << 23;
}

// Brings a row of the product, scaled by sc and B's scale, back to the norm of
// its input: first by the small correction d = sqrt(r) - 1, then by a power of
// two. r = nin / nout is near 1, and so would one factor for both be: FP32 has
// no number there between 1 and 1 + 2^-23, so that the accumulation's
// truncation, a shrinking by less than that in every block, went uncorrected
// and added up: 64 blocks in a row were 1.78e-6 off (L2) where one is 1.2e-7,
// with the correction apart 8.7e-7 and 1.1e-7; the 19-qubit 30-layer random
// circuit 2.3e-6 and 8.6e-7. Approximate quotients and roots cost it nothing
// and the 30-qubit circuit 191 -> 165 ms against full ones.
struct NormFix {
  uint64_t d, s;  // twice each
  __device__ __forceinline__ uint64_t apply(uint64_t v) const { return mul2(fma2(v, d, v), s); }
};
__device__ __forceinline__ NormFix norm_fix(float nin, float nout) {
  constexpr float kB = (float)(1 << kOperandBits);
  const uint32_t scb = norm_scale(nin);  // again: it need not stay in a register
  const float sc = __uint_as_float(scb);
  // an exact difference of near numbers: approximate quotients and roots do for the rest
  // (-1 where nin has underflowed: the row becomes zero)
  const float r = nout > 0.f ? fmaxf(__fdividef(fmaf(nin * sc, sc * (kB * kB), -nout), nout), -1.f) : 0.f;
  float q;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(q) : "f"(1.f + r));
  const uint32_t d = __float_as_uint(__fdividef(r, 1.f + q));
  const uint32_t s = ((254u - kOperandBits) << 23) - scb;  // 1 / (sc * kB)
  return {pack2(d, d), pack2(s, s)};
}

// (x, y) -> FP16 halves hi, and lo = (x, y) - hi
__device__ __forceinline__ void split2(uint64_t xy, uint32_t &hi, uint32_t &lo) {
  const float x = __uint_as_float((uint32_t)xy), y = __uint_as_float((uint32_t)(xy >> 32));
  const __half2 h2 = __floats2half2_rn(x, y);
  hi = *reinterpret_cast<const uint32_t *>(&h2);
  float dx, dy;
  asm("{\n\t.reg .b16 a, b, m;\n\t"
      "mov.b32 {a, b}, %2;\n\t"
      "mov.b16 m, 0xBC00;\n\t"  // -1
      "fma.rn.f32.f16 %0, a, m, %3;\n\t"
      "fma.rn.f32.f16 %1, b, m, %4;\n\t}\n"
      : "=f"(dx), "=f"(dy)
      : "r"(hi), "f"(x), "f"(y));
  lo = pack_half2(dx, dy);
}

__global__ void __launch_bounds__(kTtThreads, kTtPerSm) k_tc_tile(const __grid_constant__ TtParam p) {
  constexpr uint32_t SBO = 8u * 128u, LBO = 128u;
  constexpr uint32_t IDESC = make_idesc_f16(128, 64);
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t mma_done;
  __shared__ __align__(8) uint64_t b_full;  // B has landed
  __shared__ uint32_t tmem_slot;
  __shared__ int next_slot;
  __shared__ TtBlock blk[kTcTileMaxBlocks];  // read with a varying index: faster from here than from the parameters
  const int tid = threadIdx.x, warp = tid >> 5;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "n"(kTtCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mma_done)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&b_full)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  for (int j = tid; j < p.n_blocks * 4; j += kTtThreads)
    reinterpret_cast<uint4 *>(blk)[j] = reinterpret_cast<const uint4 *>(p.blk)[j];
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
  const uint32_t done = smem_addr(&mma_done), full = smem_addr(&b_full);
  const uint32_t s_tile = smem_addr(smem), s_b = s_tile + kTtTileBytes;

  // Loads and stores: chunk tid + 128 k holds tile bits 1..7 = tid, 8..11 = k
  uint64_t toff = 2u * (uint64_t)(tid & 7);
  uint32_t taddr = 0;
#pragma unroll
  for (int j = 0; j < 7; j++)
    if ((tid >> j) & 1) {
      if (j >= 3) toff += 1ull << p.tq[1 + j];
      taddr ^= tt_addr(1 + j);
    }
  auto chunk_off = [&](int k) {
    uint64_t o = toff;
#pragma unroll
    for (int j = 0; j < 4; j++)
      if ((k >> j) & 1) o += 1ull << p.tq[8 + j];
    return o;
  };
  auto chunk_addr = [&](int k) {
    uint32_t x = taddr;
#pragma unroll
    for (int j = 0; j < 4; j++)
      if ((k >> j) & 1) x ^= tt_addr(8 + j);
    return x;
  };
  auto variant = [&](int i, uint64_t base) {
    const TtBlock &x = blk[i];
    uint32_t v = 0;
#pragma unroll
    for (int j = 0; j < kTcTileSel; j++)
      if (j < x.nsel) v |= (uint32_t)((base >> x.sel[j]) & 1) << j;
    return v;
  };
  // the first block from i on that is not the identity on this tile
  auto next_block = [&](int i, uint64_t base) {
    while (i < p.n_blocks && ((blk[i].skip >> variant(i, base)) & 1)) i++;
    return i;
  };
  auto b_of = [&](int i, uint64_t base) {
    return p.b + (size_t)(blk[i].mat + variant(i, base)) * (kTtMatBytes / 16);
  };
  // one thread fetches B; its arrival flips the phase of b_full
  auto load_b = [&](const uint4 *src) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full), "n"(kTtMatBytes) : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s_b), "l"(src),
        "n"(kTtMatBytes), "r"(full)
        : "memory");
  };
  // the next tile with something to do, from t on
  auto seek = [&](long long &t, uint64_t &base, int &i) {
    for (; t < p.n_tiles; t += gridDim.x) {
      base = insert_zeros((uint64_t)t, p.tq, M);
      i = next_block(0, base);
      if (i < p.n_blocks) return;
    }
  };
  struct Addr {
    uint32_t g, dt[5];  // shared-memory address of the thread's group, XORs of the targets
  };
  auto addr_of = [&](int i) {
    Addr x;
    x.g = 0;
#pragma unroll
    for (int j = 0; j < kTtGroups; j++)
      if ((tid >> j) & 1) x.g ^= blk[i].df[j];
#pragma unroll
    for (int j = 0; j < 5; j++) x.dt[j] = blk[i].dt[j];
    return x;
  };

  long long t = blockIdx.x;
  uint64_t base = 0;
  int i = 0;
  uint32_t parity = 0;  // of both barriers: every block flips each once
  bool aborted = false;
  seek(t, base, i);
  if (t < p.n_tiles) {
#pragma unroll 4
    for (int k = 0; k < 16; k++) cp_async16(s_tile + chunk_addr(k), p.a + base + chunk_off(k));
    if (tid == 32) load_b(b_of(i, base));
  }
  while (t < p.n_tiles) {
    long long t1 = t + gridDim.x;  // the tile after this one
    uint64_t base1 = 0;
    int i1 = 0;
    seek(t1, base1, i1);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // the tile is in
    while (i < p.n_blocks) {
      const Addr cur = addr_of(i);
      auto slot_addr = [&](int s) {
        uint32_t x = cur.g;
#pragma unroll
        for (int j = 0; j < 5; j++)
          if ((s >> j) & 1) x ^= cur.dt[j];
        return x;
      };
      const bool pair = cur.dt[0] == tt_addr(0);  // bit 0 is a target: slots 2 j and 2 j + 1 are adjacent
      uint64_t v[32];
      if (pair) {
#pragma unroll
        for (int s = 0; s < 32; s += 2) {
          const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(smem + slot_addr(s));
          v[s] = x.x;
          v[s + 1] = x.y;
        }
      } else {
#pragma unroll
        for (int s = 0; s < 32; s++) v[s] = *reinterpret_cast<const uint64_t *>(smem + slot_addr(s));
      }
      uint64_t s2[2] = {0, 0};  // four chains
#pragma unroll
      for (int s = 0; s < 32; s++) s2[s & 1] = fma2(v[s], v[s], s2[s & 1]);
      const float nin = sum4(s2);
      const uint32_t sc1 = norm_scale(nin);
      const uint64_t sc = pack2(sc1, sc1);
      // slot s (re, im) -> column s of A hi and of A lo
#pragma unroll
      for (int hh = 0; hh < 2; hh++) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int s = 0; s < 16; s++) split2(mul2(v[16 * hh + s], sc), hi[s], lo[s]);
        TmemSt<16>::run(lane_base + 64 + 16 * hh, hi);
        TmemSt<16>::run(lane_base + 96 + 16 * hh, lo);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncthreads();  // A is in
      asm volatile("tcgen05.fence::after_thread_sync;");
      if (tid == 0 && mbar_wait(full, parity)) {
        const uint32_t b_hi = s_b, b_lo = b_hi + kTtMatBytes / 2;
        const uint32_t a_hi = tmem + 64, a_lo = tmem + 96;
#pragma unroll
        for (int ks = 0; ks < 4; ks++)
          mma_f16_ta(tmem, a_hi + 8u * ks, make_desc(b_lo + 2u * LBO * ks, LBO, SBO), IDESC, ks > 0 ? 1u : 0u);
#pragma unroll
        for (int ks = 0; ks < 4; ks++)
          mma_f16_ta(tmem, a_lo + 8u * ks, make_desc(b_hi + 2u * LBO * ks, LBO, SBO), IDESC, 1u);
#pragma unroll
        for (int ks = 0; ks < 4; ks++)
          mma_f16_ta(tmem, a_hi + 8u * ks, make_desc(b_hi + 2u * LBO * ks, LBO, SBO), IDESC, 1u);
        if (!p.withhold_commit) mma_commit(done);
      }
      // meanwhile one thread looks up the next block and its B
      const uint4 *nxt_b = nullptr;
      if (tid == 32) {
        const int in = next_block(i + 1, base);
        next_slot = in;
        if (in < p.n_blocks) nxt_b = b_of(in, base);
        else if (t1 < p.n_tiles) nxt_b = b_of(i1, base1);
      }
      const bool ok = __all_sync(0xffffffffu, mbar_wait(done, parity));
      parity ^= 1;
      if (ok) {
        if (tid == 32 && nxt_b) load_b(nxt_b);  // the MMAs have read B
        asm volatile("tcgen05.fence::after_thread_sync;");
        uint32_t y[64];
        TmemLd<64>::run(lane_base, y);
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        uint64_t o2[2] = {0, 0};
#pragma unroll
        for (int s = 0; s < 32; s++) {
          v[s] = pack2(y[2 * s], y[2 * s + 1]);
          o2[s & 1] = fma2(v[s], v[s], o2[s & 1]);
        }
        const NormFix f = norm_fix(nin, sum4(o2));
        if (pair) {
#pragma unroll
          for (int s = 0; s < 32; s += 2)
            *reinterpret_cast<ulonglong2 *>(smem + slot_addr(s)) = make_ulonglong2(f.apply(v[s]), f.apply(v[s + 1]));
        } else {
#pragma unroll
          for (int s = 0; s < 32; s++) *reinterpret_cast<uint64_t *>(smem + slot_addr(s)) = f.apply(v[s]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
      }
      if (!__syncthreads_and(ok)) {
        if (tid == 0) atomicExch(p.err, 1);
        aborted = true;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      i = next_slot;
    }
    if (aborted) break;
    // a thread stores its chunks and refills them with the next tile's
#pragma unroll
    for (int k0 = 0; k0 < 16; k0 += 8) {
      float4 x[8];
#pragma unroll
      for (int k = 0; k < 8; k++) x[k] = *reinterpret_cast<const float4 *>(smem + chunk_addr(k0 + k));
#pragma unroll
      for (int k = 0; k < 8; k++) *reinterpret_cast<float4 *>(p.a + base + chunk_off(k0 + k)) = x[k];
      if (t1 < p.n_tiles) {
#pragma unroll
        for (int k = 0; k < 8; k++) cp_async16(s_tile + chunk_addr(k0 + k), p.a + base1 + chunk_off(k0 + k));
      }
    }
    t = t1;
    base = base1;
    i = i1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (aborted) {
    // MMAs and a copy of B may still be in flight: have the MMAs' completion
    // signalled and give both a bounded chance to land (where no copy is in
    // flight the second wait runs out)
    if (tid == 0) {
      mma_commit(done);
      mbar_wait(done, parity ^ 1);
      mbar_wait(full, parity);
    }
    __syncthreads();
  }
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTtCols));
}

// The gates of a plan's members as uploaded: a table of (member's place in
// 16-byte words, variant), one entry per product, padded to a multiple of
// two; then per member its gate count and gates (16 bytes each), and their
// matrices, row-major FP64.
struct TtGate {
  int8_t nq, at[3];  // as Block::Member
  uint32_t mat;      // 16-byte words from the member's start
  uint32_t pad[2];
};
static_assert(sizeof(TtGate) == 16, "16-byte words");

// Applies a gate on NT of the product's five bits: thread (warp w, lane c)
// updates column c of every fourth group of rows. z is the gate's matrix,
// off[l] the row bits of its index l. Zeros and unchanged rows, the same for
// all threads, are skipped; the tests are on bits, since comparisons would
// share the FP64 pipe.
template <int NT>
__device__ __forceinline__ void left_apply(double2 (&m)[32][32], const double2 *z, int tm, const int (&off)[8]) {
  constexpr int D = 1 << NT;
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto bits_zero = [](double v) { return (__double2hiint(v) << 1 | __double2loint(v)) == 0; };
  auto is_one = [&](double2 v) {
    return __double2hiint(v.x) == 0x3ff00000 && __double2loint(v.x) == 0 && bits_zero(v.y);
  };
  for (int q = w; q < (32 >> NT); q += 4) {
    int row = q;  // the q-th row whose target bits are 0
#pragma unroll
    for (int j = 0; j < 5; j++)
      if ((tm >> j) & 1) row = ((row >> j) << (j + 1)) | (row & ((1 << j) - 1));
    double2 x[D];
#pragma unroll
    for (int l = 0; l < D; l++) x[l] = m[row | off[l]][c];
#pragma unroll
    for (int r = 0; r < D; r++) {
      double2 s = make_double2(0.0, 0.0);
      bool same = true, first = true;
#pragma unroll
      for (int l = 0; l < D; l++) {
        const double2 g = z[r * D + l];
        const bool re = !bits_zero(g.x), im = !bits_zero(g.y);
        if (!re && !im) {
          same = same && l != r;
          continue;
        }
        if (is_one(g)) {
          same = same && l == r;
          if (first) s = x[l];
          else s.x += x[l].x, s.y += x[l].y;
          first = false;
          continue;
        }
        same = first = false;
        if (re) {
          s.x = fma(g.x, x[l].x, s.x);
          s.y = fma(g.x, x[l].y, s.y);
        }
        if (im) {
          s.x = fma(-g.y, x[l].y, s.x);
          s.y = fma(g.y, x[l].x, s.y);
        }
      }
      if (!same) m[row | off[r]][c] = s;
    }
  }
}

// One product per CTA: the 32 x 32 matrix in FP64, gate by gate from the left
// in shared memory, then B: its real embedding, rounded to FP32, scaled, split
// into FP16 halves and laid out in the MMA's core matrices (as operands.cu
// does). The next gate's matrix is fetched while one is applied. Bound by the
// FP64 rate, two multiply-adds per clock and SM (a one-qubit gate of real and
// imaginary entries is 4096 clocks): 65 us for the 158 products of the 19-qubit
// 30-layer random circuit, 178 us with one loop for all gate sizes, FP64
// comparisons and the matrix read from global memory entry by entry.
__global__ void __launch_bounds__(128) k_tc_tile_product(const uint4 *__restrict__ prog, uint4 *__restrict__ b) {
  __shared__ double2 m[32][32];
  __shared__ double2 z[2][64];
  const int tid = threadIdx.x, c = tid & 31, w = tid >> 5;
  const uint2 entry = reinterpret_cast<const uint2 *>(prog)[blockIdx.x];
  const uint4 *member = prog + entry.x;
  const int n_gates = (int)member->x;
  struct Gate {
    int nt, tm;    // its bits inside the product
    double2 e;     // thread i < 4^nt: entry i of its matrix
    int off[8];
  };
  auto fetch = [&](int i) {
    Gate o;
    const TtGate g = reinterpret_cast<const TtGate *>(member + 1)[i];
    int fixed = 0, bit[3] = {0, 0, 0}, at[3] = {0, 0, 0};
    o.nt = o.tm = 0;
#pragma unroll
    for (int j = 0; j < 3; j++) {
      if (j >= g.nq) continue;
      if (g.at[j] < 0) {
        fixed |= (int)((entry.y >> (-1 - g.at[j])) & 1) << j;
        continue;
      }
      o.tm |= 1 << g.at[j];
#pragma unroll
      for (int u = 0; u < 3; u++)
        if (u == o.nt) bit[u] = 1 << j, at[u] = 1 << g.at[j];
      o.nt++;
    }
#pragma unroll
    for (int l = 0; l < 8; l++) {
      o.off[l] = 0;
#pragma unroll
      for (int u = 0; u < 3; u++)
        if ((l >> u) & 1) o.off[l] |= at[u];
    }
    // the entry's row and column in the gate's own matrix: the outer bits fixed
    int r = fixed, k = fixed;
#pragma unroll
    for (int u = 0; u < 3; u++) {
      if ((tid >> u) & 1 && u < o.nt) k |= bit[u];
      if ((tid >> (o.nt + u)) & 1 && u < o.nt) r |= bit[u];
    }
    o.e = make_double2(0.0, 0.0);
    if (tid < 1 << (2 * o.nt)) o.e = reinterpret_cast<const double2 *>(member + g.mat)[(r << g.nq) + k];
    return o;
  };
  for (int r = w; r < 32; r += 4) m[r][c] = make_double2(r == c ? 1.0 : 0.0, 0.0);
  Gate cur = fetch(0);
  for (int i = 0; i < n_gates; i++) {
    if (tid < 64) z[i & 1][tid] = cur.e;
    __syncthreads();
    Gate nxt = cur;
    if (i + 1 < n_gates) nxt = fetch(i + 1);
    switch (cur.nt) {
      case 1: left_apply<1>(m, z[i & 1], cur.tm, cur.off); break;
      case 2: left_apply<2>(m, z[i & 1], cur.tm, cur.off); break;
      case 3: left_apply<3>(m, z[i & 1], cur.tm, cur.off); break;
      default: {  // a phase of the outer bits alone
        int none[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        left_apply<0>(m, z[i & 1], 0, none);
      }
    }
    cur = nxt;
  }
  __syncthreads();
  // one 16-byte row of a core matrix at a time
  uint4 *out = b + (size_t)blockIdx.x * (kTtMatBytes / 16);
  for (int x = tid; x < 512; x += 128) {
    const int row = (x >> 3) & 63, cg = x & 7;
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const double2 u = m[row >> 1][cg * 4 + e];
      operand_halves(row & 1, (float)u.x, (float)u.y, hi[e], lo[e]);
    }
    uint4 *o = out + (row >> 3) * 64 + cg * 8 + (row & 7);
    o[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    o[kTtMatBytes / 32] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

}  // namespace

size_t tc_tile_mats(const Block &b) {
  size_t m = 0;
  for (const Block &s : b.sub) m += (size_t)1 << s.nsel;
  return m;
}

cudaError_t run_tc_tile(float2 *a, int n, const Block &b, const void *dev_b, int *err, cudaStream_t s,
                        LaunchShape *shape) {
  static thread_local TtParam p;
  if (b.k != M || b.sub.size() > (size_t)kTcTileMaxBlocks) return cudaErrorInvalidValue;
  std::memset(&p, 0, sizeof(p));
  p.a = a;
  p.b = (const uint4 *)dev_b;
  p.err = err;
  p.n_tiles = 1ll << (n - M);
  p.withhold_commit = b.withhold_commit ? 1 : 0;
  for (int j = 0; j < M; j++) p.tq[j] = b.tile_q[j];
  uint32_t mat = 0;
  for (const Block &m : b.sub) {
    TtBlock &o = p.blk[p.n_blocks++];
    if (m.k != 5) return cudaErrorInvalidValue;
    uint32_t tmask = 0;
    for (int j = 0, at = 0; j < 5; j++) {
      while (at < M && b.tile_q[at] != m.q[j]) at++;
      if (at == M) return cudaErrorInvalidValue;
      o.dt[j] = tt_addr(at);
      tmask |= 1u << at;
    }
    // free bits to thread bits: bit 0 first where it is free, then one bit of
    // each class, then the others
    int order[kTtGroups], cnt = 0;
    uint32_t left = ((1u << M) - 1) & ~tmask;
    auto take = [&](int bit) {
      order[cnt++] = bit;
      left &= ~(1u << bit);
    };
    if (left & 1) take(0);
    for (int c = 0; c < 3; c++)
      for (int bit = 1 + c; bit < M; bit += 3)
        if ((left >> bit) & 1) {
          take(bit);
          break;
        }
    for (int bit = 0; bit < M; bit++)
      if ((left >> bit) & 1) take(bit);
    for (int j = 0; j < kTtGroups; j++) o.df[j] = tt_addr(order[j]);
    o.mat = mat;
    o.nsel = (uint8_t)m.nsel;
    for (int j = 0; j < m.nsel; j++) o.sel[j] = (uint8_t)m.sel[j];
    o.skip = m.skip;
    mat += 1u << m.nsel;
  }
  const size_t smem = kTtTileBytes + kTtMatBytes;
  static thread_local int configured = -1;
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured != dev) {
    cudaError_t e = cudaFuncSetAttribute(k_tc_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    configured = dev;
  }
  const int grid = tc_grid((long long)kTtPerSm * dev_info().sms, p.n_tiles, b.tc_max_ctas);
  if (shape) {
    shape->tiles = p.n_tiles;
    shape->ctas = grid;
  }
  k_tc_tile<<<grid, kTtThreads, smem, s>>>(p);
  return cudaGetLastError();
}

}  // namespace kern

using namespace kern;

size_t operand_program_bytes(const Block *blocks, size_t count) {
  size_t products = 0, words = 0;
  for (size_t i = 0; i < count; i++) {
    const Block &b = blocks[i];
    if (!dev_operand_bytes(b)) continue;
    products += tc_tile_mats(b);
    for (const Block &m : b.sub) words += 1 + m.gates.size() + m.mat.size();
  }
  return 16 * ((products + 1) / 2 + words);
}

void fill_operand_program(const std::vector<Block> &plan, void *out) {
  static_assert(sizeof(cd) == 16, "matrix entries are 16-byte words");
  size_t products = 0;
  for (const Block &b : plan)
    if (dev_operand_bytes(b)) products += tc_tile_mats(b);
  uint32_t *table = (uint32_t *)out;
  size_t at = (products + 1) / 2;
  for (const Block &b : plan) {
    if (!dev_operand_bytes(b)) continue;
    for (const Block &m : b.sub) {
      for (uint32_t v = 0; v < (1u << m.nsel); v++) {
        *table++ = (uint32_t)at;
        *table++ = v;
      }
      unsigned char *p = (unsigned char *)out + 16 * at;
      const uint32_t head[4] = {(uint32_t)m.gates.size(), 0, 0, 0};
      std::memcpy(p, head, 16);
      uint32_t mat = 1 + (uint32_t)m.gates.size();
      std::memcpy(p + 16 * (size_t)mat, m.mat.data(), 16 * m.mat.size());
      for (size_t i = 0; i < m.gates.size(); i++) {
        TtGate g = {m.gates[i].nq, {m.gates[i].at[0], m.gates[i].at[1], m.gates[i].at[2]}, mat, {0, 0}};
        std::memcpy(p + 16 * (1 + i), &g, 16);
        mat += 1u << (2 * g.nq);
      }
      at += mat;
    }
  }
}

cudaError_t build_dev_operands(const void *program, void *out, size_t bytes, cudaStream_t s) {
  k_tc_tile_product<<<(unsigned)(bytes / kTcTileBBytes), 128, 0, s>>>((const uint4 *)program, (uint4 *)out);
  return cudaGetLastError();
}

}  // namespace qs
