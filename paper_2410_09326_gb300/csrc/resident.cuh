// Running a list of fused blocks on complex64 amplitudes that one CTA holds in
// shared memory: the encoded records and the device code that applies them.
// Used by narrow states (resident.cu: the whole state) and by batches
// (batch.cu: a narrow circuit's state, or a tile of a wide one's).
//
// A record is a header followed by the block's matrix, phase table or
// angles, in 16-byte words; the next record follows it. Bit positions are
// those inside the CTA's array; a tile's controls outside it are in gmask.
#pragma once
#include <cstdint>
#include <vector>

#include "kernels_common.cuh"

namespace qs {
namespace kern {

constexpr int kResidentPhaseBits = 14;  // widest state whose phase polynomials can be encoded

struct RecHead {
  uint32_t words;     // record length in 16-byte words, header included
  uint8_t kind;       // BlockKind: dense, diagonal, exchange, phase polynomial
  uint8_t k;          // dense targets, table qubits
  uint8_t nf;         // fixed bits of the index: targets and controls (diagonal: controls)
  uint8_t wide;       // phase polynomial seen tile by tile: the state's qubits, else 0
  uint32_t cmask;     // control bits
  uint32_t gmask;     // control bits outside the tile, as bits of the state's index
  uint8_t fixed[kMaxFixed];
  uint8_t tq[16];     // targets, table qubits, exchanged bits
  uint8_t pad3[8];
};
static_assert(sizeof(RecHead) == 64, "record header");

// Angles of a phase polynomial as 32-bit fractions of a turn (sums wrap as
// angles do, and add without rounding): constant, one per bit, one per pair.
struct RecPhase {
  uint32_t c, pad[3];
  uint32_t a[16];
  uint32_t b[kResidentPhaseBits][16];  // symmetric
};

// The same for a state of nb qubits seen tile by tile: the constant, then a
// row of nb angles, then nb rows of the symmetric pair angles, rows padded to
// a multiple of four.
inline uint32_t wide_phase_row(int nb) { return (uint32_t)(nb + 3) & ~3u; }

// Host side (resident.cu). record_encodable is false for a block the records
// do not cover. tile_q (m entries) makes a record for a tile over those bits
// of an n-qubit state; null for the whole state.
bool record_encodable(const Block &b, int n, int max_k);
size_t record_words(const Block &b, int n = 0, const int *tile_q = nullptr);
void record_encode(const Block &b, uint4 *out, int n = 0, const int *tile_q = nullptr, int m = 0);

#ifdef __CUDACC__

__device__ __forceinline__ uint32_t rec_insert(uint32_t j, const RecHead &h) {
  for (int i = 0; i < h.nf; i++) {
    const int p = h.fixed[i];
    j = ((j >> p) << (p + 1)) | (j & ((1u << p) - 1));
  }
  return j;
}

// One thread per G groups, blockDim.x apart from first; the matrix is read from
// shared memory two entries at a time, the same address for the whole warp.
// Those reads bound a mat-vec of one group, so two groups share them where
// there are that many (a batch of 192 QAOA circuits 3.37 -> 2.97 ms a run).
// Four groups, with two CTAs per SM instead of three: 3.03 ms. Entries kept as
// (x, x, -y, y) for packed multiply-adds, twice the words, 3.58 ms.
template <int K, int G>
__device__ __forceinline__ void rec_dense_groups(float2 *a, const RecHead &h, const float4 *m, uint32_t first) {
  constexpr int D = 1 << K;
  uint32_t d[K];
#pragma unroll
  for (int j = 0; j < K; j++) d[j] = 1u << h.tq[j];
  auto off = [&](int s) {
    uint32_t o = 0;
#pragma unroll
    for (int j = 0; j < K; j++)
      if ((s >> j) & 1) o += d[j];
    return o;
  };
  float2 *p[G];
  float2 v[G][D];
#pragma unroll
  for (int g = 0; g < G; g++) {
    p[g] = a + (rec_insert(first + g * blockDim.x, h) | h.cmask);
#pragma unroll
    for (int s = 0; s < D; s++) v[g][s] = p[g][off(s)];
  }
#pragma unroll
  for (int r = 0; r < D; r++) {
    float re0[G], im0[G], re1[G], im1[G];
#pragma unroll
    for (int g = 0; g < G; g++) re0[g] = im0[g] = re1[g] = im1[g] = 0.f;
#pragma unroll
    for (int c = 0; c < D; c += 2) {
      const float4 w = m[r * (D / 2) + c / 2];
#pragma unroll
      for (int g = 0; g < G; g++) {
        re0[g] = fmaf(w.x, v[g][c].x, fmaf(-w.y, v[g][c].y, re0[g]));
        im0[g] = fmaf(w.x, v[g][c].y, fmaf(w.y, v[g][c].x, im0[g]));
        re1[g] = fmaf(w.z, v[g][c + 1].x, fmaf(-w.w, v[g][c + 1].y, re1[g]));
        im1[g] = fmaf(w.z, v[g][c + 1].y, fmaf(w.w, v[g][c + 1].x, im1[g]));
      }
    }
#pragma unroll
    for (int g = 0; g < G; g++) p[g][off(r)] = make_float2(re0[g] + re1[g], im0[g] + im1[g]);
  }
}

template <int K> __device__ __forceinline__ void rec_dense(float2 *a, int n, const RecHead &h, const float4 *m) {
  const uint32_t groups = 1u << (n - h.nf);
  if (K <= 3 && groups >= 2 * blockDim.x) {  // powers of two: whole pairs
    if constexpr (K <= 3)
      for (uint32_t g = threadIdx.x; g < groups; g += 2 * blockDim.x) rec_dense_groups<K, 2>(a, h, m, g);
    return;
  }
  for (uint32_t g = threadIdx.x; g < groups; g += blockDim.x) rec_dense_groups<K, 1>(a, h, m, g);
}

__device__ __forceinline__ float2 rec_cmul(float2 w, float2 v) {
  return make_float2(fmaf(w.x, v.x, -w.y * v.y), fmaf(w.x, v.y, w.y * v.x));
}

// exp(2 pi i p / 2^32): the nearest quarter turn is taken off exactly, so the
// rest converts to FP32 with an error below 2^-27 of a turn.
__device__ __forceinline__ float2 turn(uint32_t p) {
  const uint32_t q = (p + 0x20000000u) >> 30;
  const float f = (float)(int32_t)(p - (q << 30)) * 4.656612873e-10f;  // half turns, 2^-31
  float s, c;
  sincospif(f, &s, &c);
  const float x = (q & 1) ? -s : c, y = (q & 1) ? c : s;
  return (q & 2) ? make_float2(-x, -y) : make_float2(x, y);
}

// A thread's amplitudes differ only in the bits above the thread index: the
// terms among and with the lower bits are summed once, those of the bits above
// the lowest three of them once for eight amplitudes. (Summed anew for each
// amplitude, these integer additions took as many issue slots as all else that
// a batch's tile kernel does.)
__device__ __forceinline__ void rec_phase(float2 *a, int n, const RecPhase &ph) {
  const int tb = 31 - __clz(blockDim.x);  // a power of two of threads
  const uint32_t t = threadIdx.x;
  uint32_t phi0 = ph.c;
  for (int i = 0; i < min(tb, n); i++) {
    uint32_t s = ph.a[i];
    for (int l = 0; l < i; l++)
      if ((t >> l) & 1) s += ph.b[i][l];
    if ((t >> i) & 1) phi0 += s;
  }
  // terms of the bits above with the lower ones (256 threads and 14 qubits: 6 bits)
  uint32_t up[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < 6; i++)
    if (tb + i < n) {
      up[i] = ph.a[tb + i];
      for (int l = 0; l < tb; l++)
        if ((t >> l) & 1) up[i] += ph.b[tb + i][l];
    }
  uint32_t pair[3] = {0, 0, 0};  // among the lowest three: (1, 0), (2, 0), (2, 1)
  if (tb + 1 < n) pair[0] = ph.b[tb + 1][tb];
  if (tb + 2 < n) pair[1] = ph.b[tb + 2][tb], pair[2] = ph.b[tb + 2][tb + 1];
  const uint32_t all = 1u << n;
  for (uint32_t j = 0; 8 * j * blockDim.x < all; j++) {
    uint32_t base = phi0, u[3] = {up[0], up[1], up[2]};
#pragma unroll
    for (int i = 0; i < 3; i++)
      if ((j >> i) & 1) {  // bit tb + 3 + i is set
        const uint32_t *row = ph.b[tb + 3 + i] + tb;
        base += up[3 + i];
#pragma unroll
        for (int l = 0; l < 3; l++) u[l] += row[l];
#pragma unroll
        for (int l = 0; l < i; l++)
          if ((j >> l) & 1) base += row[3 + l];
      }
#pragma unroll
    for (uint32_t e = 0; e < 8; e++) {
      const uint32_t x = t + (8 * j + e) * blockDim.x;
      uint32_t phi = base;
      if (e & 1) phi += u[0];
      if (e & 2) phi += u[1] + ((e & 1) ? pair[0] : 0u);
      if (e & 4) phi += u[2] + ((e & 1) ? pair[1] : 0u) + ((e & 2) ? pair[2] : 0u);
      if (x < all) a[x] = rec_cmul(turn(phi), a[x]);
    }
  }
}

// The tile's own polynomial: the bits outside it are fixed (base), so their
// terms join the constant and the linear angles.
__device__ __forceinline__ void tile_phase(const uint32_t *w, int nb, int m, const int *tile_q, uint32_t base,
                                           RecPhase &out) {
  const int row = (nb + 3) & ~3;
  const uint32_t *la = w + 4, *lb = la + row;
  uint32_t inside = 0;
  for (int j = 0; j < m; j++) inside |= 1u << tile_q[j];
  const uint32_t set = base & ~inside;
  for (int t = threadIdx.x; t < m + m * m + 1; t += blockDim.x) {
    if (t < m) {
      const int q = tile_q[t];
      uint32_t s = la[q];
      for (uint32_t r = set; r; r &= r - 1) s += lb[q * row + __ffs(r) - 1];
      out.a[t] = s;
    } else if (t < m + m * m) {
      const int i = (t - m) / m, l = (t - m) % m;
      out.b[i][l] = lb[tile_q[i] * row + tile_q[l]];
    } else {
      uint32_t s = w[0];
      for (uint32_t r = set; r; r &= r - 1) {
        const int q = __ffs(r) - 1;
        s += la[q];
        for (uint32_t r2 = r & (r - 1); r2; r2 &= r2 - 1) s += lb[q * row + __ffs(r2) - 1];
      }
      out.c = s;
    }
  }
  __syncthreads();
}

// Applies one record; ends with the CTA synchronised. MAXT bounds the
// registers: the 5- and 6-target mat-vecs exist where it is at most 256.
// TILE: a is a tile over the n bits tile_q, at base in the state; its blocks
// have at most four targets.
template <int MAXT, bool TILE = false>
__device__ __forceinline__ void rec_apply(float2 *a, int n, const uint4 *rec, uint32_t base = 0,
                                          const int *tile_q = nullptr, RecPhase *scratch = nullptr) {
  const RecHead &h = *reinterpret_cast<const RecHead *>(rec);
  if (TILE && (base & h.gmask) != h.gmask) return;  // the same for the whole CTA
  const uint4 *body = rec + sizeof(RecHead) / 16;
  if (h.kind == BK_DENSE) {
    const float4 *m = reinterpret_cast<const float4 *>(body);
    switch (h.k) {
      case 1: rec_dense<1>(a, n, h, m); break;
      case 2: rec_dense<2>(a, n, h, m); break;
      case 3: rec_dense<3>(a, n, h, m); break;
      case 4: rec_dense<4>(a, n, h, m); break;
      case 5:
        if constexpr (MAXT <= 256 && !TILE) rec_dense<5>(a, n, h, m);
        break;
      case 6:
        if constexpr (MAXT <= 256 && !TILE) rec_dense<6>(a, n, h, m);
        break;
      default: break;
    }
  } else if (h.kind == BK_DIAG) {
    const float2 *tab = reinterpret_cast<const float2 *>(body);
    const uint32_t amps = 1u << (n - h.nf);
    for (uint32_t j = threadIdx.x; j < amps; j += blockDim.x) {
      const uint32_t idx = rec_insert(j, h) | h.cmask;
      uint32_t l = 0;
      for (int t = 0; t < h.k; t++) l |= ((idx >> h.tq[t]) & 1) << t;
      a[idx] = rec_cmul(tab[l], a[idx]);
    }
  } else if (h.kind == BK_PERMUTE) {
    const uint32_t b0 = 1u << h.tq[0], b1 = 1u << h.tq[1];
    for (uint32_t j = threadIdx.x; j < (1u << (n - 2)); j += blockDim.x) {
      const uint32_t i = rec_insert(j, h);
      const float2 x = a[i | b0];
      a[i | b0] = a[i | b1];
      a[i | b1] = x;
    }
  } else if constexpr (TILE) {
    tile_phase(reinterpret_cast<const uint32_t *>(body), h.wide, n, tile_q, base, *scratch);
    rec_phase(a, n, *scratch);
  } else {
    rec_phase(a, n, *reinterpret_cast<const RecPhase *>(body));
  }
  __syncthreads();
}

#endif  // __CUDACC__

}  // namespace kern
}  // namespace qs
