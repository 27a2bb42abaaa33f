// Dense fused blocks of 4 and 5 targets in complex128 on the tensor cores.
//
// GB300 runs about two FP64 multiply-adds per SM and clock (1.2 TFLOP/s in
// all), so an FP64 mat-vec of 5 targets -- 128 of them per amplitude -- takes
// 45 times as long as reading and writing the state. The FP16 tensor cores
// are exact on small integers, and that is what this kernel uses: both
// operands become fixed-point numbers cut into balanced base-256 digits, all
// digit products of one weight are summed exactly in an FP32 accumulator, and
// the accumulators are put together as 64-bit integers and rounded to FP64
// once. (Splitting floating-point matrix products into exact slices: Ozaki,
// Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012.)
//
//  - A: a group's 2^(K+1) reals, scaled by the power of two that brings the
//    group's largest into [1/4, 1/2), then x = sum_i a_i 2^(-7-8i), i = 0..6,
//    |a_i| <= 128. The last digit's weight is 2^-55, at most half the spacing
//    of FP64 numbers at the group's largest.
//  - B: the real embedding of the block matrix, u = sum_j b_j 2^(-7-8j),
//    j = 0..7 (operands.cu).
//  - Level s = i + j = 0..7: acc_s = sum over i + j = s and the 2^(K+1) columns
//    of a_i b_j, an integer of at most 8 * 64 * 2^14 = 2^23, so FP32 sums it
//    exactly in any order. The terms left out (i + j >= 8) are below 2^-64 each.
//  - y = sum_s acc_s 2^(-14-8s) as an integer in units of 2^-60 (|y| < 4 since
//    the block is unitary), converted to FP64 with one rounding.
// One rounding per output instead of the FP64 kernel's 64: random 4- and
// 5-target blocks on random unit states are off the product in 113-bit
// arithmetic by 5e-17 to 8e-17 (L2), the FP64 kernel by 1.8e-16 to 2.8e-16;
// with amplitudes spread over 2^60 by 1.0e-16 to 1.5e-16 against 1.8e-16 to
// 2.8e-16.
//
// The digits keep 54 bits of a group's largest amplitude, and as much less of a
// small one as it is smaller. FP64 sums lose that too where the matrix mixes
// the large amplitude into every result, but keep small amplitudes' own 53
// bits where it holds them apart (zeros of the matrix) or brings little over
// (small entries). So groups are looked at where the matrix has entries below
// 2^-20: if an amplitude lies below 2^-20 of the largest (zeros count where
// small entries are not zero), the group takes the FP64 mat-vec (exact_groups).
// The look costs 1% (24 qubits, 10 layers, median of 30 random circuits 8.41 ->
// 8.52 ms); a block whose groups all span more, as early layers with an angle
// near a multiple of pi leave them, costs an FP64 pass: of 60 such circuits
// three took 1.25 to 1.9 times as long (with 2^-16, seven).
//
// Measured at n = 25 (1 GiB read and written), FP64 kernel -> this one: 5
// targets 6930 -> 430 us, 4 targets 4080 -> 330 us (3.2 TB/s); bits 0..4:
// 499 us, bits 0..3: 403 us. What bounds it is issue and latency: about 75
// instructions per real, of which a third are the digits and a quarter the
// way back; the tensor pipe is busy 26% of the time.
//
// One CTA takes 128 groups, a thread eight amplitudes of one group (2 or 4
// threads per group). All digit planes of A times the stacked digit planes of
// B: A_i times [B_0 .. B_(7-i)] lands in the adjacent columns of levels i..7,
// so one MMA covers up to 256 columns and A is re-read from shared memory as
// rarely as possible. The columns come in two halves (the block's highest
// target 0, then 1), each with its own completion, so that the first half is
// read out and stored while the second is computed.
#include <cuda_fp16.h>

#include <cmath>

#include "tc16_common.cuh"

namespace qs {
namespace kern {

namespace {

constexpr int kDigitsA = 7;
constexpr int kLevels = 8;  // digits of B, accumulated levels

template <int K> struct Tc64 {
  static constexpr int D = 1 << K;
  static constexpr int KR = 2 * D;        // reals per group
  static constexpr int TPR = D / 8;       // threads per group
  static constexpr int NT = 128 * TPR;    // threads per CTA
  static constexpr uint32_t A_BYTES = 128u * KR * 2u;                     // one digit plane
  static constexpr uint32_t B_BYTES = (uint32_t)kLevels * KR * KR * 2u;  // all digit planes
  static constexpr uint32_t SBO = (KR / 8) * 128u;
  static constexpr uint32_t LBO = 128u;
  static constexpr uint32_t NCOLS = (uint32_t)kLevels * KR;  // TMEM columns
  static constexpr int CTAS = 512 / NCOLS;                   // per SM: 2 (K = 4), 1 (K = 5)
  static constexpr size_t SMEM = (size_t)kDigitsA * A_BYTES + B_BYTES;
};

__device__ __forceinline__ void tmem_ld4(uint32_t t, uint32_t *r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(t));
}
// x's fixed-point digits: byte 7 - i of the result is a_i + 128 (byte 0 is
// below the last digit and only rounds it). gexp is the group's exponent
// field; a shift of 64 or more gives 0. The complement stands for the
// negative: one unit of 2^-63 off, far below the last digit.
__device__ __forceinline__ uint64_t to_digits(double x, int gexp) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const uint32_t mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const uint64_t m = (((uint64_t)mh << 32) | lo) << 9;
  uint64_t f;
  asm("shr.b64 %0, %1, %2;" : "=l"(f) : "l"(m), "r"(gexp - max(e, 1)));
  const uint64_t neg = (uint64_t)((int64_t)(int32_t)hi >> 31);
  return (f ^ neg) + 0x8080808080808080ull;
}

// digit byte B of two numbers as packed FP16 integers
template <int B> __device__ __forceinline__ uint32_t digit_pair(uint64_t x, uint64_t y) {
  const uint32_t xw = (uint32_t)(B >= 4 ? x >> 32 : x), yw = (uint32_t)(B >= 4 ? y >> 32 : y);
  // the digit bytes in bytes 0 and 2, under the exponent of 1024
  constexpr uint32_t lo = B & 3, hi = (B & 3) + 4;
  const uint32_t h = (__byte_perm(xw, yw, lo | (lo << 4) | (hi << 8) | (hi << 12)) & 0x00ff00ffu) | 0x64006400u;
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6480));  // 1024 + 128
  const __half2 v = __hsub2(*reinterpret_cast<const __half2 *>(&h), off);
  return *reinterpret_cast<const uint32_t *>(&v);
}

template <int I, int K>
__device__ __forceinline__ void store_digits(const uint64_t (&f)[8], unsigned char *sA, uint32_t off) {
  if constexpr (I < kDigitsA) {
    const uint4 w = make_uint4(digit_pair<7 - I>(f[0], f[1]), digit_pair<7 - I>(f[2], f[3]),
                               digit_pair<7 - I>(f[4], f[5]), digit_pair<7 - I>(f[6], f[7]));
    *reinterpret_cast<uint4 *>(sA + I * Tc64<K>::A_BYTES + off) = w;
    store_digits<I + 1, K>(f, sA, off);
  }
}

// The eight level sums of one output as an integer in units of 2^-60. Levels
// 0..3 are at most 2^22, so adding 1.5 * 2^23 leaves the integer in the low
// bits of the sum (the constant is taken off once, at the end); levels 4 and
// 5 are converted; 6 and 7, at most 2^21 units, are rounded to whole ones.
__device__ __forceinline__ long long levels_to_fixed(const float (&a)[kLevels]) {
  constexpr float kMagic = 12582912.f;  // 1.5 * 2^23, bits 0x4B400000
  constexpr long long kBits = 0x4B400000ll;
  constexpr unsigned long long kOff = ((unsigned long long)kBits << 46) + ((unsigned long long)kBits << 38) +
                                      ((unsigned long long)kBits << 30) + ((unsigned long long)kBits << 22) + kBits;
  long long v = (long long)__float_as_int(fmaf(fmaf(a[7], 0.00390625f, a[6]), 0.25f, kMagic));
  v += (long long)__float2int_rn(a[5]) * 64;
  v += (long long)__float2int_rn(a[4]) * 16384;
  v += (long long)__float_as_int(a[3] + kMagic) * (1 << 22);
  v += (long long)__float_as_int(a[2] + kMagic) * (1 << 30);
  unsigned long long u = (unsigned long long)v - kOff;
  u += (unsigned long long)((uint32_t)__float_as_int(a[1] + kMagic) << 6) << 32;
  u += (unsigned long long)((uint32_t)__float_as_int(a[0] + kMagic) << 14) << 32;
  return (long long)u;
}

// v * 2^(gexp - 1081) where that can leave FP64's normal range (gexp the
// group's exponent field)
__device__ __noinline__ double scale_back_slow(long long v, int gexp) {
  return scalbn(__ll2double_rn(v), gexp - 1081);
}

// The tile's groups that `rows` marks, by the FP64 mat-vec, a warp a group and
// a lane a result. Their amplitudes are still the block's input.
template <int K>
__device__ __noinline__ void exact_groups(double2 *a, const double2 *mat, const TcParam &p, long long tile,
                                          const uint32_t *rows) {
  constexpr int D = 1 << K;
  const int lane = threadIdx.x & 31, r = lane & (D - 1);
  uint64_t off = 0;
#pragma unroll
  for (int j = 0; j < K; j++)
    if ((r >> j) & 1) off += 1ull << p.tq[j];
  for (int row = threadIdx.x >> 5; row < 128; row += Tc64<K>::NT / 32) {
    if (!((rows[row >> 5] >> (row & 31)) & 1)) continue;  // the same for the whole warp
    double2 *x = a + ((insert_zeros((uint64_t)(tile * 128 + row), p.fixed, p.nf) | p.cmask) + off);
    const double2 v = *x;
    double re = 0, im = 0;
    for (int c = 0; c < D; c++) {
      const double2 w = mat[r * D + c];
      const double vx = __shfl_sync(0xffffffffu, v.x, c), vy = __shfl_sync(0xffffffffu, v.y, c);
      re = fma(w.x, vx, re);
      re = fma(-w.y, vy, re);
      im = fma(w.x, vy, im);
      im = fma(w.y, vx, im);
    }
    if (lane < D) *x = make_double2(re, im);
  }
}

template <int K>
__global__ void __launch_bounds__(Tc64<K>::NT, Tc64<K>::CTAS)
    k_dense_tc64(double2 *__restrict__ a, const uint4 *__restrict__ bmat, const __grid_constant__ TcParam p, int check,
                 int *__restrict__ err) {
  using C = Tc64<K>;
  constexpr int KR = C::KR, NT = C::NT;
  constexpr int HR = KR / 2;  // reals of a half: the outputs of one value of the highest target
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char *sA = smem;
  unsigned char *sB = smem + kDigitsA * C::A_BYTES;
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ uint32_t red[NT];
  __shared__ uint32_t exact_rows[4];

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int r = tid & 127;  // row of A = TMEM lane
  const int q = tid >> 7;   // this thread's amplitudes: 4 q .. 4 q + 3 of both halves of the group

  for (int i = tid; i < (int)(C::B_BYTES / 16); i += NT) reinterpret_cast<uint4 *>(sB)[i] = bmat[i];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "r"(C::NCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar[1])));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  const uint32_t mbar_a[2] = {smem_addr(&mbar[0]), smem_addr(&mbar[1])};
  const uint32_t a_addr = smem_addr(sA), b_addr = smem_addr(sB);

  // offsets of this thread's amplitudes: slot bits 0 and 1 vary, the bits
  // between them and the highest come from q
  uint64_t q_off = 0;
#pragma unroll
  for (int j = 2; j < K - 1; j++)
    if ((q >> (j - 2)) & 1) q_off += 1ull << p.tq[j];
  const uint64_t d0 = 1ull << p.tq[0], d1 = 1ull << p.tq[1], dh = 1ull << p.tq[K - 1];
  auto offset = [&](int u) { return ((u & 1) ? d0 : 0) + ((u & 2) ? d1 : 0) + ((u & 4) ? dh : 0); };
  const uint32_t row_off = (uint32_t)(r >> 3) * C::SBO + (uint32_t)(r & 7) * 16u;

  uint32_t phase = 0;
  bool ok = true;
  long long tile = blockIdx.x;
  double2 v[8];
  double2 *base = a;
  bool valid = false;
  auto gather = [&](long long t) {
    const long long g = t * 128 + r;
    valid = t < p.n_tiles && g < p.n_groups;
    if (valid) {
      base = a + ((insert_zeros((uint64_t)g, p.fixed, p.nf) | p.cmask) + q_off);
#pragma unroll
      for (int u = 0; u < 8; u++) v[u] = base[offset(u)];
    } else {
#pragma unroll
      for (int u = 0; u < 8; u++) v[u] = make_double2(0.0, 0.0);
    }
  };
  gather(tile);

  for (; tile < p.n_tiles; tile += gridDim.x) {
    // the group's exponent: the largest high word without its sign; and that
    // of its smallest amplitude (check 1: of the nonzero ones), both in one word
    uint32_t mx = 0, mn = 0xffffffffu;
    const uint32_t skip_zero = check == 1;  // 0 - 1 is the largest
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const uint32_t m = max((uint32_t)__double2hiint(v[u].x) & 0x7fffffffu, (uint32_t)__double2hiint(v[u].y) & 0x7fffffffu);
      mx = max(mx, m);
      mn = min(mn, m - skip_zero);
    }
    uint32_t span = (mx >> 20 << 16) | (0xffffu - (mn >> 20));
    red[tid] = span;
    if (!__syncthreads_and(ok)) break;  // a wait of the last tile ran out
#pragma unroll
    for (int o = 1; o < C::TPR; o++) span = __vmaxu2(span, red[(tid + o * 128) % NT]);
    const int gexp = max((int)(span >> 16), 1);  // subnormals count from exponent 1
    const bool exact = check && gexp < 2047 && gexp - (int)(0xffffu - (span & 0xffffu)) > kDigitSpan;
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      uint64_t f[8];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        f[2 * u] = to_digits(v[4 * hh + u].x, gexp);
        f[2 * u + 1] = to_digits(v[4 * hh + u].y, gexp);
      }
      store_digits<0, K>(f, sA, row_off + (uint32_t)(hh * C::TPR + q) * C::LBO);
    }
    if (check && tid < 128) {  // warps 0..3 have every row once
      const uint32_t rows = __ballot_sync(0xffffffffu, exact);
      if ((tid & 31) == 0) exact_rows[warp] = rows;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (tid == 0) {
#pragma unroll 1
      for (int hh = 0; hh < 2; hh++) {
        // half hh: TMEM columns and B rows [8 HR hh, 8 HR (hh + 1)), level by level
        const uint32_t tm = tmem + (uint32_t)(hh * kLevels * HR);
        const uint32_t bh = b_addr + (uint32_t)hh * (C::B_BYTES / 2);
#pragma unroll 1
        for (int i = 0; i < kDigitsA; i++) {
          const uint32_t idesc = make_idesc_f16(128, (kLevels - i) * HR);
#pragma unroll
          for (int ks = 0; ks < KR / 16; ks++) {
            const uint32_t koff = (uint32_t)ks * 2u * C::LBO;
            const uint64_t da = make_desc(a_addr + i * C::A_BYTES + koff, C::LBO, C::SBO);
            const uint64_t db = make_desc(bh + koff, C::LBO, C::SBO);
            mma_f16(tm + (uint32_t)(i * HR), da, db, idesc, (i > 0 || ks > 0) ? 1u : 0u);
          }
        }
        if (!p.withhold_commit) mma_commit(mbar_a[hh]);
      }
    }
    double2 *const cur = base;
    const bool cur_valid = valid;
    gather(tile + gridDim.x);  // next tile, in flight during the MMAs
    // the results' exponents: 1023..1085 + gexp - 1081, within FP64's normal range or not
    const bool normal = gexp >= 59 && gexp <= 2041;
    const int shift = (gexp - 1081) << 20;
    const bool not_finite = gexp == 2047;  // an infinity or NaN makes the whole group NaN
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      ok = __all_sync(0xffffffffu, ok && mbar_wait(mbar_a[hh], phase));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t col = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(hh * kLevels * HR + q * 8);
#pragma unroll
      for (int c = 0; c < 2; c++) {
        uint32_t lv[kLevels][4];
#pragma unroll
        for (int s = 0; s < kLevels; s++) tmem_ld4(col + (uint32_t)(s * HR + c * 4), lv[s]);
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        double y[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
          float lvl[kLevels];
#pragma unroll
          for (int s = 0; s < kLevels; s++) lvl[s] = __uint_as_float(lv[s][i]);
          const long long fx = levels_to_fixed(lvl);
          const double t = __ll2double_rn(fx);
          const int hi = __double2hiint(t);
          y[i] = __hiloint2double(hi ? hi + shift : 0, __double2loint(t));
          if (!normal && fx != 0) y[i] = scale_back_slow(fx, gexp);
          if (not_finite) y[i] = __hiloint2double(0x7ff80000, 0);
        }
        if (cur_valid && !exact) {
          cur[offset(4 * hh + 2 * c)] = make_double2(y[0], y[1]);
          cur[offset(4 * hh + 2 * c + 1)] = make_double2(y[2], y[3]);
        }
      }
    }
    phase ^= 1;
    if (check && (exact_rows[0] | exact_rows[1] | exact_rows[2] | exact_rows[3])) {
      exact_groups<K>(a, reinterpret_cast<const double2 *>(bmat + C::B_BYTES / 16), p, tile, exact_rows);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  if (!__syncthreads_and(ok)) {
    // MMAs may still be in flight: have their completion signalled, give them
    // a bounded chance to land, then return the columns
    if (tid == 0) {
      atomicExch(err, 1);
      mma_commit(mbar_a[1]);
    }
    mbar_wait(mbar_a[1], phase ^ 1);
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::NCOLS));
}

template <int K>
cudaError_t run_tc64(double2 *a, int n, const Block &b, const void *dev_b, int *err, cudaStream_t s,
                     LaunchShape *shape) {
  TcParam p;
  p.n_groups = 1ll << (n - K - b.nctrl);
  p.n_tiles = (p.n_groups + 127) / 128;
  p.cmask = b.cmask;
  p.withhold_commit = b.withhold_commit ? 1 : 0;
  fill_fixed(b, p.fixed, p.nf);
  for (int j = 0; j < K; j++) p.tq[j] = b.q[j];
  static thread_local int configured = -1;
  static thread_local int per_sm = 1;
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured != dev) {
    cudaError_t e = cudaFuncSetAttribute(k_dense_tc64<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Tc64<K>::SMEM);
    if (e != cudaSuccess) return e;
    const int occ = resident_ctas((const void *)k_dense_tc64<K>, Tc64<K>::NT, Tc64<K>::SMEM);
    per_sm = occ < Tc64<K>::CTAS ? occ : Tc64<K>::CTAS;  // the CTAs' TMEM columns stay within 512
    configured = dev;
  }
  const int grid = tc_grid((long long)dev_info().sms * per_sm, p.n_tiles, b.tc_max_ctas);
  if (shape) {
    shape->tiles = p.n_tiles;
    shape->ctas = grid;
  }
  k_dense_tc64<K><<<grid, Tc64<K>::NT, Tc64<K>::SMEM, s>>>(a, (const uint4 *)dev_b, p, b.digit_check, err);
  return cudaGetLastError();
}

}  // namespace

size_t tc64_b_bytes(int k) { return (size_t)kLevels * (2u << k) * (2u << k) * 2u; }

cudaError_t run_dense_tc64(double2 *a, int n, const Block &b, const void *dev_b, int *err, cudaStream_t s,
                           LaunchShape *shape) {
  switch (b.k) {
    case 4: return run_tc64<4>(a, n, b, dev_b, err, s, shape);
    case 5: return run_tc64<5>(a, n, b, dev_b, err, s, shape);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace kern
}  // namespace qs
