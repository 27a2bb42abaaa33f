// Operands of single tensor-core blocks, made on the device.
//
// The upload leaves a block's matrix (FP32 for complex64, FP64 for complex128)
// at the start of the space its B operand takes, or behind it where tc64.cu
// needs the matrix too; one launch per call turns every matrix into B: FP16
// halves for tc16.cu and tc16x.cu, digit planes for tc64.cu. The host made them before, two software FP16
// conversions per entry and half: 50 us a 5-target block, 230 us one of 6,
// 105 us a complex128 one, spread over the host's threads while the GPU
// waited. One CTA per block: it reads the matrix into shared memory, then
// writes B (over it, for complex64). The complex128 digits are bound by the FP64 rate (80
// operations an entry at two per clock).
#include <cstring>

#include "tc16_common.cuh"

namespace qs {
namespace kern {

namespace {

constexpr int kLevels = 8;  // digit planes of a complex128 B (tc64.cu)
constexpr int kJobs = 1000;
constexpr int kSrcBytes = 32 * 1024;  // 64 x 64 complex64, the largest matrix

struct Job {
  uint32_t at;     // of the block's operand, in 256 bytes
  uint16_t src;    // of its matrix behind that, in 256 bytes
  uint8_t c128, k;
  uint8_t slot[6]; // slot bit -> target's position (complex64)
};

struct Jobs {
  unsigned char *base;
  Job job[kJobs];
};
static_assert(sizeof(Jobs) <= 32764, "kernel parameter space");

__global__ void __launch_bounds__(256) k_operands(const __grid_constant__ Jobs p) {
  __shared__ __align__(16) unsigned char src[kSrcBytes];
  __shared__ uint8_t pi[64];  // row or column of the matrix for one of B
  const Job j = p.job[blockIdx.x];
  unsigned char *op = p.base + ((size_t)j.at << 8);
  const unsigned char *in = op + ((size_t)j.src << 8);
  const int D = 1 << j.k, KR = 2 * D;
  const int words = (D * D * (j.c128 ? 16 : 8)) / 16;
  for (int i = threadIdx.x; i < words; i += 256)
    reinterpret_cast<uint4 *>(src)[i] = reinterpret_cast<const uint4 *>(in)[i];
  if (threadIdx.x < D) {
    int s = 0;
    for (int b = 0; b < j.k; b++)
      if ((threadIdx.x >> b) & 1) s |= 1 << j.slot[b];
    pi[threadIdx.x] = (uint8_t)s;
  }
  __syncthreads();
  if (!j.c128) {
    // the real embedding, 16 bytes (eight columns of a row) at a time, at
    // (row / 8) * KR + (column / 8) * 8 + row % 8 in 16-byte words; hi, then lo
    const float2 *m = reinterpret_cast<const float2 *>(src);
    uint4 *out = reinterpret_cast<uint4 *>(op);
    const int rows = KR * (KR / 8);
    for (int x = threadIdx.x; x < rows; x += 256) {
      const int row = x / (KR / 8), cg = x % (KR / 8);
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const float2 u = m[pi[row >> 1] * D + pi[cg * 4 + e]];
        operand_halves(row & 1, u.x, u.y, hi[e], lo[e]);
      }
      const int at = (row >> 3) * KR + cg * 8 + (row & 7);
      out[at] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      out[rows + at] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
    return;
  }
  // balanced base-256 digits u = sum_l d_l 2^(-7 - 8 l), stacked along B's rows:
  // those of the outputs with the highest target 0 first, then the others
  const double2 *m = reinterpret_cast<const double2 *>(src);
  __half2 *out = reinterpret_cast<__half2 *>(op);
  for (int i = threadIdx.x; i < D * D; i += 256) {
    const int r = i / D, c = i % D;
    double re = m[i].x * 128.0, im = m[i].y * 128.0;
    for (int l = 0; l < kLevels; l++) {
      const double dr = rint(re), di = rint(im);
      re = (re - dr) * 256.0;
      im = (im - di) * 256.0;
      const int row = r < D / 2 ? l * D + 2 * r : (kLevels + l) * D + 2 * r - D;
      // halves (row, 2 c) and (row, 2 c + 1); rows row and row + 1 share a group of eight
      __half2 *o = out + (((size_t)(row >> 3) * (KR / 8) + (c >> 2)) * 64 + (row & 7) * 8 + 2 * (c & 3)) / 2;
      o[0] = __floats2half2_rn((float)dr, (float)-di);
      o[4] = __floats2half2_rn((float)di, (float)dr);
    }
  }
}

}  // namespace

static void job_of(const Block &b, bool c128, size_t at, Job &j) {
  j.at = (uint32_t)(at >> 8);
  j.src = (uint16_t)(dev_matrix_at(b, c128) >> 8);
  j.c128 = c128;
  j.k = (uint8_t)b.k;
  for (int s = 0; s < 6; s++) j.slot[s] = (uint8_t)s;
  // lane-exchange blocks take the matrix with rows and columns in slot order:
  // entry (rho, sigma) = U(pi(rho), pi(sigma)), pi(rho) = sum over the slot
  // bits set of 1 << (their target's position). The layout depends on the
  // targets and controls only (the planner checked that n admits it), so any
  // n above the fixed bits gives the same slots.
  TcXLayout x;
  if (b.tc_xg && tc_exchange_layout(64, b, x))
    for (int s = 0; s < b.k; s++) j.slot[s] = (uint8_t)x.slot_mat[s];
}

}  // namespace kern

using namespace kern;

size_t dev_matrix_at(const Block &b, bool c128) { return c128 ? tc64_b_bytes(b.k) : 0; }

bool made_on_device(const Block &b) { return b.kind == BK_DENSE && b.tc && !b.tc_tf32; }

cudaError_t make_dev_operands(const std::vector<Block> &plan, const std::vector<size_t> &off, bool c128, void *base,
                              cudaStream_t s) {
  static thread_local Jobs p;  // large: kept off the stack; the launch copies it
  p.base = (unsigned char *)base;
  for (size_t i = 0; i < plan.size();) {
    int n = 0;
    for (; i < plan.size() && n < kJobs; i++)
      if (made_on_device(plan[i])) job_of(plan[i], c128, off[i], p.job[n++]);
    if (!n) continue;
    k_operands<<<n, 256, 0, s>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace qs
