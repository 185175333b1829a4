// zo_update_blocks.cu -- the fused update of fp32 lists that are views off the
// 32-byte grid, without a leading perturbation (packing 1).
//
// A thread takes sixteen weights: a block, or a view's two 32-byte chunks that
// hold the tail of one block and the head of the next (lut8_block_info). Each
// lane sums its own block, from the two 16-entry 4-probe tables per group that
// update_items_kernel uses, the same partials in the same order as every update,
// and a view's sums are then moved over two lanes once, where the kernels with
// a table per lane move every group's words, and for fp32 make a block's words
// twice. 64 registers, so 32 warps to an SM with nothing held but the sums:
// theta is read after them. Bound by issue (69 % of it, ALU 59 %, K = 32)
// from three groups on, by HBM below.
//
// fp32 views, us here / in the table-per-lane kernels: 221 M weights, K = 8 273 /
// 290, K = 24 364 / 387, K = 32 433 / 455, K = 40 505 / 516; 45 M, K = 8 62 / 66,
// K = 32 99 / 110, K = 40 114 / 124, K = 48 129 / 132; 11 M, K = 32 29 / 35,
// K = 40 33 / 39. K = 16 is not faster (305 / 303), nor is a list with a leading
// perturbation (221 M, K = 32 498 / 464). Not adopted: 80 registers (K = 32 502),
// theta loaded before the sums, eight waves of CTAs (45 M, K = 32 101).
#include "zo_blocks.cuh"
#include "zo_launch.h"

namespace zo {

namespace {

constexpr int kBlockThreads = 256;
constexpr int kCtasPerSm = 4;  // resident at 64 registers; four waves of them are launched
constexpr uint32_t kFrame = 256;  // bytes from one group's tables to the next's: T_lo at 0, T_hi at 64

__device__ __forceinline__ float lds_f32_hi(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1+64];" : "=f"(v) : "r"(addr));
  return v;
}

}  // namespace

__global__ void __launch_bounds__(kBlockThreads, kCtasPerSm)
    update_blocks_kernel(const __grid_constant__ UpdateParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (P.status != nullptr && *P.status != 0) return;
  const int G = P.groups;
  float* a_s = reinterpret_cast<float*>(smem);  // 8 G coefficients
  const uint32_t after = static_cast<uint32_t>(__cvta_generic_to_shared(a_s + 8 * G));
  const uint32_t frame0 = (after + kFrame - 1u) & ~(kFrame - 1u);
  float* lut = a_s + 8 * G + (frame0 - after) / 4u;
  for (int k = threadIdx.x; k < 8 * G; k += kBlockThreads)
    a_s[k] = k < P.K ? __double2float_rn(P.coef_mul * P.coef[k]) : 0.0f;
  __syncthreads();
  for (int i = threadIdx.x; i < 32 * G; i += kBlockThreads) {
    const int h = i >> 4;  // quad of probes
    lut[(h >> 1) * (kFrame / 4) + (h & 1) * 16 + (i & 15)] = quad_partial(a_s + 4 * h, static_cast<uint32_t>(i) & 15u);
  }
  __syncthreads();
  const TensorTable& tab = P.tab;
  const uint32_t lane = threadIdx.x & 31u;
  const uint4 none = make_uint4(0u, 0u, 0u, 0u);
  int t = 0;
  for (uint32_t bl = blockIdx.x * kBlockThreads + threadIdx.x; bl - lane < tab.blk_total;
       bl += gridDim.x * kBlockThreads) {
    t = advance_tensor(tab, t, bl - lane);
    const Lut8Block k = lut8_block_info<true>(tab, t, bl);
    float acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.0f;
    uint32_t frame = frame0;
#pragma unroll 1
    for (int q = 0; q < G; ++q, frame += kFrame) {
      const uint4 x = block_bits(k.b, static_cast<uint32_t>(q), P.keys);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const uint32_t w = word_of(x, m);
        const uint32_t lo4 = (w << 2) & 0x3C3C3C3Cu;  // byte j: 4 * low nibble of byte j of w
        const uint32_t hi4 = (w >> 2) & 0x3C3C3C3Cu;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t sel = 0x7650u | static_cast<uint32_t>(j);
          acc[4 * m + j] =
              __fadd_rn(acc[4 * m + j], __fadd_rn(lds_f32(__byte_perm(lo4, frame, sel)),
                                                  lds_f32_hi(__byte_perm(hi4, frame, sel))));
        }
      }
    }
    if (k.fl & kShift) window16f(acc, 16u - k.a);  // the same in all lanes
    const uint8_t dt = k.fl & kDtypeMask;
    if (k.vec) {
      char* p = static_cast<char*>(k.base) + k.e0 * (dt == kF32 ? 4 : 2);
      uint32_t v[8];
      if (dt == kF32) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          ld256(p + 32 * half, v);
#pragma unroll
          for (int r = 0; r < 8; ++r) v[r] = __float_as_uint(__fadd_rn(__uint_as_float(v[r]), acc[8 * half + r]));
          st256(p + 32 * half, v);
        }
      } else {
        ld256(p, v);
        if (dt == kBF16)
          update_regs16<kBF16>(v, acc, none, false, P.pre);
        else
          update_regs16<kF16>(v, acc, none, false, P.pre);
        st256(p, v);
      }
    } else if (k.act) {
      lut8_apply_elements(k, acc, none, P, true);
    }
  }
}

// Which updates: mostly fp32 off the 32-byte grid (`weights` of them), packing
// 1, no leading perturbation, and longer than the short lists'. One group from
// 30 M weights on (24 M: 34 / 31 us, 45 M: 62 / 66), three to five always, six and
// seven below 70 M (45 M, K = 48: 130 / 132; 118 M: 293 / 286), eight to ten below
// 6 M (5 M, K = 64 25.3 / 28.3; 8 M 36.3 / 34.9).
bool update_blocks_takes(const UpdateParams& u, int64_t weights, int sms) {
  if (u.packing != kPacking1 || u.has_pre) return false;
  const int64_t per_sm = weights / sms;
  if (u.groups <= 2) return u.groups == 1 && per_sm > 200000;
  return u.groups <= 5 || (u.groups <= 7 && per_sm < 460000) || (u.groups <= 10 && per_sm < 40000);
}

cudaError_t launch_update_blocks(const UpdateParams& p, int sms, cudaStream_t stream) {
  const int64_t want = (static_cast<int64_t>(p.tab.blk_total) + kBlockThreads - 1) / kBlockThreads;
  const int64_t cap = static_cast<int64_t>(sms) * kCtasPerSm * 4;
  const size_t smem = static_cast<size_t>(p.groups) * (32 + kFrame) + kFrame;
  update_blocks_kernel<<<static_cast<int>(want < cap ? want : cap), kBlockThreads, smem, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace zo
