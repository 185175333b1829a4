// zo_blocks.cuh -- a thread's place in the fused update's kernels that work on
// blocks of sixteen weights (update_lut8_kernel, update_blocks_kernel), and the
// blocks across a tensor's end.
#pragma once

#include "zo_device.cuh"

namespace zo {

// A thread's block, or, of a tensor off the 32-byte grid
// (kShift), its 32-byte aligned chunk of sixteen elements: chunk c holds
// elements 16c - a .. 16c - a + 15 (a = the base's offset from the boundary
// below it, in elements), the tail of block c - 1 and the head of block c.
struct Lut8Block {
  int64_t b;       // virtual block whose probes the lane sums (Philox counter)
  int64_t e0;      // first element of the block or chunk inside its tensor (below 0 in a tensor's first chunk)
  int64_t numel;   // elements of the tensor
  void* base;      // tensor base pointer
  uint32_t a;      // chunks: a; blocks: 0
  uint8_t fl;      // tensor flags
  bool act;        // there are elements here for this lane
  bool vec;        // all sixteen, 32-byte aligned
};

// The update element by element, of a block or chunk across an end of its
// tensor; do_sum false: the leading perturbation alone.
__device__ __forceinline__ void lut8_apply_elements(const Lut8Block& k, const float (&acc)[16], const uint4& xp,
                                                    const UpdateParams& P, bool do_sum) {
  const uint8_t dt = k.fl & kDtypeMask;
  float v[16];  // all loads before the first store: there are registers for it here
#pragma unroll
  for (int i = 0; i < 16; ++i)
    v[i] = k.e0 + i >= 0 && k.e0 + i < k.numel ? load_elem(k.base, dt, k.e0 + i) : 0.0f;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int64_t e = k.e0 + i;
    if (e < 0 || e >= k.numel) continue;
    float th = v[i];
    if (P.has_pre) th = round_to_storage(dt, add_signed(th, xp, i, P.pre));
    if (do_sum) th = __fadd_rn(th, acc[i]);
    store_elem(k.base, dt, e, th);
  }
}

// Launch block bl, of tensor t: its place. (t of the warp's first block: every
// tensor starts on a multiple of 32 launch blocks, so the 32 blocks of a warp
// lie in one tensor or in the padding after it.) ANY: the launch may hold
// kShift tensors. Of those each warp takes 31 chunks: lane l sums block
// 31 w + l - 1 of the tensor and works on the chunk of that number, with the
// sums of the block below from lane l - 1; lane 0 only sums.
template <bool ANY>
__device__ __forceinline__ Lut8Block lut8_block_info(const TensorTable& tab, int t, uint32_t bl) {
  Lut8Block k;
  const uint32_t tb = tensor_blk_begin(tab, t);
  const uint32_t d = bl - tb;
  k.fl = tab.flags[t];
  k.numel = tab.numel[t];
  k.base = reinterpret_cast<void*>(tab.ptr[t]);
  k.a = 0u;
  if (ANY && (k.fl & kShift)) {
    const uint32_t lane = d & 31u;
    k.a = static_cast<uint32_t>(tab.ptr[t] & 31u) / ((k.fl & kDtypeMask) == kF32 ? 4u : 2u);
    const int64_t c = static_cast<int64_t>(d >> 5) * 31 + lane - 1;
    k.b = virtual_block(tab, t, tb) + c;
    k.e0 = 16 * c - k.a;
    k.act = lane > 0 && k.e0 < k.numel;
    k.vec = k.act && k.e0 >= 0 && k.e0 + 16 <= k.numel;
  } else {
    k.b = virtual_block(tab, t, bl);
    k.e0 = static_cast<int64_t>(d) * 16;
    k.act = bl < tab.blk_end[t];
    k.vec = k.act && k.e0 + 16 <= k.numel && (k.fl & kVec32);
  }
  return k;
}

}  // namespace zo
