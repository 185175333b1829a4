// zo_stream_kernels.cu -- the HBM-streaming kernels of the 1.5-SPSA step:
// fused perturb (Algorithm 1, ApplyPackedPerturbation), the out-of-place pair
// of perturbations and the debug views of a probe.
//
// All passes work on 32-byte items, one per thread (perturb_items_kernel,
// pair_items_kernel).
#include "zo_device.cuh"

namespace zo {

// ---------------------------------------------------------------------------
// Perturb: theta <- rn(fp32(theta) + scale * z_k) in place.
//
// z_k[g] is bit `bit` of byte (g mod 16) of Philox(b = g/16, ctr2) (packing 1:
// ctr2 = k/8, bit = k mod 8; packing 8: ctr2 = k, bit = 0). Byte m sits at
// bits 8(m mod 4).. of word m/4; shifting the word left by
// 31 - 8(m mod 4) - bit puts the probe bit in the sign position, which then
// flips -scale into +scale (bit 1 -> z = +1). The product scale * z is exact,
// so the element result is one fp32 add and one rounding to storage.
//
// A launch may apply two perturbations in sequence (zo_perturb2): the value
// is rounded to storage after each, exactly as two separate passes would,
// but theta crosses HBM once.
// ---------------------------------------------------------------------------
// The same with the sign moved by a multiply (PerturbOp::mul), in the vector
// loops: it moves half of the sign injection from the integer ALU, the busiest
// pipe of these loops, to the multiply-add pipe (measured: single-op pass
// -1.1 to -1.7 % time on the OPT-30B / OPT-13B-shaped sets).
__device__ __forceinline__ uint32_t sign_bit_mul(const uint4& x, int i, const PerturbOp& op) {
  return (word_of(x, i >> 2) * op.mul[i & 3]) & 0x80000000u;
}

__device__ __forceinline__ float add_signed_mul(float th, const uint4& x, int i, const PerturbOp& op) {
  return __fadd_rn(th, __uint_as_float(op.nscale_bits ^ sign_bit_mul(x, i, op)));
}

// Sixteen 16-bit weights in registers (element 2r in the low half of v[r]),
// NOPS perturbations one after the other, each rounded to storage. The adds
// are packed fp32x2 adds, the same round-to-nearest sum per element: 732
// against 756 us for the two-op pass on the OPT-1.3B-shaped bf16 set, 1156
// against 1205 us on Qwen3-8B-shaped layers when its probes fall in two groups.
template <uint8_t DT, int NOPS>
__device__ __forceinline__ void perturb_regs16(uint32_t (&v)[8], const uint4 (&x)[2], const PerturbOp (&op)[2]) {
#pragma unroll
  for (int r = 0; r < 8; ++r) {
#pragma unroll
    for (int o = 0; o < NOPS; ++o) {
      float2 f = unpack2<DT>(v[r]);
      fadd2_rn(f.x, f.y, __uint_as_float(op[o].nscale_bits ^ sign_bit_mul(x[o], 2 * r, op[o])),
               __uint_as_float(op[o].nscale_bits ^ sign_bit_mul(x[o], 2 * r + 1, op[o])));
      v[r] = pack2<DT>(f.x, f.y);
    }
  }
}

// ---------------------------------------------------------------------------
// One 32-byte item of theta per thread, every kind of tensor in one launch.
//
// Bound: HBM (2 x the list's bytes). A CTA is 256 threads of 32 registers, so
// an SM holds 2048 threads, each with one 256-bit load and store in flight,
// and the CTAs come in order, where a persistent grid of 1024 threads per SM
// had each prefetch its next block. Before -> after, OPT-1.3B-shaped set (2 d B =
// 5.26 GB in bf16; a plain copy was measured at 6794 GB/s):
//   one operation    bf16 783 -> 740 us (7110 GB/s), fp32 1650 -> 1474 us
//   two operations   bf16 807 -> 732 us (7190 GB/s), fp32 1592 -> 1472 us
//   as slices of one flat buffer, bf16: 860 -> 736 us, two operations 903 -> 809
// two operations whose probes fall in two groups of 8 (Qwen3-8B-shaped layers)
// 1192 -> 1156 us; 200 tensors of 40 M bf16 weights 33 -> 23 us, of 1 M 12.9 ->
// 7.5 us; 12 fp32 tensors of 270 k weights 8.5 -> 5.5 us.
// What an item costs besides its elements has to be small for that: its tensor
// is found from a hint (one constant load and a compare; a binary search per
// warp took 832 us), positions are 32-bit, rounds 0-1 of Philox are split
// (philox_start), the load is issued before the Philox call, and what only a
// partial item needs is computed there (1104 against 1031 us for two
// operations). Not adopted: 4, 8 or 16 items per warp with the next one
// prefetched (865, 808, 791 us).
//
// Tensors off the 32-byte grid (views at an element offset) move in their
// aligned 32-byte chunks: chunk i holds elements 16 i - a .. 16 i - a + 15 (8 of
// fp32; a = the base's distance from the boundary below it, in elements), the
// tail of one block (half block) and the head of the next, whose signs come
// from the neighbouring lane (item_signs).
//
// HIU: the launch's virtual blocks share the counter's high word (any launch
// below 2^36 weights); otherwise all ten rounds run.
// ---------------------------------------------------------------------------
// An item at p. full: its sixteen (eight) elements are in v; otherwise those of
// the tensor are loaded here, together.
template <uint8_t DT, int NOPS>
__device__ __forceinline__ void items_16(char* p, bool full, const ItemsEntry& e, int32_t i, uint32_t (&v)[8],
                                         const uint4 (&x)[2], const PerturbOp (&op)[2]) {
  uint16_t* q = reinterpret_cast<uint16_t*>(p);
  int lo = 0, hi = 0;
  if (!full) {
    item_range(e, i, &lo, &hi);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const uint32_t l = 2 * r >= lo && 2 * r < hi ? q[2 * r] : 0u;
      const uint32_t h = 2 * r + 1 >= lo && 2 * r + 1 < hi ? q[2 * r + 1] : 0u;
      v[r] = l | (h << 16);
    }
  }
  perturb_regs16<DT, NOPS>(v, x, op);
  if (full) {
    st256(p, v);
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      if (2 * r >= lo && 2 * r < hi) q[2 * r] = static_cast<uint16_t>(v[r]);
      if (2 * r + 1 >= lo && 2 * r + 1 < hi) q[2 * r + 1] = static_cast<uint16_t>(v[r] >> 16);
    }
  }
}

template <int NOPS>
__device__ __forceinline__ void items_32(char* p, bool full, const ItemsEntry& e, int32_t i, uint32_t (&v)[8],
                                         const uint4 (&x)[2], const PerturbOp (&op)[2]) {
  uint32_t* q = reinterpret_cast<uint32_t*>(p);
  int lo = 0, hi = 0;
  if (!full) {
    item_range(e, i, &lo, &hi);
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = r >= lo && r < hi ? q[r] : 0u;
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
#pragma unroll
    for (int o = 0; o < NOPS; ++o) v[r] = __float_as_uint(add_signed_mul(__uint_as_float(v[r]), x[o], r, op[o]));
  }
  if (full) {
    st256(p, v);
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r >= lo && r < hi) q[r] = v[r];
  }
}

template <int NOPS, bool CROSS, bool HIU, int N>
__global__ void __launch_bounds__(256) perturb_items_kernel(const __grid_constant__ ItemsParams<N> P) {
  if (P.status != nullptr && *P.status != 0) return;
  PerturbOp op[2] = {P.op[0], P.op[1]};
  if (P.coef != nullptr)
    op[0].nscale_bits = __float_as_uint(__double2float_rn(P.coef_mul * P.coef[P.probe])) ^ 0x80000000u;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x, wb = b - lane;  // the warp's items lie in one tensor
  if (wb >= P.total) return;
  int t = P.hint[wb >> P.hint_shift];
  while (wb >= P.e[t].end) ++t;
  const ItemsEntry e = P.e[t];
  const uint8_t dt = static_cast<uint8_t>(e.meta & kDtypeMask);
  const bool f32 = dt == kF32, shift = (e.meta & kShift) != 0;
  const uint32_t a = e.meta >> 16;
  const ItemPlace k = item_place(e, b);
  const int64_t vb = item_block(e, k.i);
  char* p = reinterpret_cast<char*>(e.base) + static_cast<int64_t>(k.i) * 32;
  uint32_t v[8];
  // (two Philox calls: the load after them keeps a resident block more)
  if (!CROSS && k.full) ld256(p, v);
  uint4 x[2];
  if constexpr (HIU) {
    const BlockRound01 r = block_round01(static_cast<uint32_t>(vb), P.keys);
    x[0] = philox_finish(philox_start(r, P.g[0]), P.keys);
    x[1] = CROSS ? philox_finish(philox_start(r, P.g[1]), P.keys) : x[0];
  } else {
    x[0] = block_bits(vb, op[0].ctr2, P.keys);
    x[1] = CROSS ? block_bits(vb, op[1].ctr2, P.keys) : x[0];
  }
  x[0] = item_signs(x[0], f32, (k.i & 1) != 0, shift, a);
  x[1] = CROSS ? item_signs(x[1], f32, (k.i & 1) != 0, shift, a) : x[0];
  if (!k.act) return;
  if (CROSS && k.full) ld256(p, v);
  if (f32)
    items_32<NOPS>(p, k.full, e, k.i, v, x, op);
  else if (dt == kBF16)
    items_16<kBF16, NOPS>(p, k.full, e, k.i, v, x, op);
  else
    items_16<kF16, NOPS>(p, k.full, e, k.i, v, x, op);
}

// ---------------------------------------------------------------------------
// Out-of-place pair: plus <- rn(fp32(theta) + v), minus <- rn(fp32(theta) - v)
// with v = scale z_k[g] (exact), theta untouched. One read of theta and two
// writes instead of the three read-modify-write passes of +eps / -2 eps /
// +eps, and both forward points are one rounding away from theta.
// ---------------------------------------------------------------------------
template <uint8_t DT>
__device__ __forceinline__ void pair_regs16(const uint32_t (&v)[8], const uint4& x, const PerturbOp& op,
                                            uint32_t (&p)[8], uint32_t (&m)[8]) {  // p may alias v
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float2 f = unpack2<DT>(v[r]);
    const float d0 = __uint_as_float(op.nscale_bits ^ sign_bit_mul(x, 2 * r, op));
    const float d1 = __uint_as_float(op.nscale_bits ^ sign_bit_mul(x, 2 * r + 1, op));
    p[r] = pack2<DT>(__fadd_rn(f.x, d0), __fadd_rn(f.y, d1));
    m[r] = pack2<DT>(__fsub_rn(f.x, d0), __fsub_rn(f.y, d1));
  }
}

// Bytes bo .. bo + 31 (bo even, 0..30) of the 64-byte string lo ++ hi.
__device__ __forceinline__ void window32(const uint32_t (&lo)[8], const uint32_t (&hi)[8], uint32_t bo,
                                         uint32_t (&out)[8]) {
  const uint32_t q = bo >> 2, sh = 8u * (bo & 3u);
  uint32_t e4[12], e2[10], e1[9];
#pragma unroll
  for (int i = 0; i < 12; ++i) {
    const uint32_t a = i < 8 ? lo[i] : hi[i - 8];
    const uint32_t b = i + 4 < 8 ? lo[i + 4] : hi[i - 4];
    e4[i] = (q & 4u) ? b : a;
  }
#pragma unroll
  for (int i = 0; i < 10; ++i) e2[i] = (q & 2u) ? e4[i + 2] : e4[i];
#pragma unroll
  for (int i = 0; i < 9; ++i) e1[i] = (q & 1u) ? e2[i + 1] : e2[i];
#pragma unroll
  for (int i = 0; i < 8; ++i) out[i] = __funnelshift_r(e1[i], e1[i + 1], sh);
}

// The 32 bytes of theta that belong to an item, at any element offset: the one
// or two aligned 32-byte segments that hold them (the shared one is also a
// neighbouring lane's, whose read hits L1).
__device__ __forceinline__ void ld_item(uint64_t src, uint32_t (&v)[8]) {
  const uint32_t mis = static_cast<uint32_t>(src & 31u);  // the same in all lanes
  if (mis == 0u) {
    ld256(reinterpret_cast<const void*>(src), v);
  } else {
    uint32_t lo[8], hi[8];
    ld256(reinterpret_cast<const void*>(src - mis), lo);
    ld256(reinterpret_cast<const void*>(src - mis + 32u), hi);
    window32(lo, hi, mis, v);
  }
}

template <uint8_t DT>
__device__ __forceinline__ void pair_item(const PairItemsEntry& e, const ItemPlace& k, const uint32_t (&v)[8],
                                          const uint4& x, const PerturbOp& op) {
  const int64_t at = static_cast<int64_t>(k.i) * 32;
  if (k.full) {
    uint32_t p[8], m[8];
    if constexpr (DT == kF32) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float d = __uint_as_float(op.nscale_bits ^ sign_bit_mul(x, r, op));
        p[r] = __float_as_uint(__fadd_rn(__uint_as_float(v[r]), d));
        m[r] = __float_as_uint(__fsub_rn(__uint_as_float(v[r]), d));
      }
    } else {
      pair_regs16<DT>(v, x, op, p, m);
    }
    st256(reinterpret_cast<void*>(e.base + at), p);
    if ((e.minus & 31u) == 0u)
      st256(reinterpret_cast<void*>(e.minus + at), m);
    else
      st16x16(reinterpret_cast<uint16_t*>(e.minus + at), m);
    return;
  }
  int lo, hi;
  item_range(e, k.i, &lo, &hi);
  const void* src = reinterpret_cast<const void*>(e.src + at);
#pragma unroll 1
  for (int h = lo & ~3; h < hi; h += 4) {  // four loads before their first store
    float th[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) th[j] = h + j >= lo && h + j < hi ? load_elem(src, DT, h + j) : 0.0f;
    const uint32_t w = word_of(x, h >> 2);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (h + j < lo || h + j >= hi) continue;
      const float d = signed_scale_word(w, j, op);
      store_elem(reinterpret_cast<void*>(e.base + at), DT, h + j, __fadd_rn(th[j], d));
      store_elem(reinterpret_cast<void*>(e.minus + at), DT, h + j, __fsub_rn(th[j], d));
    }
  }
}

// One 32-byte item of plus per thread, as perturb_items_kernel. Bound: HBM (3 x
// the list's bytes). Before (a persistent grid of three blocks per SM, and a
// kernel of its own for fp32 and for tensors off the 32-byte grid) -> after:
// an OPT-30B-shaped fp16 layer and its embedding 902 -> 839 us (7090 GB/s), as
// slices of flat buffers 953 -> 838, as fp32 1896 -> 1673 us; Qwen3-8B-shaped
// layers 1640 -> 1521 us.
template <bool HIU, int N>
__global__ void __launch_bounds__(256) pair_items_kernel(const __grid_constant__ PairItemsParams<N> P) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x, wb = b - lane;  // the warp's items lie in one tensor
  if (wb >= P.total) return;
  int t = P.hint[wb >> P.hint_shift];
  while (wb >= P.e[t].end) ++t;
  const PairItemsEntry e = P.e[t];
  const uint8_t dt = static_cast<uint8_t>(e.meta & kDtypeMask);
  const ItemPlace k = item_place(e, b);
  const int64_t vb = item_block(e, k.i);
  uint32_t v[8];
  if (k.full) ld_item(e.src + static_cast<int64_t>(k.i) * 32, v);
  uint4 x;
  if constexpr (HIU)
    x = philox_finish(philox_start(block_round01(static_cast<uint32_t>(vb), P.keys), P.g), P.keys);
  else
    x = block_bits(vb, P.op.ctr2, P.keys);
  x = item_signs(x, dt == kF32, (k.i & 1) != 0, (e.meta & kShift) != 0, e.meta >> 16);
  if (!k.act) return;
  if (dt == kF32)
    pair_item<kF32>(e, k, v, x, P.op);
  else if (dt == kBF16)
    pair_item<kBF16>(e, k, v, x, P.op);
  else
    pair_item<kF16>(e, k, v, x, P.op);
}

// ---------------------------------------------------------------------------
// Debug views: probe k packed one bit per element (Appendix F layout) and the
// unpacked int8 signs, over a range of the virtual index space.
// ---------------------------------------------------------------------------
__global__ void probe_bytes_kernel(RoundKeys keys, uint32_t q, uint32_t j, int64_t first, int64_t n, uint8_t* out) {
  const int64_t b_first = first >> 1, b_last = (first + n - 1) >> 1;  // packed bytes 2b, 2b+1 <- block b
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t b = b_first + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; b <= b_last; b += stride) {
    const uint4 x = philox10(static_cast<uint32_t>(b), static_cast<uint32_t>(static_cast<uint64_t>(b) >> 32), q, 0u,
                             keys);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int64_t jb = 2 * b + half;
      if (jb < first || jb >= first + n) continue;
      uint32_t v = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int m = 8 * half + i;
        v |= ((word_of(x, m >> 2) >> (8 * (m & 3) + j)) & 1u) << i;
      }
      out[jb - first] = static_cast<uint8_t>(v);
    }
  }
}

__global__ void probe_signs_kernel(RoundKeys keys, uint32_t q, uint32_t j, int64_t first, int64_t n, int8_t* out) {
  const int64_t b_first = first >> 4, b_last = (first + n - 1) >> 4;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t b = b_first + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; b <= b_last; b += stride) {
    const uint4 x = philox10(static_cast<uint32_t>(b), static_cast<uint32_t>(static_cast<uint64_t>(b) >> 32), q, 0u,
                             keys);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int64_t g = 16 * b + m;
      if (g < first || g >= first + n) continue;
      const uint32_t bit = (word_of(x, m >> 2) >> (8 * (m & 3) + j)) & 1u;
      out[g - first] = bit ? static_cast<int8_t>(1) : static_cast<int8_t>(-1);
    }
  }
}

}  // namespace zo

// ---------------------------------------------------------------------------
// Launch wrappers.
// ---------------------------------------------------------------------------
#include "zo_launch.h"

namespace zo {

template <bool HIU, int N>
void launch_items_cfg(const ItemsParams<N>& p, cudaStream_t stream) {
  const int grid = static_cast<int>((p.total + (kThreads - 1u)) / kThreads);
  if (p.nops == 1)
    perturb_items_kernel<1, false, HIU, N><<<grid, kThreads, 0, stream>>>(p);
  else if (p.op[0].ctr2 == p.op[1].ctr2)
    perturb_items_kernel<2, false, HIU, N><<<grid, kThreads, 0, stream>>>(p);
  else
    perturb_items_kernel<2, true, HIU, N><<<grid, kThreads, 0, stream>>>(p);
}

template <int N>
cudaError_t launch_perturb_items(const ItemsParams<N>& p, cudaStream_t stream) {
  launch_items_cfg<true>(p, stream);
  return cudaGetLastError();
}
template cudaError_t launch_perturb_items(const ItemsParams<kItemsFew>& p, cudaStream_t stream);
template cudaError_t launch_perturb_items(const ItemsParams<kItemsSome>& p, cudaStream_t stream);
template cudaError_t launch_perturb_items(const ItemsParams<kItemsMany>& p, cudaStream_t stream);

cudaError_t launch_perturb_items_any_high(const ItemsParams<kItemsMany>& p, cudaStream_t stream) {
  launch_items_cfg<false>(p, stream);
  return cudaGetLastError();
}
static_assert(sizeof(ItemsParams<kItemsMany>) <= 32764 && sizeof(PairItemsParams<kPairItemsMany>) <= 32764,
              "items table exceeds the kernel parameter space");

static_assert(sizeof(SmallUpdateParams) <= 32764,
              "tensor table exceeds the kernel parameter space");

template <int N>
cudaError_t launch_pair_items(const PairItemsParams<N>& p, bool one_high, cudaStream_t stream) {
  const int grid = static_cast<int>((p.total + (kThreads - 1u)) / kThreads);
  if (one_high)
    pair_items_kernel<true, N><<<grid, kThreads, 0, stream>>>(p);
  else
    pair_items_kernel<false, N><<<grid, kThreads, 0, stream>>>(p);
  return cudaGetLastError();
}
template cudaError_t launch_pair_items(const PairItemsParams<kItemsFew>& p, bool one_high, cudaStream_t stream);
template cudaError_t launch_pair_items(const PairItemsParams<kItemsSome>& p, bool one_high, cudaStream_t stream);
template cudaError_t launch_pair_items(const PairItemsParams<kPairItemsMany>& p, bool one_high, cudaStream_t stream);

cudaError_t launch_probe_bytes(const RoundKeys& keys, uint32_t ctr2, uint32_t bit, int64_t first, int64_t n,
                               uint8_t* out, int grid, cudaStream_t stream) {
  probe_bytes_kernel<<<grid, kThreads, 0, stream>>>(keys, ctr2, bit, first, n, out);
  return cudaGetLastError();
}

cudaError_t launch_probe_signs(const RoundKeys& keys, uint32_t ctr2, uint32_t bit, int64_t first, int64_t n,
                               int8_t* out, int grid, cudaStream_t stream) {
  probe_signs_kernel<<<grid, kThreads, 0, stream>>>(keys, ctr2, bit, first, n, out);
  return cudaGetLastError();
}

}  // namespace zo
