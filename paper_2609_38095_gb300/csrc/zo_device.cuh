// zo_device.cuh -- launch structures and device helpers shared by the kernels
// of the 1.5-SPSA parameter-space step (sm_103a).
#pragma once

#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace zo {

// Tensors described by one launch. The whole table travels in the kernel's
// parameter space (a 32 KB limit), so the library never allocates device
// memory for it; longer lists are split over several launches.
constexpr int kMaxTensorsPerLaunch = 1024;
constexpr int kMaxProbes = 1024;      // must match ZO_MAX_PROBES
constexpr int kMaxGroups = kMaxProbes / 8;

// Storage codes (match zo_dtype) and the per-tensor "vector path" flag.
constexpr uint8_t kF32 = 0, kBF16 = 1, kF16 = 2;
constexpr uint8_t kDtypeMask = 0x3;
constexpr uint8_t kVec32 = 0x80;      // base pointer is 32-byte aligned
constexpr uint8_t kShift = 0x40;      // not 32-byte aligned: worked on in aligned chunks

// Elements are addressed by a virtual index g: tensor t starts at a multiple
// of 16, so each 16-element Philox block lies inside one tensor. Blocks are
// the unit of work: block B covers g in [16 B, 16 B + 16). Inside a launch
// blocks get 32-bit launch numbers b in which every tensor starts at a
// multiple of kLaunchAlign (the blocks in between belong to no tensor and
// are skipped), so the 32 consecutive blocks a warp takes never straddle a
// tensor's start: a warp's 256-bit accesses then cover whole 1 KB pieces of
// a tensor. (Measured on the Qwen3-8B-shaped set, whose 128-element q/k
// norm weights shift every later tensor by half a warp: the two-op pass
// 91.6 -> 95 % of the copy bandwidth.) Block b of tensor t has virtual block
// B = blk_base + b - vdelta[t]; a launch covers fewer than 2^31 launch blocks.
constexpr int64_t kMaxLaunchBlocks = INT64_C(1) << 31;
constexpr uint32_t kLaunchAlign = 32;

struct TensorTable {
  int32_t n;            // tensors in this launch
  uint32_t blk_total;   // launch blocks of this launch (padding included)
  int64_t blk_base;     // virtual index of the launch's first block
  uint32_t blk_end[kMaxTensorsPerLaunch];  // one past the last launch block of tensor t
  uint32_t vdelta[kMaxTensorsPerLaunch];   // launch block minus virtual block (relative to blk_base) in tensor t
  uint64_t ptr[kMaxTensorsPerLaunch];
  int64_t numel[kMaxTensorsPerLaunch];
  uint8_t flags[kMaxTensorsPerLaunch];    // dtype | kVec32
};

// Philox4x32 round keys, expanded on the host from the 64-bit step seed:
// key of round r = (seed_lo + r * W0, seed_hi + r * W1) mod 2^32.
struct RoundKeys {
  uint32_t k0[10];
  uint32_t k1[10];
};

// Probe packing: one generated bit per (weight, probe) -- byte g mod 16 of
// Philox(g/16, k/8) holds 8 probes, probe k in bit k mod 8 -- or one
// generated byte per (weight, probe) -- Philox(g/16, k), sign in bit 0.
constexpr int kPacking1 = 1, kPacking8 = 8;

// One in-place perturbation theta <- rn(theta + scale z_k): the third Philox
// counter word of probe k (k/8 for packing 1, k for packing 8), the bit of
// the element's byte holding its sign (k mod 8, or 0) and -scale's bits.
// mul[m] = 2^(31 - 8m - bit): a 32-bit word times mul[m] has the sign of the
// element in byte m at bit 31 (the same bit a left shift puts there, computed
// on the multiply-add pipe instead of the integer ALU).
struct PerturbOp {
  uint32_t ctr2;
  uint32_t bit;
  uint32_t nscale_bits;
  uint32_t mul[4];
};

// Tensors off the 32-byte grid are worked on in 32-byte aligned chunks, 31 per
// warp (lane 0 only generates the block below the first).
constexpr int kShiftLanes = 31;

// Table of a launch by items (perturb_items_kernel). Work is numbered in 32-byte items
// (sixteen 16-bit or eight fp32 elements), tensors starting on multiples of 32;
// a tensor off the 32-byte grid by a elements takes 32 items per 31 of its
// aligned 32-byte chunks. A tensor's fields lie together, and the tensor of an
// item is found from a hint per 2^hint_shift items, then by walking on. Three
// sizes: a launch of few tensors is bound by latency, and 25 KB of parameters
// cost it 1 us (8 KB: 0.2).
constexpr int kItemsFew = 64, kItemsSome = 256, kItemsMany = 960;
constexpr int kItemsHints = 256;
constexpr uint32_t kItemsCont = 0x20;  // the entry is a later piece of its tensor

struct ItemsEntry {
  uint64_t base;         // the tensor's address, rounded down to 32 bytes
  int64_t vb;            // virtual block of its first element
  uint32_t begin, end;   // its first and one-past-last item
  uint32_t whole;        // (elements + a) / elements per item: chunks wholly before its end
  uint32_t meta;         // dtype, kShift and kItemsCont | elements past the whole chunks << 8 | a << 16
};

// Philox rounds 0-1 as far as they depend on the probe group alone (the
// launch's virtual blocks sharing the counter's high word).
struct GroupRound01 {
  uint32_t x0;    // lo(M1 q) ^ k0[1]
  uint32_t x2;    // hi(M0 u) ^ k1[1], u = hi(M1 q) ^ bhi ^ k0[0]
  uint32_t lpa1;  // lo(M0 u)
};

// Launch item b of its entry: the 32-byte chunk i (from the entry's base) that
// it works on, and the virtual block (fp32: half block) whose signs its lane
// generates.
struct ItemPlace {
  int32_t i;      // chunk; -1: lane 0 of a tensor's first warp off the grid
  bool act;       // the lane has elements to change
  bool full;      // all of the chunk's
};

__host__ __device__ __forceinline__ ItemPlace item_place(const ItemsEntry& e, uint32_t b) {
  const bool shift = (e.meta & kShift) != 0;
  const uint32_t d = b - e.begin, lane = d & 31u;
  ItemPlace k;
  // off the grid a warp takes 31 chunks, and lane 0 only generates
  k.i = static_cast<int32_t>(shift ? (d >> 5) * static_cast<uint32_t>(kShiftLanes) + lane - 1u : d);
  const bool some = !(shift && lane == 0u);
  // the first chunk of a tensor off the grid is not full, unless this is a later piece of it
  k.full = some && k.i < static_cast<int32_t>(e.whole) && (k.i > 0 || !shift || (e.meta & kItemsCont));
  k.act = some && k.i < static_cast<int32_t>(e.whole) + ((e.meta & 0xFF00u) != 0u ? 1 : 0);
  return k;
}

__host__ __device__ __forceinline__ int64_t item_block(const ItemsEntry& e, int32_t i) {
  return e.vb + ((e.meta & kDtypeMask) == kF32 ? i >> 1 : i);
}

// An active item's elements lo .. hi - 1 of its chunk.
__host__ __device__ __forceinline__ void item_range(const ItemsEntry& e, int32_t i, int* lo, int* hi) {
  *lo = i == 0 && !(e.meta & kItemsCont) ? static_cast<int>(e.meta >> 16) : 0;
  *hi = i < static_cast<int32_t>(e.whole) ? ((e.meta & kDtypeMask) == kF32 ? 8 : 16)
                                          : static_cast<int>((e.meta >> 8) & 255u);
}

template <int N>
struct ItemsParams {
  static constexpr int kEntries = N;
  ItemsEntry e[N];       // non-empty tensors
  uint16_t hint[kItemsHints];
  int32_t n;
  int32_t hint_shift;
  uint32_t total;
  RoundKeys keys;
  PerturbOp op[2];         // applied in order, each rounded to storage; op[1] only when nops == 2
  GroupRound01 g[2];       // their groups' Philox parts
  int32_t nops;            // 1 or 2
  uint32_t probe;          // probe index k of op[0] (for coef)
  const double* coef;      // optional: op[0]'s scale = fp32(coef_mul * coef[probe])
  double coef_mul;
  const int32_t* status;   // optional: skip everything unless *status == 0
};

// Out-of-place pair of perturbations (zo_perturb_pair): theta is read once and
// theta + scale z_k, theta - scale z_k are written to two other lists of the
// same shapes. Items are plus's; src and minus are where the same elements of
// the item at `base` lie in theta and in minus.
constexpr int kPairItemsMany = 640;

struct PairItemsEntry : ItemsEntry {
  uint64_t src;
  uint64_t minus;
};

template <int N>
struct PairItemsParams {
  static constexpr int kEntries = N;
  PairItemsEntry e[N];
  uint16_t hint[kItemsHints];
  int32_t n;
  int32_t hint_shift;
  uint32_t total;
  RoundKeys keys;
  PerturbOp op;
  GroupRound01 g;
};

struct UpdateParams {
  TensorTable tab;
  RoundKeys keys;
  const double* coef;      // K coefficients c_k (device)
  double coef_mul;         // -(lr / K)
  int32_t K;
  int32_t groups;          // ceil(K / 8): 8 probes per shared-memory frame
  int32_t packing;         // kPacking1 or kPacking8
  int32_t has_pre;         // apply `pre` (and round to storage) before adding the probe sum
  PerturbOp pre;
  const int32_t* status;   // optional: when *status != 0 only `pre` is applied
};

// The update at one to kSmallGroups probe groups: the groups' and the leading
// perturbation's Philox parts beside it. In its table launch blocks are
// 32-byte items: half blocks of fp32 tensors, and 32 per 31 aligned chunks of
// tensors off the 32-byte grid (kShift).
constexpr int kSmallGroups = 4;
struct SmallUpdateParams {
  UpdateParams u;
  GroupRound01 g[kSmallGroups];
  GroupRound01 gp;
  int32_t f32_blocks;  // mostly fp32 on the 32-byte grid
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 products;
// the high halves are xored with the other two counter words and the round
// key, the low halves pass through. Round keys come from parameter space so
// they feed the xors without extra instructions.
// ---------------------------------------------------------------------------
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

__device__ __forceinline__ void philox_round(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3, uint32_t k0,
                                             uint32_t k1) {
  const uint64_t pa = static_cast<uint64_t>(kPhiloxM0) * c0;
  const uint64_t pb = static_cast<uint64_t>(kPhiloxM1) * c2;
  const uint32_t n0 = static_cast<uint32_t>(pb >> 32) ^ c1 ^ k0;
  const uint32_t n2 = static_cast<uint32_t>(pa >> 32) ^ c3 ^ k1;
  c1 = static_cast<uint32_t>(pb);
  c3 = static_cast<uint32_t>(pa);
  c0 = n0;
  c2 = n2;
}

__device__ __forceinline__ uint4 philox10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                          const RoundKeys& rk) {
#pragma unroll
  for (int r = 0; r < 10; ++r) philox_round(c0, c1, c2, c3, rk.k0[r], rk.k1[r]);
  return make_uint4(c0, c1, c2, c3);
}

// Philox4x32-10 with rounds 0 and 1 split by what they depend on, for a
// launch whose virtual blocks share the counter's high word bhi (every launch
// below 2^36 weights). The counter is (b_lo, bhi, q, 0). Round 0 multiplies
// b_lo (per block) and q (per group); round 1 multiplies the word that came
// from q and bhi (per group) and the one that came from b_lo (per block), so
// both rounds' products are computed once per group (GroupRound01, shared by
// every block) and once per block (BlockRound01, shared by the pair's two
// groups); only their xors and rounds 2-9 are per (block, group). The output
// equals philox10(b_lo, bhi, q, 0) bit for bit.
struct BlockRound01 {
  uint32_t lpa0;  // lo(M0 b_lo)
  uint32_t hpb1;  // hi(M1 v), v = hi(M0 b_lo) ^ k1[0]
  uint32_t lpb1;  // lo(M1 v)
};
__host__ __device__ __forceinline__ GroupRound01 group_round01(uint32_t q, uint32_t bhi, const RoundKeys& rk) {
  const uint64_t pb0 = static_cast<uint64_t>(kPhiloxM1) * q;
  const uint32_t u = static_cast<uint32_t>(pb0 >> 32) ^ bhi ^ rk.k0[0];
  const uint64_t pa1 = static_cast<uint64_t>(kPhiloxM0) * u;
  GroupRound01 g;
  g.x0 = static_cast<uint32_t>(pb0) ^ rk.k0[1];
  g.x2 = static_cast<uint32_t>(pa1 >> 32) ^ rk.k1[1];
  g.lpa1 = static_cast<uint32_t>(pa1);
  return g;
}
__device__ __forceinline__ BlockRound01 block_round01(uint32_t blo, const RoundKeys& rk) {
  const uint64_t pa0 = static_cast<uint64_t>(kPhiloxM0) * blo;
  const uint32_t v = static_cast<uint32_t>(pa0 >> 32) ^ rk.k1[0];
  const uint64_t pb1 = static_cast<uint64_t>(kPhiloxM1) * v;
  BlockRound01 k;
  k.lpa0 = static_cast<uint32_t>(pa0);
  k.hpb1 = static_cast<uint32_t>(pb1 >> 32);
  k.lpb1 = static_cast<uint32_t>(pb1);
  return k;
}

// A Philox call after its first two rounds.
struct PhiloxState {
  uint32_t c0, c1, c2, c3;
};

__device__ __forceinline__ uint4 philox_finish(PhiloxState s, const RoundKeys& rk) {
#pragma unroll
  for (int r = 2; r < 10; ++r) philox_round(s.c0, s.c1, s.c2, s.c3, rk.k0[r], rk.k1[r]);
  return make_uint4(s.c0, s.c1, s.c2, s.c3);
}

__device__ __forceinline__ PhiloxState philox_start(const BlockRound01& k, const GroupRound01& g) {
  return {k.hpb1 ^ g.x0, k.lpb1, g.x2 ^ k.lpa0, g.lpa1};
}

__device__ __forceinline__ uint32_t word_of(const uint4& x, int m) {
  return m == 0 ? x.x : (m == 1 ? x.y : (m == 2 ? x.z : x.w));
}

// 256-bit global accesses (sm_100+): one per 16-element block of a 16-bit
// tensor, two for fp32. The caller guarantees 32-byte alignment.
__device__ __forceinline__ void ld256(const void* p, uint32_t (&r)[8]) {
  asm volatile("ld.global.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(p));
}

__device__ __forceinline__ void st256(void* p, const uint32_t (&r)[8]) {
  asm volatile("st.global.v8.u32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// Thirty-two bytes to an address that is only 2-byte aligned (a view at an odd
// offset): the widest accesses it allows.
__device__ __forceinline__ void st16x16(uint16_t* p, const uint32_t (&v)[8]) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  if ((a & 15u) == 0) {
    uint4* q = reinterpret_cast<uint4*>(p);
    q[0] = make_uint4(v[0], v[1], v[2], v[3]);
    q[1] = make_uint4(v[4], v[5], v[6], v[7]);
  } else if ((a & 3u) == 0) {
    uint32_t* w = reinterpret_cast<uint32_t*>(p);
#pragma unroll
    for (int r = 0; r < 8; ++r) w[r] = v[r];
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      p[2 * r] = static_cast<uint16_t>(v[r]);
      p[2 * r + 1] = static_cast<uint16_t>(v[r] >> 16);
    }
  }
}

// a0, a1 <- rn(a0 + b0), rn(a1 + b1): one packed fp32x2 add (sm_100 and
// later), the same IEEE round-to-nearest sum per element as two scalar adds.
// Used on probe sums, and on 16-bit weights whose result is then rounded to
// storage (the special-value tests run every bf16 and fp16 pattern, NaNs
// included, through those paths); fp32 weights keep scalar adds.
__device__ __forceinline__ void fadd2_rn(float& a0, float& a1, float b0, float b1) {
  asm("{\n .reg .b64 pa, pb;\n mov.b64 pa, {%0, %1};\n mov.b64 pb, {%2, %3};\n add.rn.f32x2 pa, pa, pb;\n"
      " mov.b64 {%0, %1}, pa;\n}"
      : "+f"(a0), "+f"(a1)
      : "f"(b0), "f"(b1));
}

// Widen / round 16-bit storage. A 32-bit register holds elements 2r (low
// half) and 2r + 1 (high half).
template <uint8_t DT>
__device__ __forceinline__ float2 unpack2(uint32_t u) {
  if constexpr (DT == kBF16) {
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
  } else {
    __half2 h = *reinterpret_cast<__half2*>(&u);
    return __half22float2(h);
  }
}

template <uint8_t DT>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  if constexpr (DT == kBF16) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
  } else {
    __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
  }
}

// Value of v after rounding to the storage format and widening back.
__device__ __forceinline__ float round_to_storage(uint8_t dt, float v) {
  if (dt == kBF16) return __bfloat162float(__float2bfloat16_rn(v));
  if (dt == kF16) return __half2float(__float2half_rn(v));
  return v;
}

// Scalar element access for the element-wise path.
__device__ __forceinline__ float load_elem(const void* base, uint8_t dt, int64_t i) {
  if (dt == kF32) return static_cast<const float*>(base)[i];
  const uint16_t h = static_cast<const uint16_t*>(base)[i];
  if (dt == kBF16) return __uint_as_float(static_cast<uint32_t>(h) << 16);
  return __half2float(__ushort_as_half(h));
}

__device__ __forceinline__ void store_elem(void* base, uint8_t dt, int64_t i, float v) {
  if (dt == kF32) {
    static_cast<float*>(base)[i] = v;
  } else if (dt == kBF16) {
    static_cast<__nv_bfloat16*>(base)[i] = __float2bfloat16_rn(v);
  } else {
    static_cast<__half*>(base)[i] = __float2half_rn(v);
  }
}

// Elements e0 + i of a tensor, lo <= i < hi <= 16, through f(m, j, value), i =
// 4 m + j: a block or chunk across an end of its tensor, in place. AHEAD (1, 2
// or 4) loads are issued before their first store: one by one, each load
// misses the line that the store before it changed, and up to fifteen round
// trips to L2 were a fifth of a small list's pass. What AHEAD costs in
// registers its caller's loop pays, so it is as large as leaves that loop as
// it was.
template <int AHEAD, class F>
__device__ __forceinline__ void map_elements(void* base, uint8_t dt, int64_t e0, int lo, int hi, const F& f) {
#pragma unroll 1
  for (int h = lo & ~(AHEAD - 1); h < hi; h += AHEAD) {
    float v[AHEAD];
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) v[j] = h + j >= lo && h + j < hi ? load_elem(base, dt, e0 + h + j) : 0.0f;
#pragma unroll
    for (int j = 0; j < AHEAD; ++j)
      if (h + j >= lo && h + j < hi)
        store_elem(base, dt, e0 + h + j, f(h >> 2, AHEAD == 4 ? j : (h + j) & 3, v[j]));
  }
}

// Probe bit of element i (0..15) of a block, moved to bit 31.
__device__ __forceinline__ uint32_t sign_bit(const uint4& x, int i, uint32_t j) {
  return (word_of(x, i >> 2) << (31u - 8u * static_cast<uint32_t>(i & 3) - j)) & 0x80000000u;
}

// scale z of the element in byte j of a Philox word: -scale's sign flipped by
// the probe bit.
__device__ __forceinline__ float signed_scale_word(uint32_t w, int j, const PerturbOp& op) {
  return __uint_as_float(op.nscale_bits ^ ((w << (31u - 8u * static_cast<uint32_t>(j) - op.bit)) & 0x80000000u));
}

__device__ __forceinline__ float add_signed_word(float th, uint32_t w, int j, const PerturbOp& op) {
  return __fadd_rn(th, signed_scale_word(w, j, op));
}

// theta + scale z for element i of a block: -scale's sign flipped by the probe bit.
__device__ __forceinline__ float add_signed(float th, const uint4& x, int i, const PerturbOp& op) {
  return __fadd_rn(th, __uint_as_float(op.nscale_bits ^ sign_bit(x, i, op.bit)));
}

// Philox output of virtual block b for counter word ctr2.
__device__ __forceinline__ uint4 block_bits(int64_t b, uint32_t ctr2, const RoundKeys& keys) {
  return philox10(static_cast<uint32_t>(b), static_cast<uint32_t>(static_cast<uint64_t>(b) >> 32), ctr2, 0u, keys);
}

// Leading perturbation of zo_update_ex, rounded to storage (16-bit pairs).
template <uint8_t DT>
__device__ __forceinline__ uint32_t pre_regs16(uint32_t v, const uint4& xp, int r, const PerturbOp& op) {
  const float2 f = unpack2<DT>(v);
  return pack2<DT>(add_signed(f.x, xp, 2 * r, op), add_signed(f.y, xp, 2 * r + 1, op));
}

// Tensor containing launch block b, searched forward from `t` (blocks of a
// thread only increase). Zero-length tensors own no block and are skipped.
__device__ __forceinline__ int advance_tensor(const TensorTable& tab, int t, uint32_t b) {
  while (b >= tab.blk_end[t]) ++t;
  return t;
}

// First launch block of tensor t (launch blocks below it and at or above the
// previous tensor's end are padding).
__device__ __forceinline__ uint32_t tensor_blk_begin(const TensorTable& tab, int t) {
  return t == 0 ? 0u : (tab.blk_end[t - 1] + kLaunchAlign - 1u) & ~(kLaunchAlign - 1u);
}

// Virtual block (the Philox counter) of launch block b of tensor t.
__device__ __forceinline__ int64_t virtual_block(const TensorTable& tab, int t, uint32_t b) {
  return tab.blk_base + static_cast<int64_t>(b) - static_cast<int64_t>(tab.vdelta[t]);
}

// Helpers of the kernels that work on tensors off the 32-byte grid in aligned
// chunks straddling two Philox blocks.
// The windows below are of the lane below's values followed by the lane's own.
// Where the window starts is the same in all lanes of a warp, so a branch on
// its coarse part leaves only the values that are needed to be shuffled (2.5 of
// 4 words, 10 of 16 sums on average) and no selects among whole words:
// shuffles take four issue cycles each. Slices of flat buffers, shuffling and
// selecting everything -> so: update of 400 M bf16 weights, K = 32, 773 -> 745
// us, two operations on the OPT-1.3B-shaped set 809 -> 788, on Qwen3-8B-shaped
// layers in two probe groups 1390 -> 1325.
template <int Q>
__device__ __forceinline__ uint4 window16_from(const uint4& x, uint32_t sh) {
  const uint32_t own[4] = {x.x, x.y, x.z, x.w};
  uint32_t w[5];  // words Q .. Q + 4 of below ++ own
#pragma unroll
  for (int i = 0; i < 5; ++i) w[i] = Q + i < 4 ? __shfl_up_sync(0xFFFFFFFFu, own[(Q + i) & 3], 1) : own[(Q + i) & 3];
  return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh),
                    __funnelshift_r(w[2], w[3], sh), __funnelshift_r(w[3], w[4], sh));
}

// Bytes b .. b + 15 (b = 0..15) of below ++ own.
__device__ __forceinline__ uint4 window16(const uint4& x, uint32_t b) {
  const uint32_t sh = 8u * (b & 3u);
  switch (b >> 2) {
    case 0: return window16_from<0>(x, sh);
    case 1: return window16_from<1>(x, sh);
    case 2: return window16_from<2>(x, sh);
    default: return window16_from<3>(x, sh);
  }
}

template <int Q>
__device__ __forceinline__ void window16f_from(float (&v)[16], uint32_t s) {
  float t[19], u[17];  // values 4 Q .. 4 Q + 18 of below ++ own
#pragma unroll
  for (int i = 0; i < 19; ++i)
    t[i] = 4 * Q + i < 16 ? __shfl_up_sync(0xFFFFFFFFu, v[(4 * Q + i) & 15], 1) : v[(4 * Q + i) & 15];
#pragma unroll
  for (int i = 0; i < 17; ++i) u[i] = (s & 2u) ? t[i + 2] : t[i];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = (s & 1u) ? u[i + 1] : u[i];
}

// v <- values s .. s + 15 (s = 0..15) of below ++ own.
__device__ __forceinline__ void window16f(float (&v)[16], uint32_t s) {
  switch (s >> 2) {
    case 0: window16f_from<0>(v, s); break;
    case 1: window16f_from<1>(v, s); break;
    case 2: window16f_from<2>(v, s); break;
    default: window16f_from<3>(v, s); break;
  }
}

// The sign words of a 32-byte item's elements from its Philox block's words
// (all lanes of a warp, f32 / shift / a the same in all). f32: the item is the
// block's lower or upper half, its eight bytes come first. shift: a tensor off
// the 32-byte grid by a elements, whose item holds the tail of the block (f32:
// half block) below, generated by lane l - 1, and the head of its own.
__device__ __forceinline__ uint4 item_signs(const uint4& x, bool f32, bool upper, bool shift, uint32_t a) {
  if (f32) {
    uint2 y = upper ? make_uint2(x.z, x.w) : make_uint2(x.x, x.y);
    if (shift) {  // bytes 8 - a .. 15 - a of (the half below) ++ (this half), a = 1..7
      const uint32_t b0 = __shfl_up_sync(0xFFFFFFFFu, y.x, 1), b1 = __shfl_up_sync(0xFFFFFFFFu, y.y, 1);
      const uint32_t s = 8u - a, sh = 8u * (s & 3u);
      const uint32_t w0 = s >= 4u ? b1 : b0, w1 = s >= 4u ? y.x : b1, w2 = s >= 4u ? y.y : y.x;
      y = make_uint2(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh));
    }
    return make_uint4(y.x, y.y, 0u, 0u);
  }
  return shift ? window16(x, 16u - a) : x;
}

// Helpers of the fused update's kernels.
__device__ __forceinline__ float lds_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}

// One 4-probe partial ((s0 a0 + s1 a1) + s2 a2) + s3 a3 for sign nibble i.
__device__ __forceinline__ float quad_partial(const float* a, uint32_t i) {
  float s = (i & 1u) ? a[0] : -a[0];
  s = __fadd_rn(s, (i & 2u) ? a[1] : -a[1]);
  s = __fadd_rn(s, (i & 4u) ? a[2] : -a[2]);
  s = __fadd_rn(s, (i & 8u) ? a[3] : -a[3]);
  return s;
}

// theta pair + the leading perturbation's signed scales, one packed add.
__device__ __forceinline__ void add_signed2(float2& f, const uint4& x, int i, const PerturbOp& op) {
  // the probe bit moved to bit 31 by a multiply (PerturbOp::mul): the
  // multiply-add pipe instead of the integer ALU, the busier one here
  fadd2_rn(f.x, f.y, __uint_as_float(op.nscale_bits ^ ((word_of(x, i >> 2) * op.mul[i & 3]) & 0x80000000u)),
           __uint_as_float(op.nscale_bits ^ ((word_of(x, (i + 1) >> 2) * op.mul[(i + 1) & 3]) & 0x80000000u)));
}

// Sixteen 16-bit weights: the leading perturbation, rounded to storage, then
// the probe sums.
template <uint8_t DT>
__device__ __forceinline__ void update_regs16(uint32_t (&v)[8], const float (&acc)[16], const uint4& xp,
                                              bool has_pre, const PerturbOp& pre) {
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    float2 f = unpack2<DT>(v[r]);
    if (has_pre) {
      add_signed2(f, xp, 2 * r, pre);
      f = unpack2<DT>(pack2<DT>(f.x, f.y));  // the perturbed value is rounded to storage first
    }
    fadd2_rn(f.x, f.y, acc[2 * r], acc[2 * r + 1]);
    v[r] = pack2<DT>(f.x, f.y);
  }
}

// Packing 8: bit 0 of every byte of x to bit i of y's.
__device__ __forceinline__ void fold_bits(uint4& y, const uint4& x, uint32_t i) {
  const uint32_t m = 0x01010101u << i;
  y.x |= (x.x << i) & m;
  y.y |= (x.y << i) & m;
  y.z |= (x.z << i) & m;
  y.w |= (x.w << i) & m;
}

// The fused update by items (update_items_kernel): ItemsParams'
// table, and the update's own arguments as in UpdateParams.
template <int N>
struct UpdateItemsParams {
  static constexpr int kEntries = N;
  ItemsEntry e[N];
  uint16_t hint[kItemsHints];
  int32_t n;
  int32_t hint_shift;
  uint32_t total;
  uint32_t rounds;         // packing 8: items a thread takes
  int32_t f32_blocks;      // packing 8: mostly fp32 on the 32-byte grid
  uint32_t bhi;            // the virtual blocks' counter high word
  RoundKeys keys;
  const double* coef;
  double coef_mul;
  int32_t K;
  int32_t groups;
  int32_t packing;
  int32_t has_pre;
  int32_t pre_last;        // packing 8: pre's probe is one of the last group's, pre.bit its place in it
  PerturbOp pre;
  const int32_t* status;
};

}  // namespace zo
