// zo_update_lut8.cu -- the fused K-probe update (Sec. 4.2, Eqs. 5-6) with one
// table lookup per eight probes.
//
// theta <- rn(fp32(theta) + sum_k a_k z_k[g]), a_k = fp32(coef_mul * c_k).
//
// Byte m of Philox(b, q) carries the signs of probes 8q..8q+7 of element
// 16b + m (packing 1). For each probe group q the 256-entry table
//   T8_q[n] = T_lo[n & 15] + T_hi[n >> 4],
//   T_lo[i] = ((s0 a_{8q} + s1 a_{8q+1}) + s2 a_{8q+2}) + s3 a_{8q+3}  (s_j = +1 iff bit j of i)
// and T_hi likewise for probes 8q+4..8q+7, holds the group's fp32 partial sum
// for every sign byte n. An element adds one looked-up value per group, groups
// in increasing order: one byte-permute (the address), one shared load and
// half a packed fp32x2 add per eight probes. Both kernels of this file add these
// partials in this order, so they give the same bits.
//
// Bank conflicts. 32 lanes looking up random bytes of one 256-entry table
// would collide on the 32 shared-memory banks, so every lane reads its own
// copy: row n of the replicated region (256 bytes) holds T8[n] once per lane,
// lane l in word l of one half of the row (bank l), and another group's table
// in the other half. The lookup address is then
//   region + 256 n + 128 h + 4 l,
// with the region on a 64 KB boundary of the shared window: one byte-permute
// puts the sign byte n under the region's upper half-word and next to the
// lane's offset 128 h + 4 l.
//
// Loop order. The replicated tables of all groups do not fit in shared memory
// (32 KB per group), so probe groups are the outer loop: a CTA owns a chunk of
// 512 * BPT consecutive blocks (BPT = 8 but in a launch's last round), accumulates every
// block's sums over all groups and then applies them to theta (read once,
// written once). Two regions of 64 KB each hold a pair of groups (one per
// half): while the lanes look up groups 2p and 2p+1 in one region, they copy
// the next pair's tables into the other; one barrier per pair separates the
// two. The sums live in tensor memory (TMEM) between pairs, so the chunk is
// not limited by registers: per pair, each 64 KB table copy and its barrier
// serve 4096 blocks. Up to four groups' tables fit shared memory for the whole
// launch (update_lut8_small_kernel): no chunks, and the sums stay in registers.
#include <type_traits>

#include "zo_blocks.cuh"
#include "zo_device.cuh"
#include "zo_launch.h"

namespace zo {

constexpr uint32_t kLut8Region = 65536;   // 256 rows x 256 bytes: the tables of two groups
__device__ __forceinline__ void sts_f32x4(uint32_t addr, float v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "f"(v) : "memory");
}

// Add group q's partial of the 16 elements of a block (Philox output x) to acc,
// two elements per packed add. frame: the region's upper half-word, 128 h + 4 l
// in the low byte.
__device__ __forceinline__ void lut8_lookup(float (&acc)[16], const uint4& x, uint32_t frame) {
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const uint32_t w = word_of(x, m);
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
      // bytes: frame.b0 (lane offset), w.b_j (sign byte -> row), frame.b2, frame.b3 (region)
      const uint32_t a0 = __byte_perm(w, frame, 0x7604u | (static_cast<uint32_t>(j) << 4));
      const uint32_t a1 = __byte_perm(w, frame, 0x7604u | (static_cast<uint32_t>(j + 1) << 4));
      fadd2_rn(acc[4 * m + j], acc[4 * m + j + 1], lds_f32(a0), lds_f32(a1));
    }
  }
}

// Sixteen fp32 weights: the leading perturbation, then the probe sums (scalar adds, as in every fp32 path).
__device__ __forceinline__ void lut8_apply32(uint32_t (&v)[16], const float (&acc)[16], const uint4& xp,
                                             const UpdateParams& P) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float th = __uint_as_float(v[i]);
    if (P.has_pre) th = add_signed(th, xp, i, P.pre);
    v[i] = __float_as_uint(__fadd_rn(th, acc[i]));
  }
}

// Tensor-memory accumulators. A thread's sums for the blocks of its chunk live
// in TMEM between probe-group pairs: 512 threads (16 warps), warp w reaching
// TMEM lanes 32 (w mod 4) .. +31 and, of their 512 columns, the 128 from
// 128 (w / 4); a thread's block j takes 16 columns (one per element). So a CTA
// owns BPT = 8 blocks per thread (4096 blocks, 64 K elements) while its
// registers hold one block's sums at a time, and each table copy and barrier
// serves four times the elements of a register-only chunk of two blocks per
// thread. The copies are what the chunk size is for: a pair's replicated
// tables are 64 KB of shared-memory stores, against 128 KB of lookups per
// 1024 blocks.
constexpr int kLut8Threads = 512;
constexpr int kLut8Bpt = 8;  // most blocks per thread of a chunk
constexpr uint32_t kTmemCols = 512;

__device__ __forceinline__ void tm_ld16(float (&r)[16], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
        "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
      : "r"(taddr));
}

// Wait for this thread's TMEM loads; the loaded registers pass through the
// wait so that no use of them can be scheduled before it.
__device__ __forceinline__ void tm_wait_ld(float (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]), "+f"(r[7]),
                 "+f"(r[8]), "+f"(r[9]), "+f"(r[10]), "+f"(r[11]), "+f"(r[12]), "+f"(r[13]), "+f"(r[14]), "+f"(r[15])
               :
               : "memory");
}

__device__ __forceinline__ void tm_st16(uint32_t taddr, const float (&a)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16};" ::"r"(taddr),
      "f"(a[0]), "f"(a[1]), "f"(a[2]), "f"(a[3]), "f"(a[4]), "f"(a[5]), "f"(a[6]), "f"(a[7]), "f"(a[8]), "f"(a[9]),
      "f"(a[10]), "f"(a[11]), "f"(a[12]), "f"(a[13]), "f"(a[14]), "f"(a[15])
      : "memory");
}

__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tm_get16(float (&a)[16], uint32_t taddr) {
  tm_ld16(a, taddr);
  tm_wait_ld(a);
}

__device__ __forceinline__ void zero16(float (&a)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = 0.0f;
}

// Copy the tables of groups q (and q + 1 when `two`) into the two halves of a
// region, forming each entry T8[n] = T_lo[n & 15] + T_hi[n >> 4] from the
// group's 16-entry 4-probe tables (t4: T_lo then T_hi, 32 floats per group).
// Each thread owns the same 16-byte pieces (four lane copies) of 2048 / THREADS
// rows in every table: row n = p * THREADS / 8 + tid / 8, piece tid mod 8, so
// eight consecutive threads fill one half row (each quarter-warp store covers
// 128 contiguous bytes) and every address is a per-thread base plus a constant;
// a thread's rows are 64 apart, so n & 15 is the same in all of them. All loads
// are issued before the first store.
//   dst_t  region + 256 * (tid / 8) + 16 * (tid mod 8)
template <int THREADS>
__device__ __forceinline__ void lut8_replicate4(uint32_t t4, uint32_t dst_t, int q, bool two) {
  constexpr int S = 2048 / THREADS;
  constexpr uint32_t kRowStep = THREADS / 8;
  static_assert(kRowStep % 16 == 0, "rows of a thread must share n mod 16");
  const uint32_t r0 = threadIdx.x >> 3;
  float v0[S], v1[S];
  const uint32_t g0 = t4 + 128u * static_cast<uint32_t>(q);
  {
    const float lo = lds_f32(g0 + 4u * (r0 & 15u));
#pragma unroll
    for (int p = 0; p < S; ++p) v0[p] = __fadd_rn(lo, lds_f32(g0 + 64u + 4u * ((p * kRowStep + r0) >> 4)));
  }
  if (two) {
    const float lo = lds_f32(g0 + 128u + 4u * (r0 & 15u));
#pragma unroll
    for (int p = 0; p < S; ++p) v1[p] = __fadd_rn(lo, lds_f32(g0 + 192u + 4u * ((p * kRowStep + r0) >> 4)));
  }
#pragma unroll
  for (int p = 0; p < S; ++p) sts_f32x4(dst_t + p * kRowStep * 256u, v0[p]);
  if (two) {
#pragma unroll
    for (int p = 0; p < S; ++p) sts_f32x4(dst_t + 128u + p * kRowStep * 256u, v1[p]);
  }
}

// A block's part of the counter: HIU, its round-0/1 products; otherwise the
// counter itself.
template <bool HIU>
struct BlockCounter;
template <>
struct BlockCounter<true> {
  BlockRound01 k;
  // vr: the block's low word
  __device__ __forceinline__ BlockCounter(uint32_t vr, int64_t, const RoundKeys& rk) : k(block_round01(vr, rk)) {}
  __device__ __forceinline__ PhiloxState start(const GroupRound01& g, uint32_t, const RoundKeys&) const {
    return philox_start(k, g);
  }
};
template <>
struct BlockCounter<false> {
  uint32_t lo, hi;
  // vr: the block's offset from `base`
  __device__ __forceinline__ BlockCounter(uint32_t vr, int64_t base, const RoundKeys&) {
    const uint64_t b = static_cast<uint64_t>(base + vr);
    lo = static_cast<uint32_t>(b);
    hi = static_cast<uint32_t>(b >> 32);
  }
  __device__ __forceinline__ PhiloxState start(const GroupRound01&, uint32_t q, const RoundKeys& rk) const {
    PhiloxState s = {lo, hi, q, 0u};
    philox_round(s.c0, s.c1, s.c2, s.c3, rk.k0[0], rk.k1[0]);
    philox_round(s.c0, s.c1, s.c2, s.c3, rk.k0[1], rk.k1[1]);
    return s;
  }
};

// The words whose byte m holds the signs of probes 8q .. 8q + 7 of element m
// under packing 8: bit 0 of every byte of eight Philox calls, call i moved to
// bit i; r01 holds the calls' group parts (HIU). Calls past probe K - 1 are
// left out: their coefficients are 0 in the tables. A full group's calls run
// in pairs, two independent chains of multiplies per thread: with the four
// warps a scheduler has here, one chain leaves the multiply-add pipe waiting.
template <bool HIU>
__device__ __forceinline__ uint4 group_words8(const BlockCounter<HIU>& kb, uint32_t q, uint32_t K, const uint4* r01,
                                              const RoundKeys& keys) {
  const auto start = [&](uint32_t k) {
    GroupRound01 g = {0u, 0u, 0u};
    if (HIU) {
      const uint4 r = r01[k];
      g = {r.x, r.y, r.z};
    }
    return kb.start(g, k, keys);
  };
  uint4 y = make_uint4(0u, 0u, 0u, 0u);
  if (8u * q + 8u <= K) {
#pragma unroll
    for (uint32_t i = 0; i < 8u; i += 2u) {
      PhiloxState s = start(8u * q + i), t = start(8u * q + i + 1u);
#pragma unroll
      for (int r = 2; r < 10; ++r) {
        philox_round(s.c0, s.c1, s.c2, s.c3, keys.k0[r], keys.k1[r]);
        philox_round(t.c0, t.c1, t.c2, t.c3, keys.k0[r], keys.k1[r]);
      }
      fold_bits(y, make_uint4(s.c0, s.c1, s.c2, s.c3), i);
      fold_bits(y, make_uint4(t.c0, t.c1, t.c2, t.c3), i + 1u);
    }
  } else {
#pragma unroll 1
    for (uint32_t i = 0; 8u * q + i < K; ++i) fold_bits(y, philox_finish(start(8u * q + i), keys), i);
  }
  return y;
}

// One step of a probe-group pair: one block of this thread (its sums at TMEM
// address ta) over group q and, when `two`, q + 1, the groups added in order.
// Every lane takes part (an inactive lane's sums are never applied), so the
// step has no per-lane branch; the first group's Philox call runs while the
// sums come from TMEM (FIRST: they start at zero).
template <bool FIRST, bool HIU>
__device__ __forceinline__ void lut8_tm_step(uint32_t ta, const BlockCounter<HIU>& kb, uint32_t q,
                                             const GroupRound01& g0, const GroupRound01& g1, bool two, uint32_t frame,
                                             const RoundKeys& keys) {
  float acc[16];
  if (FIRST)
    zero16(acc);
  else
    tm_ld16(acc, ta);
  const uint4 x0 = philox_finish(kb.start(g0, q, keys), keys);
  if (!FIRST) tm_wait_ld(acc);
  lut8_lookup(acc, x0, frame);
  if (two) lut8_lookup(acc, philox_finish(kb.start(g1, q + 1u, keys), keys), frame | 128u);
  tm_st16(ta, acc);
}

// Rounds 2-9 of one Philox call (s: in, its state; out, its words) and, two
// elements per round, the lookups of a group whose words x are known, added
// to acc in element order; the additions trail the loads by a round. WAIT:
// acc may still be on its way from TMEM and is waited for before the first.
template <bool WAIT>
__device__ __forceinline__ void philox_with_lookups(PhiloxState& s, float (&acc)[16], const uint4& x, uint32_t frame,
                                                    const RoundKeys& rk) {
  float p0 = 0.0f, p1 = 0.0f;
#pragma unroll
  for (int r = 2; r < 10; ++r) {
    const int e = 2 * (r - 2);
    const uint32_t w = word_of(x, e >> 2);
    const uint32_t a0 = __byte_perm(w, frame, 0x7604u | (static_cast<uint32_t>(e & 3) << 4));
    const uint32_t a1 = __byte_perm(w, frame, 0x7604u | (static_cast<uint32_t>((e + 1) & 3) << 4));
    const float n0 = lds_f32(a0), n1 = lds_f32(a1);
    philox_round(s.c0, s.c1, s.c2, s.c3, rk.k0[r], rk.k1[r]);
    if (WAIT && r == 3) tm_wait_ld(acc);
    if (r > 2) fadd2_rn(acc[e - 2], acc[e - 1], p0, p1);
    p0 = n0;
    p1 = n1;
  }
  fadd2_rn(acc[14], acc[15], p0, p1);
}

// One step with the words one group ahead (x: those of group q of this block
// on entry, of group qn of the next block on return): each Philox call runs
// among the lookups of the group before it, so a warp mixes the multiplies of
// the one with the byte-permutes and shared loads of the other instead of
// waiting for each pipe in turn.
template <bool FIRST, bool HIU>
__device__ __forceinline__ void lut8_tm_step_ahead(uint32_t ta, uint4& x, BlockCounter<HIU>& kb, uint32_t q,
                                                   const GroupRound01& g1, const BlockCounter<HIU>& next, uint32_t qn,
                                                   const GroupRound01& gn, uint32_t frame, const RoundKeys& keys) {
  float acc[16];
  if (FIRST)
    zero16(acc);
  else
    tm_ld16(acc, ta);
  PhiloxState s = kb.start(g1, q + 1u, keys);
  philox_with_lookups<!FIRST>(s, acc, x, frame, keys);
  x = make_uint4(s.c0, s.c1, s.c2, s.c3);
  kb = next;
  s = kb.start(gn, qn, keys);
  philox_with_lookups<false>(s, acc, x, frame | 128u, keys);
  x = make_uint4(s.c0, s.c1, s.c2, s.c3);
  tm_st16(ta, acc);
}

// One step under packing 8.
template <bool HIU>
__device__ __forceinline__ void lut8_tm_step8(uint32_t ta, const BlockCounter<HIU>& kb, uint32_t q, uint32_t K,
                                              const uint4* r01, bool two, uint32_t frame, const RoundKeys& keys) {
  const uint4 x0 = group_words8(kb, q, K, r01, keys);
  float acc[16];
  if (q == 0u)
    zero16(acc);
  else
    tm_get16(acc, ta);
  lut8_lookup(acc, x0, frame);
  if (two) lut8_lookup(acc, group_words8(kb, q + 1u, K, r01, keys), frame | 128u);
  tm_st16(ta, acc);
}

// Shared memory besides the two regions: coefficients (8 per group), 4-probe
// tables (32 per group), under packing 8 the probes' Philox group parts (16
// bytes each), and the tensors of the chunk's blocks (one per warp and block),
// below the first region when they fit there, else after the second.
__host__ __device__ constexpr uint32_t lut8_side_bytes(int groups, bool pack8) {
  return (pack8 ? 288u : 160u) * static_cast<uint32_t>(groups) +
         4u * static_cast<uint32_t>(kLut8Threads / 32 * kLut8Bpt);
}
// Placed after the second region only when the slack below the first is
// smaller than it, so the layout ends within 2 * side + 128 KB of the window's
// start.
constexpr size_t lut8_smem_bytes(bool pack8) {
  const size_t after = 2 * static_cast<size_t>(kLut8Region) + 2 * lut8_side_bytes(kMaxGroups, pack8) + 16u;
  const size_t below = 3 * static_cast<size_t>(kLut8Region) + 16u;
  return after > below ? after : below;
}
static_assert(lut8_smem_bytes(true) <= 226 * 1024, "side data must fit the shared memory of an SM");

// HIU: every virtual block of the launch has the same counter high word (any
// launch below 2^36 weights), so the steps use the split Philox and a 32-bit
// block word (OPT-30B-shaped set, K = 256: 245.3 -> 235.9 ms, same bits).
// ANY: the launch may hold fp32 tensors and tensors off the 32-byte grid. An
// instantiation of its own: with their code in the same kernel the loop over
// the pairs is 2-3 % slower (registers), though it is the same source.
// AHEAD: the steps run with the words one group ahead (lut8_tm_step_ahead):
// faster from 24 groups on (OPT-30B-shaped layers, K = 256: 10.08 -> 9.95 ms,
// K = 1024 on the OPT-1.3B-shaped set: 40.1 -> 39.6 ms), slower below (K = 64:
// 4.23 -> 4.30 ms on Qwen3-8B-shaped layers), where the two groups' own calls
// overlap enough and the last pair weighs more.
template <bool HIU, bool ANY, bool PACK8, bool AHEAD>
__global__ void __launch_bounds__(kLut8Threads, 1) update_lut8_kernel(const __grid_constant__ UpdateParams P) {
  constexpr int THREADS = kLut8Threads, BPT = kLut8Bpt;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int skip_s;
  __shared__ uint32_t tmem_s;
  const int G = P.groups;
  const int NP = (G + 1) / 2;  // group pairs: groups 2p, 2p + 1 share one region
  const uint32_t sbase = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  const uint32_t region0 = (sbase + kLut8Region - 1u) & ~(kLut8Region - 1u);
  const uint32_t side = lut8_side_bytes(G, PACK8);
  const uint32_t hdr = region0 - sbase >= side ? sbase : region0 + 2u * kLut8Region;
  float* a_s = reinterpret_cast<float*>(smem + (hdr - sbase));  // 8 G coefficients
  float* t4 = a_s + 8 * G;                                      // 32 G 4-probe partials
  uint4* r01_s = reinterpret_cast<uint4*>(t4 + 32 * G);         // packing 8: 8 G group parts
  int* t_s = reinterpret_cast<int*>(PACK8 ? static_cast<void*>(r01_s + 8 * G) : static_cast<void*>(r01_s));

  if (threadIdx.x == 0) skip_s = (P.status != nullptr && *P.status != 0);
  for (int k = threadIdx.x; k < 8 * G; k += THREADS)
    a_s[k] = k < P.K ? __double2float_rn(P.coef_mul * P.coef[k]) : 0.0f;
  __syncthreads();
  const bool skip = skip_s != 0;
  if (skip && !P.has_pre) return;
  const TensorTable& tab = P.tab;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (skip) {  // a failed preconditioner: the leading perturbation alone
    int t = 0;
    for (uint32_t bl = blockIdx.x * THREADS + threadIdx.x; bl - lane < tab.blk_total; bl += gridDim.x * THREADS) {
      t = advance_tensor(tab, t, bl - lane);
      const Lut8Block k = lut8_block_info<ANY>(tab, t, bl);
      uint4 xp = block_bits(k.b, P.pre.ctr2, P.keys);
      if (ANY && (k.fl & kShift)) xp = window16(xp, 16u - k.a);
      if (k.vec && (k.fl & kDtypeMask) != kF32) {
        uint16_t* p = static_cast<uint16_t*>(k.base) + k.e0;
        uint32_t v[8];
        ld256(p, v);
#pragma unroll
        for (int r = 0; r < 8; ++r)
          v[r] = (k.fl & kDtypeMask) == kBF16 ? pre_regs16<kBF16>(v[r], xp, r, P.pre) : pre_regs16<kF16>(v[r], xp, r, P.pre);
        st256(p, v);
      } else if (k.act) {
        float none[16];
        zero16(none);
        lut8_apply_elements(k, none, xp, P, false);
      }
    }
    return;
  }
  const uint32_t t4_s = hdr + 32u * G;
  const uint32_t dst_t = 256u * (threadIdx.x >> 3) + 16u * (threadIdx.x & 7u);
  const uint32_t bhi = static_cast<uint32_t>(static_cast<uint64_t>(tab.blk_base) >> 32);
  for (int e = threadIdx.x; e < 32 * G; e += THREADS) {
    const float* a = a_s + 8 * (e >> 5) + ((e & 16) ? 4 : 0);
    t4[e] = quad_partial(a, static_cast<uint32_t>(e) & 15u);
  }
  if (PACK8 && HIU) {
    for (int k = threadIdx.x; k < 8 * G; k += THREADS) {
      const GroupRound01 g = group_round01(static_cast<uint32_t>(k), bhi, P.keys);
      r01_s[k] = make_uint4(g.x0, g.x2, g.lpa1, 0u);
    }
  }
  __syncthreads();
  lut8_replicate4<THREADS>(t4_s, region0 + dst_t, 0, G > 1);
  if (warp == 0) {
    __syncwarp();
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(&tmem_s));
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tm_fence_before();
  __syncthreads();
  tm_fence_after();
  // TMEM lane 32 (warp mod 4) + lane id, columns from 128 (warp / 4)
  const uint32_t trow = tmem_s + (((warp & 3u) * 32u) << 16) + (warp >> 2) * 128u;

  const uint32_t row = gridDim.x * static_cast<uint32_t>(THREADS);  // one block per thread of the launch
  const uint32_t per_round = row * static_cast<uint32_t>(BPT);
  const uint32_t rounds = (tab.blk_total + per_round - 1u) / per_round;
  uint32_t cur = 0;  // region holding the current pair (0 or 1)
  int t = 0;         // tensor of the warp's latest block
  const auto counter_word = [&](const Lut8Block& k) {
    return static_cast<uint32_t>(HIU ? static_cast<uint64_t>(k.b) : static_cast<uint64_t>(k.b - tab.blk_base));
  };

  for (uint32_t rnd = 0; rnd < rounds; ++rnd) {
    // this thread's blocks of the chunk: cb, cb + THREADS, .. The last round's chunks are shorter: its blocks
    // spread over all CTAs (20 M bf16 weights are two rounds and 0.6 %: K = 256 243 -> 185 us, K = 64 80 -> 64;
    // 3 M, a fraction of one, K = 256 60 -> 44)
    const uint32_t left = tab.blk_total - rnd * per_round;
    const int bpt = left >= per_round ? BPT : static_cast<int>((left + row - 1u) / row);
    const uint32_t cb = rnd * per_round + blockIdx.x * static_cast<uint32_t>(THREADS * bpt) + threadIdx.x;
    int jn = 0;          // blocks of the warp inside the launch
    uint32_t vr[BPT];    // their counter words (registers: 2-6 % faster than shared memory)
#pragma unroll
    for (int j = 0; j < BPT; ++j) {
      const uint32_t bl = cb + static_cast<uint32_t>(j * THREADS);
      vr[j] = 0u;
      if (j < bpt && bl - lane < tab.blk_total) {
        jn = j + 1;
        t = advance_tensor(tab, t, bl - lane);
        const Lut8Block k = lut8_block_info<ANY>(tab, t, bl);
        vr[j] = counter_word(k);
        if (lane == 0) t_s[j * (THREADS / 32) + warp] = t;
        // theta is read with the last pair: bring it into L2 meanwhile
        if (k.vec) {
          const bool f32 = ANY && (k.fl & kDtypeMask) == kF32;
          const char* p = static_cast<const char*>(k.base) + k.e0 * (f32 ? 4 : 2);
          asm volatile("prefetch.L2 [%0];" ::"l"(p));
          if (f32) asm volatile("prefetch.L2 [%0];" ::"l"(p + 32));
        }
      }
    }
    __syncwarp();
    bool others = false;  // a block of the chunk goes element by element
    uint4 ahead = make_uint4(0u, 0u, 0u, 0u);  // AHEAD: the next step's words
    for (int pr = 0; pr < NP; ++pr) {
      const uint32_t frame = ((region0 + cur * kLut8Region) & 0xFFFF0000u) | (lane << 2);
      const uint32_t q = 2u * static_cast<uint32_t>(pr);
      const bool two = static_cast<int>(q) + 1 < G;
      const GroupRound01 g0 = group_round01(q, bhi, P.keys);
      const GroupRound01 g1 = group_round01(q + 1u, bhi, P.keys);
      if (pr + 1 < NP) {
        if constexpr (PACK8) {
#pragma unroll 1
          for (int j = 0; j < jn; ++j) {
            const Lut8Block k = lut8_block_info<ANY>(tab, t_s[j * (THREADS / 32) + warp],
                                                     cb + static_cast<uint32_t>(j * THREADS));
            lut8_tm_step8<HIU>(trow + 16u * static_cast<uint32_t>(j),
                               BlockCounter<HIU>(counter_word(k), tab.blk_base, P.keys), q,
                               static_cast<uint32_t>(P.K), r01_s, two, frame, P.keys);
          }
        } else {
          const auto run_ahead = [&](auto first) {
            if (jn == 0) return;
            const GroupRound01 g2 = group_round01(q + 2u, bhi, P.keys);
            BlockCounter<HIU> kb(vr[0], tab.blk_base, P.keys);
            if (decltype(first)::value) ahead = philox_finish(kb.start(g0, q, P.keys), P.keys);
#pragma unroll
            for (int j = 0; j < BPT; ++j) {
              if (j >= jn) break;
              const bool wrap = j + 1 == jn;  // next: block 0 of the next pair
              const GroupRound01 gn = {wrap ? g2.x0 : g0.x0, wrap ? g2.x2 : g0.x2, wrap ? g2.lpa1 : g0.lpa1};
              lut8_tm_step_ahead<decltype(first)::value, HIU>(
                  trow + 16u * static_cast<uint32_t>(j), ahead, kb, q, g1,
                  BlockCounter<HIU>(wrap ? vr[0] : vr[j + 1 < BPT ? j + 1 : 0], tab.blk_base, P.keys),
                  wrap ? q + 2u : q, gn, frame, P.keys);
            }
          };
          const auto run = [&](auto first) {
            if constexpr (AHEAD) {
              run_ahead(first);
            } else {
#pragma unroll
              for (int j = 0; j < BPT; ++j) {
                if (j >= jn) break;
                lut8_tm_step<decltype(first)::value, HIU>(trow + 16u * static_cast<uint32_t>(j),
                                                          BlockCounter<HIU>(vr[j], tab.blk_base, P.keys), q, g0, g1,
                                                          two, frame, P.keys);
              }
            }
          };
          if (pr == 0)
            run(std::true_type());
          else
            run(std::false_type());
        }
        tm_wait_st();  // this pair's sums are in TMEM before the next pair reads them
      } else {
        // The last pair applies the sums to theta as they complete: the loads
        // are issued before the block's lookups, which hide them, and theta's
        // traffic spreads over the pair instead of coming in a phase of its
        // own. Blocks across a tensor's end leave their sums in TMEM for a
        // pass of their own.
        const int pre_at = !P.has_pre ? 0 : PACK8 ? 3 : P.pre.ctr2 == q ? 1 : (two && P.pre.ctr2 == q + 1u) ? 2 : 3;
#pragma unroll 1
        for (int j = 0; j < jn; ++j) {
          const uint32_t ta = trow + 16u * static_cast<uint32_t>(j);
          const Lut8Block k = lut8_block_info<ANY>(tab, t_s[j * (THREADS / 32) + warp],
                                                   cb + static_cast<uint32_t>(j * THREADS));
          const bool f32 = ANY && (k.fl & kDtypeMask) == kF32;  // the same in all lanes
          char* tp = static_cast<char*>(k.base) + k.e0 * (f32 ? 4 : 2);
          uint32_t v[16];
          uint32_t(&lo)[8] = *reinterpret_cast<uint32_t(*)[8]>(&v[0]);
          uint32_t(&hi)[8] = *reinterpret_cast<uint32_t(*)[8]>(&v[8]);
          if (k.vec) ld256(tp, lo);
          if (ANY && k.vec && f32) ld256(tp + 32, hi);
          const BlockCounter<HIU> kb(counter_word(k), tab.blk_base, P.keys);
          float acc[16];
          uint4 x, xp;  // xp: words of the leading perturbation: group q's, q + 1's or its own
          if constexpr (PACK8) {
            x = group_words8(kb, q, static_cast<uint32_t>(P.K), r01_s, P.keys);
            if (pr == 0)
              zero16(acc);
            else
              tm_get16(acc, ta);
          } else {
            if (!HIU && pr == 0)
              zero16(acc);
            else
              tm_ld16(acc, ta);
            if (AHEAD && j == 0)
              x = ahead;
            else
              x = philox_finish(kb.start(g0, q, P.keys), P.keys);
            tm_wait_ld(acc);
          }
          lut8_lookup(acc, x, frame);
          xp = x;
          if (two) {
            x = PACK8 ? group_words8(kb, q + 1u, static_cast<uint32_t>(P.K), r01_s, P.keys)
                      : philox_finish(kb.start(g1, q + 1u, P.keys), P.keys);
            lut8_lookup(acc, x, frame | 128u);
            if (pre_at == 2) xp = x;
          }
          if (__any_sync(0xFFFFFFFFu, k.act && !k.vec)) {
            tm_st16(ta, acc);
            others = true;
          }
          if (pre_at == 3) xp = block_bits(k.b, P.pre.ctr2, P.keys);
          if (ANY && (k.fl & kShift)) {  // the same in all lanes
            window16f(acc, 16u - k.a);
            if (P.has_pre) xp = window16(xp, 16u - k.a);
          }
          if (k.vec) {
            if (ANY && f32) {
              lut8_apply32(v, acc, xp, P);
              st256(tp + 32, hi);
            } else if ((k.fl & kDtypeMask) == kBF16) {
              update_regs16<kBF16>(lo, acc, xp, P.has_pre, P.pre);
            } else {
              update_regs16<kF16>(lo, acc, xp, P.has_pre, P.pre);
            }
            st256(tp, lo);
          }
        }
        if (others) {
          tm_wait_st();
#pragma unroll 1
          for (int j = 0; j < jn; ++j) {
            const Lut8Block k = lut8_block_info<ANY>(tab, t_s[j * (THREADS / 32) + warp],
                                                     cb + static_cast<uint32_t>(j * THREADS));
            const bool mine = k.act && !k.vec;
            if (!__any_sync(0xFFFFFFFFu, mine)) continue;
            float acc[16];
            tm_get16(acc, trow + 16u * static_cast<uint32_t>(j));
            uint4 xp = make_uint4(0u, 0u, 0u, 0u);
            if (P.has_pre) xp = block_bits(k.b, P.pre.ctr2, P.keys);
            if (ANY && (k.fl & kShift)) {
              window16f(acc, 16u - k.a);
              xp = window16(xp, 16u - k.a);
            }
            if (mine) lut8_apply_elements(k, acc, xp, P, true);
          }
        }
      }
      if (NP > 1) {
        // the next pair (wrapping to pair 0 for the next chunk) into the other region
        const int qn = pr + 1 < NP ? static_cast<int>(q) + 2 : 0;
        lut8_replicate4<THREADS>(t4_s, region0 + (cur ^ 1u) * kLut8Region + dst_t, qn, qn + 1 < G);
        __syncthreads();
        cur ^= 1u;
      }
    }
  }
  tm_fence_before();
  __syncthreads();
  tm_fence_after();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_s), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------
// One to four probe groups (K <= 32): the tables stay in shared memory for the
// whole launch, so there is no chunking and no barrier. The kernel walks
// 32-byte items of theta grid-stride like the perturbation passes (sixteen
// 16-bit or eight fp32 elements, half a Philox block), the next item's 256-bit
// load issued before the current one is computed: the same sums, in the same
// order (0 + T8_0 + T8_1 ...), as the chunk kernel.
//
// At K <= 16 the bound is one pass over HBM, 379 cycles per warp and item at
// 2.07 GHz, and what the SM has to issue in that time: two Philox calls cost
// about 180 (a 32x32->64 multiply holds the issue for four), so the rest has
// to be short:
//  * Philox rounds 0-1 split as in the chunk kernel, the groups' parts from
//    the host (parameter space, no registers);
//  * group 0's table holds 0 + T8_0, so its addition to 0 is gone;
//  * with the leading perturbation's probe in the last group (the fused
//    schedule's restore of probe K - 1), that group's entries are pairs (T8,
//    the signed scale): one 64-bit lookup gives both, in place of a multiply
//    and a logic operation per element. Its sums are scalar adds: packed ones
//    would need the two elements' halves moved into register pairs first
//    (0.95 against 0.90 ms at K = 16, 1.00 against 0.79 ms at K = 8).
// OPT-1.3B-shaped bf16 set (one pass at the copy bandwidth: 0.775 ms), with
// the leading perturbation: K = 8 0.845 -> 0.787 ms, K = 16 0.941 -> 0.903 ms
// (fp16 0.962 -> 0.880); without it 0.822 -> 0.780 and 0.880 -> 0.810 ms. fp32
// and tensors off the 32-byte grid ran element by element or in a kernel of
// their own before: 205 M fp32 weights, K = 16: 0.332 -> 0.249 ms; 400 M bf16
// weights in one flat buffer, K = 16: 0.749 -> 0.381 ms. Not adopted: a
// prefetch of the item after the next into L2 (K = 16 -2 %, K = 8 +10 %).
// ---------------------------------------------------------------------------
// Threads of a CTA: three and four groups' words take more registers than 64
// (OPT-1.3B-shaped set, ms at 512 / 768 / 1024 threads: three groups 1.107 /
// 1.122 / 1.219 with the leading perturbation, 1.018 / 1.000 / 1.131 without;
// four 1.386 / 1.629 / 1.612 and 1.284 / 1.270 / 1.474; 400 M weights in one
// flat buffer 0.472 / 0.451 / 0.521 and 0.584 / 0.640 / 0.621).
__host__ __device__ constexpr int small_threads(int G) { return G <= 2 ? 1024 : G == 3 ? 768 : 512; }
// The last group's (T8, signed scale) pairs fill a region, plain tables half of one.
__host__ __device__ constexpr uint32_t small_regions(int G, bool pairs) {
  return pairs ? 1u + static_cast<uint32_t>(G) / 2u : (static_cast<uint32_t>(G) + 1u) / 2u;
}
constexpr size_t small_smem_bytes(int G, bool pairs) {
  return (1 + small_regions(G, pairs)) * static_cast<size_t>(kLut8Region) + 16u;
}

__device__ __forceinline__ void lds_pair(uint32_t addr, float& a, float& b) {
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(a), "=f"(b) : "r"(addr));
}

// Shared address of element i's entry: its sign byte in byte i mod 4 of w.
template <int I>
__device__ __forceinline__ uint32_t entry_addr(uint32_t w, uint32_t frame) {
  return __byte_perm(w, frame, 0x7604u | (static_cast<uint32_t>(I & 3) << 4));
}

// The leading perturbation in the small kernel: none, in the last group's
// table, with Philox words of its own, with the last group's words (four
// groups, whose tables leave no room for pairs), or with another group's.
constexpr int kPreNone = 0, kPreTable = 1, kPreOwn = 2, kPreLast = 3, kPreGroup = 4;

// Element I's partial sums, and with kPreTable its leading perturbation (d).
// x: the groups' words; f0, fl: frames of group 0's and the last group's tables.
template <int I, int PRE, int G>
__device__ __forceinline__ void small_sums(const uint4 (&x)[G], uint32_t f0, uint32_t fl, float (&t)[G], float& d) {
#pragma unroll
  for (int g = 0; g < G - 1; ++g)
    t[g] = lds_f32(entry_addr<I>(word_of(x[g], I >> 2), f0 + (g & 1) * 128u + (g >> 1) * kLut8Region));
  if constexpr (PRE == kPreTable)
    lds_pair(entry_addr<I>(word_of(x[G - 1], I >> 2), fl), t[G - 1], d);
  else
    t[G - 1] = lds_f32(entry_addr<I>(word_of(x[G - 1], I >> 2), fl));
}

// Elements 2R and 2R + 1, 16-bit.
template <uint8_t DT, int PRE, int G, int R>
__device__ __forceinline__ void small_pair16(uint32_t& v, const uint4 (&x)[G], const uint4& xp, uint32_t f0,
                                             uint32_t fl, const UpdateParams& P) {
  constexpr int e = 2 * R;
  float2 f = unpack2<DT>(v);
  float t[G], u[G], d0 = 0.0f, d1 = 0.0f;
  small_sums<e, PRE, G>(x, f0, fl, t, d0);
  small_sums<e + 1, PRE, G>(x, f0, fl, u, d1);
  if constexpr (PRE != kPreNone) {
    if constexpr (PRE == kPreTable) {
      f.x = __fadd_rn(f.x, d0);
      f.y = __fadd_rn(f.y, d1);
    } else {
      add_signed2(f, xp, e, P.pre);
    }
    f = unpack2<DT>(pack2<DT>(f.x, f.y));  // the perturbed value is rounded to storage first
  }
#pragma unroll
  for (int g = 1; g < G - 1; ++g) fadd2_rn(t[0], u[0], t[g], u[g]);
  if constexpr (PRE == kPreTable) {
    if constexpr (G > 1) {
      t[0] = __fadd_rn(t[0], t[G - 1]);
      u[0] = __fadd_rn(u[0], u[G - 1]);
    }
    f.x = __fadd_rn(f.x, t[0]);
    f.y = __fadd_rn(f.y, u[0]);
  } else {
    if constexpr (G > 1) fadd2_rn(t[0], u[0], t[G - 1], u[G - 1]);
    fadd2_rn(f.x, f.y, t[0], u[0]);
  }
  v = pack2<DT>(f.x, f.y);
}

template <uint8_t DT, int PRE, int G>
__device__ __forceinline__ void small_item16(uint32_t (&v)[8], const uint4 (&x)[G], const uint4& xp, uint32_t f0,
                                             uint32_t fl, const UpdateParams& P) {
  small_pair16<DT, PRE, G, 0>(v[0], x, xp, f0, fl, P);
  small_pair16<DT, PRE, G, 1>(v[1], x, xp, f0, fl, P);
  small_pair16<DT, PRE, G, 2>(v[2], x, xp, f0, fl, P);
  small_pair16<DT, PRE, G, 3>(v[3], x, xp, f0, fl, P);
  small_pair16<DT, PRE, G, 4>(v[4], x, xp, f0, fl, P);
  small_pair16<DT, PRE, G, 5>(v[5], x, xp, f0, fl, P);
  small_pair16<DT, PRE, G, 6>(v[6], x, xp, f0, fl, P);
  small_pair16<DT, PRE, G, 7>(v[7], x, xp, f0, fl, P);
}

// One fp32 element (scalar adds, as every fp32 path).
template <int PRE, int G, int I>
__device__ __forceinline__ void small_one32(uint32_t& v, const uint4 (&x)[G], const uint4& xp, uint32_t f0, uint32_t fl,
                                            const UpdateParams& P) {
  float th = __uint_as_float(v);
  float t[G], d = 0.0f;
  small_sums<I, PRE, G>(x, f0, fl, t, d);
  if constexpr (PRE == kPreTable)
    th = __fadd_rn(th, d);
  else if constexpr (PRE != kPreNone)
    th = add_signed(th, xp, I, P.pre);
#pragma unroll
  for (int g = 1; g < G; ++g) t[0] = __fadd_rn(t[0], t[g]);
  v = __float_as_uint(__fadd_rn(th, t[0]));
}

template <int PRE, int G>
__device__ __forceinline__ void small_item32(uint32_t (&v)[8], const uint4 (&x)[G], const uint4& xp, uint32_t f0,
                                             uint32_t fl, const UpdateParams& P) {
  small_one32<PRE, G, 0>(v[0], x, xp, f0, fl, P);
  small_one32<PRE, G, 1>(v[1], x, xp, f0, fl, P);
  small_one32<PRE, G, 2>(v[2], x, xp, f0, fl, P);
  small_one32<PRE, G, 3>(v[3], x, xp, f0, fl, P);
  small_one32<PRE, G, 4>(v[4], x, xp, f0, fl, P);
  small_one32<PRE, G, 5>(v[5], x, xp, f0, fl, P);
  small_one32<PRE, G, 6>(v[6], x, xp, f0, fl, P);
  small_one32<PRE, G, 7>(v[7], x, xp, f0, fl, P);
}

// An item across an end of its tensor, element by element (not inlined: it
// is rare and would otherwise hold registers in the loop). e0: the item's
// first element; do_sum false: the leading perturbation alone.
// x0, mid, xl: the groups' words (one group: xl)
template <int PRE, int G, class... Mid>
__device__ __noinline__ void small_elements(void* base, uint8_t dt, int64_t e0, int64_t numel, uint4 x0, uint4 xl,
                                            uint4 xp, uint32_t f0, uint32_t fl, bool do_sum, PerturbOp pre, Mid... mid) {
  const uint4 x[G > 1 ? G - 1 : 1] = {x0, mid...};
  const int per = dt == kF32 ? 8 : 16;
  const int lo = e0 < 0 ? static_cast<int>(-e0) : 0;
  const int hi = static_cast<int>(min(static_cast<int64_t>(per), numel - e0));
  map_elements<2>(base, dt, e0, lo, hi, [&](int m, int j, float v) {
    float th = v, t = 0.0f, l = 0.0f, d = 0.0f;
    if (do_sum) {
      const uint32_t sel = 0x7604u | (static_cast<uint32_t>(j) << 4);
#pragma unroll
      for (int g = 0; g < G - 1; ++g) {
        const float p = lds_f32(__byte_perm(word_of(x[g], m), f0 + (g & 1) * 128u + (g >> 1) * kLut8Region, sel));
        t = g == 0 ? p : __fadd_rn(t, p);
      }
      const uint32_t at = __byte_perm(word_of(xl, m), fl, sel);
      if constexpr (PRE == kPreTable)
        lds_pair(at, l, d);
      else
        l = lds_f32(at);
    }
    if (PRE != kPreNone) {
      th = do_sum && PRE == kPreTable ? __fadd_rn(th, d) : add_signed_word(th, word_of(xp, m), j, pre);
      th = round_to_storage(dt, th);
    }
    return do_sum ? __fadd_rn(th, G > 1 ? __fadd_rn(t, l) : l) : th;
  });
}

// A warp's position in the table: its 32 items lie in one tensor.
struct SmallCursor {
  int t;
  uint32_t tb, te;   // first and one-past-last launch item
  uint32_t full;     // full aligned items from tb (0: tensors off the 32-byte grid)
  uint32_t vb;       // low word of the virtual block of the tensor's first element
  char* p;           // base pointer
  uint8_t fl;        // flags
  uint32_t a;        // kShift: the base's offset from the 32-byte boundary below it, in elements
};

template <bool ANY>
__device__ __forceinline__ void small_seek(const TensorTable& tab, SmallCursor& c, uint32_t b) {
  c.t = advance_tensor(tab, c.t, b);
  c.tb = tensor_blk_begin(tab, c.t);
  c.te = tab.blk_end[c.t];
  c.fl = tab.flags[c.t];
  c.p = reinterpret_cast<char*>(tab.ptr[c.t]);
  c.vb = static_cast<uint32_t>(static_cast<uint64_t>(virtual_block(tab, c.t, c.tb)));
  const bool f32 = ANY && (c.fl & kDtypeMask) == kF32;
  c.full = (c.fl & kVec32) ? static_cast<uint32_t>(tab.numel[c.t] / (f32 ? 8 : 16)) : 0u;
  c.a = ANY ? static_cast<uint32_t>(tab.ptr[c.t] & 31u) / (f32 ? 4u : 2u) : 0u;
}

// A lane's item. Tensors off the 32-byte grid (kShift): each warp takes 31 of
// their aligned 32-byte chunks, lane l the chunk 31 w + l - 1 and the signs of
// the elements that fall into the block (fp32: half block) below from lane
// l - 1; lane 0 only generates.
struct SmallItem {
  char* p;        // the item's address (full)
  uint32_t blk;   // low word of the Philox block it generates
  int64_t e0;     // its first element
  bool upper;     // fp32: the block's upper half
  bool full;      // all its elements exist, 32-byte aligned
  bool act;       // some do
};

template <bool ANY>
__device__ __forceinline__ SmallItem small_item(const TensorTable& tab, const SmallCursor& c, uint32_t b) {
  SmallItem k;
  const uint32_t d = b - c.tb;
  if constexpr (!ANY) {
    k.full = d < c.full;
    k.act = b < c.te;
    k.p = c.p + static_cast<size_t>(d) * 32;
    k.blk = c.vb + d;
    k.e0 = static_cast<int64_t>(d) * 16;
    k.upper = false;
  } else {
    const bool f32 = (c.fl & kDtypeMask) == kF32;
    const int per = f32 ? 8 : 16;
    int64_t i = d;  // item number inside the tensor
    if (c.fl & kShift) i = static_cast<int64_t>(d >> 5) * kShiftLanes + static_cast<int64_t>(d & 31u) - 1;
    k.e0 = i * per - c.a;
    const int64_t numel = tab.numel[c.t];
    k.act = (c.fl & kShift) ? (d & 31u) != 0u && k.e0 < numel : b < c.te;
    k.full = k.act && k.e0 >= 0 && k.e0 + per <= numel;
    k.p = c.p + k.e0 * (f32 ? 4 : 2);
    k.blk = c.vb + static_cast<uint32_t>(static_cast<uint64_t>(f32 ? i >> 1 : i));
    k.upper = f32 && (i & 1) != 0;
  }
  return k;
}

__device__ __forceinline__ uint4 small_window(const SmallCursor& c, const SmallItem& k, const uint4& x) {
  return item_signs(x, (c.fl & kDtypeMask) == kF32, k.upper, (c.fl & kShift) != 0, c.a);
}

// The groups' words of an aligned fp32 item. Lanes 2 j and 2 j + 1 hold the
// halves of one block, so of every two groups each lane makes one's words and
// hands the other lane the half that it needs. 205 M fp32 weights, K = 16 / 24 /
// 32 (the last in the chunk kernel before): 265 / 337 / 379 -> 249 / 291 / 336 us;
// 40 M, K = 24: 72 -> 64 us.
template <int G>
__device__ __forceinline__ void small_pair_words(uint4 (&x)[G], const BlockCounter<true>& kb,
                                                 const GroupRound01 (&gs)[kSmallGroups], bool upper,
                                                 const RoundKeys& keys) {
#pragma unroll
  for (int g = 0; g + 1 < G; g += 2) {
    const GroupRound01 mine = {upper ? gs[g + 1].x0 : gs[g].x0, upper ? gs[g + 1].x2 : gs[g].x2,
                               upper ? gs[g + 1].lpa1 : gs[g].lpa1};
    const uint4 y = philox_finish(kb.start(mine, 0u, keys), keys);
    const uint32_t a = __shfl_xor_sync(0xFFFFFFFFu, upper ? y.x : y.z, 1);
    const uint32_t b = __shfl_xor_sync(0xFFFFFFFFu, upper ? y.y : y.w, 1);
    x[g] = make_uint4(upper ? a : y.x, upper ? b : y.y, 0u, 0u);
    x[g + 1] = make_uint4(upper ? y.z : a, upper ? y.w : b, 0u, 0u);
  }
  if (G & 1) {
    const uint4 y = philox_finish(kb.start(gs[G - 1], 0u, keys), keys);
    x[G - 1] = upper ? make_uint4(y.z, y.w, 0u, 0u) : make_uint4(y.x, y.y, 0u, 0u);
  }
}

// ANY: the launch may hold fp32 tensors (numbered in half blocks) and tensors
// off the 32-byte grid (32 launch items per 31 chunks). BLOCKS: mostly aligned
// fp32, whose words a pair of lanes makes once (small_pair_words); in the
// general instantiation that code costs views 4 % (586 -> 607 us, K = 32).
template <int PRE, int G, bool ANY, bool BLOCKS>
__global__ void __launch_bounds__(small_threads(G), 1)
    update_lut8_small_kernel(const __grid_constant__ SmallUpdateParams S) {
  constexpr int kThreads = small_threads(G);
  const UpdateParams& P = S.u;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int skip_s;
  constexpr uint32_t kRegions = small_regions(G, PRE == kPreTable);
  const uint32_t sbase = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  const uint32_t region0 = (sbase + kLut8Region - 1u) & ~(kLut8Region - 1u);
  // coefficients and unreplicated tables (1 KB per group) below the region, or after it when the window starts on
  // a 64 KB boundary
  const uint32_t hdr = region0 - sbase >= 32u * G + 1024u * G ? sbase : region0 + kRegions * kLut8Region;
  float* a_s = reinterpret_cast<float*>(smem + (hdr - sbase));
  float* t8 = a_s + 8 * G;
  if (threadIdx.x == 0) skip_s = (P.status != nullptr && *P.status != 0);
  for (int k = threadIdx.x; k < 8 * G; k += kThreads)
    a_s[k] = k < P.K ? __double2float_rn(P.coef_mul * P.coef[k]) : 0.0f;
  __syncthreads();
  const bool do_sum = skip_s == 0;  // a failed preconditioner still gets the leading perturbation
  if (!do_sum && PRE == kPreNone) return;
  if (do_sum) {
    for (int e = threadIdx.x; e < 256 * G; e += kThreads) {
      const float* a = a_s + 8 * (e >> 8);
      const uint32_t n = static_cast<uint32_t>(e) & 255u;
      const float v = __fadd_rn(quad_partial(a, n & 15u), quad_partial(a + 4, n >> 4));
      t8[e] = e < 256 ? __fadd_rn(0.0f, v) : v;
    }
    __syncthreads();
    // rows of 256 bytes. Pairs: (T8, signed scale) of the last group, lane l in 8-byte word l of the last region;
    // plain tables: group g in region g / 2, lane l in word l of half g mod 2 of the row
    constexpr int kPieces = 256 * 16;  // 16-byte pieces of a region
    for (int i = threadIdx.x; i < kPieces; i += kThreads) {
      const uint32_t n = static_cast<uint32_t>(i) >> 4, piece = static_cast<uint32_t>(i) & 15u;
#pragma unroll
      for (uint32_t r = 0; r < kRegions; ++r) {
        const uint32_t row = region0 + r * kLut8Region + 256u * n + 16u * piece;
        if (PRE == kPreTable && r == kRegions - 1u) {
          const float v = t8[256 * (G - 1) + n];
          const float d = __uint_as_float(P.pre.nscale_bits ^ (((n >> P.pre.bit) & 1u) << 31));
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %1, %2};" ::"r"(row), "f"(v), "f"(d) : "memory");
        } else {
          const int g = static_cast<int>(2u * r + (piece >> 3));
          if (g < (PRE == kPreTable ? G - 1 : G)) sts_f32x4(row, t8[256 * g + static_cast<int>(n)]);
        }
      }
    }
    __syncthreads();
  }
  const TensorTable& tab = P.tab;
  const uint32_t total = tab.blk_total;
  const uint32_t stride = gridDim.x * kThreads;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t f0 = (region0 & 0xFFFF0000u) | (lane << 2);
  const uint32_t fl = PRE == kPreTable
                          ? ((region0 + (kRegions - 1u) * kLut8Region) & 0xFFFF0000u) | (lane << 3)
                          : f0 + ((G - 1) & 1) * 128u + ((G - 1) >> 1) * kLut8Region;
  uint32_t b = blockIdx.x * kThreads + threadIdx.x;
  if (b - lane >= total) return;
  SmallCursor c;
  c.t = 0;
  small_seek<ANY>(tab, c, b - lane);
  const auto edge = [&](const SmallCursor& at, const SmallItem& i, const uint4 (&x)[G], const uint4& xp, bool sum) {
    const uint8_t dt = at.fl & kDtypeMask;
    const int64_t n = tab.numel[at.t];
    if constexpr (G <= 2)
      small_elements<PRE, G>(at.p, dt, i.e0, n, x[0], x[G - 1], xp, f0, fl, sum, P.pre);
    else if constexpr (G == 3)
      small_elements<PRE, G>(at.p, dt, i.e0, n, x[0], x[2], xp, f0, fl, sum, P.pre, x[1]);
    else
      small_elements<PRE, G>(at.p, dt, i.e0, n, x[0], x[3], xp, f0, fl, sum, P.pre, x[1], x[2]);
  };
  if (!do_sum) {
    for (; b - lane < total; b += stride) {
      if (b - lane >= c.te) small_seek<ANY>(tab, c, b - lane);
      const SmallItem k = small_item<ANY>(tab, c, b);
      const BlockCounter<true> kb(k.blk, 0, P.keys);
      uint4 xp = philox_finish(kb.start(S.gp, 0u, P.keys), P.keys);
      if (ANY) xp = small_window(c, k, xp);
      uint4 x[G];  // not looked at
#pragma unroll
      for (int g = 0; g < G; ++g) x[g] = xp;
      if (k.act) edge(c, k, x, xp, false);
    }
    return;
  }
  SmallItem k = small_item<ANY>(tab, c, b);
  uint32_t v[8];
  if (k.full) ld256(k.p, v);
  while (true) {
    const uint32_t bn = b + stride;
    const bool more = bn - lane < total;
    SmallCursor cn = c;
    SmallItem kn = k;
    uint32_t vn[8];
    if (more) {
      if (bn - lane >= c.te) small_seek<ANY>(tab, cn, bn - lane);
      kn = small_item<ANY>(tab, cn, bn);
      if (kn.full) ld256(kn.p, vn);
    }
    const BlockCounter<true> kb(k.blk, 0, P.keys);
    uint4 x[G];
    uint4 xp = make_uint4(0u, 0u, 0u, 0u);
    if (BLOCKS && (c.fl & kDtypeMask) == kF32 && !(c.fl & kShift)) {
      small_pair_words<G>(x, kb, S.g, k.upper, P.keys);
      if (PRE == kPreOwn) xp = small_window(c, k, philox_finish(kb.start(S.gp, 0u, P.keys), P.keys));
    } else {
      x[0] = philox_finish(kb.start(S.g[0], 0u, P.keys), P.keys);
#pragma unroll
      for (int g = 1; g < G; ++g) x[g] = philox_finish(kb.start(S.g[g], static_cast<uint32_t>(g), P.keys), P.keys);
      if (PRE == kPreOwn) xp = philox_finish(kb.start(S.gp, 0u, P.keys), P.keys);
      if (ANY) {
        x[0] = small_window(c, k, x[0]);
#pragma unroll
        for (int g = 1; g < G; ++g) x[g] = small_window(c, k, x[g]);
        if (PRE == kPreOwn) xp = small_window(c, k, xp);
      }
    }
    if (PRE == kPreLast) xp = x[G - 1];
    if constexpr (PRE == kPreGroup) {  // the same group in all lanes
      xp = x[0];
#pragma unroll
      for (int g = 1; g + 1 < G; ++g)
        if (P.pre.ctr2 == static_cast<uint32_t>(g)) xp = x[g];
    }
    if (k.full) {
      if (ANY && (c.fl & kDtypeMask) == kF32)
        small_item32<PRE, G>(v, x, xp, f0, fl, P);
      else if ((c.fl & kDtypeMask) == kBF16)
        small_item16<kBF16, PRE, G>(v, x, xp, f0, fl, P);
      else
        small_item16<kF16, PRE, G>(v, x, xp, f0, fl, P);
      st256(k.p, v);
    } else if (k.act) {
      edge(c, k, x, xp, true);
    }
    if (!more) break;
    b = bn;
    c = cn;
    k = kn;
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = vn[r];
  }
}

template <bool HIU, bool ANY, bool PACK8, bool AHEAD = false>
cudaError_t launch_lut8_cfg(const UpdateParams& p, int sms, cudaStream_t stream) {
  // one CTA per SM, or per 512 blocks of a short list
  const int64_t want = (static_cast<int64_t>(p.tab.blk_total) + kLut8Threads - 1) / kLut8Threads;
  const int grid = static_cast<int>(want < sms ? want : sms);
  update_lut8_kernel<HIU, ANY, PACK8, AHEAD><<<grid, kLut8Threads, lut8_smem_bytes(PACK8), stream>>>(p);
  return cudaGetLastError();
}

template <bool HIU, bool ANY, bool PACK8, bool AHEAD = false>
cudaError_t lut8_limit() {
  return cudaFuncSetAttribute(update_lut8_kernel<HIU, ANY, PACK8, AHEAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(lut8_smem_bytes(PACK8)));
}

template <int PRE, int G, bool ANY, bool BLOCKS = false>
cudaError_t small_limit() {
  return cudaFuncSetAttribute(update_lut8_small_kernel<PRE, G, ANY, BLOCKS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(small_smem_bytes(G, PRE == kPreTable)));
}

// Whether there is a BLOCKS instantiation (see lut8_small_takes).
constexpr bool small_has_blocks(int pre, int G) { return G > 1 && !(pre == kPreGroup && G == 4); }

template <int PRE, int G>
cudaError_t small_limits() {
  cudaError_t e = small_limit<PRE, G, false>();
  if (e == cudaSuccess) e = small_limit<PRE, G, true>();
  if constexpr (small_has_blocks(PRE, G))
    if (e == cudaSuccess) e = small_limit<PRE, G, true, true>();
  return e;
}

cudaError_t lut8_prepare() {
  cudaError_t e = small_limits<kPreNone, 1>();
  if (e == cudaSuccess) e = small_limits<kPreNone, 2>();
  if (e == cudaSuccess) e = small_limits<kPreNone, 3>();
  if (e == cudaSuccess) e = small_limits<kPreNone, 4>();
  if (e == cudaSuccess) e = small_limits<kPreTable, 1>();
  if (e == cudaSuccess) e = small_limits<kPreTable, 2>();
  if (e == cudaSuccess) e = small_limits<kPreTable, 3>();
  if (e == cudaSuccess) e = small_limits<kPreLast, 4>();
  if (e == cudaSuccess) e = small_limits<kPreOwn, 1>();
  if (e == cudaSuccess) e = small_limits<kPreOwn, 2>();
  if (e == cudaSuccess) e = small_limits<kPreGroup, 2>();
  if (e == cudaSuccess) e = small_limits<kPreGroup, 3>();
  if (e == cudaSuccess) e = small_limits<kPreGroup, 4>();
  if (e == cudaSuccess) e = lut8_limit<true, false, false>();
  if (e == cudaSuccess) e = lut8_limit<true, false, false, true>();
  if (e == cudaSuccess) e = lut8_limit<true, true, false>();
  if (e == cudaSuccess) e = lut8_limit<false, true, false>();
  if (e == cudaSuccess) e = lut8_limit<true, true, true>();
  if (e == cudaSuccess) e = lut8_limit<false, true, true>();
  return e;
}

constexpr int kAheadGroups = 24;  // see AHEAD

bool one_high_word(const TensorTable& tab) {
  // every virtual block that a lane sums lies in [blk_base, blk_base + blk_total), except the one below a
  // tensor's first chunk, whose sums nothing uses
  const uint64_t first = static_cast<uint64_t>(tab.blk_base);
  const uint64_t last = first + (tab.blk_total > 0 ? tab.blk_total - 1u : 0u);
  return (first >> 32) == (last >> 32);
}

template <int PRE, int G>
void launch_small_cfg(const SmallUpdateParams& p, bool any, int sms, cudaStream_t stream) {
  constexpr size_t sm = small_smem_bytes(G, PRE == kPreTable);
  constexpr int threads = small_threads(G);
  const int64_t want = (static_cast<int64_t>(p.u.tab.blk_total) + threads - 1) / threads;
  const int grid = static_cast<int>(want < sms ? want : sms);
  if constexpr (small_has_blocks(PRE, G)) {
    if (any && p.f32_blocks) {
      update_lut8_small_kernel<PRE, G, true, true><<<grid, threads, sm, stream>>>(p);
      return;
    }
  }
  if (any)
    update_lut8_small_kernel<PRE, G, true, false><<<grid, threads, sm, stream>>>(p);
  else
    update_lut8_small_kernel<PRE, G, false, false><<<grid, threads, sm, stream>>>(p);
}

// Which updates the small kernel takes. Three and four groups only with the
// leading perturbation's probe in one of them, or none: words of its own
// would be a fifth Philox call's registers. (Its probe in another group than the
// last: 400 M bf16 weights, K = 16 / 24 / 32: 322 / 584 / 664 us with a call of its
// own or in the chunk kernel -> 284 / 362 / 448; in one flat buffer 475 / 753 / 827 ->
// 370 / 472 / 634; fp32 699 / 676 -> 495 / 571, but with four groups 754 -> 797, so
// those stay.) Views of fp32 make a block's words
// twice here, once per half, where the chunk kernel makes them once: with four
// groups that costs them more than the chunks' tables and barriers do (205 M
// fp32 weights in one flat buffer, K = 32: 0.450 ms here, 0.425 there; K = 24:
// 0.363 and 0.386). Before, K from 17 on walked the chunks: OPT-1.3B-shaped bf16
// set with the leading perturbation, K = 24 / 32: 1.612 / 1.857 -> 1.122 / 1.386
// ms; 400 M bf16 weights in one flat buffer 0.677 / 0.747 -> 0.451 / 0.584 ms.
bool lut8_small_takes(const UpdateParams& u, bool f32_blocks, bool f32_views) {
  if (u.packing != kPacking1 || u.groups > kSmallGroups || (u.groups == 4 && f32_views)) return false;
  const uint32_t groups = static_cast<uint32_t>(u.groups);
  if (u.groups <= 2 || !u.has_pre || u.pre.ctr2 + 1u == groups) return true;
  return u.pre.ctr2 < groups && !(u.groups == 4 && f32_blocks);
}

cudaError_t launch_update_lut8_small(SmallUpdateParams& p, bool any, int sms, cudaStream_t stream) {
  const UpdateParams& u = p.u;
  const uint32_t bhi = static_cast<uint32_t>(static_cast<uint64_t>(u.tab.blk_base) >> 32);
  for (uint32_t g = 0; g < static_cast<uint32_t>(kSmallGroups); ++g) p.g[g] = group_round01(g, bhi, u.keys);
  p.gp = group_round01(u.pre.ctr2, bhi, u.keys);
  const bool last = u.pre.ctr2 + 1u == static_cast<uint32_t>(u.groups);
  const bool group = !last && u.pre.ctr2 < static_cast<uint32_t>(u.groups);
  if (u.groups == 1)
    !u.has_pre ? launch_small_cfg<kPreNone, 1>(p, any, sms, stream)
    : last     ? launch_small_cfg<kPreTable, 1>(p, any, sms, stream)
               : launch_small_cfg<kPreOwn, 1>(p, any, sms, stream);
  else if (u.groups == 2)
    !u.has_pre ? launch_small_cfg<kPreNone, 2>(p, any, sms, stream)
    : last     ? launch_small_cfg<kPreTable, 2>(p, any, sms, stream)
    : group    ? launch_small_cfg<kPreGroup, 2>(p, any, sms, stream)
               : launch_small_cfg<kPreOwn, 2>(p, any, sms, stream);
  else if (u.groups == 3)
    !u.has_pre ? launch_small_cfg<kPreNone, 3>(p, any, sms, stream)
    : last     ? launch_small_cfg<kPreTable, 3>(p, any, sms, stream)
               : launch_small_cfg<kPreGroup, 3>(p, any, sms, stream);
  else
    !u.has_pre ? launch_small_cfg<kPreNone, 4>(p, any, sms, stream)
    : last     ? launch_small_cfg<kPreLast, 4>(p, any, sms, stream)
               : launch_small_cfg<kPreGroup, 4>(p, any, sms, stream);
  return cudaGetLastError();
}

cudaError_t launch_update_lut8(const UpdateParams& p, bool any, int sms, cudaStream_t stream) {
  const bool pack8 = p.packing == kPacking8;
  // a launch of one or two groups comes here when the small kernel cannot take it: rare, on the general form
  if (!one_high_word(p.tab) || (!pack8 && p.groups <= 2))
    return pack8 ? launch_lut8_cfg<false, true, true>(p, sms, stream)
                 : launch_lut8_cfg<false, true, false>(p, sms, stream);
  if (pack8) return launch_lut8_cfg<true, true, true>(p, sms, stream);
  if (any) return launch_lut8_cfg<true, true, false>(p, sms, stream);
  return p.groups >= kAheadGroups ? launch_lut8_cfg<true, false, false, true>(p, sms, stream)
                                  : launch_lut8_cfg<true, false, false>(p, sms, stream);
}

}  // namespace zo
