// zo_update_items.cu -- the fused K-probe update by 32-byte items: short lists,
// and most of packing 8.
//
// theta <- rn(fp32(theta) + sum_k a_k z_k[g]), the sums formed from the same
// 8-probe partials T_lo + T_hi in the same order as in zo_update_lut8.cu, so
// the bits are the same. What differs is what a launch costs before and after
// its lookups: the kernels there copy a group's 256-entry table once per lane
// (32 KB per group, for one lookup per element and group without bank
// conflicts), which short lists do not repay. Here a group's two 16-entry
// 4-probe tables lie in 128 bytes as they are: sixteen entries in sixteen
// banks, so lanes that read different ones do not conflict, and lanes that
// read the same one share it. Two lookups per element and group, nothing to
// copy, 128 threads to a CTA so that few items still reach every SM; one
// 32-byte item per thread, every kind of tensor in one launch
// (perturb_items_kernel). Bound by its chain of latencies: launch, table,
// coefficients, one Philox call and sixteen lookups per group, theta. 300 k
// bf16 weights in 12 tensors, K = 8 / 32 / 64 / 256: 10.5 / 13.5 / 17.0 / 34.5
// -> 8.7 / 8.2 / 8.8 / 15.1 us; as fp32, K = 32 15.0 -> 8.2; in one flat buffer
// 23.3 -> 8.6; packing 8, K = 32 14.5 -> 10.2 (calls back to back 5.5 / 6.0 / 6.2 /
// 12.3; 5.3; 6.4; 8.3). Not adopted: a grid of 8 to 64
// CTAs per SM that walks the items (K = 256, 8 M weights 97.5 -> 98-107 us).
//
// Packing 8 has eight Philox calls per group and is bound by them (85 to 90
// cycles per warp and call on an SM's quarter). A full group's calls are
// unrolled, several chains in flight per thread, and a thread of a long list
// takes several items. A leading perturbation whose probe is one of the last
// group's, as a step's restore has it, takes that group's words instead of a
// call of its own. 205 M bf16 weights, K = 4 / 8 / 16, without / with it: 249 /
// 315 / 562 and 284 / 346 / 593 us (a persistent grid with plain Philox calls
// took 312 / 312 / 564 and 380 / 379 / 632; a call of its own 313 / 377 / 627);
// 60 M, K = 24: 245 and 255 (247 and 268; 264). Not adopted: the calls in twos
// or fours (K = 8 445 / 432 us), registers capped at 40 for more warps (spills;
// 409), CTAs of 256 threads (406), the counters' group parts computed instead of
// read (60 M, K = 8 99 -> 105).
//
// Aligned fp32 is taken by whole blocks, two items of a lane at a time (an
// instantiation of its own, 88 registers), so that a block's words are made
// once, its calls' bits folded where the lookups take them (16-bit items would
// pay for that when they are views: 100 M, K = 24 426 -> 438). 205 M fp32
// weights, K = 4 / 8 / 16, without / with the leading perturbation: 278 / 322 /
// 562 and 296 / 348 / 591 us (the persistent grid: 321 / 322 / 562 and 364 / 364 /
// 610). Not adopted there: 76 registers, six CTAs to an SM (K = 16 580), theta
// loaded after the calls (100 M, K = 8 164 -> 177).
#include "zo_device.cuh"
#include "zo_launch.h"

namespace zo {

namespace {

constexpr int kItemThreads = 128;
constexpr uint32_t kFrame = 256;  // bytes from one group's tables to the next's: T_lo at 0, T_hi at 64

__device__ __forceinline__ float lds_f32_hi(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1+64];" : "=f"(v) : "r"(addr));
  return v;
}

__device__ __forceinline__ uint4 shift_left(const uint4& x, uint32_t n) {
  return make_uint4(x.x << n, x.y << n, x.z << n, x.w << n);
}

// Add a group's partial of elements 4 M .. 4 M + 3: their bytes of lo4 and hi4 hold four times the signs of the
// group's probes 0-3 and 4-7.
template <int M>
__device__ __forceinline__ void add_word(float (&acc)[16], uint32_t lo4, uint32_t hi4, uint32_t frame) {
#pragma unroll
  for (int j = 0; j < 4; j += 2) {
    const uint32_t s0 = 0x7650u | static_cast<uint32_t>(j), s1 = s0 + 1u;
    float p0 = lds_f32(__byte_perm(lo4, frame, s0)), p1 = lds_f32(__byte_perm(lo4, frame, s1));
    fadd2_rn(p0, p1, lds_f32_hi(__byte_perm(hi4, frame, s0)), lds_f32_hi(__byte_perm(hi4, frame, s1)));
    fadd2_rn(acc[4 * M + j], acc[4 * M + j + 1], p0, p1);
  }
}

// The same of the first WORDS words of sign bytes.
template <int WORDS>
__device__ __forceinline__ void add_group(float (&acc)[16], const uint4& x, uint32_t frame) {
  add_word<0>(acc, (x.x << 2) & 0x3C3C3C3Cu, (x.x >> 2) & 0x3C3C3C3Cu, frame);
  add_word<1>(acc, (x.y << 2) & 0x3C3C3C3Cu, (x.y >> 2) & 0x3C3C3C3Cu, frame);
  if (WORDS == 2) return;
  add_word<2>(acc, (x.z << 2) & 0x3C3C3C3Cu, (x.z >> 2) & 0x3C3C3C3Cu, frame);
  add_word<3>(acc, (x.w << 2) & 0x3C3C3C3Cu, (x.w >> 2) & 0x3C3C3C3Cu, frame);
}

size_t update_items_smem_bytes(int groups, int packing) {
  // a_k, the tables on a 256-byte boundary, the counters' group parts
  return static_cast<size_t>(groups) * (32 + kFrame + 16 * (packing == kPacking8 ? 8 : 1)) + kFrame;
}

}  // namespace

// What a launch holds: packing 1, packing 8, packing 8 and mostly fp32 on the 32-byte grid, or packing 1 with at most
// two groups on more CTAs than 7 per SM.
constexpr int kPlain = 0, kBytes = 1, kBytesF32 = 2, kPlainMany = 3;

// LAST: packing 8, the leading perturbation's probe is one of the last group's, whose words it takes. The second launch
// bound leaves a group's calls and lookups the registers that they are interleaved with: 5 CTAs of kBytesF32, 7 of
// kPlain (70 registers). Without it kPlain takes 56 and holds 9 CTAs, us: 24 tensors, 2 M bf16 weights, K = 16 / 96 /
// 520 5.8 / 13.3 / 55.7, with it 5.7 / 13.0 / 54.3; 0.03 M, K = 520 23.5, with it 18.0. Only a second wave costs more
// where little is left to interleave, 3 M bf16 weights, K = 8 / 16: 6.2 / 7.1 in place of kPlainMany's 5.8 / 6.9.
template <int KIND, bool LAST, int N>
__global__ void __launch_bounds__(kItemThreads, KIND == kPlain ? 7 : KIND == kBytesF32 ? 5 : 0) update_items_kernel(const __grid_constant__ UpdateItemsParams<N> P) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int skip_s;
  constexpr bool PACK8 = KIND == kBytes || KIND == kBytesF32, WIDE = KIND == kBytesF32;
  const int G = P.groups;
  constexpr int kCalls = PACK8 ? 8 : 1;  // Philox calls per group
  uint4* r01_s = reinterpret_cast<uint4*>(smem);            // kCalls G group parts
  float* a_s = reinterpret_cast<float*>(r01_s + kCalls * G);  // 8 G coefficients
  const uint32_t after = static_cast<uint32_t>(__cvta_generic_to_shared(a_s + 8 * G));
  const uint32_t frame0 = (after + kFrame - 1u) & ~(kFrame - 1u);
  float* lut = a_s + 8 * G + (frame0 - after) / 4u;
  if (threadIdx.x == 0) skip_s = (P.status != nullptr && *P.status != 0);
  for (int k = threadIdx.x; k < 8 * G; k += kItemThreads)
    a_s[k] = k < P.K ? __double2float_rn(P.coef_mul * P.coef[k]) : 0.0f;
  for (int k = threadIdx.x; k < kCalls * G; k += kItemThreads) {
    const GroupRound01 g = group_round01(static_cast<uint32_t>(k), P.bhi, P.keys);
    r01_s[k] = make_uint4(g.x0, g.x2, g.lpa1, 0u);
  }
  // this thread's item, its load on the way while the tables are made
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t left = PACK8 ? P.rounds : 1u;  // a warp's items are consecutive
  uint32_t b = (blockIdx.x * (kItemThreads / 32u) + (threadIdx.x >> 5)) * 32u * left + lane;
  bool here = false;  // the same in all lanes
  ItemsEntry e;
  uint8_t dt = 0;
  bool f32 = false, shift = false;
  uint32_t a = 0;
  ItemPlace k;
  char* p = nullptr;
  uint32_t v[8], v2[8];
  bool pairs = WIDE;
  bool wide = false;  // WIDE: lane l takes items 2 l and 2 l + 1 of the next 64, an fp32 block (the same in all lanes)
  const auto seek = [&] {
    const uint32_t wb = b - lane;
    here = wb < P.total;
    int t = here ? P.hint[wb >> P.hint_shift] : 0;
    while (here && wb >= P.e[t].end) ++t;
    e = P.e[t];
    dt = static_cast<uint8_t>(e.meta & kDtypeMask);
    f32 = dt == kF32;
    shift = (e.meta & kShift) != 0;
    a = e.meta >> 16;
    wide = pairs && here && f32 && !shift && left >= 2u && wb - e.begin + 64u <= e.whole;
    k = item_place(e, wide ? b + lane : b);
    k.full = k.full && here;
    k.act = k.act && here;
    p = reinterpret_cast<char*>(e.base) + static_cast<int64_t>(k.i) * 32;
    if (k.full) ld256(p, v);
    if (WIDE && wide) ld256(p + 32, v2);
  };
  seek();
  __syncthreads();
  const bool do_sum = skip_s == 0;  // a failed preconditioner still gets the leading perturbation
  if (!do_sum && !P.has_pre) return;
  if (WIDE && !do_sum) {  // element by element, below
    pairs = false;
    seek();
  }
  for (int i = threadIdx.x; i < 32 * G; i += kItemThreads) {
    const int h = i >> 4;  // quad of probes
    lut[(h >> 1) * (kFrame / 4) + (h & 1) * 16 + (i & 15)] = quad_partial(a_s + 4 * h, static_cast<uint32_t>(i) & 15u);
  }
  __syncthreads();
  if (!here) return;
  const auto item = [&] {
    const BlockRound01 blk = block_round01(static_cast<uint32_t>(item_block(e, k.i)), P.keys);
    const auto call = [&](uint32_t c) {
      const uint4 r = r01_s[c];
      return philox_finish(philox_start(blk, {r.x, r.y, r.z}), P.keys);
    };
    const auto own = [&](const uint4& x) { return item_signs(x, f32, (k.i & 1) != 0, shift, a); };
    uint4 last = make_uint4(0u, 0u, 0u, 0u);  // LAST: the last group's sign bytes
    float acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.0f;
    if (do_sum) {
      uint32_t frame = frame0;
      uint4 lo, hi;  // WIDE: the bits of probes 0-3 and 4-7, where the lookups take them
#pragma unroll 1
      for (int q = 0; q < G; ++q, frame += kFrame) {
        uint4 x = make_uint4(0u, 0u, 0u, 0u);  // the sign bytes of this lane's elements
        if constexpr (WIDE) {
          lo = hi = x;
          if (8 * q + 8 <= P.K) {
#pragma unroll
            for (int i = 0; i < 8; ++i) fold_bits(i < 4 ? lo : hi, call(static_cast<uint32_t>(8 * q + i)), i & 3);
          } else {
#pragma unroll 1
            for (int i = 0; i < 4 && 8 * q + i < P.K; ++i) fold_bits(lo, call(static_cast<uint32_t>(8 * q + i)), i);
#pragma unroll 1
            for (int i = 4; i < 8 && 8 * q + i < P.K; ++i) fold_bits(hi, call(static_cast<uint32_t>(8 * q + i)), i & 3);
          }
          if (!wide) x = make_uint4(lo.x + (hi.x << 4), lo.y + (hi.y << 4), lo.z + (hi.z << 4), lo.w + (hi.w << 4));
          if (wide) {
            lo = shift_left(lo, 2u);
            hi = shift_left(hi, 2u);
            add_word<0>(acc, lo.x, hi.x, frame);
            add_word<1>(acc, lo.y, hi.y, frame);
            add_word<2>(acc, lo.z, hi.z, frame);
            add_word<3>(acc, lo.w, hi.w, frame);
          }
        } else if constexpr (PACK8) {
          if (8 * q + 8 <= P.K) {
#pragma unroll
            for (int i = 0; i < 8; ++i) fold_bits(x, call(static_cast<uint32_t>(8 * q + i)), i);
          } else {
#pragma unroll 2
            for (int i = 0; i < 8 && 8 * q + i < P.K; ++i) fold_bits(x, call(static_cast<uint32_t>(8 * q + i)), i);
          }
        } else {
          x = call(static_cast<uint32_t>(q));
        }
        if (!(WIDE && wide)) {
          x = own(x);
          if (f32)
            add_group<2>(acc, x, frame);
          else
            add_group<4>(acc, x, frame);
        }
        if (LAST && !(WIDE && wide)) last = x;
      }
      if constexpr (LAST && WIDE) {
        if (wide)  // both were shifted for the lookups
          last = make_uint4((lo.x >> 2) + (hi.x << 2), (lo.y >> 2) + (hi.y << 2), (lo.z >> 2) + (hi.z << 2), (lo.w >> 2) + (hi.w << 2));
      }
    }
    uint4 xp = last;
    if (P.has_pre && !(LAST && do_sum)) {
      const GroupRound01 g = group_round01(P.pre.ctr2, P.bhi, P.keys);
      xp = philox_finish(philox_start(blk, g), P.keys);
      if (LAST) xp = shift_left(xp, P.pre.bit);
      if (!(WIDE && wide)) xp = own(xp);
    }
    if (!k.act) return;
    if (k.full && do_sum) {
      if (f32) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float th = __uint_as_float(v[i]);
          if (P.has_pre) th = add_signed(th, xp, i, P.pre);
          v[i] = __float_as_uint(__fadd_rn(th, acc[i]));
        }
        if (WIDE && wide) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float th = __uint_as_float(v2[i]);
            if (P.has_pre) th = add_signed(th, xp, 8 + i, P.pre);
            v2[i] = __float_as_uint(__fadd_rn(th, acc[8 + i]));
          }
          st256(p + 32, v2);
        }
      } else if (dt == kBF16) {
        update_regs16<kBF16>(v, acc, xp, P.has_pre, P.pre);
      } else {
        update_regs16<kF16>(v, acc, xp, P.has_pre, P.pre);
      }
      st256(p, v);
      return;
    }
    // an item across a tensor's end, or the leading perturbation alone
    int lo, hi;
    item_range(e, k.i, &lo, &hi);
    float th[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) th[i] = i >= lo && i < hi ? load_elem(p, dt, i) : 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (i < lo || i >= hi) continue;
      if (P.has_pre) th[i] = round_to_storage(dt, add_signed(th[i], xp, i, P.pre));
      if (do_sum) th[i] = __fadd_rn(th[i], acc[i]);
      store_elem(p, dt, i, th[i]);
    }
  };
  if constexpr (PACK8) {
    while (here) {
      item();
      const uint32_t took = WIDE && wide ? 2u : 1u;
      left -= took;
      if (left == 0u) break;
      b += 32u * took;
      seek();
    }
  } else {
    item();
  }
}

template <int N>
cudaError_t launch_update_items(const UpdateItemsParams<N>& p, int sms, cudaStream_t stream) {
  const uint32_t per = kItemThreads * (p.packing == kPacking8 ? p.rounds : 1u);
  const int grid = static_cast<int>((static_cast<uint64_t>(p.total) + (per - 1u)) / per);
  const size_t smem = update_items_smem_bytes(p.groups, p.packing);
  const auto go = [&](auto kernel) -> cudaError_t {
    if (smem > 48 * 1024) {
      const cudaError_t e = cudaFuncSetAttribute(
          kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(update_items_smem_bytes(kMaxGroups, kPacking8)));
      if (e != cudaSuccess) return e;
    }
    kernel<<<grid, kItemThreads, smem, stream>>>(p);
    return cudaGetLastError();
  };
  if (p.packing != kPacking8)
    return p.groups <= 2 && grid > 7 * sms ? go(update_items_kernel<kPlainMany, false, N>) : go(update_items_kernel<kPlain, false, N>);
  if (p.pre_last != 0)
    return p.f32_blocks ? go(update_items_kernel<kBytesF32, true, N>) : go(update_items_kernel<kBytes, true, N>);
  return p.f32_blocks ? go(update_items_kernel<kBytesF32, false, N>) : go(update_items_kernel<kBytes, false, N>);
}
template cudaError_t launch_update_items(const UpdateItemsParams<kItemsFew>& p, int sms, cudaStream_t stream);
template cudaError_t launch_update_items(const UpdateItemsParams<kItemsSome>& p, int sms, cudaStream_t stream);
template cudaError_t launch_update_items(const UpdateItemsParams<kItemsMany>& p, int sms, cudaStream_t stream);

}  // namespace zo
