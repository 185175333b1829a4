// zo_quad_step.cu -- every forward point of one step of the small quadratic
// workload in one launch (zo_quadratic_points).
//
// Algorithm 1 with f(theta) = 1/2 sum a_i theta_i^2 as the forward pass: the
// clean loss, then per probe theta <- rn(theta + eps z_k) and its loss,
// theta <- rn(theta - 2 eps z_k) and its loss, theta <- rn(theta + eps z_k).
// A weight's chain of perturbations depends on no other weight and on no
// loss, so a thread takes its weights through all 2 K + 1 points in registers
// (theta and a are read once, theta written once) and only the 2 K + 1 sums
// cross threads.
//
// Bound: fp32 arithmetic (seven packed operations per weight and point, below,
// and an addition and a sign flip per weight and move) and the grid's size; d =
// 2^20 and K = 8 are 17.8 M terms.
//
// Sums. Each term a t^2 is formed without rounding as a pair of fp32 values
// (Dekker's product by fused multiply-add: a t = p + pe, p t = q + qe, term =
// q + fma(pe, t, qe)) and summed into an fp32 pair with Knuth's two-sum, two
// weights per packed fp32x2 operation. The products are exact while a stays
// in [2^-40, 2^40] or 0 and |t| in [2^-30, 2^30] in magnitude; a thread whose
// eight weights leave that range at a point (zeros, infinities, tiny or huge
// weights) redoes the point weight by weight, adding terms whose products
// leave the exact range in fp64. NaN needs no such care: it reaches the sum
// either way.
//
// Reduction. A thread ends four probes with eight pairs, which a warp's
// butterfly folds by halving the values as it doubles the lanes (9 exchanges
// for the 8 values; a tree for each would be 40). From the warp on, over its
// rounds in shared memory and over the CTA's warps, eight lanes to a point, a
// sum is three fp32 values that carry the pairs' rounding errors: two alone put
// a loss 1.6 times as far from the exact sum as a launch per point does, whose
// sums are fp64 from the warp on (root mean square over 60 losses 1.9e-16, 1.2e-16
// so and there); fp64 here took the slow pipe 2 us (d = 2^20, K = 8: 31 -> 33).
// The CTA that finishes last (a ticket counter in the workspace, reset by that
// CTA) folds the CTAs' fp64 partials in index order and writes the loss table.
// No CTA waits for another; for a given size every order is fixed, so the
// losses are bit-reproducible.
#include <type_traits>

#include "zo_device.cuh"
#include "zo_launch.h"
#include "zo_precond.cuh"

namespace zo {

namespace {

constexpr int kItem = 8;            // weights per thread and round: half a Philox block
constexpr int kPointsMaxThreads = 896;

struct f2 {  // two fp32 values in one 64-bit register
  unsigned long long v;
};
__device__ __forceinline__ f2 pack_f2(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack_f2(f2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

struct Ds {  // s + l, an unevaluated fp32 pair
  float s, l;
};

// a + b by Knuth's two-sum of the high parts.
__device__ __forceinline__ Ds ds_sum(Ds a, Ds b) {
  const float s = __fadd_rn(a.s, b.s);
  const float bb = __fsub_rn(s, a.s);
  const float e = __fadd_rn(__fsub_rn(a.s, __fsub_rn(s, bb)), __fsub_rn(b.s, bb));
  return {s, __fadd_rn(a.l, __fadd_rn(e, b.l))};
}

// x <- fl(x + y); its rounding error.
__device__ __forceinline__ float two_sum(float& x, float y) {
  const float s = __fadd_rn(x, y);
  const float bb = __fsub_rn(s, x);
  const float e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)), __fsub_rn(y, bb));
  x = s;
  return e;
}

struct Ts {  // s + l + m
  float s, l, m;
};

// a + b, the errors of the first two parts' sums kept.
__device__ __forceinline__ Ts ts_sum(Ts a, Ts b) {
  const float e = two_sum(a.s, b.s);
  const float f = two_sum(a.l, b.l);
  const float g = two_sum(a.l, e);
  a.m = __fadd_rn(__fadd_rn(a.m, b.m), __fadd_rn(f, g));
  return a;
}

constexpr float kMinA = 0x1p-40f, kMaxA = 0x1p40f, kMinT = 0x1p-30f, kMaxT = 0x1p30f;

// The eight terms of one point as a pair; with CHECK, *ok: every |t| in [kMinT,
// kMaxT]. na = -a: the error of a product by one fused multiply-add needs the
// product's negative, so p and -p are both formed, and the errors come out
// negated (u = p - a t, w = q - p t, a term's low part is -(u t + w)). q is the
// rounded product p t + 0, with a zero that the compiler cannot see: a packed
// multiply whose result is only added is fused with those additions (ptxas
// does so in spite of .rn), and the sums then lose q's rounding error twice
// over.
template <bool CHECK>
__device__ __forceinline__ Ds point_terms(const f2 (&t)[kItem / 2], const f2 (&a)[kItem / 2], const f2 (&na)[kItem / 2],
                                          f2 zero, bool* ok) {
  f2 s, l;
  float mx = 0.0f, mn = 1.0f;
#pragma unroll
  for (int i = 0; i < kItem / 2; ++i) {
    if (CHECK) {
      const float2 tv = unpack_f2(t[i]);
      mx = fmaxf(mx, fmaxf(fabsf(tv.x), fabsf(tv.y)));
      mn = fminf(mn, fminf(fabsf(tv.x), fabsf(tv.y)));
    }
    const f2 p = mul2(a[i], t[i]);
    const f2 np = mul2(na[i], t[i]);
    const f2 u = fma2(na[i], t[i], p);
    const f2 q = fma2(p, t[i], zero);
    const f2 r = fma2(u, t[i], fma2(np, t[i], q));  // minus the low part
    if (i == 0) {
      s = q;
      l = sub2(zero, r);
    } else {
      const f2 sn = add2(s, q);
      const f2 bb = sub2(sn, s);
      const f2 e = add2(sub2(s, sub2(sn, bb)), sub2(q, bb));
      l = add2(l, sub2(e, r));
      s = sn;
    }
  }
  *ok = !CHECK || (mx <= kMaxT && mn >= kMinT);
  const float2 sv = unpack_f2(s), lv = unpack_f2(l);
  return ds_sum({sv.x, lv.x}, {sv.y, lv.y});
}

// The same weight by weight: terms whose products leave the exact range (or
// are not finite) go to *wide in fp64. cnt weights of the item exist.
__device__ __noinline__ Ds point_terms_any(const f2 (&t)[kItem / 2], const f2 (&a)[kItem / 2], int cnt, double* wide) {
  Ds sum = {0.0f, 0.0f};
  double w = 0.0;
  for (int i = 0; i < cnt; ++i) {
    const float2 tp = unpack_f2(t[i >> 1]), ap = unpack_f2(a[i >> 1]);
    const float tv = (i & 1) ? tp.y : tp.x, av = (i & 1) ? ap.y : ap.x;
    const float p = __fmul_rn(av, tv);
    const float pe = __fmaf_rn(av, tv, -p);
    const float q = __fmul_rn(p, tv);
    const float qe = __fmaf_rn(p, tv, -q);
    const float mp = fabsf(p), mq = fabsf(q);
    if (mp >= 0x1p-100f && mp < 0x1p100f && mq >= 0x1p-100f && mq < 0x1p100f) {
      sum = ds_sum(sum, {q, __fmaf_rn(pe, tv, qe)});
    } else {
      const double td = tv;
      w = __dadd_rn(w, __dmul_rn(static_cast<double>(av), __dmul_rn(td, td)));
    }
  }
  *wide = w;
  return sum;
}

// The coefficient of one probe as zo_precondition forms it (alpha = 0.1,
// lambda_reg = 1, two-sided); false when a loss, the curvature or it is not
// finite. Not inlined: pow would take registers from the loop over the probes.
__device__ __noinline__ bool probe_coefficient(double lp, double lm, double l0, double eps, double* c) {
  const double cv = probe_curvature(lp, lm, l0, eps);
  *c = __dmul_rn(probe_weight(cv, 0.1, 1.0), central_difference(lp, lm, eps));
  return isfinite(lp) && isfinite(lm) && isfinite(l0) && isfinite(cv) && isfinite(*c);
}

// Sum over a warp, fp64 (fixed tree), in every lane.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
  return v;
}

__device__ __forceinline__ Ds shfl_xor_ds(Ds a, int off) {
  return {__shfl_xor_sync(0xFFFFFFFFu, a.s, off), __shfl_xor_sync(0xFFFFFFFFu, a.l, off)};
}

// Fold eight values over a warp: lane l ends with the sum over all lanes of
// value l >> 2 (the lanes of a quad hold it up to the order of the last adds).
__device__ __forceinline__ Ds butterfly8(Ds (&v)[8], int lane) {
#pragma unroll
  for (int step = 0; step < 3; ++step) {
    const int off = 16 >> step, half = 4 >> step;
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const Ds keep = hi ? v[i + half] : v[i], send = hi ? v[i] : v[i + half];
      v[i] = ds_sum(keep, shfl_xor_ds(send, off));
    }
  }
  Ds r = v[0];
  r = ds_sum(r, shfl_xor_ds(r, 2));
  return ds_sum(r, shfl_xor_ds(r, 1));
}

}  // namespace

// Shared memory per warp: the sums' fp32 values (in launches of several rounds
// a third one, below 2^-46 of the first, as bf16) and fp64 parts of 16 points per
// group of 8 probes, then of the clean loss (slot 16 G).
size_t quad_points_smem_bytes(int groups, int warps, bool several) {
  return static_cast<size_t>(warps) * (16u * static_cast<size_t>(groups) + 1u) * (several ? 18u : 16u);
}

struct QuadPointsParams {
  float* theta;
  const float* a;
  int64_t n;
  RoundKeys keys;
  int32_t K, groups;
  uint32_t neps_bits;    // -fp32(eps)
  uint32_t nmeps_bits;   // -fp32(-2 eps)
  double* losses;        // K rows (L+, L-, L0)
  double* partial;       // (2 K + 1) x gridDim.x
  uint32_t* ticket;      // zero before the launch; the last CTA zeroes it again
  float zero;            // 0.0f
  float drift;           // (K + 1) 2^-21
  int32_t several;       // rounds
  double eps;            // for the coefficients
  double* c;             // K coefficients and their status, or null
  int32_t* status;
};

template <bool PACK8, bool VEC>
__global__ void __launch_bounds__(kPointsMaxThreads, 1) quad_points_kernel(const __grid_constant__ QuadPointsParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ bool last_s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int slots = 16 * P.groups + 1;
  double* wide_s = reinterpret_cast<double*>(smem);                     // [slots][warps]
  float2* pair_s = reinterpret_cast<float2*>(wide_s + slots * warps);   // [slots][warps]
  __nv_bfloat16* third_s = reinterpret_cast<__nv_bfloat16*>(pair_s + slots * warps);  // [slots][warps]
  for (int i = threadIdx.x; i < slots * warps; i += blockDim.x) {
    wide_s[i] = 0.0;
    pair_s[i] = make_float2(0.0f, 0.0f);
    if (P.several) third_s[i] = __float2bfloat16_rn(0.0f);
  }
  __syncthreads();

  // The terms of one point of this thread's weights, redone weight by weight
  // where a lane's leave the exact range; fp64 parts to the warp's slot.
  const f2 zero = pack_f2(P.zero, P.zero);
  bool a_ok = true;
  int cnt = 0;
  f2 t[kItem / 2], a[kItem / 2], na[kItem / 2];
  const auto point = [&](auto check, int slot) -> Ds {
    bool ok;
    Ds r = point_terms<decltype(check)::value>(t, a, na, zero, &ok);
    if constexpr (decltype(check)::value) {
      ok = ok && a_ok;
      if (__any_sync(0xFFFFFFFFu, !ok)) {
        double w = 0.0;
        if (!ok) r = point_terms_any(t, a, cnt, &w);
        if (__any_sync(0xFFFFFFFFu, w != 0.0)) {
          w = warp_sum(w);
          if (lane == 0) wide_s[slot * warps + warp] = __dadd_rn(wide_s[slot * warps + warp], w);
        }
      }
    }
    return r;
  };
  bool again = false;  // not the warp's first round
  const auto store_sum = [&](int slot, Ds v) {
    float2& c = pair_s[slot * warps + warp];
    if (!again) {
      c = make_float2(v.s, v.l);
      return;
    }
    __nv_bfloat16& m = third_s[slot * warps + warp];
    const Ts r = ts_sum({c.x, c.y, __bfloat162float(m)}, {v.s, v.l, 0.0f});
    c = make_float2(r.s, r.l);
    m = __float2bfloat16_rn(r.m);
  };

  const int64_t items = (P.n + kItem - 1) / kItem;
  // warps take 32 items each, first one per CTA, then a second, ..: few items still use every SM
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t base = (static_cast<int64_t>(warp) * gridDim.x + blockIdx.x) * 32; base < items; base += stride) {
    const int64_t item = base + lane;
    const int64_t e0 = item * kItem;
    cnt = static_cast<int>(max(static_cast<int64_t>(0), min(static_cast<int64_t>(kItem), P.n - e0)));
    if (VEC && cnt == kItem) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float4 x = reinterpret_cast<const float4*>(P.theta + e0)[j];
        const float4 y = reinterpret_cast<const float4*>(P.a + e0)[j];
        t[2 * j] = pack_f2(x.x, x.y);
        t[2 * j + 1] = pack_f2(x.z, x.w);
        a[2 * j] = pack_f2(y.x, y.y);
        a[2 * j + 1] = pack_f2(y.z, y.w);
      }
    } else {
#pragma unroll
      for (int i = 0; i < kItem / 2; ++i) {
        // past the end: a = 0, whose terms are exact zeros
        t[i] = pack_f2(2 * i < cnt ? P.theta[e0 + 2 * i] : 1.0f, 2 * i + 1 < cnt ? P.theta[e0 + 2 * i + 1] : 1.0f);
        a[i] = pack_f2(2 * i < cnt ? P.a[e0 + 2 * i] : 0.0f, 2 * i + 1 < cnt ? P.a[e0 + 2 * i + 1] : 0.0f);
      }
    }
    a_ok = true;
#pragma unroll
    for (int i = 0; i < kItem / 2; ++i) {
      const float2 y = unpack_f2(a[i]);
      na[i] = pack_f2(-y.x, -y.y);
      const float ax = fabsf(y.x), ay = fabsf(y.y);
      a_ok = a_ok && (ax >= kMinA || ax == 0.0f) && ax <= kMaxA && (ay >= kMinA || ay == 0.0f) && ay <= kMaxA;
    }
    Ds clean = point(std::true_type(), 16 * P.groups);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) clean = ds_sum(clean, shfl_xor_ds(clean, off));
    Ds mine = {0.0f, 0.0f};
    const int64_t b = item >> 1;
    const bool upper = (item & 1) != 0;  // words 2, 3 of the block's Philox output
    uint32_t w0 = 0, w1 = 0;
    const auto probes = [&](auto check) {
#pragma unroll 1
    for (int h = 0; 4 * h < P.K; ++h) {  // four probes at a time
      Ds v[8];
      if (!PACK8 && (h & 1) == 0) {
        const uint4 x = block_bits(b, static_cast<uint32_t>(h >> 1), P.keys);
        w0 = upper ? x.z : x.x;
        w1 = upper ? x.w : x.y;
      }
      // packing 1: the probe's bit of every byte moved to the byte's bit 7
      const uint32_t up = PACK8 ? 0u : ((h & 1) ? 0u : 4u);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[2 * j] = {0.0f, 0.0f};
        v[2 * j + 1] = {0.0f, 0.0f};
        const int k = 4 * h + j;
        if (k >= P.K) continue;
        uint32_t u0, u1;  // sign bit of weight i at bit 7 of byte i
        if (PACK8) {
          const uint4 x = block_bits(b, static_cast<uint32_t>(k), P.keys);
          u0 = (upper ? x.z : x.x) << 7;
          u1 = (upper ? x.w : x.y) << 7;
        } else {
          u0 = (w0 << up) << (3 - j);
          u1 = (w1 << up) << (3 - j);
        }
        // scalar adds, as every fp32 perturbation (the same NaN encoding)
        float d[kItem];
#pragma unroll
        for (int i = 0; i < kItem; ++i)
          d[i] = __uint_as_float(P.neps_bits ^ (((i < 4 ? u0 : u1) << (24 - 8 * (i & 3))) & 0x80000000u));
        const auto move = [&](uint32_t flip) {
#pragma unroll
          for (int i = 0; i < kItem / 2; ++i) {
            const float2 x = unpack_f2(t[i]);
            t[i] = pack_f2(__fadd_rn(x.x, __uint_as_float(__float_as_uint(d[2 * i]) ^ flip)),
                           __fadd_rn(x.y, __uint_as_float(__float_as_uint(d[2 * i + 1]) ^ flip)));
          }
        };
        move(0u);
        v[2 * j] = point(check, 16 * (k >> 3) + 2 * (k & 7));
        move(P.neps_bits ^ P.nmeps_bits);
        v[2 * j + 1] = point(check, 16 * (k >> 3) + 2 * (k & 7) + 1);
        move(0u);
      }
      // of eight probes' sums, lanes 4 i take the first four's, lanes 4 i + 1 the others', and with the last ones
      // lane 2 the clean loss: one store
      const Ds r = butterfly8(v, lane);
      if ((lane & 3) == (h & 1)) mine = r;
      const bool last = 4 * (h + 1) >= P.K;
      if ((h & 1) != 0 || last) {
        const bool c = last && lane == 2;
        if (c) mine = clean;
        if ((lane & 3) <= (h & 1) || c) store_sum(c ? 16 * P.groups : 8 * ((h & ~1) + (lane & 3)) + (lane >> 2), mine);
      }
    }
    };
    // The points lie at theta +- eps up to the restores' drift (three roundings
    // per probe, each at most 2^-24 of |theta| + 2 eps). Far enough from 0 for
    // all of them, no point needs a check of its own.
    bool far_ok = a_ok;
    const float eps = fabsf(__uint_as_float(P.neps_bits)), drift = P.drift;
#pragma unroll
    for (int i = 0; i < kItem / 2; ++i) {
      const float2 x = unpack_f2(t[i]);
      const float mx = fabsf(x.x) + 2.0f * eps, my = fabsf(x.y) + 2.0f * eps;
      far_ok = far_ok && fabsf(fabsf(x.x) - eps) >= fmaf(drift, mx, 2.0f * kMinT) && mx <= 0.5f * kMaxT &&
               fabsf(fabsf(x.y) - eps) >= fmaf(drift, my, 2.0f * kMinT) && my <= 0.5f * kMaxT;
    }
    if (__any_sync(0xFFFFFFFFu, !far_ok))
      probes(std::true_type());
    else
      probes(std::false_type());
    again = true;
    if (VEC && cnt == kItem) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 x = unpack_f2(t[2 * j]), y = unpack_f2(t[2 * j + 1]);
        reinterpret_cast<float4*>(P.theta + e0)[j] = make_float4(x.x, x.y, y.x, y.y);
      }
    } else {
#pragma unroll
      for (int i = 0; i < kItem / 2; ++i) {
        const float2 x = unpack_f2(t[i]);
        if (2 * i < cnt) P.theta[e0 + 2 * i] = x.x;
        if (2 * i + 1 < cnt) P.theta[e0 + 2 * i + 1] = x.y;
      }
    }
  }
  __syncthreads();
  // the CTA's sums: of each eight lanes, lane i takes warps i, i + 8, .., then a fixed tree over the lanes (rolled: a
  // launch this short waits for every line of code)
  const int points = 2 * P.K + 1;
  for (int p0 = 4 * warp; p0 < points; p0 += 4 * warps) {
    const int p = p0 + (lane >> 3), row = (p == 2 * P.K ? 16 * P.groups : p) * warps;
    Ts r = {0.0f, 0.0f, 0.0f};
    double w = 0.0;
#pragma unroll 1
    for (int i = lane & 7; p < points && i < warps; i += 8) {
      r = ts_sum(r, {pair_s[row + i].x, pair_s[row + i].y, P.several ? __bfloat162float(third_s[row + i]) : 0.0f});
      const double x = wide_s[row + i];
      if (__double_as_longlong(x) != 0) w = __dadd_rn(w, x);
    }
#pragma unroll 1
    for (int off = 4; off > 0; off >>= 1)
      r = ts_sum(r, {__shfl_xor_sync(0xFFFFFFFFu, r.s, off), __shfl_xor_sync(0xFFFFFFFFu, r.l, off),
                     __shfl_xor_sync(0xFFFFFFFFu, r.m, off)});
    const bool any_wide = __any_sync(0xFFFFFFFFu, __double_as_longlong(w) != 0);
#pragma unroll 1
    for (int off = any_wide ? 4 : 0; off > 0; off >>= 1) w = __dadd_rn(w, __shfl_xor_sync(0xFFFFFFFFu, w, off));
    if (p < points && (lane & 7) == 0) {
      double sum = __dadd_rn(static_cast<double>(r.s), __dadd_rn(static_cast<double>(r.l), static_cast<double>(r.m)));
      if (any_wide) sum = __dadd_rn(sum, w);
      P.partial[static_cast<int64_t>(p) * gridDim.x + blockIdx.x] = sum;
    }
  }
  __threadfence();  // the partials are visible before the ticket counts them
  __syncthreads();
  if (threadIdx.x == 0) last_s = atomicAdd(P.ticket, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  double* loss_s = reinterpret_cast<double*>(smem);  // the warps' sums are done with: 2 K + 1 losses, K coefficients
  double* c_s = loss_s + points;
  for (int p = warp; p < points; p += warps) {
    const double* row = P.partial + static_cast<int64_t>(p) * gridDim.x;
    double s = 0.0;
    for (int i = lane; i < static_cast<int>(gridDim.x); i += 32) s = __dadd_rn(s, __ldcg(row + i));
    const double f = __dmul_rn(0.5, warp_sum(s));
    if (p == 2 * P.K) {
      for (int k = lane; k < P.K; k += 32) P.losses[3 * k + 2] = f;
    } else if (lane == 0) {
      P.losses[3 * (p >> 1) + (p & 1)] = f;
    }
    if (lane == 0) loss_s[p] = f;
  }
  if (P.c != nullptr) {
    __syncthreads();
    bool bad = false;
    for (int k = threadIdx.x; k < P.K; k += blockDim.x) {
      double ck;
      bad = !probe_coefficient(loss_s[2 * k], loss_s[2 * k + 1], loss_s[2 * P.K], P.eps, &ck) || bad;
      c_s[k] = ck;
    }
    bad = __syncthreads_or(bad);  // one bad probe: nothing but the status is written
    if (threadIdx.x == 0) *P.status = bad ? static_cast<int32_t>(kStatusNonFinite) : 0;
    for (int k = threadIdx.x; !bad && k < P.K; k += blockDim.x) P.c[k] = c_s[k];
  }
  if (threadIdx.x == 0) *P.ticket = 0u;
}

// Threads per CTA (at most one CTA per SM): as many rounds as the largest CTA
// needs, then just enough warps for that many, so the last round is not
// nearly empty. Many probes leave room for fewer warps' sums.
cudaError_t launch_quad_points(float* theta, const float* a, int64_t n, const RoundKeys& keys, int packing, int K,
                               double eps, double* losses, double* c, int32_t* status, double* partial,
                               uint32_t* ticket, int num_sms, cudaStream_t stream) {
  QuadPointsParams P;
  P.theta = theta;
  P.a = a;
  P.n = n;
  P.keys = keys;
  P.K = K;
  P.groups = (K + 7) / 8;
  P.neps_bits = __builtin_bit_cast(uint32_t, static_cast<float>(eps)) ^ 0x80000000u;
  P.nmeps_bits = __builtin_bit_cast(uint32_t, static_cast<float>(-2.0 * eps)) ^ 0x80000000u;
  P.losses = losses;
  P.partial = partial;
  P.ticket = ticket;
  P.zero = 0.0f;
  P.drift = static_cast<float>(K + 1) * 0x1p-21f;
  P.eps = eps;
  P.c = c;
  P.status = status;
  int max_warps = kPointsMaxThreads / 32;
  while (max_warps > 1 && quad_points_smem_bytes(P.groups, max_warps, true) > kQuadPointsMaxSmem) --max_warps;
  const int64_t items = (n + kItem - 1) / kItem;
  const int64_t cap = static_cast<int64_t>(num_sms) * max_warps * 32;
  const int64_t rounds = items > cap ? (items + cap - 1) / cap : 1;
  const int64_t per_round = static_cast<int64_t>(num_sms) * rounds * 32;
  int64_t warps = (items + per_round - 1) / per_round;
  if (warps < 8) warps = 8;  // the sums' folds, which take a warp per point
  if (warps > max_warps) warps = max_warps;
  const int threads = static_cast<int>(warps) * 32;
  int64_t grid = (items + 31) / 32;
  if (grid < 1) grid = 1;
  if (grid > num_sms) grid = num_sms;
  if (grid > kQuadPointsMaxCtas) grid = kQuadPointsMaxCtas;  // the workspace's partials
  const bool vec = reinterpret_cast<uintptr_t>(theta) % 16 == 0 && reinterpret_cast<uintptr_t>(a) % 16 == 0;
  P.several = items > grid * warps * 32;
  const size_t smem = quad_points_smem_bytes(P.groups, static_cast<int>(warps), P.several != 0);
  const auto go = [&](auto kernel) -> cudaError_t {
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           static_cast<int>(kQuadPointsMaxSmem));
      if (e != cudaSuccess) return e;
    }
    kernel<<<static_cast<int>(grid), threads, smem, stream>>>(P);
    return cudaGetLastError();
  };
  if (packing == kPacking8) return vec ? go(quad_points_kernel<true, true>) : go(quad_points_kernel<true, false>);
  return vec ? go(quad_points_kernel<false, true>) : go(quad_points_kernel<false, false>);
}

}  // namespace zo
