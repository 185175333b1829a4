// zo_api.cu -- the extern "C" entry points declared in include/zo.h: argument
// validation, Philox key expansion, tensor-table planning and launch sizing.
// Everything here runs on the host and only enqueues kernels.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include <cuda_runtime.h>

#include "zo.h"
#include "zo_items.h"
#include "zo_launch.h"

namespace {

using zo::RoundKeys;
using zo::TensorTable;
using zo::UpdateParams;

thread_local char g_last_cuda_error[256] = "";

int cuda_fail(cudaError_t e, const char* where) {
  std::snprintf(g_last_cuda_error, sizeof(g_last_cuda_error), "%s: %s (%s)", where, cudaGetErrorName(e),
                cudaGetErrorString(e));
  return ZO_ERR_CUDA;
}

// Philox4x32 key schedule: round r uses (lo + r * W0, hi + r * W1) mod 2^32.
RoundKeys expand_keys(uint64_t seed) {
  RoundKeys k;
  uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    k.k0[r] = k0;
    k.k1[r] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return k;
}

int elem_size(int32_t dtype) { return dtype == ZO_F32 ? 4 : 2; }

// Probe packing of every later call (1 or 8 generated bits per weight and probe).
std::atomic<int> g_packing{zo::kPacking1};

// Third Philox counter word and sign bit of probe k under the current packing.
void probe_counter(uint32_t k, int packing, uint32_t* ctr2, uint32_t* bit) {
  if (packing == zo::kPacking8) {
    *ctr2 = k;
    *bit = 0;
  } else {
    *ctr2 = k >> 3;
    *bit = k & 7u;
  }
}

// An operand's sign taken from bit `bit` of a weight's byte.
void set_bit(zo::PerturbOp& op, uint32_t bit) {
  op.bit = bit;
  for (uint32_t m = 0; m < 4; ++m) op.mul[m] = 1u << (31u - 8u * m - bit);
}

// theta <- rn(theta + scale z_k) as a kernel operand.
zo::PerturbOp make_op(uint32_t k, float scale, int packing) {
  zo::PerturbOp op;
  uint32_t bit = 0, u;
  probe_counter(k, packing, &op.ctr2, &bit);
  set_bit(op, bit);
  std::memcpy(&u, &scale, sizeof(u));
  op.nscale_bits = u ^ 0x80000000u;  // -scale: the probe bit flips it to +scale
  return op;
}

// Most items per SM of a list that update_items_kernel takes, in as many
// launches as its tensors fill tables (packing 8, K = 8, 1000 tensors of 1 M bf16
// weights in all: 42 -> 21 us). It does two
// lookups per element and group where the table-per-lane kernels do one, but
// copies no tables; the lines lie where the two cross on 12 or 24 tensors (us,
// items against tables):
//   packing 1   K = 16: 3 M weights 10.5 / 12.9, 8 M 17.1 / 15.8
//               K = 20: 5 M 14.7 / 15.1, 8 M 19.2 / 18.8;  K = 32: 16.8 / 17.1, 23.0 / 21.2
//               K = 64: 3 M 16.8 / 19.1, 8 M 33.4 / 31.6;  K = 256: 43.6 / 43.6, 97 / 80
// (3 M weights are 1233 items per SM; the items' side before kPlain's launch bound,
// which takes 3 to 7 % off K = 64 and more). Under packing 8 generating the bits is
// most of the work and many small CTAs do it best, whatever the size, but for
// 16-bit lists of many groups:
//   fp32          K = 3: 100 M 134 / 151;  K = 24: 399 / 450;  K = 64: 50 M 506 / 531, 205 M 2010 / 2081
//                 K = 256: 50 M 1944 / 1978, 205 M 7800 / 7880
//   16 bits       K = 3: 205 M 219 / 268;  K = 24: 809 / 862;  K = 64: 50 M 512 / 522, 205 M 2049 / 2047
//                 K = 96: 50 M 756 / 763, 80 M 1203 / 1199;  K = 256: 20 M 804 / 832, 50 M 1977 / 1967
//   16-bit views  K = 3: 205 M 235 / 316;  K = 48: 1650 / 1649;  K = 64: 20 M 224 / 227, 205 M 2179 / 2154
//                 K = 128: 10 M 224 / 233, 20 M 434 / 429, 50 M 1070 / 1040
//   fp32 views    K = 3: 3 M 14.7 / 17.0, 6 M 23.1 / 21.3;  K = 24: 1 M 14.8 / 17.0, 3 M 31.4 / 28.2
//                 K = 64: 1 M 27.3 / 24.8
// (1 M fp32 weights are 822 items per SM; those off the 32-byte grid make a
// block's words twice. With a leading perturbation, whose words the items have
// for nothing, they gain up to 1 %: K = 64, 205 M 2076 / 2100.) Between 1 and
// 0.05 M weights of packing 1 all of these take about 9 us here, 11 to 35 with
// the tables. f32, views: mostly so, by weights.
int64_t update_items_per_sm(int packing, int groups, bool f32, bool views) {
  if (packing != zo::kPacking8) return groups == 3 || groups == 4 ? 2400 : 1600;
  constexpr int64_t any = INT64_C(1) << 40;
  if (f32 && views) return groups == 1 ? 3000 : groups <= 4 ? 1200 : 400;
  if (f32 || groups < 8) return any;
  if (views) return groups == 8 ? 24000 : 8000;
  return groups == 8 ? any : 24000;
}

// Which kernel an update's list goes to.
enum UpdateRoute { kByItems, kByBlocks, kResidentTables, kByChunks };

struct UpdatePlan {
  UpdateRoute route;
  bool f32_blocks;  // mostly fp32 on the 32-byte grid
};

UpdatePlan plan_update(const zo_tensor* params, int32_t n, const UpdateParams& up, int sms) {
  int64_t f32 = 0, f32_off = 0, off = 0, all = 0;  // weights: fp32 on and off the 32-byte grid, any off it, all
  int64_t items = 0;                               // of the list by items
  for (int32_t i = 0; i < n; ++i) {
    const bool on = reinterpret_cast<uintptr_t>(params[i].ptr) % 32 == 0;
    items += zo::tensor_items(params[i]);
    all += params[i].numel;
    if (!on) off += params[i].numel;
    if (params[i].dtype == ZO_F32) (on ? f32 : f32_off) += params[i].numel;
  }
  const bool f32_blocks = 2 * f32 > all, f32_views = 2 * f32_off > all;
  const int64_t most_items =
      update_items_per_sm(up.packing, up.groups, f32_blocks || f32_views, f32_views || (!f32_blocks && 2 * off > all)) *
      sms;
  UpdatePlan p = {kByChunks, f32_blocks};
  if (items <= most_items && all / 16 + n <= INT64_C(1) << 32)  // the items' counter high word is 0
    p.route = kByItems;
  else if (f32_views && zo::update_blocks_takes(up, f32_off, sms))
    p.route = kByBlocks;
  else if (zo::lut8_small_takes(up, f32_blocks, f32_views))
    p.route = kResidentTables;
  return p;
}

// Per-device launch facts, filled once per device.
struct DeviceInfo {
  int sms = 0;
  bool lut8_ready = false;                // the update kernels' shared-memory limits are raised
};
constexpr int kMaxDevices = 64;
DeviceInfo g_dev[kMaxDevices];
std::mutex g_dev_mu;

int device_info(DeviceInfo** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return ZO_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_dev_mu);
  DeviceInfo& d = g_dev[dev];
  if (d.sms == 0) {
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    d.sms = sms;
  }
  *out = &d;
  return ZO_OK;
}

// Raises the update kernels' dynamic shared-memory limits, once per device.
int lut8_ready(DeviceInfo* d) {
  std::lock_guard<std::mutex> lock(g_dev_mu);
  if (!d->lut8_ready) {
    cudaError_t e = zo::lut8_prepare();
    if (e != cudaSuccess) return cuda_fail(e, "shared-memory limit(update_lut8)");
    d->lut8_ready = true;
  }
  return ZO_OK;
}

// Checks a parameter list; *packing (optional) receives the probe packing
// its tensors ask for (zo_tensor.packing: 0 = the process default, else 1
// or 8, the same for every tensor of the list) resolved to 1 or 8.
int validate_params(const zo_tensor* params, int32_t n, int* packing = nullptr) {
  if (n < 0) return ZO_ERR_ARG;
  if (n > 0 && params == nullptr) return ZO_ERR_ARG;
  int64_t blocks = 0;
  const int32_t pk = n > 0 ? params[0].packing : 0;
  if (pk != 0 && pk != zo::kPacking1 && pk != zo::kPacking8) return ZO_ERR_ARG;
  if (packing != nullptr) *packing = pk != 0 ? pk : g_packing.load();
  for (int32_t t = 0; t < n; ++t) {
    const zo_tensor& p = params[t];
    if (p.numel < 0 || p.packing != pk) return ZO_ERR_ARG;
    if (p.dtype != ZO_F32 && p.dtype != ZO_BF16 && p.dtype != ZO_F16) return ZO_ERR_DTYPE;
    if (p.numel > 0 && p.ptr == nullptr) return ZO_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(p.ptr) % static_cast<uintptr_t>(elem_size(p.dtype)) != 0) return ZO_ERR_ALIGN;
    const int64_t nb = (p.numel + 15) / 16;
    if (nb >= zo::kMaxLaunchBlocks) return ZO_ERR_ARG;          // one tensor must fit one launch
    if (nb > (INT64_C(1) << 58) - blocks) return ZO_ERR_ARG;   // virtual index space
    blocks += nb;
  }
  return ZO_OK;
}

// Fill `tab` with tensors t0, t0+1, ... while the launch holds fewer than
// kMaxTensorsPerLaunch tensors and fewer than kMaxLaunchBlocks launch blocks;
// the launch's first block has virtual index blk_base. In the launch
// numbering every tensor starts on a multiple of kLaunchAlign blocks (see
// TensorTable). Returns the first tensor not taken; *nblocks receives the
// virtual blocks the launch covers (tab.blk_total its launch blocks).
// kSlots: tensors off the 32-byte grid are flagged kShift and take 32 launch
// blocks per 31 of their aligned chunks (the update kernels). kItems: so, and
// launch blocks are 32-byte items, of which fp32 tensors have two per block; a
// tensor whose items alone exceed a launch is not taken.
enum Numbering { kBlocks, kSlots, kItems };

int32_t fill_table(TensorTable& tab, const zo_tensor* params, int32_t t0, int32_t n, int64_t blk_base,
                   int64_t* nblocks, Numbering numbering = kBlocks) {
  const bool slots = numbering != kBlocks;
  tab.n = 0;
  tab.blk_base = blk_base;
  int64_t b = 0;  // launch blocks so far
  int64_t v = 0;  // virtual blocks so far
  int32_t t = t0;
  for (; t < n && tab.n < zo::kMaxTensorsPerLaunch; ++t) {
    const zo_tensor& p = params[t];
    const int64_t nb = (p.numel + 15) / 16;
    const int64_t start = (b + zo::kLaunchAlign - 1) / zo::kLaunchAlign * zo::kLaunchAlign;
    const uint32_t off = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(p.ptr) % 32);
    const int64_t per = numbering == kItems && p.dtype == ZO_F32 ? 8 : 16;  // elements per launch block
    int64_t span = (p.numel + per - 1) / per;  // launch blocks of the tensor
    if (slots && off != 0 && nb > 0) {
      const int64_t chunks = (p.numel + off / elem_size(p.dtype) + per - 1) / per;
      span = (chunks + zo::kShiftLanes - 1) / zo::kShiftLanes * zo::kLaunchAlign;
    }
    if ((tab.n > 0 || numbering == kItems) && start + span >= zo::kMaxLaunchBlocks) break;
    const int i = tab.n++;
    tab.vdelta[i] = static_cast<uint32_t>(start - v);
    b = start + span;
    v += nb;
    tab.blk_end[i] = static_cast<uint32_t>(b);
    tab.ptr[i] = reinterpret_cast<uint64_t>(p.ptr);
    tab.numel[i] = p.numel;
    uint8_t fl = static_cast<uint8_t>(p.dtype);
    if (off == 0) fl |= zo::kVec32;
    if (slots && off != 0 && nb > 0) fl |= zo::kShift;
    tab.flags[i] = fl;
  }
  tab.blk_total = static_cast<uint32_t>(b);
  *nblocks = v;
  return t;
}

int grid_for(int64_t blocks, int sms, int bps) {
  const int64_t want = (blocks + zo::kThreads - 1) / zo::kThreads;
  const int64_t cap = static_cast<int64_t>(sms) * bps;
  const int64_t g = want < cap ? want : cap;
  return static_cast<int>(g < 1 ? 1 : g);
}

thread_local zo::ItemsParams<zo::kItemsFew> tl_items_few;
thread_local zo::ItemsParams<zo::kItemsSome> tl_items_some;
thread_local zo::ItemsParams<zo::kItemsMany> tl_items_many;

// One perturbation pass over a list.
struct PerturbPass {
  RoundKeys keys;
  zo::PerturbOp op[2];
  int32_t nops;
  uint32_t probe;
  const double* coef;
  double coef_mul;
  const int32_t* status;
};

template <int N>
void set_pass(zo::ItemsParams<N>& ip, const PerturbPass& pp) {
  ip.keys = pp.keys;
  ip.op[0] = pp.op[0];
  ip.op[1] = pp.op[1];
  const uint32_t high = static_cast<uint32_t>(static_cast<uint64_t>(ip.e[0].vb) >> 32);
  ip.g[0] = zo::group_round01(pp.op[0].ctr2, high, pp.keys);
  ip.g[1] = zo::group_round01(pp.op[1].ctr2, high, pp.keys);
  ip.nops = pp.nops;
  ip.probe = pp.probe;
  ip.coef = pp.coef;
  ip.coef_mul = pp.coef_mul;
  ip.status = pp.status;
}

// Launches over the whole list, each with the smallest table that holds it
// (kItemsMany per launch when the virtual blocks cross a counter high word).
int run_perturb(const zo_tensor* params, int32_t n, const PerturbPass& pp, cudaStream_t s) {
  zo::ItemsCursor cur;
  const auto launch = [&](auto& ip) -> cudaError_t {
    const zo::ItemsCursor from = cur;
    const auto no_more = [](auto&, int32_t, int64_t) {};
    if (zo::fill_items(ip, params, n, cur, no_more)) {
      if (ip.n == 0) return cudaSuccess;
      set_pass(ip, pp);
      return zo::launch_perturb_items(ip, s);
    }
    cur = from;
    zo::fill_items(tl_items_many, params, n, cur, no_more);
    set_pass(tl_items_many, pp);
    return zo::launch_perturb_items_any_high(tl_items_many, s);
  };
  while (cur.t < n) {
    const int32_t left = n - cur.t;
    const cudaError_t e = left <= zo::kItemsFew    ? launch(tl_items_few)
                          : left <= zo::kItemsSome ? launch(tl_items_some)
                                                   : launch(tl_items_many);
    if (e != cudaSuccess) return cuda_fail(e, "perturb_items_kernel");
  }
  return ZO_OK;
}

thread_local zo::PairItemsParams<zo::kItemsFew> tl_pair_few;
thread_local zo::PairItemsParams<zo::kItemsSome> tl_pair_some;
thread_local zo::PairItemsParams<zo::kPairItemsMany> tl_pair_many;
thread_local zo::SmallUpdateParams tl_update;
thread_local zo::UpdateItemsParams<zo::kItemsFew> tl_update_few;
thread_local zo::UpdateItemsParams<zo::kItemsSome> tl_update_some;
thread_local zo::UpdateItemsParams<zo::kItemsMany> tl_update_many;

}  // namespace

extern "C" {

const char* zo_status_string(int status) {
  switch (status) {
    case ZO_OK: return "ZO_OK";
    case ZO_ERR_ARG: return "ZO_ERR_ARG: invalid argument";
    case ZO_ERR_DTYPE: return "ZO_ERR_DTYPE: unknown dtype";
    case ZO_ERR_ALIGN: return "ZO_ERR_ALIGN: pointer not aligned to its element size";
    case ZO_ERR_NONFINITE: return "ZO_ERR_NONFINITE: non-finite loss, curvature or coefficient";
    case ZO_ERR_CUDA: return "ZO_ERR_CUDA: CUDA runtime error";
    case ZO_ERR_TOO_MANY_PROBES: return "ZO_ERR_TOO_MANY_PROBES: K exceeds ZO_MAX_PROBES";
    case ZO_ERR_WORKSPACE: return "ZO_ERR_WORKSPACE: workspace missing or too small";
    default: return "unknown zo_status";
  }
}

const char* zo_last_cuda_error(void) { return g_last_cuda_error; }

int zo_version(void) { return 10500; }

int zo_set_packing(int32_t bits_per_value) {
  if (bits_per_value != zo::kPacking1 && bits_per_value != zo::kPacking8) return ZO_ERR_ARG;
  g_packing.store(bits_per_value);
  return ZO_OK;
}

int zo_get_packing(void) { return g_packing.load(); }

int zo_perturb(const zo_tensor* params, int32_t n_tensors, uint64_t seed, uint32_t probe, float scale,
               void* stream) {
  int packing = zo::kPacking1;
  int rc = validate_params(params, n_tensors, &packing);
  if (rc != ZO_OK) return rc;
  if (!std::isfinite(scale)) return ZO_ERR_ARG;
  if (n_tensors == 0) return ZO_OK;
  PerturbPass pp;
  pp.keys = expand_keys(seed);
  pp.probe = probe;
  pp.op[0] = make_op(probe, scale, packing);
  pp.op[1] = pp.op[0];
  pp.nops = 1;
  pp.coef = nullptr;
  pp.coef_mul = 0.0;
  pp.status = nullptr;
  return run_perturb(params, n_tensors, pp, static_cast<cudaStream_t>(stream));
}

int zo_perturb2(const zo_tensor* params, int32_t n_tensors, uint64_t seed, uint32_t probe_a, float scale_a,
                uint32_t probe_b, float scale_b, void* stream) {
  int packing = zo::kPacking1;
  int rc = validate_params(params, n_tensors, &packing);
  if (rc != ZO_OK) return rc;
  if (!std::isfinite(scale_a) || !std::isfinite(scale_b)) return ZO_ERR_ARG;
  if (n_tensors == 0) return ZO_OK;
  PerturbPass pp;
  pp.keys = expand_keys(seed);
  pp.probe = probe_a;
  pp.op[0] = make_op(probe_a, scale_a, packing);
  pp.op[1] = make_op(probe_b, scale_b, packing);
  pp.nops = 2;
  pp.coef = nullptr;
  pp.coef_mul = 0.0;
  pp.status = nullptr;
  return run_perturb(params, n_tensors, pp, static_cast<cudaStream_t>(stream));
}

int zo_perturb_pair(const zo_tensor* theta, const zo_tensor* plus, const zo_tensor* minus, int32_t n_tensors,
                    uint64_t seed, uint32_t probe, float scale, void* stream) {
  int packing = zo::kPacking1, pk_plus = 0, pk_minus = 0;
  int rc = validate_params(theta, n_tensors, &packing);
  if (rc != ZO_OK) return rc;
  if ((rc = validate_params(plus, n_tensors, &pk_plus)) != ZO_OK) return rc;
  if ((rc = validate_params(minus, n_tensors, &pk_minus)) != ZO_OK) return rc;
  // plus and minus follow theta's probes: they may name no packing or the same one
  if (n_tensors > 0 && ((plus[0].packing != 0 && pk_plus != packing) ||
                        (minus[0].packing != 0 && pk_minus != packing)))
    return ZO_ERR_ARG;
  if (!std::isfinite(scale)) return ZO_ERR_ARG;
  for (int32_t t = 0; t < n_tensors; ++t) {
    if (plus[t].numel != theta[t].numel || minus[t].numel != theta[t].numel) return ZO_ERR_ARG;
    if (plus[t].dtype != theta[t].dtype || minus[t].dtype != theta[t].dtype) return ZO_ERR_ARG;
    if (theta[t].numel > 0 && plus[t].ptr == minus[t].ptr) return ZO_ERR_ARG;
  }
  if (n_tensors == 0) return ZO_OK;
  zo::ItemsCursor cur;
  const auto launch = [&](auto& ip) -> cudaError_t {
    const bool one_high = zo::fill_items(ip, plus, n_tensors, cur, [&](auto& e, int32_t t, int64_t bytes) {
      e.src = static_cast<uint64_t>(reinterpret_cast<uintptr_t>(theta[t].ptr)) + static_cast<uint64_t>(bytes);
      e.minus = static_cast<uint64_t>(reinterpret_cast<uintptr_t>(minus[t].ptr)) + static_cast<uint64_t>(bytes);
    });
    if (ip.n == 0) return cudaSuccess;
    ip.keys = expand_keys(seed);
    ip.op = make_op(probe, scale, packing);
    ip.g = zo::group_round01(ip.op.ctr2, static_cast<uint32_t>(static_cast<uint64_t>(ip.e[0].vb) >> 32), ip.keys);
    return zo::launch_pair_items(ip, one_high, static_cast<cudaStream_t>(stream));
  };
  while (cur.t < n_tensors) {
    const int32_t left = n_tensors - cur.t;
    const cudaError_t e = left <= zo::kItemsFew    ? launch(tl_pair_few)
                          : left <= zo::kItemsSome ? launch(tl_pair_some)
                                                   : launch(tl_pair_many);
    if (e != cudaSuccess) return cuda_fail(e, "pair_items_kernel");
  }
  return ZO_OK;
}

static int check_update_args(const zo_tensor* params, int32_t n, const double* c, int32_t K, double lr,
                             int* packing) {
  int rc = validate_params(params, n, packing);
  if (rc != ZO_OK) return rc;
  if (K < 1) return ZO_ERR_ARG;
  if (K > ZO_MAX_PROBES) return ZO_ERR_TOO_MANY_PROBES;
  if (c == nullptr || !std::isfinite(lr)) return ZO_ERR_ARG;
  return ZO_OK;
}

int zo_update(const zo_tensor* params, int32_t n_tensors, uint64_t seed, const double* c, int32_t K, double lr,
              const int32_t* status, void* stream) {
  return zo_update_ex(params, n_tensors, seed, c, K, lr, status, 0, 0u, 0.0f, stream);
}

int zo_update_ex(const zo_tensor* params, int32_t n_tensors, uint64_t seed, const double* c, int32_t K, double lr,
                 const int32_t* status, int32_t has_pre, uint32_t pre_probe, float pre_scale, void* stream) {
  int packing = zo::kPacking1;
  int rc = check_update_args(params, n_tensors, c, K, lr, &packing);
  if (rc != ZO_OK) return rc;
  if (has_pre != 0 && !std::isfinite(pre_scale)) return ZO_ERR_ARG;
  if (n_tensors == 0) return rc;
  DeviceInfo* d = nullptr;
  if ((rc = device_info(&d)) != ZO_OK) return rc;
  UpdateParams& up = tl_update.u;
  up.keys = expand_keys(seed);
  up.coef = c;
  up.coef_mul = -(lr / static_cast<double>(K));
  up.K = K;
  up.groups = (K + 7) / 8;
  up.packing = packing;
  up.has_pre = has_pre != 0;
  up.pre = make_op(pre_probe, has_pre != 0 ? pre_scale : 0.0f, up.packing);
  up.status = status;
  const UpdatePlan plan = plan_update(params, n_tensors, up, d->sms);
  const bool f32_blocks = plan.f32_blocks;
  zo::ItemsCursor cur;
  const auto by_items = [&](auto& ip) -> cudaError_t {
    zo::fill_items(ip, params, n_tensors, cur, [](auto&, int32_t, int64_t) {});
    if (ip.n == 0) return cudaSuccess;
    // packing 8: several items per thread where about eight waves of CTAs remain, which spread a CTA's tables over
    // more work (205 M bf16 weights, K = 8, one / eight / ten items: 396 / 317 / 315 us; as fp32 with 32 / 64 at most
    // 326 / 322; 30 M bf16 weights one / two 58.4 / 55.7)
    const int64_t unit = INT64_C(8) * 128 * 8 * d->sms, waves = (ip.total + unit / 2) / unit, cap = f32_blocks ? 64 : 16;
    ip.f32_blocks = f32_blocks;
    ip.rounds = static_cast<uint32_t>(waves < 1 ? 1 : waves > cap ? cap : waves);
    if (f32_blocks && ip.rounds % 2 == 1) ++ip.rounds;  // fp32: whole blocks, two items each
    ip.bhi = 0;
    ip.keys = up.keys;
    ip.coef = c;
    ip.coef_mul = up.coef_mul;
    ip.K = up.K;
    ip.groups = up.groups;
    ip.packing = up.packing;
    ip.has_pre = up.has_pre;
    ip.pre = up.pre;
    // not where one wave of fp32 goes through many groups, whose loop is slower so than a call saved (us, with / without:
    // 0.3 M weights, K = 256 / 520 44.7 / 43.8, 86.6 / 84.6; 1 M 74.9 / 76.0, 147.9 / 149.7)
    const bool one_wave = f32_blocks && up.groups > 8 && ip.total < 500 * static_cast<int64_t>(d->sms);
    ip.pre_last = up.has_pre && up.packing == zo::kPacking8 && pre_probe < static_cast<uint32_t>(K) &&
                  pre_probe / 8u + 1u == static_cast<uint32_t>(up.groups) && !one_wave;
    if (ip.pre_last) set_bit(ip.pre, pre_probe & 7u);
    ip.status = status;
    return zo::launch_update_items(ip, d->sms, static_cast<cudaStream_t>(stream));
  };
  if (plan.route == kByItems) {
    while (cur.t < n_tensors) {
      const int32_t left = n_tensors - cur.t;
      const cudaError_t e = left <= zo::kItemsFew    ? by_items(tl_update_few)
                            : left <= zo::kItemsSome ? by_items(tl_update_some)
                                                     : by_items(tl_update_many);
      if (e != cudaSuccess) return cuda_fail(e, "update_items_kernel");
    }
    return ZO_OK;
  }
  const bool by_blocks = plan.route == kByBlocks, few = plan.route == kResidentTables;
  tl_update.f32_blocks = f32_blocks;
  if ((rc = lut8_ready(d)) != ZO_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int64_t blk = 0;
  for (int32_t t0 = 0; t0 < n_tensors;) {
    int64_t nb = 0;
    const int32_t first = t0;
    t0 = fill_table(up.tab, params, first, n_tensors, blk, &nb, few ? kItems : kSlots);
    const bool small = few && t0 > first && zo::one_high_word(up.tab);
    if (few && !small) t0 = fill_table(up.tab, params, first, n_tensors, blk, &nb, kSlots);
    blk += nb;
    if (nb == 0) continue;
    bool any = false;  // a non-empty tensor that is not 16-bit and aligned
    for (int i = 0; i < up.tab.n && !any; ++i)
      any = up.tab.numel[i] > 0 &&
            ((up.tab.flags[i] & zo::kShift) || (up.tab.flags[i] & zo::kDtypeMask) == zo::kF32);
    const cudaError_t e = by_blocks ? zo::launch_update_blocks(up, d->sms, s)
                          : small   ? zo::launch_update_lut8_small(tl_update, any, d->sms, s)
                                    : zo::launch_update_lut8(up, any, d->sms, s);
    if (e != cudaSuccess)
      return cuda_fail(e, by_blocks ? "update_blocks_kernel" : small ? "update_lut8_small_kernel" : "update_lut8_kernel");
  }
  return ZO_OK;
}

// Not part of the public interface: the kernel that zo_update_ex sends a list to
// on a device of `sms` SMs (UpdateRoute), for the tests of each kernel.
int zo_internal_update_route(const zo_tensor* params, int32_t n_tensors, int32_t K, int32_t has_pre,
                             uint32_t pre_probe, int32_t sms) {
  UpdateParams& up = tl_update.u;
  int rc = validate_params(params, n_tensors, &up.packing);
  if (rc != ZO_OK) return rc;
  up.groups = (K + 7) / 8;
  up.has_pre = has_pre != 0;
  up.pre = make_op(pre_probe, 0.0f, up.packing);
  return plan_update(params, n_tensors, up, sms).route;
}

int zo_update_sequential(const zo_tensor* params, int32_t n_tensors, uint64_t seed, const double* c, int32_t K,
                         double lr, const int32_t* status, void* stream) {
  int packing = zo::kPacking1;
  int rc = check_update_args(params, n_tensors, c, K, lr, &packing);
  if (rc != ZO_OK || n_tensors == 0) return rc;
  PerturbPass pp;
  pp.keys = expand_keys(seed);
  pp.coef = c;
  pp.coef_mul = -(lr / static_cast<double>(K));
  pp.status = status;
  pp.nops = 1;
  for (int32_t k = 0; k < K; ++k) {
    pp.probe = static_cast<uint32_t>(k);
    pp.op[0] = make_op(pp.probe, 0.0f, packing);  // scale read from c on the device
    pp.op[1] = pp.op[0];
    if ((rc = run_perturb(params, n_tensors, pp, static_cast<cudaStream_t>(stream))) != ZO_OK) return rc;
  }
  return ZO_OK;
}

static int check_precondition_args(const double* losses, int32_t K, double eps, double alpha, double lambda_reg,
                                   const double* c, const int32_t* status) {
  if (K < 1) return ZO_ERR_ARG;
  if (K > ZO_MAX_PROBES) return ZO_ERR_TOO_MANY_PROBES;
  if (losses == nullptr || c == nullptr || status == nullptr) return ZO_ERR_ARG;
  if (!(eps > 0.0) || !std::isfinite(eps)) return ZO_ERR_ARG;
  if (!(alpha >= 0.0) || !(alpha <= 1.0)) return ZO_ERR_ARG;
  if (!(lambda_reg > 0.0) || !std::isfinite(lambda_reg)) return ZO_ERR_ARG;
  return ZO_OK;
}

int zo_precondition_ex(const double* losses, int32_t K, double eps, double alpha, double lambda_reg,
                       int32_t flags, double* c, double* w, double* curv, int32_t* status, void* stream) {
  int rc = check_precondition_args(losses, K, eps, alpha, lambda_reg, c, status);
  if (rc != ZO_OK) return rc;
  if ((flags & ~(ZO_PRECOND_ONE_SIDED | ZO_PRECOND_RELATIVE_CURVATURE)) != 0) return ZO_ERR_ARG;
  static_assert(ZO_PRECOND_ONE_SIDED == zo::kPrecondOneSided && ZO_PRECOND_RELATIVE_CURVATURE == zo::kPrecondRelative,
                "flag values");
  cudaError_t e = zo::launch_precondition(losses, K, eps, alpha, lambda_reg, flags, c, w, curv, status,
                                          static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ZO_OK : cuda_fail(e, "precondition_kernel");
}

int zo_precondition(const double* losses, int32_t K, double eps, double* c, int32_t* status, void* stream) {
  return zo_precondition_ex(losses, K, eps, 0.1, 1.0, 0, c, nullptr, nullptr, status, stream);
}

static int probe_view_grid(int64_t blocks, int* grid) {
  DeviceInfo* d = nullptr;
  int rc = device_info(&d);
  if (rc != ZO_OK) return rc;
  *grid = grid_for(blocks, d->sms, 8);
  return ZO_OK;
}

int zo_probe_bytes(uint64_t seed, uint32_t probe, int64_t first, int64_t n, uint8_t* out, void* stream) {
  if (first < 0 || n < 0 || (n > 0 && out == nullptr)) return ZO_ERR_ARG;
  if (n > (INT64_C(1) << 58) - first) return ZO_ERR_ARG;
  if (n == 0) return ZO_OK;
  int grid = 1;
  int rc = probe_view_grid((n + 1) / 2 + 1, &grid);
  if (rc != ZO_OK) return rc;
  uint32_t ctr2 = 0, bit = 0;
  probe_counter(probe, g_packing.load(), &ctr2, &bit);
  cudaError_t e = zo::launch_probe_bytes(expand_keys(seed), ctr2, bit, first, n, out, grid,
                                         static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ZO_OK : cuda_fail(e, "probe_bytes_kernel");
}

int zo_probe_signs(uint64_t seed, uint32_t probe, int64_t first, int64_t n, int8_t* out, void* stream) {
  if (first < 0 || n < 0 || (n > 0 && out == nullptr)) return ZO_ERR_ARG;
  if (n > (INT64_C(1) << 58) - first) return ZO_ERR_ARG;
  if (n == 0) return ZO_OK;
  int grid = 1;
  int rc = probe_view_grid(n / 16 + 2, &grid);
  if (rc != ZO_OK) return rc;
  uint32_t ctr2 = 0, bit = 0;
  probe_counter(probe, g_packing.load(), &ctr2, &bit);
  cudaError_t e = zo::launch_probe_signs(expand_keys(seed), ctr2, bit, first, n, out, grid,
                                         static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ZO_OK : cuda_fail(e, "probe_signs_kernel");
}

int64_t zo_quadratic_loss_workspace_size(int64_t n) {
  (void)n;
  return static_cast<int64_t>(zo::kMaxLossPartials) * static_cast<int64_t>(sizeof(double));
}

int zo_quadratic_loss(const float* theta, const float* a, int64_t n, double* out, void* workspace,
                      int64_t workspace_bytes, void* stream) {
  if (n < 0 || out == nullptr || (n > 0 && (theta == nullptr || a == nullptr))) return ZO_ERR_ARG;
  if (workspace == nullptr || workspace_bytes < zo_quadratic_loss_workspace_size(n)) return ZO_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % sizeof(double) != 0) return ZO_ERR_ALIGN;
  DeviceInfo* d = nullptr;
  int rc = device_info(&d);
  if (rc != ZO_OK) return rc;
  cudaError_t e = zo::launch_quadratic_loss(theta, a, n, out, static_cast<double*>(workspace), zo::kMaxLossPartials,
                                            d->sms, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ZO_OK : cuda_fail(e, "quadratic_loss");
}

int64_t zo_perturb_quadratic_loss_workspace_size(int64_t n) {
  (void)n;
  // the partials, then the ticket counter (8 bytes keep the size a multiple of 8)
  return static_cast<int64_t>(zo::kMaxQuadPassPartials) * static_cast<int64_t>(sizeof(double)) + 8;
}

int zo_perturb_quadratic_loss(float* theta, const float* a, int64_t n, uint64_t seed, int32_t packing, int32_t nops,
                              uint32_t probe_a, float scale_a, uint32_t probe_b, float scale_b, double* out,
                              int32_t out_copies, int64_t out_stride, void* workspace, int64_t workspace_bytes,
                              void* stream) {
  if (n < 0 || out == nullptr || (n > 0 && (theta == nullptr || a == nullptr))) return ZO_ERR_ARG;
  if (nops < 0 || nops > 2 || out_copies < 1 || out_stride < 1) return ZO_ERR_ARG;
  if (packing != 0 && packing != zo::kPacking1 && packing != zo::kPacking8) return ZO_ERR_ARG;
  if ((nops >= 1 && !std::isfinite(scale_a)) || (nops == 2 && !std::isfinite(scale_b))) return ZO_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(theta) % sizeof(float) != 0 || reinterpret_cast<uintptr_t>(a) % sizeof(float) != 0)
    return ZO_ERR_ALIGN;
  if (workspace == nullptr || workspace_bytes < zo_perturb_quadratic_loss_workspace_size(n)) return ZO_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % sizeof(double) != 0) return ZO_ERR_ALIGN;
  DeviceInfo* d = nullptr;
  int rc = device_info(&d);
  if (rc != ZO_OK) return rc;
  const int pk = packing != 0 ? packing : g_packing.load();
  const zo::RoundKeys keys = expand_keys(seed);
  const zo::PerturbOp ops[2] = {make_op(probe_a, scale_a, pk), make_op(probe_b, scale_b, pk)};
  double* partial = static_cast<double*>(workspace);
  uint32_t* ticket = reinterpret_cast<uint32_t*>(partial + zo::kMaxQuadPassPartials);
  cudaError_t e = zo::launch_perturb_quad_loss(theta, a, n, keys, ops, nops, out, out_copies, out_stride, partial,
                                               ticket, zo::kMaxQuadPassPartials, d->sms,
                                               static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ZO_OK : cuda_fail(e, "perturb_quad_loss");
}

int64_t zo_quadratic_points_workspace_size(int32_t K) {
  const int64_t points = 2 * static_cast<int64_t>(K < 1 ? 1 : K) + 1;
  return points * zo::kQuadPointsMaxCtas * static_cast<int64_t>(sizeof(double)) + 8;  // the partials, then the ticket
}

int zo_quadratic_points(float* theta, const float* a, int64_t n, uint64_t seed, int32_t packing, int32_t K, double eps,
                        double* losses, double* c, int32_t* status, void* workspace, int64_t workspace_bytes,
                        void* stream) {
  if (n < 0 || losses == nullptr || (n > 0 && (theta == nullptr || a == nullptr)) || K < 1) return ZO_ERR_ARG;
  if ((c == nullptr) != (status == nullptr) || (c != nullptr && !(eps > 0.0))) return ZO_ERR_ARG;
  if (K > ZO_MAX_PROBES) return ZO_ERR_TOO_MANY_PROBES;
  if (packing != 0 && packing != zo::kPacking1 && packing != zo::kPacking8) return ZO_ERR_ARG;
  const float scale = static_cast<float>(eps), mscale = static_cast<float>(-2.0 * eps);
  if (!std::isfinite(scale) || !std::isfinite(mscale)) return ZO_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(theta) % sizeof(float) != 0 || reinterpret_cast<uintptr_t>(a) % sizeof(float) != 0)
    return ZO_ERR_ALIGN;
  if (workspace == nullptr || workspace_bytes < zo_quadratic_points_workspace_size(K)) return ZO_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % sizeof(double) != 0) return ZO_ERR_ALIGN;
  DeviceInfo* d = nullptr;
  int rc = device_info(&d);
  if (rc != ZO_OK) return rc;
  double* partial = static_cast<double*>(workspace);
  uint32_t* ticket =
      reinterpret_cast<uint32_t*>(partial + (2 * static_cast<int64_t>(K) + 1) * zo::kQuadPointsMaxCtas);
  cudaError_t e = zo::launch_quad_points(theta, a, n, expand_keys(seed), packing != 0 ? packing : g_packing.load(), K,
                                         eps, losses, c, status, partial, ticket, d->sms,
                                         static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ZO_OK : cuda_fail(e, "quad_points");
}

int zo_quadratic_loss_static(const float* theta, const float* a, int64_t n, double* out, void* stream) {
  if (n < 0 || out == nullptr || (n > 0 && (theta == nullptr || a == nullptr))) return ZO_ERR_ARG;
  if (n > ZO_QUADRATIC_LOSS_STATIC_MAX_N) return ZO_ERR_WORKSPACE;
  static_assert(ZO_QUADRATIC_LOSS_STATIC_MAX_N == zo::kStaticLossPartials * zo::kStaticLossSlice,
                "static scratch capacity and the documented limit must agree");
  cudaError_t e = zo::launch_quadratic_loss_static(theta, a, n, out, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ZO_OK : cuda_fail(e, "quadratic_loss_static");
}

}  // extern "C"
