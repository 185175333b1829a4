// zo_launch.h -- host-side launch wrappers shared between the kernel files and
// the C ABI layer (not part of the public interface).
#pragma once

#include <cuda_runtime.h>

#include "zo_device.cuh"

namespace zo {

constexpr int kStatusNonFinite = -4;  // ZO_ERR_NONFINITE
constexpr int kPrecondOneSided = 1;   // ZO_PRECOND_ONE_SIDED
constexpr int kPrecondRelative = 2;   // ZO_PRECOND_RELATIVE_CURVATURE
constexpr int kThreads = 256;         // threads per block of the streaming kernels
constexpr int kMaxLossPartials = 2048;
constexpr int kStaticLossPartials = 4096;   // fixed scratch of the allocation-free loss (32 KB)
constexpr int kMaxQuadPassPartials = 4096;  // CTAs of the one-pass perturbation + loss
constexpr int kQuadPointsMaxCtas = 256;     // CTAs of the launch that takes a step through all its forward points
constexpr size_t kQuadPointsMaxSmem = 224 * 1024;  // and its shared memory per CTA
constexpr int64_t kStaticLossSlice = 2048;  // elements per partial in that variant

// Perturbation by 32-byte items, one per thread.
template <int N>
cudaError_t launch_perturb_items(const ItemsParams<N>& p, cudaStream_t stream);
// The same when the launch's virtual blocks differ in the counter's high word.
cudaError_t launch_perturb_items_any_high(const ItemsParams<kItemsMany>& p, cudaStream_t stream);
// The out-of-place pair; one_high: the launch's virtual blocks share the
// counter's high word.
template <int N>
cudaError_t launch_pair_items(const PairItemsParams<N>& p, bool one_high, cudaStream_t stream);
// Fused update: what lut8_small_takes (packing 1, at most kSmallGroups probe
// groups) with virtual blocks that share the counter's high word; ...
bool lut8_small_takes(const UpdateParams& u, bool f32_blocks, bool f32_views);  // mostly fp32 on, off the 32-byte grid
cudaError_t launch_update_lut8_small(SmallUpdateParams& p, bool any, int sms, cudaStream_t stream);
// ... and every other one. any: the launch holds fp32 tensors or tensors off
// the 32-byte grid (those flagged kShift, in slots of 32 launch blocks per 31
// chunks).
cudaError_t launch_update_lut8(const UpdateParams& p, bool any, int sms, cudaStream_t stream);
cudaError_t lut8_prepare();  // raises both kernels' shared-memory limits (once per device)
bool one_high_word(const TensorTable& tab);  // of the launch's virtual blocks
// Fused update of fp32 views without a leading perturbation (weights: of the list's, those fp32 off the 32-byte grid).
bool update_blocks_takes(const UpdateParams& u, int64_t weights, int sms);
cudaError_t launch_update_blocks(const UpdateParams& p, int sms, cudaStream_t stream);
// Fused update by items; its virtual blocks share the counter's high word.
template <int N>
cudaError_t launch_update_items(const UpdateItemsParams<N>& p, int sms, cudaStream_t stream);
cudaError_t launch_probe_bytes(const RoundKeys& keys, uint32_t ctr2, uint32_t bit, int64_t first, int64_t n,
                               uint8_t* out, int grid, cudaStream_t stream);
cudaError_t launch_probe_signs(const RoundKeys& keys, uint32_t ctr2, uint32_t bit, int64_t first, int64_t n,
                               int8_t* out, int grid, cudaStream_t stream);
cudaError_t launch_precondition(const double* losses, int K, double eps, double alpha, double lambda_reg,
                                int flags, double* c, double* w, double* curv, int32_t* status,
                                cudaStream_t stream);
cudaError_t launch_quadratic_loss(const float* theta, const float* a, int64_t n, double* out, double* partial,
                                  int max_partials, int num_sms, cudaStream_t stream);
cudaError_t launch_quadratic_loss_static(const float* theta, const float* a, int64_t n, double* out,
                                         cudaStream_t stream);
// ops: nops (0, 1 or 2) perturbations; partial: max_partials doubles; ticket:
// a zeroed counter, zeroed again by the launch.
cudaError_t launch_perturb_quad_loss(float* theta, const float* a, int64_t n, const RoundKeys& keys,
                                     const PerturbOp* ops, int nops, double* out, int out_copies, int64_t out_stride,
                                     double* partial, uint32_t* ticket, int max_partials, int num_sms,
                                     cudaStream_t stream);

// Every forward point of a step, and its coefficients when c is given; partial:
// (2 K + 1) * kQuadPointsMaxCtas doubles; ticket: as above.
cudaError_t launch_quad_points(float* theta, const float* a, int64_t n, const RoundKeys& keys, int packing, int K,
                               double eps, double* losses, double* c, int32_t* status, double* partial,
                               uint32_t* ticket, int num_sms, cudaStream_t stream);

}  // namespace zo
