// vbq_kernels.h — launchers of the library's CUDA kernels (internal; called by
// the C ABI in vbq_api.cu). Each returns the cudaError_t of its launch.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include "vbq_common.cuh"

namespace vbq {

// Pack-time kernels (vbq_pack.cu): per unit, item counts per width and warp
// tasks (counts[5u ..]); then the blobs. *err (a word the host can read) is
// set to 1 by launch_count for a width outside {1,2,4,8}, by launch_scatter
// for a code >= 2^b of its group.
cudaError_t launch_count(const uint8_t* widths, int64_t N, int G, int C, int nrb, int units,
                         uint32_t* counts, uint32_t* err, cudaStream_t s);
cudaError_t launch_scatter(const uint8_t* codes, const uint8_t* widths, const uint16_t* scales,
                           const uint32_t* counts, const LayoutView& L, uint8_t* blobs, uint32_t* err,
                           cudaStream_t s);
cudaError_t launch_dequant(const LayoutView& L, uint8_t* codes_out, uint8_t* widths_out,
                           uint16_t* scales_out, float* w_out, cudaStream_t s);

// Quantisation (vbq_quant.cu): validation (err[0] set to 1 for a width outside
// {1,2,4,8}, err[1] for a NaN weight; words the host can read), then codes and
// FP16 scales per group.
cudaError_t launch_quant_validate(const float* w, const uint8_t* widths, int64_t N, int64_t K, uint32_t* err,
                                  cudaStream_t s);
cudaError_t launch_quantize(const float* w, const uint8_t* widths, int64_t N, int64_t K, uint8_t* codes,
                            uint16_t* scales, cudaStream_t s);

// Training-time soft-quantised forward (vbq_soft.cu): w_soft (N x K), and per
// group the expected width (exp_bits, may be null) and the hardened width
// (hard, may be null). gumbel may be null (no noise).
cudaError_t launch_soft_quant(const float* w, const float* logits, const float* gumbel, float tau, int64_t N,
                              int64_t K, float* w_soft, float* exp_bits, uint8_t* hard, cudaStream_t s);

// Batches of 2..GEMV1_MAX_B rows may run on the batch-1 table kernel, two
// rows per launch; tables_for_batch (vbq_plan.cu) says whether the layout's
// width mix makes that cheaper than the tensor-core kernel.
constexpr int GEMV1_MAX_B = 4;
bool tables_for_batch(const LayoutView& L, int B);

// Layouts planned so that the batch-1 product can run one unit per block, a row
// block's S slabs a cluster (gemv1_unit_kernel, vbq_gemv.cu): units of at most
// 8 columns (a wider unit's 2048 groups on one block's 16 warps take longer
// than the hand-over saves: 4096x4096 as 128 16-column units 4.6 -> 5.1 us),
// clusters of at most 16 blocks, every cluster resident at once (two blocks
// per SM, less what clusters leave unused of a GPC's SMs: 276..296 blocks fit
// for up to 8 slabs, 196..253 above; in several waves of clusters 14336x4096
// takes 8.3 -> 10.9 us), and fewer than 200,000 groups (below).
constexpr int MAX_CLUSTER = 16;
constexpr int64_t UNIT_MAX_GROUPS = 200000;
inline bool unit_plan_fits(int64_t C, int64_t S, int64_t units, int64_t groups, int sms) {
    return C <= 8 && S <= MAX_CLUSTER && groups < UNIT_MAX_GROUPS && 4 * units <= (S <= 8 ? 7 : 5) * (int64_t)sms;
}
// Whether it does run them so. The unit kernel gains where its neighbours on
// the stream are unit kernels too, whose blocks share SMs with it; next to a
// persistent block of 226 KB its clusters wait for whole SMs. A ~9B layer's
// fused products (4096x4096, 262,144 groups, between 6144x4096 and
// 28672x4096) take 36.9 us with 4096x4096 on the persistent kernel and 39.0 on
// this one, and its 1024x4096 products among 4096x4096 ones cost the unfused
// layer 0.5 us; a ~1B layer, of which only the down projection (2048x5632) stays
// off it, takes 22.8 instead of 26.1. So a matrix stays off it when it, or a
// square matrix on its input, has 200,000 groups or more: K stands for what the
// neighbours are like, which a call cannot see (a single 1024x4096 product, or
// one among small ones, is kept off it too).
inline bool unit_neighbours(int64_t G) { return GROUP * G * G < UNIT_MAX_GROUPS; }
inline bool runs_unit_per_block(const LayoutView& L, int sms) {
    return unit_neighbours(L.G) && unit_plan_fits(L.C, L.S, L.units, L.N * L.G, sms);
}

// Products (vbq_gemv.cu). Y is B x N, overwritten (no zeroing needed).
cudaError_t launch_gemv(const LayoutView& L, const uint16_t* X, float* Y, int B, cudaStream_t s);

// How a batch-1 launch orders itself against the previous kernel on its
// stream (programmatic dependent launch):
//   DEP_BEFORE       lets the next kernel launch at once, then waits for the
//                    previous kernel before touching x, y or control words
//                    (every product call: x may be the previous output);
//   DEP_GROUP_FIRST  waits first, then lets the next kernel launch, so the
//                    rest of a group starts only after earlier stream work;
//   DEP_GROUP_NEXT   lets the next kernel launch and works without waiting
//                    (its inputs predate the group), then waits for the
//                    previous kernel before it completes, so kernels still
//                    complete in stream order.
enum Dep : int { DEP_BEFORE = 0, DEP_GROUP_FIRST = 1, DEP_GROUP_NEXT = 2 };

// count independent batch-1 products (distinct layouts and outputs) as one
// group: launch i > 0 overlaps the tail of launch i - 1.
cudaError_t launch_gemv_group(const LayoutView* const* Ls, const uint16_t* const* xs, float* const* ys, int count,
                              cudaStream_t s);

// Batch 1 on a gate-up matrix whose rows alternate (gate i, up i) with the
// SwiGLU epilogue: y (N floats) as launch_gemv writes it, and h (N/2 BF16 bit
// patterns) = silu(gate) * up. Uses the layout's slab counts (control words
// 2 + nrb ..) when a row spans several slabs.
cudaError_t launch_gemv_swiglu(const LayoutView& L, const uint16_t* x, float* y, uint16_t* h, cudaStream_t s);

// Batch 1 whose activations are h_k = silu(gu[2k]) * gu[2k + 1], computed in
// fp32 while the activation tables are built (gu: 2K floats, the y of a
// gate-up product with alternating rows); h never reaches memory.
cudaError_t launch_gemv_swiglu_in(const LayoutView& L, const float* gu, float* y, cudaStream_t s);

// A chain of count batch-1 products in one persistent launch of blocks
// blocks (every product's ChainItem::rot computed for that count). cctl:
// 3 + count zero-initialised words owned by the chain (call counter, one
// completion count per product, then the count of blocks that have zeroed
// their split-K rows).
cudaError_t launch_chain(const ChainItem* items, int count, uint32_t* cctl, int blocks, cudaStream_t s);
int device_sms(int* sms);   // the current device's SM count (0 on success)

// Batch 1 with the split-K control words in a fixed device array (no
// allocation anywhere); usable for layouts with at most STATIC_CTL_WORDS - 2
// row blocks.
constexpr int STATIC_CTL_WORDS = 2 + 8192;
cudaError_t launch_gemv1_static(const LayoutView& L, const uint16_t* x, float* y, cudaStream_t s);

// Batch 2..16 on the tensor cores (vbq_gemm.cu); Y is B x N, overwritten.
cudaError_t launch_gemm_small(const LayoutView& L, const uint16_t* X, float* Y, int B, cudaStream_t s);

// Bounded-wait report: synchronise s, read and clear the device status words
// of both product files (nonzero when some wait gave up); and the self-test
// that makes one wait run out after limit_ns.
cudaError_t read_device_status(uint32_t* status, cudaStream_t s);
cudaError_t read_device_status_gemm(uint32_t* status);
cudaError_t launch_selftest_timeout(unsigned long long limit_ns, cudaStream_t s);

}  // namespace vbq
