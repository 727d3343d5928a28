// Host-side declarations shared by the translation units of libmsla.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <atomic>

#include "../../include/msla.h"

namespace msla {

// Carving of the attention core's scratch: fp32 partial states
// [BH][S][d*(d+1)] at partial_off, combined states [BH][d*(d+1)] at state_off.
struct CorePlan {
  int S;       // number of token chunks per (batch, head)
  int chunk;   // tokens per chunk (multiple of 64)
  int ne;      // d*(d+1) state entries
  int apply_tokens;  // tokens per CTA of the tuned apply kernel (multiple of 128)
  size_t partial_off, state_off, bytes;
};

CorePlan make_core_plan(long long BH, int N, int d);

// Records a thread-local message and returns `st`.
msla_status_t fail(msla_status_t st, const char* fmt, ...);
// MSLA_OK, or MSLA_ERR_CUDA if a launch since the last check failed.
msla_status_t check_launch(const char* what);

void count_launches(int n);

// Function attributes (the dynamic shared-memory limit) belong to one device: a launch site keeps an
// atomic mask of the devices on which it has set them.  Bit of the current device; 0 for device numbers
// past 63, which makes the site set the attribute on every call there.
inline unsigned long long current_device_bit() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
  return (dev >= 0 && dev < 64) ? 1ull << dev : 0ull;
}

// Raises the dynamic shared-memory limit of `kernel` to `bytes` on the current device, once per device
// (two threads racing on the first call both set it, which is harmless).
template <typename Kernel>
inline msla_status_t ensure_smem_attr(std::atomic<unsigned long long>& done, Kernel kernel, int bytes) {
  const unsigned long long bit = current_device_bit();
  if (bit && (done.load(std::memory_order_acquire) & bit)) return MSLA_OK;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
    cudaGetLastError();
    return fail(MSLA_ERR_CUDA, "cannot reserve %d bytes of shared memory for a kernel", bytes);
  }
  done.fetch_or(bit, std::memory_order_release);
  return MSLA_OK;
}

// Number of SMs of the current device (looked up once per device).
int device_sm_count();

// Launches `kernel` with programmatic stream serialization allowed: it may become resident before the
// previous kernel of the stream has finished, and orders itself with pdl_wait() (msla_common.cuh).
template <typename... KArgs, typename... Args>
inline void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);  // errors surface in check_launch()
}

// The same for a kernel that runs as clusters of two CTAs (grid.x must be even).
template <typename... KArgs, typename... Args>
inline void launch_pdl_cluster2(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);  // errors surface in check_launch()
}

struct HeadView;
// Tuned attention core for 16-bit storage, bf16 or (f16 = true) fp16 (d in {16, 32}); all view strides must be multiples of 8 elements.
// `phases` selects what runs: CORE_STATE the partial states (at ws + p.partial_off, p.S per head), CORE_COMBINE their
// fixed-order sum (at ws + p.state_off), CORE_APPLY the apply step reading that sum; without CORE_APPLY `out` and `ov` are unused.
enum : int { CORE_STATE = 1, CORE_COMBINE = 2, CORE_APPLY = 4, CORE_ALL = 7 };
msla_status_t run_core_bf16(const void* q, const void* k, const void* v, void* out, HeadView in, HeadView ov, int B,
                            int heads, int N, int d, float eps, const CorePlan& p, void* ws, cudaStream_t st,
                            cudaEvent_t mid, int phases, bool f16 = false);

// FFN with a depthwise convolution (gemm_tcgen05.cu, ffn_dw_bf16.cu): bf16; the hidden tensor is planes of 32 channels
// [B][Ch / 32][N][32] after the first layer, planes of 64 channels [B][Ch / 64][N][64] after the depthwise convolution.
// act: 0 none, 1 ReLU, 2 hard-swish.
bool ffn_bf16_supported(int C, int Ch, int Cout);
// ldx, ldy: elements between rows (tokens of one channel) of x, and of y and the residual; multiples of 8, as tensor maps need.
// first: first kernel of a call (msla_common.cuh).
msla_status_t run_ffn_expand_bf16(const void* x, int ldx, const void* w1, const void* b1, void* h, int B, int C, int Ch, int N, int act,
                                  cudaStream_t st, bool f16, bool first);
msla_status_t run_ffn_dw3x3_bf16(const void* h, const void* w_dw, const void* b_dw, void* g, int B, int Ch, int H, int W, int act,
                                 cudaStream_t st, bool f16 = false);
msla_status_t run_ffn_project_bf16(const void* g, const void* w2, const void* b2, const void* residual, void* y, int ldy, int B, int Ch,
                                   int Cout, int N, cudaStream_t st, bool f16 = false);

// Apply step and output projection as one GEMM per image (fused_out.cu): bf16, d in {16, 32}, at most 512 attention
// channels and 256 output channels.  q: planar query matrices [N][d], head h of image b at q + b*q_sb + h*q_sh
// (elements).
bool fused_out_bf16_supported(int Ht, int d, int Cout);
size_t fused_out_scratch_bytes(int B, int Ht, int d, int Cout);
int fused_timeout_flag();
int dw_timeout_flag();

// bf16 projections on tcgen05 tensor cores (gemm_tcgen05.cu).
bool project_in_bf16_supported(int C, int Cout, int ldx, int d);
msla_status_t run_project_in_bf16(const void* x, int ldx, const void* w, void* y, int B, int C, int Cout, int N, int d,
                                  long long y_batch_stride, cudaStream_t st, bool f16, bool first);
bool project_out_bf16_supported(int Cin, int Cout, int ldy);
// residual: nullptr, or a tensor shaped like y that is added to it
msla_status_t run_project_out_bf16(const void* a, const void* w, const void* bias, const void* residual, void* y, int ldy, int B, int Cin,
                                   int Cout, int N, cudaStream_t st, bool f16, bool first);
bool project_out_planar_bf16_supported(int Cin, int Cout);
msla_status_t run_project_out_planar_bf16(const void* a, const void* w, const void* bias, const void* residual, void* y, int ldy, int B,
                                          int Cin, int Cout, int N, cudaStream_t st, bool f16 = false);
int gemm_timeout_flag();

// fp32 projections on tensor cores (gemm_f32_split.cu); K a multiple of 8, 16-byte aligned tensors.
msla_status_t run_project_in_split(const float* x, const float* w, float* y, int B, int C, int Cout, int N, int d, long long y_sb, cudaStream_t st, bool first);
msla_status_t run_project_out_split(const float* a, bool token_major, const float* w, const float* bias, int act, const float* residual, float* y, int B, int K,
                                    int Cout, int N, cudaStream_t st, bool first);
int split_gemm_timeout_flag();
int run_wait_selftest(long long limit_cycles, int* scratch, cudaStream_t st);

// bf16 aggregation (d = 16 or 32, Ch a multiple of 32): TMA halo tiles, depthwise filter as banded matrices on
// tensor cores (agg_bf16.cu).  weights_ready: an earlier kernel of the call has waited, and none of its wrote w_dw.  dst_sb must be a multiple of the plane size H*W*d.
bool aggregate_bf16_supported(int H, int W, int Ch, int d);
msla_status_t run_aggregate_bf16(const void* src, long long src_planes_total, int src_ppb, const void* w_dw,
                                 const void* w_pw, void* dst, long long dst_sb, int B, int H, int W, int Ch, int d,
                                 cudaStream_t st, bool f16, bool weights_ready);
int agg_timeout_flag();

// Rows of n 16-bit elements to and from rows `pitch` (a multiple of 8) elements apart (repack.cu).
msla_status_t run_pad_rows(const void* src, void* dst, long long rows, int n, int pitch, cudaStream_t st);
msla_status_t run_unpad_rows(const void* src, void* dst, long long rows, int n, int pitch, cudaStream_t st);

// ---- The 16-bit module path on channel-blocked planes: a plane (q, k or v of one head) is [H][W / 8][d][8], W a multiple of 8,
// i.e. eight horizontally neighbouring pixels of one channel are 16 contiguous bytes.
//
// Aggregation and state sums (agg_state.cu).  The grid's CTAs take contiguous runs of tiles, of equal cost; CTA c writes the
// part of segment s (a pair of blocks of one image: s = pair * B + image) that it summed to slot s + c (unique, because both
// grow along the list of tiles).  The runs are cut for `batch` images; a call that has images first .. first + B - 1 of them takes
// those tiles of every run, so that its sums are added as the whole batch adds them.
constexpr int AGG_STATE_CTAS = 148;
struct AggStatePlan {
  int kv_tiles_x, q_tiles_x, tiles_y, grid, slot_floats, kv_cost, q_cost, batch, first;
  long long kv_tiles, kv_units, cost;  // kv_units, cost: of the batch
  size_t partial_bytes;
};
AggStatePlan make_agg_state_plan(int B, int heads, int H, int W, int d, int batch, int first);
// First tile of CTA c; the CTA that has key/value tile u.
__host__ __device__ inline long long agg_state_first_unit(long long cost, int kv_cost, int q_cost, long long kv_units, long long c, long long grid) {
  const long long at = cost * c / grid, kv = kv_cost * kv_units;
  return at < kv ? (at + kv_cost - 1) / kv_cost : kv_units + (at - kv + q_cost - 1) / q_cost;
}
__host__ __device__ inline long long agg_state_cta_of(long long cost, int kv_cost, long long u, long long grid) { return (grid * (kv_cost * u + 1) - 1) / cost; }
// Tiles of the batch's list before `u` (`tiles` per plane; pair of blocks, image, tile) that belong to images first .. first + B - 1.
__host__ __device__ inline long long agg_state_part_units(long long u, long long tiles, int batch, int first, int B) {
  const long long pb = u / tiles, pair = pb / batch, b = pb - pair * batch - first;
  return b < 0 ? pair * B * tiles : b >= B ? (pair + 1) * B * tiles : (pair * B + b) * tiles + (u - pb * tiles);
}
// ms0: [B][3*heads] planes; q1: [B][heads] planes; rows [row_lo, row_hi) count in the states.
msla_status_t run_agg_state(const void* ms0, void* q1, float* partial, const void* w_dw, const void* w_pw, const AggStatePlan& plan, int B,
                            int heads, int H, int W, int d, int row_lo, int row_hi, bool with_scale0, cudaStream_t st, bool f16);
int agg_state_timeout_flag();

// Input projection into scale-0 planes (proj_planes.cu), the first kernel of its call: x [B][C][Np], Np a multiple of 8.
msla_status_t run_project_planes(const void* x, const void* w, void* y, int B, int C, int Cout, int Np, int d, long long y_sb, cudaStream_t st, bool f16);
int project_planes_timeout_flag();

// Where the partial states lie that the fold adds: [B*Ht][S][d][d+1] (slots.grid == 0), or the slots of the aggregation launches,
// one per aggregated branch, with the grouped 1x1 weights whose value rows are still to be applied.
struct FoldStates {
  const float* partial;
  int S;
  const float* slots[2];
  const void* w_pw[2];
  AggStatePlan plan;
};
// Queries of all scales in channel-blocked planes: query head h of image b at scale 0 is plane (b*heads + h)*3 of q0, at branch s
// plane ((s-1)*B + b)*heads + h of q1.
struct PlanesQueries {
  const void *q0, *q1;
  int heads;                            // per scale
  long long plane_tokens, first_token;  // tokens of a plane; first one used (a multiple of 8)
};
// Fold and fused output kernel (see above); planes: nullptr, or the query planes that take the place of q.
msla_status_t run_fused_out_bf16(const void* q, long long q_sb, long long q_sh, const PlanesQueries* planes, const FoldStates& states, void* scratch,
                                 const void* w, const void* bias, const void* residual, void* y, int ldy, int B, int Ht, int d, int N, int Cout,
                                 float eps, cudaStream_t st, bool f16 = false);
// The sum of the partial states [B*Ht][d][d+1] (planes path where steps 4 and 5 stay apart, and bands).
msla_status_t run_sum_states(const FoldStates& in, float* state_out, int B, int heads, int Ht, int d, cudaStream_t st, bool f16);
// The apply step on such planes; att token-major or paired planes (ov).  sum_tokens: tokens the states were summed over.
msla_status_t run_apply_planes(const PlanesQueries& q, const float* state, void* att, HeadView ov, int B, int Ht, int N, int d, float eps,
                               long long sum_tokens, cudaStream_t st, bool f16);

}  // namespace msla
