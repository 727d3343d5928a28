// Step 1 of the module (Section 3.1: Q = xW_Q, K = xW_K, V = xW_V) on the 5th-generation tensor cores, writing
// channel-blocked planes:  y[b][o / d][n / 8][o % d][n % 8] = sum_c w[o][c] * x[b][c][n],  fp32 accumulate.
//
// The product is taken with output channels as MMA rows and tokens as columns: A = weights (K-major), B = the x tile
// straight from NCHW (tokens contiguous: an MN-major operand).  A lane of tensor memory is then one output channel and a
// thread reads eight neighbouring tokens of it in a row, i.e. one 16-byte piece of the layout; the 32 lanes of a warp
// are the channels of one plane (d = 16: of two), so 8 tokens are 512 contiguous bytes and 32 tokens one bulk copy.
//
// Persistent CTAs, one per SM, warp-specialised: warp 0 issues the copies, warp 1 the MMAs, warps 2-9 drain the
// accumulators (two sets, so that the drain of a tile overlaps the MMAs of the next).  A CTA serves one block of
// 128 * HALVES output channels for its whole life and streams 128-token tiles of x.
//   HALVES = 2: 256 weight rows resident in shared memory (K <= 256): x is read once per 256 output channels
//   HALVES = 1: 128 rows resident (K <= 512); also taken where 256-row blocks would leave SMs without work
//   STREAM    : weights too large to stay (K > 512): their k-slices go through the ring beside x's
// HBM-bound at large sizes: it writes three bytes for every byte it reads.  Every wait is bounded.
#include <cuda.h>

#include "msla_common.cuh"
#include "msla_host.h"
#include "tma_host.h"
#include "tcgen05_util.cuh"

namespace msla {
namespace {

using bf16 = __nv_bfloat16;

constexpr int PP_TOK = 128, PP_BK = 64;
constexpr int PP_X_STAGE = PP_TOK * PP_BK * 2;       // 16 KB: two boxes of 64 tokens x 64 channels
constexpr int PP_W_SLICE = 128 * PP_BK * 2;          // 16 KB: 128 weight rows x 64 channels
constexpr int PP_THREADS = 320;
constexpr int PP_STAGING_WARP = 2 * 2048;            // two blocks of 32 channels x 32 tokens
constexpr int PP_STAGING = 8 * PP_STAGING_WARP;
constexpr int PP_MAX_STAGES = 8;
constexpr int PP_BAR_BYTES = 256;
constexpr int PP_SMEM_LIMIT = 226 * 1024;

__device__ int g_pp_timeout_flag = 0;

struct ProjPlanesParams {
  int Np, K, Cout, d;       // tokens per image (a multiple of 8), channels in, channels out, channels per plane
  int tok_tiles, tiles;     // 128-token tiles per image, and of all images
  int blocks, workers;      // output-channel blocks; CTAs per block
  int stages;
  long long out_sb;         // elements between images of the output
  bf16* out;
};

template <int HALVES, bool STREAM, bool F16>
__global__ void __launch_bounds__(PP_THREADS, 1)
project_planes_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW, ProjPlanesParams p) {
  constexpr int STAGE = PP_X_STAGE + (STREAM ? PP_W_SLICE : 0);
  constexpr int ROWS = 128 * HALVES;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;  // swizzle atoms need 1024-byte alignment
  const int k_iters = (p.K + PP_BK - 1) / PP_BK;
  const uint32_t ring = smem_base + (STREAM ? 0u : (uint32_t)(k_iters * HALVES * PP_W_SLICE));
  const uint32_t staging = ring + (uint32_t)(p.stages * STAGE);
  const uint32_t bars = staging + PP_STAGING;
  const uint32_t full_bar = bars, empty_bar = bars + 8 * PP_MAX_STAGES;
  const uint32_t tfull_bar = bars + 16 * PP_MAX_STAGES, tempty_bar = tfull_bar + 16;
  const uint32_t res_bar = tempty_bar + 16, tmem_slot = res_bar + 8;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blk = blockIdx.x % p.blocks, worker = blockIdx.x / p.blocks;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < p.stages; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar + 8 * a, 1); mbar_init(tempty_bar + 8 * a, 8); }
    mbar_init(res_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (threadIdx.x == 0) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(tmem_slot));
    tmem_base_sh = v;
  }
  __syncthreads();
  const uint32_t tmem_base = tmem_base_sh;

  if (warp == 0) {
    // ------------------------------------------------------------ copies
    if (lane == 0) {
      pdl_first_wait();
      if (!STREAM) {
        mbar_expect_tx(res_bar, (uint32_t)(k_iters * HALVES * PP_W_SLICE));
        for (int kb = 0; kb < k_iters; ++kb) tma_load_3d(smem_base + kb * (HALVES * PP_W_SLICE), &tmW, res_bar, kb * PP_BK, blk * ROWS, 0);
      }
      uint32_t s = 0, ph = 0;
      bool ok = true;
      for (int tile = worker; ok && tile < p.tiles; tile += p.workers) {
        const int b = tile / p.tok_tiles, n0 = (tile - b * p.tok_tiles) * PP_TOK;
        for (int kb = 0; ok && kb < k_iters; ++kb) {
          ok = mbar_wait(empty_bar + 8 * s, ph ^ 1, &abort_flag);
          if (!ok) break;
          const uint32_t dst = ring + s * STAGE;
          mbar_expect_tx(full_bar + 8 * s, STAGE);
          tma_load_3d(dst, &tmX, full_bar + 8 * s, n0, kb * PP_BK, b);
          tma_load_3d(dst + PP_X_STAGE / 2, &tmX, full_bar + 8 * s, n0 + 64, kb * PP_BK, b);
          if (STREAM) tma_load_3d(dst + PP_X_STAGE, &tmW, full_bar + 8 * s, kb * PP_BK, blk * ROWS, 0);
          if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      // instruction descriptor: D = f32, A K-major, B MN-major, N = 128 tokens, M = 128 channels
      const uint32_t idesc = (1u << 4) | (F16 ? 0u : ((1u << 7) | (1u << 10))) | (1u << 16) | ((uint32_t)(PP_TOK >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      uint32_t s = 0, ph = 0, local = 0;
      bool ok = STREAM || mbar_wait(res_bar, 0, &abort_flag);
      for (int tile = worker; ok && tile < p.tiles; tile += p.workers, ++local) {
        const uint32_t acc = local & 1, acc_ph = (local >> 1) & 1;
        ok = mbar_wait(tempty_bar + 8 * acc, acc_ph ^ 1, &abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * (HALVES * PP_TOK);
        for (int kb = 0; ok && kb < k_iters; ++kb) {
          ok = mbar_wait(full_bar + 8 * s, ph, &abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint32_t xs = ring + s * STAGE, ws = STREAM ? xs + PP_X_STAGE : smem_base + kb * (HALVES * PP_W_SLICE);
#pragma unroll
          for (int kk = 0; kk < PP_BK / 16; ++kk) {
            const uint64_t bd = make_desc(xs + kk * 2048, (PP_X_STAGE / 2) >> 4, 1024 >> 4);
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf)
              umma_bf16(d_tmem + hf * PP_TOK, make_desc(ws + hf * PP_W_SLICE + kk * 32, 1, 1024 >> 4), bd, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
          }
          umma_commit(empty_bar + 8 * s);
          if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1; }
        }
        if (ok) umma_commit(tfull_bar + 8 * acc);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // warp % 4 selects the tensor-memory lanes (a hardware rule); the other bit the half of the block's channels
    // (HALVES = 2) or of the tile's tokens
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const int ch0 = blk * ROWS + (HALVES == 2 ? part * 128 : 0) + quarter * 32;
    const uint32_t stage = staging + (uint32_t)(warp - 2) * PP_STAGING_WARP;
    const uint32_t lane_off = p.d == 32 ? (uint32_t)lane * 16u : (uint32_t)((lane >> 4) * 1024 + (lane & 15) * 16);
    const uint32_t octet = (uint32_t)p.d * 16u;  // bytes of eight tokens of a plane
    constexpr int CHUNKS = HALVES == 2 ? 4 : 2;  // of 32 tokens
    uint32_t local = 0, nbuf = 0;
    bool ok = true;
    pdl_wait();  // no global write before the previous kernel is done with the output buffer
    for (int tile = worker; ok && tile < p.tiles; tile += p.workers, ++local) {
      const int b = tile / p.tok_tiles, n_tile = (tile - b * p.tok_tiles) * PP_TOK + (HALVES == 2 ? 0 : part * 64);
      const uint32_t acc = local & 1, acc_ph = (local >> 1) & 1;
      ok = mbar_wait(tfull_bar + 8 * acc, acc_ph, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + acc * (HALVES * PP_TOK) + (uint32_t)(part * (HALVES == 2 ? PP_TOK : 64)) + ((uint32_t)(quarter * 32) << 16);
      uint32_t r[2][32];
      tmem_ld32(taddr, r[0]);
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        tmem_ld_wait();
        if (c + 1 < CHUNKS) tmem_ld32(taddr + (c + 1) * 32, r[(c + 1) & 1]);  // next chunk streams in meanwhile
        const uint32_t(&rc)[32] = r[c & 1];
        const int n0 = n_tile + c * 32;
        if (n0 >= p.Np || ch0 >= p.Cout) continue;  // warp-uniform
        const uint32_t buf = stage + (nbuf & 1) * 2048u;
        ++nbuf;
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");  // the block stored from this buffer before has been read
        __syncwarp();
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float lo = __uint_as_float(rc[8 * v + 2 * e]), hi = __uint_as_float(rc[8 * v + 2 * e + 1]);
            if constexpr (F16) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(w[e]) : "f"(hi), "f"(lo));
            else w[e] = pack2(lo, hi);
          }
          asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(buf + lane_off + v * octet), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          const uint32_t bytes = (uint32_t)(min(32, p.Np - n0) * p.d * 2);
          bf16* dst = p.out + (long long)b * p.out_sb + ((long long)(ch0 / p.d) * p.Np + n0) * p.d;
          asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(buf), "r"(bytes) : "memory");
          if (p.d == 16 && ch0 + 16 < p.Cout)
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst + (long long)p.Np * 16), "r"(buf + 1024), "r"(bytes) : "memory");
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty_bar + 8 * acc);
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  tc_fence_before();
  __syncthreads();
  if (abort_flag) {
    for (int i = 0; i < 64; ++i) __nanosleep(1000);  // copies and MMAs still in flight land before memory is released
    if (threadIdx.x == 0) atomicExch(&g_pp_timeout_flag, 1);
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

template <int HALVES, bool STREAM, bool F16>
msla_status_t launch_pp(const CUtensorMap& tmX, const CUtensorMap& tmW, ProjPlanesParams p, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done{0};
  const msla_status_t s = ensure_smem_attr(attr_done, project_planes_kernel<HALVES, STREAM, F16>, PP_SMEM_LIMIT);
  if (s != MSLA_OK) return s;
  const int k_iters = (p.K + PP_BK - 1) / PP_BK;
  const int fixed = (STREAM ? 0 : k_iters * HALVES * PP_W_SLICE) + PP_STAGING + PP_BAR_BYTES + 1024;
  constexpr int STAGE = PP_X_STAGE + (STREAM ? PP_W_SLICE : 0);
  p.stages = (PP_SMEM_LIMIT - fixed) / STAGE;
  if (p.stages > PP_MAX_STAGES) p.stages = PP_MAX_STAGES;
  p.blocks = (p.Cout + 128 * HALVES - 1) / (128 * HALVES);
  p.workers = device_sm_count() / p.blocks;
  if (p.workers < 1) p.workers = 1;
  if (p.workers > p.tiles) p.workers = p.tiles;
  launch_pdl(project_planes_kernel<HALVES, STREAM, F16>, dim3((unsigned)(p.blocks * p.workers)), dim3(PP_THREADS), (size_t)(fixed + p.stages * STAGE), st, tmX, tmW, p);
  count_launches(1);
  return check_launch("input projection (tcgen05, channel-blocked planes)");
}

}  // namespace

// x: [B][C][Np] 16-bit, Np a multiple of 8; w: [Cout][C]; y: planes [Np / 8][d][8], image stride y_sb elements.
msla_status_t run_project_planes(const void* x, const void* w, void* y, int B, int C, int Cout, int Np, int d, long long y_sb, cudaStream_t st, bool f16) {
  ProjPlanesParams p{};
  p.Np = Np; p.K = C; p.Cout = Cout; p.d = d;
  p.tok_tiles = (Np + PP_TOK - 1) / PP_TOK;
  const long long tiles = (long long)B * p.tok_tiles;
  if (tiles > 0x7fffffffLL) return fail(MSLA_ERR_UNSUPPORTED, "too many token tiles");
  p.tiles = (int)tiles;
  p.out_sb = y_sb; p.out = (bf16*)y;
  // 256 resident rows re-read x half as often; 128 rows where K does not allow them or where they leave SMs idle
  const long long work2 = (long long)p.tiles * ((Cout + 255) / 256);
  const int halves = C <= 256 && work2 >= device_sm_count() ? 2 : 1;
  CUtensorMap tmX, tmW;
  const cuuint64_t dx[3] = {(cuuint64_t)Np, (cuuint64_t)C, (cuuint64_t)B}, dw[3] = {(cuuint64_t)C, (cuuint64_t)Cout, 1};
  const cuuint64_t sx[2] = {(cuuint64_t)Np * 2, (cuuint64_t)C * Np * 2}, sw[2] = {(cuuint64_t)C * 2, (cuuint64_t)C * Cout * 2};
  const cuuint32_t bx[3] = {64, PP_BK, 1}, bw[3] = {PP_BK, (cuuint32_t)(128 * halves), 1};
  if (!tma_make_map_bf16(&tmX, x, 3, dx, sx, bx, CU_TENSOR_MAP_SWIZZLE_128B) || !tma_make_map_bf16(&tmW, w, 3, dw, sw, bw, CU_TENSOR_MAP_SWIZZLE_128B))
    return fail(MSLA_ERR_CUDA, "cuTensorMapEncodeTiled failed for the input projection");
  if (halves == 2) return f16 ? launch_pp<2, false, true>(tmX, tmW, p, st) : launch_pp<2, false, false>(tmX, tmW, p, st);
  if (C <= 512) return f16 ? launch_pp<1, false, true>(tmX, tmW, p, st) : launch_pp<1, false, false>(tmX, tmW, p, st);
  return f16 ? launch_pp<1, true, true>(tmX, tmW, p, st) : launch_pp<1, true, false>(tmX, tmW, p, st);
}

int project_planes_timeout_flag() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_pp_timeout_flag, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return v;
}

}  // namespace msla
