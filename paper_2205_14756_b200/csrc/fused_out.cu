// Steps 4 and 5 of the module (Section 3.1: apply step of Eq. 3, head concat,
// final linear projection) as one tensor-core GEMM per image.
//
// Eq. 3 gives, for head h and token n,  O_h[n][c] = sum_a relu(q_h[n][a]) S_h[a][c] / den_h[n]
// with den_h[n] = sum_a relu(q_h[n][a]) ks_h[a] + eps, and the projection is
// y[m][n] = sum_h sum_c w[m][h*d + c] O_h[n][c] + bias[m].  Re-associating the two sums,
//
//   y[m][n] = sum_h sum_a  M[m][h*d + a] * qt[h*d + a][n]  + bias[m],
//   M[m][h*d + a] = sum_c w[m][h*d + c] S_h[a][c]          (per image, C_out x 2C', tiny)
//   qt[h*d + a][n] = relu(q_h[n][a]) / den_h[n]            (the queries, scaled per head and token)
//
// which is exact in real arithmetic: the d x d contraction of the apply step moves
// from every token into the small matrix M, and what is left per token and head is
// one d-term dot product (the normaliser) and a scaling.  M and qt are rounded to
// bf16 where the unfused path rounds S and O.
//
// state_fold_kernel : sums the partial states in index order (fixed order, so the result
//                     is reproducible bit for bit), writes ks and M (fp32 accumulate, bf16 out).
// fused_out_kernel  : clusters of two CTAs, paired tensor-core MMAs (cta_group::2, M = 256).
//   Each CTA keeps its 128 rows of M (<= 128 KB) in shared memory while the image lasts and
//   owns 128 of the pair's 256 tokens per tile.  The unit handed from role to role is a pair of
//   heads (two slices of d query channels in one ring slot, one set of barriers): the thread that
//   issues the MMAs pays a wait and a commit per unit, and its serial chain is what bounds the kernel.
//     warp 0       TMA: per unit one box of 2 heads x 128 tokens x d channels of the heads' planar [N][d]
//                  query matrices (contiguous 8 KB pieces for d = 32; swizzle span = the row)
//     warps 2-13   turn q into qt in place (normaliser on the fp32 pipes, one token per lane);
//                  three groups of four warps, each taking every third slice
//     warp 1       loads the rows of M and the key sums; in the leader CTA issues tcgen05.mma 256 x 256 x 16: A = M,
//                  B = qt, both K-major, fp32 accumulators in both CTAs' tensor memory
//     warps 14-17  drain the accumulators: TMEM -> bf16 (+ bias) -> swizzled staging -> TMA
//                  stores of 32-channel x 64-token blocks into the NCHW output
//                  (RES kernels: the same block of a residual tensor, fetched by TMA into a block of its own one
//                  block ahead of its use, is added before the conversion: the residual connection around the module)
//   Two accumulator sets (2 x 256 TMEM columns) let the drain of a tile overlap the next.
//   A small problem (one tile of 64 tokens per CTA) is the latency of this chain: six transform groups of two warps, a ring that
//   holds every unit, one copy per unit and M requested by a warp of its own took [1, 256, 32, 32] from 24.7 to 23.8 us a
//   forward, [1, 192, 64, 128] from 30.6 to 29.8, f16 [8, 128, 45, 80] from 50.2 to 49.4.  Waiting for M slice by slice is slower (25.1):
//   the waits lengthen the issuing thread's chain.
// Queries come in one of two layouts: planes [token][d] (above), or (PL) channel-blocked planes [token / 8][d][8], where eight
// tokens of one channel are 16 contiguous bytes.  PL kernels fetch a head's 128 tokens by one bulk copy (contiguous in the
// plane); a transform warp takes 32 tokens through ldmatrix.trans, which gives a lane the same two channels of every channel
// octet for four tokens, the four lanes of a token add their parts of the normaliser, and stmatrix.trans puts the scaled queries
// back; the MMA reads them as they lie (tokens contiguous: an MN-major operand of 8 x 8 core matrices without swizzle).
// No TMA load is multicast: each CTA loads its own operands; only tcgen05.commit signals
// both CTAs' barriers.  Every mbarrier wait is bounded as in the GEMM.
#include <cuda.h>

#include "msla_common.cuh"
#include "msla_host.h"
#include "tma_host.h"
#include "tcgen05_util.cuh"

namespace msla {
namespace {

using bf16 = __nv_bfloat16;

constexpr int OT = 128;                  // tokens per CTA and tile (256 per pair); 64 where that spreads a small problem over more pairs
constexpr int OM = 128;                  // output channels per CTA (256 per pair)
constexpr int OKS = 64;                  // k-extent of one resident slice of M (one 128-byte swizzle span)
constexpr int O_A_SLICE = OM * OKS * 2;  // 16 KB: 128 rows of M x 64 k
constexpr int O_MAX_KS = 8;              // K = 2C' <= 512
constexpr int O_MIN_STAGES = 2, O_MAX_STAGES = 16;  // query ring: as many slots (of two slices each) as shared memory holds (the host decides)
constexpr int O_XWARPS = 12;             // transform warps: three groups of four, each taking every third slice
constexpr int O_THREADS = 32 * (2 + O_XWARPS + 4);
constexpr int O_STAGING_WARP = 32 * 128;
constexpr int O_STAGING = 4 * O_STAGING_WARP;
constexpr int O_BAR_BYTES = 512;
constexpr int O_KS_BYTES = O_MAX_KS * OKS * 4;  // the image's key sums
constexpr int O_SMEM_FIXED = O_STAGING + O_BAR_BYTES + O_KS_BYTES;  // besides the rows of M, the ring and the residual blocks
constexpr int O_SMEM_LIMIT = 227 * 1024;                     // all of it dynamic
static_assert(24 * O_MAX_STAGES + 16 + 16 + 8 + 8 + 8 + 4 * 8 + 8 + 8 + 8 + 8 <= O_BAR_BYTES, "barrier block");

__device__ int g_fused_timeout_flag = 0;

struct OutParams {
  const unsigned char *q0, *q1;      // PL: see PlanesQueries (msla_host.h)
  long long plane_bytes, tok_bytes;  // PL: bytes of a plane; offset of the first token inside it
  int heads;                         // PL: heads per scale
  const float* ks;   // [B][Ht][d] key sums
  const bf16* bias;  // [Cout] or nullptr
  const bf16* residual;  // RES kernels: [B][Cout][N], added to the output (the residual connection around the module)
  int B, N, Cout, Ht, d;
  int kslices;       // 64-wide k-slices of M: ceil(Ht * d / 64)
  int ot;            // tokens per CTA and tile: 128 or 64
  int stages;        // slots of the query ring (a slot holds the slices of two consecutive heads)
  int tiles_per_image, num_tiles;  // tiles of 2 * ot tokens
  float eps;
};

// ---- cluster helpers
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {  // shared::cta address -> shared::cluster address in CTA `rank`
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P1;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, P1;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait on a barrier that other CTAs of the cluster (or tcgen05.commit) arrive on.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait_cluster(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > WAIT_LIMIT_CYCLES) {
      *abort_flag = 1;
      return false;
    }
  }
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// K-major shared-memory matrix descriptor whose swizzle span is the row: rows of 64 bytes (mode 4) or 32 bytes (mode 6);
// sbo16 = distance between groups of 8 rows in 16-byte units.
__device__ __forceinline__ uint64_t make_desc_kmajor(uint32_t addr, uint32_t sbo16, uint64_t mode) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)sbo16 << 32) | (1ull << 46) | (mode << 61);
}
// Descriptor of an MN-major operand without swizzle: core matrices of 8 k x 8 tokens (16-byte rows, 128 contiguous bytes);
// lbo16 = distance between groups of 8 k, sbo16 = between groups of 8 tokens, in 16-byte units.
__device__ __forceinline__ uint64_t make_desc_octets(uint32_t addr, uint32_t lbo16, uint32_t sbo16) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)lbo16 << 16) | ((uint64_t)sbo16 << 32) | (1ull << 46);
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void umma2_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrives (once the MMAs issued so far have completed) on the barrier at this shared-memory offset in both CTAs of the pair.
__device__ __forceinline__ void umma2_commit_both(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((unsigned short)3) : "memory");
}

// F16 kernels: the 16-bit storage type is IEEE binary16 instead of bfloat16.  The values travel untyped; the conversions,
// the packed maximum and the MMA's operand format differ.
template <bool F16> __device__ __forceinline__ float lo16(uint32_t w) {
  if constexpr (F16) return __low2float(*reinterpret_cast<const __half2*>(&w));
  else return __uint_as_float(w << 16);
}
template <bool F16> __device__ __forceinline__ float hi16(uint32_t w) {
  if constexpr (F16) return __high2float(*reinterpret_cast<const __half2*>(&w));
  else return __uint_as_float(w & 0xffff0000u);
}
template <bool F16> __device__ __forceinline__ uint32_t pack16(float lo, float hi) {
  if constexpr (F16) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
  } else {
    return pack2(lo, hi);
  }
}

// F16: two queries times their key sums and the reciprocal of the normaliser, the products of both in one instruction each.
__device__ __forceinline__ uint32_t scale_pair(uint32_t w, float k0, float k1, float inv) {
  float lo = lo16<true>(w), hi = hi16<true>(w);
  asm("{\n\t.reg .b64 q, k, i;\n\tmov.b64 q, {%0, %1};\n\tmov.b64 k, {%2, %3};\n\tmov.b64 i, {%4, %4};\n\t"
      "mul.rn.f32x2 q, q, k;\n\tmul.rn.f32x2 q, q, i;\n\tmov.b64 {%0, %1}, q;\n\t}" : "+f"(lo), "+f"(hi) : "f"(k0), "f"(k1), "f"(inv));
  return pack16<true>(lo, hi);
}

// ---------------------------------------------------------------------------
// Second level of the state reduction (Eq. 3) and the fold of the state into the projection weights.
// Grid (B * Ht, D / DA): a CTA takes one head and DA of its key channels a, i.e. DA consecutive rows of the head's state.
// partial: [B*Ht][S][D*(D+1)] fp32, entry [a][c], column D = key sum.
//   ks[bh][a]            = sum_s partial[bh][s][a][D]
//   M[b][m][hh*D + a]    = sum_c w[m][hh*D + c] * (sum_s partial[bh][s][a][c])        (16 bit, row stride K), all m < Cout
// SLOTS: the partial states are the slots that the aggregation's CTAs wrote (msla_host.h, AggStatePlan): a contiguous run of
// them, and those of aggregated scales still lack the grouped 1x1 of the values, S[a][c] = sum_c' Wv[c][c'] (sum_s ..)[a][c'].
// With M == nullptr the states go to state_out [B*Ht][D][D+1] instead.
// Fixed summation order, the same for every DA: the S partial states are cut into eight runs of consecutive indices, each run
// is summed in index order (eight 16-byte loads in flight) and the run sums are added in run order.  With few heads every run
// has threads of its own, otherwise a thread sums FOLD_RUNS / GROUPS of them.
// The product runs on mma.sync with output channels as rows, key channels as columns and c along the contraction.  The
// weights are 16-bit already; the fp32 state is cut into PIECES 16-bit pieces (bf16: three, which hold all 24 bits; fp16:
// two, 22 bits of a value that is rounded to 11).  Contraction slots and columns are assigned so that a lane loads 16
// consecutive bytes of a weight row (8 for D = 16) and, where the CTA has whole rows of M (DA = D), stores as many.
// Latency bounds it with few heads (one memory round trip, two barriers), the write of M with many.  Against the version
// that did the product on the fp32 pipes with 1024 threads per CTA: 1024 heads (64 images, S = 1) 73.4 -> 13.7 us, 256
// heads 22.9 -> 6.4 us, 16 heads (S = 37) 7.0 -> 4.3 us.
// ---------------------------------------------------------------------------
constexpr int FOLD_RUNS = 8;
template <int D, int DA> struct FoldShape {
  static constexpr int GROUPS = DA == 8 ? 8 : DA * D >= 1024 ? 1 : 4;  // threads that share the runs of a vector
  static constexpr int NV = DA * (D + 1) / 4;                       // 16-byte vectors of the CTA's rows of a state
  static constexpr int THREADS = (NV * GROUPS + 31) / 32 * 32;        // 288, 544, 544 for D = 32 and DA = 32, 16, 8; 288 for D = 16
};

template <bool F16>
__device__ __forceinline__ void fold_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  if constexpr (F16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// F16: row a of the state is divided by its key sum (0 where that is 0), and the output kernel multiplies its queries by it,
//   M[m][hd + a] = sum_c w[m][hd + c] S_h[a][c] / ks_h[a],   qt[hd + a][n] = relu(q_h[n][a]) ks_h[a] / den_h[n] <= 1,
// so that both stay inside binary16's range whatever N and the key sums are.  relu(q) / den alone does not: where the keys have nothing
// above zero in the channels that a query has, den is eps, and infinity times the zero column of M is not a number.
struct FoldParams {
  const float* partial;      // [B*Ht][S][D][D+1]
  int S;
  const float* slots[2];     // SLOTS: per aggregated branch (the first also carries scale 0)
  const bf16* w_pw[2];       // SLOTS: the branches' grouped 1x1 weights
  int slot_floats, grid, kv_cost, batch, first_image;  // SLOTS: of the aggregation
  long long tiles, cost;
  const bf16* w;             // projection weights [Cout][K]
  bf16* M;
  float *ks, *state_out;
  int B, heads, Ht, Cout, K;
};
template <int D, int DA, bool F16, bool SLOTS>
__global__ void __launch_bounds__(FoldShape<D, DA>::THREADS, DA == D ? 4 : 1)
state_fold_kernel(FoldParams p) {
  constexpr int GROUPS = FoldShape<D, DA>::GROUPS, NV = FoldShape<D, DA>::NV, THREADS = FoldShape<D, DA>::THREADS;
  constexpr int D1 = D + 1, NE4 = D * D1 / 4, WARPS = THREADS / 32;
  constexpr int KS = D / 16, NT = DA / 8, PIECES = F16 ? 2 : 3;
  __shared__ float4 run_sum[GROUPS == 1 ? 1 : FOLD_RUNS][NV];
  __shared__ uint32_t rounded[PIECES][DA][D / 2 + 1];  // pairs of neighbouring c
  __shared__ float wv[SLOTS ? D : 1][D + 1];           // SLOTS: Wv transposed, [c'][c]
  float* st = reinterpret_cast<float*>(run_sum[0]);
  pdl_launch_dependents();
  const int Ht = p.Ht, Cout = p.Cout, K = p.K;
  const bf16* w = p.w;
  const int bh = blockIdx.x, b = bh / Ht, hh = bh % Ht, a0 = blockIdx.y * DA;
  const int branch = SLOTS ? hh / p.heads : 0, h = SLOTS ? hh - branch * p.heads : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  // A fragments of 16 output channels: lane (g, t) holds c = t*D/4 .. + D/4 - 1 of rows g and g + 8
  auto load_weights = [&](int m0, uint32_t (&x)[2][D / 8]) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const bf16* src = w + (long long)(m0 + g + 8 * r) * K + hh * D + t * (D / 4);
      const bool ok = m0 + g + 8 * r < Cout;
      if constexpr (D == 32) {
        const uint4 v = ok ? __ldg(reinterpret_cast<const uint4*>(src)) : make_uint4(0u, 0u, 0u, 0u);
        x[r][0] = v.x; x[r][1] = v.y; x[r][2] = v.z; x[r][3] = v.w;
      } else {
        const uint2 v = ok ? __ldg(reinterpret_cast<const uint2*>(src)) : make_uint2(0u, 0u);
        x[r][0] = v.x; x[r][1] = v.y;
      }
    }
  };
  uint32_t x[2][D / 8];
  // the weights do not come from the previous kernel: fetched while it drains; the partial states do
  if (p.M) load_weights(16 * warp, x);
  if (SLOTS && branch > 0) {
    const bf16* src = (branch == 2 ? p.w_pw[1] : p.w_pw[0]) + (long long)(3 * h + 2) * D * D;
    for (int i = tid; i < D * D / 2; i += THREADS) {
      const uint32_t v = __ldg(reinterpret_cast<const uint32_t*>(src) + i);
      const int c = i / (D / 2), k = i % (D / 2) * 2;
      wv[k][c] = lo16<F16>(v);
      wv[k + 1][c] = hi16<F16>(v);
    }
  }
  pdl_wait();
  int S = p.S;
  long long stride4 = NE4;
  const float* first = p.partial + (long long)bh * S * (D * D1);
  if constexpr (SLOTS) {
    constexpr int HPB = 32 / D;  // heads per slot
    const long long seg = (long long)(h / HPB) * p.B + b, of_batch = (long long)(h / HPB) * p.batch + p.first_image + b;
    const long long c0 = agg_state_cta_of(p.cost, p.kv_cost, of_batch * p.tiles, p.grid), c1 = agg_state_cta_of(p.cost, p.kv_cost, (of_batch + 1) * p.tiles - 1, p.grid);
    S = (int)(c1 - c0) + 1;
    stride4 = p.slot_floats / 4;
    first = (branch == 2 ? p.slots[1] : p.slots[0]) + (seg + c0) * p.slot_floats + ((h % HPB) * 2 + (branch > 0 ? 1 : 0)) * (D * D1);
  }
  const float4* sp = reinterpret_cast<const float4*>(first + a0 * D1);
  auto add = [](float4& v, const float4& x) { v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w; };
  if (tid < GROUPS * NV) {
    const int group = tid / NV, e = tid - group * NV;
    float4 total = make_float4(0.f, 0.f, 0.f, 0.f);
    if (GROUPS == 1 && S <= 8) {  // a run has one partial state or none
      float4 q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = u < S ? ld_dep128f(sp + u * stride4 + e) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) add(total, q[u]);
    } else {
#pragma unroll 1
      for (int j = group * (FOLD_RUNS / GROUPS); j < (group + 1) * (FOLD_RUNS / GROUPS); ++j) {
        const int s0 = S * j / FOLD_RUNS, s1 = S * (j + 1) / FOLD_RUNS;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = s0; s < s1; s += 8) {
          float4 q[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) q[u] = s + u < s1 ? ld_dep128f(sp + (s + u) * stride4 + e) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int u = 0; u < 8; ++u) add(v, q[u]);
        }
        if (GROUPS == 1) add(total, v);
        else run_sum[j][e] = v;
      }
    }
    if (GROUPS == 1) run_sum[0][e] = total;
  }
  __syncthreads();
  if (GROUPS > 1) {
    if (tid < NV) {
      float4 v = run_sum[0][tid];
#pragma unroll
      for (int j = 1; j < FOLD_RUNS; ++j) add(v, run_sum[j][tid]);
      run_sum[0][tid] = v;  // st[al * D1 + c], al = a - a0
    }
    __syncthreads();
  }
  if (SLOTS && branch > 0) {  // the grouped 1x1 of the values: an entry of the CTA's rows per thread and round
    constexpr int PER = (DA * D + THREADS - 1) / THREADS;
    float mixed[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int i = tid + r * THREADS, al = i / D, c = i % D;
      float v = 0.f;
      if (i < DA * D) {
#pragma unroll
        for (int k = 0; k < D; ++k) v = fmaf(wv[k][c], st[al * D1 + k], v);
      }
      mixed[r] = v;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int i = tid + r * THREADS;
      if (i < DA * D) st[i / D * D1 + i % D] = mixed[r];
    }
    __syncthreads();
  }
  if (!p.M) {
    for (int i = tid; i < DA * D1; i += THREADS) p.state_out[(long long)bh * (D * D1) + a0 * D1 + i] = st[i];
    return;
  }
  if (tid < DA) p.ks[(long long)bh * D + a0 + tid] = st[tid * D1 + D];
  for (int i = tid; i < DA * D / 2; i += THREADS) {
    const int al = i / (D / 2), c2 = i - al * (D / 2);
    float v0 = st[al * D1 + 2 * c2], v1 = st[al * D1 + 2 * c2 + 1];
    if (F16) {
      const float sum = st[al * D1 + D], r = sum > 0.f ? 1.f / sum : 0.f;
      v0 *= r; v1 *= r;
    }
#pragma unroll
    for (int k = 0; k < PIECES; ++k) {
      const uint32_t word = pack16<F16>(v0, v1);
      rounded[k][al][c2] = word;
      v0 -= lo16<F16>(word); v1 -= hi16<F16>(word);
    }
  }
  __syncthreads();
  // B fragments: column g of tile j is key channel al(j), contraction slots of step i: c = t*D/4 + 4*i + {0 .. 3}; read when
  // they are needed (held for the whole loop they cost 48 registers, and two of four CTAs per SM)
  const uint32_t pieces = smem_u32(&rounded[0][0][0]) + (uint32_t)((DA == D ? (g >> 1) * (D / 4) + (g & 1) : g) * (D / 2 + 1) + t * (D / 8)) * 4u;
  for (int m0 = 16 * warp; m0 < Cout; m0 += 16 * WARPS) {
    if (m0 != 16 * warp) load_weights(m0, x);
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
#pragma unroll
      for (int k = PIECES - 1; k >= 0; --k)  // small pieces first
#pragma unroll
        for (int i = 0; i < KS; ++i) {
          const uint32_t A[4] = {x[0][2 * i], x[1][2 * i], x[0][2 * i + 1], x[1][2 * i + 1]};
          const uint32_t at = pieces + (uint32_t)((k * DA + (DA == D ? 2 : 8) * j) * (D / 2 + 1) + 2 * i) * 4u;
          uint32_t b0, b1;
          asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b0) : "r"(at));
          asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b1) : "r"(at + 4));
          fold_mma<F16>(acc[j], A, b0, b1);
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int m = m0 + g + 8 * r;
      if (m >= Cout) continue;
      bf16* row = p.M + ((long long)b * Cout + m) * K + hh * D + a0;
      if constexpr (DA == D) {
        uint32_t o[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) o[j] = pack16<F16>(acc[j][2 * r], acc[j][2 * r + 1]);
        if constexpr (D == 32) *reinterpret_cast<uint4*>(row + 8 * t) = make_uint4(o[0], o[1], o[2], o[3]);
        else *reinterpret_cast<uint2*>(row + 4 * t) = make_uint2(o[0], o[1]);
      } else {
#pragma unroll
        for (int j = 0; j < NT; ++j) *reinterpret_cast<uint32_t*>(row + 8 * j + 2 * t) = pack16<F16>(acc[j][2 * r], acc[j][2 * r + 1]);
      }
    }
  }
}

template <int D, bool RES, bool F16, bool PL>
__global__ void __launch_bounds__(O_THREADS, 1)
fused_out_kernel(const __grid_constant__ CUtensorMap tmM, const __grid_constant__ CUtensorMap tmQ,
                 const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmR, OutParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];  // swizzle atoms need 1024-byte alignment
  const uint32_t smem_base = smem_u32(smem_raw);
  const uint32_t a_base = smem_base;                                  // resident rows of M: kslices x 16 KB
  const uint32_t SLICE = (uint32_t)p.ot * D * 2;                       // one head's queries of this CTA's tokens
  const uint32_t SLOT = 2 * SLICE;                                     // ring slot: two consecutive heads
  constexpr int ROWB = D * 2;                                          // bytes per token row = the swizzle span (not PL)
  const int xwarps = p.ot / 32;                                        // transform warps per group: one token per lane
  constexpr int OCTET = D * 16;                                        // PL: bytes of eight tokens
  const uint32_t ring = a_base + (uint32_t)p.kslices * O_A_SLICE;
  const uint32_t staging = ring + (uint32_t)p.stages * SLOT;
  const uint32_t resbuf = staging + O_STAGING;           // RES: one 32-channel x 64-token block of the residual per epilogue warp
  const uint32_t bars = resbuf + (RES ? O_STAGING : 0);
  const uint32_t full_bar = bars;                        // [stage] both heads' boxes landed (own CTA)
  const uint32_t empty_bar = bars + 8 * O_MAX_STAGES;        // [stage] MMAs have read the slice (commit, both CTAs)
  const uint32_t ready_bar = bars + 16 * O_MAX_STAGES;       // [stage] both CTAs' slices transformed (leader only)
  const uint32_t tfull_bar = bars + 24 * O_MAX_STAGES;       // [acc] accumulator complete (commit, both CTAs)
  const uint32_t tempty_bar = tfull_bar + 16;            // [acc] both CTAs' epilogues have drained it (leader only)
  const uint32_t res_bar = tempty_bar + 16;              // rows of M landed (own CTA)
  const uint32_t peer_res_bar = res_bar + 8;             // the peer's rows of M landed (leader only)
  const uint32_t tmem_slot = peer_res_bar + 8;
  const uint32_t resid_bar = tmem_slot + 8;              // [epilogue warp] RES: the warp's residual block landed
  const uint32_t mfree_bar = resid_bar + 32;             // the MMAs of an image are complete: its rows of M may be replaced (commit, both CTAs)
  const uint32_t ks_bar = mfree_bar + 8;                 // the image's key sums landed (own CTA)
  const uint32_t ks_sm = bars + O_BAR_BYTES;
  const uint32_t kseen_bar = ks_bar + 8;                 // every transform warp has seen the image's key sums land (own CTA)
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + (kseen_bar + 8 - smem_base));

  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();               // 0 = leader of the pair
  // A pair works on a run of consecutive tiles, so that it changes image (and reloads its rows of M) as seldom as possible.
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int tiles_per_pair = (p.num_tiles + npairs - 1) / npairs;
  const int tile_first = min(pair * tiles_per_pair, p.num_tiles), tile_end = min(tile_first + tiles_per_pair, p.num_tiles);

  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(full_bar + 8 * s, 1);
      mbar_init(empty_bar + 8 * s, 1);
      mbar_init(ready_bar + 8 * s, 2 * 2 * xwarps);  // per head the warps of one transform group, in both CTAs
    }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar + 8 * a, 1); mbar_init(tempty_bar + 8 * a, 2 * 4); }
    mbar_init(res_bar, 1);
    mbar_init(peer_res_bar, 1);
    mbar_init(mfree_bar, 1);
    mbar_init(ks_bar, 1);
    mbar_init(kseen_bar, O_XWARPS);
    if (RES)
      for (int w = 0; w < 4; ++w) mbar_init(resid_bar + 8 * w, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {  // one warp of each CTA of the pair: all 512 tensor-memory columns in both
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_sync_all();  // both CTAs' barriers exist before anything arrives on them from the other CTA
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));
  pdl_wait();  // queries, states and M come from earlier kernels

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (each CTA for itself)
    if (lane == 0) {
      if (!PL) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmQ) : "memory");
      uint32_t s = 0, ph = 0;  // ring slot and the parity of its current use
      bool ok = true;
      for (int tile = tile_first; ok && tile < tile_end; ++tile) {
        const int b = tile / p.tiles_per_image, nt = tile % p.tiles_per_image;
        const int n0 = nt * (2 * p.ot) + (int)rank * p.ot;
        for (int h = 0; ok && h < p.Ht; h += 2) {
          ok = mbar_wait_cluster(empty_bar + 8 * s, ph ^ 1, abort_flag);
          if (!ok) break;
          if constexpr (PL) {
            const bool two = h + 1 < p.Ht;  // an odd head count leaves the last slot half used
            // tokens past the last one are not copied: their accumulator columns are never stored
            const uint32_t bytes = (uint32_t)max(0, min(p.ot, p.N - n0)) * (D * 2);
            auto query = [&](int hq) -> const unsigned char* {
              const int sc = hq / p.heads, hd = hq - sc * p.heads;
              const unsigned char* plane = sc == 0 ? p.q0 + ((long long)b * p.heads + hd) * 3 * p.plane_bytes
                                                   : p.q1 + (((long long)(sc - 1) * p.B + b) * p.heads + hd) * p.plane_bytes;
              return plane + p.tok_bytes + (long long)n0 * (D * 2);
            };
            mbar_expect_tx(full_bar + 8 * s, (two ? 2u : 1u) * bytes);
            if (bytes) {
              bulk_load(ring + s * SLOT, query(h), bytes, full_bar + 8 * s);
              if (two) bulk_load(ring + s * SLOT + SLICE, query(h + 1), bytes, full_bar + 8 * s);
            }
          } else {  // one box of two heads; rows past the last token (and the head past an odd count) are filled with zeros
            mbar_expect_tx(full_bar + 8 * s, SLOT);
            tma_load_4d(ring + s * SLOT, &tmQ, full_bar + 8 * s, 0, n0, h, b);
          }
          if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ rows of M and key sums (each CTA for itself), MMA issuer (leader)
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmM) : "memory");
      // instruction descriptor: D = f32, A = B = bf16, both K-major (PL: B MN-major), N = 256, M = 256 (pair)
      const uint32_t idesc = (1u << 4) | (F16 ? 0u : ((1u << 7) | (1u << 10))) | (PL ? 1u << 16 : 0u) | ((uint32_t)((2 * p.ot) >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      const uint32_t peer_res_remote = map_to_cta(peer_res_bar, 0);
      uint32_t local = 0, res_ph = 0, mfree_ph = 0, s = 0, ph = 0;  // s, ph: ring slot and the parity of its current use
      // Matrix descriptors: the high words are constants; the low words carry the start address in 16-byte units
      // (A: the 128B-swizzled rows of M; B: the slice, K-major, the swizzle span being the token row).
      const uint64_t a_hi = make_desc(0, 1, 1024 >> 4), b_hi = PL ? make_desc_octets(0, 128 >> 4, OCTET >> 4) : make_desc_kmajor(0, (8 * ROWB) >> 4, D == 32 ? 4ull : 6ull);
      const uint32_t a_lo0 = (a_base & 0x3FFFFu) >> 4, b_lo0 = (ring & 0x3FFFFu) >> 4;
      int cur_b = -1;
      bool ok = true;
      for (int tile = tile_first; ok && tile < tile_end; ++tile, ++local) {
        const int b = tile / p.tiles_per_image;
        if (b != cur_b) {
          if (cur_b >= 0) {
            // Every MMA that reads the previous image's rows of M must be complete (and with them every scaling that reads its key
            // sums).  The accumulators' barriers cannot tell: a parity two phases back looks complete.
            ok = mbar_wait_cluster(mfree_bar, mfree_ph, abort_flag);
            if (!ok) break;
            // Nor does a group of transform warps that took no slice of that image (two heads, one tile) hold anything back: without its
            // sign-off it could find ks_bar a phase further on, and wait for good.
            ok = mbar_wait(kseen_bar, mfree_ph, abort_flag);
            if (!ok) break;
            mfree_ph ^= 1;
          }
          cur_b = b;
          mbar_expect_tx(ks_bar, (uint32_t)(p.Ht * D * 4));
          bulk_load(ks_sm, p.ks + (long long)b * p.Ht * D, (uint32_t)(p.Ht * D * 4), ks_bar);
          mbar_expect_tx(res_bar, (uint32_t)(p.kslices * O_A_SLICE));
          for (int ks = 0; ks < p.kslices; ++ks) tma_load_3d(a_base + ks * O_A_SLICE, &tmM, res_bar, ks * OKS, (int)rank * OM, b);
          ok = mbar_wait(res_bar, res_ph, abort_flag);  // own rows of M
          if (!ok) break;
          if (rank == 0) {
            ok = mbar_wait_cluster(peer_res_bar, res_ph, abort_flag);  // the peer's rows of M
            if (!ok) break;
          } else {
            mbar_arrive_cluster(peer_res_remote);
          }
          res_ph ^= 1;
        }
        if (rank != 0) continue;
        const uint32_t acc = local & 1, acc_ph = (local >> 1) & 1;
        ok = mbar_wait_cluster(tempty_bar + 8 * acc, acc_ph ^ 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * 256;
        uint32_t a_lo = a_lo0;  // the unit's columns of M: 32 bytes per 16 columns, 64-column slices O_A_SLICE apart
        for (int h = 0; ok && h < p.Ht; h += 2) {
          ok = mbar_wait_cluster(ready_bar + 8 * s, ph, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint32_t b_lo = b_lo0 + s * (SLOT >> 4);
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            umma2_bf16(d_tmem, a_hi | (a_lo + 2u * kk), b_hi | (b_lo + (PL ? 16u : 2u) * kk), idesc, (h > 0 || kk > 0) ? 1u : 0u);
          if (h + 1 < p.Ht) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              umma2_bf16(d_tmem, a_hi | (a_lo + 2u * (D / 16 + kk)), b_hi | (b_lo + (SLICE >> 4) + (PL ? 16u : 2u) * kk), idesc, 1u);
          }
          // two heads of 32 fill a 64-column slice, two heads of 16 half of one
          a_lo += D == 32 || (h & 2) ? (uint32_t)((O_A_SLICE - (D == 32 ? 0 : 64)) >> 4) : 4u;
          umma2_commit_both(empty_bar + 8 * s);  // both CTAs may refill the slot once these MMAs have read it
          if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1; }
        }
        if (ok) umma2_commit_both(tfull_bar + 8 * acc);
        if (ok && tile + 1 < tile_end && (tile + 1) / p.tiles_per_image != b) umma2_commit_both(mfree_bar);
      }
    }
  } else if (warp < 2 + O_XWARPS) {
    // ------------------------------------------------------------ transform warps: q -> relu(q) / den, in place
    // Groups of as many warps as a CTA's tile has token rows for (three groups of four, or six of two) take the slices in
    // turn, starting with slice xg; a lane owns one token row (d channels: 64 or 32 bytes, 16-byte pieces XOR-swizzled with
    // the row as the TMA unit wrote them and as the MMA reads them; eight consecutive rows cover all banks once).
    constexpr int PCS = D / 8;     // 16-byte pieces per token row
    const int xw = warp - 2, xg = xw / xwarps, wig = xw - xg * xwarps, groups = O_XWARPS / xwarps;
    const uint32_t ready_remote = map_to_cta(ready_bar, 0);
    const uint32_t row = (uint32_t)(wig * 32 + lane);
    const uint32_t swz = D == 32 ? (row >> 1) & 3u : (row >> 2) & 1u;
    const uint32_t row_off = row * ROWB;
    uint32_t s = 0, ph = 0, turn = 0;  // ring slot, the parity of its current use, and the group whose turn it is
    const int h_end = (p.Ht + 1) & ~1;  // an odd head count: the empty half of the last slot still has to be signed off
    uint32_t ks_ph = 0;
    int cur_b = -1;
    bool ok = true;
    for (int tile = tile_first; ok && tile < tile_end; ++tile) {
      const int b = tile / p.tiles_per_image;
      if (b != cur_b) {
        cur_b = b;
        ok = mbar_wait(ks_bar, ks_ph, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        ks_ph ^= 1;
        if (lane == 0) mbar_arrive(kseen_bar);
      }
      for (int h = 0; ok && h < h_end; ++h) {
        const uint32_t cs = s, cph = ph;  // this slice's slot; the counters move on to the next slice
        const bool mine = (int)turn == xg;
        if (h & 1) { if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1; } }
        if ((int)++turn == groups) turn = 0;
        if (!mine) continue;
        if constexpr (PL) {
          constexpr int CB = D / 8;  // channel octets; register (o, cb) of lane (g, t) holds channels 8 cb + 2t, + 1 of token 8 o + g
          const int t = lane & 3;
          float2 kk[CB];  // the lane's key sums
          const uint32_t ksp = ks_sm + (uint32_t)(min(h, p.Ht - 1) * D + 2 * t) * 4u;
#pragma unroll
          for (int cb = 0; cb < CB; ++cb) asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(kk[cb].x), "=f"(kk[cb].y) : "r"(ksp + 32u * cb));
          ok = mbar_wait(full_bar + 8 * cs, cph, abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (h >= p.Ht) {
            if (lane == 0) mbar_arrive_cluster(ready_remote + 8 * cs);
            continue;
          }
          const uint32_t base = ring + cs * SLOT + (uint32_t)(h & 1) * SLICE + (uint32_t)(wig * 4 * OCTET + lane * 16);
          uint32_t q[4 * CB];  // q[o * CB + cb]
#pragma unroll
          for (int i = 0; i < CB; ++i)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(q[4 * i]), "=r"(q[4 * i + 1]), "=r"(q[4 * i + 2]), "=r"(q[4 * i + 3]) : "r"(base + i * 512) : "memory");
          float den[4];
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            float d0 = 0.f, d1 = 0.f;
#pragma unroll
            for (int cb = 0; cb < CB; ++cb) {
              uint32_t& w = q[o * CB + cb];
              if constexpr (F16) asm("max.f16x2 %0, %1, %2;" : "=r"(w) : "r"(w), "r"(0u));
              else asm("max.bf16x2 %0, %1, %2;" : "=r"(w) : "r"(w), "r"(0u));
              d0 = fmaf(lo16<F16>(w), kk[cb].x, d0);
              d1 = fmaf(hi16<F16>(w), kk[cb].y, d1);
            }
            den[o] = d0 + d1;
          }
          // sum over the four lanes of a token; lane t ends up with octet 2 (t & 1) + (t >> 1)
          const bool odd = t & 1, up = t & 2;
          const float k0 = (odd ? den[2] : den[0]) + __shfl_xor_sync(0xffffffffu, odd ? den[0] : den[2], 1);
          const float k1 = (odd ? den[3] : den[1]) + __shfl_xor_sync(0xffffffffu, odd ? den[1] : den[3], 1);
          const float tot = (up ? k1 : k0) + __shfl_xor_sync(0xffffffffu, up ? k0 : k1, 2);
          const float inv = __frcp_rn(tot + p.eps);
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            const float io = __shfl_sync(0xffffffffu, inv, (lane & ~3) | (o >> 1) | ((o & 1) << 1));
#pragma unroll
            for (int cb = 0; cb < CB; ++cb) {
              uint32_t& w = q[o * CB + cb];
              w = F16 ? scale_pair(w, kk[cb].x, kk[cb].y, io) : pack16<F16>(lo16<F16>(w) * io, hi16<F16>(w) * io);
            }
          }
#pragma unroll
          for (int i = 0; i < CB; ++i)
            asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(base + i * 512), "r"(q[4 * i]), "r"(q[4 * i + 1]),
                         "r"(q[4 * i + 2]), "r"(q[4 * i + 3]) : "memory");
        } else {
        float kk[D];  // the head's key sums
        const uint32_t ksp = ks_sm + (uint32_t)(min(h, p.Ht - 1) * D) * 4u;
#pragma unroll
        for (int a4 = 0; a4 < D / 4; ++a4)
          asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(kk[4 * a4]), "=f"(kk[4 * a4 + 1]), "=f"(kk[4 * a4 + 2]), "=f"(kk[4 * a4 + 3]) : "r"(ksp + 16u * a4));
        ok = mbar_wait(full_bar + 8 * cs, cph, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const uint32_t rbase = ring + cs * SLOT + (uint32_t)(h & 1) * SLICE + row_off;
        if (h >= p.Ht) {
          if (lane == 0) mbar_arrive_cluster(ready_remote + 8 * cs);
          continue;
        }
        uint32_t q[D / 2];  // word w = channels 2w (low half), 2w+1 (high half)
#pragma unroll
        for (int c = 0; c < PCS; ++c)
          asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(q[4 * c]), "=r"(q[4 * c + 1]), "=r"(q[4 * c + 2]), "=r"(q[4 * c + 3])
                       : "r"(rbase + (((uint32_t)c ^ swz) << 4)));
        float den[4] = {0.f, 0.f, 0.f, 0.f};  // four chains
#pragma unroll
        for (int w = 0; w < D / 2; ++w) {
          if constexpr (F16) asm("max.f16x2 %0, %1, %2;" : "=r"(q[w]) : "r"(q[w]), "r"(0u));
          else asm("max.bf16x2 %0, %1, %2;" : "=r"(q[w]) : "r"(q[w]), "r"(0u));
          den[2 * (w & 1)] = fmaf(lo16<F16>(q[w]), kk[2 * w], den[2 * (w & 1)]);
          den[2 * (w & 1) + 1] = fmaf(hi16<F16>(q[w]), kk[2 * w + 1], den[2 * (w & 1) + 1]);
        }
        const float inv = __frcp_rn((den[0] + den[1]) + (den[2] + den[3]) + p.eps);
#pragma unroll
        for (int w = 0; w < D / 2; ++w)
          q[w] = F16 ? scale_pair(q[w], kk[2 * w], kk[2 * w + 1], inv) : pack16<F16>(lo16<F16>(q[w]) * inv, hi16<F16>(q[w]) * inv);
#pragma unroll
        for (int c = 0; c < PCS; ++c)
          asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(rbase + (((uint32_t)c ^ swz) << 4)), "r"(q[4 * c]), "r"(q[4 * c + 1]),
                       "r"(q[4 * c + 2]), "r"(q[4 * c + 3]) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the tensor cores read what was just written
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(ready_remote + 8 * cs);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // Four warps; warp % 4 selects the TMEM lane quarter (a hardware rule).  A lane owns one output
    // channel of this CTA's 128; the accumulator's 256 columns are the pair's 256 tokens.
    const int quarter = warp & 3;
    const uint32_t stage = staging + (uint32_t)(warp - 2 - O_XWARPS) * O_STAGING_WARP;
    const uint32_t my_row = stage + lane * 128, sw = (uint32_t)(lane & 7);
    const int row0 = (int)rank * OM + quarter * 32;
    const float bias = !(p.bias && row0 + lane < p.Cout) ? 0.f : F16 ? __half2float(reinterpret_cast<const __half*>(p.bias)[row0 + lane]) : __bfloat162float(p.bias[row0 + lane]);
    const uint32_t tempty_remote = map_to_cta(tempty_bar, 0);
    // RES: the residual arrives by TMA, one 32-channel x 64-token block per warp and request, a block ahead of its use
    const uint32_t my_resid_bar = resid_bar + 8 * (uint32_t)(warp - 2 - O_XWARPS);
    const uint32_t my_res = resbuf + (uint32_t)(warp - 2 - O_XWARPS) * O_STAGING_WARP, my_res_row = my_res + lane * 128;
    uint32_t res_count = 0;
    auto request_residual = [&](int t2, int j2) {  // one lane
      mbar_expect_tx(my_resid_bar, O_STAGING_WARP);
      tma_load_3d(my_res, &tmR, my_resid_bar, (t2 % p.tiles_per_image) * (2 * p.ot) + j2 * 64, row0, t2 / p.tiles_per_image);
    };
    if (RES && lane == 0 && row0 < p.Cout && tile_first < tile_end) request_residual(tile_first, 0);
    uint32_t local = 0;
    bool ok = true;
    for (int tile = tile_first; ok && tile < tile_end; ++tile, ++local) {
      const int b = tile / p.tiles_per_image, nt = tile % p.tiles_per_image;
      const uint32_t acc = local & 1, acc_ph = (local >> 1) & 1;
      ok = mbar_wait_cluster(tfull_bar + 8 * acc, acc_ph, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + acc * 256 + ((uint32_t)(quarter * 32) << 16);
      uint32_t r[2][32];
      tmem_ld32(taddr, r[0]);
      const int chunks = (2 * p.ot) / 32;  // the accumulator's columns are the pair's tokens
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (c >= chunks) break;
        tmem_ld_wait();
        if (c + 1 < chunks) tmem_ld32(taddr + (c + 1) * 32, r[(c + 1) & 1]);  // next chunk streams in meanwhile
        const uint32_t(&rc)[32] = r[c & 1];
        const int n0 = nt * (2 * p.ot) + (c >> 1) * 64;  // first token of the 64-token block
        if (n0 >= p.N || row0 >= p.Cout) continue;    // warp-uniform
        if ((c & 1) == 0) {  // the previous block must have been read out of the staging buffer
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          __syncwarp();
          if (RES) {           // this block of the residual was requested one block ago
            ok = mbar_wait(my_resid_bar, res_count & 1, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            ++res_count;
          }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const uint32_t pc = (uint32_t)((c & 1) * 4 + v);
          uint4 rv = make_uint4(0u, 0u, 0u, 0u);  // the same 16-byte piece of the lane's row in the residual block (same box, same swizzle)
          if (RES) asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(rv.x), "=r"(rv.y), "=r"(rv.z), "=r"(rv.w) : "r"(my_res_row + ((pc ^ sw) << 4)));
          const uint32_t rw[4] = {rv.x, rv.y, rv.z, rv.w};
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float f0 = __uint_as_float(rc[v * 8 + 2 * e]) + bias, f1 = __uint_as_float(rc[v * 8 + 2 * e + 1]) + bias;
            if (RES) { f0 += lo16<F16>(rw[e]); f1 += hi16<F16>(rw[e]); }
            w[e] = pack16<F16>(f0, f1);
          }
          asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(my_row + ((pc ^ sw) << 4)), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                       "r"(w[3]) : "memory");
        }
        if (c & 1) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // also orders the reads of the residual block before its refill
          __syncwarp();
          if (lane == 0) {
            tma_store_3d(&tmO, stage, n0, row0, b);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            if (RES) {  // request the next block this warp will drain: the next 64 tokens of this tile, else the next tile's first
              int t2 = tile, j2 = (c >> 1) + 1;
              if (j2 * 64 >= 2 * p.ot || (t2 % p.tiles_per_image) * (2 * p.ot) + j2 * 64 >= p.N) { ++t2; j2 = 0; }
              if (t2 < tile_end) request_residual(t2, j2);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty_remote + 8 * acc);  // this warp's quarter of the accumulator is drained
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // stores done before the CTA retires
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies and MMAs still in flight time to land before memory is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    if (threadIdx.x == 0) atomicExch(&g_fused_timeout_flag, 1);
    __syncthreads();
  }
  cluster_sync_all();  // neither CTA leaves (or frees tensor memory) while the other may still touch its barriers or shared memory
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

}  // namespace

bool fused_out_bf16_supported(int Ht, int d, int Cout) {
  return (d == 16 || d == 32) && Ht >= 1 && Ht * d <= O_MAX_KS * OKS && Cout >= 1 && Cout <= 2 * OM && Cout % 8 == 0;
}

// Scratch: M [B][Cout][Ht*d] bf16, then ks [B][Ht][d] fp32 (256-byte aligned).
static size_t fused_out_m_bytes(int B, int Ht, int d, int Cout) { return ((size_t)B * Cout * Ht * d * 2 + 255) / 256 * 256; }
size_t fused_out_scratch_bytes(int B, int Ht, int d, int Cout) { return fused_out_m_bytes(B, Ht, d, Cout) + (size_t)B * Ht * d * sizeof(float); }

// y[b][m][n] = sum_h sum_c w[m][h*d + c] * att[b][h][n][c] + bias[m], att = Eq. 3 applied to query head h with the
// state of (b, h) = sum over s < S of partial[(b * Ht + h) * S + s] ([d][d+1] fp32 each: KV, then the key sum in
// column d).  q: planar bf16 query matrices [N][d], head h of image b at q + b*q_sb + h*q_sh (elements); y (and
// residual): [B, Cout, N] with rows ldy elements apart.
namespace {
template <int D, bool RES, bool F16, bool PL>
msla_status_t launch_fused(dim3 grid, int smem, cudaStream_t st, const CUtensorMap& tmM, const CUtensorMap& tmQ, const CUtensorMap& tmO,
                           const CUtensorMap& tmR, const OutParams& p) {
  static std::atomic<unsigned long long> attr_done{0};
  const msla_status_t s = ensure_smem_attr(attr_done, fused_out_kernel<D, RES, F16, PL>, O_SMEM_LIMIT);
  if (s != MSLA_OK) return s;
  launch_pdl_cluster2(fused_out_kernel<D, RES, F16, PL>, grid, dim3(O_THREADS), (size_t)smem, st, tmM, tmQ, tmO, tmR, p);
  count_launches(1);
  return check_launch("fused apply + output projection (tcgen05, paired CTAs)");
}
template <bool F16, bool PL>
msla_status_t launch_fused_for(int d, bool res, dim3 grid, int smem, cudaStream_t st, const CUtensorMap& tmM, const CUtensorMap& tmQ,
                               const CUtensorMap& tmO, const CUtensorMap& tmR, const OutParams& p) {
  if (d == 32) return res ? launch_fused<32, true, F16, PL>(grid, smem, st, tmM, tmQ, tmO, tmR, p) : launch_fused<32, false, F16, PL>(grid, smem, st, tmM, tmQ, tmO, tmR, p);
  return res ? launch_fused<16, true, F16, PL>(grid, smem, st, tmM, tmQ, tmO, tmR, p) : launch_fused<16, false, F16, PL>(grid, smem, st, tmM, tmQ, tmO, tmR, p);
}

template <int D, bool F16, bool SLOTS>
msla_status_t launch_fold(const FoldParams& p, cudaStream_t st) {
  // few heads: a head's key channels are shared out, to one or two CTAs per SM (two: [8, 256, 64, 64] 84.0 -> 80.2 us a forward, f16
  // [8, 128, 45, 80] 49.4 -> 48.6; four are slower, [16, 192, 30, 30] 46.6 -> 49.5)
  const int heads = p.B * p.Ht, sms = device_sm_count();
  if (D == 32 && 4 * heads <= sms) launch_pdl(state_fold_kernel<D, 8, F16, SLOTS>, dim3(heads, D / 8), dim3(FoldShape<D, 8>::THREADS), 0, st, p);
  else if (heads <= sms) launch_pdl(state_fold_kernel<D, D / 2, F16, SLOTS>, dim3(heads, 2), dim3(FoldShape<D, D / 2>::THREADS), 0, st, p);
  else launch_pdl(state_fold_kernel<D, D, F16, SLOTS>, dim3(heads), dim3(FoldShape<D, D>::THREADS), 0, st, p);
  count_launches(1);
  return check_launch("sum of the partial states");
}
msla_status_t run_fold(const FoldStates& in, FoldParams& f, int d, cudaStream_t st, bool f16) {
  f.partial = in.partial; f.S = in.S;
  const bool slots = in.plan.grid > 0;
  for (int i = 0; i < 2; ++i) { f.slots[i] = in.slots[i]; f.w_pw[i] = (const bf16*)in.w_pw[i]; }
  f.slot_floats = in.plan.slot_floats; f.grid = in.plan.grid; f.kv_cost = in.plan.kv_cost; f.tiles = in.plan.kv_tiles; f.cost = in.plan.cost;
  f.batch = in.plan.batch; f.first_image = in.plan.first;
  if (!slots && f.S < 1) return fail(MSLA_ERR_UNSUPPORTED, "fused apply + projection: %d partial states per head", f.S);
  if (d == 32) {
    if (slots) return f16 ? launch_fold<32, true, true>(f, st) : launch_fold<32, false, true>(f, st);
    return f16 ? launch_fold<32, true, false>(f, st) : launch_fold<32, false, false>(f, st);
  }
  if (slots) return f16 ? launch_fold<16, true, true>(f, st) : launch_fold<16, false, true>(f, st);
  return f16 ? launch_fold<16, true, false>(f, st) : launch_fold<16, false, false>(f, st);
}
}  // namespace

msla_status_t run_sum_states(const FoldStates& in, float* state_out, int B, int heads, int Ht, int d, cudaStream_t st, bool f16) {
  FoldParams f{};
  f.state_out = state_out;
  f.B = B; f.heads = heads; f.Ht = Ht;
  return run_fold(in, f, d, st, f16);
}

// f16: queries, weights, bias, residual and output are IEEE binary16 instead of bfloat16 (see FoldParams).
// planes: nullptr, or the channel-blocked query planes that take the place of q.
msla_status_t run_fused_out_bf16(const void* q, long long q_sb, long long q_sh, const PlanesQueries* planes, const FoldStates& states, void* scratch,
                                 const void* w, const void* bias, const void* residual, void* y, int ldy, int B, int Ht, int d, int N, int Cout,
                                 float eps, cudaStream_t st, bool f16) {
  if (!fused_out_bf16_supported(Ht, d, Cout) || ldy % 8 != 0 || q_sb % 8 != 0 || q_sh % 8 != 0 || (planes && N % 8 != 0))
    return fail(MSLA_ERR_UNSUPPORTED, "fused apply + projection: %d heads of %d channels, %d output channels, %d tokens", Ht, d, Cout, N);
  const int K = Ht * d;
  // 256-token tiles per pair of CTAs; 128-token tiles for problems so small that half the pairs would have nothing
  // to do (the larger tile is the more efficient one as soon as every pair has work)
  const int sms = device_sm_count();
  const int ot = 2LL * B * ((N + 2 * OT - 1) / (2 * OT)) <= sms / 2 ? OT / 2 : OT;
  bf16* M = (bf16*)scratch;
  float* ks = (float*)((char*)scratch + fused_out_m_bytes(B, Ht, d, Cout));
  CUtensorMap tmM, tmQ, tmO, tmR;
  {
    const cuuint64_t dM[3] = {(cuuint64_t)K, (cuuint64_t)Cout, (cuuint64_t)B};
    const cuuint64_t sM[2] = {(cuuint64_t)K * 2, (cuuint64_t)K * Cout * 2};
    const cuuint32_t bM[3] = {OKS, OM, 1};
    const cuuint64_t dQ[4] = {(cuuint64_t)d, (cuuint64_t)N, (cuuint64_t)Ht, (cuuint64_t)B};
    const cuuint64_t sQ[3] = {(cuuint64_t)d * 2, (cuuint64_t)q_sh * 2, (cuuint64_t)q_sb * 2};
    const cuuint32_t bQ[4] = {(cuuint32_t)d, (cuuint32_t)ot, 2, 1};
    const cuuint64_t dO[3] = {(cuuint64_t)N, (cuuint64_t)Cout, (cuuint64_t)B};
    const cuuint64_t sO[2] = {(cuuint64_t)ldy * 2, (cuuint64_t)Cout * ldy * 2};
    const cuuint32_t bO[3] = {64, 32, 1};
    if (!tma_make_map_bf16(&tmM, M, 3, dM, sM, bM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        (!planes && !tma_make_map_bf16(&tmQ, q, 4, dQ, sQ, bQ, d == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B)) ||
        !tma_make_map_bf16(&tmO, y, 3, dO, sO, bO, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !tma_make_map_bf16(&tmR, residual ? residual : y, 3, dO, sO, bO, CU_TENSOR_MAP_SWIZZLE_128B))
      return fail(MSLA_ERR_CUDA, "cuTensorMapEncodeTiled failed for the fused apply + output projection");
    if (planes) tmQ = tmM;  // not read
  }
  FoldParams f{};
  f.w = (const bf16*)w; f.M = M; f.ks = ks;
  f.B = B; f.heads = planes ? planes->heads : Ht; f.Ht = Ht; f.Cout = Cout; f.K = K;
  msla_status_t s = run_fold(states, f, d, st, f16);
  if (s != MSLA_OK) return s;
  OutParams p{};
  if (planes) {
    p.q0 = (const unsigned char*)planes->q0; p.q1 = (const unsigned char*)planes->q1; p.heads = planes->heads;
    p.plane_bytes = planes->plane_tokens * d * 2; p.tok_bytes = planes->first_token * d * 2;
  }
  p.ks = ks; p.bias = (const bf16*)bias; p.residual = (const bf16*)residual;
  p.B = B; p.N = N; p.Cout = Cout; p.Ht = Ht; p.d = d; p.eps = eps;
  p.kslices = (K + OKS - 1) / OKS;
  p.ot = ot;
  p.tiles_per_image = (N + 2 * ot - 1) / (2 * ot);
  const long long tiles = (long long)B * p.tiles_per_image;
  if (tiles > 0x7fffffffLL) return fail(MSLA_ERR_UNSUPPORTED, "too many token tiles");
  p.num_tiles = (int)tiles;
  // the query ring takes what shared memory is left beside the rows of M (and the residual blocks)
  const int smem_fixed = p.kslices * O_A_SLICE + O_SMEM_FIXED + (residual ? O_STAGING : 0), slot = 2 * ot * d * 2;
  p.stages = (O_SMEM_LIMIT - smem_fixed) / slot;
  if (p.stages > O_MAX_STAGES) p.stages = O_MAX_STAGES;
  if (p.stages < O_MIN_STAGES) return fail(MSLA_ERR_UNSUPPORTED, "fused apply + projection: no room for the query ring (%d slots)", p.stages);
  const int smem = smem_fixed + p.stages * slot;
  long long pairs = sms / 2;
  if (pairs > tiles) pairs = tiles;
  if (pairs < 1) pairs = 1;
  const dim3 grid((unsigned)(2 * pairs));
  const bool res = residual != nullptr;
  if (planes) return f16 ? launch_fused_for<true, true>(d, res, grid, smem, st, tmM, tmQ, tmO, tmR, p) : launch_fused_for<false, true>(d, res, grid, smem, st, tmM, tmQ, tmO, tmR, p);
  return f16 ? launch_fused_for<true, false>(d, res, grid, smem, st, tmM, tmQ, tmO, tmR, p) : launch_fused_for<false, false>(d, res, grid, smem, st, tmM, tmQ, tmO, tmR, p);
}

int fused_timeout_flag() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_fused_timeout_flag, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return v;
}

}  // namespace msla
