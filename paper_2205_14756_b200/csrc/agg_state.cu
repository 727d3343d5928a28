// Steps 2 and 3 of the module (Section 3.1) in one kernel, on channel-blocked planes: the multi-scale aggregation
// (5x5 depthwise + grouped 1x1) and both scales' state sums  sum_n relu(k[n])^T [v[n] | 1]  of Eq. 3.
//
// Layout of a plane (the q, k or v of one head): [H][W / 8][D][8], W a multiple of 8: eight horizontally neighbouring
// pixels of one channel are 16 contiguous bytes (a pixel octet), and the D channels of an octet are contiguous.
//
// What is computed where:
//   * queries: the aggregated plane is written, as the output step needs it token by token;
//   * keys and values: the aggregated tokens are needed by the state sums only, so they are never written.  The state
//     of the aggregated scale is accumulated from the tile in shared memory, and so is the un-aggregated scale's, from
//     the staged input rows.  The grouped 1x1 of the values commutes with the sum over tokens,
//       sum_n relu(k1[n])[a] * (Wv dv[n])[c] = sum_c' Wv[c][c'] * (sum_n relu(k1[n])[a] * dv[n][c']),
//     so the kernel sums over the depthwise output dv and the reader of the partial states applies Wv to the d x d
//     result (in fp32).
//
// The depthwise filter runs on tensor cores as banded (Toeplitz) matrices: for one channel and filter row dy,
//   out[y][x] += sum_k in[y + dy - 2][x' + k] * T[k][x]
// is one mma.sync.m16n8k16 per 16 rows x 8 output pixels.  MMA row g is image row 2g, row g + 8 image row 2g + 1: the fragment
// for dy + 1 reuses half of the one for dy.  Every operand is an aligned 16-byte row that ldmatrix takes from the staged tile
// as it was copied: no pass that turns the tile around (the token-major kernel spends a third of its shared-memory cycles on
// it).  The five taps of eight outputs reach over twelve pixels, and which octets those lie in depends on the outputs:
//   * keys and values: the order of the tokens inside a tile does not matter to the sums, so the outputs are taken two pixels to
//     the left of the octets, x = 8o - 2 .. 8o + 5.  Their window is then exactly the octets o - 1 and o.
//   * queries are written back in octets, so the outputs are an octet, and the window is that octet and a mixed one: slots
//     6, 7 hold the last two pixels of the octet to the left, slots 0, 1 the first two of the octet to the right (lanes t = 3
//     and t = 0 of a fragment), the others meet zero weights.
//
// One persistent CTA per SM with a contiguous run of 16 x 16-pixel tiles: first of pairs of 32-channel blocks (K and V of one
// head; d = 16: of two heads), then of blocks of queries.  Tiles run down bands of four tile rows, column by column, so that the
// halo rows and columns shared with the neighbours are still in L2.  Warps are specialised, so that the phases of neighbouring
// tiles overlap (all warps taking the phases in turn, 16 of them, kept the tensor pipe 43 % busy):
//   warps 0-15   depthwise step of four channels each (queries: two), Toeplitz fragments in registers while the head lasts; fp32
//                sums rounded once into a [channel][pixel] tile, double buffered
//   warps 16-23  keys and values: 16 key channels x 4 image rows of both states each, accumulators in registers while the (head,
//                image) lasts: the un-aggregated scale from the staged rows, the aggregated one from the depthwise tile, keys
//                through their grouped 1x1 first (transposed: channels x pixels, whose accumulator layout is the A-fragment
//                layout of the state's MMA)
//                queries: grouped 1x1 of two image rows each, staged
//   warp 24      requests the tiles: 20 rows x 3 (queries: 4) octets per block by TMA, even and odd image rows apart (two tensor maps), so that
//                the rows of an ldmatrix matrix (2g + r, g = 0 .. 7) are neighbours: a box of 8 channels x 8 pixels (128 bytes, 128B
//                swizzle) x 10 rows x octets x channel groups lands as [group][octet][row][128 bytes], and eight consecutive rows
//                fall on different banks.  Rows and octets outside the image are zero-filled = the padding.  Two buffers (queries: four)
//   warp 25      writes the staged query tiles, one TMA store each
// Issuing a copy takes a thread about 0.14 us.  With the copies issued by the summing warps (per tile of queries two loads by one of
// them and two row copies by each) a tile of queries took 1.32 us against 1.12 now: the warps wait for one another in turn.
// In each role the next operands are fetched before the stores that wait for the current products.
// Shared-memory wavefronts, the MMA rate and issue slots bound it together (per 16 x 16 tile of a head's K, V and Q: about 3400
// wavefronts and 1540 MMAs of two cycles; leaving out the depthwise MMAs, the state of either scale or the loads takes 16, 12, 12
// or 3 % off the keys and values).  [1, 256, 512, 512]: 192 us (212 before the copies had warps of their own), where the
// token-major aggregation (209 us) and the state kernel (98 us) took 307; [1, 128, 512, 512] d = 16: 97 (119); whole
// forward 415 -> 393, 251 -> 229, [16, 256, 64, 64] 141.5 -> 136, building block [1, 256, 128, 256] / 1024 160.5 -> 157.
// All waits are bounded; on time-out every warp leaves its loop and a flag is raised.
#include <cuda.h>

#include "msla_common.cuh"
#include "msla_host.h"
#include "tma_host.h"
#include "tcgen05_util.cuh"

namespace msla {
namespace {

using bf16 = __nv_bfloat16;

constexpr int AS_DW_WARPS = 16, AS_SUM_WARPS = 8, AS_COPY_WARPS = 4;  // of the last four one requests loads and one stores
constexpr int AS_THREADS = 32 * (AS_DW_WARPS + AS_SUM_WARPS + AS_COPY_WARPS);
constexpr int AS_LOAD_WARP = AS_DW_WARPS + AS_SUM_WARPS, AS_STORE_WARP = AS_LOAD_WARP + 1;
// Registers a thread: the launch's 72, shared out (80 for 24 warps alike spilled in both computing roles)
constexpr int AS_DW_REGS = 64, AS_SUM_REGS = 104, AS_COPY_REGS = 40;
static_assert(AS_DW_WARPS * AS_DW_REGS + AS_SUM_WARPS * AS_SUM_REGS + AS_COPY_WARPS * AS_COPY_REGS == AS_THREADS / 32 * 72, "shares of the launch's registers");
constexpr int AS_TW = 16, AS_TH = 16, AS_ROWS = AS_TH + 4;
constexpr int AS_DWO_CH = AS_TW * AS_TH * 2 + 16;   // depthwise output: bytes per channel (33 * 16)
constexpr int AS_DWO_SIDE = 32 * AS_DWO_CH;          // of one block
constexpr int AS_STAGE = AS_TH * 1024;              // staged query output: 16 rows x 16 pixels x 32 channels, double buffered
constexpr int AS_BAND = 4;                          // tile rows per band of the traversal
// Staged tile of the two roles: SIDES blocks of OCT octets per row; [block][row parity][channel group of 8][octet][row / 2][128 bytes].
template <int SIDES_, int OCT_, int BUFS_> struct AsStage {
  static constexpr int SIDES = SIDES_, OCT = OCT_, BUFS = BUFS_, ROWS2 = AS_ROWS / 2;
  static constexpr int PAR = 4 * OCT * ROWS2 * 128;           // one parity of one block
  static constexpr int SIDE = 2 * PAR, BUF = SIDES * SIDE;    // one block; all
  static constexpr int DWO = SIDES * AS_DWO_SIDE;
};
using AsKv = AsStage<2, 3, 2>;
using AsQ = AsStage<1, 4, 4>;
constexpr int AS_RED = 2 * AS_SUM_WARPS * 16 * 33 * 4;  // the warps' states on their way to the partial sums
constexpr int AS_SMEM_KV = AsKv::BUFS * AsKv::BUF + 2 * AsKv::DWO + AS_RED, AS_SMEM_Q = AsQ::BUFS * AsQ::BUF + 2 * AsQ::DWO + 2 * AS_STAGE;
constexpr int AS_SMEM = (AS_SMEM_KV > AS_SMEM_Q ? AS_SMEM_KV : AS_SMEM_Q) + 1024;  // + slack to align the base (the swizzle is a function of the address)
static_assert(AsKv::PAR % 1024 == 0 && AsQ::PAR % 1024 == 0 && (AS_DWO_CH / 16) % 2 == 1, "swizzle atoms; conflict-free pitch");
static_assert(AS_SMEM + 256 <= 227 * 1024, "dynamic and static shared memory of a CTA");

__device__ int g_aggstate_timeout_flag = 0;

struct AggStateParams {
  float* partial;            // slots of 2 states per head of the block: [.., un-aggregated, aggregated][d][d + 1]
  const bf16* w_dw;          // [3 * heads * d][5][5]
  const bf16* w_pw;          // [3 * heads * d][d]
  int heads, B, H, W, Wb;
  int tiles_y, kv_tiles_x, q_tiles_x, kv_tiles, q_tiles;  // tiles per plane
  int row_lo, row_hi;           // image rows that count in the states
  int with_scale0;
  int batch, first;             // see AggStatePlan
  long long kv_units;           // of the batch: (block, image, tile), tile fastest; keys and values first, then queries
  long long cost;               // of all units, and of one
  int kv_cost, q_cost;
};

template <bool F16>
__device__ __forceinline__ uint32_t as_pack(float lo, float hi) {
  uint32_t r;
  if constexpr (F16) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
template <bool F16>
__device__ __forceinline__ uint32_t as_pack_relu(float lo, float hi) {  // max(x, 0), then rounded
  uint32_t r;
  if constexpr (F16) asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  else asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
template <bool F16>
__device__ __forceinline__ uint32_t as_relu(uint32_t x) {
  uint32_t r;
  if constexpr (F16) asm("max.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0u));
  else asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0u));
  return r;
}
template <bool F16>
__device__ __forceinline__ void as_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  if constexpr (F16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
template <bool F16>
__device__ __forceinline__ void as_mma_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  const float z = 0.f;
  if constexpr (F16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(z));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(z));
}
__device__ __forceinline__ void as_ldsm4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
__device__ __forceinline__ void as_ldsm2(uint32_t& r0, uint32_t& r1, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}
__device__ __forceinline__ void as_ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void as_ldsm2t(uint32_t& r0, uint32_t& r1, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t as_lds32(uint32_t addr) {
  uint32_t r;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(addr) : "memory");
  return r;
}
__device__ __forceinline__ void as_sts32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void as_tma_load(uint32_t dst, const CUtensorMap* map, uint32_t bar, int row2, int oct, int plane) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(row2), "r"(oct), "r"(0), "r"(plane) : "memory");
}
__device__ __forceinline__ void as_tma_store(const CUtensorMap* map, uint32_t src, int piece, int row, int plane) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
               ::"l"(map), "r"(src), "r"(0), "r"(piece), "r"(row), "r"(plane) : "memory");
}

// A tile of the run: pair of blocks, image, position.  Advanced without divisions.
struct AsUnit {
  int p, b;
  int tx, ty, band_end;  // band_end: first tile row below the current band
};
__device__ __forceinline__ AsUnit as_locate(const AggStateParams& p, long long v, int tiles_x, int tiles) {
  const long long pb = v / tiles;
  const int tile = (int)(v - pb * tiles);
  AsUnit r;
  const int band = tile / (AS_BAND * tiles_x), rem = tile - band * (AS_BAND * tiles_x);
  r.band_end = min(band * AS_BAND + AS_BAND, p.tiles_y);
  const int bh = r.band_end - band * AS_BAND;
  r.tx = rem / bh;
  r.ty = band * AS_BAND + rem - r.tx * bh;
  r.p = (int)(pb / p.B);
  r.b = (int)(pb - (long long)r.p * p.B);
  return r;
}
__device__ __forceinline__ void as_advance(const AggStateParams& p, AsUnit& u, int tiles_x) {
  if (++u.ty < u.band_end) return;
  if (++u.tx < tiles_x) { u.ty = (u.band_end - 1) / AS_BAND * AS_BAND; return; }
  u.tx = 0;
  u.ty = u.band_end;
  if (u.ty == p.tiles_y) {
    u.ty = 0;
    if (++u.b == p.B) { u.b = 0; ++u.p; }
  }
  u.band_end = min(u.ty + AS_BAND, p.tiles_y);
}

// Words of Toeplitz B fragments of N channels from `ch` on: taps i, i + 1 of every filter row (zero outside the five).  No branches: all
// loads of a thread are in flight together.
template <int N>
__device__ __forceinline__ void as_load_taps(const bf16* w_dw, int ch, int i, uint32_t (&bt)[N][5]) {
#pragma unroll
  for (int cc = 0; cc < N; ++cc)
#pragma unroll
    for (int dy = 0; dy < 5; ++dy) {
      const unsigned short* row = reinterpret_cast<const unsigned short*>(w_dw) + (long long)(ch + cc) * 25 + dy * 5;
      auto tap = [&](int j) -> uint32_t {
        const uint32_t v = ld_dep16(row + min(max(j, 0), 4));
        return j >= 0 && j < 5 ? v : 0u;
      };
      bt[cc][dy] = tap(i) | (tap(i + 1) << 16);
    }
}
// Pixel pair (row 2g + half, columns 8nb + 2t, + 1): word t of octet (2nb + half) * 8 + g of the channel.
template <bool F16>
__device__ __forceinline__ void as_put_depthwise(uint32_t dst, const float (&acc)[2][4]) {
#pragma unroll
  for (int nb = 0; nb < 2; ++nb)
#pragma unroll
    for (int half = 0; half < 2; ++half) as_sts32(dst + (uint32_t)((2 * nb + half) * 128), as_pack<F16>(acc[nb][2 * half], acc[nb][2 * half + 1]));
}

template <int D, bool F16>
__global__ void __launch_bounds__(AS_THREADS, 1)
agg_state_kernel(const __grid_constant__ CUtensorMap kv_even, const __grid_constant__ CUtensorMap kv_odd, const __grid_constant__ CUtensorMap q_even,
                 const __grid_constant__ CUtensorMap q_odd, const __grid_constant__ CUtensorMap q_out, AggStateParams p) {
  constexpr bool D16 = D == 16;
  constexpr int NE = D * (D + 1);
  constexpr int HPB = 32 / D;        // heads per 32-channel block
  constexpr int NJ = D / 8;          // 8-channel column blocks of a state
  extern __shared__ unsigned char smem_raw[];
  const uint32_t box = (smem_u32(smem_raw) + 1023u) & ~1023u;
  __shared__ __align__(8) unsigned long long bar_storage[25];
  __shared__ int abort_flag;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;

  const long long run_first = agg_state_first_unit(p.cost, p.kv_cost, p.q_cost, p.kv_units, blockIdx.x, gridDim.x),
                  run_end = agg_state_first_unit(p.cost, p.kv_cost, p.q_cost, p.kv_units, blockIdx.x + 1, gridDim.x);
  long long u_first = min(run_first, p.kv_units), u_end = min(run_end, p.kv_units);
  long long q_first = max(run_first, p.kv_units) - p.kv_units, q_end = max(run_end, p.kv_units) - p.kv_units;
  if (p.batch != p.B) {  // this call's tiles of the run are a run of its own list
    u_first = agg_state_part_units(u_first, p.kv_tiles, p.batch, p.first, p.B);
    u_end = agg_state_part_units(u_end, p.kv_tiles, p.batch, p.first, p.B);
    q_first = agg_state_part_units(q_first, p.q_tiles, p.batch, p.first, p.B);
    q_end = agg_state_part_units(q_end, p.q_tiles, p.batch, p.first, p.B);
  }
  const int kv_count = (int)(u_end - u_first), q_count = (int)(q_end - q_first);

  // Plane (inside an image's 3 * heads): block `pr` of queries (s = 0), keys (1) or values (2), sub-block `sub`; an absent head
  // (odd counts, d = 16) repeats the last.
  auto plane_of = [&](int s, int pr, int sub) { return 3 * min(HPB * pr + sub, p.heads - 1) + s; };
  // Address of the 16 bytes of channel c (of the block's 32) in staged row r, octet o.
  auto at = [&](auto stage, int s, int r, int o, int c) -> uint32_t {
    using ST = decltype(stage);
    const int idx = ((c >> 3) * ST::OCT + o) * ST::ROWS2 + (r >> 1);
    return (uint32_t)(s * ST::SIDE + (r & 1) * ST::PAR + idx * 128 + (((c & 7) ^ (idx & 7)) << 4));
  };

  // Barriers, a set per role: a staged tile has landed / been read, a depthwise tile is complete / been read.
  const uint32_t bars = smem_u32(bar_storage);
  auto full = [&](int role, uint32_t buf) { return bars + 64 * role + 8 * buf; };
  auto freed = [&](int role, uint32_t buf) { return bars + 64 * role + (role ? 32 : 16) + 8 * buf; };
  auto dwo_full = [&](int role, uint32_t buf) { return bars + 64 * role + (role ? 64 : 32) + 8 * buf; };
  auto dwo_freed = [&](int role, uint32_t buf) { return bars + 64 * role + (role ? 80 : 48) + 8 * buf; };
  auto staged = [&](uint32_t buf) { return bars + 160 + 8 * buf; };       // queries: the output tile is staged / has been copied out
  auto staging_freed = [&](uint32_t buf) { return bars + 176 + 8 * buf; };
  const uint32_t sums_meet = bars + 192;                                  // the summing warps, twice per (head, image)
  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int r = 0; r < 2; ++r) {
      for (int i = 0; i < (r == 0 ? AsKv::BUFS : AsQ::BUFS); ++i) {
        mbar_init(full(r, i), 1);
        mbar_init(freed(r, i), r == 0 ? AS_DW_WARPS + AS_SUM_WARPS : AS_DW_WARPS);
      }
      for (int i = 0; i < 2; ++i) {
        mbar_init(dwo_full(r, i), AS_DW_WARPS);
        mbar_init(dwo_freed(r, i), AS_SUM_WARPS);
      }
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(staged(i), AS_SUM_WARPS);
      mbar_init(staging_freed(i), 1);
    }
    mbar_init(sums_meet, AS_SUM_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
    ok = mbar_wait(bar, parity, &abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    return ok;
  };
  auto arrive = [&](uint32_t bar) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };
  // Requests tile `un` of keys and values / of queries and moves the cursor on.
  auto request_kv = [&](AsUnit& un, uint32_t buf) {
    if (lane == 0) {
      mbar_expect_tx(full(0, buf), AsKv::BUF);
      const int row2 = un.ty * (AS_TH / 2) - 1, oct = un.tx * 2 - 1;  // rows 16 ty - 2 + {0, 2, ..} and + {1, 3, ..}
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int sub = 0; sub < HPB; ++sub) {
          const int plane = un.b * 3 * p.heads + plane_of(1 + s, un.p, sub);
          const uint32_t dst = box + buf * AsKv::BUF + s * AsKv::SIDE + sub * (AsKv::PAR / HPB);
          as_tma_load(dst, &kv_even, full(0, buf), row2, oct, plane);
          as_tma_load(dst + AsKv::PAR, &kv_odd, full(0, buf), row2, oct, plane);
        }
    }
    as_advance(p, un, p.kv_tiles_x);
  };
  auto request_q = [&](AsUnit& un, uint32_t buf) {
    if (lane == 0) {
      mbar_expect_tx(full(1, buf), AsQ::BUF);
      const int row2 = un.ty * (AS_TH / 2) - 1, oct = un.tx * 2 - 1;
#pragma unroll
      for (int sub = 0; sub < HPB; ++sub) {
        const int plane = un.b * 3 * p.heads + plane_of(0, un.p, sub);
        const uint32_t dst = box + buf * AsQ::BUF + sub * (AsQ::PAR / HPB);
        as_tma_load(dst, &q_even, full(1, buf), row2, oct, plane);
        as_tma_load(dst + AsQ::PAR, &q_odd, full(1, buf), row2, oct, plane);
      }
    }
    as_advance(p, un, p.q_tiles_x);
  };
  pdl_wait();  // the planes are the previous kernel's output; q1 and the partial states may still be read by an earlier one

  // Roles.  Each branch ends the keys and values at the same barrier, after which the queries' tiles take over the shared memory (in
  // one piece of code per role: where branches with different register counts meet, the compiler allows the smallest).
  auto end_of_kv = [&]() -> bool {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("bar.sync 2, %0;" ::"n"(AS_THREADS) : "memory");
    ok = ok && !*(volatile int*)&abort_flag;
    return ok && q_count > 0;
  };
  if (warp < AS_DW_WARPS) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(AS_DW_REGS));
    {
      // ---------------------------------------------------------------- depthwise: keys and values
      using ST = AsKv;
      const int side = warp >> 3, c0 = 4 * (warp & 7);
      const uint32_t dwo = box + 2 * ST::BUF + (uint32_t)(side * AS_DWO_SIDE + c0 * AS_DWO_CH + lane * 4);
      // matrix (r, o) = staged rows 2g' + r, octet o of channel c0; lane l supplies row l % 8 of matrix l / 8.  Channel c0 + cc: XOR
      // cc << 4 (the swizzle permutes the 16-byte pieces of a row by XOR).
      auto mat = [&](int r, int o) { return box + at(ST{}, side, 2 * (lane & 7) + r, o, c0); };
      const int mi = lane >> 3;
      const uint32_t a0 = mi < 3 ? mat(0, mi) : mat(1, 0), a1 = mi < 2 ? mat(1, 1 + mi) : mat(2, mi - 2), a2 = mi == 0 ? mat(2, 2) : mat(3, mi - 1),
                     a3 = mi < 3 ? mat(4, mi) : mat(5, 0), a4 = mat(5, 1 + (mi & 1));
      // Toeplitz B fragments: window pixel k, output pixel n: tap k - n - 4.  Of a lane's two words (k = 2t, + 1 and 2t + 8, + 9) one at
      // most meets the five taps, the same one throughout.
      uint32_t bt[4][5];
      const bool low = 2 * t - g - 4 >= -1;
      int change = 0;        // tile at which the pair of blocks changes
#pragma unroll 1
      for (int i = 0; i < kv_count; ++i) {
        const uint32_t buf = i & 1, ph = (i >> 1) & 1;
        if (i == change) {
          const long long per_pair = (long long)p.kv_tiles * p.B;
          const int pr = (int)((u_first + i) / per_pair);
          change = (int)min((pr + 1) * per_pair - u_first, (long long)kv_count);
          as_load_taps<4>(p.w_dw, plane_of(1 + side, pr, D16 ? c0 >> 4 : 0) * D + (c0 & (D - 1)), low ? 2 * t - g - 4 : 2 * t - g + 4, bt);
        }
        if (!wait(full(0, buf), ph)) break;
        if (!wait(dwo_freed(0, buf), ph ^ 1)) break;
        const uint32_t ro = buf * ST::BUF, dw = dwo + buf * ST::DWO;
        uint32_t R[6][3];
        auto load = [&](int cc) {
          as_ldsm4(R[0][0], R[0][1], R[0][2], R[1][0], (a0 + ro) ^ (uint32_t)(cc << 4));
          as_ldsm4(R[1][1], R[1][2], R[2][0], R[2][1], (a1 + ro) ^ (uint32_t)(cc << 4));
          as_ldsm4(R[2][2], R[3][0], R[3][1], R[3][2], (a2 + ro) ^ (uint32_t)(cc << 4));
          as_ldsm4(R[4][0], R[4][1], R[4][2], R[5][0], (a3 + ro) ^ (uint32_t)(cc << 4));
          as_ldsm2(R[5][1], R[5][2], (a4 + ro) ^ (uint32_t)(cc << 4));
        };
        load(0);
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          float acc[2][4];
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) as_mma_first<F16>(acc[nb], R[0][nb], R[1][nb], R[0][nb + 1], R[1][nb + 1], low ? bt[cc][0] : 0u, low ? 0u : bt[cc][0]);
#pragma unroll
          for (int dy = 1; dy < 5; ++dy)
#pragma unroll
            for (int nb = 0; nb < 2; ++nb) as_mma<F16>(acc[nb], R[dy][nb], R[dy + 1][nb], R[dy][nb + 1], R[dy + 1][nb + 1], low ? bt[cc][dy] : 0u, low ? 0u : bt[cc][dy]);
          if (cc < 3) load(cc + 1);  // ahead of the stores below, which wait for the products
          if (cc == 2) arrive(freed(0, buf));
          as_put_depthwise<F16>(dw + cc * AS_DWO_CH, acc);
        }
        arrive(dwo_full(0, buf));
      }
    }
    if (end_of_kv()) {
      // ---------------------------------------------------------------- depthwise
      using ST = AsQ;
      const int c0 = 2 * warp;
      const uint32_t dwo = box + ST::BUFS * ST::BUF + (uint32_t)(c0 * AS_DWO_CH + lane * 4);
      uint32_t main_off[3], edge_off[3];  // octets 1, 2 of staged rows 2g + r (r = 2k + lane bit 3), and the neighbours' pixel pairs
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        main_off[k] = box + at(ST{}, 0, 2 * (lane & 7) + 2 * k + ((lane >> 3) & 1), 1 + (lane >> 4), c0);
        edge_off[k] = box + at(ST{}, 0, 2 * g + 2 * k, t >= 2 ? 0 : 3, c0) + (t >= 2 ? 12 : 0);
      }
      // Toeplitz B fragments: [0] the octet itself, tap k - n + 2; [1] the mixed octet: left neighbour's pixel 6 (= -2) in lane t = 3,
      // right neighbour's pixel 0 (= 8) in lane t = 0
      uint32_t b0[2][5], b1[2][5];
      int change = 0;
#pragma unroll 1
      for (int i = 0; i < q_count; ++i) {
        const uint32_t buf = i & 1, ph = (i >> 1) & 1;
        if (i == change) {
          const long long per_block = (long long)p.q_tiles * p.B;
          const int pr = (int)((q_first + i) / per_block);
          change = (int)min((pr + 1) * per_block - q_first, (long long)q_count);
          as_load_taps<2>(p.w_dw, plane_of(0, pr, D16 ? c0 >> 4 : 0) * D + (c0 & (D - 1)), 2 * t - g + 2, b0);
          as_load_taps<2>(p.w_dw, plane_of(0, pr, D16 ? c0 >> 4 : 0) * D + (c0 & (D - 1)), t == 3 ? -g : t == 0 ? 10 - g : -8, b1);
        }
        const uint32_t sbuf = i % ST::BUFS;
        if (!wait(full(1, sbuf), (i / ST::BUFS) & 1)) break;
        if (!wait(dwo_freed(1, buf), ph ^ 1)) break;
        const uint32_t ro = sbuf * ST::BUF, dw = dwo + buf * ST::DWO;
        uint32_t R[6][2], E[6];
        auto load = [&](int cc) {
#pragma unroll
          for (int k = 0; k < 3; ++k) as_ldsm4(R[2 * k][0], R[2 * k + 1][0], R[2 * k][1], R[2 * k + 1][1], (main_off[k] + ro) ^ (uint32_t)(cc << 4));
#pragma unroll
          for (int r = 0; r < 6; ++r) E[r] = as_lds32(((edge_off[r >> 1] + ro) ^ (uint32_t)(cc << 4)) + (r & 1) * ST::PAR);
        };
        load(0);
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          float acc[2][4];
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) {
            uint32_t X[6];  // the mixed octet: left neighbour in lanes t >= 2, right neighbour in lanes t < 2
#pragma unroll
            for (int r = 0; r < 6; ++r) X[r] = nb == 0 ? (t >= 2 ? E[r] : R[r][1]) : (t >= 2 ? R[r][0] : E[r]);
            as_mma_first<F16>(acc[nb], R[0][nb], R[1][nb], X[0], X[1], b0[cc][0], b1[cc][0]);
#pragma unroll
            for (int dy = 1; dy < 5; ++dy) as_mma<F16>(acc[nb], R[dy][nb], R[dy + 1][nb], X[dy], X[dy + 1], b0[cc][dy], b1[cc][dy]);
          }
          if (cc == 0) {  // ahead of the stores below, which wait for the products
            load(1);
            arrive(freed(1, sbuf));
          }
          as_put_depthwise<F16>(dw + cc * AS_DWO_CH, acc);
        }
        arrive(dwo_full(1, buf));
      }
    }
  } else if (warp >= AS_LOAD_WARP) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(AS_COPY_REGS));
    // ---------------------------------------------------------------- copies
    if (warp == AS_LOAD_WARP && kv_count > 0) {
      AsUnit nxt = as_locate(p, u_first, p.kv_tiles_x, p.kv_tiles);
#pragma unroll 1
      for (int i = 0; i < kv_count; ++i) {
        if (i >= 2 && !wait(freed(0, i & 1), ((i - 2) >> 1) & 1)) break;
        request_kv(nxt, i & 1);
      }
    }
    const bool more = end_of_kv();
    if (more && warp == AS_LOAD_WARP) {
      // ---------------------------------------------------------------- copies: staged tiles
      AsUnit nxt = as_locate(p, q_first, p.q_tiles_x, p.q_tiles);
#pragma unroll 1
      for (int i = 0; i < q_count; ++i) {
        if (i >= AsQ::BUFS && !wait(freed(1, i % AsQ::BUFS), (i / AsQ::BUFS - 1) & 1)) break;
        request_q(nxt, i % AsQ::BUFS);
      }
    } else if (more && warp == AS_STORE_WARP) {
      // ---------------------------------------------------------------- copies: output tiles (rows and octets outside the image are clipped)
      const uint32_t stage0 = box + AsQ::BUFS * AsQ::BUF + 2 * AsQ::DWO;
      AsUnit un = as_locate(p, q_first, p.q_tiles_x, p.q_tiles);
#pragma unroll 1
      for (int i = 0; i < q_count; ++i, as_advance(p, un, p.q_tiles_x)) {
        const uint32_t buf = i & 1;
        if (!wait(staged(buf), (i >> 1) & 1)) break;
        if (lane == 0) {
#pragma unroll
          for (int sub = 0; sub < HPB; ++sub) {
            const int h = HPB * un.p + sub;
            if (h < p.heads) as_tma_store(&q_out, stage0 + buf * AS_STAGE + sub * (AS_STAGE / HPB), un.tx * (D / 4), un.ty * AS_TH, un.b * p.heads + h);
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          mbar_arrive(staging_freed(buf));
        }
      }
      if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // stores done before the CTA retires
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(AS_SUM_REGS));
    if (kv_count > 0) {
      // ---------------------------------------------------------------- states
      using ST = AsKv;
      const int sw = warp - AS_DW_WARPS, mh = sw >> 2, rg = sw & 3;  // key channels 16 mh .. + 15 of the block (d = 16: head mh of the pair), image rows 4 rg .. + 3
      const uint32_t dwo = box + 2 * ST::BUF;
      AsUnit un = as_locate(p, u_first, p.kv_tiles_x, p.kv_tiles);
      const uint32_t ONES = F16 ? 0x3C003C00u : 0x3F803F80u;
      const uint32_t ones0 = (g & 1) ? 0u : ONES, ones1 = (g & 1) ? ONES : 0u;  // even columns count scale 0, odd ones the aggregated scale
      float acc0[NJ][4], acc1[NJ][4], accs[4];
      auto clear = [&] {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          accs[e] = 0.f;
#pragma unroll
          for (int j = 0; j < NJ; ++j) acc0[j][e] = acc1[j][e] = 0.f;
        }
      };
      clear();
      uint32_t wk[D / 16][4];  // A fragments of the keys' grouped 1x1, rows 16 mh .. + 15
      int cur_p = -1;
      // depthwise tile: row 2g' + half of column block nb is octet (2nb + half) * 8 + g'; this warp's rows are g' = 2 rg, 2 rg + 1
      const uint32_t k1_off = dwo + (uint32_t)((D16 ? 16 * mh + (lane & 15) : lane) * AS_DWO_CH + rg * 32);
      const uint32_t v1_off = dwo + AS_DWO_SIDE + (uint32_t)(((D16 ? 16 * mh : 0) + 8 * (lane >> 4) + (lane & 7)) * AS_DWO_CH + ((lane >> 3) & 1) * 256 + rg * 32);
      // staged row of image row 4 rg (+ PAR: 4 rg + 1; + 128 and another swizzle phase: 4 rg + 2), octets 1 and 2; keys: channels
      // 16 mh + .., values: from channel 0 (d = 16: 16 mh) on
      uint32_t k0_off[2], v0_off[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        k0_off[e] = box + at(ST{}, 0, 4 * rg + 2 * e + 2, 1 + (lane >> 4), 16 * mh + (lane & 15));
        v0_off[e] = box + at(ST{}, 1, 4 * rg + 2 * e + 2, 1 + ((lane >> 3) & 1), (D16 ? 16 * mh : 0) + 8 * (lane >> 4) + (lane & 7));
      }
      // two channel groups further on: 60 rows of 128 bytes, i.e. the swizzle phase changes by 4
      static_assert(2 * ST::OCT * ST::ROWS2 % 8 == 4, "phase of the second pair of channel groups");
      constexpr uint32_t V0_STEP = 2 * ST::OCT * ST::ROWS2 * 128;
#pragma unroll 1
      for (int i = 0; i < kv_count; ++i) {
        const uint32_t buf = i & 1, ph = (i >> 1) & 1;
        if (un.p != cur_p) {
          cur_p = un.p;
          const uint32_t* wp = reinterpret_cast<const uint32_t*>(p.w_pw + ((long long)plane_of(1, cur_p, D16 ? mh : 0) * D + (D16 ? 0 : 16 * mh)) * D);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t* a = wp + (g * D + 16 * ks) / 2 + t;
            wk[ks][0] = __ldg(a); wk[ks][1] = __ldg(a + 4 * D); wk[ks][2] = __ldg(a + 4); wk[ks][3] = __ldg(a + 4 * D + 4);
          }
        }
        const int y = un.ty * AS_TH + 4 * rg, x0 = un.tx * AS_TW - 2;
        const bool edge_y = un.ty * AS_TH < p.row_lo || un.ty * AS_TH + AS_TH > p.row_hi;
        const bool edge = edge_y || x0 < 0 || x0 + AS_TW > p.W;
        // ---- un-aggregated scale: octets 2 tx, 2 tx + 1 of the staged rows
        if (!wait(full(0, buf), ph)) break;
        if (p.with_scale0) {
          uint32_t k[4], v[NJ / 2][4];  // one image row's operands, fetched while the row before is multiplied
          auto load = [&](int r) {
            const uint32_t ro = buf * ST::BUF + (r & 1) * ST::PAR;
            as_ldsm4(k[0], k[1], k[2], k[3], k0_off[r >> 1] + ro);
#pragma unroll
            for (int j = 0; j < NJ / 2; ++j) as_ldsm4(v[j][0], v[j][1], v[j][2], v[j][3], j == 0 ? v0_off[r >> 1] + ro : (v0_off[r >> 1] + ro + V0_STEP) ^ 64u);
          };
          load(0);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            uint32_t a[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) a[e] = as_relu<F16>(k[e]);
            if (edge_y) {
              const bool in = y + r >= p.row_lo && y + r < p.row_hi;
#pragma unroll
              for (int e = 0; e < 4; ++e) a[e] = in ? a[e] : 0u;
            }
            as_mma<F16>(accs, a[0], a[1], a[2], a[3], ones0, ones0);
#pragma unroll
            for (int j = 0; j < NJ / 2; ++j) {
              as_mma<F16>(acc0[2 * j], a[0], a[1], a[2], a[3], v[j][0], v[j][1]);
              as_mma<F16>(acc0[2 * j + 1], a[0], a[1], a[2], a[3], v[j][2], v[j][3]);
            }
            if (r < 3) load(r + 1);
          }
        }
        arrive(freed(0, buf));
        // ---- aggregated scale
        if (!wait(dwo_full(0, buf), ph)) break;
        uint32_t kb[2][4];  // one image row of keys, both column blocks, fetched a row ahead
        auto load_keys = [&](int r) {
          const uint32_t ro = buf * ST::DWO + (r >> 1) * 16 + (r & 1) * 128;
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) {
            if constexpr (D16) as_ldsm2t(kb[nb][0], kb[nb][1], k1_off + ro + nb * 256);
            else as_ldsm4t(kb[nb], k1_off + ro + nb * 256);
          }
        };
        load_keys(0);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const uint32_t ro = buf * ST::DWO + (r >> 1) * 16 + (r & 1) * 128;
          uint32_t v[NJ / 2][4];
#pragma unroll
          for (int j = 0; j < NJ / 2; ++j) as_ldsm4(v[j][0], v[j][1], v[j][2], v[j][3], v1_off + ro + (uint32_t)(j * 16 * AS_DWO_CH));
          float c[2][4];
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) as_mma_first<F16>(c[nb], wk[0][0], wk[0][1], wk[0][2], wk[0][3], kb[nb][0], kb[nb][1]);
          if constexpr (!D16) {
#pragma unroll
            for (int nb = 0; nb < 2; ++nb)
              as_mma<F16>(c[nb], wk[D / 16 - 1][0], wk[D / 16 - 1][1], wk[D / 16 - 1][2], wk[D / 16 - 1][3], kb[nb][2], kb[nb][3]);
          }
          if (r < 3) load_keys(r + 1);
          uint32_t a[4];
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) {
            a[2 * nb] = as_pack_relu<F16>(c[nb][0], c[nb][1]);
            a[2 * nb + 1] = as_pack_relu<F16>(c[nb][2], c[nb][3]);
            if (edge) {  // outputs that do not exist or do not count
              const int x = x0 + 8 * nb + 2 * t;
              const bool in = y + r >= p.row_lo && y + r < p.row_hi;
              const uint32_t m = in ? (x >= 0 && x < p.W ? 0xFFFFu : 0u) | (x + 1 >= 0 && x + 1 < p.W ? 0xFFFF0000u : 0u) : 0u;
              a[2 * nb] &= m; a[2 * nb + 1] &= m;
            }
          }
          as_mma<F16>(accs, a[0], a[1], a[2], a[3], ones1, ones1);
#pragma unroll
          for (int j = 0; j < NJ / 2; ++j) {
            as_mma<F16>(acc1[2 * j], a[0], a[1], a[2], a[3], v[j][0], v[j][1]);
            as_mma<F16>(acc1[2 * j + 1], a[0], a[1], a[2], a[3], v[j][2], v[j][3]);
          }
        }
        arrive(dwo_freed(0, buf));

        const int pb = un.p * p.B + un.b;
        as_advance(p, un, p.kv_tiles_x);
        if (i + 1 < kv_count && un.p * p.B + un.b == pb) continue;
        // The run leaves this (head, image): add the warps' sums in warp order and write them to this CTA's slot.
        float* red = reinterpret_cast<float*>(smem_raw + (dwo + 2 * ST::DWO - smem_u32(smem_raw)));  // [state][warp][16][D + 1]
        float* mine = red + sw * 16 * (D + 1);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int r = g + 8 * (e >> 1);
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            mine[r * (D + 1) + 8 * j + 2 * t + (e & 1)] = acc0[j][e];
            mine[AS_SUM_WARPS * 16 * (D + 1) + r * (D + 1) + 8 * j + 2 * t + (e & 1)] = acc1[j][e];
          }
          if (t == 0) mine[(e & 1) * AS_SUM_WARPS * 16 * (D + 1) + r * (D + 1) + D] = accs[e];
        }
        clear();
        arrive(sums_meet);  // a bounded wait here too: a warp that has given up does not come
        if (!wait(sums_meet, 0)) break;
        // [state][mh][r][c] of the block: d = 32: rows 16 mh + r of one head's states; d = 16: rows r of head mh's
        float* out = p.partial + ((long long)pb + blockIdx.x) * (HPB * 2 * NE);
        for (int e = threadIdx.x - 32 * AS_DW_WARPS; e < HPB * 2 * NE; e += 32 * AS_SUM_WARPS) {
          const int s = D16 ? (e / NE) & 1 : e / NE, r = e - (e / NE) * NE;
          const int half = D16 ? e / (2 * NE) : r / (16 * (D + 1)), rr = D16 ? r : r - half * 16 * (D + 1);
          const float* src = red + (s * AS_SUM_WARPS + half * 4) * 16 * (D + 1) + rr;
          float sum = src[0];
#pragma unroll
          for (int w = 1; w < 4; ++w) sum += src[w * 16 * (D + 1)];
          out[e] = sum;
        }
        arrive(sums_meet);
        if (!wait(sums_meet, 1)) break;
      }
    }
    if (end_of_kv()) {
      // ---------------------------------------------------------------- grouped 1x1 of image rows 2 sw, 2 sw + 1 of the tile
      using ST = AsQ;
      const int sw = warp - AS_DW_WARPS;
      const uint32_t q_off = box + ST::BUFS * ST::BUF + (uint32_t)(lane * AS_DWO_CH + sw * 16);
      // staging: [row][octet][32 channels][8 pixels] (d = 16: [head][row][octet][16 channels][8 pixels])
      const uint32_t stage0 = box + ST::BUFS * ST::BUF + 2 * ST::DWO + (uint32_t)(sw * 2 * (D16 ? 512 : 1024) + g * 16 + t * 4);
      uint32_t wq[2][D / 16][4];  // A fragments of the queries' grouped 1x1: 16-row block m, contraction step ks (d = 16: only ks = m exists)
      int cur_p = -1;
      AsUnit un = as_locate(p, q_first, p.q_tiles_x, p.q_tiles);
#pragma unroll 1
      for (int i = 0; i < q_count; ++i, as_advance(p, un, p.q_tiles_x)) {
        const uint32_t buf = i & 1, ph = (i >> 1) & 1;
        if (un.p != cur_p) {
          cur_p = un.p;
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const uint32_t* wp = reinterpret_cast<const uint32_t*>(p.w_pw + ((long long)plane_of(0, cur_p, D16 ? m : 0) * D + (D16 ? 0 : 16 * m)) * D);
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint32_t* a = wp + (g * D + 16 * ks) / 2 + t;
              wq[m][ks][0] = __ldg(a); wq[m][ks][1] = __ldg(a + 4 * D); wq[m][ks][2] = __ldg(a + 4); wq[m][ks][3] = __ldg(a + 4 * D + 4);
            }
          }
        }
        if (!wait(dwo_full(1, buf), ph)) break;
        const uint32_t my_stage = stage0 + buf * AS_STAGE;
        uint32_t b[4][4];  // block q = 2 nb + half: image row `half`, pixels 8 nb .. + 7
#pragma unroll
        for (int q = 0; q < 4; ++q) as_ldsm4t(b[q], q_off + buf * ST::DWO + (uint32_t)(q * 128));
        float c[4][2][4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            if constexpr (D16) as_mma_first<F16>(c[q][m], wq[m][0][0], wq[m][0][1], wq[m][0][2], wq[m][0][3], b[q][2 * m], b[q][2 * m + 1]);
            else as_mma_first<F16>(c[q][m], wq[m][0][0], wq[m][0][1], wq[m][0][2], wq[m][0][3], b[q][0], b[q][1]);
          }
        if constexpr (!D16) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int m = 0; m < 2; ++m)
              as_mma<F16>(c[q][m], wq[m][D / 16 - 1][0], wq[m][D / 16 - 1][1], wq[m][D / 16 - 1][2], wq[m][D / 16 - 1][3], b[q][2], b[q][3]);
        }
        if (!wait(staging_freed(buf), ph ^ 1)) break;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const int half = q & 1, nb = q >> 1;
            const uint32_t o = my_stage + (uint32_t)(D16 ? m * (AS_STAGE / 2) + half * 512 + nb * 256 : half * 1024 + nb * 512 + m * 256);
            as_sts32(o, as_pack<F16>(c[q][m][0], c[q][m][1]));
            as_sts32(o + 128, as_pack<F16>(c[q][m][2], c[q][m][3]));
          }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        arrive(dwo_freed(1, buf));
        arrive(staged(buf));
      }
    }
  }
  if (!ok && lane == 0) {
    for (int k = 0; k < 64; ++k) __nanosleep(1000);  // copies still in flight land before the CTA retires
    atomicExch(&g_aggstate_timeout_flag, 1);
  }
}

template <int D, bool F16>
msla_status_t launch_agg_state(int grid, const CUtensorMap (&m)[5], const AggStateParams& p, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done{0};
  const msla_status_t s = ensure_smem_attr(attr_done, agg_state_kernel<D, F16>, AS_SMEM);
  if (s != MSLA_OK) return s;
  launch_pdl(agg_state_kernel<D, F16>, dim3((unsigned)grid), dim3(AS_THREADS), AS_SMEM, st, m[0], m[1], m[2], m[3], m[4], p);
  count_launches(1);
  return check_launch(F16 ? "token aggregation and states (fp16)" : "token aggregation and states (bf16)");
}

}  // namespace

AggStatePlan make_agg_state_plan(int B, int heads, int H, int W, int d, int batch, int first) {
  AggStatePlan pl;
  pl.batch = batch;
  pl.first = first;
  const int hpb = 32 / d;
  pl.kv_tiles_x = (W + 2 + AS_TW - 1) / AS_TW;
  pl.q_tiles_x = (W + AS_TW - 1) / AS_TW;
  pl.tiles_y = (H + AS_TH - 1) / AS_TH;
  pl.kv_tiles = (long long)pl.kv_tiles_x * pl.tiles_y;
  const long long blocks = (heads + hpb - 1) / hpb;  // of 32 channels
  pl.kv_units = blocks * batch * pl.kv_tiles;
  const long long q_units = blocks * batch * pl.q_tiles_x * pl.tiles_y, units = pl.kv_units + q_units;
  pl.grid = (int)(units < AGG_STATE_CTAS ? units : AGG_STATE_CTAS);
  // a tile of keys and values takes about 1.85 times one of queries; counted alike where a CTA has few (each must get one)
  pl.kv_cost = units >= 8 * pl.grid ? 37 : 1;
  pl.q_cost = units >= 8 * pl.grid ? 20 : 1;
  pl.cost = pl.kv_cost * pl.kv_units + pl.q_cost * q_units;
  pl.slot_floats = hpb * 2 * d * (d + 1);
  pl.partial_bytes = (size_t)(blocks * B + pl.grid) * pl.slot_floats * sizeof(float);
  return pl;
}

msla_status_t run_agg_state(const void* ms0, void* q1, float* partial, const void* w_dw, const void* w_pw, const AggStatePlan& pl, int B,
                            int heads, int H, int W, int d, int row_lo, int row_hi, bool with_scale0, cudaStream_t st, bool f16) {
  if (H < 2) return fail(MSLA_ERR_UNSUPPORTED, "aggregation on channel-blocked planes: one row");  // no odd rows to map
  if (pl.kv_tiles > 0x7fffffffLL || pl.cost / pl.grid >= 0x7fffffffLL) return fail(MSLA_ERR_UNSUPPORTED, "too many aggregation tiles");
  AggStateParams p{};
  p.partial = partial;
  p.w_dw = (const bf16*)w_dw; p.w_pw = (const bf16*)w_pw;
  p.heads = heads; p.B = B; p.H = H; p.W = W; p.Wb = W / 8;
  p.tiles_y = pl.tiles_y; p.kv_tiles_x = pl.kv_tiles_x; p.q_tiles_x = pl.q_tiles_x;
  p.kv_tiles = (int)pl.kv_tiles; p.q_tiles = pl.q_tiles_x * pl.tiles_y;
  p.row_lo = row_lo; p.row_hi = row_hi; p.with_scale0 = with_scale0 ? 1 : 0;
  p.batch = pl.batch; p.first = pl.first;
  p.kv_units = pl.kv_units; p.cost = pl.cost; p.kv_cost = pl.kv_cost; p.q_cost = pl.q_cost;
  // [plane][8-channel group][octet][row of this parity][64 elements]
  CUtensorMap maps[5];
  const cuuint64_t row = (cuuint64_t)p.Wb * d * 16;
  for (int i = 0; i < 4; ++i) {
    const int odd = i & 1;
    const cuuint64_t dims[5] = {64, (cuuint64_t)((H + 1 - odd) / 2), (cuuint64_t)p.Wb, (cuuint64_t)(d / 8), (cuuint64_t)B * 3 * heads};
    const cuuint64_t strides[4] = {2 * row, (cuuint64_t)d * 16, 128, row * H};
    const cuuint32_t bx[5] = {64, AS_ROWS / 2, (cuuint32_t)(i < 2 ? 3 : 4), (cuuint32_t)(d / 8), 1};
    if (!tma_make_map_bf16(&maps[i], (const char*)ms0 + odd * row, 5, dims, strides, bx, CU_TENSOR_MAP_SWIZZLE_128B))
      return fail(MSLA_ERR_CUDA, "cuTensorMapEncodeTiled failed for the aggregation");
  }
  {  // output of the queries: [plane][row][piece of 64 elements]
    const cuuint64_t dims[4] = {64, (cuuint64_t)p.Wb * d / 8, (cuuint64_t)H, (cuuint64_t)B * heads};
    const cuuint64_t strides[3] = {128, row, row * H};
    const cuuint32_t bx[4] = {64, (cuuint32_t)d / 4, AS_TH, 1};
    if (!tma_make_map_bf16(&maps[4], q1, 4, dims, strides, bx, CU_TENSOR_MAP_SWIZZLE_NONE))
      return fail(MSLA_ERR_CUDA, "cuTensorMapEncodeTiled failed for the aggregation's output");
  }
  if (d == 32) return f16 ? launch_agg_state<32, true>(pl.grid, maps, p, st) : launch_agg_state<32, false>(pl.grid, maps, p, st);
  return f16 ? launch_agg_state<16, true>(pl.grid, maps, p, st) : launch_agg_state<16, false>(pl.grid, maps, p, st);
}

int agg_state_timeout_flag() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_aggstate_timeout_flag, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return v;
}

}  // namespace msla
