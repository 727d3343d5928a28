// Kernels on the fp32 pipes for every stage of the module, templated on the storage
// type.  They are the fp32 path (a TF32 tensor-core product would not meet the
// fp32 accuracy bound) and the fallback for 16-bit shapes the tensor-core kernels do
// not cover.  All accumulate in fp32 and are deterministic.
//
// What bounds them is how many multiply-adds a shared-memory access feeds: every inner loop works on a register tile
// (4 x 4 to 8 x 4 outputs) read in 16-byte pieces.  Module [1, 192, 64, 128], d = 32, fp32: 333 us per forward with one or
// two shared-memory loads per multiply-add, F32_NEW us now; [1, 64, 16, 16], d = 16 (all latency): 71 -> F32_SMALL us.
#pragma once

#include "msla_common.cuh"

namespace msla {
namespace generic {

// ---------------------------------------------------------------------------
// Strided GEMM for the two 1x1 projections (Section 3.1: Q = xW_Q, K = xW_K,
// V = xW_V; final linear projection):
//   D(m, n) = sum_k A(m, k) * W[n, k] (+ bias[n]),   m = token, n = out channel
// A(m, k) = A[b*sAb + m*sAm + k*sAk];
// D(m, n) = D[b*sDb + (n / group)*sDg + m*sDm + (n % group)*sDn]: out channels
// may be split into groups of `group` that live in separate planes.
// ---------------------------------------------------------------------------
struct GemmArgs {
  long long sAb, sAm, sAk;
  long long sDb, sDm, sDn, sDg;
  int M, Nc, K;  // tokens, out channels, in channels
  int group;     // out channels per plane (>= Nc: one plane)
  int act;       // applied to the sum + bias: 0 none, 1 ReLU, 2 hard-swish
  const void* residual;  // nullptr, or a tensor laid out like D, added after the activation
};

__device__ __forceinline__ float act_f32(float v, int act) {
  if (act == 1) return fmaxf(v, 0.f);
  if (act == 2) return v * fminf(fmaxf(v + 3.f, 0.f), 6.f) / 6.f;
  return v;
}

// Four consecutive elements, aligned to their total size.
template <typename T> __device__ __forceinline__ float4 load4(const T* p) {
  if constexpr (sizeof(T) == 4) {
    return __ldg(reinterpret_cast<const float4*>(p));
  } else {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    const T* e = reinterpret_cast<const T*>(&v);
    return make_float4(to_f32(e[0]), to_f32(e[1]), to_f32(e[2]), to_f32(e[3]));
  }
}
template <typename T> __device__ __forceinline__ void store4(T* p, const float (&v)[4]) {
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    uint2 o;
    T* e = reinterpret_cast<T*>(&o);
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = from_f32<T>(v[i]);
    *reinterpret_cast<uint2*>(p) = o;
  }
}

// Tile BM x BN, a thread owns TM x 4 outputs (TM / 4 runs of four consecutive tokens, four consecutive channels); the next
// BK-slice of both operands is fetched into registers while the current one is multiplied.  Threads run along whichever
// output index is contiguous in memory.  vec: four consecutive outputs along that index are an aligned vector.
template <typename T, int BM, int BN, int BK, int TM>
__global__ void __launch_bounds__((BM / TM) * (BN / 4))
gemm_kernel(const T* __restrict__ A, const T* __restrict__ Wt, const T* __restrict__ bias,
            T* __restrict__ D, GemmArgs g, bool vec) {
  constexpr int TX = BM / TM, THREADS = TX * (BN / 4);
  constexpr int LA = BM * BK / THREADS, LW = BN * BK / THREADS;
  static_assert(BM * BK % THREADS == 0 && BN * BK % THREADS == 0 && TM % 4 == 0, "tile shape");
  __shared__ __align__(16) float As[2][BK][BM + 4];
  __shared__ __align__(16) float Ws[2][BK][BN + 4];
  pdl_launch_dependents();
  const int tid = threadIdx.x;
  const long long m0 = (long long)blockIdx.x * BM;
  const int n0 = blockIdx.y * BN;
  const int b = blockIdx.z;
  const bool a_m_contig = (g.sAm == 1);
  const bool d_m_contig = (g.sDm == 1);
  const int tm = d_m_contig ? tid % TX : tid / (BN / 4), tn = d_m_contig ? tid / TX : tid % (BN / 4);
  const T* Ab = A + (long long)b * g.sAb;
  float ra[LA], rw[LW];
  auto fetch_w = [&](int k0) {
#pragma unroll
    for (int i = 0; i < LW; ++i) {
      const int e = tid + i * THREADS, k = e % BK, n = e / BK;
      rw[i] = n0 + n < g.Nc && k0 + k < g.K ? to_f32(__ldg(Wt + (long long)(n0 + n) * g.K + k0 + k)) : 0.f;
    }
  };
  auto fetch_a = [&](int k0) {
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + i * THREADS, m = a_m_contig ? e % BM : e / BK, k = a_m_contig ? e / BM : e % BK;
      ra[i] = m0 + m < g.M && k0 + k < g.K ? to_f32(Ab[(m0 + m) * g.sAm + (long long)(k0 + k) * g.sAk]) : 0.f;
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + i * THREADS;
      if (a_m_contig) As[buf][e / BM][e % BM] = ra[i];
      else As[buf][e % BK][e / BK] = ra[i];
    }
#pragma unroll
    for (int i = 0; i < LW; ++i) {
      const int e = tid + i * THREADS;
      Ws[buf][e % BK][e / BK] = rw[i];
    }
  };
  float acc[TM][4] = {};
  fetch_w(0);
  pdl_wait();  // the weights do not come from the previous kernel
  fetch_a(0);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < g.K; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < g.K;
    if (more) { fetch_w(k0 + BK); fetch_a(k0 + BK); }
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM];
#pragma unroll
      for (int r = 0; r < TM / 4; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(&As[buf][k][r * (TX * 4) + tm * 4]);
        a[4 * r] = v.x; a[4 * r + 1] = v.y; a[4 * r + 2] = v.z; a[4 * r + 3] = v.w;
      }
      const float4 w = *reinterpret_cast<const float4*>(&Ws[buf][k][tn * 4]);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        acc[i][0] = fmaf(a[i], w.x, acc[i][0]);
        acc[i][1] = fmaf(a[i], w.y, acc[i][1]);
        acc[i][2] = fmaf(a[i], w.z, acc[i][2]);
        acc[i][3] = fmaf(a[i], w.w, acc[i][3]);
      }
    }
    if (more) put(buf ^ 1);  // last read before the previous barrier
    __syncthreads();
  }
  T* Db = D + (long long)b * g.sDb;
  const T* Rb = static_cast<const T*>(g.residual) + (g.residual ? (long long)b * g.sDb : 0);
  const int n = n0 + tn * 4;  // Nc is a multiple of 8: all four channels exist or none does
  if (n >= g.Nc) return;
  float bv[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) bv[j] = bias ? to_f32(bias[n + j]) : 0.f;
  const long long at_n = (long long)(n / g.group) * g.sDg + (long long)(n % g.group) * g.sDn;  // four channels share a plane
#pragma unroll
  for (int r = 0; r < TM / 4; ++r) {
    const long long m = m0 + r * (TX * 4) + tm * 4;
#pragma unroll
    for (int u = 0; u < 4; ++u) {  // a vector: four tokens of channel n + u, or four channels of token m + u
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = act_f32(d_m_contig ? acc[4 * r + e][u] + bv[u] : acc[4 * r + u][e] + bv[e], g.act);
      const long long at = at_n + (d_m_contig ? m * g.sDm + u * g.sDn : (m + u) * g.sDm);
      const int count = d_m_contig ? (int)min(4LL, g.M - m) : (m + u < g.M ? 4 : 0);
      const long long step = d_m_contig ? g.sDm : g.sDn;
      if (vec && count == 4) {
        if (g.residual) {
          const float4 x = load4(Rb + at);
          v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
        }
        store4(Db + at, v);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e < count) Db[at + e * step] = from_f32<T>(g.residual ? v[e] + to_f32(Rb[at + e * step]) : v[e]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The depthwise 3x3 convolution inside the FFN (Section 3.1, Fig. 2 left) with its bias and activation, on NCHW:
//   g[b,c,y,x] = act(sum_{dy,dx} w[c,dy,dx] * h[b,c,y+dy-1,x+dx-1] + bias[c]), zero padding 1.  One thread per output.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
ffn_dw3x3_nchw_kernel(const T* __restrict__ h, const T* __restrict__ w, const T* __restrict__ bias, T* __restrict__ g,
                      int Ch, int H, int W, int act, long long total) {
  const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
  if (idx >= total) return;
  const int x = (int)(idx % W), y = (int)((idx / W) % H);
  const long long bc = idx / ((long long)W * H);
  const int c = (int)(bc % Ch);
  const T* hp = h + bc * H * W;
  float acc = bias ? to_f32(bias[c]) : 0.f;
  for (int dy = 0; dy < 3; ++dy) {
    const int yy = y + dy - 1;
    if (yy < 0 || yy >= H) continue;
    for (int dx = 0; dx < 3; ++dx) {
      const int xx = x + dx - 1;
      if (xx < 0 || xx >= W) continue;
      acc = fmaf(to_f32(w[(long long)c * 9 + dy * 3 + dx]), to_f32(hp[(long long)yy * W + xx]), acc);
    }
  }
  g[idx] = from_f32<T>(act_f32(acc, act));
}

// 3x3 depthwise taps embedded in a 5x5 filter with a ring of zeros: w5[c][r][s] = w3[c][r-1][s-1] inside, 0 outside.
template <typename T>
__global__ void __launch_bounds__(256)
embed_taps_kernel(const T* __restrict__ w3, T* __restrict__ w5, long long total) {
  const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
  if (idx >= total) return;
  const long long c = idx / 25;
  const int r = (int)(idx % 25) / 5, s = (int)(idx % 5);
  const bool inside = r >= 1 && r <= 3 && s >= 1 && s <= 3;
  w5[idx] = inside ? w3[c * 9 + (r - 1) * 3 + (s - 1)] : from_f32<T>(0.f);
}

// ---------------------------------------------------------------------------
// Multi-scale token aggregation (Section 3.1): 5x5 depthwise convolution
// (cross-correlation, zero padding 2) followed by the grouped 1x1 convolution,
// on planar activations [B, groups, H*W, D].  One CTA = one tile of TH x TW pixels of
// one group.  src(b, g, n, i) = src[b*src_sb + (g*H*W + n)*D + i]; dst likewise with dst_sb.
// A lane keeps one channel (D = 16: the half-warps take different pixels): the depthwise step slides down a strip of
// four pixel columns and eight rows with five rows of sums in registers (8 shared-memory loads per 100 multiply-adds), the
// 1x1 step holds the channel's D weights in registers and reads the depthwise results as broadcast 16-byte pieces.
// ---------------------------------------------------------------------------
template <typename T, int D, int TH, int TW>
__global__ void __launch_bounds__(TH * TW * D / 32)
aggregate_kernel(const T* __restrict__ src, const T* __restrict__ w_dw, const T* __restrict__ w_pw,
                 T* __restrict__ dst, int H, int W, long long src_sb, long long dst_sb) {
  constexpr int THREADS = TH * TW * D / 32;  // a strip of 32 pixels per lane
  constexpr int HW_ = TW + 4, HH = TH + 4, CV = D / 4;
  static_assert(TH % 8 == 0 && TW % 4 == 0, "strips of 4 x 8 pixels");
  extern __shared__ __align__(16) float agg_smem[];
  float* tile = agg_smem;                  // [HH][HW_][D]
  float* dwo = agg_smem + HH * HW_ * D;    // [TH * TW][D]
  pdl_launch_dependents();
  const int tid = threadIdx.x;
  const int tiles_x = (W + TW - 1) / TW;
  const int x0 = (blockIdx.x % tiles_x) * TW, y0 = (blockIdx.x / tiles_x) * TH;
  const int ch0 = blockIdx.y * D;
  const int b = blockIdx.z;
  const int c = tid % D, strip = tid / D;  // strips: row-major over (TH / 8) x (TW / 4)
  float taps[25], pw[D];
#pragma unroll
  for (int i = 0; i < D; i += 4) {
    const float4 v = load4(w_pw + (long long)(ch0 + c) * D + i);
    pw[i] = v.x; pw[i + 1] = v.y; pw[i + 2] = v.z; pw[i + 3] = v.w;
  }
  pdl_wait();  // the 1x1 weights do not come from the previous kernel; the taps may (a 3x3 filter embedded in 5x5)
#pragma unroll
  for (int i = 0; i < 25; ++i) taps[i] = to_f32(__ldg(w_dw + (long long)(ch0 + c) * 25 + i));
  const T* sb = src + (long long)b * src_sb + (long long)blockIdx.y * H * W * D;
  for (int e = tid; e < HH * HW_ * CV; e += THREADS) {
    const int cv = e % CV, p = e / CV;
    const int yy = y0 + p / HW_ - 2, xx = x0 + p % HW_ - 2;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (yy >= 0 && yy < H && xx >= 0 && xx < W) v = load4(sb + ((long long)yy * W + xx) * D + cv * 4);
    *reinterpret_cast<float4*>(tile + p * D + cv * 4) = v;
  }
  __syncthreads();
  {
    const int sx = (strip % (TW / 4)) * 4, sy = strip / (TW / 4) * 8;
    const float* t0 = tile + (sy * HW_ + sx) * D + c;
    float acc[5][4];
#pragma unroll
    for (int r = 0; r < 12; ++r) {  // staged row r feeds output rows r - 4 .. r of the strip
      float in[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) in[x] = t0[(r * HW_ + x) * D];
#pragma unroll
      for (int dy = 0; dy < 5; ++dy) {
        const int o = r - dy;
        if (o < 0 || o >= 8) continue;
        float (&a)[4] = acc[o % 5];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          float v = dy == 0 ? 0.f : a[x];
#pragma unroll
          for (int dx = 0; dx < 5; ++dx) v = fmaf(taps[dy * 5 + dx], in[x + dx], v);
          a[x] = v;
        }
      }
      if (r >= 4) {
#pragma unroll
        for (int x = 0; x < 4; ++x) dwo[((sy + r - 4) * TW + sx + x) * D + c] = acc[(r - 4) % 5][x];
      }
    }
  }
  __syncthreads();
  T* db = dst + (long long)b * dst_sb + (long long)blockIdx.y * H * W * D;
#pragma unroll 2
  for (int i = 0; i < 32; ++i) {
    const int p = strip + i * (THREADS / D);
    const int yy = y0 + p / TW, xx = x0 + p % TW;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int k = 0; k < D; k += 4) {
      const float4 v = *reinterpret_cast<const float4*>(dwo + p * D + k);
      a0 = fmaf(pw[k], v.x, a0); a1 = fmaf(pw[k + 1], v.y, a1); a2 = fmaf(pw[k + 2], v.z, a2); a3 = fmaf(pw[k + 3], v.w, a3);
    }
    if (yy < H && xx < W) db[((long long)yy * W + xx) * D + c] = from_f32<T>((a0 + a1) + (a2 + a3));
  }
}
template <int D, int TH, int TW> constexpr int aggregate_smem() { return ((TH + 4) * (TW + 4) + TH * TW) * D * 4; }

// ---------------------------------------------------------------------------
// KV-state reduction, first level (Eq. 3): for one (batch, head) and one chunk
// of tokens,  part[a][c] = sum_j relu(k[j,a]) * v[j,c]  for c < d and
// part[a][d] = sum_j relu(k[j,a]).   Partials: [BH][S][d*(d+1)] fp32.
// ---------------------------------------------------------------------------
// Every warp stages 16 tokens of K and V at a time in its own part of shared memory (the next 16 in registers meanwhile) and
// keeps a whole state in registers, 4 x 8 entries per lane (D = 16: four lane groups take every fourth token): three
// 16-byte shared-memory loads per 32 multiply-adds.  Sums are added in lane-group, then warp order.
template <typename T, int D>
__global__ void __launch_bounds__(128)
kv_partial_kernel(const T* __restrict__ k, const T* __restrict__ v, float* __restrict__ partial,
                  HeadView kv, int heads, int N, int S, int chunk) {
  constexpr int WARPS = 4, TT = 16, D1 = D + 1, NE = D * D1, CV = D / 4;
  constexpr int LANES = (D / 4) * (D / 8), SUB = 32 / LANES;  // lanes per state, states per warp
  constexpr int LD = TT * CV / 32;                            // 16-byte loads per lane and operand
  __shared__ __align__(16) float sm[(WARPS * 2 * TT * D > WARPS * SUB * NE) ? WARPS * 2 * TT * D : WARPS * SUB * NE];
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bh = blockIdx.x, s = blockIdx.y;
  const int b = bh / heads, h = bh % heads;
  const long long base = (long long)b * kv.batch + (long long)h * kv.head;
  const int n_begin = s * chunk, n_end = min(N, n_begin + chunk);
  float* Ks = sm + warp * (2 * TT * D);
  float* Vs = Ks + TT * D;
  const int sub = lane / LANES, li = lane % LANES, a0 = li / (D / 8) * 4, c0 = li % (D / 8) * 8;
  float acc[4][8] = {}, ks[4] = {};
  float4 rk[LD], rv[LD];
  auto fetch = [&](int n0) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = lane + 32 * i, n = n0 + e / CV;
      const bool ok = n < n_end;
      const long long off = base + (long long)(ok ? n : n_begin) * kv.ld + e % CV * 4;
      rk[i] = ok ? load4(k + off) : make_float4(0.f, 0.f, 0.f, 0.f);
      rv[i] = ok ? load4(v + off) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  int n0 = n_begin + warp * TT;
  if (n0 < n_end) fetch(n0);
  for (; n0 < n_end; n0 += WARPS * TT) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = lane + 32 * i;
      const float4 r = make_float4(fmaxf(rk[i].x, 0.f), fmaxf(rk[i].y, 0.f), fmaxf(rk[i].z, 0.f), fmaxf(rk[i].w, 0.f));
      *reinterpret_cast<float4*>(Ks + e * 4) = r;
      *reinterpret_cast<float4*>(Vs + e * 4) = rv[i];
    }
    __syncwarp();
    if (n0 + WARPS * TT < n_end) fetch(n0 + WARPS * TT);
#pragma unroll 4
    for (int t = sub; t < TT; t += SUB) {
      const float4 a = *reinterpret_cast<const float4*>(Ks + t * D + a0);
      const float4 x = *reinterpret_cast<const float4*>(Vs + t * D + c0), y = *reinterpret_cast<const float4*>(Vs + t * D + c0 + 4);
      const float av[4] = {a.x, a.y, a.z, a.w}, cv[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ks[i] += av[i];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], cv[j], acc[i][j]);
      }
    }
    __syncwarp();
  }
  __syncthreads();  // every warp has left its staging
  float* mine = sm + (warp * SUB + sub) * NE;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = 0; j < 8; ++j) mine[(a0 + i) * D1 + c0 + j] = acc[i][j];
    if (c0 == 0) mine[(a0 + i) * D1 + D] = ks[i];
  }
  __syncthreads();
  float* out = partial + ((long long)bh * S + s) * NE;
  for (int e = threadIdx.x; e < NE; e += WARPS * 32) {
    float sum = sm[e];
#pragma unroll
    for (int w = 1; w < WARPS * SUB; ++w) sum += sm[w * NE + e];
    out[e] = sum;
  }
}

// Second level: state[bh][e] = partial[bh][0][e] + partial[bh][1][e] + ... in
// index order, so the result does not depend on scheduling.
__global__ void __launch_bounds__(256)
kv_combine_kernel(const float* __restrict__ partial, float* __restrict__ state, int S, int ne,
                  long long total) {
  pdl_launch_dependents();
  pdl_wait();
  const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
  if (idx >= total) return;
  const long long bh = idx / ne;
  const int e = (int)(idx % ne);
  const float* p = partial + bh * S * ne + e;
  float acc = 0.f;
  for (int s = 0; s < S; ++s) acc += p[(long long)s * ne];
  state[idx] = acc;
}

// Token-sharded forward: state[i] = states[0][i] + states[1][i] + ... over the R bands of the image in band
// order (Eq. 3's sums over tokens, cut into bands), the same order on every rank.
__global__ void __launch_bounds__(256)
band_state_sum_kernel(const float* __restrict__ states, float* __restrict__ state, int R, long long total) {
  const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
  if (idx >= total) return;
  float acc = 0.f;
  for (int r = 0; r < R; ++r) acc += states[(long long)r * total + idx];
  state[idx] = acc;
}

// ---------------------------------------------------------------------------
// Apply step (Eq. 3): out[i,c] = relu(q[i]) . KV[:,c] / (relu(q[i]) . ks + eps),
// written at channel offset head*D of the output view (head concat).
// One thread per token with its D sums in registers; state [BH][D*(D+1)] fp32 staged in shared memory with rows of
// D + 4 floats, read as broadcast 16-byte pieces (one per four multiply-adds).
// ---------------------------------------------------------------------------
template <typename T, int D>
__global__ void __launch_bounds__(128)
apply_kernel(const T* __restrict__ q, const float* __restrict__ state, T* __restrict__ out,
             HeadView qv, HeadView ov, int heads, int N, float eps) {
  constexpr int D1 = D + 1, P = D + 4;
  __shared__ __align__(16) float st[D * P];
  pdl_launch_dependents();
  pdl_wait();
  const int bh = blockIdx.y;
  const int b = bh / heads, h = bh % heads;
  for (int e = threadIdx.x; e < D * D1; e += 128) st[e / D1 * P + e % D1] = state[(long long)bh * D * D1 + e];
  const int n = blockIdx.x * 128 + threadIdx.x;
  const T* qp = q + (long long)b * qv.batch + (long long)h * qv.head + (long long)min(n, N - 1) * qv.ld;
  float qr[D];
#pragma unroll
  for (int a = 0; a < D; a += 4) {
    const float4 x = load4(qp + a);
    qr[a] = fmaxf(x.x, 0.f); qr[a + 1] = fmaxf(x.y, 0.f); qr[a + 2] = fmaxf(x.z, 0.f); qr[a + 3] = fmaxf(x.w, 0.f);
  }
  __syncthreads();
  if (n >= N) return;
  T* op = out + (long long)b * ov.batch + (long long)h * ov.head + (long long)n * ov.ld;
  float den = 0.f, num[D];
#pragma unroll
  for (int c = 0; c < D; ++c) num[c] = 0.f;
#pragma unroll
  for (int a = 0; a < D; ++a) {
#pragma unroll
    for (int c = 0; c < D; c += 4) {
      const float4 x = *reinterpret_cast<const float4*>(st + a * P + c);
      num[c] = fmaf(qr[a], x.x, num[c]); num[c + 1] = fmaf(qr[a], x.y, num[c + 1]);
      num[c + 2] = fmaf(qr[a], x.z, num[c + 2]); num[c + 3] = fmaf(qr[a], x.w, num[c + 3]);
    }
    den = fmaf(qr[a], st[a * P + D], den);
  }
  const float inv = 1.f / (den + eps);
#pragma unroll
  for (int c = 0; c < D; c += 4) {
    const float o[4] = {num[c] * inv, num[c + 1] * inv, num[c + 2] * inv, num[c + 3] * inv};
    store4(op + c, o);
  }
}

}  // namespace generic
}  // namespace msla
