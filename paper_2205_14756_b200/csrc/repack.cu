// Rows of a length that is no multiple of eight 16-bit elements (feature maps of 14x14, 7x7, ... tokens), to and from rows
// padded to one: tensor maps need row strides of whole 16-byte units, so the tensor-core projections read and write
// padded copies, and these two kernels make the copies.
//
// Both are bound by memory: a thread writes one aligned 16-byte piece and reads the (unaligned) eight elements that go into
// it as aligned 32-bit words, which the lanes of a warp share through L1.  [64, 256, 14, 14] (6.4 MB): about 4 us each way,
// where the plain kernels that such shapes ran on before took 410 us for the two projections, the tensor-core ones about 25.
#include "msla_common.cuh"
#include "msla_host.h"

namespace msla {
namespace {

constexpr int RP_THREADS = 256;

// Elements s .. s + 7 of a 16-bit array (4-byte aligned base) of `total` elements; what lies beyond the end reads as 0.
__device__ __forceinline__ uint4 load8(const unsigned short* __restrict__ src, long long s, long long total) {
  const uint32_t* words = reinterpret_cast<const uint32_t*>(src) + (s >> 1);
  const bool odd = s & 1;
  const long long left = total - (s & ~1LL);  // elements from the first word on
  uint32_t w[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    if (2 * i + 1 < left && (i < 4 || odd)) w[i] = ld_dep32(words + i);
    else if (2 * i < left && (i < 4 || odd)) w[i] = ld_dep16(src + (s & ~1LL) + 2 * i);
    else w[i] = 0u;
  }
  if (!odd) return make_uint4(w[0], w[1], w[2], w[3]);
  return make_uint4(__byte_perm(w[0], w[1], 0x5432), __byte_perm(w[1], w[2], 0x5432), __byte_perm(w[2], w[3], 0x5432), __byte_perm(w[3], w[4], 0x5432));
}

// dst[row][0 .. pitch) <- src[row][0 .. n); the padding holds elements of the next row (no reader looks at it).
__global__ void __launch_bounds__(RP_THREADS)
pad_rows_kernel(const unsigned short* __restrict__ src, uint4* __restrict__ dst, int n, int pieces, long long total, long long count) {
  pdl_first_wait();  // the first kernel of its call
  const long long i = (long long)blockIdx.x * RP_THREADS + threadIdx.x;
  if (i >= count) return;
  const long long row = count <= 0xffffffffLL ? (uint32_t)i / (uint32_t)pieces : i / pieces;
  const int col = (int)(i - row * pieces) * 8;
  dst[i] = load8(src, row * n + col, total);
}

// dst[row][0 .. n) <- src[row][0 .. n) of rows `pitch` apart; a thread writes eight consecutive elements of dst.
__global__ void __launch_bounds__(RP_THREADS)
unpad_rows_kernel(const unsigned short* __restrict__ src, unsigned short* __restrict__ dst, int n, int pitch, long long src_total, long long total) {
  pdl_launch_dependents();
  pdl_wait();
  const long long f = ((long long)blockIdx.x * RP_THREADS + threadIdx.x) * 8;
  if (f >= total) return;
  long long row = total <= 0xffffffffLL ? (uint32_t)f / (uint32_t)n : f / n;
  int col = (int)(f - row * n);
  if (col + 8 <= n) {  // then f + 8 <= total, and f is a multiple of 8: an aligned piece
    *reinterpret_cast<uint4*>(dst + f) = load8(src, row * pitch + col, src_total);
    return;
  }
  unsigned short v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (col == n) { col = 0; ++row; }
    v[e] = f + e < total ? (unsigned short)ld_dep16(src + row * pitch + col) : (unsigned short)0;
    ++col;
  }
  if (f + 8 <= total) {
    uint4 o;
    o.x = v[0] | (uint32_t)v[1] << 16; o.y = v[2] | (uint32_t)v[3] << 16; o.z = v[4] | (uint32_t)v[5] << 16; o.w = v[6] | (uint32_t)v[7] << 16;
    *reinterpret_cast<uint4*>(dst + f) = o;
  } else {
    for (int e = 0; e < 8 && f + e < total; ++e) dst[f + e] = v[e];
  }
}

}  // namespace

msla_status_t run_pad_rows(const void* src, void* dst, long long rows, int n, int pitch, cudaStream_t st) {
  const int pieces = pitch / 8;
  const long long count = rows * pieces;
  if (ceil_div_ll(count, RP_THREADS) > 0x7fffffffLL) return fail(MSLA_ERR_UNSUPPORTED, "too many elements to repack");
  launch_pdl(pad_rows_kernel, dim3((unsigned)ceil_div_ll(count, RP_THREADS)), dim3(RP_THREADS), 0, st, (const unsigned short*)src, (uint4*)dst, n, pieces,
             rows * n, count);
  count_launches(1);
  return check_launch("padding of rows");
}

msla_status_t run_unpad_rows(const void* src, void* dst, long long rows, int n, int pitch, cudaStream_t st) {
  const long long total = rows * n, blocks = ceil_div_ll(total, 8LL * RP_THREADS);
  if (blocks > 0x7fffffffLL) return fail(MSLA_ERR_UNSUPPORTED, "too many elements to repack");
  launch_pdl(unpad_rows_kernel, dim3((unsigned)blocks), dim3(RP_THREADS), 0, st, (const unsigned short*)src, (unsigned short*)dst, n, pitch, rows * pitch, total);
  count_launches(1);
  return check_launch("unpadding of rows");
}

}  // namespace msla
