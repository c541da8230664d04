// cache_fp8.cuh -- the write of the E4M3 reference cache (the approximate
// variant of the exact cache of Sec. 3.3, Eq. 2): the cached rows' K and V
// quantised per (128-row tile of one request, head) with one fp32 scale each:
//   amax = max |x| over the tile's rows and the head's 128 columns
//   s    = amax / 448,  code = E4M3(x * (448 / amax))   (0 when amax = 0)
// with IEEE fp32 division and multiply and round-to-nearest-even conversion.
// Layout of one layer:
//   k8     [rows_pad, H, 128]   codes, rows in cache order
//   vt8    [H, 128, rows_pad]   codes of V, transposed per head (K-major B
//                               operand of the P.V MMA)
//   scales [rows_pad / 128, H]  float4 (s_K, s_V, log2 s_V, 1 / s_V); the last
//                               two (0 when s_V = 0) spare the attention kernel a
//                               logarithm and a division per tile
// Each request's rows start on a 128-row boundary; pad rows hold code 0.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

#include "ptx.cuh"

namespace rc {

// One 128-row tile of the cache: rows [src_row0, src_row0 + valid) of the
// prefill tensors go to rows [dst_row0, dst_row0 + 128) of the cache.
struct QuantTile {
  int32_t src_row0, valid, dst_row0, pad;
};

__device__ __forceinline__ float block_amax_256(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = red[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) r = fmaxf(r, red[w]);
  return r;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// grid (H, tiles, 2): blockIdx.z = 0 quantises the tile's K, 1 its V (heads
// fastest, so that CTAs running together read neighbouring bytes of the same
// rows); 256 threads.
//
// Bound by memory: 4 bytes read and 2 written per cached element of K and V.
// Every warp instruction moves whole 128-byte lines: 16 lanes take one head of a
// row (8 columns = 16 bytes each), so a load covers two rows, and thread
// (row group g = i / 16, c = i % 16) holds rows [8 g, 8 g + 8), columns
// [8 c, 8 c + 8).  K codes leave as they lie (8 bytes a lane).  V codes are
// transposed 8 x 8 in registers and through shared memory: the 8-byte word of
// rows [8 g, 8 g + 8) of column d is word g ^ ((d / 8) % 16) of the column's 128
// bytes, which spreads both the stores (16 columns 8 apart) and the reads (a
// column's 128 bytes) over all banks.  (With a lane per four rows each load and K
// store touched 32 rows' sectors, and the build of a 1024^2 request with two
// references, 42 us of it here, took 3 % longer.)
//
// Like copy_rows_kernel it reads only the static inputs and goes behind the
// prefill as its programmatic dependent: its CTAs fill in as the prefill's leave.
// (Before the prefill a build of nine heads, two requests of 740 and 5694 cached
// rows, took 112 us, behind it 107.)
struct QuantArgs {
  const QuantTile* tiles;
  int32_t n_tiles, num_heads;
  const uint4 *src_k, *src_v;
  uint8_t *k8, *vt8;
  float4* scales;
  int64_t rows_pad;
};
constexpr int kQuantThreads = 256;
__global__ void __launch_bounds__(kQuantThreads, 3) quantize_cache_kernel(const QuantArgs a) {
  if (threadIdx.x == 0) grid_launch_dependents();
  constexpr int D = 128;
  const int H = a.num_heads;
  const int64_t rows_pad = a.rows_pad;
  __shared__ float red[8];
  __shared__ __align__(16) uint2 vt[D][16];  // V^T codes of the tile: [d][word of 8 rows, swizzled]
  const QuantTile t = a.tiles[blockIdx.y];
  const int h = blockIdx.x;
  const bool is_v = blockIdx.z != 0;
  const int g = threadIdx.x >> 4;  // rows 8 g .. 8 g + 7
  const int c = threadIdx.x & 15;  // columns 8 c .. 8 c + 7
  const int64_t row_u4 = static_cast<int64_t>(H) * D / 8;
  const uint4* src = (is_v ? a.src_v : a.src_k) + static_cast<int64_t>(t.src_row0 + 8 * g) * row_u4 + h * (D / 8) + c;
  uint4 x[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) x[r] = 8 * g + r < t.valid ? src[r * row_u4] : make_uint4(0, 0, 0, 0);
  float m = 0.f;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint32_t w[4] = {x[r].x, x[r].y, x[r].z, x[r].w};
#pragma unroll
    for (int e = 0; e < 4; ++e) m = fmax3(m, fabsf(bf16_lo(w[e])), fabsf(bf16_hi(w[e])));
  }
  const float amax = block_amax_256(m, red);
  const float inv = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
  // codes of the 8 columns of row r: two words of four codes
  uint2 cw[8];
#pragma unroll
  for (int r = 0; r < 8; ++r)
    cw[r] = make_uint2(pack_e4m3x4(__fmul_rn(bf16_lo(x[r].x), inv), __fmul_rn(bf16_hi(x[r].x), inv),
                                   __fmul_rn(bf16_lo(x[r].y), inv), __fmul_rn(bf16_hi(x[r].y), inv)),
                       pack_e4m3x4(__fmul_rn(bf16_lo(x[r].z), inv), __fmul_rn(bf16_hi(x[r].z), inv),
                                   __fmul_rn(bf16_lo(x[r].w), inv), __fmul_rn(bf16_hi(x[r].w), inv)));
  if (!is_v) {
    const int64_t row = static_cast<int64_t>(H) * D;
    uint8_t* dst = a.k8 + (t.dst_row0 + 8 * g) * row + static_cast<int64_t>(h) * D + 8 * c;
#pragma unroll
    for (int r = 0; r < 8; ++r) *reinterpret_cast<uint2*>(dst + r * row) = cw[r];
    if (threadIdx.x == 0) a.scales[static_cast<int64_t>(t.dst_row0 >> 7) * H + h].x = __fdiv_rn(amax, 448.f);
    grid_dependency_wait();
    return;
  }
  // column 8 c + 4 w + e: byte e of word w of each of the eight rows
#pragma unroll
  for (int w = 0; w < 2; ++w)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      uint32_t col[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t r0 = w ? cw[4 * u].y : cw[4 * u].x, r1 = w ? cw[4 * u + 1].y : cw[4 * u + 1].x;
        const uint32_t r2 = w ? cw[4 * u + 2].y : cw[4 * u + 2].x, r3 = w ? cw[4 * u + 3].y : cw[4 * u + 3].x;
        col[u] = __byte_perm(__byte_perm(r0, r1, 0x0040 + e * 0x0011), __byte_perm(r2, r3, 0x0040 + e * 0x0011), 0x5410);
      }
      vt[8 * c + 4 * w + e][g ^ c] = make_uint2(col[0], col[1]);
    }
  __syncthreads();
  // V^T rows: 128 d rows of 128 codes, 16 bytes per thread and step: words
  // 2 ch and 2 ch + 1 of row d lie side by side, exchanged where d / 8 is odd
  uint8_t* vbase = a.vt8 + static_cast<int64_t>(h) * D * rows_pad + t.dst_row0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int idx = threadIdx.x + 256 * i;  // 0..1023 = d * 8 + chunk
    const int d = idx >> 3, ch = idx & 7, z = d >> 3;
    const uint4 y = *reinterpret_cast<const uint4*>(&vt[d][2 * (ch ^ (z >> 1))]);
    *reinterpret_cast<uint4*>(vbase + static_cast<int64_t>(d) * rows_pad + 16 * ch) =
        z & 1 ? make_uint4(y.z, y.w, y.x, y.y) : y;
  }
  if (threadIdx.x == 0) {
    const float sv = __fdiv_rn(amax, 448.f);
    float4* dst = &a.scales[static_cast<int64_t>(t.dst_row0 >> 7) * H + h];
    dst->y = sv;
    dst->z = sv > 0.f ? log2f(sv) : 0.f;
    dst->w = sv > 0.f ? __frcp_rn(sv) : 0.f;
  }
  grid_dependency_wait();
}

}  // namespace rc
