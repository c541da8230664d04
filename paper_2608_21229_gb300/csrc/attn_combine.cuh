// attn_combine.cuh -- merge the parts of split items.
//
// When the items of a launch do not divide evenly over the GPU's CTA pairs,
// the last items are split by key range into parts that run on otherwise idle
// pairs.  Each part p of an item leaves, for every query row, its own
// normalised output O_p = (sum_j p_j v_j) / l_p and L_p = m_p + log l_p over
// its keys.  Over all keys of the item the softmax normaliser is
// l = sum_p exp(L_p), so the item's output is
//   O = sum_p exp(L_p - L) O_p   with   L = log sum_p exp(L_p),
// computed here with L_max subtracted first.
//
// Parts lie in the workspace as [part][D / 4][rows_per_part] float4 (the layout
// in which the attention kernel's epilogue, a row per thread, writes whole
// lines); a warp takes 32 rows and reads runs of 512 bytes, and the outputs go
// through shared memory so that rows are written whole.
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"
#include "ptx.cuh"

namespace rc {

constexpr int kMaxParts = 8;
constexpr int kCombineRows = 32;

// grid = (ceil(rows / 32), jobs, D / (32 kQ)), 256 threads: lane = row, kQ column
// quads per thread.
//
// Two forms.  Few jobs leave the SMs idle and wait for memory, part after part: with
// kAhead all parts' loads are in flight before the first is used, and a block takes
// 64 columns.  Many jobs are bound by the L2's bandwidth and by the number of blocks
// that fit on an SM (57 registers against 92): a block takes all columns, part after
// part.  us a call, back to back, 256 rows of 128 columns, ahead / part after part:
//   jobs     2 parts       4 parts        8 parts
//      4   2.0 /  2.7    2.1 /  3.5     2.4 /  4.6
//     12   2.4 /  2.8    2.5 /  3.6     2.9 /  4.7
//     18   2.4 /  2.9    2.6 /  3.7     3.1 /  4.8
//     24   3.5 /  3.0    4.0 /  3.8     4.8 /  5.1
//     76   7.2 /  4.0    7.7 /  5.2    10.6 /  7.4
// (A step with 256 live and 8192 cached rows, 4 heads, 8 parts: 17.6 us part after
// part, 13.8 ahead.)
// The line (launch_combine) lies where the blocks of the first form fill two per SM.
template <int D, int kQ, bool kAhead>
__global__ void __launch_bounds__(256) combine_parts_kernel(const CombineJob* __restrict__ jobs,
                                                            const float* __restrict__ part_o,
                                                            const float* __restrict__ part_lse, int rows_per_part,
                                                            __nv_bfloat16* __restrict__ out, float* __restrict__ lse,
                                                            int64_t row_stride, int num_heads) {
  static_assert(D % (32 * kQ) == 0, "eight warps of kQ column quads");
  constexpr int kCols = 32 * kQ;     // columns of this block
  constexpr int kPitch = kCols + 8;  // bf16 elements of a staged row (16 bytes of padding)
  __shared__ __align__(16) __nv_bfloat16 tile[kCombineRows * kPitch];
  const CombineJob job = jobs[blockIdx.y];  // written when the cache was created
  const int r0 = blockIdx.x * kCombineRows, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = r0 + lane, col0 = kCols * blockIdx.z;
  grid_dependency_wait();  // the attention kernel's parts are complete
  if (threadIdx.x == 0) grid_launch_dependents();
  if (r0 >= job.q_rows) return;
  const bool ok = r < job.q_rows;
  const int np = min(job.nparts, kMaxParts);
  const float4* src = reinterpret_cast<const float4*>(part_o) +
                      (static_cast<int64_t>(job.part0) * (D / 4) + col0 / 4 + warp) * rows_per_part + r;
  auto load = [&](int p, int c) { return src[(static_cast<int64_t>(p) * (D / 4) + 8 * c) * rows_per_part]; };
  float w[kMaxParts];
  float4 ahead[kMaxParts][kQ];
#pragma unroll
  for (int p = 0; p < kMaxParts; ++p) {
    w[p] = p < np && ok ? part_lse[static_cast<int64_t>(job.part0 + p) * rows_per_part + r] : -INFINITY;
    if (kAhead && p < np && ok) {
#pragma unroll
      for (int c = 0; c < kQ; ++c) ahead[p][c] = load(p, c);
    }
  }
  float lmax = -INFINITY;
#pragma unroll
  for (int p = 0; p < kMaxParts; ++p) lmax = fmaxf(lmax, w[p]);
  float wsum = 0.f;
#pragma unroll
  for (int p = 0; p < kMaxParts; ++p) {
    w[p] = p < np && ok ? expf(w[p] - lmax) : 0.f;
    wsum += w[p];
  }
  float4 acc[kQ];
#pragma unroll
  for (int c = 0; c < kQ; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int p = 0; p < kMaxParts; ++p) {
    if (p < np && ok) {
#pragma unroll
      for (int c = 0; c < kQ; ++c) {
        const float4 x = kAhead ? ahead[p][c] : load(p, c);
        acc[c].x += w[p] * x.x, acc[c].y += w[p] * x.y, acc[c].z += w[p] * x.z, acc[c].w += w[p] * x.w;
      }
    }
  }
  const float inv = 1.0f / wsum;
#pragma unroll
  for (int c = 0; c < kQ; ++c) {
    uint2 packed;
    packed.x = pack_bf16x2(acc[c].x * inv, acc[c].y * inv);
    packed.y = pack_bf16x2(acc[c].z * inv, acc[c].w * inv);
    *reinterpret_cast<uint2*>(&tile[lane * kPitch + 4 * (warp + 8 * c)]) = packed;
  }
  if (lse && blockIdx.z == 0 && warp == 0 && ok)
    lse[(static_cast<int64_t>(job.q_row0) + r) * num_heads + job.head] = lmax + logf(wsum);
  __syncthreads();
  constexpr int kNC = kCols / 8;  // 16-byte chunks of a row
  for (int i = threadIdx.x; i < kCombineRows * kNC; i += 256) {
    const int rr = i / kNC, ch = i % kNC;
    if (r0 + rr < job.q_rows)
      *reinterpret_cast<uint4*>(out + (static_cast<int64_t>(job.q_row0) + r0 + rr) * row_stride +
                                static_cast<int64_t>(job.head) * D + col0 + 8 * ch) =
          *reinterpret_cast<const uint4*>(&tile[rr * kPitch + 8 * ch]);
  }
}

}  // namespace rc
