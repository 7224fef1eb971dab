// A [rows][cols] matrix of float values as its tf32 high and low parts, written transposed ([cols][rows] each): the operands of
// the weight gradients, whose contraction runs over the rows.
#pragma once
#include "hbp_internal.h"

namespace hbp {

// 64 x 64 tiles through shared memory, 16 bytes per access on both sides where alignment and the row count allow it.  Bound by
// bytes.  Tiles of one row group run one after the other, so that what several columns are formed from (the upstream gradient
// of a gated cell, read for each of four coefficient blocks) comes from L2.  Value: four neighbouring values of a row.
// 131072 x 512 x gradient times tanh' (1.07 GB): 258 -> 163 us (32 x 32 tiles, 4 bytes per access, before); GRU 32768 x 4 x 512 270 ->
// 144; LSTM 32768 x 4 x 512 331 -> 169; GRU 131072 x 4 x 64 133 -> 69.
template <typename Value>
__global__ void __launch_bounds__(256) split_transposed_kernel(const Value value, float* __restrict__ hiT, float* __restrict__ loT, int64_t rows,
                                                               int cols, int col_tiles) {
  // element (column c, row r) of the tile at c * 64 + r, the groups of four rows of a column permuted by c / 4: the four columns
  // that a thread writes and the four rows that one reads then meet at most one other thread in a bank
  __shared__ __align__(16) float tile[64 * 64];
  const int64_t r0 = (int64_t)(blockIdx.x / col_tiles) * 64;
  const int c0 = (int)(blockIdx.x % col_tiles) * 64, t = threadIdx.x;
  {
    const int cq = t & 15, c = c0 + 4 * cq;
    float4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t r = r0 + (t >> 4) + 16 * i;
      v[i] = r < rows && c < cols ? value(r, c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);  // (cols is a multiple of 4)
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int rr = (t >> 4) + 16 * i, at = ((rr >> 2) ^ cq) * 4 + (rr & 3);
      tile[(4 * cq) * 64 + at] = v[i].x;
      tile[(4 * cq + 1) * 64 + at] = v[i].y;
      tile[(4 * cq + 2) * 64 + at] = v[i].z;
      tile[(4 * cq + 3) * 64 + at] = v[i].w;
    }
  }
  __syncthreads();
  const int rq = t & 15;
  const int64_t r = r0 + 4 * rq;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int cc = (t >> 4) + 16 * i, c = c0 + cc;
    if (c >= cols || r >= rows) continue;
    const float4 v = *reinterpret_cast<const float4*>(tile + cc * 64 + ((rq ^ (cc >> 2)) & 15) * 4);
    const float4 h = make_float4(round_tf32(v.x), round_tf32(v.y), round_tf32(v.z), round_tf32(v.w));
    const float4 l = make_float4(round_tf32(v.x - h.x), round_tf32(v.y - h.y), round_tf32(v.z - h.z), round_tf32(v.w - h.w));
    float *ph = hiT + (int64_t)c * rows + r, *pl = loT + (int64_t)c * rows + r;
    if (rows % 4 == 0) {
      *reinterpret_cast<float4*>(ph) = h;
      *reinterpret_cast<float4*>(pl) = l;
    } else {
      const float hs[4] = {h.x, h.y, h.z, h.w}, ls[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (r + k < rows) {
          ph[k] = hs[k];
          pl[k] = ls[k];
        }
    }
  }
}
template <typename Value>
void launch_split_transposed(Launcher& lc, const Value& value, float* hiT, float* loT, int64_t rows, int cols) {
  const int col_tiles = (cols + 63) / 64;
  split_transposed_kernel<Value><<<(unsigned)((rows + 63) / 64 * col_tiles), 256, 0, lc.stream>>>(value, hiT, loT, rows, cols, col_tiles);
  lc.count();
  lc.check();
}

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 mul4(const float4& a, const float4& b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }

}  // namespace hbp
