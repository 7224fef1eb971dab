// A float as three bf16 parts that add up to it: the form in which float operands reach the tensor cores.
#pragma once
#include <cuda.h>

#include "hbp_internal.h"

namespace hbp {

__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void split_rest2(uint32_t h, float ra, float rb, uint32_t& m, uint32_t& l) {
  m = pack_bf16(ra, rb);
  l = pack_bf16(ra - __uint_as_float(m << 16), rb - __uint_as_float(m & 0xffff0000u));
}
// a and b, each as three bf16 parts that add up to it exactly (24 bits; below 2^-109 the low part runs into the denormals and
// loses bits), packed in pairs.  For magnitudes (as bits) below kPlainParts, whose high part rounds to a finite value (from there on
// a part is infinite or NaN).
constexpr uint32_t kPlainParts = 0x7f7f8000u;
__device__ __forceinline__ void split_plain2(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack_bf16(a, b);
  split_rest2(h, a - __uint_as_float(h << 16), b - __uint_as_float(h & 0xffff0000u), m, l);
}
// The same for any: where rounding the high part would make a finite value infinite it is cut off instead; an infinity or a NaN
// is its high part, the others zero.  So the sum of the parts is the value, whatever it is.
__device__ __forceinline__ void split_parts2(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  const uint32_t ua = __float_as_uint(a) & 0x7fffffffu, ub = __float_as_uint(b) & 0x7fffffffu;
  if (max(ua, ub) < kPlainParts) return split_plain2(a, b, h, m, l);
  const uint32_t inf = 0x7f800000u;
  h = pack_bf16(a, b);
  if (ua >= kPlainParts && ua < inf) h = (h & 0xffff0000u) | (__float_as_uint(a) >> 16);
  if (ub >= kPlainParts && ub < inf) h = (h & 0x0000ffffu) | (__float_as_uint(b) & 0xffff0000u);
  split_rest2(h, ua < inf ? a - __uint_as_float(h << 16) : 0.0f, ub < inf ? b - __uint_as_float(h & 0xffff0000u) : 0.0f, m, l);
}

// The tensor core truncates: the sums of 32 of K are 4.5e-8 of themselves (normal operands) to 5.1e-8 (of one sign) too small on
// average, which adds up over the products of a stack where the float sums' roundings do not (weight gradients of 8 layers: 2.7 times
// the error).  Three of eight blocks of a row, others in the next row, count 2^-23 = 1.19e-7 more.
constexpr float kOneUp = 1.00000011920928955f;

// A matrix [batch][rows][cols] held as three such planes, columns contiguous: part q of element (b, r, c) at
// p[q * plane + b * sb + r * ld + c].  ld is a multiple of 16 (32 bytes) or 64, what lies beyond cols is never read.
struct Planes {
  bf16* p = nullptr;
  int64_t ld = 0, sb = 0, plane = 0;
  Planes at(int64_t b) const {
    Planes r = *this;
    r.p += b * sb;
    return r;
  }
};
// Four neighbouring elements.
__device__ __forceinline__ void store_parts4(bf16* at, int64_t plane, const float4& v) {
  uint32_t h0, m0, l0, h1, m1, l1;
  split_parts2(v.x, v.y, h0, m0, l0);
  split_parts2(v.z, v.w, h1, m1, l1);
  *reinterpret_cast<uint2*>(at) = make_uint2(h0, h1);
  *reinterpret_cast<uint2*>(at + plane) = make_uint2(m0, m1);
  *reinterpret_cast<uint2*>(at + 2 * plane) = make_uint2(l0, l1);
}

namespace tc {
// Tensor map of planes of a matrix with `cols` columns and `rows` rows per batch entry: boxes of box_c x box_r x one entry x all
// parts (gemm_parts.cu).
bool map_planes(CUtensorMap* tm, const Planes& P, int cols, int rows, int batch, int box_c, int box_r, CUtensorMapSwizzle swizzle);
}  // namespace tc

// D(m, n) = sum_k A(m, k) B(n, k) of operands held as planes (gemm_parts.cu).  a_mn / b_mn: the plane's columns are the
// operand's rows (else they are k).  Epilogues as in GemmArgs, float: EPI_STORE, EPI_GELU_FWD (gelu(acc) to Dp, gelu'(acc) to D2),
// EPI_MUL (acc * E to Dp), EPI_RESID (D, with relu the mask to D2).
struct PartsGemm {
  int M = 0, N = 0, K = 0, batch = 1;
  Planes A, B;
  bool a_mn = false, b_mn = false;
  int epi = EPI_STORE;
  float* D = nullptr;
  int64_t ldd = 0, d_sb = 0;
  Planes Dp;
  float* D2 = nullptr;
  int64_t ldd2 = 0, d2_sb = 0;
  const float* E = nullptr;
  int64_t lde = 0, e_sb = 0;
  const float* gate = nullptr;
  bool relu = false;
};
// false: not launched (the device refuses launches in clusters, no tensor map could be made, or D is not 16-byte aligned in
// another epilogue than EPI_STORE); nothing has run then.
bool gemm_parts(Launcher& lc, const PartsGemm& g, int* status_word);
// Whether `batch` products with M x N outputs have tiles for half of the CTA pairs.
bool parts_fill(int M, int N, int batch);
// src [rows][cols] (cols contiguous and a multiple of 4, any alignment) -> dst rows of the first batch entry on
void split_parts(Launcher& lc, const float* src, const Planes& dst, int64_t rows, int cols);

// The left operand of a recurrent kind's all-step products, formed while it is loaded (gemm_cell.cu): g = g_{t+1} of every step
// (LSTM: rows of 2d), coef = the forward pass's coefficients (tanh', C4, C5), both 16-byte aligned; d = units, a multiple of 4.
struct CellOperand {
  const float* g = nullptr;
  const float* coef = nullptr;
  int64_t rows = 0;
  int d = 0;
};
// out (rows ld apart) = operand times W, W's planes [1, 3 or 4 times d][d]; + delta (laid out like out) unless null.  LSTM: out and delta are
// the hidden halves, and uc = fg g_h c_h (+ delta_c), the cell halves, rows of 2d.  false (of either): nothing was launched.
bool cell_vjp(Launcher& lc, int kind, const CellOperand& o, const Planes& W, const float* delta, float* out, int64_t ld, const float* fg,
              const float* delta_c, float* uc, int* status_word);
// dW = operand^T H (rows of H ldh apart, 16-byte aligned), dU = operand^T X (X of any alignment, rows of `in`)
bool cell_wgrad(Launcher& lc, int kind, const CellOperand& o, const float* H, int64_t ldh, const float* X, int in, float* dW, float* dU,
                float* partial, size_t partial_floats, int* status_word);

}  // namespace hbp
