// CUDA-core (FFMA) GEMM with arbitrary operand strides, fp32 accumulation and fused epilogues.
// Serves the float products that the split-operand tensor-core kernel declines (few rows, short contractions, unaligned
// operands) and every bf16 problem whose shape the tcgen05 kernel does not take.
#include "hbp_internal.h"

namespace hbp {

namespace {

template <typename T>
__device__ __forceinline__ float load_a(const T* A, const T* A2, int64_t off) {
  float v = to_f(A[off]);
  if (A2) v *= to_f(A2[off]);
  return v;
}

template <typename T>
__device__ __forceinline__ void epilogue_store(const GemmArgs& g, int b, int m, int n, float acc) {
  const int64_t dn = (int64_t)m * g.ldd + n;
  switch (g.epi) {
    case EPI_STORE_LN:
    case EPI_STORE: {
      if (g.d_f32) ((float*)g.D)[b * g.d_sb + dn] = acc;
      else ((T*)g.D)[b * g.d_sb + dn] = from_f<T>(acc);
    } break;
    case EPI_GELU_FWD: {
      ((T*)g.D)[b * g.d_sb + dn] = from_f<T>(gelu_f(acc));
      ((T*)g.D2)[b * g.d2_sb + (int64_t)m * g.ldd2 + n] = from_f<T>(gelu_prime_f(acc));
    } break;
    case EPI_RESID: {
      float gate = g.gate ? to_f(((const T*)g.gate)[b * g.gate_sb + n]) : 1.0f;
      float r = g.R ? g.R[(int64_t)m * g.N + n] : to_f(((const T*)g.E)[b * g.e_sb + (int64_t)m * g.lde + n]);
      float v = gate * r + acc;
      if (g.relu) {
        ((T*)g.D2)[b * g.d2_sb + (int64_t)m * g.ldd2 + n] = from_f<T>(v > 0.0f ? 1.0f : 0.0f);
        v = fmaxf(v, 0.0f);
      }
      if (g.R) g.R[(int64_t)m * g.N + n] = v;
      ((T*)g.D)[b * g.d_sb + dn] = from_f<T>(v);
    } break;
    case EPI_ADD: {
      float e = to_f(((const T*)g.E)[b * g.e_sb + (int64_t)m * g.lde + n]);
      if (g.d_f32) ((float*)g.D)[b * g.d_sb + dn] = acc + e;
      else ((T*)g.D)[b * g.d_sb + dn] = from_f<T>(acc + e);
    } break;
    case EPI_MUL: {
      float e = to_f(((const T*)g.E)[b * g.e_sb + (int64_t)m * g.lde + n]);
      ((T*)g.D)[b * g.d_sb + dn] = from_f<T>(acc * e);
    } break;
    case EPI_AFFINE: {
      float gate = g.gate ? to_f(((const T*)g.gate)[b * g.gate_sb + n]) : 1.0f;
      float e = g.E ? to_f(((const T*)g.E)[b * g.e_sb + (int64_t)m * g.lde + n]) : 0.0f;
      float e2 = to_f(((const T*)g.E2)[b * g.e2_sb + (int64_t)m * g.lde2 + n]);
      ((T*)g.D)[b * g.d_sb + dn] = from_f<T>(e + gate * e2 + acc);
    } break;
    case EPI_RNN_FWD: {
      float gate = g.gate ? to_f(((const T*)g.gate)[b * g.gate_sb + n]) : 1.0f;
      float z = acc + to_f(((const T*)g.E)[b * g.e_sb + (int64_t)m * g.lde + n]);
      // tanh and its derivative 1 - tanh^2 = 4e / (1 + e)^2 with e = exp(-2|z|): no cancellation near |c| = 1
      float e = expf(-2.0f * fabsf(z));
      float c = copysignf((1.0f - e) / (1.0f + e), z);
      float h = to_f(((const T*)g.E2)[b * g.e2_sb + (int64_t)m * g.lde2 + n]);
      ((T*)g.D2)[b * g.d2_sb + (int64_t)m * g.ldd2 + n] = from_f<T>(4.0f * e / ((1.0f + e) * (1.0f + e)));
      ((T*)g.D)[b * g.d_sb + dn] = from_f<T>(gate * h + c);
    } break;
  }
}

// 256 threads, BM x BN output tile, BK = 16, (BM/16) x (BN/16) register micro-tile.  The next block of K is loaded into
// registers while the current one is multiplied (1900 x 1560 x 520, 12 at once: 1980 -> 1660 us).
template <typename T, int BM, int BN>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const GemmArgs g) {
  constexpr int BK = 16, TM = BM / 16, TN = BN / 16, NA = BM * BK / 256, NB = BN * BK / 256;
  __shared__ float As[BK][BM + 4];
  __shared__ float Bs[BK][BN + 4];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int b = blockIdx.z / g.splitk, split = blockIdx.z % g.splitk;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const T* A = (const T*)g.A + (int64_t)b * g.a_sb;
  const T* A2 = g.A2 ? (const T*)g.A2 + (int64_t)b * g.a_sb : nullptr;
  const T* B = (const T*)g.B + (int64_t)b * g.b_sb;
  // K range of this split (multiples of 16 except the last)
  const int ktiles = (g.K + 15) / 16;
  const int per = (ktiles + g.splitk - 1) / g.splitk;
  const int kbeg = split * per * 16;
  const int kend = min(g.K, (split + 1) * per * 16);

  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;

  const bool a_kmajor = (g.a_sk == 1), b_kmajor = (g.b_sk == 1);
  float av[NA], bv[NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int idx = tid + i * 256, kk = a_kmajor ? idx % BK : idx / BM, mm = a_kmajor ? idx / BK : idx % BM;
      const int m = m0 + mm, k = k0 + kk;
      av[i] = (m < g.M && k < kend) ? load_a<T>(A, A2, (int64_t)m * g.a_sm + (int64_t)k * g.a_sk) : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int idx = tid + i * 256, kk = b_kmajor ? idx % BK : idx / BN, nn = b_kmajor ? idx / BK : idx % BN;
      const int n = n0 + nn, k = k0 + kk;
      bv[i] = (n < g.N && k < kend) ? to_f(B[(int64_t)n * g.b_sn + (int64_t)k * g.b_sk]) : 0.0f;
    }
  };
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int idx = tid + i * 256;
      As[a_kmajor ? idx % BK : idx / BM][a_kmajor ? idx / BK : idx % BM] = av[i];
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int idx = tid + i * 256;
      Bs[b_kmajor ? idx % BK : idx / BN][b_kmajor ? idx / BK : idx % BN] = bv[i];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[TM], bb[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < TM; ++i) {
    int m = m0 + ty + 16 * i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      int n = n0 + tx + 16 * j;
      if (n >= g.N) continue;
      if (g.splitk > 1) {
        g.partial[(((int64_t)split * g.batch + b) * g.M + m) * g.N + n] = acc[i][j];
      } else {
        epilogue_store<T>(g, b, m, n, acc[i][j]);
      }
    }
  }
}

// At most 32 rows and a long contraction: 32 x 32 tiles, a few blocks on an idle GPU, so what counts is the time of one block.  64 of K per block
// (one exposed memory latency, the next block's loads in flight meanwhile); four groups of 64 threads take 16 of them each
// with a 4 x 4 micro-tile, because with one group of 256 threads and 2 x 2 the shared-memory loads bound it, and the groups'
// sums are added in a fixed order.  32 x 64 x 256: 16.5 -> 8.5 us, 32 x 512 x
// 1024: 51 -> 23.
template <typename T>
__global__ void __launch_bounds__(256) gemm_small_kernel(const GemmArgs g) {
  constexpr int BM = 32, BN = 32, BK = 64, P = 36, N4 = BM * BK / 256;
  __shared__ __align__(16) float As[BK][P];
  __shared__ __align__(16) float Bs[BK][P];
  __shared__ float red[4][BM][BN + 1];
  const int tid = threadIdx.x, grp = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
  const int b = blockIdx.z / g.splitk, split = blockIdx.z % g.splitk;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const T* A = (const T*)g.A + (int64_t)b * g.a_sb;
  const T* A2 = g.A2 ? (const T*)g.A2 + (int64_t)b * g.a_sb : nullptr;
  const T* B = (const T*)g.B + (int64_t)b * g.b_sb;
  const int ktiles = (g.K + 15) / 16, per = (ktiles + g.splitk - 1) / g.splitk;
  const int kbeg = split * per * 16, kend = min(g.K, (split + 1) * per * 16);
  const bool a_kmajor = g.a_sk == 1, b_kmajor = g.b_sk == 1;
  float acc[4][4] = {}, av[N4], bv[N4];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < N4; ++i) {
      const int idx = tid + i * 256;
      const int ka = k0 + (a_kmajor ? idx % BK : idx / BM), m = m0 + (a_kmajor ? idx / BK : idx % BM);
      const int kb = k0 + (b_kmajor ? idx % BK : idx / BN), n = n0 + (b_kmajor ? idx / BK : idx % BN);
      av[i] = (m < g.M && ka < kend) ? load_a<T>(A, A2, (int64_t)m * g.a_sm + (int64_t)ka * g.a_sk) : 0.0f;
      bv[i] = (n < g.N && kb < kend) ? to_f(B[(int64_t)n * g.b_sn + (int64_t)kb * g.b_sk]) : 0.0f;
    }
  };
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int i = 0; i < N4; ++i) {
      const int idx = tid + i * 256;
      As[a_kmajor ? idx % BK : idx / BM][a_kmajor ? idx / BK : idx % BM] = av[i];
      Bs[b_kmajor ? idx % BK : idx / BN][b_kmajor ? idx / BK : idx % BN] = bv[i];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK / 4; ++kk) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[grp * (BK / 4) + kk][ty * 4]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[grp * (BK / 4) + kk][tx * 4]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) red[grp][ty * 4 + i][tx * 4 + j] = acc[i][j];
  __syncthreads();
  const int nn = tid & 31, n = n0 + nn;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int mm = (tid >> 5) + 8 * i, m = m0 + mm;
    if (m >= g.M || n >= g.N) continue;
    const float v = (red[0][mm][nn] + red[1][mm][nn]) + (red[2][mm][nn] + red[3][mm][nn]);
    if (g.splitk > 1) g.partial[(((int64_t)split * g.batch + b) * g.M + m) * g.N + n] = v;
    else epilogue_store<T>(g, b, m, n, v);
  }
}

__global__ void reduce_splitk_kernel(const float* __restrict__ partial, float* __restrict__ out, int splits,
                                     int64_t elems) {
  chain_next();
  chain_wait();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= elems) return;
  double s = 0.0;
#pragma unroll 8
  for (int k = 0; k < splits; ++k) s += (double)partial[(int64_t)k * elems + i];  // fixed order: deterministic
  out[i] = (float)s;
}
// The same for many splits of few elements, whose loads a thread would wait for one batch after the other: eight warps take an eighth
// of the splits each (reduce_eighths), 32 elements a block.  512 elements, 256 splits: 21 us a thread each.
__global__ void __launch_bounds__(256) reduce_eighths_kernel(const float* __restrict__ partial, float* __restrict__ out, int splits, int64_t elems) {
  chain_next();
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  const double s = reduce_eighths(partial + i, i < elems, splits, elems);
  if (threadIdx.x < 32 && i < elems) out[i] = (float)s;
}

template <typename T>
void launch_simt(Launcher& lc, const GemmArgs& g) {
  const int64_t ctas128 = (int64_t)((g.M + 127) / 128) * ((g.N + 127) / 128) * g.batch * g.splitk;
  if (ctas128 >= 148 && g.M >= 128 && g.N >= 128) {
    dim3 grid((g.N + 127) / 128, (g.M + 127) / 128, g.batch * g.splitk);
    gemm_simt_kernel<T, 128, 128><<<grid, 256, 0, lc.stream>>>(g);
  } else if (g.M > 32) {
    dim3 grid((g.N + 63) / 64, (g.M + 63) / 64, g.batch * g.splitk);
    gemm_simt_kernel<T, 64, 64><<<grid, 256, 0, lc.stream>>>(g);
  } else {
    // At most 32 rows.  Few tiles, or a long contraction, are the small kernel's; but a block of it takes 64 of K at a time and 1
    // to 2 us however short the contraction, which counts where an SM gets several: 32 x 1024 x 64, 16 at once (512 tiles), 14.7
    // us against 10.7 for the plain kernel; 32 x 2048 x 32, 64 at once, 82 against 31.  Up to 128 tiles the two are the same at 64
    // of K (7.9 us with the launch); from 192 of K on the small one is never slower (a few tiles 8 against 10.5).
    dim3 grid((g.N + 31) / 32, (g.M + 31) / 32, g.batch * g.splitk);
    if (g.K <= 128 * g.splitk && (int64_t)grid.x * grid.y * grid.z > 148) gemm_simt_kernel<T, 32, 32><<<grid, 256, 0, lc.stream>>>(g);
    else gemm_small_kernel<T><<<grid, 256, 0, lc.stream>>>(g);
  }
  lc.ran(HBP_FORM_GEMM_SIMT);
  lc.count();
  lc.check();
}

}  // namespace

void reduce_splitk(Launcher& lc, const float* partial, float* out, int splits, int64_t elems) {
  if (splits >= kManySplits) launch_chained(lc, reduce_eighths_kernel, dim3((unsigned)((elems + 31) / 32)), 256, 0, 1, partial, out, splits, elems);
  else launch_chained(lc, reduce_splitk_kernel, dim3((unsigned)((elems + 255) / 256)), 256, 0, 1, partial, out, splits, elems);
}

void gemm_simt(Launcher& lc, const GemmArgs& g) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return;
  if (g.in_dtype == HBP_F32) launch_simt<float>(lc, g);
  else launch_simt<bf16>(lc, g);
  // split-K supports a plain contiguous float store only
  if (g.splitk > 1) reduce_splitk(lc, g.partial, (float*)g.D, g.splitk, (int64_t)g.batch * g.M * g.N);
}

}  // namespace hbp
