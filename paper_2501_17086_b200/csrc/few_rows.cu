// Float MLP stacks of few rows and narrow layers: the whole forward pass as one launch, and all iterations of a Highway-BP backward
// pass (with the scans between them) as another.  Layer by layer each product is a launch of 4 to 8 us that keeps a few blocks
// busy for one; rows are independent of each other, so here a cluster of 8 CTAs takes 4 rows through all layers or iterations, and only
// its CTAs wait for one another (hardware cluster barriers).
//   forward   the hidden units are split over the cluster: every CTA forms its units' activations from the state (a copy in each),
//             then its part of the block's output for all channels; the parts are added in rank order through distributed shared
//             memory by every CTA alike.  One cluster barrier per layer.
//   backward  the layers are split over the cluster: every CTA forms the vector-Jacobian products of its layers from the iterate it
//             holds for them; then the scan, one thread per element, reads them from all CTAs in descending order of the layers and
//             hands each CTA its next iterate.  Two cluster barriers per iteration.
// Bound by latency: weights come from L2 (16 bytes a lane along a row forward, coalesced columns backward), 4 rows to a load.
// 8 layers 64 (256), 32 rows: see few_rows_take for the times on both sides and where the rule draws the line.
#include "few_rows.cuh"
#include "tc_common.cuh"

namespace hbp {

using namespace tc;

namespace {

constexpr int kCluster = 8, kRows = 4, kThreads = 256, kWarps = kThreads / 32;
constexpr size_t kMostSmem = 160 << 10;

__device__ __forceinline__ float ld_peer(uint32_t own_addr, int rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(map_to_cta(own_addr, (uint32_t)rank)) : "memory");
  return v;
}
__device__ __forceinline__ void st_peer(uint32_t own_addr, int rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_to_cta(own_addr, (uint32_t)rank)), "f"(v) : "memory");
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float c) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ const float* gate_of(const FewRows& a, int l) {
  return a.gate == HBP_GATE_ONE ? nullptr : a.a + (a.gate == HBP_GATE_CHANNEL_PER_STEP ? (int64_t)l * a.d : 0);
}

// Eight lanes form one output of kRows rows: a row of weights against rows of shared memory; lane r of the eight gets row r's.
// x: rows of `pitch` floats; count: a multiple of 4.
__device__ __forceinline__ float eight_lane_dot(const float* __restrict__ w, const float* x, int pitch, int count) {
  const int lane8 = threadIdx.x & 7;
  float acc[kRows] = {};
#pragma unroll 4
  for (int k = lane8 * 4; k < count; k += 32) {
    const float4 wv = __ldg(reinterpret_cast<const float4*>(w + k));
#pragma unroll
    for (int r = 0; r < kRows; ++r) acc[r] = dot4(wv, *reinterpret_cast<const float4*>(x + r * pitch + k), acc[r]);
  }
  float mine = 0.0f;
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
    if (lane8 == r) mine = acc[r];
  }
  return mine;
}

__global__ void __launch_bounds__(kThreads) few_rows_forward_kernel(const FewRows a) {
  extern __shared__ __align__(16) float smem[];
  const int rank = (int)cluster_ctarank(), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lane8 = lane & 7;
  const int d = a.d, h = a.h, hs = (h + 4 * kCluster - 1) / (4 * kCluster) * 4;  // hidden units of a CTA, a multiple of 4
  const int h0 = min(h, rank * hs), mine = min(h, h0 + hs) - h0;
  const int64_t row0 = (int64_t)(blockIdx.x / kCluster) * kRows, state = a.N * d;
  float* xs = smem;                       // [kRows][d] the state
  float* xn = xs + kRows * d;             // [kRows][d] normalised (pre-LN)
  float* act = xn + kRows * d;            // [kRows][hs]
  float* part = act + kRows * hs;         // [2][kRows][d] this CTA's part of the block's output
  chain_next();
  chain_wait();
  for (int e = tid; e < kRows * d; e += kThreads) {
    const int64_t row = row0 + e / d;
    const float v = row < a.N ? a.x0[row0 * d + e] : 0.0f;
    xs[e] = v;
    if (rank == 0 && row < a.N) a.x_all[row0 * d + e] = v;
  }
  __syncthreads();
  for (int l = 0; l < a.L; ++l) {
    const float* op = xs;
    if (a.preln) {
      op = xn;
      if (warp < kRows) {
        const float* x = xs + warp * d;
        float s1 = 0.0f, s2 = 0.0f;
        for (int c = lane; c < d; c += 32) s1 += x[c];
        const float mu = warp_sum(s1) / (float)d;
        for (int c = lane; c < d; c += 32) s2 = fmaf(x[c] - mu, x[c] - mu, s2);
        const float r = rsqrtf(warp_sum(s2) / (float)d + a.eps);
        const int64_t row = row0 + warp;
        const bool store = rank == 0 && row < a.N;
        if (store && lane == 0) a.rstd[l * a.N + row] = r;
        for (int c = lane; c < d; c += 32) {
          const float v = (x[c] - mu) * r;
          xn[warp * d + c] = v;
          if (store) a.Y[l * state + row * d + c] = v;
        }
      }
      __syncthreads();
    }
    const float* W1 = a.W1 + (int64_t)l * h * d;
    for (int u0 = warp * 4; u0 < mine; u0 += 4 * kWarps) {  // (warps go round together: the lanes exchange their sums)
      const int u = u0 + (lane >> 3);
      const float z = eight_lane_dot(W1 + (int64_t)(h0 + min(u, mine - 1)) * d, op, d, d);
      if (u < mine && lane8 < kRows) {
        const float v = gelu_f(z);
        act[lane8 * hs + u] = v;
        const int64_t row = row0 + lane8;
        if (row < a.N) {
          const int64_t at = ((int64_t)l * a.N + row) * h + h0 + u;
          a.ACT[at] = v;
          a.DACT[at] = gelu_prime_f(z);
        }
      }
    }
    __syncthreads();
    const float* W2 = a.W2 + (int64_t)l * d * h + h0;
    float* out = part + (l & 1) * kRows * d;
    for (int c0 = warp * 4; c0 < d; c0 += 4 * kWarps) {  // (d is a multiple of 4)
      const int c = c0 + (lane >> 3);
      const float y = eight_lane_dot(W2 + (int64_t)c * h, act, hs, mine);
      if (lane8 < kRows) out[lane8 * d + c] = y;
    }
    cluster_sync();  // (the parts of the layer before the last have been read by all)
    const float* gate = gate_of(a, l);
    const uint32_t at = smem_u32(out);
    for (int e = tid; e < kRows * d; e += kThreads) {
      float p[kCluster];
#pragma unroll
      for (int j = 0; j < kCluster; ++j) p[j] = ld_peer(at + 4u * e, j);
      float y = p[0];
#pragma unroll
      for (int j = 1; j < kCluster; ++j) y += p[j];
      const float v = (gate ? gate[e % d] : 1.0f) * xs[e] + y;
      xs[e] = v;
      if (rank == 0 && row0 + e / d < a.N) a.x_all[(l + 1) * state + row0 * d + e] = v;
    }
    __syncthreads();
  }
  cluster_sync();  // no CTA leaves while another may read its part
}

// k iterations from g^0, all states of the last estimate to g_all; with dZ also gelu'(Z) times what the block is differentiated against in
// the last estimate, the parameter gradients' operand.
__global__ void __launch_bounds__(kThreads) few_rows_backward_kernel(const FewRows a) {
  extern __shared__ __align__(16) float smem[];
  const int rank = (int)cluster_ctarank(), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = a.d, h = a.h, L = a.L, slots = (L + kCluster - 1) / kCluster, rd = kRows * d;
  const int64_t row0 = (int64_t)(blockIdx.x / kCluster) * kRows, state = a.N * d;
  float* G = smem;               // [slots][kRows][d]: g_{l+1} of this CTA's layers l = slot * kCluster + rank
  float* U = G + slots * rd;     // [slots][kRows][d]: their vector-Jacobian products
  float* dz = U + slots * rd;    // [kRows][h]
  float* red = dz + kRows * h;   // [groups][kRows][cols]
  const uint32_t G_at = smem_u32(G), U_at = smem_u32(U);
  chain_next();
  chain_wait();
  // One thread per element of the cluster's rows walks the layers down: g_l = delta_l + a_l g_{l+1} (+ u_l).
  auto scan = [&](bool with_u, bool last) {
    for (int e = rank * kThreads + tid; e < rd; e += kCluster * kThreads) {
      const int c = e % d;
      const int64_t row = row0 + e / d, at = row * d + c;
      const bool in = row < a.N;
      float g = in ? a.delta[(a.every ? L * state : 0) + at] : 0.0f;
      if (last && in) a.g_all[L * state + at] = g;
      st_peer(G_at + 4u * ((L - 1) / kCluster * rd + e), (L - 1) % kCluster, g);
      for (int top = L - 1; top >= 0; top -= 8) {
        float u[8], dl[8], gt[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int l = top - j;
          u[j] = dl[j] = 0.0f;
          gt[j] = 1.0f;
          if (l < 0) continue;
          if (with_u) u[j] = ld_peer(U_at + 4u * (l / kCluster * rd + e), l % kCluster);
          if (a.every && in) dl[j] = a.delta[l * state + at];
          const float* gate = gate_of(a, l);
          if (gate) gt[j] = gate[c];
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int l = top - j;
          if (l < 0) continue;
          g = gt[j] * g;
          g += u[j];
          g += dl[j];
          if (last && in) a.g_all[l * state + at] = g;
          if (l > 0) st_peer(G_at + 4u * ((l - 1) / kCluster * rd + e), (l - 1) % kCluster, g);
        }
      }
    }
    cluster_sync();
  };
  const int cols = min(d, kThreads), groups = kThreads / cols, group = tid / cols, col = tid % cols;
  auto vjp = [&](bool to_memory) {
    for (int s = 0; s < slots; ++s) {
      const int l = s * kCluster + rank;
      if (l >= L) break;
      const float* g = G + s * rd;
      const float* W2 = a.W2 + (int64_t)l * d * h;
      for (int i = tid; i < h; i += kThreads) {
        float acc[kRows] = {};
#pragma unroll 4
        for (int k = 0; k < d; k += 4) {
          float4 w;
          w.x = __ldg(W2 + (int64_t)k * h + i);
          w.y = __ldg(W2 + (int64_t)(k + 1) * h + i);
          w.z = __ldg(W2 + (int64_t)(k + 2) * h + i);
          w.w = __ldg(W2 + (int64_t)(k + 3) * h + i);
#pragma unroll
          for (int r = 0; r < kRows; ++r) acc[r] = dot4(w, *reinterpret_cast<const float4*>(g + r * d + k), acc[r]);
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          const int64_t at = ((int64_t)l * a.N + row0 + r) * h + i;
          const float v = row0 + r < a.N ? acc[r] * a.DACT[at] : 0.0f;
          dz[r * h + i] = v;
          if (to_memory && row0 + r < a.N) a.dZ[at] = v;
        }
      }
      __syncthreads();
      if (to_memory) continue;  // (the next layer's dz may be written: nobody reads this one's)
      const float* W1 = a.W1 + (int64_t)l * h * d;
      float* u = U + s * rd;
      for (int c0 = 0; c0 < d; c0 += cols) {
        const int c = c0 + col;
        if (group < groups && c < d) {
          float acc[kRows] = {};
#pragma unroll 4
          for (int i = 4 * group; i < h; i += 4 * groups) {
            float4 w;
            w.x = __ldg(W1 + (int64_t)i * d + c);
            w.y = __ldg(W1 + (int64_t)(i + 1) * d + c);
            w.z = __ldg(W1 + (int64_t)(i + 2) * d + c);
            w.w = __ldg(W1 + (int64_t)(i + 3) * d + c);
#pragma unroll
            for (int r = 0; r < kRows; ++r) acc[r] = dot4(w, *reinterpret_cast<const float4*>(dz + r * h + i), acc[r]);
          }
#pragma unroll
          for (int r = 0; r < kRows; ++r) red[(group * kRows + r) * cols + col] = acc[r];
        }
        __syncthreads();
        for (int e = tid; e < kRows * cols; e += kThreads) {
          const int r = e / cols, cc = e % cols;
          if (c0 + cc >= d) continue;
          float y = red[e];
          for (int q = 1; q < groups; ++q) y += red[q * kRows * cols + e];
          u[r * d + c0 + cc] = y;
        }
        __syncthreads();
      }
      if (a.preln && warp < kRows) {  // through the LayerNorm: rstd (dy - mean dy - xhat mean(dy xhat))
        const int64_t row = row0 + warp;
        const bool in = row < a.N;
        const float* xh = a.Y + l * state + row * d;
        float* y = u + warp * d;
        float s1 = 0.0f, s2 = 0.0f;
        for (int c = lane; c < d; c += 32) {
          s1 += y[c];
          s2 = fmaf(y[c], in ? xh[c] : 0.0f, s2);
        }
        const float m1 = warp_sum(s1) / (float)d, m2 = warp_sum(s2) / (float)d, r = in ? a.rstd[l * a.N + row] : 0.0f;
        for (int c = lane; c < d; c += 32) y[c] = r * (y[c] - m1 - (in ? xh[c] : 0.0f) * m2);
      }
    }
  };
  cluster_sync();  // every CTA's shared memory may be written from here on
  scan(false, a.k == 0);
  for (int it = 0; it < a.k; ++it) {
    vjp(false);
    cluster_sync();
    scan(true, it + 1 == a.k);
  }
  if (a.dZ) vjp(true);
}

size_t forward_smem(const FewRows& a) {
  const int hs = (a.h + 4 * kCluster - 1) / (4 * kCluster) * 4;
  return (size_t)4 * kRows * (4 * a.d + hs);
}
size_t backward_smem(const FewRows& a) {
  const int slots = (a.L + kCluster - 1) / kCluster, cols = a.d < kThreads ? a.d : kThreads;
  return (size_t)4 * kRows * (2 * slots * a.d + a.h + kThreads / cols * cols);
}

bool launch(Launcher& lc, void (*kernel)(const FewRows), size_t smem, const FewRows& a) {
  if (smem > kMostSmem) return false;
  if (smem > (48 << 10) && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const unsigned clusters = (unsigned)((a.N + kRows - 1) / kRows);
  if (try_launch_chained(lc, kernel, dim3(clusters * kCluster), kThreads, smem, kCluster, a) != cudaSuccess) return false;
  lc.ran(HBP_FORM_FEW_ROWS);
  return true;
}
bool aligned(const void* p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

bool few_rows_take(int64_t N, int d, int h) { return N <= 32 && (int64_t)d * h <= 64 * 1024; }

bool few_rows_forward(Launcher& lc, const FewRows& a) {
  if (!aligned(a.W1) || !aligned(a.W2)) return false;
  return launch(lc, few_rows_forward_kernel, forward_smem(a), a);
}
bool few_rows_backward(Launcher& lc, const FewRows& a) { return launch(lc, few_rows_backward_kernel, backward_smem(a), a); }

}  // namespace hbp
