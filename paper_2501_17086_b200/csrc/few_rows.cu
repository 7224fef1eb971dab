// Float MLP stacks of few rows and narrow layers: the whole forward pass as one launch, and all iterations of a Highway-BP backward
// pass (with the scans between them) as another.  Layer by layer each product is a launch of 4 to 8 us that keeps a few blocks
// busy for one; rows are independent of each other, so here a cluster of 8 CTAs takes 3 rows through all layers or iterations, and only
// its CTAs wait for one another (hardware cluster barriers, one per layer or iteration).
//   forward   the hidden units are split over the cluster: every CTA forms its units' activations from the state (a copy in each),
//             then its part of the block's output for all channels, which it writes to all CTAs; each adds the parts in rank order.
//   backward  the layers are split over the cluster: every CTA forms the vector-Jacobian products of its layers from the iterate it
//             holds for them and writes them to all CTAs; each then scans all layers for itself and keeps the iterates it needs.
//   exact     the same split with one layer at a time: its CTA forms the product, all add it to the running gradient.
// Weights lie in shared memory: forward two layers' at a time (the next layer's are copied while one is worked on), backward those of the
// CTA's layers for all iterations where they fit.  Bound by latency and shared-memory bandwidth (a 16-byte broadcast takes four clocks:
// a thread forms four neighbouring outputs of all rows).  Results that go to memory are stored after the barrier, not before: a
// cluster-scope release waits for all stores before it, 1000 clocks.
// 8 layers 64 (256), 32 rows, training step: see few_rows_take for the times on both sides and where the rule draws the line.
#include "few_rows.cuh"
#include "tc_common.cuh"

namespace hbp {

using namespace tc;

namespace {

// 15 clusters of 8 CTAs run at a time where a CTA fills an SM: three rows to a cluster take 32 rows at once (two, in 16 clusters, twice
// the time: backward 38 us instead of 21, forward 38 instead of 20).
constexpr int kCluster = 8, kRows = 3, kThreads = 256, kWarps = kThreads / 32;
constexpr size_t kMostSmem = 224 << 10;

__device__ __forceinline__ void st_peer(uint32_t own_addr, int rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_to_cta(own_addr, (uint32_t)rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float c) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}
__device__ __forceinline__ const float4& vec4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void copy16_async(float* to, const float* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(to)), "l"(from) : "memory");
}
__device__ __forceinline__ void copy_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ const float* gate_of(const FewRows& a, int l) {
  return a.gate == HBP_GATE_ONE ? nullptr : a.a + (a.gate == HBP_GATE_CHANNEL_PER_STEP ? (int64_t)l * a.d : 0);
}

// Eight lanes form one output of kRows rows: a row of weights against rows of shared memory (`pitch` floats apart, count a multiple of
// 4); all eight get the sums.
__device__ __forceinline__ void eight_lane_dot(const float* w, const float* x, int pitch, int count, float (&acc)[kRows]) {
  const int lane8 = threadIdx.x & 7;
#pragma unroll
  for (int r = 0; r < kRows; ++r) acc[r] = 0.0f;
#pragma unroll 4
  for (int k = lane8 * 4; k < count; k += 32) {
    const float4 wv = vec4(w + k);
#pragma unroll
    for (int r = 0; r < kRows; ++r) acc[r] = dot4(wv, vec4(x + r * pitch + k), acc[r]);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1)
#pragma unroll
    for (int r = 0; r < kRows; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
}

__device__ __host__ inline int units_per_cta(int h) { return (h + 4 * kCluster - 1) / (4 * kCluster) * 4; }

__global__ void __launch_bounds__(kThreads, 1) few_rows_forward_kernel(const FewRows a) {
  extern __shared__ __align__(16) float smem[];
  const int rank = (int)cluster_ctarank(), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lane8 = lane & 7;
  const int d = a.d, h = a.h, hs = units_per_cta(h), rd = kRows * d;
  const int h0 = min(h, rank * hs), mine = min(h, h0 + hs) - h0;  // this CTA's hidden units
  const int64_t row0 = (int64_t)(blockIdx.x / kCluster) * kRows, state = a.N * d;
  const int rows = (int)min((int64_t)kRows, a.N - row0);
  float* xs = smem;                           // [kRows][d] the state
  float* xn = xs + rd;                        // [kRows][d] normalised (pre-LN)
  float* act = xn + rd;                       // [kRows][hs] gelu(z)
  float* prime = act + kRows * hs;            // [kRows][hs] gelu'(z)
  float* parts = prime + kRows * hs;          // [2][kCluster][kRows][d] the CTAs' parts of the block's output
  float* weights = parts + 2 * kCluster * rd;  // [2] rows of W1 [hs][d] and columns of W2 [d][hs]
  chain_next();
  chain_wait();
  // a layer's weights, while the layer before is worked on
  const int quads = max(mine / 4, 1), c_first = tid / quads, q_first = tid % quads, c_step = kThreads / quads, q_step = kThreads % quads;
  auto fetch = [&](int l) {
    if (l < a.L && mine > 0) {
      float* to = weights + (l & 1) * 2 * hs * d;
      const float* W1 = a.W1 + ((int64_t)l * h + h0) * d;
      for (int e = tid * 4; e < mine * d; e += 4 * kThreads) copy16_async(to + e, W1 + e);
      const float* W2 = a.W2 + (int64_t)l * d * h + h0;
      for (int c = c_first, q = q_first; c < d;) {
        copy16_async(to + hs * d + c * hs + 4 * q, W2 + (int64_t)c * h + 4 * q);
        c += c_step;
        q += q_step;
        if (q >= quads) {
          q -= quads;
          ++c;
        }
      }
    }
    copy_group();
  };
  fetch(0);
  for (int e = tid; e < rd; e += kThreads) {
    const float v = e < rows * d ? a.x0[row0 * d + e] : 0.0f;
    xs[e] = v;
    if (rank == 0 && e < rows * d) a.x_all[row0 * d + e] = v;
  }
  cluster_sync();  // every CTA's shared memory may be written from here on
  for (int l = 0; l < a.L; ++l) {
    fetch(l + 1);  // (into the place of layer l - 1's)
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
        const bool store = rank == 0 && warp < rows;
        if (store && lane == 0) a.rstd[l * a.N + row0 + warp] = r;
        for (int c = lane; c < d; c += 32) {
          const float v = (x[c] - mu) * r;
          xn[warp * d + c] = v;
          if (store) a.Y[l * state + (row0 + warp) * d + c] = v;
        }
      }
    }
    copy_wait<1>();
    __syncthreads();
    const float* W1 = weights + (l & 1) * 2 * hs * d;
    for (int u0 = warp * 4; u0 < mine; u0 += 4 * kWarps) {  // (warps go round together: the lanes exchange their sums)
      const int u = u0 + (lane >> 3);
      float z[kRows];
      eight_lane_dot(W1 + min(u, mine - 1) * d, op, d, d, z);
      float zr = z[0];
#pragma unroll
      for (int r = 1; r < kRows; ++r)
        if (lane8 == r) zr = z[r];
      if (u < mine && lane8 < kRows) {
        act[lane8 * hs + u] = gelu_f(zr);
        prime[lane8 * hs + u] = gelu_prime_f(zr);
      }
    }
    __syncthreads();
    const float* W2 = W1 + hs * d;
    float* part = parts + (l & 1) * kCluster * rd;
    const uint32_t to = smem_u32(part + rank * rd);
    for (int c0 = warp * 4; c0 < d; c0 += 4 * kWarps) {  // (d is a multiple of 4)
      const int c = c0 + (lane >> 3);
      float y[kRows];
      eight_lane_dot(W2 + c * hs, act, hs, mine, y);
#pragma unroll
      for (int r = 0; r < kRows; ++r) st_peer(to + 4u * (r * d + c), lane8, y[r]);  // lane j of the eight to CTA j
    }
    cluster_arrive();
    for (int r = 0; r < rows; ++r) {
      const int64_t at = ((int64_t)l * a.N + row0 + r) * h + h0;
      for (int u = tid; u < mine; u += kThreads) {
        a.ACT[at + u] = act[r * hs + u];
        a.DACT[at + u] = prime[r * hs + u];
      }
    }
    cluster_wait();
    const float* gate = gate_of(a, l);
    for (int e = tid; e < rd; e += kThreads) {
      float p[kCluster];
#pragma unroll
      for (int j = 0; j < kCluster; ++j) p[j] = part[j * rd + e];
      float y = p[0];
#pragma unroll
      for (int j = 1; j < kCluster; ++j) y += p[j];
      const float v = (gate ? gate[e % d] : 1.0f) * xs[e] + y;
      xs[e] = v;
      if (rank == 0 && e < rows * d) a.x_all[(l + 1) * state + row0 * d + e] = v;
    }
    __syncthreads();
  }
}

// Four neighbouring columns of kRows products of rows x (of shared memory, `pitch` apart) with a matrix w [count][width], over the rows of w
// in blocks of four from `first` on, `step` apart.
__device__ __forceinline__ void four_columns(const float* w, int width, const float* x, int pitch, int count, int first, int step, float4 (&acc)[kRows]) {
#pragma unroll
  for (int r = 0; r < kRows; ++r) acc[r] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
  for (int k = first; k < count; k += step) {
    const float4 w0 = vec4(w + (int64_t)k * width), w1 = vec4(w + (int64_t)(k + 1) * width), w2 = vec4(w + (int64_t)(k + 2) * width),
                 w3 = vec4(w + (int64_t)(k + 3) * width);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const float4 v = vec4(x + r * pitch + k);
      acc[r].x = fmaf(w3.x, v.w, fmaf(w2.x, v.z, fmaf(w1.x, v.y, fmaf(w0.x, v.x, acc[r].x))));
      acc[r].y = fmaf(w3.y, v.w, fmaf(w2.y, v.z, fmaf(w1.y, v.y, fmaf(w0.y, v.x, acc[r].y))));
      acc[r].z = fmaf(w3.z, v.w, fmaf(w2.z, v.z, fmaf(w1.z, v.y, fmaf(w0.z, v.x, acc[r].z))));
      acc[r].w = fmaf(w3.w, v.w, fmaf(w2.w, v.z, fmaf(w1.w, v.y, fmaf(w0.w, v.x, acc[r].w))));
    }
  }
}
// How the threads share a product `width` wide: `quads` of them a pass, each for four columns, `groups` of those splitting the sum.
struct Share {
  int quads, groups;
};
__device__ __host__ inline Share share_of(int width) {
  const int quads = width / 4 < kThreads ? width / 4 : kThreads;
  return {quads, kThreads / quads};
}
__device__ __host__ inline int share_floats(int width) { return share_of(width).groups * kRows * 4 * share_of(width).quads; }

// k iterations from g^0 (or exact backpropagation), all states of the last estimate to g_all; with dZ also gelu'(Z) times what the block is differentiated against in
// the last estimate, the parameter gradients' operand.
__global__ void __launch_bounds__(kThreads, 1) few_rows_backward_kernel(const FewRows a) {
  extern __shared__ __align__(16) float smem[];
  const int rank = (int)cluster_ctarank(), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = a.d, h = a.h, L = a.L, slots = (L + kCluster - 1) / kCluster, rd = kRows * d;
  const int64_t row0 = (int64_t)(blockIdx.x / kCluster) * kRows, state = a.N * d;
  const int rows = (int)min((int64_t)kRows, a.N - row0);
  float* G = smem;                     // [slots][kRows][d]: g_{l+1} of this CTA's layers l = slot * kCluster + rank
  float* U = G + (a.exact ? 0 : slots * rd);  // [2][L][kRows][d]: all layers' vector-Jacobian products, of alternating iterations
  float* dz = U + 2 * (a.exact ? 1 : L) * rd; // [kRows][h]  (exact: no G, and two layers' products in turn)
  float* y = dz + kRows * h;           // [kRows][d]: a layer's product before its LayerNorm
  float* last_delta = y + rd;          // [kRows][d]: delta of the last state
  float* red = last_delta + rd;        // [groups][kRows][columns of a pass]
  // where they fit, kept for all iterations: W2 [d][h], W1 [h][d], gelu' [kRows][h] of every slot
  float* kept = red + max(share_floats(d), share_floats(h));
  const int per_slot = 2 * d * h + kRows * h;
  chain_next();
  chain_wait();
  if (a.resident) {
    for (int s = 0; s < slots; ++s) {
      const int l = s * kCluster + rank;
      if (l >= L) break;
      float* to = kept + s * per_slot;
      for (int e = tid * 4; e < d * h; e += 4 * kThreads) {
        copy16_async(to + e, a.W2 + (int64_t)l * d * h + e);
        copy16_async(to + d * h + e, a.W1 + (int64_t)l * d * h + e);
      }
      for (int e = tid * 4; e < rows * h; e += 4 * kThreads) copy16_async(to + 2 * d * h + e, a.DACT + ((int64_t)l * a.N + row0) * h + e);
    }
    copy_group();
  }
  for (int e = tid; e < rd; e += kThreads) last_delta[e] = e < rows * d ? a.delta[(a.every ? L * state : 0) + row0 * d + e] : 0.0f;  // (each its own)
  // Every CTA walks the layers down for all elements: g_l = delta_l + a_l g_{l+1} (+ u_l), and keeps the iterates of its own.  The running
  // value is a double, as in the scans of scan.cu: a state is rounded where it is stored, not on the way to the next one.
  auto scan = [&](const float* u, bool last) {
    for (int e = tid; e < rd; e += kThreads) {
      const int c = e % d;
      const bool in = e < rows * d;
      const int64_t at = row0 * d + e;
      double g = last_delta[e];
      if (last && in && L % kCluster == rank) a.g_all[L * state + at] = (float)g;
      for (int top = L - 1; top >= 0; top -= kCluster) {  // eight layers' operands at a time, then their chain
        float ul[kCluster], dl[kCluster], gt[kCluster];
#pragma unroll
        for (int j = 0; j < kCluster; ++j) {
          const int l = top - j;
          ul[j] = dl[j] = 0.0f;
          gt[j] = 1.0f;
          if (l < 0) continue;
          if (u) ul[j] = u[l * rd + e];
          if (a.every && in) dl[j] = a.delta[l * state + at];
          if (a.gate != HBP_GATE_ONE) gt[j] = gate_of(a, l)[c];
        }
#pragma unroll
        for (int j = 0; j < kCluster; ++j) {
          const int l = top - j;
          if (l < 0) continue;
          if (l % kCluster == rank) G[l / kCluster * rd + e] = (float)g;
          g = gt[j] * g + ul[j];
          g += dl[j];
          if (last && in && l % kCluster == rank) a.g_all[l * state + at] = (float)g;
        }
      }
    }
    __syncthreads();
  };
  // The sum of the groups' parts of a pass over four columns each
  auto add_groups = [&](const Share& sh, int e) {
    float v = red[e];
#pragma unroll 8
    for (int q = 1; q < sh.groups; ++q) v += red[q * kRows * 4 * sh.quads + e];
    return v;
  };
  auto product = [&](const float* w, int width, const float* x, int pitch, int count, auto store) {  // store(row, column, sum)
    const Share sh = share_of(width);
    const int group = tid / sh.quads, quad = tid % sh.quads;
    for (int q0 = 0; q0 < width / 4; q0 += sh.quads) {
      if (group < sh.groups && q0 + quad < width / 4) {
        float4 acc[kRows];
        four_columns(w + 4 * (q0 + quad), width, x, pitch, count, 4 * group, 4 * sh.groups, acc);
#pragma unroll
        for (int r = 0; r < kRows; ++r) *reinterpret_cast<float4*>(red + ((group * kRows + r) * sh.quads + quad) * 4) = acc[r];
      }
      __syncthreads();
      for (int e = tid; e < kRows * 4 * sh.quads; e += kThreads) {
        const int r = e / (4 * sh.quads), c = 4 * q0 + e % (4 * sh.quads);
        if (c < width) store(r, c, add_groups(sh, e));
      }
      __syncthreads();
    }
  };
  auto layer = [&](int s, const float* x, float* u, bool to_memory) {
    const int l = s * kCluster + rank;
    const float *W2 = a.W2 + (int64_t)l * d * h, *W1 = a.W1 + (int64_t)l * h * d, *prime = a.DACT + ((int64_t)l * a.N + row0) * h;
    if (a.resident) {
      W2 = kept + s * per_slot;
      W1 = W2 + d * h;
      prime = W1 + d * h;
    }
    product(W2, h, x, d, d, [&](int r, int i, float v) {
      v = r < rows ? v * prime[r * h + i] : 0.0f;
      dz[r * h + i] = v;
      if (to_memory && r < rows) a.dZ[((int64_t)l * a.N + row0 + r) * h + i] = v;
    });
    if (to_memory) return;
    const uint32_t to = smem_u32(u + l * rd);
    if (!a.preln) {
      product(W1, d, dz, h, h, [&](int r, int c, float v) {
#pragma unroll
        for (int j = 0; j < kCluster; ++j) st_peer(to + 4u * (r * d + c), j, v);
      });
      return;
    }
    product(W1, d, dz, h, h, [&](int r, int c, float v) { y[r * d + c] = v; });
    if (warp < kRows) {  // through the LayerNorm: rstd (dy - mean dy - xhat mean(dy xhat))
      const bool in = warp < rows;
      const float *xh = a.Y + l * state + (row0 + warp) * d, *dy = y + warp * d;
      float s1 = 0.0f, s2 = 0.0f;
      for (int c = lane; c < d; c += 32) {
        s1 += dy[c];
        s2 = fmaf(dy[c], in ? xh[c] : 0.0f, s2);
      }
      const float m1 = warp_sum(s1) / (float)d, m2 = warp_sum(s2) / (float)d, r = in ? a.rstd[l * a.N + row0 + warp] : 0.0f;
      for (int c = lane; c < d; c += 32) {
        const float v = r * (dy[c] - m1 - (in ? xh[c] : 0.0f) * m2);
#pragma unroll
        for (int j = 0; j < kCluster; ++j) st_peer(to + 4u * (warp * d + c), j, v);
      }
    }
    // (y is written again only after the next product's barriers)
  };
  if (a.exact) {  // step by step: one CTA forms a layer's product, all add it to the running gradient (in place of last_delta)
    for (int e = tid; e < rows * d; e += kThreads)
      if (L % kCluster == rank) a.g_all[L * state + row0 * d + e] = last_delta[e];
    copy_wait<0>();
    cluster_sync();  // every CTA's shared memory may be written from here on
    for (int l = L - 1; l >= 0; --l) {
      const bool own = l % kCluster == rank;
      const float* u = U + (l & 1) * rd;
      if (own) layer(l / kCluster, last_delta, U + ((l & 1) - l) * rd, false);
      cluster_sync();
      for (int e = tid; e < rd; e += kThreads) {
        const bool in = e < rows * d;
        const int64_t at = l * state + row0 * d + e;
        double sum = last_delta[e];  // (rounded once a layer)
        if (a.gate != HBP_GATE_ONE) sum *= gate_of(a, l)[e % d];
        sum += u[e];
        if (a.every && in) sum += a.delta[at];
        const float g = (float)sum;
        last_delta[e] = g;
        if (own && in) a.g_all[at] = g;
      }
      if (own && a.dZ)
        for (int e = tid; e < rows * h; e += kThreads) a.dZ[((int64_t)l * a.N + row0) * h + e] = dz[e];
      __syncthreads();
    }
    return;
  }
  auto vjp = [&](float* u, bool to_memory) {
    for (int s = 0; s * kCluster + rank < L; ++s) layer(s, G + s * rd, u, to_memory);
  };
  scan(nullptr, a.k == 0);
  copy_wait<0>();
  cluster_sync();  // every CTA's shared memory may be written from here on
  for (int it = 0; it < a.k; ++it) {
    float* u = U + (it & 1) * L * rd;
    vjp(u, false);
    cluster_sync();
    scan(u, it + 1 == a.k);
  }
  if (a.dZ) vjp(nullptr, true);
}

// Weight gradients of every layer, dW2 = G^T gelu(Z) and dW1 = dZ^T y: sums over at most 32 rows, 64 x 64 outputs a block.  Eight
// rows add up at a time: the error is that of sums of eight and of four.
constexpr int kTile = 64, kMostRows = 32;
__global__ void __launch_bounds__(kThreads, 1) few_rows_wgrad_kernel(const FewRows a, const float* g, const float* y, float* dW1, float* dW2) {
  __shared__ __align__(16) float sa[kMostRows][kTile], sb[kMostRows][kTile];
  const int tid = threadIdx.x, d = a.d, h = a.h, N = (int)a.N;
  const int dt = (d + kTile - 1) / kTile, ht = (h + kTile - 1) / kTile;  // as many blocks for either product
  const int block = (int)(blockIdx.x % (dt * ht)), product = (int)(blockIdx.x / (dt * ht)), l = product >> 1;
  const bool first = product & 1;  // dW1 [h][d], else dW2 [d][h]
  const int M = first ? h : d, K = first ? d : h, across = first ? dt : ht, m0 = block / across * kTile, n0 = block % across * kTile;
  chain_next();
  chain_wait();
  const float* A = first ? a.dZ + (int64_t)l * N * h : g + (int64_t)(l + 1) * N * d;
  const float* B = first ? y + (int64_t)l * N * d : a.ACT + (int64_t)l * N * h;
  const int quad = tid % (kTile / 4) * 4;
#pragma unroll
  for (int i = 0; i < kMostRows * kTile / 4 / kThreads; ++i) {
    const int r = tid / (kTile / 4) + i * (kThreads / (kTile / 4));
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    *reinterpret_cast<float4*>(&sa[r][quad]) = r < N && m0 + quad < M ? vec4(A + (int64_t)r * M + m0 + quad) : zero;
    *reinterpret_cast<float4*>(&sb[r][quad]) = r < N && n0 + quad < K ? vec4(B + (int64_t)r * K + n0 + quad) : zero;
  }
  __syncthreads();
  const int m = tid / 16 * 4, n = tid % 16 * 4;
  float4 sum[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) sum[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
  for (int r0 = 0; r0 < kMostRows; r0 += 8) {
    if (r0 >= N) break;
    float4 acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int r = r0; r < r0 + 8; ++r) {
      const float4 av = vec4(&sa[r][m]), bv = vec4(&sb[r][n]);
      const float am[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[i].x = fmaf(am[i], bv.x, acc[i].x);
        acc[i].y = fmaf(am[i], bv.y, acc[i].y);
        acc[i].z = fmaf(am[i], bv.z, acc[i].z);
        acc[i].w = fmaf(am[i], bv.w, acc[i].w);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) sum[i] = make_float4(sum[i].x + acc[i].x, sum[i].y + acc[i].y, sum[i].z + acc[i].z, sum[i].w + acc[i].w);
  }
  float* D = (first ? dW1 : dW2) + (int64_t)l * d * h;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (m0 + m + i < M && n0 + n < K) {
      float* at = D + (int64_t)(m0 + m + i) * K + n0 + n;
      const float v[4] = {sum[i].x, sum[i].y, sum[i].z, sum[i].w};
      if (((uintptr_t)D & 15u) == 0) *reinterpret_cast<float4*>(at) = sum[i];
      else
        for (int j = 0; j < 4; ++j) at[j] = v[j];
    }
}

size_t forward_smem(const FewRows& a) {
  const int hs = units_per_cta(a.h);
  return (size_t)4 * (kRows * (2 * a.d + 2 * hs + 2 * kCluster * a.d) + 4 * hs * a.d);
}
size_t backward_smem(const FewRows& a) {
  const int slots = (a.L + kCluster - 1) / kCluster, red_d = share_floats(a.d), red_h = share_floats(a.h);
  const int states = a.exact ? 2 : slots + 2 * a.L;
  return (size_t)4 * (kRows * (states * a.d + a.h + 2 * a.d) + (red_d > red_h ? red_d : red_h) + (a.resident ? slots * (2 * a.d * a.h + kRows * a.h) : 0));
}

// The kernel's limit is set once per device and for any size: one set for a call could be lowered by another thread's before the launch.
template <void (*kernel)(const FewRows)>
bool launch(Launcher& lc, size_t smem, const FewRows& a, bool* refused) {
  if (smem > kMostSmem) return false;
  *refused = true;
  static PerDevice<bool> attr_done;
  if (!attr_done.here()) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMostSmem) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    attr_done.here() = true;
  }
  const unsigned clusters = (unsigned)((a.N + kRows - 1) / kRows);
  if (try_launch_chained(lc, kernel, dim3(clusters * kCluster), kThreads, smem, kCluster, a) != cudaSuccess) return false;
  *refused = false;
  lc.ran(HBP_FORM_FEW_ROWS);
  return true;
}
bool aligned(const void* p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

// 32 rows, forward pass in us here and with a launch per product: 8 layers 64 (256) 22 and 133, 128 (512) 37 and 166, 256 (256) 43 and 159, 2
// layers 64 (128) 9 and 31, 64 layers 64 (256) 162 and 1050, 64 layers 128 (512) 278 and 1313; 1 row, 8 layers 64 (256) 20 and 101.  Beyond 64 K
// weights a matrix its two layers no longer fit shared memory, and backward passes gain less (8 layers 256 (1024) 79, 200 and 82, 214).
// 32 rows are where the products move to the tensor cores (hbp_api.cu, keeps_parts), not where these kernels stop gaining.
bool few_rows_take(int64_t N, int d, int h) { return N <= 32 && (int64_t)d * h <= 64 * 1024; }

bool few_rows_forward(Launcher& lc, const FewRows& a, bool* refused) {
  if (!aligned(a.W1) || !aligned(a.W2)) return false;
  return launch<few_rows_forward_kernel>(lc, forward_smem(a), a, refused);
}
// Which backward passes gain.  A CTA works its layers off one by one, every 8 layers take an iteration 4 to 13 us more, where the batched
// products of all layers hardly take longer for more of them (and from 32 layers on their scan runs in the ring).  Backward(1) and (4)
// without gradients in us here and with a launch per product, 32 rows: 64 (256) 8 layers 10, 22 and 29, 91; 24 layers 21, 69 and 40, 126; 32
// layers 27, 89 and 34, 95; 64 layers 48, 168 and 44, 118; 200 layers 32 (128) 91, 321 and 78, 164.  Matrices of more than 32 K weights, as
// long as neither side makes the batched products long too (64 (1024), 24 layers 45, 163 and 59, 203), break even at one layer a CTA: 256
// (256) 8 layers 20, 63 and 29, 97; 9 layers 32, 109 and 29, 97, of which the gradient pass makes 48, 125 and 57, 126 (pre-LN 49, 131
// and 55, 121); 512 (128) pre-LN, 9 layers 43, 141 and 32, 106, with gradients 57, 155 and 64, 138.
// The exact pass always gains (32 rows 8 layers 64 (256) 38 and 163, 64 layers 337 and 1197, with gradients) until the weights of such
// matrices, read from L2 by a CTA at a time, and the gradients written no longer fit there: 256 (256), 3 rows with gradients 64 layers
// (34 + 34 MB) 957 and 1452, 100 layers 2213 and 2283, pre-LN 2311 and 2073, 400 layers 9069 and 9006, 9482 and 8197; with more
// clusters to wait for them 9 rows 200 layers 4208 and 4834, 32 rows 4132 and 4628, but pre-LN 4334 and 4227.
static bool backward_gains(const FewRows& a) {
  const int64_t weights = (int64_t)a.d * a.h;
  const bool heavy = weights > 32 * 1024 && a.d < 1024 && a.h < 1024;
  if (a.exact) return !heavy || 8 * a.L * weights * (a.dZ ? 2 : 1) <= (72 << 20) || (!a.preln && a.N > 8);
  if (a.L <= kCluster) return true;
  return heavy ? a.L <= 2 * kCluster && a.dZ && a.d <= 256 && a.k <= 3 : a.L <= 3 * kCluster;
}
bool few_rows_backward(Launcher& lc, const FewRows& args, bool* refused) {
  FewRows a = args;
  if (!aligned(a.W1) || !aligned(a.W2) || !backward_gains(a)) return false;
  a.resident = true;
  if (backward_smem(a) > kMostSmem) a.resident = false;
  return launch<few_rows_backward_kernel>(lc, backward_smem(a), a, refused);
}

void few_rows_wgrad(Launcher& lc, const FewRows& a, const float* g, const float* y, float* dW1, float* dW2) {
  const unsigned dt = (unsigned)((a.d + kTile - 1) / kTile), ht = (unsigned)((a.h + kTile - 1) / kTile);
  launch_chained(lc, few_rows_wgrad_kernel, dim3(dt * ht * 2 * (unsigned)a.L), kThreads, 0, 1, a, g, y, dW1, dW2);
}

}  // namespace hbp
