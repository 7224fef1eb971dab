// Forward recurrence of the gated tanh RNN, h_{t+1} = a * h_t + tanh(W h_t + U x_t) (Section 5.2), as ONE launch over
// all T steps on the FP64 matrix instruction: the same clusters, exchange and bounded waits as cell_cluster.cu.
//
// With gates near one this network amplifies the last bit of its pre-activations by many orders of magnitude over a few
// thousand steps, so the sums are taken in EXACTLY the order of the kernels this one stands in for, and the states agree
// with theirs bit for bit.  The matrix instruction makes that possible: it adds its four products one after the other,
// each rounded like an FMA, in ascending order of the contraction index (checked against an FMA chain on random data).
//   parts    (128, 256, 512 units; rnn_persistent.cu): 16 consecutive parts of the contraction, added pairwise, plus
//            U x_t formed beforehand as one ascending sum
//   classes  (other widths; rnn_step_staged_kernel in rnn.cu): the concatenation [h | x_t] in 8 residue classes mod 8;
//            a trailing half block of 4 elements goes to classes 0 and 1
// A chain (part or class) is one accumulator tile; step i of a chain covers its elements 4i .. 4i + 3, one per lane of a
// quad.  State and weights lie in shared memory in that order, so neither is ever rearranged in the loop.
//
// Bound by the FP64 rate plus, per step, one exchange and one exponential.  What it gains over rnn_persistent.cu is rows
// per cluster: that form takes 4 rows per cluster of 16 CTAs and 7 such clusters run at a time, so more than 28 rows
// queue; here a cluster takes up to 24 rows at the cost of one, two or three 8-row tiles.  Measured (us per step): 32 rows, 512
// units, 256 inputs 5.5 -> 3.2; 192 rows, 128 units 3.7 -> 1.6; per-step widths: 50 rows, 300 units 12.4 -> 3.0.
#include "cell_common.cuh"

namespace hbp {

using namespace cell;

namespace {

constexpr int kMaxThreads = 256;

struct RnnArgs {
  const void *W, *U, *X, *x0, *gate;
  const double* P;    // parts: U x_t of every step [T][B][u]
  float4* Wp;         // weights by [unit tile][step][4 chains][32]
  void *states, *deriv;
  int* status;
  int T, B, u, in;
  int rows, uc, res;  // rows per cluster, units per CTA, chain steps whose weights stay in shared memory
};

// Chain and place in it of element k of the contraction (n elements), and back (-1: padding).
__host__ __device__ __forceinline__ int chain_of(bool parts, int n, int k) {
  if (parts) return k / (n / 16);
  return (n & 4) && k >= n - 2 ? k - (n - 2) : k & 7;
}
__host__ __device__ __forceinline__ int place_of(bool parts, int n, int k) {
  if (parts) return k % (n / 16);
  return (n & 4) && k >= n - 2 ? (n >> 3) + 1 : k >> 3;
}
__host__ __device__ __forceinline__ int element_at(bool parts, int n, int chain, int place) {
  if (parts) return place < n / 16 ? chain * (n / 16) + place : -1;
  const int q = n >> 3;
  if (place < q) return 8 * place + chain;
  if (!(n & 4) || chain > 1 || place > q + 1) return -1;
  return place == q ? 8 * q + chain : n - 2 + chain;
}
__host__ __device__ __forceinline__ int chain_steps(bool parts, int n) {
  return parts ? n / 64 : ((n >> 3) + ((n & 4) ? 2 : 0) + 3) / 4;
}

template <typename T, int MT, int NCW, bool PARTS>
__global__ void __launch_bounds__(kMaxThreads, 1) rnn_cluster_kernel(const RnnArgs p) {
  constexpr int NC = PARTS ? 16 : 8, KS = NC / NCW;  // chains; warps that share an 8-unit tile's chains out
  constexpr int kAhead = 2;                          // streamed chain steps in flight per warp
  constexpr int kOuts = (2 * MT + KS - 1) / KS;      // outputs per thread
  const int kThreads = (int)blockDim.x, R = p.rows, u = p.u, in = p.in, uc = p.uc, ntu = uc / 8;
  const int n_k = PARTS ? u : u + in, steps = chain_steps(PARTS, n_k);
  const int cs = (int)cluster_size(), rank = (int)tc::cluster_ctarank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nt = warp % ntu, ks = warp / ntu;
  const int row0 = (int)cluster_index() * R, live_rows = min(R, p.B - row0);
  const int outs = 8 * MT * uc;

  extern __shared__ __align__(16) unsigned char rnn_smem[];
  const uint32_t buf_bytes = (uint32_t)steps * NC * MT * 256u;
  const uint32_t x_bytes = PARTS ? 0u : (uint32_t)R * in * (uint32_t)sizeof(T);
  unsigned char* xs = rnn_smem + 2 * buf_bytes;                                  // classes: inputs of two steps
  double* red = reinterpret_cast<double*>(xs + ((2 * x_bytes + 15u) & ~15u));    // [chain][outs]
  float4* wres = reinterpret_cast<float4*>(red + NC * outs);                     // [warp][res][NCW / 4][32]
  uint64_t* bars = reinterpret_cast<uint64_t*>(wres + ntu * KS * p.res * (NCW / 4) * 32);  // h x 2, inputs x 2
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 4);
  const uint32_t vbuf = tc::smem_u32(rnn_smem), bar0 = tc::smem_u32(bars), xbar0 = bar0 + 16;

  // byte offset of (row, element k) in a buffer: elements k, k + 1 (k even) of a row are neighbours in both orders
  auto v_offset = [&](int row, int k) {
    const int c = chain_of(PARTS, n_k, k), place = place_of(PARTS, n_k, k), i = place >> 2, l = (row & 7) * 4 + (place & 3);
    if (PARTS) return (uint32_t)(((i * NC + c) * MT + (row >> 3)) * 256 + l * 8);
    return (uint32_t)(((i * (NC / 2) + (c >> 1)) * MT + (row >> 3)) * 512 + l * 16 + (c & 1) * 8);
  };
  const float4* gW = p.Wp + ((rank * ntu + nt) * steps * NC / 4 + ks * (NCW / 4)) * 32 + lane;
  auto load_w = [&](int i, float4* b) {
#pragma unroll
    for (int q = 0; q < NCW / 4; ++q) b[q] = __ldg(gW + (i * (NC / 4) + q) * 32);
  };
  const int res = min(p.res, steps);
  const float4* my_w = wres + warp * p.res * (NCW / 4) * 32 + lane;

  auto fetch_x = [&](int t) {  // one thread: the rows of a step are one contiguous block
    fetch_rows(tc::smem_u32(xs) + (t & 1) * x_bytes, (const T*)p.X + ((int64_t)t * p.B + row0) * in,
               (uint32_t)live_rows * in * (uint32_t)sizeof(T), xbar0 + 8 * (t & 1));
  };
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) tc::mbar_init(bar0 + 8 * i, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (!PARTS && p.T > 1) fetch_x(1);
  }
  for (int i = tid; i < (int)(2 * buf_bytes / 16); i += kThreads) reinterpret_cast<double2*>(rnn_smem)[i] = make_double2(0.0, 0.0);
  for (int i = 0; i < res; ++i) {
    float4 b[NCW / 4];
    load_w(i, b);
#pragma unroll
    for (int q = 0; q < NCW / 4; ++q) wres[((warp * p.res + i) * (NCW / 4) + q) * 32 + lane] = b[q];
  }
  __syncthreads();
  for (int row = 0; row < live_rows; ++row) {  // h_0 (and x_0), every CTA its own copy
    for (int k = tid; k < u; k += kThreads)
      *reinterpret_cast<double*>(rnn_smem + v_offset(row, k)) = (double)to_f(((const T*)p.x0)[(int64_t)(row0 + row) * u + k]);
    if (!PARTS)
      for (int k = tid; k < in; k += kThreads)
        *reinterpret_cast<double*>(rnn_smem + v_offset(row, u + k)) = (double)to_f(((const T*)p.X)[(int64_t)(row0 + row) * in + k]);
  }
  // this thread's outputs, in the order a tile's lanes hold the sums: (row, units 2c, 2c + 1)
  int o_row[kOuts], o_unit[kOuts];
  bool o_on[kOuts], o_live[kOuts];
  double a_gate[kOuts];
  uint32_t voff[kOuts];
#pragma unroll
  for (int it = 0; it < kOuts; ++it) {
    const int o = min(tid + it * kThreads, outs - 1), tile = o >> 6, l = (o & 63) >> 1;
    o_row[it] = (tile / ntu) * 8 + (l >> 2);
    o_unit[it] = rank * uc + (tile % ntu) * 8 + 2 * (l & 3) + (o & 1);
    o_on[it] = tid + it * kThreads < outs && o_row[it] < R;
    o_live[it] = o_on[it] && o_unit[it] < u && o_row[it] < live_rows;
    a_gate[it] = (p.gate && o_live[it]) ? (double)to_f(((const T*)p.gate)[o_unit[it]]) : 1.0;
    voff[it] = o_unit[it] < u ? v_offset(o_row[it], o_unit[it]) : 0u;
  }
  // padding units (an 8-unit tile that reaches past u) are not sent: their elements do not exist in a buffer
  const uint32_t step_bytes = (uint32_t)u * R * 8u;
  __syncthreads();
  tc::cluster_sync();  // every CTA of the cluster has started: barriers and buffers exist

  bool ok = true;
  for (int t = 0; t < p.T; ++t) {
    const uint32_t cur = t & 1, nxt = cur ^ 1;
    if (tid == 0) {
      if (t + 1 < p.T) tc::mbar_expect_tx(bar0 + 8 * nxt, step_bytes);
      if (!PARTS && t + 2 < p.T) fetch_x(t + 2);  // (its buffer was read before the last barrier)
    }
    double add[kOuts];
#pragma unroll
    for (int it = 0; it < kOuts; ++it) {
      add[it] = 0.0;
      if (PARTS && o_live[it]) {
        const double* P = p.P + ((int64_t)t * p.B + row0 + o_row[it]) * u + o_unit[it];
        add[it] = __ldg(P);
        if (t + 3 < p.T) prefetch_l2(P + (int64_t)3 * p.B * u);
      }
    }
    if (!PARTS && t + 1 < p.T) {  // x_{t+1} as double into the next buffer (last read before the last barrier)
      ok = bar_wait_cluster(xbar0 + 8 * nxt, (uint32_t)(((t + 1) >> 1) - (int)cur) & 1u, abort_flag) && ok;
      const T* x = reinterpret_cast<const T*>(xs + nxt * x_bytes);
      for (int row = 0; row < live_rows; ++row)
        for (int k = tid; k < in; k += kThreads)
          *reinterpret_cast<double*>(rnn_smem + nxt * buf_bytes + v_offset(row, u + k)) = (double)to_f(x[row * in + k]);
    }
    double2 acc[NCW][MT];
#pragma unroll
    for (int c = 0; c < NCW; ++c)
#pragma unroll
      for (int m = 0; m < MT; ++m) acc[c][m] = make_double2(0.0, 0.0);
    float4 pre[kAhead][NCW / 4];
#pragma unroll
    for (int s = 0; s < kAhead; ++s) load_w(min(res + s, steps - 1), pre[s]);
    if (t > 0) ok = bar_wait_cluster(bar0 + 8 * cur, (uint32_t)(((t - 1) >> 1) & 1), abort_flag) && ok;
    if (ok) {
      const unsigned char* vb = rnn_smem + cur * buf_bytes;
      auto multiply = [&](int i, const float4* b) {
        if (PARTS) {
#pragma unroll
          for (int c = 0; c < NCW; ++c) {
            const double bv = (double)lane4(b[c / 4], c & 3);
#pragma unroll
            for (int m = 0; m < MT; ++m)
              dmma(acc[c][m], *reinterpret_cast<const double*>(vb + ((i * NC + ks * NCW + c) * MT + m) * 256 + lane * 8), bv);
          }
        } else {
#pragma unroll
          for (int c = 0; c < NCW; c += 2) {
            const double b0 = (double)lane4(b[c / 4], c & 3), b1 = (double)lane4(b[c / 4], (c & 3) + 1);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
              const double2 a = *reinterpret_cast<const double2*>(vb + ((i * (NC / 2) + (ks * NCW + c) / 2) * MT + m) * 512 + lane * 16);
              dmma(acc[c][m], a.x, b0);
              dmma(acc[c + 1][m], a.y, b1);
            }
          }
        }
      };
#pragma unroll 2
      for (int i = 0; i < res; ++i) {
        float4 b[NCW / 4];
#pragma unroll
        for (int q = 0; q < NCW / 4; ++q) b[q] = my_w[(i * (NCW / 4) + q) * 32];
        multiply(i, b);
      }
      int i = res;
      for (; i + kAhead <= steps; i += kAhead) {
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
          multiply(i + s, pre[s]);
          load_w(min(i + s + kAhead, steps - 1), pre[s]);
        }
      }
      if (i < steps) multiply(i, pre[0]);
#pragma unroll
      for (int c = 0; c < NCW; ++c)
#pragma unroll
        for (int m = 0; m < MT; ++m)
          *reinterpret_cast<double2*>(red + (ks * NCW + c) * outs + ((m * ntu + nt) * 32 + lane) * 2) = acc[c][m];
    }
    if (__syncthreads_or(!ok)) {  // the chains' sums are in place; or the whole CTA leaves together
      ok = false;
      break;
    }
#pragma unroll
    for (int it = 0; it < kOuts; ++it) {
      const int o = min(tid + it * kThreads, outs - 1);
      double q[NC], z, th, sl;
#pragma unroll
      for (int c = 0; c < NC; ++c) q[c] = red[c * outs + o];
      if (PARTS) {
#pragma unroll
        for (int w = 1; w < NC; w *= 2)  // ((q0 + q1) + (q2 + q3)) + ...
#pragma unroll
          for (int c = 0; c < NC; c += 2 * w) q[c] += q[c + w];
        z = q[0] + add[it];
      } else {
        z = ((q[0] + q[2]) + (q[4] + q[6])) + ((q[1] + q[3]) + (q[5] + q[7]));
      }
      const double e = exp(-2.0 * fabs(z));
      if (PARTS) {  // (the two forms' own last operations: their results differ in the last bit)
        const double rcp = 1.0 / (1.0 + e);
        th = copysign((1.0 - e) * rcp, z);
        sl = 4.0 * e * rcp * rcp;
      } else {
        th = copysign((1.0 - e) / (1.0 + e), z);
        sl = 4.0 * e / ((1.0 + e) * (1.0 + e));
      }
      const double hp = *reinterpret_cast<const double*>(rnn_smem + cur * buf_bytes + voff[it]);
      double hn = a_gate[it] * hp + th;
      if (!o_live[it]) hn = 0.0;
      if (t + 1 < p.T) {  // nobody reads what the last step would send; the even lane of a pair sends both units
        const double other = __shfl_down_sync(0xffffffffu, hn, 1);
        if (o_on[it] && o_unit[it] < u && !(tid & 1)) {
          const uint32_t dst = vbuf + nxt * buf_bytes + voff[it], bar = bar0 + 8 * nxt;
          for (int r = 0; r < cs; ++r) {
            const int to = rank + r < cs ? rank + r : rank + r - cs;  // each CTA starts with another peer
            send16(tc::map_to_cta(dst, to), hn, other, tc::map_to_cta(bar, to));
          }
        }
      }
      if (o_live[it]) {
        const int64_t at = ((int64_t)t * p.B + row0 + o_row[it]) * u + o_unit[it];
        ((T*)p.states)[at + (int64_t)p.B * u] = from_f<T>((float)hn);
        ((T*)p.deriv)[at] = from_f<T>((float)sl);
      }
    }
  }
  if (!ok) after_timeout(p.status);
  tc::cluster_sync();
}

// Weights in chain order: element (lane, j) of (unit tile, step, 4 chains) belongs to unit 8 tile + lane / 4, chain
// 4 group + j, place 4 step + lane % 4.
template <typename T>
__global__ void __launch_bounds__(256) rnn_pack_kernel(const T* __restrict__ W, const T* __restrict__ U, float4* __restrict__ out, int u,
                                                       int in, int parts, int steps, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int groups = parts ? 4 : 2, n_k = parts ? u : u + in;
  const int lane = i & 31, grp = (i >> 5) % groups, step = (i >> 5) / groups % steps, tile = (i >> 5) / groups / steps;
  const int unit = tile * 8 + (lane >> 2);
  float v[4];
  for (int j = 0; j < 4; ++j) {
    const int k = element_at(parts != 0, n_k, 4 * grp + j, 4 * step + (lane & 3));
    v[j] = k < 0 || unit >= u ? 0.0f : (k < u ? to_f(W[unit * u + k]) : to_f(U[unit * in + k - u]));
  }
  out[i] = make_float4(v[0], v[1], v[2], v[3]);
}

struct RnnPlan {
  int uc = 0, cs = 0, mt = 0, ncw = 0, rows = 0, res = 0, threads = 0;
  size_t smem = 0;
};

// As make_plan in cell_cluster.cu: matrix instructions at 16 clocks each on a warp's quarter of the SM, the exchange, 1200
// clocks for the rest of a step, times the waves of clusters.
template <typename ActiveClusters>
bool make_rnn_plan(bool parts, int es, int B, int u, int in, ActiveClusters active, RnnPlan* best) {
  const int nc = parts ? 16 : 8, n_k = parts ? u : u + in, steps = chain_steps(parts, n_k);
  double best_cost = 0.0;
  best->uc = 0;
  for (int uc = 8; uc <= 64; uc += 8) {
    const int cs = (u + uc - 1) / uc, ntu = uc / 8;
    if (cs > kMaxCluster || uc >= u + 8) continue;
    for (int ncw = 4; ncw <= 8; ncw += 4) {
      const int warps = ntu * (nc / ncw);
      if (warps > kMaxThreads / 32) continue;
      for (int mt = 1; mt <= 3; ++mt) {
        const int at_once = active(mt, ncw, cs);
        if (at_once <= 0) continue;
        RnnPlan q;
        const int spread = (B + at_once - 1) / at_once;
        q.uc = uc; q.cs = cs; q.mt = mt; q.ncw = ncw; q.threads = 32 * warps;
        q.rows = spread < 8 * mt ? spread : 8 * mt;
        if (q.rows <= 8 * (mt - 1)) continue;
        const size_t base = (size_t)2 * steps * nc * mt * 256 + (parts ? 0 : ((size_t)2 * q.rows * in * es + 15) / 16 * 16) +
                            (size_t)nc * 8 * mt * uc * 8 + 64;
        if (base > (size_t)kSmemLimit) continue;
        const int waves = ((B + q.rows - 1) / q.rows + at_once - 1) / at_once;
        const double cost = waves * (16.0 * steps * ncw * mt * ((warps + 3) / 4) + 1200.0 + 150.0 * mt +
                                     exchange_clocks(cs, q.rows, uc));
        if (best->uc && cost >= best_cost) continue;
        const size_t block = (size_t)warps * (ncw / 4) * 512, left = (size_t)kSmemLimit - base;
        q.res = (int)(left / block < (size_t)steps ? left / block : (size_t)steps);
        q.smem = base + q.res * block;
        *best = q;
        best_cost = cost;
      }
    }
  }
  return best->uc != 0;
}

template <typename T, int MT, int NCW, bool PARTS>
int active_rnns(int cs) {
  return active_clusters<rnn_cluster_kernel<T, MT, NCW, PARTS>>(cs, kMaxThreads);
}

template <typename T, bool PARTS>
bool run_rnn(Launcher& lc, RnnArgs a) {
  auto active = [](int mt, int ncw, int cs) {
    if (ncw == 4) return mt == 1 ? active_rnns<T, 1, 4, PARTS>(cs) : (mt == 2 ? active_rnns<T, 2, 4, PARTS>(cs) : active_rnns<T, 3, 4, PARTS>(cs));
    return mt == 1 ? active_rnns<T, 1, 8, PARTS>(cs) : (mt == 2 ? active_rnns<T, 2, 8, PARTS>(cs) : active_rnns<T, 3, 8, PARTS>(cs));
  };
  RnnPlan q;
  if (!make_rnn_plan(PARTS, (int)sizeof(T), a.B, a.u, a.in, active, &q)) return false;
  const int steps = chain_steps(PARTS, PARTS ? a.u : a.u + a.in), n = q.cs * (q.uc / 8) * steps * (PARTS ? 4 : 2) * 32;
  rnn_pack_kernel<T><<<(n + 255) / 256, 256, 0, lc.stream>>>((const T*)a.W, (const T*)a.U, a.Wp, a.u, a.in, PARTS, steps, n);
  lc.count();
  lc.check();
  a.rows = q.rows; a.uc = q.uc; a.res = q.res;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  launch_config(cfg, attr, (a.B + q.rows - 1) / q.rows, q.cs, q.threads, q.smem, lc.stream);
  auto launch = [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, a); };
  cudaError_t e;
  if (q.ncw == 4)
    e = q.mt == 1 ? launch(rnn_cluster_kernel<T, 1, 4, PARTS>) : (q.mt == 2 ? launch(rnn_cluster_kernel<T, 2, 4, PARTS>) : launch(rnn_cluster_kernel<T, 3, 4, PARTS>));
  else
    e = q.mt == 1 ? launch(rnn_cluster_kernel<T, 1, 8, PARTS>) : (q.mt == 2 ? launch(rnn_cluster_kernel<T, 2, 8, PARTS>) : launch(rnn_cluster_kernel<T, 3, 8, PARTS>));
  if (e != cudaSuccess) {  // clusters of this size cannot be placed here: the caller runs another form
    cudaGetLastError();
    return false;
  }
  lc.ran(HBP_FORM_RNN_CLUSTER);
  lc.count();
  lc.check();
  return true;
}

}  // namespace

size_t rnn_cluster_pack_bytes(int u, int in_dim) {
  const bool parts = u == 128 || u == 256 || u == 512;
  size_t most = 0;
  for (int uc = 8; uc <= 64; uc += 8) {
    const int cs = (u + uc - 1) / uc;
    if (cs > kMaxCluster) continue;
    const size_t n = (size_t)cs * (uc / 8) * chain_steps(parts, parts ? u : u + in_dim) * (parts ? 4 : 2) * 32 * sizeof(float4);
    if (n > most) most = n;
  }
  return most;
}

bool rnn_forward_cluster(Launcher& lc, int dtype, const void* W, const void* U, const void* X, const void* gate, const void* x0,
                         double* P, void* x_all, void* deriv, int T, int B, int u, int in_dim, void* pack, int* status) {
  const bool parts = u == 128 || u == 256 || u == 512;
  // the other widths stand in for the staged per-step kernel, so only where that is what would run
  if (!pack || T <= 0 || B <= 0 || (parts ? !P : !rnn_step_is_staged(u, in_dim)) || ((uintptr_t)X & 15u)) return false;
  RnnArgs a = {};
  a.W = W; a.U = U; a.X = X; a.x0 = x0; a.gate = gate; a.P = P; a.Wp = (float4*)pack; a.states = x_all; a.deriv = deriv; a.status = status;
  a.T = T; a.B = B; a.u = u; a.in = in_dim;
  if (parts) {
    rnn_project(lc, dtype, X, U, P, (int64_t)T * B, u, in_dim);
    return dtype == HBP_F32 ? run_rnn<float, true>(lc, a) : run_rnn<bf16, true>(lc, a);
  }
  return dtype == HBP_F32 ? run_rnn<float, false>(lc, a) : run_rnn<bf16, false>(lc, a);
}

}  // namespace hbp
