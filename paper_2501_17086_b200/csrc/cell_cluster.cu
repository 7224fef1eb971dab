// The recurrences of the gated cells as ONE launch over all T steps, up to 1536 units (16 CTAs of 96):
//     forward     (GRU, LSTM) next state, stored state and the coefficients of the backward pass, from h_0 and all inputs
//     exact BPTT  (tanh RNN, GRU, LSTM) g_t from g_{t+1}, delta_t and the stored coefficients (Section 2.2)
// both carried in double, contractions on the FP64 matrix instruction (mma.m8n8k4.f64).
//
// Batch rows are independent, so a thread-block cluster owns up to 24 rows (one to three 8-row matrix tiles, or one tile
// and a ninth row on the plain FP64 units) and never waits for another cluster.  CTA `rank` of a cluster owns `uc` units (a multiple of 8) and the rows of W that
// belong to them.
//   forward: z = h W^T for its own units, all gates, K = all units.  Every CTA holds the whole vector h of its rows in
//     shared memory (two buffers) and sends the units it computed to all CTAs of the cluster.
//   backward: v = g * coefficients is local to the owner of a unit, so the CTA multiplies its own v (K = its units, all
//     gates) with the same rows of W and sends each other CTA that CTA's share of the partial sums; the receiver adds
//     the shares in rank order.  Neither g nor the coefficients are ever broadcast.
// The exchange uses asynchronous distributed-shared-memory stores that count bytes on the receiver's mbarrier; the
// arrival of the data is the only synchronisation between CTAs.  The input projection U x_t of a step does not depend
// on h and is accumulated while the CTA waits for the exchange.
//
// What bounds it: the FP64 rate (124 FMA per ns and SM measured, 64 per clock) plus, per step, one exchange and the
// gates' exponentials.  The matrix instruction reaches that rate with 4 warps where the FMA loop it replaces (32 x 32
// tiles, one launch per step) ran at a third of it, limited by shared-memory operands.  A small kernel
// first copies W and U into the order the lanes consume them (float, zero-padded): every load of a block is 512
// contiguous bytes per warp.  As many blocks as fit stay in shared memory for the whole sequence, the others are streamed
// from L2 into registers a few blocks ahead; read from the rows of W as they lie, eight 64-byte pieces per load, that
// streaming ran at 12 bytes per clock and SM and cost more than the products.
//
// Measured against one launch per step (128 rows, 512 units, 212 inputs, us per step): GRU forward 35.2 -> 17.5, exact
// 43.1 -> 11.8; LSTM forward 44.8 -> 21.1, exact 65.6 -> 14.8.  128 rows, 64 units, 4 inputs: GRU 12.4 -> 2.0 and 8.6 -> 1.8.
// What is left of a 512-unit GRU's forward step: 18 of 34 thousand clocks are h's products, 10 the input projection, the
// rest the exchange and the gates.
//
// Waits are bounded (2 s): a wait that gives up records HBP_ERR_TIMEOUT, the CTA leaves the loop together and still
// meets its peers at the final cluster barrier, so no CTA ends while a peer may still write into its shared memory.
#include "cell_common.cuh"

namespace hbp {

using namespace cell;

namespace {

// one 8-row tile per cluster leaves registers for up to 12 warps, so that a CTA can own up to 96 units
constexpr int max_threads(int mt, int ex) { return mt == 1 && ex == 0 ? 384 : 256; }
template <int N>
struct Const {
  static constexpr int value = N;
};
enum { CELL_RNN = 0, CELL_GRU = 1, CELL_LSTM = 2 };
template <int CELL>
struct Cell;
template <>
struct Cell<CELL_RNN> {
  static constexpr int kGates = 1, kCoef = 1;
};
template <>
struct Cell<CELL_GRU> {  // sums: r, z, W_n h, U_n x
  static constexpr int kGates = 3, kAcc = 4, kCoef = 4;
};
template <>
struct Cell<CELL_LSTM> {
  static constexpr int kGates = 4, kAcc = 4, kCoef = 5;
};

struct CellArgs {
  const void *W, *U;    // [G u][u], [G u][in]
  float4 *Wp, *Up;      // the same in blocks: forward [unit tile][k block][G][32], backward [CTA][column group][k block][4][32]
  const void* X;        // forward: [T][B][in]
  const void* x0;       // forward: [B][S]
  const void* gate;     // backward, RNN: [u] or null (ones)
  void* states;         // forward: x_all [T+1][B][S] (entry 0 is the caller's);  backward: g [T+1][B][S], g[T] given
  void* keep;           // diagonal of K per step: GRU z [T][B][u], LSTM [f | 0] [T][B][2u] (RNN: unused)
  void* coef;           // RNN tanh' [T][B][u], GRU [T B][4u], LSTM [T B][5u]
  const void* delta;    // backward: [T+1][B][S] or null
  int* status;
  int T, B, u, in;
  int rows;             // batch rows per cluster, at most 8 MT
  int uc;               // units per CTA
  int ksplit;           // forward: warps that share one 8-unit tile's contraction
  int res, res_x;       // blocks of W (U) per warp that stay in shared memory
  int kc, padding;      // backward: blocks of 16 of a CTA's own contraction, blocks of zeros among them
  int stage_x;          // forward: the inputs of a step are copied to shared memory one step ahead
};

// e^x for x <= 0 (or NaN), below -708 the value there, 3.3e-308 (zero in float): x = k ln 2 + r with |r| <= ln 2 / 2 and
// the Taylor polynomial of degree 13 in r (remainder 4e-18), evaluated pairwise: within one unit in the last place.  Without
// branches, so that the gates of the two units a thread owns run interleaved: with exp() and the division operator a GRU's
// step spent 2870 clocks here.
__device__ __forceinline__ double exp_nonpos(double x) {
  x = x < -708.0 ? -708.0 : x;
  constexpr double kRound = 6755399441055744.0;  // 1.5 * 2^52: adding it leaves the nearest integer in the low word
  double kf = fma(x, 1.4426950408889634, kRound);
  const int k = __double2loint(kf);
  kf -= kRound;
  double r = fma(kf, -0.69314718055994531, x);
  r = fma(kf, -2.3190468138462996e-17, r);
  const double r2 = r * r, r4 = r2 * r2, r8 = r4 * r4;
  const double a1 = fma(r, 1.0 / 6.0, 0.5), a2 = fma(r, 1.0 / 120.0, 1.0 / 24.0), a3 = fma(r, 1.0 / 5040.0, 1.0 / 720.0);
  const double a4 = fma(r, 1.0 / 362880.0, 1.0 / 40320.0), a5 = fma(r, 1.0 / 39916800.0, 1.0 / 3628800.0);
  const double a6 = fma(r, 1.0 / 6227020800.0, 1.0 / 479001600.0);
  const double b1 = fma(r2, a2, a1), b2 = fma(r2, a4, a3), b3 = fma(r2, a6, a5);
  const double p = 1.0 + fma(r2, fma(r8, b3, fma(r4, b2, b1)), r);
  return p * __hiloint2double((1023 + k) << 20, 0);
}
// 1 / d for d in [1, 2], within one unit in the last place, by Newton's iteration from the hardware's estimate
__device__ __forceinline__ double recip(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}
// sigmoid(v) and 1 - sigmoid(v) from one exponential and one reciprocal, neither by cancellation
__device__ __forceinline__ void sigmoid_pair(double v, double& s, double& s1) {
  const double e = exp_nonpos(-fabs(v)), big = recip(1.0 + e), small = e * big;
  s = v >= 0.0 ? big : small;
  s1 = v >= 0.0 ? small : big;
}
// tanh(v) and 1 - tanh(v)^2 = 4e / (1 + e)^2 with e = exp(-2|v|)
__device__ __forceinline__ void tanh_pair(double v, double& t, double& s) {
  const double e = exp_nonpos(-2.0 * fabs(v)), q = recip(1.0 + e);
  t = copysign((1.0 - e) * q, v);
  s = 4.0 * e * q * q;
}

// The warps that share a tile's contraction take its blocks in turn: warp ks takes blocks ks, ks + ks_n, ...  How many those
// are: none for a warp beyond the last block (few inputs have one block of U for up to eight warps).
__host__ __device__ constexpr int block_share(int blocks, int ks, int ks_n) { return ks < blocks ? (blocks - ks + ks_n - 1) / ks_n : 0; }
// Where its share starts.  A warp without one reads the last block, and uses nothing of it: a branch around its loads costs the
// others 3 % of a step (GRU, 512 units, 212 inputs: 5975 -> 6137 us for 256 steps and the backward pass).
__host__ __device__ constexpr int first_block(int blocks, int ks) { return ks < blocks ? ks : blocks - 1; }
// Which block of a share of n, with `res` of them resident, ring slot s starts with (the last one again past the end).
__host__ __device__ constexpr int ahead_block(int res, int s, int n) { return res + s < n ? res + s : (n > 0 ? n - 1 : 0); }

// ------------------------------------------------------------------------------------------------ forward
// The contraction index runs in blocks of 16 units; within a block lane c = l % 4 holds units 4c .. 4c + 3, one per
// matrix instruction, so that a lane's share of W is one 16-byte load and its share of h two.  Outputs are finished one
// unit per thread (FP64 latency is about 20 clocks per operation: more threads, not more work per thread, hide it).
template <typename T, int CELL, int MT, int EX>
__global__ void __launch_bounds__(max_threads(MT, EX), 1) cell_forward_kernel(const CellArgs p) {
  constexpr int G = Cell<CELL>::kGates, GA = Cell<CELL>::kAcc;
  constexpr int kChains = MT * G < 4 ? 2 : 1;  // independent sums per output, so that few tiles still fill the pipe
  // streamed blocks in flight per warp, as many as the registers hold
  constexpr int kAhead = MT == 3 || (MT == 1 && EX == 0 && G == 4) ? 2 : (EX ? 4 : 3);
  const int kThreads = (int)blockDim.x, R = p.rows;
  const int u = p.u, in = p.in, uc = p.uc, ntu = uc / 8, ks_n = p.ksplit;
  const int cs = (int)cluster_size(), rank = (int)tc::cluster_ctarank();
  const int kbh = (cs * uc + 15) / 16, kbx = (in + 15) / 16;
  const int S = CELL == CELL_LSTM ? 2 * u : u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lr = lane >> 2, lc = lane & 3;
  const int nt = warp % ntu, ks = warp / ntu;
  const int row0 = (int)cluster_index() * R, live_rows = min(R, p.B - row0);
  const int outs = (8 * MT + EX) * uc;  // outputs of this CTA, rows beyond R among them
  constexpr int kOuts = 2 * MT + EX;    // outputs a thread may own (there are at least 4 threads per unit)

  extern __shared__ __align__(16) unsigned char cell_smem[];
  const uint32_t tile_bytes = (uint32_t)kbh * MT * 1024u, buf_bytes = tile_bytes + (uint32_t)kbh * EX * 128u;
  const uint32_t x_bytes = p.stage_x ? (uint32_t)R * in * (uint32_t)sizeof(T) : 0u;
  unsigned char* xs = cell_smem + 2 * buf_bytes;                                      // inputs of two steps
  double* red = reinterpret_cast<double*>(xs + ((2 * x_bytes + 15u) & ~15u));         // [ks][GA][outs]
  double* cst = red + ks_n * GA * outs;                                               // LSTM cell state [outs]
  float4* wres = reinterpret_cast<float4*>(cst + (CELL == CELL_LSTM ? outs : 0));     // [warp][res][G][32]
  float4* ures = wres + ntu * ks_n * p.res * G * 32;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ures + ntu * ks_n * p.res_x * G * 32); // h x 2, inputs x 2
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 4);
  const uint32_t vbuf = tc::smem_u32(cell_smem), bar0 = tc::smem_u32(bars), xbar0 = bar0 + 16;

  const float4* gW = p.Wp + ((rank * ntu + nt) * kbh + first_block(kbh, ks)) * G * 32 + lane;
  const float4* gU = p.Up + ((rank * ntu + nt) * kbx + first_block(kbx, ks)) * G * 32 + lane;
  auto load_rows = [&](const float4* M, int j, float4* b) {  // block ks + j ks_n
#pragma unroll
    for (int g = 0; g < G; ++g) b[g] = __ldg(M + (j * ks_n * G + g) * 32);
  };
  const int jh = block_share(kbh, ks, ks_n), jx = block_share(kbx, ks, ks_n);
  const int res = min(p.res, jh), res_x = min(p.res_x, jx);
  const float4* my_w = wres + warp * p.res * G * 32 + lane;
  const float4* my_u = ures + warp * p.res_x * G * 32 + lane;

  auto fetch_x = [&](int t) {  // one thread: the rows of a step are one contiguous block
    fetch_rows(tc::smem_u32(xs) + (t & 1) * x_bytes, (const T*)p.X + ((int64_t)t * p.B + row0) * in,
               (uint32_t)live_rows * in * (uint32_t)sizeof(T), xbar0 + 8 * (t & 1));
  };
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) tc::mbar_init(bar0 + 8 * i, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (p.stage_x) fetch_x(0);
  }
  for (int i = tid; i < (int)(2 * buf_bytes / 16); i += kThreads) reinterpret_cast<double2*>(cell_smem)[i] = make_double2(0.0, 0.0);
  for (int j = 0; j < res; ++j) {
    float4 b[G];
    load_rows(gW, j, b);
#pragma unroll
    for (int g = 0; g < G; ++g) wres[((warp * p.res + j) * G + g) * 32 + lane] = b[g];
  }
  for (int j = 0; j < res_x; ++j) {
    float4 b[G];
    load_rows(gU, j, b);
#pragma unroll
    for (int g = 0; g < G; ++g) ures[((warp * p.res_x + j) * G + g) * 32 + lane] = b[g];
  }
  __syncthreads();
  // byte offset of (row, unit k) in a buffer: matrix-tile order, the ninth row behind the tile
  auto v_offset = [&](int row, int k) {
    if (EX && row >= 8 * MT) return tile_bytes + (uint32_t)k * 8u;
    return (uint32_t)((((k >> 4) * MT + (row >> 3)) * 2 + ((k >> 1) & 1)) * 512 + ((row & 7) * 4 + ((k >> 2) & 3)) * 16 + (k & 1) * 8);
  };
  for (int i = tid; i < live_rows * u; i += kThreads) {  // h_0 of all units, every CTA its own copy
    const int row = i / u, k = i - row * u;
    *reinterpret_cast<double*>(cell_smem + v_offset(row, k)) =
        (double)to_f(((const T*)p.x0)[(int64_t)(row0 + row) * S + (CELL == CELL_LSTM ? u : 0) + k]);
  }
  // this thread's outputs.  Outputs of a tile come in the order its lanes hold the sums: (row, units 2c, 2c + 1)
  int o_row[kOuts] = {}, o_unit[kOuts] = {};
  bool o_on[kOuts], o_live[kOuts];
#pragma unroll
  for (int it = 0; it < kOuts; ++it) {
    const int o = tid + it * kThreads;
    if (o < MT * ntu * 64) {
      const int tile = o >> 6, l = (o & 63) >> 1;
      o_row[it] = (tile / ntu) * 8 + (l >> 2);
      o_unit[it] = rank * uc + (tile % ntu) * 8 + 2 * (l & 3) + (o & 1);
    } else {
      o_row[it] = 8 * MT;
      o_unit[it] = rank * uc + o - MT * ntu * 64;
    }
    o_on[it] = o < outs && o_row[it] < R;
    o_live[it] = o_on[it] && o_unit[it] < u && o_row[it] < live_rows;
    if (CELL == CELL_LSTM && o < outs)
      cst[o] = o_live[it] ? (double)to_f(((const T*)p.x0)[(int64_t)(row0 + o_row[it]) * S + o_unit[it]]) : 0.0;
  }
  __syncthreads();
  tc::cluster_sync_whole_warps();  // every CTA of the cluster has started: barriers and buffers exist

  bool ok = true;
  for (int t = 0; t < p.T; ++t) {
    const uint32_t cur = t & 1, nxt = cur ^ 1;
    if (tid == 0 && t + 1 < p.T) {
      tc::mbar_expect_tx(bar0 + 8 * nxt, (uint32_t)(cs * uc * R * 8));
      if (p.stage_x) fetch_x(t + 1);  // (its buffer was last read two barriers ago)
    }
    double2 acc[kChains][MT][GA];
    double ex[EX ? GA : 1];
#pragma unroll
    for (int g = 0; g < GA; ++g) {
      if (EX) ex[g] = 0.0;
#pragma unroll
      for (int s = 0; s < kChains; ++s)
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[s][m][g] = make_double2(0.0, 0.0);
    }
    // U x_t: independent of the exchange
    const T* x_t = p.stage_x ? reinterpret_cast<const T*>(xs + cur * x_bytes) : (const T*)p.X + ((int64_t)t * p.B + row0) * in;
    {
      auto multiply_x = [&](int j, const float4* b) {
        const int k = (ks + j * ks_n) * 16 + 4 * lc;
        float4 a[MT], e = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int m = 0; m < MT; ++m)
          a[m] = (8 * m + lr < live_rows && k < in) ? load4(x_t + (8 * m + lr) * in + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (EX && 8 * MT < live_rows && k < in) e = load4(x_t + 8 * MT * in + k);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const double bv = (double)lane4(b[g], i);
            const int to = CELL == CELL_GRU && g == 2 ? GA - 1 : g;
#pragma unroll
            for (int m = 0; m < MT; ++m) dmma(acc[i % kChains][m][to], (double)lane4(a[m], i), bv);
            if (EX) ex[to] = fma((double)lane4(e, i), bv, ex[to]);
          }
      };
      float4 pre[kAhead][G];
#pragma unroll
      for (int s = 0; s < kAhead; ++s) load_rows(gU, ahead_block(res_x, s, jx), pre[s]);
      if (p.stage_x) ok = bar_wait_cluster(xbar0 + 8 * cur, (uint32_t)((t >> 1) & 1), abort_flag) && ok;
      for (int j = 0; j < res_x; ++j) {
        float4 b[G];
#pragma unroll
        for (int g = 0; g < G; ++g) b[g] = my_u[(j * G + g) * 32];
        multiply_x(j, b);
      }
      int j = res_x;
      for (; j + kAhead <= jx; j += kAhead) {
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
          multiply_x(j + s, pre[s]);
          load_rows(gU, min(j + s + kAhead, jx - 1), pre[s]);
        }
      }
#pragma unroll
      for (int s = 0; s < kAhead - 1; ++s)
        if (j + s < jx) multiply_x(j + s, pre[s]);
    }
    float4 pre[kAhead][G];  // the first streamed blocks of W do not depend on the exchange either
#pragma unroll
    for (int s = 0; s < kAhead; ++s) load_rows(gW, ahead_block(res, s, jh), pre[s]);
    if (t > 0) ok = bar_wait_cluster(bar0 + 8 * cur, (uint32_t)(((t - 1) >> 1) & 1), abort_flag) && ok;
    if (ok) {
      const unsigned char* vb = cell_smem + cur * buf_bytes;
      auto multiply = [&](int j, const float4* b) {
        const int kb = ks + j * ks_n;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          double2 a[MT], e = make_double2(0.0, 0.0);
#pragma unroll
          for (int m = 0; m < MT; ++m) a[m] = *reinterpret_cast<const double2*>(vb + ((kb * MT + m) * 2 + h) * 512 + lane * 16);
          if (EX) e = *reinterpret_cast<const double2*>(vb + tile_bytes + (kb * 16 + 4 * lc + 2 * h) * 8);
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int g = 0; g < G; ++g) {
              const double bv = (double)lane4(b[g], 2 * h + i);
#pragma unroll
              for (int m = 0; m < MT; ++m) dmma(acc[i % kChains][m][g], i == 0 ? a[m].x : a[m].y, bv);
              if (EX) ex[g] = fma(i == 0 ? e.x : e.y, bv, ex[g]);
            }
        }
      };
      for (int j = 0; j < res; ++j) {
        float4 b[G];
#pragma unroll
        for (int g = 0; g < G; ++g) b[g] = my_w[(j * G + g) * 32];
        multiply(j, b);
      }
      // no branches between the loads of a round: ptxas otherwise waits for all of them at the first use of one
      int j = res;
      for (; j + kAhead <= jh; j += kAhead) {
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
          multiply(j + s, pre[s]);
          load_rows(gW, min(j + s + kAhead, jh - 1), pre[s]);
        }
      }
#pragma unroll
      for (int s = 0; s < kAhead - 1; ++s)
        if (j + s < jh) multiply(j + s, pre[s]);
#pragma unroll
      for (int g = 0; g < GA; ++g) {
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          double2 v = acc[0][m][g];
          if (kChains == 2) { v.x += acc[kChains - 1][m][g].x; v.y += acc[kChains - 1][m][g].y; }
          *reinterpret_cast<double2*>(red + (ks * GA + g) * outs + ((m * ntu + nt) * 32 + lane) * 2) = v;
        }
        if (EX) {
          double v = ex[g];
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          if (lc == 0) red[(ks * GA + g) * outs + MT * ntu * 64 + nt * 8 + lr] = v;
        }
      }
    }
    if (__syncthreads_or(!ok)) {  // partial sums are in place; or the whole CTA leaves together
      ok = false;
      break;
    }
    // Outputs are finished up to three at a time: first their sums, then straight-line arithmetic, so that the chains of
    // dependent FP64 operations (about 50 long) of a thread's outputs run interleaved, then the sends.
    auto finish = [&](auto first_c, auto count_c) {
      constexpr int kFirst = decltype(first_c)::value, N = decltype(count_c)::value;
      double z[N][GA], hn[N], kept[N], cell[N], coef[N][Cell<CELL>::kCoef], hp[N], cp[N];
      uint32_t voff[N];
#pragma unroll
      for (int n = 0; n < N; ++n) {
        const int o = min(tid + (kFirst + n) * kThreads, outs - 1);
#pragma unroll
        for (int g = 0; g < GA; ++g) z[n][g] = red[g * outs + o];
        voff[n] = v_offset(o_row[kFirst + n], o_unit[kFirst + n]);
        hp[n] = o_on[kFirst + n] ? *reinterpret_cast<const double*>(cell_smem + cur * buf_bytes + voff[n]) : 0.0;
        cp[n] = CELL == CELL_LSTM ? cst[o] : 0.0;
      }
      for (int k = 1; k < ks_n; ++k)  // fixed order
#pragma unroll
        for (int n = 0; n < N; ++n)
#pragma unroll
          for (int g = 0; g < GA; ++g) z[n][g] += red[(k * GA + g) * outs + min(tid + (kFirst + n) * kThreads, outs - 1)];
#pragma unroll
      for (int n = 0; n < N; ++n) {
        kept[n] = cell[n] = 0.0;
        double* c = coef[n];
        if constexpr (CELL == CELL_GRU) {
          double r, r1, z1, nn, dn;
          sigmoid_pair(z[n][0], r, r1);
          sigmoid_pair(z[n][1], kept[n], z1);
          const double rec = z[n][2];
          tanh_pair(z[n][3] + r * rec, nn, dn);
          hn[n] = kept[n] * hp[n] + z1 * nn;
          c[3] = z1 * dn;
          c[0] = c[3] * rec * r * r1;
          c[1] = (hp[n] - nn) * kept[n] * z1;
          c[2] = c[3] * r;
        } else {
          double i, i1, f1, og, o1, g, dg, tch, dtc;
          sigmoid_pair(z[n][0], i, i1);
          sigmoid_pair(z[n][1], kept[n], f1);
          tanh_pair(z[n][2], g, dg);
          sigmoid_pair(z[n][3], og, o1);
          cell[n] = kept[n] * cp[n] + i * g;
          tanh_pair(cell[n], tch, dtc);
          hn[n] = og * tch;
          c[0] = g * i * i1;
          c[1] = cp[n] * kept[n] * f1;
          c[2] = i * dg;
          c[3] = tch * og * o1;
          c[4] = og * dtc;
        }
        if (!o_live[kFirst + n]) hn[n] = cell[n] = 0.0;
      }
      if (t + 1 < p.T) {  // nobody reads what the last step would send; the even lane of a pair sends both units
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const double other = __shfl_down_sync(0xffffffffu, hn[n], 1);
          if (o_on[kFirst + n] && !(tid & 1)) {
            const uint32_t dst = vbuf + nxt * buf_bytes + voff[n], bar = bar0 + 8 * nxt;
            for (int q = 0; q < cs; ++q) {
              const int to = rank + q < cs ? rank + q : rank + q - cs;  // each CTA starts with another peer
              send16(tc::map_to_cta(dst, to), hn[n], other, tc::map_to_cta(bar, to));
            }
          }
        }
      }
#pragma unroll
      for (int n = 0; n < N; ++n) {
        constexpr int NC = Cell<CELL>::kCoef;
        if (!o_live[kFirst + n]) continue;
        if (CELL == CELL_LSTM) cst[tid + (kFirst + n) * kThreads] = cell[n];
        const int unit = o_unit[kFirst + n];
        const int64_t at = (int64_t)t * p.B + row0 + o_row[kFirst + n];  // row of the [T B] arrays
        T* out = (T*)p.states + (at + p.B) * S + unit;
        out[CELL == CELL_LSTM ? u : 0] = from_f<T>((float)hn[n]);
        T* c = (T*)p.coef + at * NC * u + unit;
#pragma unroll
        for (int q = 0; q < NC; ++q) c[q * u] = from_f<T>((float)coef[n][q]);
        T* k = (T*)p.keep + at * S + unit;
        k[0] = from_f<T>((float)kept[n]);
        if (CELL == CELL_LSTM) {
          k[u] = from_f<T>(0.0f);
          out[0] = from_f<T>((float)cell[n]);
        }
      }
    };
    const int rounds = (outs + kThreads - 1) / kThreads;
    if (rounds == 1) finish(Const<0>{}, Const<1>{});
    else if constexpr (kOuts == 2) finish(Const<0>{}, Const<2>{});
    else if constexpr (kOuts == 3) finish(Const<0>{}, Const<3>{});
    else {
      finish(Const<0>{}, Const<2>{});
      if (rounds > 2) finish(Const<2>{}, Const<2>{});
      if constexpr (kOuts > 4)
        if (rounds > 4) finish(Const<4>{}, Const<2>{});
    }
  }
  if (!ok) after_timeout(p.status);
  tc::cluster_sync();
}

// ------------------------------------------------------------------------------------------------ backward
template <int MT>
constexpr int kAheadBackward = MT == 1 ? 4 : 2;

// Output columns run in groups of 32; within a group lane r = l / 4 holds columns 4r .. 4r + 3, one per matrix tile, so
// that a lane's share of a row of W is one 16-byte load and its results are 8 consecutive columns.
template <typename T, int CELL, int MT, int EX>
__global__ void __launch_bounds__(max_threads(MT, EX), 1) cell_backward_kernel(const CellArgs p) {
  constexpr int G = Cell<CELL>::kGates, NC = Cell<CELL>::kCoef;
  constexpr int kAhead = kAheadBackward<MT>;  // streamed blocks in flight per warp
  constexpr int kItems = MT + EX;          // pairs of units a thread may own
  const int kThreads = (int)blockDim.x, kWarps = kThreads / 32, R = p.rows;
  const int u = p.u, uc = p.uc;
  const int cs = (int)cluster_size(), rank = (int)tc::cluster_ctarank();
  const int S = CELL == CELL_LSTM ? 2 * u : u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lr = lane >> 2, lc = lane & 3;
  const int row0 = (int)cluster_index() * R;
  const int half = uc / 2, items = R * half;
  // Blocks of 16 of the own contraction.  The same number either way; as a parameter the GRU's loop is 5 % slower (512 units, 128
  // rows: 2990 -> 3152 us for 256 steps), computed the LSTM's is 4 % (3787 -> 3944).
  const int kc = CELL == CELL_LSTM ? p.kc : (G * uc + 15) / 16 + p.padding;
  const int groups = (cs * uc + 31) / 32;
  const int my_groups = groups > warp ? (groups - warp + kWarps - 1) / kWarps : 0;
  const int rb = p.res, nb = kc - rb;                     // blocks of each group that are resident; streamed

  extern __shared__ __align__(16) unsigned char cell_smem[];
  const uint32_t buf_bytes = (uint32_t)cs * items * 16u;  // partial sums from every CTA of the cluster
  double* va = reinterpret_cast<double*>(cell_smem + 2 * buf_bytes);       // own v in matrix-tile order, [kc * 4][MT][32]
  double* ve = va + kc * 4 * MT * 32;                                      // ... and of the ninth row, [kc * 16]
  const int v_elems = kc * 4 * MT * 32 + EX * kc * 16;
  float4* wres = reinterpret_cast<float4*>(va + v_elems);                  // [group][res][4][32]
  uint64_t* bars = reinterpret_cast<uint64_t*>(wres + groups * rb * 4 * 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 2);
  const uint32_t rbuf = tc::smem_u32(cell_smem), bar0 = tc::smem_u32(bars);

  const float4* gW = p.Wp + rank * groups * kc * 128 + lane;
  auto load_w = [&](int grp, int blk, float4* b) {
#pragma unroll
    for (int i = 0; i < 4; ++i) b[i] = __ldg(gW + ((grp * kc + blk) * 4 + i) * 32);
  };
  if (tid == 0) {
    tc::mbar_init(bar0, 1);
    tc::mbar_init(bar0 + 8, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < v_elems; i += kThreads) va[i] = 0.0;
  for (int grp = warp; grp < groups; grp += kWarps)
    for (int blk = 0; blk < rb; ++blk) {
      float4 b[4];
      load_w(grp, blk, b);
#pragma unroll
      for (int i = 0; i < 4; ++i) wres[((grp * rb + blk) * 4 + i) * 32 + lane] = b[i];
    }
  // this thread's pairs of units: running gradient (LSTM: of the cell state and of h)
  int i_row[kItems] = {}, i_unit[kItems] = {};
  bool i_on[kItems], i_live[kItems];
  double2 g[kItems], gc[kItems];
  float2 coef[kItems][NC];
  auto load_coef = [&](int it, int t) {
    const int64_t at = (int64_t)t * p.B + row0 + i_row[it];
#pragma unroll
    for (int q = 0; q < NC; ++q)
      if (!(CELL == CELL_GRU && q == 3)) coef[it][q] = load2((const T*)p.coef + at * NC * u + (int64_t)q * u + i_unit[it]);
  };
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int item = tid + it * kThreads;
    i_on[it] = item < items;
    i_row[it] = i_on[it] ? item / half : 0;
    i_unit[it] = rank * uc + 2 * (item - i_row[it] * half);
    i_live[it] = i_on[it] && i_unit[it] < u && row0 + i_row[it] < p.B;
    g[it] = gc[it] = make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < NC; ++q) coef[it][q] = make_float2(0.f, 0.f);
    if (i_live[it]) {
      const T* last = (const T*)p.states + ((int64_t)p.T * p.B + row0 + i_row[it]) * S + i_unit[it];
      const float2 v = load2(last + (CELL == CELL_LSTM ? u : 0));
      g[it] = make_double2((double)v.x, (double)v.y);
      if (CELL == CELL_LSTM) {
        const float2 c = load2(last);
        gc[it] = make_double2((double)c.x, (double)c.y);
      }
      load_coef(it, p.T - 1);
    }
  }
  __syncthreads();
  tc::cluster_sync_whole_warps();

  bool ok = true;
  for (int s = 0; s < p.T; ++s) {
    const int t = p.T - 1 - s;
    const uint32_t cur = s & 1;
    if (tid == 0) tc::mbar_expect_tx(bar0 + 8 * cur, buf_bytes);
    float4 pre[kAhead][4];
    int l_grp = warp, l_blk = rb;  // the next block to load; past the last one the last group's blocks again
    const int l_end = warp + (my_groups - 1) * kWarps;
    auto load_next = [&](float4* b) {
      load_w(l_grp, l_blk, b);
      const bool wrap = ++l_blk == kc;
      l_blk = wrap ? rb : l_blk;
      l_grp = wrap ? min(l_grp + kWarps, l_end) : l_grp;
    };
    if (my_groups > 0 && nb > 0) {
#pragma unroll
      for (int a = 0; a < kAhead; ++a) load_next(pre[a]);
    }
    // v_t = g_{t+1} * coefficients
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      if (!i_on[it]) continue;
      const int ul = i_unit[it] - rank * uc, row = i_row[it];
#pragma unroll
      for (int q = 0; q < G; ++q) {
        double2 b = g[it];
        if (CELL == CELL_LSTM && q < 3) {  // what reaches the cell state
          b.x = gc[it].x + g[it].x * (double)coef[it][NC - 1].x;
          b.y = gc[it].y + g[it].y * (double)coef[it][NC - 1].y;
        }
        const int kk = q * uc + ul;
        double* dst = EX && row >= 8 * MT ? ve + kk : va + (((kk >> 2) * MT + (row >> 3)) * 32 + (row & 7) * 4 + (kk & 3));
        *reinterpret_cast<double2*>(dst) = make_double2(b.x * (double)coef[it][q].x, b.y * (double)coef[it][q].y);
      }
    }
    if (__syncthreads_or(!ok)) {  // v_t is in place; or a wait of the previous step gave up and the whole CTA leaves
      ok = false;
      break;
    }
    // operands of the end of this step and the coefficients of the next one, requested before the products
    float2 add[kItems], addc[kItems], keep[kItems], ch[kItems];
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      add[it] = addc[it] = make_float2(0.f, 0.f);
      keep[it] = make_float2(1.f, 1.f);
      ch[it] = coef[it][NC - 1];
      if (!i_live[it]) continue;
      const int64_t at = (int64_t)t * p.B + row0 + i_row[it];
      if (CELL == CELL_RNN) {
        if (p.gate) keep[it] = load2((const T*)p.gate + i_unit[it]);
      } else {
        keep[it] = load2((const T*)p.keep + at * S + i_unit[it]);
      }
      if (p.delta) {
        add[it] = load2((const T*)p.delta + at * S + (CELL == CELL_LSTM ? u : 0) + i_unit[it]);
        if (CELL == CELL_LSTM) addc[it] = load2((const T*)p.delta + at * S + i_unit[it]);
      }
      if (t > 0) load_coef(it, t - 1);
      if (t > 3) {  // from HBM: four steps ahead into L2
        const int64_t far = at - (int64_t)3 * p.B;
#pragma unroll
        for (int q = 0; q < NC; ++q) prefetch_l2((const T*)p.coef + (far - p.B) * NC * u + (int64_t)q * u + i_unit[it]);
        if (CELL != CELL_RNN) prefetch_l2((const T*)p.keep + far * S + i_unit[it]);
        if (p.delta) prefetch_l2((const T*)p.delta + far * S + i_unit[it]);
        if (p.delta && CELL == CELL_LSTM) prefetch_l2((const T*)p.delta + far * S + u + i_unit[it]);
      }
    }
    double2 acc[MT][4];
    double ex[4];
    auto multiply = [&](int blk, const float4* b) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        double a[MT];
        const double e = EX ? ve[blk * 16 + 4 * i + lc] : 0.0;
#pragma unroll
        for (int m = 0; m < MT; ++m) a[m] = va[((blk * 4 + i) * MT + m) * 32 + lane];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const double bv = (double)lane4(b[i], n);
#pragma unroll
          for (int m = 0; m < MT; ++m) dmma(acc[m][n], a[m], bv);
          if (EX) ex[n] = fma(e, bv, ex[n]);
        }
      }
    };
    const uint32_t mine = rbuf + cur * buf_bytes + (uint32_t)(rank * items) * 16u;
    for (int grp = warp; grp < groups; grp += kWarps) {
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        ex[n] = 0.0;
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[m][n] = make_double2(0.0, 0.0);
      }
      for (int blk = 0; blk < rb; ++blk) {
        float4 b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = wres[((grp * rb + blk) * 4 + i) * 32 + lane];
        multiply(blk, b);
      }
      for (int blk = rb; blk < kc; blk += kAhead) {  // (a multiple of kAhead blocks; no branches between the loads)
#pragma unroll
        for (int a = 0; a < kAhead; ++a) {
          multiply(blk + a, pre[a]);
          load_next(pre[a]);
        }
      }
      // hand the group's sums to the owners of its units: columns n .. n + 7 are this lane's
      const int n = grp * 32 + 8 * lc, to = n / uc, ul = n - to * uc;
      if (to < cs) {
        const uint32_t bar = tc::map_to_cta(bar0 + 8 * cur, to);
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          if (m * 8 + lr >= R) break;
          const uint32_t dst = tc::map_to_cta(mine + (uint32_t)((m * 8 + lr) * half + ul / 2) * 16u, to);
          send16(dst, acc[m][0].x, acc[m][1].x, bar);
          send16(dst + 16, acc[m][2].x, acc[m][3].x, bar);
          send16(dst + 32, acc[m][0].y, acc[m][1].y, bar);
          send16(dst + 48, acc[m][2].y, acc[m][3].y, bar);
        }
      }
      if (EX) {  // the ninth row: this lane holds a quarter of the sums of columns 4 lr .. 4 lr + 3
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          ex[q] += __shfl_xor_sync(0xffffffffu, ex[q], 1);
          ex[q] += __shfl_xor_sync(0xffffffffu, ex[q], 2);
        }
        const int ne = grp * 32 + 4 * lr, toe = ne / uc, ule = ne - toe * uc;
        if (lc == 0 && toe < cs && 8 * MT < R) {
          const uint32_t bar = tc::map_to_cta(bar0 + 8 * cur, toe);
          const uint32_t dst = tc::map_to_cta(mine + (uint32_t)(8 * MT * half + ule / 2) * 16u, toe);
          send16(dst, ex[0], ex[1], bar);
          send16(dst + 16, ex[2], ex[3], bar);
        }
      }
    }
    __syncthreads();  // v_t has been read: the next step's may be written once its sums are here
    ok = bar_wait_cluster(bar0 + 8 * cur, (uint32_t)((s >> 1) & 1), abort_flag);
    if (ok) {
#pragma unroll
      for (int it = 0; it < kItems; ++it) {
        if (!i_on[it]) continue;
        if (!i_live[it]) continue;  // padding units stay at zero: their sums may be an infinity times zero weights
        const double2* r = reinterpret_cast<const double2*>(cell_smem + cur * buf_bytes) + tid + it * kThreads;
        double2 sum = r[0];
        for (int q = 1; q < cs; ++q) {  // rank order: the same bits every run
          const double2 v = r[q * items];
          sum.x += v.x;
          sum.y += v.y;
        }
        if (CELL == CELL_LSTM) {
          gc[it].x = (double)addc[it].x + (double)keep[it].x * (gc[it].x + g[it].x * (double)ch[it].x);
          gc[it].y = (double)addc[it].y + (double)keep[it].y * (gc[it].y + g[it].y * (double)ch[it].y);
          g[it].x = (double)add[it].x + sum.x;
          g[it].y = (double)add[it].y + sum.y;
        } else {
          g[it].x = (double)add[it].x + (double)keep[it].x * g[it].x + sum.x;
          g[it].y = (double)add[it].y + (double)keep[it].y * g[it].y + sum.y;
        }
        if (i_live[it]) {
          T* out = (T*)p.states + ((int64_t)t * p.B + row0 + i_row[it]) * S + i_unit[it];
          if (CELL == CELL_LSTM) {
            store2(out, gc[it].x, gc[it].y);
            store2(out + u, g[it].x, g[it].y);
          } else {
            store2(out, g[it].x, g[it].y);
          }
        }
      }
    }
  }
  if (__syncthreads_or(!ok)) after_timeout(p.status);
  tc::cluster_sync_whole_warps();
}

// the functions of the gates on their own: out[i] = {e^-|v|, 1 / (1 + e^-|v|), sigmoid(v), 1 - sigmoid(v), tanh(v), 1 - tanh(v)^2}
__global__ void __launch_bounds__(256) gate_math_kernel(const double* __restrict__ v, double* __restrict__ out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  double* o = out + 6 * i;
  o[0] = exp_nonpos(-fabs(v[i]));
  o[1] = recip(1.0 + o[0]);
  sigmoid_pair(v[i], o[2], o[3]);
  tanh_pair(v[i], o[4], o[5]);
}

// ------------------------------------------------------------------------------------------------ weights in blocks
// forward: element (lane, i) of block (unit tile, k block, gate) is M[gate u + 8 tile + lane / 4][16 block + 4 (lane % 4) + i]
template <typename T>
__global__ void __launch_bounds__(256) pack_forward_kernel(const T* __restrict__ M, float4* __restrict__ out, int u, int width, int gates,
                                                           int kb, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int lane = i & 31, g = (i >> 5) % gates, b = (i >> 5) / gates % kb, tile = (i >> 5) / gates / kb;
  const int unit = tile * 8 + (lane >> 2), k = b * 16 + 4 * (lane & 3);
  out[i] = (unit < u && k < width) ? load4(M + (g * u + unit) * width + k) : make_float4(0.f, 0.f, 0.f, 0.f);
}
// backward: element (lane, j) of (CTA, column group, k block, i) is row kk = 16 block + 4 i + lane % 4 of the CTA's
// [gates][uc] rows of W, column 32 group + 4 (lane / 4) + j
template <typename T>
__global__ void __launch_bounds__(256) pack_backward_kernel(const T* __restrict__ W, float4* __restrict__ out, int u, int gates, int uc,
                                                            int kc, int groups, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int lane = i & 31, q4 = (i >> 5) & 3, b = (i >> 7) % kc, grp = (i >> 7) / kc % groups, rank = (i >> 7) / kc / groups;
  const int kk = b * 16 + 4 * q4 + (lane & 3), q = kk / uc, unit = rank * uc + kk - q * uc, col = grp * 32 + 4 * (lane >> 2);
  out[i] = (q < gates && unit < u && col < u) ? load4(W + (q * u + unit) * u + col) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// ------------------------------------------------------------------------------------------------ host
struct Packed {
  int w, x;  // float4 values of W (and U)
};
Packed packed_size(bool bwd, int gates, int u, int in, int uc, int kc) {  // (kc: backward only)
  const int cs = (u + uc - 1) / uc;
  if (bwd) return {cs * ((cs * uc + 31) / 32) * kc * 128, 0};
  return {cs * (uc / 8) * ((cs * uc + 15) / 16) * gates * 32, cs * (uc / 8) * ((in + 15) / 16) * gates * 32};
}

struct Plan {
  int uc = 0, cs = 0, mt = 0, ex = 0, rows = 0, ksplit = 1, threads = 0, res = 0, res_x = 0, stage_x = 0, kc = 0;
  size_t smem = 0;
};

constexpr size_t v_block_bytes(int mt, int ex) { return mt * 1024 + ex * 128; }  // a block of 16 of the backward contraction's v

size_t smem_without_weights(int cell, bool bwd, int uc, int cs, int mt, int ex, int rows, int ksplit, size_t x_bytes) {
  const int gates = cell == CELL_RNN ? 1 : (cell == CELL_GRU ? 3 : 4), acc = 4;  // (the tanh cell: backward only)
  if (bwd) return (size_t)2 * cs * rows * (uc / 2) * 16 + (gates * uc + 15) / 16 * v_block_bytes(mt, ex) + 64;
  const size_t outs = (size_t)(8 * mt + ex) * uc, kbh = (cs * uc + 15) / 16;
  return 2 * kbh * (mt * 1024 + ex * 128) + (2 * x_bytes + 15) / 16 * 16 + (ksplit * acc + (cell == CELL_LSTM)) * outs * 8 + 64;
}

// Clocks of a step of the per-step forward kernels (gru.cu, lstm.cu) at 1.92 GHz, fitted to 400 measurements at 8 to 1536 units and
// 1 to 2304 rows (standard deviation 6 %): 32 x 32 tiles, the contraction split over two CTAs where that still leaves at most
// two per SM, the CTAs of an SM sharing its FP64 units.
double per_step_clocks(int gates, int64_t B, int u, int in) {
  const int64_t cols = (u + 31) / 32, tiles = cols * ((B + 31) / 32);
  const int split = tiles <= 148 && cols >= 8 ? 2 : 1;
  const int64_t per_sm = (tiles * split + 147) / 148;
  return 17000.0 + 6800.0 * (per_sm - 1) + gates * (u + in) * 2.0 / split * (per_sm == 1 ? 20.6 : 17.7 * per_sm);
}

// The split with the smallest estimated time of a step, in clocks per SM: matrix instructions at 16 clocks each on a
// warp's quarter of the SM (at least 60 between two that add to the same sums), the exchange (500 clocks of latency and
// 17 bytes per clock received, both measured; the input projection overlaps it in the forward pass) and the elementwise
// end of a step, times the waves that the clusters need.  `active` = clusters of a size that run at a time: 7 of 11 to 16
// CTAs, 11 of 10, 15 of 7 to 9, 22 of 6 (fewer than 148 / size: a cluster stays within one GPC), so the rows are spread
// over what runs at once before a cluster takes a second tile of rows.  128 rows of 512 units: 15 clusters of 8 CTAs with
// 9 rows each (8 clusters of 16 with 16 rows would need two waves, 6 with 24 rows compute a third more).
template <typename ActiveClusters>
bool make_plan(int cell, bool bwd, int es, int64_t B, int u, int in, ActiveClusters active, Plan* best) {
  const int gates = cell == CELL_RNN ? 1 : (cell == CELL_GRU ? 3 : 4);
  double best_cost = 0.0;
  int best_waves = 0;
  best->uc = 0;
  for (int uc = 8; uc <= 96; uc += 8) {
    const int cs = (u + uc - 1) / uc, ntu = uc / 8;
    if (cs > kMaxCluster || uc >= u + 8) continue;
    for (int form = 0; form < 4; ++form) {  // one tile of rows, one and a ninth row, two, three
      const int mt = form < 2 ? 1 : form, ex = form == 1;
      const int at_once = active(mt, ex, cs), max_rows = 8 * mt + ex;
      if (at_once <= 0 || (uc > 64 && form > 0)) continue;
      const int64_t spread = (B + at_once - 1) / at_once;
      Plan q;
      q.uc = uc; q.cs = cs; q.mt = mt; q.ex = ex;
      q.rows = (int)(spread < max_rows ? spread : max_rows);
      if (q.rows <= max_rows - (ex ? 1 : 8)) continue;
      const int waves = (int)(((B + q.rows - 1) / q.rows + at_once - 1) / at_once);
      const int kbh = (cs * uc + 15) / 16, kbx = (in + 15) / 16;
      const int kc = (gates * uc + 15) / 16, groups = (cs * uc + 31) / 32;
      const int max_warps = max_threads(mt, ex) / 32;
      const double tile_clocks = 16.0 * mt + 2.0 * ex;  // 8 columns, 4 of the contraction
      int first = bwd ? 1 : max_warps / ntu;
      if (first > kbh) first = kbh;
      if (first > 8) first = 8;
      for (q.ksplit = first; q.ksplit >= 1; --q.ksplit) {
        // backward: a thread per pair of units and tile of rows, and 8 or 12 warps for the columns
        const int warps = bwd ? (uc > 64 || (groups > 8 && groups <= max_warps) ? max_warps : 8) : ntu * q.ksplit;
        if (!bwd && warps < 4 && ntu * first >= 4) continue;
        q.threads = 32 * warps;
        const size_t x_bytes = (size_t)q.rows * in * es;
        q.stage_x = !bwd && smem_without_weights(cell, bwd, uc, cs, mt, ex, q.rows, q.ksplit, x_bytes) <= (size_t)kSmemLimit;
        const size_t base = smem_without_weights(cell, bwd, uc, cs, mt, ex, q.rows, q.ksplit, q.stage_x ? x_bytes : 0);
        if (base > (size_t)kSmemLimit) continue;
        const double exchange = exchange_clocks(cs, q.rows, uc);
        double cost;
        if (bwd) {
          cost = (double)kc * 16 * tile_clocks * ((groups + 3) / 4) + exchange;
        } else {
          const int chains = gates * mt * (mt * gates < 4 ? 2 : 1) * ((warps + 3) / 4);  // sums in flight per quarter
          const double block = 4.0 * gates * tile_clocks * ((warps + 3) / 4) * (chains < 4 ? 4.0 / chains : 1.0) + 30.0;
          const double x_part = block * ((kbx + q.ksplit - 1) / q.ksplit) * (q.stage_x ? 1.0 : 2.0);
          cost = block * ((kbh + q.ksplit - 1) / q.ksplit) + (x_part > exchange ? x_part : exchange) + 60.0 * q.ksplit;
        }
        cost = (cost + 800.0 + 100.0 * mt) * waves;
        if (best->uc && cost >= best_cost) continue;
        // what is left of the shared memory holds blocks of W, then of U
        size_t left = (size_t)kSmemLimit - base;
        if (bwd) {
          // as many blocks of every column group as fit, the streamed rest a multiple of the blocks in flight: with blocks
          // of zeros behind it where not even the remainder fits
          const int ahead = mt == 1 ? kAheadBackward<1> : kAheadBackward<2>;
          const size_t block = (size_t)groups * 2048;
          q.res = (int)(left / block < (size_t)kc ? left / block : (size_t)kc);
          q.res = kc - (kc - q.res + ahead - 1) / ahead * ahead;
          const int padding = q.res < 0 ? -q.res : 0;
          if (padding * v_block_bytes(mt, ex) > left) continue;
          q.res += padding;
          q.kc = kc + padding;
          q.smem = base + padding * v_block_bytes(mt, ex) + q.res * block;
        } else {
          const size_t block = (size_t)warps * gates * 512;
          const int jh = (kbh + q.ksplit - 1) / q.ksplit, jx = (kbx + q.ksplit - 1) / q.ksplit;
          q.res = (int)(left / block < (size_t)jh ? left / block : (size_t)jh);
          left -= q.res * block;
          q.res_x = (int)(left / block < (size_t)jx ? left / block : (size_t)jx);
          q.smem = base + (q.res + q.res_x) * block;
        }
        *best = q;
        best_cost = cost;
        best_waves = waves;
      }
    }
  }
  // The estimate ranks splits; against another kernel it is short of 4100 clocks and 3.3 per unit a wave, 6100 more with a ninth
  // row and 3600 per further tile of rows (the same measurements, 6 %; weights streamed from L2 add nothing).  One launch per
  // step is the faster forward pass where the last wave of 7 clusters is nearly empty and the per-step tiles just fill the
  // chip: 1056 to 1184 units with 57 to 64 or 113 to 128 rows (GRU, 1152 units: 70 us a step against 56 with 64 rows, 101 against
  // 90 with 128), LSTM, 512 units, 288 rows (67 against 62).  Elsewhere one launch is up to 6 times as fast, and exact
  // backpropagation 1.3 to 10 times at all sizes.
  if (!bwd && best->uc) {
    const double one = 1.04 * best_cost + best_waves * (4100.0 + 3.3 * u + 6100.0 * best->ex + 3600.0 * (best->mt - 1));
    if (per_step_clocks(gates, B, u, in) < 0.95 * one) best->uc = 0;
  }
  return best->uc != 0;
}

// One past the last 16-byte word of the packed weights (W, then U) that any lane reads under a plan, by the kernels' own
// index arithmetic: the last warps of the last CTA reach furthest.
int64_t packed_words_read(bool bwd, int gates, int in, const Plan& q) {
  if (bwd) return packed_size(true, gates, q.cs * q.uc, in, q.uc, q.kc).w;  // group < groups, block < kc by construction
  const int kbh = (q.cs * q.uc + 15) / 16, kbx = (in + 15) / 16;
  const int64_t tiles = (int64_t)q.cs * q.uc / 8, n_w = tiles * kbh * gates * 32;
  int64_t end = 0;
  for (int ks = 0; ks < q.ksplit; ++ks) {
    const int jh = block_share(kbh, ks, q.ksplit), jx = block_share(kbx, ks, q.ksplit);
    const int64_t w = ((tiles - 1) * kbh + first_block(kbh, ks)) * gates * 32, x = n_w + ((tiles - 1) * kbx + first_block(kbx, ks)) * gates * 32;
    auto reach = [&](int64_t base, int j) {
      const int64_t e = base + ((int64_t)j * q.ksplit * gates + gates) * 32;
      if (e > end) end = e;
    };
    for (int j = 0; j < jh; ++j) reach(w, j);
    for (int j = 0; j < jx; ++j) reach(x, j);
    for (int s = 0; s < 4; ++s) {
      reach(w, ahead_block(q.res, s, jh));
      reach(x, ahead_block(q.res_x, s, jx));
    }
  }
  return end;
}

template <typename T, int CELL, bool BWD, int MT, int EX>
constexpr auto cell_kernel() {
  if constexpr (BWD) return cell_backward_kernel<T, CELL, MT, EX>;
  else return cell_forward_kernel<T, CELL, MT, EX>;
}
template <typename T, int CELL, bool BWD, int MT, int EX>
int active_cells(int cs) {
  return active_clusters<cell_kernel<T, CELL, BWD, MT, EX>()>(cs, max_threads(MT, EX));
}

template <typename T, int CELL, bool BWD>
bool run_cell(Launcher& lc, CellArgs a) {
  auto active = [](int mt, int ex, int cs) {
    return ex        ? active_cells<T, CELL, BWD, 1, 1>(cs)
           : mt == 1 ? active_cells<T, CELL, BWD, 1, 0>(cs)
           : mt == 2 ? active_cells<T, CELL, BWD, 2, 0>(cs)
                     : active_cells<T, CELL, BWD, 3, 0>(cs);
  };
  Plan q;
  if (!make_plan(CELL, BWD, (int)sizeof(T), a.B, a.u, a.in, active, &q)) return false;
  const Packed n = packed_size(BWD, Cell<CELL>::kGates, a.u, a.in, q.uc, q.kc);
  a.Up = a.Wp + n.w;
  if (BWD) {
    const int groups = (q.cs * q.uc + 31) / 32;
    pack_backward_kernel<T><<<(n.w + 255) / 256, 256, 0, lc.stream>>>((const T*)a.W, a.Wp, a.u, Cell<CELL>::kGates, q.uc, q.kc, groups, n.w);
    lc.count();
  } else {
    pack_forward_kernel<T><<<(n.w + 255) / 256, 256, 0, lc.stream>>>((const T*)a.W, a.Wp, a.u, a.u, Cell<CELL>::kGates, (q.cs * q.uc + 15) / 16, n.w);
    pack_forward_kernel<T><<<(n.x + 255) / 256, 256, 0, lc.stream>>>((const T*)a.U, a.Up, a.u, a.in, Cell<CELL>::kGates, (a.in + 15) / 16, n.x);
    lc.count(2);
  }
  lc.check();
  a.rows = q.rows; a.uc = q.uc; a.ksplit = q.ksplit; a.res = q.res; a.res_x = q.res_x; a.stage_x = q.stage_x; a.kc = q.kc; a.padding = q.kc - (Cell<CELL>::kGates * q.uc + 15) / 16;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  launch_config(cfg, attr, (a.B + q.rows - 1) / q.rows, q.cs, q.threads, q.smem, lc.stream);
  cudaError_t e = q.ex        ? cudaLaunchKernelEx(&cfg, cell_kernel<T, CELL, BWD, 1, 1>(), a)
                  : q.mt == 1 ? cudaLaunchKernelEx(&cfg, cell_kernel<T, CELL, BWD, 1, 0>(), a)
                  : q.mt == 2 ? cudaLaunchKernelEx(&cfg, cell_kernel<T, CELL, BWD, 2, 0>(), a)
                              : cudaLaunchKernelEx(&cfg, cell_kernel<T, CELL, BWD, 3, 0>(), a);
  if (e != cudaSuccess) {  // clusters of this size cannot be placed here: the caller runs another form
    cudaGetLastError();
    return false;
  }
  lc.ran(HBP_FORM_CELL_CLUSTER);
  lc.count();
  lc.check();
  return true;
}

template <bool BWD>
bool dispatch_cell(Launcher& lc, int dtype, int block, const CellArgs& a) {
  const bool f32 = dtype == HBP_F32;
  if (!a.Wp) return false;
  // vector loads: four weights or inputs, two states
  for (const void* ptr : {a.W, a.U, a.X, a.gate, a.delta})
    if ((uintptr_t)ptr & 15u) return false;
  if (a.T <= 0 || a.B <= 0) return false;
  switch (block) {
    case HBP_BLOCK_RNN_TANH:  // backward only: its forward pass keeps an order of sums of its own (rnn_cluster.cu)
      if constexpr (!BWD) return false;
      else return f32 ? run_cell<float, CELL_RNN, BWD>(lc, a) : run_cell<bf16, CELL_RNN, BWD>(lc, a);
    case HBP_BLOCK_GRU: return f32 ? run_cell<float, CELL_GRU, BWD>(lc, a) : run_cell<bf16, CELL_GRU, BWD>(lc, a);
    case HBP_BLOCK_LSTM: return f32 ? run_cell<float, CELL_LSTM, BWD>(lc, a) : run_cell<bf16, CELL_LSTM, BWD>(lc, a);
  }
  return false;
}

}  // namespace

size_t cell_pack_bytes(int block, int u, int in_dim) {
  const int gates = block == HBP_BLOCK_GRU ? 3 : (block == HBP_BLOCK_LSTM ? 4 : 1);
  size_t most = 0;
  for (int uc = 8; uc <= 96; uc += 8) {
    if ((u + uc - 1) / uc > kMaxCluster) continue;
    const int kc = (gates * uc + 15) / 16 + 3;  // with the most padding a plan adds (fewer blocks than are in flight)
    const Packed f = packed_size(false, gates, u, in_dim, uc, 0), b = packed_size(true, gates, u, in_dim, uc, kc);
    const size_t n = (size_t)(f.w + f.x > b.w ? f.w + f.x : b.w) * sizeof(float4);
    if (n > most) most = n;
  }
  return most;
}

bool cell_plan(int block, int dtype, bool backward, int64_t B, int u, int in_dim, const int32_t* at_once, int64_t* out) {
  const int cell = block == HBP_BLOCK_GRU ? CELL_GRU : (block == HBP_BLOCK_LSTM ? CELL_LSTM : CELL_RNN);
  const int gates = cell == CELL_RNN ? 1 : (cell == CELL_GRU ? 3 : 4), in = backward ? 0 : in_dim;
  Plan q;
  if (!make_plan(cell, backward, dtype == HBP_F32 ? 4 : 2, B, u, in, [&](int, int, int cs) { return (int)at_once[cs]; }, &q)) return false;
  const Packed n = packed_size(backward, gates, u, in, q.uc, q.kc);
  const int64_t v[8] = {q.uc, q.cs, q.rows, q.ksplit, q.threads, (int64_t)q.smem, (int64_t)n.w + n.x, packed_words_read(backward, gates, in, q)};
  for (int i = 0; i < 8; ++i) out[i] = v[i];
  return true;
}

void cell_gate_math(Launcher& lc, const double* v, double* out, int64_t n) {
  gate_math_kernel<<<(unsigned)((n + 255) / 256), 256, 0, lc.stream>>>(v, out, n);
  lc.count();
  lc.check();
}

bool cell_forward_cluster(Launcher& lc, int dtype, int block, const void* W, const void* U, const void* X, const void* x0,
                          void* x_all, void* keep, void* coef, int T, int B, int u, int in_dim, void* pack, int* status) {
  CellArgs a = {};
  a.Wp = (float4*)pack;
  a.W = W; a.U = U; a.X = X; a.x0 = x0; a.states = x_all; a.keep = keep; a.coef = coef; a.status = status;
  a.T = T; a.B = B; a.u = u; a.in = in_dim;
  return dispatch_cell<false>(lc, dtype, block, a);
}

bool cell_backward_cluster(Launcher& lc, int dtype, int block, const void* W, const void* gate, const void* keep, const void* coef,
                           const void* delta, void* g_all, int T, int B, int u, void* pack, int* status) {
  CellArgs a = {};
  a.Wp = (float4*)pack;
  a.W = W; a.gate = gate; a.keep = const_cast<void*>(keep); a.coef = const_cast<void*>(coef); a.delta = delta; a.states = g_all;
  a.status = status;
  a.T = T; a.B = B; a.u = u; a.in = 0;
  return dispatch_cell<true>(lc, dtype, block, a);
}

}  // namespace hbp
