// Reverse diagonal scan over depth or time (Eq. 9 / Eq. 12 with diagonal K) and the row-wise
// elementwise kernels around it.  All access is 128-bit and coalesced along the channel axis; the
// running value is kept in float and rounded only when stored.
#include "float_parts.cuh"
#include "hbp_internal.h"
#include "split_transposed.cuh"

namespace hbp {

namespace {

template <typename T>
struct Vec;  // 16-byte vector of T
template <>
struct Vec<float> {
  static constexpr int N = 4;
  float4 raw;
  template <typename F>
  __device__ __forceinline__ void get(F* f) const { f[0] = raw.x; f[1] = raw.y; f[2] = raw.z; f[3] = raw.w; }
  template <typename F>
  __device__ __forceinline__ void set(const F* f) { raw = make_float4((float)f[0], (float)f[1], (float)f[2], (float)f[3]); }
};
template <>
struct Vec<bf16> {
  static constexpr int N = 8;
  uint4 raw;
  template <typename F>
  __device__ __forceinline__ void get(F* f) const {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 t = __bfloat1622float2(p[i]);
      f[2 * i] = t.x;
      f[2 * i + 1] = t.y;
    }
  }
  template <typename F>
  __device__ __forceinline__ void set(const F* f) {
    __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = __floats2bfloat162_rn((float)f[2 * i], (float)f[2 * i + 1]);
  }
};

// The running value of the recurrence: double for float data (thousands of steps must stay within 1e-5 of
// an exact evaluation), float for bf16 data.
template <typename T>
struct Acc {
  typedef float type;
};
template <>
struct Acc<float> {
  typedef double type;
};

template <typename T>
__device__ __forceinline__ Vec<T> ldv(const T* p) {
  Vec<T> v;
  v.raw = *reinterpret_cast<const decltype(v.raw)*>(p);
  return v;
}
template <typename T>
__device__ __forceinline__ Vec<T> ldv_stream(const T* p) {  // read-once data: evict first
  Vec<T> v;
  v.raw = __ldcs(reinterpret_cast<const decltype(v.raw)*>(p));
  return v;
}
template <typename T>
__device__ __forceinline__ void stv(T* p, const Vec<T>& v) {
  *reinterpret_cast<decltype(v.raw)*>(p) = v.raw;
}

// delta pointer for state l (nullptr = zero)
template <typename T>
__device__ __forceinline__ const T* delta_at(const ScanArgs& s, int l, int64_t state_elems) {
  if (!s.delta) return nullptr;
  if (s.loss == HBP_LOSS_EVERY_STEP) return (s.u_has_delta && l < s.L) ? nullptr : (const T*)s.delta + (int64_t)l * state_elems;
  return (l == s.L) ? (const T*)s.delta : nullptr;
}
// gate vector of step l for the 16-byte group at element `off` of the state, channel `ch` (nullptr = ones)
template <typename T>
__device__ __forceinline__ const T* gate_at(const ScanArgs& s, int l, int64_t state_elems, int64_t off, int ch) {
  if (s.gate == HBP_GATE_ONE || s.gate == kGateRow || !s.a) return nullptr;
  if (s.gate == kGateElement) return (const T*)s.a + (int64_t)l * state_elems + off;
  return (const T*)s.a + (s.gate == HBP_GATE_CHANNEL_PER_STEP ? (int64_t)l * s.d : 0) + ch;
}

// One step of the recurrence for a 16-byte channel group: val = a * carry + u + delta.
template <typename T>
__device__ __forceinline__ void scan_step(const ScanArgs& s, int l, int64_t state_elems, int64_t off, int ch,
                                          const typename Acc<T>::type* carry, typename Acc<T>::type* val,
                                          int64_t row = 0) {
  constexpr int V = Vec<T>::N;
  const T* gp = gate_at<T>(s, l, state_elems, off, ch);
  if (s.gate == kGateRow) {  // one gate value per row and step (a float table [L][rows])
    const float a = s.keep * __ldg(s.row_gate + (int64_t)l * s.rows + row);
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] = a * carry[i];
  } else if (gp) {
    float a[V];
    ldv<T>(gp).get(a);
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] = a[i] * carry[i];
  } else {
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] = s.keep * carry[i];
  }
  if (s.u2) {
    float w[V];
    ldv_stream<T>((const T*)s.u2 + (int64_t)l * state_elems + off).get(w);
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] += w[i];
  }
  if (s.u) {
    float u[V];
    ldv_stream<T>((const T*)s.u + (int64_t)l * state_elems + off).get(u);
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] += u[i];
  }
  const T* dp = delta_at<T>(s, l, state_elems);
  if (dp) {
    float dl[V];
    ldv_stream<T>(dp + off).get(dl);
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] += dl[i];
  }
}

// ---- depth scan, no LayerNorm: one thread per 16-byte channel group, serial over l -----------------
// kShift: the shifted split (gamma > 0), which also reads the previous iterate; compiled apart so that the plain
// scan carries no registers for it
template <typename T, bool kShift>
__global__ void __launch_bounds__(256) scan_depth_kernel(const ScanArgs s) {
  constexpr int V = Vec<T>::N;
  const int64_t state_elems = s.rows * s.d;
  const int64_t nvec = state_elems / V;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nvec) return;
  const int64_t off = v * V;
  const int64_t row = off / s.d;  // once per thread: the per-row gate of post-LN layers is looked up by it
  const int ch = (int)(off - row * s.d);
  T* g = (T*)s.g;
  typedef typename Acc<T>::type A;
  A carry[V];
  ldv<T>(g + (int64_t)s.l_hi * state_elems + off).get(carry);
  float old_next[kShift ? V : 1];  // shifted split: g_{l+1} of the previous iterate
  if (kShift) {
#pragma unroll
    for (int i = 0; i < V; ++i) old_next[i] = (float)carry[i];
  }
#pragma unroll 4
  for (int l = s.l_hi - 1; l >= s.l_lo; --l) {  // unrolled: the loads of four steps in flight per thread
    A val[V];
    scan_step<T>(s, l, state_elems, off, ch, carry, val, row);
    if (kShift) {
      // the shifted part of the split acts on the previous iterate: gamma * a * g_{l+1} (a = 1 unless the gate is per row)
      const float ga = s.gate == kGateRow ? s.gamma * __ldg(s.row_gate + (int64_t)l * s.rows + row) : s.gamma;
#pragma unroll
      for (int i = 0; i < V; ++i) val[i] += ga * old_next[i];
      ldv<T>(g + (int64_t)l * state_elems + off).get(old_next);  // before it is overwritten below
    }
    Vec<T> out;
    out.set(val);
    stv<T>(g + (int64_t)l * state_elems + off, out);
#pragma unroll
    for (int i = 0; i < V; ++i) carry[i] = val[i];
  }
}

// ---- depth scan with the LayerNorm-backward finish from prepared row statistics ---------------------
// Same streaming form as above: lnstat[l][row] = {rstd, mean(dy), mean(dy * xhat)} comes from the GEMM that
// produced dy, so no reduction is needed here.  u holds dy, the VJP is rstd * (dy - m1 - xhat * m2).
template <typename T, bool kShift>
__global__ void __launch_bounds__(256) scan_depth_lnstat_kernel(const ScanArgs s) {
  chain_next();
  chain_wait();
  constexpr int V = Vec<T>::N;
  const int64_t state_elems = s.rows * s.d;
  const int64_t nvec = state_elems / V;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nvec) return;
  const int64_t off = v * V;
  const int64_t row = off / s.d;
  const int ch = (int)(off - row * s.d);
  T* g = (T*)s.g;
  float carry[V], old_next[kShift ? V : 1];
  ldv<T>(g + (int64_t)s.l_hi * state_elems + off).get(carry);
  if (kShift) {
#pragma unroll
    for (int i = 0; i < V; ++i) old_next[i] = carry[i];
  }
  // the loads of a step do not depend on the running value: unrolled, those of four steps are in flight per thread
#pragma unroll 4
  for (int l = s.l_hi - 1; l >= s.l_lo; --l) {
    float dy[V], xh[V], val[V];
    ldv_stream<T>((const T*)s.u + (int64_t)l * state_elems + off).get(dy);
    ldv_stream<T>((const T*)s.xhat + (int64_t)l * state_elems + off).get(xh);
    const float4 st = __ldg(s.lnstat + (int64_t)l * s.rows + row);
    const T* gp = gate_at<T>(s, l, state_elems, off, ch);
    if (gp) {
      float a[V];
      ldv<T>(gp).get(a);
#pragma unroll
      for (int i = 0; i < V; ++i) val[i] = a[i] * carry[i];
    } else {
#pragma unroll
      for (int i = 0; i < V; ++i) val[i] = s.keep * carry[i];
    }
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] += st.x * (dy[i] - st.y - xh[i] * st.z);
    if (kShift) {
#pragma unroll
      for (int i = 0; i < V; ++i) val[i] += s.gamma * old_next[i];
      ldv<T>(g + (int64_t)l * state_elems + off).get(old_next);
    }
    const T* dp = delta_at<T>(s, l, state_elems);
    if (dp) {
      float dl[V];
      ldv_stream<T>(dp + off).get(dl);
#pragma unroll
      for (int i = 0; i < V; ++i) val[i] += dl[i];
    }
    Vec<T> out;
    out.set(val);
    stv<T>(g + (int64_t)l * state_elems + off, out);
#pragma unroll
    for (int i = 0; i < V; ++i) carry[i] = val[i];
  }
}

// One step of it (the exact pass goes step by step), with the row statistics formed here from the GEMM's partial sums, in ln_stats_finish's
// order, while the step's operands are on their way: a launch of 2 us less in a chain of 10 a layer.
__global__ void __launch_bounds__(256) scan_one_lnstat_kernel(const ScanArgs s) {
  chain_next();
  chain_wait();
  constexpr int V = Vec<bf16>::N;
  __shared__ float4 stat[256 + 2];  // of the rows that the block's groups of channels lie in (d is a multiple of V)
  const int l = s.l_lo;
  const int64_t state_elems = s.rows * s.d, off = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V;
  const bool in = off < state_elems;
  const int64_t row = off / s.d, row0 = (int64_t)blockIdx.x * blockDim.x * V / s.d;
  const int ch = (int)(off - row * s.d);
  const int64_t at = (int64_t)l * state_elems + off;
  bf16* g = (bf16*)s.g;
  Vec<bf16> carry, dy, xh, gate, delta;
  const bf16 *gp = gate_at<bf16>(s, l, state_elems, off, ch), *dp = delta_at<bf16>(s, l, state_elems);
  if (in) {
    carry = ldv<bf16>(g + at + state_elems);
    dy = ldv_stream<bf16>((const bf16*)s.u + at);
    xh = ldv_stream<bf16>((const bf16*)s.xhat + at);
    if (gp) gate = ldv<bf16>(gp);
    if (dp) delta = ldv_stream<bf16>(dp + off);
  }
  const int64_t last = min(s.rows - 1, (((int64_t)blockIdx.x + 1) * blockDim.x * V - 1) / s.d);
  for (int r = threadIdx.x; r <= (int)(last - row0); r += blockDim.x) {
    const float2* part = s.lnpart + ((int64_t)l * s.rows + row0 + r) * s.ln_slots;
    float s1 = 0.0f, s2 = 0.0f;
#pragma unroll 8
    for (int k = 0; k < s.ln_slots; ++k) {
      const float2 t = part[k];
      s1 += t.x;
      s2 += t.y;
    }
    const float inv_d = 1.0f / (float)s.d;
    stat[r] = make_float4(s.rstd[(int64_t)l * s.rows + row0 + r], s1 * inv_d, s2 * inv_d, 0.0f);
  }
  __syncthreads();
  if (!in) return;
  const float4 st = stat[row - row0];
  float c[V], y[V], x[V], val[V], more[V];
  carry.get(c);
  dy.get(y);
  xh.get(x);
  if (gp) gate.get(more);
#pragma unroll
  for (int i = 0; i < V; ++i) val[i] = (gp ? more[i] : s.keep) * c[i];
#pragma unroll
  for (int i = 0; i < V; ++i) val[i] += st.x * (y[i] - st.y - x[i] * st.z);
  if (dp) {
    delta.get(more);
#pragma unroll
    for (int i = 0; i < V; ++i) val[i] += more[i];
  }
  Vec<bf16> out;
  out.set(val);
  stv<bf16>(g + at, out);
}

__global__ void ln_stats_finish_kernel(const float2* __restrict__ stats, int slots, const float* __restrict__ rstd,
                                       float4* __restrict__ lnstat, int64_t count, float inv_d) {
  chain_next();
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  float s1 = 0.0f, s2 = 0.0f;
  for (int k = 0; k < slots; ++k) {  // fixed order: deterministic
    const float2 t = stats[i * slots + k];
    s1 += t.x;
    s2 += t.y;
  }
  lnstat[i] = make_float4(rstd[i], s1 * inv_d, s2 * inv_d, 0.0f);
}

// ---- depth scan with the LayerNorm-backward finish: one block per row ------------------------------
// u holds dY = dL/d(LN(x)); the step's VJP is rstd * (dy - mean(dy) - xhat * mean(dy * xhat)).
template <typename T>
__global__ void __launch_bounds__(1024) scan_depth_ln_kernel(const ScanArgs s) {
  chain_next();
  chain_wait();
  constexpr int V = Vec<T>::N;
  __shared__ float red[2][32][2];
  const int64_t row = blockIdx.x;
  const int tpr = s.d / V;
  const bool active = (int)threadIdx.x < tpr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
  const int64_t state_elems = s.rows * s.d;
  const int64_t off = row * s.d + (int64_t)threadIdx.x * V;
  T* g = (T*)s.g;
  float carry[V], dy[V], xh[V], old_next[V];
#pragma unroll
  for (int i = 0; i < V; ++i) carry[i] = dy[i] = xh[i] = old_next[i] = 0.0f;
  if (active) {
    ldv<T>(g + (int64_t)s.l_hi * state_elems + off).get(carry);
    ldv<T>(g + (int64_t)s.l_hi * state_elems + off).get(old_next);
    ldv_stream<T>((const T*)s.u + (int64_t)(s.l_hi - 1) * state_elems + off).get(dy);
    ldv_stream<T>((const T*)s.xhat + (int64_t)(s.l_hi - 1) * state_elems + off).get(xh);
  }
  const float inv_d = 1.0f / (float)s.d;
  for (int l = s.l_hi - 1; l >= s.l_lo; --l) {
    float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
    for (int i = 0; i < V; ++i) {
      s1 += dy[i];
      s2 = fmaf(dy[i], xh[i], s2);
    }
    // fetch the next step's operands before waiting on the reduction
    float ndy[V], nxh[V];
#pragma unroll
    for (int i = 0; i < V; ++i) ndy[i] = nxh[i] = 0.0f;
    if (active && l > s.l_lo) {
      ldv_stream<T>((const T*)s.u + (int64_t)(l - 1) * state_elems + off).get(ndy);
      ldv_stream<T>((const T*)s.xhat + (int64_t)(l - 1) * state_elems + off).get(nxh);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    const int buf = l & 1;  // two buffers: one barrier per step is enough
    if (lane == 0) {
      red[buf][warp][0] = s1;
      red[buf][warp][1] = s2;
    }
    __syncthreads();
    float t1 = 0.0f, t2 = 0.0f;
    for (int w = 0; w < nwarps; ++w) {
      t1 += red[buf][w][0];
      t2 += red[buf][w][1];
    }
    const float m1 = t1 * inv_d, m2 = t2 * inv_d;
    const float r = s.rstd[(int64_t)l * s.rows + row];
    if (active) {
      float val[V];
      const T* gp = gate_at<T>(s, l, state_elems, off, (int)threadIdx.x * V);
      if (gp) {
        float a[V];
        ldv<T>(gp).get(a);
#pragma unroll
        for (int i = 0; i < V; ++i) val[i] = a[i] * carry[i];
      } else {
#pragma unroll
        for (int i = 0; i < V; ++i) val[i] = s.keep * carry[i];
      }
#pragma unroll
      for (int i = 0; i < V; ++i) val[i] += r * (dy[i] - m1 - xh[i] * m2);
      if (s.gamma != 0.0f) {
#pragma unroll
        for (int i = 0; i < V; ++i) val[i] += s.gamma * old_next[i];
        ldv<T>(g + (int64_t)l * state_elems + off).get(old_next);
      }
      const T* dp = delta_at<T>(s, l, state_elems);
      if (dp) {
        float dl[V];
        ldv_stream<T>(dp + off).get(dl);
#pragma unroll
        for (int i = 0; i < V; ++i) val[i] += dl[i];
      }
      Vec<T> out;
      out.set(val);
      stv<T>(g + (int64_t)l * state_elems + off, out);
#pragma unroll
      for (int i = 0; i < V; ++i) carry[i] = val[i];
    }
#pragma unroll
    for (int i = 0; i < V; ++i) {
      dy[i] = ndy[i];
      xh[i] = nxh[i];
    }
  }
}

// ---- time-chunked scan for long L and few channels (three phases) ----------------------------------
// Phase 1: per (chunk, channel group) local scan with zero carry-in -> S (value at the chunk's first
// step) and P (product of the gates over the chunk).  Phase 2: per channel, serial over the chunks:
// carry-in of chunk c = G_{c+1}, G_c = S_c + P_c * G_{c+1}.  Phase 3: local scan again with the
// carry-in, writing g.  Scratch: S (then the carry-ins) [nchunks][rows*d] and P likewise, in the
// accumulator type (double for float data).
constexpr int kChunk = 32;

template <typename T, bool kApply>
__global__ void __launch_bounds__(128) scan_chunk_kernel(const ScanArgs s, typename Acc<T>::type* __restrict__ S,
                                                         typename Acc<T>::type* __restrict__ P) {
  typedef typename Acc<T>::type A;
  constexpr int V = Vec<T>::N;
  const int64_t state_elems = s.rows * s.d;
  const int64_t nvec = state_elems / V;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nvec) return;
  const int c = blockIdx.y;
  const int lo = s.l_lo + c * kChunk, hi = min(s.l_hi, lo + kChunk);
  const int64_t off = v * V;
  const int ch = (int)(off % s.d);
  T* g = (T*)s.g;
  A carry[V], prod[V];
#pragma unroll
  for (int i = 0; i < V; ++i) {
    carry[i] = kApply ? S[(int64_t)c * state_elems + off + i] : (A)0;
    prod[i] = (A)1;
  }
  for (int l = hi - 1; l >= lo; --l) {
    A val[V];
    scan_step<T>(s, l, state_elems, off, ch, carry, val);
    if (kApply) {
      Vec<T> out;
      out.set(val);
      stv<T>(g + (int64_t)l * state_elems + off, out);
    } else {
      const T* gp = gate_at<T>(s, l, state_elems, off, ch);
      if (gp) {
        float a[V];
        ldv<T>(gp).get(a);
#pragma unroll
        for (int i = 0; i < V; ++i) prod[i] *= a[i];
      }
    }
#pragma unroll
    for (int i = 0; i < V; ++i) carry[i] = val[i];
  }
  if (!kApply) {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      S[(int64_t)c * state_elems + off + i] = carry[i];
      P[(int64_t)c * state_elems + off + i] = prod[i];
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(128) scan_carry_kernel(const ScanArgs s, typename Acc<T>::type* __restrict__ S,
                                                         const typename Acc<T>::type* __restrict__ P, int nchunks) {
  typedef typename Acc<T>::type A;
  const int64_t state_elems = s.rows * s.d;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= state_elems) return;
  A G = (A)to_f(((const T*)s.g)[(int64_t)s.l_hi * state_elems + e]);
  for (int c = nchunks - 1; c >= 0; --c) {
    const A sc = S[(int64_t)c * state_elems + e], pc = P[(int64_t)c * state_elems + e];
    S[(int64_t)c * state_elems + e] = G;  // carry-in of chunk c
    G = sc + pc * G;
  }
}

// ---- row-wise helpers ----------------------------------------------------------------------------
template <typename T>
__global__ void copy_kernel(T* __restrict__ dst, const T* __restrict__ src, int64_t nvec) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v < nvec) stv<T>(dst + v * Vec<T>::N, ldv<T>(src + v * Vec<T>::N));
}

template <typename T>
__global__ void mul_kernel(T* __restrict__ dst, const T* __restrict__ a, const T* __restrict__ b, int64_t nvec) {
  constexpr int V = Vec<T>::N;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nvec) return;
  float x[V], y[V];
  ldv_stream<T>(a + v * V).get(x);
  ldv_stream<T>(b + v * V).get(y);
#pragma unroll
  for (int i = 0; i < V; ++i) x[i] *= y[i];
  Vec<T> out;
  out.set(x);
  stv<T>(dst + v * V, out);
}

// states[s] += carry for every state s (the carry of a scan whose gates are all one, applied after the fact)
template <typename T>
__global__ void add_to_states_kernel(T* __restrict__ states, const T* __restrict__ carry, int64_t elems) {
  constexpr int V = Vec<T>::N;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v * V >= elems) return;
  T* p = states + (int64_t)blockIdx.y * elems + v * V;
  float a[V], c[V];
  ldv<T>(p).get(a);
  ldv<T>(carry + v * V).get(c);
#pragma unroll
  for (int i = 0; i < V; ++i) a[i] += c[i];
  Vec<T> out;
  out.set(a);
  stv<T>(p, out);
}

template <typename T>
__global__ void to_f32_kernel(const T* __restrict__ src, float* __restrict__ dst, int64_t n) {
  chain_next();
  chain_wait();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = to_f(src[i]);
}

// xhat = (x - mean) * rstd over the last axis, biased variance, two passes in registers.  `wpr` warps (1, 2 or 4) of a block
// of four hold a row, NV float4 per lane, so that a row's loads are all in flight at once and a row of up to 2048 needs no
// block barrier.  Bound: bytes.  8192 x 1024 float -> bf16, with the state written too (67 MB): 17.6 -> 9.4 us (one block per
// row before, without the state).  master receives the normalised values in float (post-LN layers: the float copy of the
// residual stream continues from them), state the row itself in T (the float copy is the only one kept during the pass), parts
// (float data) the output again as the next product reads it.
__device__ __forceinline__ void store4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(bf16* p, const float4& v) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}
__global__ void from_f32_kernel(const float* __restrict__ src, bf16* __restrict__ dst, int64_t nvec) {
  chain_next();
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nvec) store4(dst + 4 * i, *reinterpret_cast<const float4*>(src + 4 * i));
}

constexpr int kLnWarps = 4;
template <typename T, int NV>
__global__ void __launch_bounds__(kLnWarps * 32) layernorm_fwd_kernel(const float* __restrict__ x, T* __restrict__ xhat,
                                                                      float* __restrict__ rstd, int64_t rows, int d, float eps,
                                                                      float* __restrict__ master, T* __restrict__ state, Planes parts, int wpr) {
  chain_next();
  chain_wait();
  __shared__ float red[2][kLnWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t row = (int64_t)blockIdx.x * (kLnWarps / wpr) + warp / wpr;
  const int first = (warp % wpr) * 32 + lane, nvec = row < rows ? d / 4 : 0;
  const float* xr = x + row * d;
  float4 v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int c = first + i * wpr * 32;
    v[i] = c < nvec ? *reinterpret_cast<const float4*>(xr + 4 * c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  auto row_sum = [&](float s, int k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (wpr > 1) {
      if (lane == 0) red[k][warp] = s;
      __syncthreads();
      s = 0.0f;
      for (int w = 0; w < wpr; ++w) s += red[k][warp / wpr * wpr + w];
    }
    return s;
  };
  float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
  for (int i = 0; i < NV; ++i) s1 += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  const float mu = row_sum(s1, 0) / (float)d;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    if (first + i * wpr * 32 >= nvec) continue;
    const float a = v[i].x - mu, b = v[i].y - mu, c = v[i].z - mu, e = v[i].w - mu;
    s2 += fmaf(a, a, b * b) + fmaf(c, c, e * e);
  }
  const float r = rsqrtf(row_sum(s2, 1) / (float)d + eps);
  if (first == 0 && row < rows) rstd[row] = r;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int c = first + i * wpr * 32;
    if (c >= nvec) continue;
    const float4 o = make_float4((v[i].x - mu) * r, (v[i].y - mu) * r, (v[i].z - mu) * r, (v[i].w - mu) * r);
    store4(xhat + row * d + 4 * c, o);
    if (master) store4(master + row * d + 4 * c, o);
    if (state) store4(state + row * d + 4 * c, v[i]);
    if (sizeof(T) == 4 && parts.p) store_parts4(parts.p + row * parts.ld + 4 * c, parts.plane, o);
  }
}

// Post-LN layers: per row, t = LayerNorm-backward of g through the layer's own output xo (the normalised state):
// t = rstd (g - mean g - xo mean(g xo)), and c = t - rstd g, the part of the layer's VJP that is not the block's.
template <typename T>
__global__ void __launch_bounds__(1024) postln_prepass_kernel(const T* __restrict__ g, const T* __restrict__ xo,
                                                              const float* __restrict__ rstd, T* __restrict__ t_out,
                                                              T* __restrict__ c_out, int d) {
  constexpr int V = Vec<T>::N;
  __shared__ float red[2][32];
  const int64_t row = blockIdx.x;
  const bool active = (int)threadIdx.x * V < d;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
  const int64_t off = row * d + (int64_t)threadIdx.x * V;
  float gv[V], xv[V];
#pragma unroll
  for (int i = 0; i < V; ++i) gv[i] = xv[i] = 0.0f;
  if (active) {
    ldv<T>(g + off).get(gv);
    ldv<T>(xo + off).get(xv);
  }
  float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    s1 += gv[i];
    s2 = fmaf(gv[i], xv[i], s2);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  if (lane == 0) {
    red[0][warp] = s1;
    red[1][warp] = s2;
  }
  __syncthreads();
  float t1 = 0.0f, t2 = 0.0f;
  for (int w = 0; w < nwarps; ++w) {
    t1 += red[0][w];
    t2 += red[1][w];
  }
  if (!active) return;
  const float m1 = t1 / (float)d, m2 = t2 / (float)d, r = rstd[row];
  float tv[V], cv[V];
#pragma unroll
  for (int i = 0; i < V; ++i) {
    cv[i] = r * (-m1 - xv[i] * m2);
    tv[i] = fmaf(r, gv[i], cv[i]);
  }
  Vec<T> a, b;
  a.set(tv);
  b.set(cv);
  stv<T>(t_out + off, a);
  stv<T>(c_out + off, b);
}

// partial[b][c] = sum over the block's rows of g[r][c] * x[r][c]
template <typename T>
__global__ void __launch_bounds__(256) gate_grad_kernel(const T* __restrict__ g, const T* __restrict__ x,
                                                        int64_t rows, int d, float* __restrict__ partial) {
  constexpr int V = Vec<T>::N;
  __shared__ float red[256 * V];
  const int64_t per = (rows + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = (int64_t)blockIdx.x * per, r1 = min(rows, r0 + per);
  // 16 bytes per load; where a row has fewer of them than the block threads, several rows at a time
  const int vecs = d / V, cols = min(vecs, 256), groups = 256 / cols, group = threadIdx.x / cols, col = threadIdx.x % cols;
  for (int c0 = 0; c0 < vecs; c0 += cols) {
    const int c = (c0 + col) * V;
    float sum[V];
#pragma unroll
    for (int i = 0; i < V; ++i) sum[i] = 0.0f;
    if (group < groups && c < d) {
      // four running sums over interleaved rows: eight loads in flight per thread, fixed order
      float acc[4][V];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < V; ++i) acc[k][i] = 0.0f;
      int64_t r = r0 + group;
      for (; r + 3 * groups < r1; r += 4 * groups) {
        Vec<T> gv[4], xv[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          gv[k] = ldv_stream<T>(g + (r + k * groups) * d + c);
          xv[k] = ldv_stream<T>(x + (r + k * groups) * d + c);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float a[V], b[V];
          gv[k].get(a);
          xv[k].get(b);
#pragma unroll
          for (int i = 0; i < V; ++i) acc[k][i] = fmaf(a[i], b[i], acc[k][i]);
        }
      }
      for (; r < r1; r += groups) {
        float a[V], b[V];
        ldv_stream<T>(g + r * d + c).get(a);
        ldv_stream<T>(x + r * d + c).get(b);
#pragma unroll
        for (int i = 0; i < V; ++i) acc[0][i] = fmaf(a[i], b[i], acc[0][i]);
      }
#pragma unroll
      for (int i = 0; i < V; ++i) sum[i] = (acc[0][i] + acc[1][i]) + (acc[2][i] + acc[3][i]);
    }
#pragma unroll
    for (int i = 0; i < V; ++i) red[threadIdx.x * V + i] = sum[i];
    __syncthreads();
    if (group == 0 && c < d)
#pragma unroll
      for (int i = 0; i < V; ++i) {
        float s = sum[i];
        for (int q = 1; q < groups; ++q) s += red[(q * cols + col) * V + i];
        partial[(int64_t)blockIdx.x * d + c + i] = s;
      }
    __syncthreads();
  }
}

// v = a * b (b optional); hi = v rounded to tf32 precision, lo = the same rounding of v - hi.  hi + lo carries
// 21+ bits of v, and both are exact tf32 operands.
__global__ void split_tf32_kernel(const float4* __restrict__ a, const float4* __restrict__ b, float4* __restrict__ hi,
                                  float4* __restrict__ lo, int64_t nvec) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nvec) return;
  float4 v = a[i];
  if (b) {
    const float4 w = b[i];
    v.x *= w.x; v.y *= w.y; v.z *= w.z; v.w *= w.w;
  }
  float4 h, l;
  h.x = round_tf32(v.x); h.y = round_tf32(v.y); h.z = round_tf32(v.z); h.w = round_tf32(v.w);
  l.x = round_tf32(v.x - h.x); l.y = round_tf32(v.y - h.y); l.z = round_tf32(v.z - h.z); l.w = round_tf32(v.w - h.w);
  hi[i] = h;
  lo[i] = l;
}

// a, or a * b, with ld elements between rows
struct ProductValue {
  const float *a, *b;
  int64_t ld;
  __device__ __forceinline__ float4 operator()(int64_t r, int c) const {
    const float4 v = load4(a + r * ld + c);
    return b ? mul4(v, load4(b + r * ld + c)) : v;
  }
};
// the same where a is not 16-byte aligned (a caller's inputs or weights)
struct UnalignedValue {
  const float* a;
  int64_t ld;
  __device__ __forceinline__ float4 operator()(int64_t r, int c) const {
    const float* p = a + r * ld + c;
    return make_float4(p[0], p[1], p[2], p[3]);
  }
};

inline int row_block_threads(int d, int V) {
  int t = (d / V + 31) / 32 * 32;
  return t < 32 ? 32 : t;
}

}  // namespace

size_t scan_scratch_bytes(int dtype, int L, int64_t rows, int d) {
  const int V = dtype == HBP_F32 ? 4 : 8;
  const int64_t nvec = rows * d / V;
  if (nvec >= 148 * 512 || L < 4 * kChunk) return 0;  // enough channels (or too short) for the serial form
  const int nchunks = (L + kChunk - 1) / kChunk;
  return (size_t)2 * nchunks * rows * d * (dtype == HBP_F32 ? sizeof(double) : sizeof(float));
}

void scan_reverse(Launcher& lc, const ScanArgs& s) {
  if (s.l_hi <= s.l_lo || s.rows <= 0) return;
  const int V = s.dtype == HBP_F32 ? 4 : 8;
  const int64_t nvec = s.rows * s.d / V;
  if (s.xhat && s.lnpart) {
    launch_chained(lc, scan_one_lnstat_kernel, dim3((unsigned)((nvec + 255) / 256)), 256, 0, 1, s);
    return;
  }
  if (s.xhat && s.lnstat) {
    const unsigned grid = (unsigned)((nvec + 255) / 256);
    const bool shift = s.gamma != 0.0f;
    if (s.dtype == HBP_F32) {
      if (shift) launch_chained(lc, scan_depth_lnstat_kernel<float, true>, dim3(grid), 256, 0, 1, s);
      else launch_chained(lc, scan_depth_lnstat_kernel<float, false>, dim3(grid), 256, 0, 1, s);
    } else {
      if (shift) launch_chained(lc, scan_depth_lnstat_kernel<bf16, true>, dim3(grid), 256, 0, 1, s);
      else launch_chained(lc, scan_depth_lnstat_kernel<bf16, false>, dim3(grid), 256, 0, 1, s);
    }
    return;
  }
  if (s.xhat) {
    const int threads = row_block_threads(s.d, V);
    if (s.dtype == HBP_F32) launch_chained(lc, scan_depth_ln_kernel<float>, dim3((unsigned)s.rows), threads, 0, 1, s);
    else launch_chained(lc, scan_depth_ln_kernel<bf16>, dim3((unsigned)s.rows), threads, 0, 1, s);
    return;
  }
  const int steps = s.l_hi - s.l_lo;
  const size_t need = scan_scratch_bytes(s.dtype, steps, s.rows, s.d);
  // One serial pass in time behind a ring of TMA loads reads and writes every byte once, from 32 steps on and for any number of channels: the
  // threads of the serial depth scan wait for their own loads step by step where they are few, and reach some 80 % of the copy rate
  // where they are many.  Depth scan / ring, us: float, 64 steps of 20480 channels 60 / 17 (88 / 16 with a loss on every step), 100 of
  // 288000 98 / 50, 40 of 8 M 497 / 435, 128 of 2.4 M with a loss on every step 726 / 571; bf16, 300 of 900000 297 / 186, 64 of 8 M 369 / 349.
  // Where the depth scan would run (need == 0) the ring too adds two float streams up in double.  The three-phase form below remains
  // for what the ring does not take (a gate table per step).
  const bool depth_only = s.u2 || s.gate == kGateRow;  // forms only the serial depth scan takes
  if (!depth_only && scan_ring(lc, s, need == 0)) return;
  if (need > 0 && !depth_only && s.scratch && s.scratch_bytes >= need && s.keep == 1.0f && s.gamma == 0.0f) {
    const int nchunks = (steps + kChunk - 1) / kChunk;
    dim3 grid((unsigned)((nvec + 127) / 128), nchunks);
    const unsigned cgrid = (unsigned)((s.rows * s.d + 127) / 128);
    if (s.dtype == HBP_F32) {
      double* S = (double*)s.scratch;
      double* P = S + (int64_t)nchunks * s.rows * s.d;
      scan_chunk_kernel<float, false><<<grid, 128, 0, lc.stream>>>(s, S, P);
      scan_carry_kernel<float><<<cgrid, 128, 0, lc.stream>>>(s, S, P, nchunks);
      scan_chunk_kernel<float, true><<<grid, 128, 0, lc.stream>>>(s, S, P);
    } else {
      float* S = (float*)s.scratch;
      float* P = S + (int64_t)nchunks * s.rows * s.d;
      scan_chunk_kernel<bf16, false><<<grid, 128, 0, lc.stream>>>(s, S, P);
      scan_carry_kernel<bf16><<<cgrid, 128, 0, lc.stream>>>(s, S, P, nchunks);
      scan_chunk_kernel<bf16, true><<<grid, 128, 0, lc.stream>>>(s, S, P);
    }
    lc.count(3);
    lc.check();
    return;
  }
  const unsigned grid = (unsigned)((nvec + 255) / 256);
  const bool shift = s.gamma != 0.0f;
  if (s.dtype == HBP_F32) {
    if (shift) scan_depth_kernel<float, true><<<grid, 256, 0, lc.stream>>>(s);
    else scan_depth_kernel<float, false><<<grid, 256, 0, lc.stream>>>(s);
  } else {
    if (shift) scan_depth_kernel<bf16, true><<<grid, 256, 0, lc.stream>>>(s);
    else scan_depth_kernel<bf16, false><<<grid, 256, 0, lc.stream>>>(s);
  }
  lc.count();
  lc.check();
}

void ln_stats_finish(Launcher& lc, const float2* stats, int slots, const float* rstd, float4* lnstat, int64_t count,
                     int d) {
  launch_chained(lc, ln_stats_finish_kernel, dim3((unsigned)((count + 255) / 256)), 256, 0, 1, stats, slots, rstd, lnstat, count, 1.0f / (float)d);
}

void copy_state(Launcher& lc, int dtype, void* dst, const void* src, int64_t elems) {
  if (dtype == HBP_F32)
    copy_kernel<float><<<(unsigned)((elems / 4 + 255) / 256), 256, 0, lc.stream>>>((float*)dst, (const float*)src, elems / 4);
  else
    copy_kernel<bf16><<<(unsigned)((elems / 8 + 255) / 256), 256, 0, lc.stream>>>((bf16*)dst, (const bf16*)src, elems / 8);
  lc.count();
  lc.check();
}

void postln_prepass(Launcher& lc, int dtype, const void* g, const void* xo, const float* rstd, void* t_out, void* c_out,
                    int64_t rows, int d) {
  const int V = dtype == HBP_F32 ? 4 : 8;
  const int threads = row_block_threads(d, V);
  if (dtype == HBP_F32)
    postln_prepass_kernel<float><<<(unsigned)rows, threads, 0, lc.stream>>>((const float*)g, (const float*)xo, rstd,
                                                                           (float*)t_out, (float*)c_out, d);
  else
    postln_prepass_kernel<bf16><<<(unsigned)rows, threads, 0, lc.stream>>>((const bf16*)g, (const bf16*)xo, rstd,
                                                                          (bf16*)t_out, (bf16*)c_out, d);
  lc.count();
  lc.check();
}

void mul_elementwise(Launcher& lc, int dtype, void* dst, const void* a, const void* b, int64_t elems) {
  const int V = dtype == HBP_F32 ? 4 : 8;
  const unsigned grid = (unsigned)((elems / V + 255) / 256);
  if (dtype == HBP_F32) mul_kernel<float><<<grid, 256, 0, lc.stream>>>((float*)dst, (const float*)a, (const float*)b, elems / V);
  else mul_kernel<bf16><<<grid, 256, 0, lc.stream>>>((bf16*)dst, (const bf16*)a, (const bf16*)b, elems / V);
  lc.count();
  lc.check();
}

void add_to_states(Launcher& lc, int dtype, void* states, const void* carry, int count, int64_t elems) {
  const int V = dtype == HBP_F32 ? 4 : 8;
  dim3 grid((unsigned)((elems / V + 255) / 256), (unsigned)count);
  if (dtype == HBP_F32) add_to_states_kernel<float><<<grid, 256, 0, lc.stream>>>((float*)states, (const float*)carry, elems);
  else add_to_states_kernel<bf16><<<grid, 256, 0, lc.stream>>>((bf16*)states, (const bf16*)carry, elems);
  lc.count();
  lc.check();
}

void convert_to_f32(Launcher& lc, int dtype, const void* src, float* dst, int64_t elems) {
  const unsigned grid = (unsigned)((elems + 255) / 256);
  if (dtype == HBP_F32) launch_chained(lc, to_f32_kernel<float>, dim3(grid), 256, 0, 1, (const float*)src, dst, elems);
  else launch_chained(lc, to_f32_kernel<bf16>, dim3(grid), 256, 0, 1, (const bf16*)src, dst, elems);
}

template <typename T>
static void layernorm_launch(Launcher& lc, const float* x, T* xhat, float* rstd, int64_t rows, int d, float eps, float* master,
                             T* state, const Planes& parts) {
  const int nvec = d / 4, wpr = nvec <= 512 ? 1 : (nvec <= 1024 ? 2 : 4);  // at most 16 float4 per lane (d <= 8192)
  const int per_lane = (nvec + 32 * wpr - 1) / (32 * wpr);
  const int64_t per_block = kLnWarps / wpr;
  const unsigned grid = (unsigned)((rows + per_block - 1) / per_block);
  auto kernel = per_lane <= 4 ? layernorm_fwd_kernel<T, 4> : (per_lane <= 8 ? layernorm_fwd_kernel<T, 8> : layernorm_fwd_kernel<T, 16>);
  launch_chained(lc, kernel, dim3(grid), kLnWarps * 32, 0, 1, x, xhat, rstd, rows, d, eps, master, state, parts, wpr);
}

void layernorm_fwd(Launcher& lc, int dtype, const float* x, void* xhat, float* rstd, int64_t rows, int d, float eps,
                   float* master, void* state, const Planes& parts) {
  if (dtype == HBP_F32) layernorm_launch<float>(lc, x, (float*)xhat, rstd, rows, d, eps, master, (float*)state, parts);
  else layernorm_launch<bf16>(lc, x, (bf16*)xhat, rstd, rows, d, eps, master, (bf16*)state, parts);
}

void convert_from_f32(Launcher& lc, const float* src, bf16* dst, int64_t elems) {
  launch_chained(lc, from_f32_kernel, dim3((unsigned)((elems / 4 + 255) / 256)), 256, 0, 1, src, dst, elems / 4);
}

void split_tf32(Launcher& lc, const float* a, const float* b, float* hi, float* lo, int64_t elems) {
  const int64_t nvec = elems / 4;
  split_tf32_kernel<<<(unsigned)((nvec + 255) / 256), 256, 0, lc.stream>>>((const float4*)a, (const float4*)b, (float4*)hi,
                                                                          (float4*)lo, nvec);
  lc.count();
  lc.check();
}

void split_tf32_transposed(Launcher& lc, const float* a, const float* b, float* hiT, float* loT, int64_t rows, int cols,
                           int64_t ld) {
  if (ld <= 0) ld = cols;
  if ((uintptr_t)a & 15u) launch_split_transposed(lc, UnalignedValue{a, ld}, hiT, loT, rows, cols);  // (never with b)
  else launch_split_transposed(lc, ProductValue{a, b, ld}, hiT, loT, rows, cols);
}

void gate_grad(Launcher& lc, int dtype, const void* g, const void* x, int64_t rows_total, int d, float* da,
               float* partial, int blocks) {
  if (dtype == HBP_F32)
    gate_grad_kernel<float><<<blocks, 256, 0, lc.stream>>>((const float*)g, (const float*)x, rows_total, d, partial);
  else
    gate_grad_kernel<bf16><<<blocks, 256, 0, lc.stream>>>((const bf16*)g, (const bf16*)x, rows_total, d, partial);
  lc.count();
  lc.check();
  reduce_splitk(lc, partial, da, blocks, d);
}

}  // namespace hbp
