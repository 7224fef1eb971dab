// Shared by the one-launch recurrences (cell_cluster.cu, rnn_cluster.cu): cluster addressing, the exchange through
// distributed shared memory, the FP64 matrix instruction, small vector loads and the launch configuration.
#pragma once
#include "tc_common.cuh"

namespace hbp {
namespace cell {

constexpr int kMaxCluster = 16;
constexpr int kSmemLimit = 232448;  // 227 KB per CTA
constexpr uint64_t kWaitLimitNs = 2000000000ull;

__device__ __forceinline__ uint32_t cluster_index() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// 16 bytes into a peer's shared memory; the peer's mbarrier counts them on arrival
__device__ __forceinline__ void send16(uint32_t addr, double a, double b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(addr),
               "l"(__double_as_longlong(a)), "l"(__double_as_longlong(b)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool bar_try_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// false once the time limit has passed or another thread of this CTA has given up
__device__ __forceinline__ bool bar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  uint64_t t0 = 0;
  for (uint32_t spin = 0;; ++spin) {
    if (bar_try_cluster(bar, parity)) return true;
    if ((spin & 255u) == 255u) {
      if (*abort_flag) return false;
      const uint64_t now = tc::global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) {
        *abort_flag = 1;
        return false;
      }
    }
  }
}
// 8 x 8 += 8 x 4 times 4 x 8.  Lane l holds A(l / 4, l % 4), B(l % 4, l / 4) and C(l / 4, 2 (l % 4) + {0, 1}).
__device__ __forceinline__ void dmma(double2& c, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c.x), "+d"(c.y) : "d"(a), "d"(b));
}
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const bf16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float2 load2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 load2(const bf16* p) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p)); }
__device__ __forceinline__ void store2(float* p, double a, double b) { *reinterpret_cast<float2*>(p) = make_float2((float)a, (float)b); }
__device__ __forceinline__ void store2(bf16* p, double a, double b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn((float)a, (float)b);
}
__device__ __forceinline__ float lane4(const float4& v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w)); }
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// One thread: `bytes` contiguous bytes (a multiple of 16, both ends aligned to 16) from global to shared memory, counted by
// the mbarrier.
__device__ __forceinline__ void fetch_rows(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  tc::mbar_expect_tx(bar, bytes);
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// The whole CTA, once a wait has given up: records it and lets copies of its own and stores of peers that may still be in
// flight arrive.
__device__ __forceinline__ void after_timeout(int* status) {
  if (threadIdx.x == 0 && status) atomicExch(status, (int)HBP_ERR_TIMEOUT);
  const uint64_t t0 = tc::global_ns();
  while (tc::global_ns() - t0 < 2000000ull) {
  }
}

// Estimated clocks of a step's exchange: 500 of latency and 17 bytes per clock received, both measured.
inline double exchange_clocks(int cs, int rows, int uc) { return cs > 1 ? 500.0 + rows * cs * uc * 8 / 17.0 : 0.0; }

inline void launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr, int64_t clusters, int cs, int threads, size_t smem, cudaStream_t stream) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)(clusters * cs));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)cs;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
}

// Clusters of `cs` CTAs with all of the shared memory that this device runs at a time; 0 if it takes none.  Also opts the
// kernel in to both (per device).
template <typename K>
int max_active_clusters(K kernel, int cs, int threads) {
  int n = 0;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  launch_config(cfg, attr, 1, cs, threads, kSmemLimit, nullptr);
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess ||
      cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 0)
    n = 0;
  cudaGetLastError();
  return n;
}

// The same, asked once per device, kernel and cluster size.
template <auto Kernel>
int active_clusters(int cs, int threads) {
  struct Known { int n[kMaxCluster + 1]; };  // 1 + the answer, 0 = not asked yet
  static PerDevice<Known> known;
  int& k = known.here().n[cs];
  if (k == 0) k = 1 + max_active_clusters(Kernel, cs, threads);
  return k - 1;
}

}  // namespace cell
}  // namespace hbp
