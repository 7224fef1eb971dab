// The end of a kernel with a ring of tile copies (gemm_tc.cu, gemm_parts.cu, gemm_cell.cu) after one of its bounded waits gave up: no CTA may
// end, and its shared memory be given away, while a copy into it is still in flight.
#pragma once
#include "tc_common.cuh"

namespace hbp {
namespace tc {

// `bytes` of an armed barrier that no copy will bring
__device__ __forceinline__ void mbar_complete_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t cluster_addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
// What a ring's producers report then, in the shared memory of the CTA that owns its full barriers: how often the owner armed a stage, and
// how often producer i issued its copies into one.
struct RingReport {
  uint32_t armed, filled[4];
};
__device__ __forceinline__ void tell_peer(volatile int* abort_flag) {
  st_cluster(map_to_cta(smem_u32((const void*)abort_flag), cluster_ctarank() ^ 1u), 1);
}
// All roles of the CTA (pair: of both) have stopped; `ok` is false in a thread one of whose waits gave up.  True if any did, in all threads of
// both.  (Costs what the barrier does: an end of 150 ns more is 1.4 % of the exact pass of a small decoder, 60 launches.)
template <bool kPair>
__device__ __forceinline__ bool roles_gave_up(volatile int* abort_flag, bool ok) {
  tc_fence_before();
  if (!kPair) {
    __syncthreads();
  } else {
    if (!ok) tell_peer(abort_flag);
    __syncwarp();
    cluster_sync();  // neither CTA leaves (or frees) while its peer may still read its tiles or signal its barriers
  }
  return *abort_flag != 0;
}
// Kernels that split the registers (setmaxnreg), which the account below would cost spilled ones, and those whose ring's
// barriers also count arrivals of other roles: a time after which every copy that was issued is over, in both CTAs.
__device__ __forceinline__ void outlast_copies() {
  const uint64_t t0 = global_ns();
  while (global_ns() - t0 < 100000000ull) {
  }
}
// One thread of the ring's owner, once roles_gave_up and all have reported: waits (bounded) for every copy that was issued.  bytes[i]: what
// producer i's copies bring a stage.  The last use of a stage may be armed but not filled by all (the bytes that nobody sends are then counted as come), or
// filled in part but never armed (then armed now for what was sent).
template <int kProducers>
__device__ __forceinline__ void drain_ring(uint32_t full0, int stages, const volatile RingReport* report, const uint32_t (&bytes)[kProducers]) {
  const uint32_t n = (uint32_t)stages;
  for (uint32_t s = 0; s < n; ++s) {
    auto last = [&](uint32_t uses) { return uses > s ? (uses - 1 - s) / n * n + s + 1 : 0u; };  // of stage s, counted from one over all stages
    const uint32_t armed = report->armed;
    uint32_t use = last(armed), all = 0, sent = 0;
#pragma unroll
    for (int i = 0; i < kProducers; ++i) use = max(use, last(report->filled[i]));
    if (use == 0) continue;
#pragma unroll
    for (int i = 0; i < kProducers; ++i) {
      all += bytes[i];
      if (report->filled[i] >= use) sent += bytes[i];
    }
    const uint32_t bar = full0 + 8u * s;
    if (armed < use) mbar_expect_tx(bar, sent);
    else if (sent < all) mbar_complete_tx(bar, all - sent);
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, ((use - 1) / n) & 1u) && global_ns() - t0 < 100000000ull) {
    }
  }
}

}  // namespace tc
}  // namespace hbp
