// The end of a kernel with a ring of tile copies (gemm_tc.cu, gemm_parts.cu, gemm_cell.cu) after one of its bounded waits gave up: no CTA may
// end, and its shared memory be given away, while a copy into it is still in flight.
#pragma once
#include "tc_common.cuh"

namespace hbp {
namespace tc {

// Of a pair: a role whose wait gave up stops the other CTA's roles too, before both meet at the end.
__device__ __forceinline__ void tell_peer(volatile int* abort_flag) {
  const uint32_t at = map_to_cta(smem_u32((const void*)abort_flag), cluster_ctarank() ^ 1u);
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(1) : "memory");
}
// Then one warp of each CTA stays for a time after which every copy is over, whoever issued it and whether its stage was ever armed.  (A
// barrier can be waited for only if what it expects is made up for, stage by stage, from the counts of all producers and other
// arrivals: with that account, known to all threads, the end of a kernel took 50 to 150 ns more, up to 1.4 % of the exact pass of a small
// decoder, 60 launches.)
__device__ __forceinline__ void outlast_copies() {
  const uint64_t t0 = global_ns();
  while (global_ns() - t0 < 100000000ull) {
  }
}

}  // namespace tc
}  // namespace hbp
