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
// The end of a pair's CTAs, for all threads of both: this CTA's roles have stopped, the other's are stopped if one of these gave up.  With
// each role telling the peer by itself, which keeps whether it gave up in a register up to here, exact passes of 20 bf16 layers 320
// (800) x 700 rows took 431 us and of 4 decoder blocks 512 x 1024 338, where this way they take 422 and 332 (426 and 335 before any peer was told);
// gemm_cell.cu, which has fewer and longer launches, gains nothing by it (LSTM, exact pass 4314 and 4321).
__device__ __forceinline__ void leave_together(volatile int* abort_flag) {
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) tell_peer(abort_flag);
  __syncwarp();
  cluster_sync_whole_warps();
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
