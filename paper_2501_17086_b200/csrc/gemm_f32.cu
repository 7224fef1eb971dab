// Float GEMM on the tensor cores for any orientation of the operands (decoders in single precision, MLP stacks up to 63 wide; wider
// ones keep their operands in parts, gemm_parts.cu, where their workspace and the device allow it):
//   D(m, n) = sum_k A(m, k) B(n, k), each operand split on the way into shared memory into three bf16 parts that add up to it
//   exactly, six bf16 products of parts (all but the three below 2^-26 of the whole), the epilogues of the CUDA-core kernel.
//
// One CTA per 128 x 128 tile (and batch entry, and split of K), 512 threads:
//   warps 0..7   load 32-wide k-blocks of A and B from global memory (two blocks ahead, in registers), split them and store
//                the parts as K-major 128-byte-swizzled rows (48 KB a stage, four stages); an operand whose row index is
//                contiguous is transposed in 4 x 4 blocks in registers on the way
//   warps 8..15  add each finished accumulator to float sums in registers; epilogue
//   warp 8       also issues 12 x tcgen05.mma 128x128x16 per k-block into one of two tensor-memory accumulators, before it
//                adds up the previous block's (a warp of its own would leave 96 registers a thread instead of 128)
// The sums leave the tensor core after every 32 of K because its accumulation truncates: the error of a long chain is a bias
// that grows with its length, while the additions in registers round to nearest.  What is left of the bias is taken out there
// (kOneUp).  Error against 64 bits, normal operands (2-norm): the CUDA-core kernel's running float sums; here; two tf32 parts
// and three products, which hold 22 bits and are biased:
//   K =   32  1.0e-7  0.7e-7  1.3e-7        K =  520  4.1e-7  1.05e-7  1.5e-7
//   K =  128  2.0e-7  0.8e-7  1.35e-7       K = 4096  1.1e-6  2.2e-7  2.4e-7
// and less for positive operands.  Weight gradients of float MLP stacks of 2 and 8 layers, 64 to 520 wide, 32 to 4000 rows (here under
// HBP_GEMM_PAIR=0; in parts they have the same bits): 0.18 to 1.0 times the error on the CUDA cores.  Contractions up to 16 stay there: a float sum of a few terms rounds no more than a
// block truncates (K = 4: 3.9e-8, 16: 7.3e-8, 20: 8.2e-8, 32: 1.03e-7 against 6.8e-8 for any K up to 32).
//
// The six bf16 products cost the tensor time of three tf32 ones (768 clocks of a k-block), the parts take 48 KB of stores
// instead of 64.  1900 x 1560 x 520, 12 at once: CUDA cores 1800 us, tf32 363, here 350 (106 TFLOP/s); rows contiguous 1700, 473,
// 467; 4096 x 1024 x 4096: 1390, 282, 254.  Bound by the loading warps, no one thing in them: of the 350 (467) us 50 (162) go
// without the global loads, 40 (19) without the split's arithmetic, 14 (38) without two of the three stores, 16 (29) without ten
// of the twelve MMAs.
#include "float_parts.cuh"
#include "tc_common.cuh"

namespace hbp {

using namespace tc;

namespace {

constexpr int BM = 128, BN = 128, BK = 32;
constexpr int kShortK = 16;  // contractions up to here are the CUDA-core kernel's
constexpr int kWorkerWarps = 8, kMmaWarp = kWorkerWarps, kAllThreads = 64 * kWorkerWarps;
constexpr int kStages = 4;
// 128 rows of 128 bytes: the high and middle parts of 32 elements of A; of B; the low parts of A and of B
constexpr uint32_t kTile = BM * 128, kStageBytes = 3 * kTile;
constexpr uint32_t kTmemCols = 256;
constexpr int kSmemBytes = kStages * (int)kStageBytes + 1024 /*alignment*/ + 256 /*barriers*/;
// what each adding warp uses of the stages once all products are done (refine's two blocks, or the epilogue's one)
constexpr int kRowPitch = 33, kColPitch = 68, kWarpFloats = BK * kRowPitch + BK * kColPitch;
static_assert(kWorkerWarps * kWarpFloats * 4 <= kStages * (int)kStageBytes && 32 * 36 <= kWarpFloats, "stages");

struct F32Params {
  GemmArgs g;
  int a_mn, b_mn;  // 1: the row index is contiguous
  int k_blocks, kb_per_split;
  int* status;
};

__device__ __forceinline__ void st_shared8(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
// Four neighbours in k (unit of 4 out of 8) of a row: high and middle parts to the operand's tile, low parts to its half
// (0 = A, 4 = B, in 16-byte units) of the common one.  An infinity, a NaN or a value whose high part rounds to one leaves a part NaN,
// so that every sum it enters is not finite, which refine settles.
__device__ __forceinline__ void store_split(uint32_t tile, uint32_t low_tile, int low_half, int row, int unit, float a, float b, float c, float d) {
  uint32_t h0, m0, l0, h1, m1, l1;
  split_plain2(a, b, h0, m0, l0);
  split_plain2(c, d, h1, m1, l1);
  const uint32_t at = (uint32_t)(unit & 1) * 8u;
  st_shared8(swz(tile, row, unit >> 1) + at, h0, h1);
  st_shared8(swz(tile, row, 4 + (unit >> 1)) + at, m0, m1);
  st_shared8(swz(low_tile, row, low_half + (unit >> 1)) + at, l0, l1);
}

// This thread's share of one operand's 128 x 32 block: four 16-byte loads.
//   K contiguous: 8 lanes read the 8 units of a row, rows 32 apart;  rows contiguous: a 4 x 4 block, lane & 7 = unit of K.
// Either way the two rows that a half-warp stores to are 4 apart (modulo 8), and the swizzle puts them on distinct banks.
struct Loader {
  const float* at;     // this thread's first element of the current block
  int64_t step, next;  // between its four loads, and from block to block
  int left, k, unit;   // rows from its first row to the end; first k of the thread in the current block
  bool mn;
  __device__ __forceinline__ int k_row() const {  // of 32, for K contiguous
    const int g = threadIdx.x >> 3;
    return (g & ~7) | ((g & 1) << 2) | ((g >> 1) & 3);
  }
  __device__ __forceinline__ void init(const void* p, int64_t s_row, int64_t s_k, int extent, int row0, int k0, bool mn_major) {
    const int tid = threadIdx.x;
    mn = mn_major;
    unit = tid & 7;
    const int row = row0 + (mn ? (tid >> 3) * 4 : k_row());
    left = extent - row;
    k = k0 + unit * 4;
    at = (const float*)p + (int64_t)row * s_row + (int64_t)k * s_k;
    step = mn ? s_k : 32 * s_row;
    next = BK * s_k;
  }
  __device__ __forceinline__ void load(int k_end, float4* v) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bool in = mn ? left > 0 && k + i < k_end : left > 32 * i && k < k_end;
      v[i] = in ? __ldg(reinterpret_cast<const float4*>(at + i * step)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    at += next;
    k += BK;
  }
  __device__ __forceinline__ void store(uint32_t tile, uint32_t low_tile, int low_half, const float4* v) const {
    if (mn) {
      const int r = (threadIdx.x >> 3) * 4;
      store_split(tile, low_tile, low_half, r, unit, v[0].x, v[1].x, v[2].x, v[3].x);
      store_split(tile, low_tile, low_half, r + 1, unit, v[0].y, v[1].y, v[2].y, v[3].y);
      store_split(tile, low_tile, low_half, r + 2, unit, v[0].z, v[1].z, v[2].z, v[3].z);
      store_split(tile, low_tile, low_half, r + 3, unit, v[0].w, v[1].w, v[2].w, v[3].w);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) store_split(tile, low_tile, low_half, k_row() + 32 * i, unit, v[i].x, v[i].y, v[i].z, v[i].w);
    }
  }
};

// Four neighbouring outputs (m, n .. n + 3); what the scalar epilogue_store does for these kinds, with 16-byte accesses.
__device__ __forceinline__ void epilogue_store4(const GemmArgs& g, int b, int m, int n, float4 acc) {
  float* D = (float*)g.D + b * g.d_sb + (int64_t)m * g.ldd + n;
  float v[4] = {acc.x, acc.y, acc.z, acc.w};
  if (g.epi == EPI_GELU_FWD) {
    float d2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      d2[i] = gelu_prime_f(v[i]);
      v[i] = gelu_f(v[i]);
    }
    *reinterpret_cast<float4*>((float*)g.D2 + b * g.d2_sb + (int64_t)m * g.ldd2 + n) = make_float4(d2[0], d2[1], d2[2], d2[3]);
  } else if (g.epi == EPI_MUL || g.epi == EPI_ADD || g.epi == EPI_RESID) {
    const float4 ev = *reinterpret_cast<const float4*>((const float*)g.E + b * g.e_sb + (int64_t)m * g.lde + n);
    const float e[4] = {ev.x, ev.y, ev.z, ev.w};
    if (g.epi == EPI_RESID) {
      float mask[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float gate = g.gate ? ((const float*)g.gate)[b * g.gate_sb + n + i] : 1.0f;
        v[i] = gate * e[i] + v[i];
        mask[i] = v[i] > 0.0f ? 1.0f : 0.0f;
        if (g.relu) v[i] = fmaxf(v[i], 0.0f);
      }
      if (g.relu) *reinterpret_cast<float4*>((float*)g.D2 + b * g.d2_sb + (int64_t)m * g.ldd2 + n) = make_float4(mask[0], mask[1], mask[2], mask[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = g.epi == EPI_MUL ? v[i] * e[i] : v[i] + e[i];
    }
  }
  *reinterpret_cast<float4*>(D) = make_float4(v[0], v[1], v[2], v[3]);
}

// Sums that the parts may not give as the operands would: infinite or NaN ones.
__device__ __forceinline__ bool in_doubt(float sum) { return !(fabsf(sum) < __uint_as_float(0x7f800000u)); }
// The sums in doubt of one warp's 32 x 64 outputs, formed again as plain float sums in ascending order of k.  Products of parts
// do not give what one product of the whole does where an operand is not finite: an infinity times a part of zero, or of the
// other sign, is NaN where infinity times the operand is infinity, a NaN may lose its payload and become an infinity, and a
// part may overflow where the sum does not.  Whatever the operands, a finite sum has met none of that.
__device__ __forceinline__ void refine(const GemmArgs& g, int b, int m0, int n0, int k_lo, int k_hi, float* smem, float (&sum)[64]) {
  const int lane = threadIdx.x & 31;
  float *As = smem, *Bs = smem + BK * kRowPitch;  // [k][row], [k][column]
  const float* A = (const float*)g.A + (int64_t)b * g.a_sb;
  const float* B = (const float*)g.B + (int64_t)b * g.b_sb;
  // a [rows] x [BK] block, lanes along the index that is contiguous
  auto stage = [&](float* to, int pitch, const float* from, int64_t s_row, int64_t s_k, int row0, int rows, int extent, int k0) {
    for (int i = lane; i < rows * BK; i += 32) {
      const int r = s_k == 1 ? i / BK : i % rows, kk = s_k == 1 ? i % BK : i / rows;
      to[kk * pitch + r] = (row0 + r < extent && k0 + kk < k_hi) ? __ldg(from + (int64_t)(row0 + r) * s_row + (int64_t)(k0 + kk) * s_k) : 0.0f;
    }
  };
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.0f;
    for (int k0 = k_lo; k0 < k_hi; k0 += BK) {
      __syncwarp();
      stage(As, kRowPitch, A, g.a_sm, g.a_sk, m0, 32, g.M, k0);
      stage(Bs, kColPitch, B, g.b_sn, g.b_sk, n0 + 32 * h, 32, g.N, k0);
      __syncwarp();
#pragma unroll 1
      for (int kk = 0; kk < min(BK, k_hi - k0); ++kk) {
        const float a = As[kk * kRowPitch + lane];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(Bs + kk * kColPitch + 4 * i);
          acc[4 * i] = fmaf(a, v.x, acc[4 * i]);
          acc[4 * i + 1] = fmaf(a, v.y, acc[4 * i + 1]);
          acc[4 * i + 2] = fmaf(a, v.z, acc[4 * i + 2]);
          acc[4 * i + 3] = fmaf(a, v.w, acc[4 * i + 3]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (in_doubt(sum[32 * h + i])) sum[32 * h + i] = acc[i];
  }
}

__global__ void __launch_bounds__(kAllThreads, 1) gemm_f32_kernel(const F32Params p) {
  const GemmArgs& g = p.g;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* aligned = smem_raw + (base - smem_u32(smem_raw));
  uint64_t* bars = reinterpret_cast<uint64_t*>(aligned + kStages * kStageBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto accf_bar = [&](int a) { return bar0 + 8u * (2 * kStages + a); };
  auto acce_bar = [&](int a) { return bar0 + 8u * (2 * kStages + 2 + a); };
  const uint32_t drain_bar = bar0 + 8u * (2 * kStages + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), kWorkerWarps);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), kWorkerWarps);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  chain_next();
  chain_wait();

  const int b = blockIdx.z / g.splitk, split = blockIdx.z % g.splitk;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int kb_lo = split * p.kb_per_split, kb_hi = min(p.k_blocks, kb_lo + p.kb_per_split);
  const int n_kb = max(0, kb_hi - kb_lo);

  if (warp < kWorkerWarps) {
    Loader la, lb;
    la.init((const float*)g.A + (int64_t)b * g.a_sb, g.a_sm, g.a_sk, g.M, m0, kb_lo * BK, p.a_mn != 0);
    lb.init((const float*)g.B + (int64_t)b * g.b_sb, g.b_sn, g.b_sk, g.N, n0, kb_lo * BK, p.b_mn != 0);
    const int k_end = min(g.K, kb_hi * BK);
    float4 va[2][4], vb[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      la.load(k_end, va[i]);
      lb.load(k_end, vb[i]);
    }
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int kb = 0; kb < n_kb && ok; kb += 2) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (kb + i >= n_kb) break;
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
        const uint32_t s0 = base + stage * kStageBytes;
        la.store(s0, s0 + 2 * kTile, 0, va[i]);
        la.load(k_end, va[i]);  // past the last block: nothing
        lb.store(s0 + kTile, s0 + 2 * kTile, 4, vb[i]);
        lb.load(k_end, vb[i]);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar(stage));
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
  } else {
    const int quarter = warp & 3, half = (warp >> 2) & 1;
    const uint32_t tsrc = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 64);
    float sum[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) sum[i] = 0.0f;
    bool ok = true;
    auto drain = [&](int kb) {  // adds k-block kb's accumulator to the sums
      const int acc = kb & 1;
      const float unbias = ((3 * kb + lane) & 7) < 3 ? kOneUp : 1.0f;
      if (!mbar_wait(accf_bar(acc), (uint32_t)((kb >> 1) & 1), abort_flag, p.status)) { ok = false; return; }
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[32];
        tc_ld32(tsrc + (uint32_t)(acc * BN + h * 32), v);
        if (h == 1) {  // read: it may be written again
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acce_bar(acc));
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) sum[h * 32 + i] = fmaf(v[i], unbias, sum[h * 32 + i]);
      }
    };
    if (warp == kMmaWarp) {
      uint32_t elected;
      asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(elected));
      const bool issuer = elected != 0;
      const uint32_t idesc = (1u << 4) /*fp32 accumulate*/ | (1u << 7) | (1u << 10) /*bf16*/ | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = 0; kb < n_kb; ++kb) {
        const int acc = kb & 1;
        ok = mbar_wait(full_bar(stage), phase, abort_flag, p.status) &&
             mbar_wait(acce_bar(acc), (uint32_t)(((kb >> 1) & 1) ^ 1), abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        if (issuer) {
          const uint32_t s0 = base + stage * kStageBytes, tmem_d = tmem_base + (uint32_t)acc * BN;
          const uint64_t a_h = make_desc(s0, 16u, 1024u), b_h = make_desc(s0 + kTile, 16u, 1024u);
          const uint64_t a_l = make_desc(s0 + 2 * kTile, 16u, 1024u), a_m = a_h + 4, b_m = b_h + 4, b_l = a_l + 4;
          const uint64_t as[6] = {a_l, a_h, a_m, a_m, a_h, a_h}, bs[6] = {b_h, b_l, b_m, b_h, b_m, b_h};  // the small terms first
#pragma unroll
          for (int q = 0; q < 6; ++q)
#pragma unroll
            for (int k = 0; k < 2; ++k) tc_mma(tmem_d, as[q] + 2 * k, bs[q] + 2 * k, idesc, q + k > 0);
          tc_commit(empty_bar(stage));
          tc_commit(accf_bar(acc));
        }
        __syncwarp();
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
        if (kb > 0) drain(kb - 1);
        if (!ok) break;
      }
      if (ok && n_kb > 0) drain(n_kb - 1);
      if (!ok) {  // let issued MMAs finish before the tensor memory is freed
        if (issuer) tc_commit(drain_bar);
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(drain_bar, 0) && global_ns() - t0 < 100000000ull) {
        }
      }
    } else {
      for (int kb = 0; kb < n_kb && ok; ++kb) drain(kb);
    }
    // All products of this CTA are done: the stages are free.  Each warp passes its 32 x 64 sums through 32 x 36 floats of
    // its own so that 8 lanes write 32 consecutive columns of a row.
    if (ok) {
      float* buf = reinterpret_cast<float*>(aligned) + (warp - kWorkerWarps) * kWarpFloats;
      bool doubt = false;
#pragma unroll
      for (int i = 0; i < 64; ++i) doubt = doubt || in_doubt(sum[i]);
      if (__any_sync(0xffffffffu, doubt))
        refine(g, b, m0 + quarter * 32, n0 + half * 64, kb_lo * BK, min(g.K, kb_hi * BK), buf, sum);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i)
          *reinterpret_cast<float4*>(buf + lane * 36 + 4 * i) =
              make_float4(sum[h * 32 + 4 * i], sum[h * 32 + 4 * i + 1], sum[h * 32 + 4 * i + 2], sum[h * 32 + 4 * i + 3]);
        __syncwarp();
        const int n = n0 + half * 64 + h * 32 + 4 * (lane & 7);
#pragma unroll 2
        for (int i = 0; i < 8; ++i) {
          const int r = 4 * i + (lane >> 3), m = m0 + quarter * 32 + r;
          if (m >= g.M || n >= g.N) continue;
          const float4 v = *reinterpret_cast<const float4*>(buf + r * 36 + 4 * (lane & 7));
          if (g.splitk > 1) *reinterpret_cast<float4*>(g.partial + (((int64_t)split * g.batch + b) * g.M + m) * g.N + n) = v;
          else epilogue_store4(g, b, m, n, v);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// An operand qualifies if one of its strides is 1, its 16-byte vectors are aligned and none straddles the end.
bool operand_ok(const void* base, int64_t s_row, int64_t s_k, int64_t s_b, int batch, int rows, int K, int* mn) {
  if ((uintptr_t)base & 15u) return false;
  if (batch > 1 && s_b % 4) return false;
  if (s_k == 1 && s_row % 4 == 0 && K % 4 == 0) { *mn = 0; return true; }
  if (s_row == 1 && s_k % 4 == 0 && rows % 4 == 0) { *mn = 1; return true; }
  return false;
}

}  // namespace

bool gemm_f32_tc(Launcher& lc, const GemmArgs& g, int* status_word) {
  if (!status_word || g.in_dtype != HBP_F32 || g.A2) return false;
  if (g.M <= 0 || g.N <= 0 || g.K <= 0 || g.batch <= 0) return false;
  // Few rows are the CUDA-core kernel's: a tile would be mostly padding, and setting up tensor memory and the pipeline takes
  // 6 us.  32 x 64 x 256: 9 us there against 14.5; 32 x 512 x 1024: 23 against 39.  (Many such products at once, 500 tiles or more,
  // would take half the time here, 32 x 1024 x 4096, 16 at once, 160 us against 290: the rule does not look at that.)  So are
  // short contractions, whose float sums have few roundings (above).
  if (g.M <= 32 || g.K <= kShortK) return false;
  // the epilogue's 16-byte accesses
  auto vec = [](const void* p, int64_t ld, int64_t sb) { return !((uintptr_t)p & 15u) && ld % 4 == 0 && sb % 4 == 0; };
  if (g.N % 4 || !vec(g.D, g.ldd, g.d_sb) || g.R) return false;
  const bool has_e = g.epi == EPI_MUL || g.epi == EPI_ADD || g.epi == EPI_RESID;
  if (!has_e && g.epi != EPI_STORE && g.epi != EPI_STORE_LN && g.epi != EPI_GELU_FWD) return false;
  if (has_e && (!g.E || !vec(g.E, g.lde, g.e_sb))) return false;
  if ((g.epi == EPI_GELU_FWD || g.relu) && (!g.D2 || !vec(g.D2, g.ldd2, g.d2_sb))) return false;
  if (g.splitk > 1 && (g.epi != EPI_STORE || ((uintptr_t)g.partial & 15u))) return false;
  F32Params p;
  p.g = g;
  if (!operand_ok(g.A, g.a_sm, g.a_sk, g.a_sb, g.batch, g.M, g.K, &p.a_mn)) return false;
  if (!operand_ok(g.B, g.b_sn, g.b_sk, g.b_sb, g.batch, g.N, g.K, &p.b_mn)) return false;
  const int64_t z = (int64_t)g.batch * g.splitk;
  if (z > 65535 || (g.M + BM - 1) / BM > 65535) return false;
  p.k_blocks = (g.K + BK - 1) / BK;
  p.kb_per_split = (p.k_blocks + g.splitk - 1) / g.splitk;
  p.status = status_word;
  static PerDevice<bool> attr_done;
  if (!attr_done.here()) {
    if (cudaFuncSetAttribute(gemm_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    attr_done.here() = true;
  }
  dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, (unsigned)z);
  launch_chained(lc, gemm_f32_kernel, grid, kAllThreads, kSmemBytes, 1, p);
  lc.ran(HBP_FORM_GEMM_F32);
  if (g.splitk > 1) reduce_splitk(lc, g.partial, (float*)g.D, g.splitk, (int64_t)g.batch * g.M * g.N);
  return true;
}

}  // namespace hbp
