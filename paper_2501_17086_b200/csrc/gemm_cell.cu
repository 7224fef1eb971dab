// The all-step products of the float recurrent kinds, whose left operand is formed while it is loaded:
//   a(r, c) = g(r, .) times the coefficients cached by the forward pass (tanh RNN g tanh'; GRU g [c_r | c_z | c_nr (| c_n)];
//   LSTM [t c_i | t c_f | t c_g | g_h c_o], t = g_c + g_h c_h), r = one of the T * B rows of the sequence.
//   VJP               u(r, n)  = sum_c a(r, c) W(c, n) (+ delta(r, n))
//   weight gradients  dW(c, n) = sum_r a(r, c) h(r, n),  dU(c, n) = sum_r a(r, c) x(r, n)
//
// Each product of floats is six bf16 products of parts (float_parts.cuh).  CTA pairs on 256 x n_tile tiles (n_tile = 32 .. 256 in
// steps of 32), persistent, 512 threads:
//   warp 0       VJP: TMA producer of W's planes
//   warp 1       MMA issuer (one lane of the even CTA): 12 x tcgen05.mma 256 x n_tile x 16 per 32 of K, the product of the high parts
//                into one accumulator, the five small ones into another (FINE: all into one), so that only every sixth addition is
//                made at full magnitude, where the tensor core's truncation counts
//   warps 4..7   epilogue: the two accumulators added, delta added (VJP), out by TMA tile copies
//   warps 8..15  load g and the coefficients (16 bytes per lane, the next blocks' loads in flight while one is worked on), multiply,
//                split and store the parts: K-major rows of 64 bytes for the VJP; MN-major rows of 128 bytes for the weight gradients,
//                whose right operand (states, inputs) they split likewise, so that nothing is ever written transposed
// FINE, the weight gradients of T * B rows that are no multiple of 4: they have always been sums of floats, 3e-8 to 1.2e-7 from 64 bits
// (tanh RNN 1.5e-7 to 7e-7), and stay so.  One accumulator per 32 rows, the small terms first, and the epilogue adds it, rounded and
// its truncation made good (float_parts.cuh), to sums kept in tensor memory; every 512 rows these go out as a set of partial
// sums, which are added in double.  Weight gradients in us as float sums before / as the other form / so: GRU 32385 x 512 1590 / 330 / 750
// (errors 7e-8 / 1.1e-6 / 7e-8), 131967 x 64 550 / 70 / 100, LSTM 32385 x 512 1720 / 500 / 1190, tanh RNN 135135 x 512 10400 / 525 / 1140 (2e-7 /
// 1.3e-6 / 7e-8).  Tiles of 96 columns 980, of 256, whose one set of accumulators holds up the products, 840 (GRU 32385 x 512).
// Nothing of the operand goes through memory.  Before, it was written as two tf32 parts by a pass (the tanh RNN's by the scan before)
// and read back by gemm_tc.cu, for the gradients transposed, their partial sums written every 512 rows.  One VJP with its pass and
// scan, before / now: tanh RNN 131072 x 512 446 / 404 us, GRU 32768 x 512 345 / 250, GRU 131072 x 64 138 / 72; the weight
// gradients 780 / 480, 550 / 310, 260 / 78, LSTM 32768 x 512 695 / 480.  Error against 64 bits: 1.6e-6 / 1.3e-6, 1.2e-6 / 1.0e-6 of
// the gradients (2-norm, all outputs).
// What bounds it: at 512 units the products (205 us of the tanh RNN's 320 at 1.68 GHz), the loading warps beside them (240 with two of
// twelve MMAs: the loads, 16 bytes a lane in flight through the first-level cache, which the shared memory leaves 60 KB of: with
// 28 KB left 342, so the loads do not allocate there and the epilogue has three buffers, not five) and the end of a tile, which
// a 256-column tile's accumulators leave uncovered (20 us of it waiting for delta); at 64 units the bytes (200 MB in 36 us).  Sixteen
// loading warps with half the rows each are no faster (339).
#include <type_traits>

#include "float_parts.cuh"
#include "ring_drain.cuh"
#include "tc_common.cuh"

namespace hbp {

using namespace tc;

namespace {

constexpr int BM = 128, BK = 32, TILE_M = 2 * BM, kMaxTileN = 256, kStages = 3, kSets = 2;
constexpr uint32_t kABytes = 3 * BM * BK * 2, kStageBytes = 2 * kABytes;
constexpr uint32_t kMnBlock = 3 * BK * 128;  // one MN-major block of 64 elements: three parts of 32 rows of 128 bytes
constexpr int kEpiWarps = 4, kLoadWarps = 8, THREADS = 256 + 32 * kLoadWarps;
// 512 threads start with 128 registers each, 65536: 128 x 56 + 128 x 168 + 256 x 144 = 65536
constexpr int kRegsFew = 56, kRegsEpi = 168, kRegsLoad = 144;
constexpr int kEpiBufs = 3;
constexpr uint32_t kFloatBuf = 4096;
constexpr uint32_t TMEM_COLS = 512;
constexpr int SMEM_BYTES = kStages * (int)kStageBytes + kEpiWarps * kEpiBufs * (int)kFloatBuf + 1024 /*alignment*/ + 512 /*barriers*/;
// The operand is multiplied by this on the way in and the sums divided by it: the low part of any normal float is then a normal
// bf16, also of gradients below 1e-34, which long recurrences have (values from 2^103 on overflow: refine).
constexpr float kScale = 16777216.0f, kUnscale = 1.0f / 16777216.0f;
// Weight gradients: rows that add up in the tensor core (32 additions at full magnitude, each of which truncates) before the sum is added,
// rounded, to the split's partial sums.  With 1024 rows (as once here) a pass takes 0.5 to 2 % less (GRU 32768 x 512 5339 for 5367 us, tanh
// RNN 131072 x 512 2715 for 2768) and is twice as far from 64 bits: dW, dU of the tanh RNN 32768 x 512 1.3e-6, 1.7e-6 (as three tf32
// products 1.2e-6, 1.6e-6) and 5.9e-7, 7.8e-7 with 512, of the GRU 1.1e-6 (1.2e-6) and 5.4e-7.  That the sums of a split are added in
// float adds 2e-9 to that.
constexpr int kDrainBlocks = 512 / BK;
// FINE: rows from which on the tensor core is used (as in gemm_f32.cu); k-blocks of a set of partial sums, more where the workspace, which
// is that of the splits, has no room for so many sets (GRU of 131967 rows, 64 units and inputs: 57 k-blocks, 3.1e-8 -> 3.7e-8 from 64 bits;
// 512 and 512: 30, 5.0e-8 -> 5.8e-8, and 4250 -> 3780 us); the widest tile that leaves two accumulators room beside the sums (three
// and four of them, on tiles of 128 and 96 columns, gain nothing: a k-block takes the loading warps as long for any width)
constexpr int kFewProducts = 17, kFineSet = 512 / BK, kFineTileN = 160;

struct Params {
  CellOperand o;
  int kind;       // hbp_block
  int blocks;     // of the VJP's operand: 1, 3, 4
  // VJP
  Planes W;
  int N, n_tiles, num_tiles, chunks;  // chunks of 32 channels, `blocks` k-blocks each
  int n_tile, has_e;
  const float* fg;        // LSTM: the cell-state half of the VJP is written beside the product
  const float* delta_c;
  float* uc;
  // weight gradients: products against the states (segment 0) and the inputs (segment 1), or against both side by side (`both`: one
  // segment of d + in columns, M of all coefficient blocks)
  struct Segment {
    const float* B;
    int64_t ldb;
    int N, n_tile, m_tiles, n_tiles, vec;
  } seg[2];
  int M, tiles, splits, k_blocks, per_split, both;
  int group, merge, sets_per_split;  // k-blocks added up in the tensor core; such sums in a set of partial sums; sets of a split
  int* status;
};

__device__ __forceinline__ float part_value(const Planes& P, int64_t at) {
  return __bfloat162float(P.p[at]) + (__bfloat162float(P.p[at + P.plane]) + __bfloat162float(P.p[at + 2 * P.plane]));
}
// block q of the operand that weight gradient rows of block q belong to: dU's third block of the GRU uses the fourth coefficient
template <int KIND>
__device__ __forceinline__ int coef_block(int q, int segment) {
  return KIND == HBP_BLOCK_GRU && segment == 1 && q == 2 ? 3 : q;
}
template <int KIND>
__device__ __forceinline__ float operand_value(const CellOperand& o, int64_t r, int q, int c) {
  if (KIND == HBP_BLOCK_RNN_TANH) return o.g[r * o.d + c] * o.coef[r * o.d + c];
  if (KIND == HBP_BLOCK_GRU) return o.g[r * o.d + c] * o.coef[r * 4 * o.d + q * o.d + c];
  const float gh = o.g[r * 2 * o.d + o.d + c];
  const float* cr = o.coef + r * 5 * o.d + c;
  return q == 3 ? gh * cr[3 * o.d] : (o.g[r * 2 * o.d + c] + gh * cr[4 * o.d]) * cr[q * o.d];
}
// Sums that the parts may not give as the operands would (infinite or NaN ones), again as plain float sums of the operands.
template <int KIND>
__device__ __forceinline__ void refine_vjp(const Params& p, int64_t row, int col0, float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int part = 0; part < 32; part += 4) {  // (few sums at a time: this code must not cost the others registers)
    float acc[4] = {};
#pragma unroll 1
    for (int q = 0; q < p.blocks; ++q)
#pragma unroll 1
      for (int c = 0; c < p.o.d; ++c) {
        const float a = row < p.o.rows ? operand_value<KIND>(p.o, row, q, c) : 0.0f;
        const float mine = col0 + lane < p.N ? part_value(p.W, (int64_t)(q * p.o.d + c) * p.W.ld + col0 + lane) : 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = fmaf(a, __shfl_sync(0xffffffffu, mine, part + i), acc[i]);
      }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (!(fabsf(v[part + i]) < __uint_as_float(0x7f800000u))) v[part + i] = acc[i];
  }
}
template <int KIND>
__device__ __forceinline__ void refine_grad(const Params& p, int segment, int m, int col0, int r_lo, int r_hi, float (&v)[32]) {
  const int lane = threadIdx.x & 31, q = coef_block<KIND>(m / p.o.d, segment), c = m % p.o.d;
  const Params::Segment& s = p.seg[segment];
#pragma unroll
  for (int part = 0; part < 32; part += 4) {
    float acc[4] = {};
#pragma unroll 1
    for (int r = r_lo; r < r_hi; ++r) {
      const float a = m < p.M ? operand_value<KIND>(p.o, r, q, c) : 0.0f;
      const int n = col0 + lane;
    const float mine = n >= s.N ? 0.0f : p.both && n >= p.o.d ? p.seg[1].B[r * p.seg[1].ldb + n - p.o.d] : s.B[r * s.ldb + n];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] = fmaf(a, __shfl_sync(0xffffffffu, mine, part + i), acc[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (!(fabsf(v[part + i]) < __uint_as_float(0x7f800000u))) v[part + i] = acc[i];
  }
}

// 32 columns of this thread's TMEM lane; tc_st_wait() before they are read back
__device__ __forceinline__ void tc_st32(uint32_t taddr, const float* v) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"
      ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]),
      "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]),
      "r"(r[31]), "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Two neighbouring floats in one register pair, for the packed float instructions.
typedef unsigned long long f2;
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 pack2(uint32_t lo, uint32_t hi) { return (f2)hi << 32 | lo; }
// a box into L2 (a hint)
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* tm, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global [%0, {%1, %2, %3}];" ::"l"(tm), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// Four neighbouring floats of a row: with 16 bytes a lane a warp's load covers whole lines (32 bytes a lane in two loads take the
// load path twice: the weight gradients of 131072 x 512 476 -> 880 us)
struct Four {
  f2 a, b;
};
__device__ __forceinline__ Four load4(const float* p) {
  ulonglong2 t;
  asm volatile("ld.global.nc.L1::no_allocate.v2.u64 {%0, %1}, [%2];" : "=l"(t.x), "=l"(t.y) : "l"(p));
  return {t.x, t.y};
}
__device__ __forceinline__ Four scaled(const Four& x) {
  const f2 s = pack2(__float_as_uint(kScale), __float_as_uint(kScale));
  return {mul2(x.a, s), mul2(x.b, s)};
}
__device__ __forceinline__ Four times(const Four& x, const Four& y) { return {mul2(x.a, y.a), mul2(x.b, y.b)}; }
// split_plain2 of a pair (an infinity or a NaN leaves a part NaN, so that every sum it enters is not finite, which refine settles)
__device__ __forceinline__ void split_pair(f2 x, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack_bf16(__uint_as_float((uint32_t)x), __uint_as_float((uint32_t)(x >> 32)));
  const f2 r = sub2(x, pack2(h << 16, h & 0xffff0000u));
  m = pack_bf16(__uint_as_float((uint32_t)r), __uint_as_float((uint32_t)(r >> 32)));
  const f2 q = sub2(r, pack2(m << 16, m & 0xffff0000u));
  l = pack_bf16(__uint_as_float((uint32_t)q), __uint_as_float((uint32_t)(q >> 32)));
}
__device__ __forceinline__ void st_shared8(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void store_parts(uint32_t at, uint32_t part, const Four& v) {
  uint32_t h0, m0, l0, h1, m1, l1;
  split_pair(v.a, h0, m0, l0);
  split_pair(v.b, h1, m1, l1);
  st_shared8(at, h0, h1);
  st_shared8(at + part, m0, m1);
  st_shared8(at + 2 * part, l0, l1);
}

// One unit of the weight gradients' work: a tile of one segment and a range of k-blocks.
struct Unit {
  int segment, m0, n0, kb_lo, kb_hi, split;
};
__device__ __forceinline__ Unit unit_of(const Params& p, int unit) {
  Unit u;
  u.split = unit / p.tiles;
  int t = unit % p.tiles;
  const int first = p.seg[0].m_tiles * p.seg[0].n_tiles;
  u.segment = t >= first ? 1 : 0;
  if (u.segment) t -= first;
  const Params::Segment& s = p.seg[u.segment];
  u.m0 = (t / s.n_tiles) * TILE_M;
  u.n0 = (t % s.n_tiles) * s.n_tile;
  u.kb_lo = u.split * p.per_split;
  u.kb_hi = min(p.k_blocks, u.kb_lo + p.per_split);
  return u;
}

template <int KIND, bool GRAD, bool FINE>
__global__ void __launch_bounds__(THREADS, 1)
gemm_cell_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmD, const __grid_constant__ CUtensorMap tmD1,
                 const __grid_constant__ CUtensorMap tmE, const __grid_constant__ Params p) {
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int first_item = (int)(blockIdx.x >> 1), item_step = (int)(gridDim.x >> 1);
  const int items = GRAD ? p.tiles * p.splits : p.num_tiles;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t epi_base = base + kStages * kStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + (base - smem_u32(smem_raw)) + kStages * kStageBytes + kEpiWarps * kEpiBufs * kFloatBuf);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto accf_bar = [&](int a) { return bar0 + 8u * (2 * kStages + a); };
  auto acce_bar = [&](int a) { return bar0 + 8u * (2 * kStages + kSets + a); };
  const uint32_t drain_bar = bar0 + 8u * (2 * kStages + 2 * kSets);
  auto epi_bar = [&](int w, int i) { return bar0 + 8u * (2 * kStages + 2 * kSets + 1 + w * kEpiBufs + i); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 2 * kSets + 1 + kEpiWarps * kEpiBufs);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), 2 * kLoadWarps + (GRAD ? 0 : 1));  // both CTAs' warps (and the copies' bytes) arrive at the leader
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < kSets; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), 2 * kEpiWarps);
    }
    mbar_init(drain_bar, 1);
    for (int w = 0; w < kEpiWarps; ++w)
      for (int i = 0; i < kEpiBufs; ++i) mbar_init(epi_bar(w, i), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  chain_next();
  chain_wait();

  // accumulators: `sets` pairs of n_tile columns (the widest tiles fill the tensor memory with one); FINE: single ones, the sums behind
  auto item_n_tile = [&](int item) { return GRAD ? p.seg[unit_of(p, item).segment].n_tile : p.n_tile; };
  const int widest = GRAD ? max(p.seg[0].n_tile, p.seg[1].n_tile) : p.n_tile;
  constexpr int kAccs = FINE ? 1 : 2;  // accumulators of a set
  const int sets = (2 * kAccs + (FINE ? 1 : 0)) * widest <= (int)TMEM_COLS ? 2 : 1;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsFew));
    if (!GRAD && warp == 0) {
      // ---------------------------------------------------------------- TMA producer of W's planes
      if (lane == 0) {
        const int half_n = p.n_tile / 2;
        const uint32_t b_bytes = (half_n > 64 ? 2 : 1) * kMnBlock;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int item = first_item; item < items && ok; item += item_step) {
          const int n0 = (item % p.n_tiles) * p.n_tile + (int)rank * half_n;
          for (int c = 0; c < p.chunks && ok; ++c)
            for (int q = 0; q < p.blocks; ++q) {
              if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
              const uint32_t sB = base + stage * kStageBytes + kABytes, fb = map_to_cta(full_bar(stage), 0);
              if (leader) mbar_expect_tx(full_bar(stage), 2 * b_bytes);
              const int k0 = q * p.o.d + c * BK;
              tma_load_4d_pair(sB, &tmW, fb, n0, k0, 0, 0);
              if (half_n > 64) tma_load_4d_pair(sB + kMnBlock, &tmW, fb, n0 + 64, k0, 0, 0);
              if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok) tell_peer(abort_flag);
      }
    } else if (warp == 1 && leader) {
      // ---------------------------------------------------------------- MMA issuer (the warp converged, one elected lane issues)
      uint32_t elected;
      asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(elected));
      const bool issuer = elected != 0;
      // in 16-byte units: from part to part, and 16 of K further
      const uint32_t a_part = (GRAD ? BK * 128u : BM * 64u) >> 4, b_part = (BK * 128u) >> 4;
      const uint32_t a_k = (GRAD ? 2048u : 32u) >> 4, b_k = 2048u >> 4;
      const uint64_t a0 = GRAD ? make_desc(base, kMnBlock, 1024u) : make_desc64(base);
      const uint64_t b0 = make_desc(base + kABytes, kMnBlock, 1024u);
      int stage = 0, set = 0;
      uint32_t phase = 0, set_phase = 0;
      bool ok = true, stage_ready = false;
      for (int item = first_item; item < items && ok; item += item_step) {
        const int n_tile = item_n_tile(item);
        const uint32_t idesc = (1u << 4) /*fp32 accumulate*/ | (1u << 7) | (1u << 10) /*bf16*/ | ((uint32_t)GRAD << 15) | (1u << 16) |
                               ((uint32_t)(n_tile >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24);
        int n_kb = p.chunks * p.blocks, group = n_kb;
        if (GRAD) {
          const Unit u = unit_of(p, item);
          n_kb = u.kb_hi - u.kb_lo;
          group = p.group;
        }
        for (int kb = 0; kb < n_kb && ok; kb += group) {
          if (!mbar_wait(acce_bar(set), set_phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
          const int end = min(n_kb, kb + group);
          const uint32_t d_high = tmem_base + (uint32_t)(set * kAccs * widest), d_small = FINE ? d_high : d_high + (uint32_t)n_tile;
          for (int i = kb; i < end; ++i) {
            if (!stage_ready && !mbar_wait(full_bar(stage), phase, abort_flag, p.status)) { ok = false; break; }
            tc_fence_after();
            const int next_stage = stage + 1 == kStages ? 0 : stage + 1;
            const uint32_t next_phase = next_stage == 0 ? phase ^ 1u : phase;
            // only tested here, so that nothing is waited for between two blocks' instructions (gemm_tc.cu)
            const bool peek = mbar_test_wait(full_bar(next_stage), next_phase);
            if (issuer) {
              const uint64_t ad = a0 + (uint64_t)((uint32_t)stage * (kStageBytes >> 4)), bd = b0 + (uint64_t)((uint32_t)stage * (kStageBytes >> 4));
              constexpr uint32_t qa[6] = {2, 0, 1, 1, 0, 0}, qb[6] = {0, 2, 1, 0, 1, 0};  // parts, 0 = high: the small terms first
#pragma unroll
              for (int q = 0; q < 6; ++q)
#pragma unroll
                for (int k = 0; k < 2; ++k)
                  tc_mma_pair(q < 5 ? d_small : d_high, ad + (uint64_t)(qa[q] * a_part + k * a_k), bd + (uint64_t)(qb[q] * b_part + k * b_k), idesc,
                              i > kb || k > 0 || (q > 0 && (FINE || q < 5)));
              tc_commit_pair(empty_bar(stage));
              if (i + 1 == end) tc_commit_pair(accf_bar(set));
            }
            stage_ready = peek;
            stage = next_stage; phase = next_phase;
          }
          if (++set == sets) { set = 0; set_phase ^= 1u; }
        }
      }
      if (!ok) {  // let issued MMAs finish before the tensor memory is freed
        if (issuer) tc_commit_pair(drain_bar);
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(drain_bar, 0) && global_ns() - t0 < 100000000ull) {
        }
        tell_peer(abort_flag);
      }
    }
  } else if (warp < 8) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    // ------------------------------------------------------------------ epilogue
    const int ew = warp - 4;  // quarter of the tile's rows
    const uint32_t buf0 = epi_base + ew * kEpiBufs * kFloatBuf;
    int set = 0, buf = 0;
    uint32_t set_phase = 0, e_phase = 0, e_flight = 0;  // e_phase, e_flight: a bit per buffer (e_flight: lane 0, a load of E is in flight)
    bool ok = true;
    auto put_floats = [&](uint32_t at, const float* v) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        st_shared16(swz(at, lane, u), make_uint4(__float_as_uint(v[4 * u]), __float_as_uint(v[4 * u + 1]), __float_as_uint(v[4 * u + 2]),
                                                 __float_as_uint(v[4 * u + 3])));
    };
    for (int item = first_item; item < items && ok; item += item_step) {
      Unit u;
      int n_kb, group, N, n_tile;
      if (GRAD) {
        u = unit_of(p, item);
        n_kb = u.kb_hi - u.kb_lo;
        group = p.group;
        n_tile = p.seg[u.segment].n_tile;
        N = p.seg[u.segment].N;
      } else {
        u.m0 = (item / p.n_tiles) * TILE_M;
        u.n0 = (item % p.n_tiles) * p.n_tile;
        u.segment = u.split = 0;
        u.kb_lo = u.kb_hi = 0;
        n_kb = group = 1;
        n_tile = p.n_tile;
        N = p.N;
      }
      const int row0 = u.m0 + (int)rank * BM + ew * 32;
      const int chunks = min(n_tile, (N - u.n0 + 31) / 32 * 32) / 32;
      const CUtensorMap* out = GRAD && u.segment ? &tmD1 : &tmD;
      int set_z = GRAD ? u.split * p.sets_per_split : 0, in_set = 0;  // the set of partial sums, and how many sums it has
      for (int kb = 0; kb < n_kb && ok; kb += group) {
        auto load_e = [&](int c, int to) {  // lane 0
          mbar_expect_tx(epi_bar(ew, to), kFloatBuf);
          tma_load_3d(buf0 + to * kFloatBuf, &tmE, epi_bar(ew, to), u.n0 + c * 32, row0, 0);
          e_flight |= 1u << to;
        };
        if (lane == 0) {
          if (GRAD && !FINE) tma_store_wait_all();  // the sums that these are added to have been written
          else tma_store_wait_read();
          if (!GRAD && p.has_e) {  // (tiles of 256 columns hold up the products until the epilogue has read them)
            for (int c = kEpiBufs - 1; c < chunks; ++c) tma_prefetch_3d(&tmE, u.n0 + c * 32, row0, 0);
            for (int c = 0; c < min(chunks, kEpiBufs - 1); ++c) load_e(c, buf + c >= kEpiBufs ? buf + c - kEpiBufs : buf + c);
          }
        }
        __syncwarp();
        if (!mbar_wait(accf_bar(set), set_phase, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tsrc = tmem_base + ((uint32_t)(ew * 32) << 16) + (uint32_t)(set * kAccs * widest);
        float v[2][32], w[2][32];
        // the second accumulator, or what the set's sums are so far
        const uint32_t tmore = FINE ? tmem_base + ((uint32_t)(ew * 32) << 16) + (uint32_t)(sets * widest) : tsrc + n_tile;
        const bool keep = FINE && in_set + 1 < p.merge && kb + group < n_kb;  // the set goes on
        tc_ld32_async(tsrc, v[0]);
        if (!FINE || in_set > 0) tc_ld32_async(tmore, w[0]);
        auto chunk = [&](int c, float (&s)[32], float (&t)[32], float (&s_next)[32], float (&t_next)[32]) {
          tc_ld_wait();
          if (c + 1 < chunks) {
            tc_ld32_async(tsrc + (c + 1) * 32, s_next);
            if (!FINE || in_set > 0) tc_ld32_async(tmore + (c + 1) * 32, t_next);
          }
          const int col = u.n0 + c * 32;
          auto release = [&]() {  // the accumulators, before the last chunk goes out
            if (c + 1 < chunks) return;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_cta(acce_bar(set), 0));
          };
          if (FINE) {
            const float factor = ((3 * kb + lane) & 7) < 3 ? kUnscale * kOneUp : kUnscale;
#pragma unroll
            for (int i = 0; i < 32; ++i) s[i] = fmaf(s[i], factor, in_set > 0 ? t[i] : 0.0f);
            if (keep) {
              release();
              tc_st32(tmore + c * 32, s);
              return;
            }
            // sums of a few products, where a truncation or a part left out counts as much as a rounding: as plain float sums (refine)
            if (p.o.rows < kFewProducts)
#pragma unroll
              for (int i = 0; i < 32; ++i) s[i] = __uint_as_float(0x7fffffffu);
          }
          f2 all = 0;  // not finite if one of the sums is not
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            f2 one = pack2(__float_as_uint(s[i]), __float_as_uint(s[i + 1]));
            if (!FINE) {
              one = mul2(add2(one, pack2(__float_as_uint(t[i]), __float_as_uint(t[i + 1]))), pack2(__float_as_uint(kUnscale), __float_as_uint(kUnscale)));
              s[i] = __uint_as_float((uint32_t)one);
              s[i + 1] = __uint_as_float((uint32_t)(one >> 32));
            }
            all = add2(all, one);
          }
          const bool doubt = !(fabsf(__uint_as_float((uint32_t)all) + __uint_as_float((uint32_t)(all >> 32))) < __uint_as_float(0x7f800000u));
          if (__any_sync(0xffffffffu, doubt)) {
            tc_ld_wait();
            if (GRAD) {
              const int first = u.kb_lo + (FINE ? kb - in_set * group : kb);  // (the whole set's, where it is one sum)
              refine_grad<KIND>(p, u.segment, row0 + lane, col, first * BK, min((int)p.o.rows, min(u.kb_hi, u.kb_lo + kb + group) * BK), s);
            } else {
              refine_vjp<KIND>(p, row0 + lane, col, s);
            }
            const int again = min(c + 1, chunks - 1) * 32;  // (so that the next chunk need not be held in registers meanwhile)
            tc_ld32(tsrc + again, s_next);
            if (!FINE || in_set > 0) tc_ld32(tmore + again, t_next);
          }
          release();
          const uint32_t at = buf0 + buf * kFloatBuf;
          if (!GRAD && p.has_e) {
            if (!mbar_wait(epi_bar(ew, buf), (e_phase >> buf) & 1u, abort_flag, p.status)) { ok = false; return; }
            e_phase ^= 1u << buf;
            e_flight &= ~(1u << buf);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const uint4 raw = ld_shared16(swz(at, lane, k));
              s[4 * k] += __uint_as_float(raw.x);
              s[4 * k + 1] += __uint_as_float(raw.y);
              s[4 * k + 2] += __uint_as_float(raw.z);
              s[4 * k + 3] += __uint_as_float(raw.w);
            }
          } else {
            if (lane == 0) tma_store_wait_read<kEpiBufs - 1>();
            __syncwarp();
          }
          put_floats(at, s);
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (GRAD && !FINE && in_set > 0) tma_add_3d(out, at, col, row0, set_z);
            else tma_store_3d(out, at, col, row0, set_z);
            if (!GRAD && p.has_e && c + kEpiBufs - 1 < chunks) {  // into the buffer that the chunk before this one went out from
              tma_store_wait_read<1>();
              load_e(c + kEpiBufs - 1, buf == 0 ? kEpiBufs - 1 : buf - 1);
            }
          }
          __syncwarp();
          if (++buf == kEpiBufs) buf = 0;
        };
#pragma unroll 1
        for (int c = 0; c < chunks && ok; c += 2) {
          chunk(c, v[0], w[0], v[1], w[1]);
          if (ok && c + 1 < chunks) chunk(c + 1, v[1], w[1], v[0], w[0]);
        }
        if (keep) tc_st_wait();
        if (GRAD && ++in_set == p.merge) { in_set = 0; ++set_z; }
        if (++set == sets) { set = 0; set_phase ^= 1u; }
      }
    }
    if (lane == 0) {
      tma_store_wait_all();
      for (int i = 0; i < kEpiBufs; ++i)  // only after an abort: do not leave with a copy into our buffers in flight
        if (e_flight & (1u << i)) {
          const uint64_t t0 = global_ns();
          while (!mbar_try_wait(epi_bar(ew, i), (e_phase >> i) & 1u) && global_ns() - t0 < 100000000ull) {
          }
        }
    }
    if (!ok) tell_peer(abort_flag);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsLoad));
    // ------------------------------------------------------------------ operands
    const int t = threadIdx.x - 256, d = p.o.d;
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    auto begin = [&]() { return mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.status); };
    auto done = [&]() {
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_cta(full_bar(stage), 0));
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    };
    if (!GRAD) {
      // this thread: four neighbouring channels (unit of 8 of a chunk) of rows r, r + 32, r + 64, r + 96
      const int unit = t & 7, r = t >> 3;
      auto store = [&](Four (&v)[4], int chunk) {
        if (chunk * BK + unit * 4 >= d)
#pragma unroll
          for (int i = 0; i < 4; ++i) v[i] = {0, 0};
        const uint32_t at = base + stage * kStageBytes + r * 64 + (((uint32_t)(unit >> 1) ^ ((r >> 1) & 3)) << 4) + (unit & 1) * 8;
#pragma unroll
        for (int i = 0; i < 4; ++i) store_parts(at + i * 32 * 64, BM * 64u, v[i]);  // (32 rows on the swizzle is the same)
      };
      // the chunks of all of this CTA's tiles as one sequence
      struct Cursor {
        int item, c;
      };
      auto next_of = [&](Cursor k) {
        if (++k.c == p.chunks) {
          k.c = 0;
          k.item += item_step;
        }
        return k;
      };
      const int last_row = (int)p.o.rows - 1;
      const int g_w = KIND == HBP_BLOCK_LSTM ? 2 * d : d, c_w = KIND == HBP_BLOCK_LSTM ? 5 * d : KIND == HBP_BLOCK_GRU ? 4 * d : d;
      auto row0_of = [&](const Cursor& k) { return (int64_t)(k.item / p.n_tiles) * TILE_M + (int)rank * BM; };
      // (Rows and columns past the end: the last ones again, without a condition.  Those rows of the result are not stored; of the
      // columns store() makes zeros.)
      auto loads = [&](const Cursor& k, const float* src, int w, int off, Four (&v)[4]) {
        const float* at = src + (off + min(k.c * BK + unit * 4, d - 4));
        const int row = (k.item / p.n_tiles) * TILE_M + (int)rank * BM + r;
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = load4(at + (int64_t)min(row + 32 * i, last_row) * w);
      };
      if (KIND == HBP_BLOCK_RNN_TANH) {
        constexpr int S = 3;
        Four g[S][4], c[S][4];
        Cursor ld = {first_item, 0}, at = ld;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          loads(ld, p.o.g, g_w, 0, g[s]);
          loads(ld, p.o.coef, c_w, 0, c[s]);
          ld = next_of(ld);
        }
        while (at.item < items && ok) {
#pragma unroll
          for (int s = 0; s < S; ++s) {
            if (at.item >= items || !ok) break;
            if (!begin()) { ok = false; break; }
            Four v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = times(scaled(g[s][i]), c[s][i]);
            loads(ld, p.o.g, g_w, 0, g[s]);
            loads(ld, p.o.coef, c_w, 0, c[s]);
            store(v, at.c);
            done();
            ld = next_of(ld);
            at = next_of(at);
          }
        }
      } else if (KIND == HBP_BLOCK_GRU) {
        Four g[4], g_next[4], c[3][4];
        Cursor at = {first_item, 0};
        loads(at, p.o.g, g_w, 0, g_next);
#pragma unroll
        for (int q = 0; q < 3; ++q) loads(at, p.o.coef, c_w, q * d, c[q]);
        while (at.item < items && ok) {
          const Cursor next = next_of(at);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            if (!begin()) { ok = false; break; }
            if (q == 0) {
#pragma unroll
              for (int i = 0; i < 4; ++i) g[i] = scaled(g_next[i]);
              loads(next, p.o.g, g_w, 0, g_next);
            }
            Four v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = times(g[i], c[q][i]);
            loads(next, p.o.coef, c_w, q * d, c[q]);
            store(v, at.c);
            done();
          }
          at = next;
        }
      } else {
        Four gc[4], gh[4], ch[4], c[4][4];  // gc: g_c as loaded, then t
        Cursor at = {first_item, 0};
        loads(at, p.o.g, g_w, 0, gc);
        loads(at, p.o.g, g_w, d, gh);
        loads(at, p.o.coef, c_w, 4 * d, ch);
#pragma unroll
        for (int q = 0; q < 4; ++q) loads(at, p.o.coef, c_w, q * d, c[q]);
        while (at.item < items && ok) {
          const Cursor next = next_of(at);
          if (p.uc && at.item % p.n_tiles == 0) {  // u_c = f g_h c_h (+ delta), from the tiles of the first columns
            const int64_t row = row0_of(at) + r;
            const int col = at.c * BK + unit * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (col < d && row + 32 * i < p.o.rows) {
                const int64_t e = (row + 32 * i) * 2 * d + col;
                Four v = times(times(load4(p.fg + e), gh[i]), ch[i]);
                if (p.delta_c) {
                  const Four dl = load4(p.delta_c + e);
                  v = {add2(v.a, dl.a), add2(v.b, dl.b)};
                }
                *reinterpret_cast<ulonglong2*>(p.uc + e) = make_ulonglong2(v.a, v.b);
              }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            gc[i] = scaled({fma2(gh[i].a, ch[i].a, gc[i].a), fma2(gh[i].b, ch[i].b, gc[i].b)});
            gh[i] = scaled(gh[i]);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (!begin()) { ok = false; break; }
            {
              Four v[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) v[i] = times(q == 3 ? gh[i] : gc[i], c[q][i]);
              store(v, at.c);
            }
            done();
            loads(next, p.o.coef, c_w, q * d, c[q]);
            if (q == 2) {
              loads(next, p.o.g, g_w, 0, gc);
              loads(next, p.o.coef, c_w, 4 * d, ch);
            }
            if (q == 3) loads(next, p.o.g, g_w, d, gh);
          }
          at = next;
        }
      }
    } else {
      // this thread: four neighbouring columns of either operand, rows w, w + 8, w + 16, w + 24 of a block
      const int w = t >> 5;
      const uint32_t off = (uint32_t)(lane >> 4) * kMnBlock + w * 128 + (((((uint32_t)lane & 15u) >> 1) ^ (uint32_t)w) << 4) + (lane & 1) * 8;
      auto store = [&](uint32_t tile, const Four (&v)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) store_parts(tile + off + i * 8 * 128, BK * 128u, v[i]);  // (8 rows on the swizzle is the same)
      };
      for (int item = first_item; item < items && ok; item += item_step) {
        const Unit u = unit_of(p, item);
        const Params::Segment& sg = p.seg[u.segment];
        // columns past the end: the last ones again (those rows and columns of the result are not stored)
        const int m = min(u.m0 + (int)rank * BM + lane * 4, p.M - 4), n = min(u.n0 + (int)rank * (sg.n_tile / 2) + lane * 4, sg.N - 4);
        const bool has_n = lane * 4 < sg.n_tile / 2;
        const int q = coef_block<KIND>(m / d, u.segment), c = m % d;
        const bool input = p.both && n >= d;
        const Params::Segment& from = p.seg[input ? 1 : u.segment];
        const float* b_at = from.B + (n - (input ? d : 0));
        const int b_ld = (int)from.ldb;
        const bool b_vec = from.vec != 0;
        const int row_lo = u.kb_lo * BK + w, last_row = (int)p.o.rows - 1;
        // block kb's share of a matrix with rows of `stride` (past the last row: that row again, without a condition; store_a makes zeros
        // of the operand's)
        auto load = [&](int kb, const float* src, int stride, Four (&v)[4]) {
          const int row = row_lo + kb * BK;
#pragma unroll
          for (int i = 0; i < 4; ++i) v[i] = load4(src + (int64_t)min(row + 8 * i, last_row) * stride);
        };
        auto load_b = [&](int kb, Four (&v)[4]) {
          if (b_vec) return load(kb, b_at, b_ld, v);
#pragma unroll
          for (int i = 0; i < 4; ++i) {  // not 16-byte aligned
            const float* at = b_at + (int64_t)min(row_lo + kb * BK + 8 * i, last_row) * b_ld;
            v[i] = {pack2(__float_as_uint(at[0]), __float_as_uint(at[1])), pack2(__float_as_uint(at[2]), __float_as_uint(at[3]))};
          }
        };
        auto store_a = [&](int kb, uint32_t tile, Four (&v)[4]) {
          const int row = row_lo + kb * BK;
          if (row - w + BK > last_row + 1)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (row + 8 * i > last_row) v[i] = {0, 0};
          store(tile, v);
        };
        const int n_kb = u.kb_hi - u.kb_lo;
        if (KIND != HBP_BLOCK_LSTM) {
          constexpr int S = 2;
          const int c_w = KIND == HBP_BLOCK_GRU ? 4 * d : d;
          const float *g_at = p.o.g + c, *c_at = p.o.coef + (KIND == HBP_BLOCK_GRU ? q * d : 0) + c;
          Four g[S][4], cf[S][4], b[S][4];
#pragma unroll
          for (int s = 0; s < S; ++s) {
            load(s, g_at, d, g[s]);
            load(s, c_at, c_w, cf[s]);
            load_b(s, b[s]);
          }
          for (int kb = 0; kb < n_kb && ok; kb += S) {
#pragma unroll
            for (int s = 0; s < S; ++s) {
              if (kb + s >= n_kb) break;
              if (!begin()) { ok = false; break; }
              const uint32_t tile = base + stage * kStageBytes;
              Four v[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) v[i] = times(scaled(g[s][i]), cf[s][i]);
              load(kb + s + S, g_at, d, g[s]);
              load(kb + s + S, c_at, c_w, cf[s]);
              store_a(kb + s, tile, v);
              if (has_n) store(tile + kABytes, b[s]);
              load_b(kb + s + S, b[s]);
              done();
            }
          }
        } else {
          const bool with_t = q != 3;  // t c_q for the first three blocks, g_h c_o for the last
          const float *g_at = p.o.g + c, *c_at = p.o.coef + c;
          Four gc[4], gh[4], ch[4], cq[4], b[4];
          auto load_a = [&](int kb) {
            load(kb, g_at + d, 2 * d, gh);
            load(kb, c_at + q * d, 5 * d, cq);
            if (with_t) {
              load(kb, g_at, 2 * d, gc);
              load(kb, c_at + 4 * d, 5 * d, ch);
            }
          };
          load_a(0);
          load_b(0, b);
          for (int kb = 0; kb < n_kb; ++kb) {
            if (!begin()) { ok = false; break; }
            const uint32_t tile = base + stage * kStageBytes;
            Four v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              v[i] = gh[i];
              if (with_t) v[i] = {fma2(gh[i].a, ch[i].a, gc[i].a), fma2(gh[i].b, ch[i].b, gc[i].b)};
              v[i] = times(scaled(v[i]), cq[i]);
            }
            load_a(kb + 1);
            store_a(kb, tile, v);
            if (has_n) store(tile + kABytes, b);
            load_b(kb + 1, b);
            done();
          }
        }
      }
    }
    if (!ok) tell_peer(abort_flag);
  }

  tc_fence_before();
  cluster_sync();  // neither CTA leaves (or frees) while its peer may still read its tiles or signal its barriers
  if (warp == 1) {
    const int gave_up = *abort_flag;
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    if (!GRAD && gave_up) outlast_copies();
  }
}

// An even split of n columns into `tiles` tiles, a multiple of 32 wide.
int even_width(int n, int tiles) { return ((n + tiles - 1) / tiles + 31) / 32 * 32; }
// Width of the VJP's tiles: the least time over the waves of CTA pairs.  A k-block takes 2400 clocks at 256 columns and 1380 at 128,
// where forming the operand bounds it, so that narrower ones gain nothing (131072 x 512 x 512 in tiles of 256 and 128: 322 and 368 us;
// 32768 x 512 x 1536, 4 waves and 7: 219 and 208).
int vjp_tile_width(int n, int64_t m_tiles) {
  const int pairs = sm_count() / 2;
  int64_t best = 0;
  int width = 0;
  for (int tiles = (n + kMaxTileN - 1) / kMaxTileN; tiles <= (n + 127) / 128; ++tiles) {
    const int w = even_width(n, tiles);
    const int64_t cost = (m_tiles * ((n + w - 1) / w) + pairs - 1) / pairs * (w <= 128 ? 1380 : 360 + 8 * w);
    if (best == 0 || cost < best) {
      best = cost;
      width = w;
    }
  }
  return width;
}

// The partial sums [split][M][d + in] of products against states and inputs side by side, added in double in ascending order of the splits:
// dW [blocks d][d] and dU [blocks d][in].  The GRU's rows have four blocks, [c_r | c_z | c_nr | c_n]: dW leaves out the last, dU the third.
__global__ void __launch_bounds__(256) reduce_both_kernel(const float* __restrict__ partial, float* __restrict__ dW, float* __restrict__ dU, int splits,
                                                          int M, int d, int in, int gru) {
  chain_next();
  chain_wait();
  const int64_t elems = (int64_t)M * (d + in), i = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  const double s = reduce_eighths(partial + i, i < elems, splits, elems);
  if (threadIdx.x >= 32 || i >= elems) return;
  const int m = (int)(i / (d + in)), n = (int)(i % (d + in)), q = m / d;
  if (gru && q == (n < d ? 3 : 2)) return;
  if (n < d) dW[(int64_t)m * d + n] = (float)s;
  else dU[(int64_t)(gru && q == 3 ? m - d : m) * in + n - d] = (float)s;
}

template <int KIND, bool GRAD, bool FINE>
bool launch(Launcher& lc, int items, const CUtensorMap& w, const CUtensorMap& d0, const CUtensorMap& d1, const CUtensorMap& e, const Params& p) {
  static PerDevice<bool> attr_done;
  if (!attr_done.here()) {
    if (cudaFuncSetAttribute(gemm_cell_kernel<KIND, GRAD, FINE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    attr_done.here() = true;
  }
  const int pairs = sm_count() / 2;
  return try_launch_chained(lc, gemm_cell_kernel<KIND, GRAD, FINE>, dim3(2 * (items < pairs ? items : pairs)), THREADS, SMEM_BYTES, 2, w, d0, d1, e, p) ==
         cudaSuccess;
}
template <bool GRAD, bool FINE>
bool launch_kind(Launcher& lc, int items, const CUtensorMap& w, const CUtensorMap& d0, const CUtensorMap& d1, const CUtensorMap& e, const Params& p) {
  if (p.kind == HBP_BLOCK_RNN_TANH) return launch<HBP_BLOCK_RNN_TANH, GRAD, FINE>(lc, items, w, d0, d1, e, p);
  if (p.kind == HBP_BLOCK_GRU) return launch<HBP_BLOCK_GRU, GRAD, FINE>(lc, items, w, d0, d1, e, p);
  return launch<HBP_BLOCK_LSTM, GRAD, FINE>(lc, items, w, d0, d1, e, p);
}
// Rows of the operand whose sums stay as exact as sums of floats are (see the FINE form of the kernel).
bool fine_sums(int64_t rows) { return rows % 4 != 0; }
// Where states and inputs fit one tile's columns the operand is loaded and split once for both: the GRU's of four blocks then.
bool both_at_once(int d, int in) { return d + in <= kMaxTileN; }
int blocks_of(int kind) { return kind == HBP_BLOCK_RNN_TANH ? 1 : kind == HBP_BLOCK_GRU ? 3 : 4; }

}  // namespace

bool cell_vjp(Launcher& lc, int kind, const CellOperand& o, const Planes& W, const float* delta, float* out, int64_t ld, const float* fg,
              const float* delta_c, float* uc, int* status_word) {
  Params p = {};
  p.o = o;
  p.kind = kind;
  p.blocks = blocks_of(kind);
  p.W = W;
  p.N = o.d;
  const int64_t m_tiles = (o.rows + TILE_M - 1) / TILE_M;
  p.n_tile = vjp_tile_width(o.d, m_tiles);
  p.n_tiles = (o.d + p.n_tile - 1) / p.n_tile;
  if (o.rows > (int64_t)1 << 30 || m_tiles * p.n_tiles > (int64_t)1 << 30) return false;
  p.num_tiles = (int)m_tiles * p.n_tiles;
  p.chunks = (o.d + BK - 1) / BK;
  p.has_e = delta != nullptr;
  p.fg = fg;
  p.delta_c = delta_c;
  p.uc = uc;
  p.status = status_word;
  CUtensorMap tmW, tmD, tmE;
  if (!map_planes(&tmW, W, o.d, p.blocks * o.d, 1, 64, BK, CU_TENSOR_MAP_SWIZZLE_128B)) return false;
  if (!make_map_epi(&tmD, out, true, (int)o.rows, o.d, 1, ld, 0)) return false;
  tmE = tmD;
  if (delta && !make_map_epi(&tmE, delta, true, (int)o.rows, o.d, 1, ld, 0)) return false;
  return launch_kind<false, false>(lc, p.num_tiles, tmW, tmD, tmD, tmE, p);
}

bool cell_wgrad(Launcher& lc, int kind, const CellOperand& o, const float* H, int64_t ldh, const float* X, int in, float* dW, float* dU,
                float* partial, size_t partial_floats, int* status_word) {
  Params p = {};
  p.o = o;
  p.kind = kind;
  p.blocks = blocks_of(kind);
  p.both = both_at_once(o.d, in);
  const bool fine = fine_sums(o.rows);
  const int widest = fine ? kFineTileN : kMaxTileN;
  auto tile_width = [&](int n) { return even_width(n, (n + widest - 1) / widest); };
  p.M = (p.both && kind == HBP_BLOCK_GRU ? 4 : p.blocks) * o.d;
  p.status = status_word;
  const int m_tiles = (p.M + TILE_M - 1) / TILE_M, n0 = p.both ? o.d + in : o.d;
  p.seg[0] = {H, ldh, n0, tile_width(n0), m_tiles, 0, 1};
  p.seg[1] = {X, in, in, tile_width(in), p.both ? 0 : m_tiles, 0, ((uintptr_t)X & 15u) == 0};
  if (p.both) p.seg[1].n_tile = p.seg[0].n_tile;
  for (auto& s : p.seg) {
    s.n_tiles = (s.N + s.n_tile - 1) / s.n_tile;
    p.tiles += s.m_tiles * s.n_tiles;
  }
  if (o.rows > (int64_t)1 << 30) return false;
  p.k_blocks = (int)((o.rows + BK - 1) / BK);
  // As many splits of the rows as give the shortest longest queue of a CTA pair, four k-blocks at least in each (of those within
  // 5 % the fewest: every split is a set of partial sums).  A wide tile costs more than a narrow one only where the tensor core bounds it.
  const int64_t outputs = (int64_t)p.M * (o.d + in);
  const int pairs = sm_count() / 2;
  int64_t best = 0;
  for (int s = 1; s <= pairs && s * outputs <= (int64_t)partial_floats && (s == 1 || s * 4 <= p.k_blocks); ++s) {
    const int64_t per = (p.k_blocks + s - 1) / s, cost = ((int64_t)p.tiles * s + pairs - 1) / pairs * (per + 4);
    if (best == 0 || 100 * cost < 95 * best) {
      best = cost;
      p.splits = s;
    }
  }
  if (best == 0) return false;
  p.group = fine ? 1 : kDrainBlocks;
  const int per = (p.k_blocks + p.splits - 1) / p.splits, groups = (per + p.group - 1) / p.group;
  p.sets_per_split = fine ? (per + kFineSet - 1) / kFineSet : 1;
  while (p.sets_per_split > 1 && p.splits * p.sets_per_split * outputs > (int64_t)partial_floats) --p.sets_per_split;
  p.merge = (groups + p.sets_per_split - 1) / p.sets_per_split;
  p.per_split = fine ? p.sets_per_split * p.merge : per;
  p.splits = (p.k_blocks + p.per_split - 1) / p.per_split;
  const int set_blocks = p.merge * p.group, last = p.k_blocks - (p.splits - 1) * p.per_split;
  const int sets = (p.splits - 1) * p.sets_per_split + (last + set_blocks - 1) / set_blocks;
  CUtensorMap tmD0, tmD1;
  if (!make_map_epi(&tmD0, partial, true, p.M, n0, sets, n0, (int64_t)p.M * n0)) return false;
  if (p.both) {
    if (!(fine ? launch_kind<true, true>(lc, p.tiles * p.splits, tmD0, tmD0, tmD0, tmD0, p)
               : launch_kind<true, false>(lc, p.tiles * p.splits, tmD0, tmD0, tmD0, tmD0, p)))
      return false;
    launch_chained(lc, reduce_both_kernel, dim3((unsigned)((outputs + 31) / 32)), 256, 0, 1, (const float*)partial, dW, dU, sets, p.M, o.d, in,
                   (int)(kind == HBP_BLOCK_GRU));
    return true;
  }
  float* part1 = partial + (int64_t)sets * p.M * o.d;
  if (!make_map_epi(&tmD1, part1, true, p.M, in, sets, in, (int64_t)p.M * in)) return false;
  if (!(fine ? launch_kind<true, true>(lc, p.tiles * p.splits, tmD0, tmD0, tmD1, tmD0, p)
             : launch_kind<true, false>(lc, p.tiles * p.splits, tmD0, tmD0, tmD1, tmD0, p)))
    return false;
  reduce_splitk(lc, partial, dW, sets, (int64_t)p.M * o.d);
  reduce_splitk(lc, part1, dU, sets, (int64_t)p.M * in);
  return true;
}

}  // namespace hbp
