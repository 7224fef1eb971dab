// Float GEMM on the tensor cores for operands that lie in memory as three bf16 planes each (float residual MLP stacks):
//   D(m, n) = sum_k A(m, k) B(n, k), six bf16 products of parts (all but the three below 2^-26 of the whole), float epilogues.
//
// The arithmetic is gemm_f32.cu's: per 32 of K the six products, the small ones first, into a fresh accumulator; each finished
// accumulator added to float sums in registers, three of eight blocks of a row counted 2^-23 more.  There every tile splits its
// operands again, by warps that load 32 floats at a time, and those warps bound it (a quarter of the tensor rate).  Here an
// operand is split once, by the kernel that produces it where there is one, and the parts arrive by TMA, either way round
// (K-major rows of 64 bytes, or MN-major blocks of 64 elements x 32 of K).
//
// CTA pairs on 256 x n_tile tiles (n_tile = 32 .. 192, chosen by gemm_parts), persistent, 384 threads:
//   warps 0, 2  TMA producers of A and of B (one lane each: a copy takes its issuer 100 clocks): three to five stages of
//               {A 128 x 32, B n_tile/2 x 32} x 3 parts, 48 KB at most
//   warp 1      MMA issuer (one lane of the even CTA): 12 x tcgen05.mma 256 x n_tile x 16 per stage, into the next of two to
//               four accumulators
//   warps 4..11 add the accumulators up (two warps per 32 rows, up to three chunks of 32 columns each) and run the epilogue
//               through 10 KB of staging per warp: every global access is a TMA tile copy
// 1900 x 1560 x 520, 12 at once: 350 us in gemm_f32.cu's kernel, 222 here with the product by gelu' and the result in parts
// (540 there); 1900 x 520 x 1560 418 -> 170; weight gradients of both 530 -> 210 to 218; one layer's 1900 x 1560 x 520 with GELU
// 53 -> 28, 1900 x 520 x 1560 61 -> 25.  At the tensor rate these take 135, 127, 137 to 160, 17 and 14.  What is left: the
// epilogue (a third of the short contraction's time: the warps that hold the sums run it), and for narrow tiles the issue of 12
// instructions and 4 commits per 32 of K (340 clocks).  Before the accumulators were handed back without a cluster-scope release
// the adding warps took 1800 clocks a block instead of 290, and all of it 3570 us instead of 2077.
#include <type_traits>

#include "float_parts.cuh"
#include "ring_drain.cuh"
#include "tc_common.cuh"

namespace hbp {

using namespace tc;

namespace {

constexpr int BM = 128, BK = 32, TILE_M = 2 * BM, kMaxTileN = 192;
constexpr int kMaxStages = 5, kMaxAcc = 4;
constexpr uint32_t kABytes = 3 * BM * BK * 2, kRingBytes = 6 * kABytes;  // 144 KB: three stages of the widest tile
constexpr uint32_t kMnBlock = 3 * BK * 128;  // one MN-major block of 64 elements: three parts of 32 rows of 128 bytes
constexpr int EPI_WARPS = 8, THREADS = 128 + 32 * EPI_WARPS;
// 384 threads start with 168 registers each, 64512; the first warpgroup keeps 56 a thread and the two others take 224:
// 128 x 56 + 256 x 224 = 64512
constexpr int kRegsFew = 56, kRegsMany = 224;
constexpr uint32_t kFloatBuf = 4096, kPartBuf = 3 * 32 * 64, kEpiBytes = kFloatBuf + kPartBuf;
constexpr uint32_t TMEM_COLS = 512;
constexpr int SMEM_BYTES = (int)kRingBytes + EPI_WARPS * (int)kEpiBytes + 1024 /*alignment*/ + 512 /*barriers*/;

struct Params {
  PartsGemm g;
  int m_tiles, n_tiles, num_tiles, k_blocks, n_tile, n_acc, stages;
  uint32_t b_bytes;  // of one stage and CTA
  int direct;        // D is not 16-byte aligned: stored element by element
  int* status;
};

__device__ __forceinline__ float part_value(const Planes& P, int64_t at) {
  return __bfloat162float(P.p[at]) + (__bfloat162float(P.p[at + P.plane]) + __bfloat162float(P.p[at + 2 * P.plane]));
}
// Sums that the parts may not give as the operands would: infinite or NaN ones (an infinity times a part that is zero is NaN).
// One warp's 32 x 32 outputs again, as plain float sums in ascending order of k of the operands themselves.
__device__ __forceinline__ void refine(const PartsGemm& g, int b, int row, int col0, float (&sum)[32]) {
  const int lane = threadIdx.x & 31;
  const int64_t ar = g.a_mn ? 1 : g.A.ld, ak = g.a_mn ? g.A.ld : 1, br = g.b_mn ? 1 : g.B.ld, bk = g.b_mn ? g.B.ld : 1;
  float acc[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = 0.0f;
#pragma unroll 1
  for (int k = 0; k < g.K; ++k) {
    const float a = row < g.M ? part_value(g.A, b * g.A.sb + row * ar + k * ak) : 0.0f;
    const float mine = col0 + lane < g.N ? part_value(g.B, b * g.B.sb + (col0 + lane) * br + k * bk) : 0.0f;
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = fmaf(a, __shfl_sync(0xffffffffu, mine, i), acc[i]);
  }
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (!(fabsf(sum[i]) < __uint_as_float(0x7f800000u))) sum[i] = acc[i];
}

__global__ void __launch_bounds__(THREADS, 1)
gemm_parts_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ CUtensorMap tmD, const __grid_constant__ CUtensorMap tmD2,
                  const __grid_constant__ CUtensorMap tmE, const __grid_constant__ CUtensorMap tmP, const __grid_constant__ Params p) {
  const PartsGemm& g = p.g;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int first_tile = (int)(blockIdx.x >> 1), tile_step = (int)(gridDim.x >> 1);
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t epi_base = base + kRingBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + (base - smem_u32(smem_raw)) + kRingBytes + EPI_WARPS * kEpiBytes);
  const uint32_t bar0 = smem_u32(bars);
  const int stages = p.stages;
  const uint32_t stage_bytes = kABytes + p.b_bytes;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
  auto accf_bar = [&](int a) { return bar0 + 8u * (2 * kMaxStages + a); };
  auto acce_bar = [&](int a) { return bar0 + 8u * (2 * kMaxStages + kMaxAcc + a); };
  const uint32_t drain_bar = bar0 + 8u * (2 * kMaxStages + 2 * kMaxAcc);
  auto epi_bar = [&](int w) { return bar0 + 8u * (2 * kMaxStages + 2 * kMaxAcc + 1 + w); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 2 * kMaxAcc + 1 + EPI_WARPS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < kMaxAcc; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), 2 * EPI_WARPS);  // both CTAs' warps arrive at the leader
    }
    mbar_init(drain_bar, 1);
    for (int w = 0; w < EPI_WARPS; ++w) mbar_init(epi_bar(w), 1);
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
  const int tiles_per_batch = p.m_tiles * p.n_tiles, half_n = p.n_tile / 2;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsFew));
    if (warp == 0 || warp == 2) {
      // ---------------------------------------------------------------- TMA producers
      if (lane == 0) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = first_tile; tile < p.num_tiles && ok; tile += tile_step) {
          const int b = tile / tiles_per_batch, r = tile % tiles_per_batch;
          const int m0 = (r / p.n_tiles) * TILE_M + (int)rank * BM, n0 = (r % p.n_tiles) * p.n_tile + (int)rank * half_n;
          for (int kb = 0; kb < p.k_blocks; ++kb) {
            if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
            const uint32_t sA = base + stage * stage_bytes, sB = sA + kABytes, fb = map_to_cta(full_bar(stage), 0);
            const int k0 = kb * BK;
            if (warp == 0) {
              if (leader) mbar_expect_tx(full_bar(stage), 2 * stage_bytes);
              if (g.a_mn) {
                tma_load_4d_pair(sA, &tmA, fb, m0, k0, b, 0);
                tma_load_4d_pair(sA + kMnBlock, &tmA, fb, m0 + 64, k0, b, 0);
              } else {
                tma_load_4d_pair(sA, &tmA, fb, k0, m0, b, 0);
              }
            } else if (g.b_mn) {
              tma_load_4d_pair(sB, &tmB, fb, n0, k0, b, 0);
              if (half_n > 64) tma_load_4d_pair(sB + kMnBlock, &tmB, fb, n0 + 64, k0, b, 0);
            } else {
              tma_load_4d_pair(sB, &tmB, fb, k0, n0, b, 0);
            }
            if (++stage == stages) { stage = 0; phase ^= 1u; }
          }
        }
      }
    } else if (warp == 1 && leader) {
      // ---------------------------------------------------------------- MMA issuer (the warp converged, one elected lane issues)
      uint32_t elected;
      asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(elected));
      const bool issuer = elected != 0;
      const uint32_t idesc = (1u << 4) /*fp32 accumulate*/ | (1u << 7) | (1u << 10) /*bf16*/ | ((uint32_t)g.a_mn << 15) |
                             ((uint32_t)g.b_mn << 16) | ((uint32_t)(p.n_tile >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24);
      // in 16-byte units: from part to part, and 16 of K further
      const uint32_t a_part = (g.a_mn ? BK * 128u : BM * 64u) >> 4, b_part = (g.b_mn ? BK * 128u : (uint32_t)half_n * 64u) >> 4;
      const uint32_t a_k = (g.a_mn ? 2048u : 32u) >> 4, b_k = (g.b_mn ? 2048u : 32u) >> 4;
      const uint64_t a0 = g.a_mn ? make_desc(base, kMnBlock, 1024u) : make_desc64(base);
      const uint64_t b0 = g.b_mn ? make_desc(base + kABytes, kMnBlock, 1024u) : make_desc64(base + kABytes);
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true, stage_ready = false, acc_ready = false;
      for (int tile = first_tile; tile < p.num_tiles && ok; tile += tile_step) {
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          if (!acc_ready && !mbar_wait(acce_bar(acc), acc_phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
          if (!stage_ready && !mbar_wait(full_bar(stage), phase, abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          const int next_stage = stage + 1 == stages ? 0 : stage + 1, next_acc = acc + 1 == p.n_acc ? 0 : acc + 1;
          const uint32_t next_phase = next_stage == 0 ? phase ^ 1u : phase, next_acc_phase = next_acc == 0 ? acc_phase ^ 1u : acc_phase;
          // only tested here, so that nothing is waited for between two blocks' instructions (gemm_tc.cu)
          const bool peek = mbar_test_wait(full_bar(next_stage), next_phase);
          const bool peek_acc = mbar_test_wait(acce_bar(next_acc), next_acc_phase ^ 1u);
          if (issuer) {
            const uint32_t tmem_d = tmem_base + (uint32_t)(acc * p.n_tile);
            const uint64_t ad = a0 + (uint64_t)((uint32_t)stage * (stage_bytes >> 4)), bd = b0 + (uint64_t)((uint32_t)stage * (stage_bytes >> 4));
            constexpr uint32_t qa[6] = {2, 0, 1, 1, 0, 0}, qb[6] = {0, 2, 1, 0, 1, 0};  // parts, 0 = high: the small terms first
#pragma unroll
            for (int q = 0; q < 6; ++q)
#pragma unroll
              for (int k = 0; k < 2; ++k)
                tc_mma_pair(tmem_d, ad + (uint64_t)(qa[q] * a_part + k * a_k), bd + (uint64_t)(qb[q] * b_part + k * b_k), idesc, q + k > 0);
            tc_commit_pair(empty_bar(stage));
            tc_commit_pair(accf_bar(acc));
          }
          stage_ready = peek; acc_ready = peek_acc;
          stage = next_stage; phase = next_phase;
          acc = next_acc; acc_phase = next_acc_phase;
        }
      }
      if (!ok) {  // let issued MMAs finish before the tensor memory is freed
        if (issuer) tc_commit_pair(drain_bar);
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(drain_bar, 0) && global_ns() - t0 < 100000000ull) {
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsMany));
    // ------------------------------------------------------------------ sums and epilogue
    const int quarter = warp & 3, half = (warp - 4) >> 2, ew = warp - 4;
    const uint32_t fbuf = epi_base + ew * kEpiBytes, pbuf = fbuf + kFloatBuf, ebar = epi_bar(ew);
    const int chunks = p.n_tile / 32, c_lo = half ? (chunks + 1) / 2 : 0, n_c = half ? chunks / 2 : (chunks + 1) / 2;
    const bool has_e = g.epi == EPI_MUL || g.epi == EPI_RESID;
    uint32_t e_phase = 0;
    bool e_pending = false, ok = true;  // e_pending: lane 0, a load of E is in flight
    int acc = 0;
    uint32_t acc_phase = 0;
    // 32 rows x 128 bytes of floats, swizzled; 3 x 32 rows x 64 bytes of parts, swizzled
    auto put_floats = [&](uint32_t buf, const float* v) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        st_shared16(swz(buf, lane, u), make_uint4(__float_as_uint(v[4 * u]), __float_as_uint(v[4 * u + 1]), __float_as_uint(v[4 * u + 2]),
                                                  __float_as_uint(v[4 * u + 3])));
    };
    auto put_parts = [&](const float* v) {
      uint32_t top = 0;  // one test for all (a branch per pair would keep their chains apart)
#pragma unroll
      for (int i = 0; i < 32; ++i) top = max(top, __float_as_uint(v[i]) & 0x7fffffffu);
      auto put = [&](auto plain) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t w[3][4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (plain.value) split_plain2(v[8 * u + 2 * i], v[8 * u + 2 * i + 1], w[0][i], w[1][i], w[2][i]);
            else split_parts2(v[8 * u + 2 * i], v[8 * u + 2 * i + 1], w[0][i], w[1][i], w[2][i]);
          }
          const uint32_t at = pbuf + lane * 64 + ((u ^ ((lane >> 1) & 3)) << 4);
#pragma unroll
          for (int q = 0; q < 3; ++q) st_shared16(at + q * 2048u, make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]));
        }
      };
      if (top < kPlainParts) put(std::true_type());
      else put(std::false_type());
    };
    auto free_buffers = [&]() {  // until this warp's copies out have been read
      if (lane == 0) tma_store_wait_read();
      __syncwarp();
    };
    for (int tile = first_tile; tile < p.num_tiles && ok; tile += tile_step) {
      const int b = tile / tiles_per_batch, r = tile % tiles_per_batch;
      const int row0 = (r / p.n_tiles) * TILE_M + (int)rank * BM + quarter * 32, col0 = (r % p.n_tiles) * p.n_tile + c_lo * 32;
      auto load_e = [&](int c) {
        mbar_expect_tx(ebar, kFloatBuf);
        tma_load_3d(fbuf, &tmE, ebar, col0 + c * 32, row0, b);
        e_pending = true;
      };
      if (has_e && lane == 0 && n_c > 0) {
        tma_store_wait_read();
        load_e(0);
      }
      float sum[3][32];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int i = 0; i < 32; ++i) sum[c][i] = 0.0f;
      auto add_blocks = [&](auto chunks_t) {  // (a loop for each number of chunks: no conditions between the reads)
        constexpr int NC = decltype(chunks_t)::value;
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          if (!mbar_wait(accf_bar(acc), acc_phase, abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          const float unbias = ((3 * kb + lane) & 7) < 3 ? kOneUp : 1.0f;
          const uint32_t tsrc = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * p.n_tile + c_lo * 32);
          float v[2][32];
          if (NC > 0) tc_ld32_async(tsrc, v[0]);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            tc_ld_wait();
            if (c + 1 < NC) tc_ld32_async(tsrc + (c + 1) * 32, v[(c + 1) & 1]);
            if (c + 1 == NC) tc_fence_before();
            if (c + 1 == NC) __syncwarp();
            if (c + 1 == NC && lane == 0) mbar_arrive_cluster(map_to_cta(acce_bar(acc), 0));  // handed back before the last addition
#pragma unroll
            for (int i = 0; i < 32; ++i) sum[c][i] = fmaf(v[c & 1][i], unbias, sum[c][i]);
          }
          if (NC == 0 && lane == 0) mbar_arrive_cluster(map_to_cta(acce_bar(acc), 0));
          if (++acc == p.n_acc) { acc = 0; acc_phase ^= 1u; }
        }
      };
      if (n_c == 3) add_blocks(std::integral_constant<int, 3>());
      else if (n_c == 2) add_blocks(std::integral_constant<int, 2>());
      else if (n_c == 1) add_blocks(std::integral_constant<int, 1>());
      else add_blocks(std::integral_constant<int, 0>());
      if (!ok) break;
#pragma unroll 1
      for (int c = 0; c < n_c; ++c) {
        float (&v)[32] = sum[0];  // the chunks move up: this code is there once
        const int col = col0 + c * 32;
        bool doubt = false;
#pragma unroll
        for (int i = 0; i < 32; ++i) doubt = doubt || !(fabsf(v[i]) < __uint_as_float(0x7f800000u));
        if (__any_sync(0xffffffffu, doubt)) refine(g, b, row0 + lane, col, v);
        float second[32];  // gelu' or the mask
        if (has_e) {
          if (!mbar_wait(ebar, e_phase, abort_flag, p.status)) { ok = false; break; }
          e_phase ^= 1u;
          e_pending = false;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const uint4 raw = ld_shared16(swz(fbuf, lane, u));
            const float e[4] = {__uint_as_float(raw.x), __uint_as_float(raw.y), __uint_as_float(raw.z), __uint_as_float(raw.w)};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int j = 4 * u + i;
              if (g.epi == EPI_MUL) {
                v[j] *= e[i];
              } else {
                const float gate = g.gate && col + j < g.N ? g.gate[col + j] : 1.0f;
                v[j] = gate * e[i] + v[j];
                second[j] = v[j] > 0.0f ? 1.0f : 0.0f;
                if (g.relu) v[j] = fmaxf(v[j], 0.0f);
              }
            }
          }
          __syncwarp();
          if (g.epi == EPI_MUL && lane == 0 && c + 1 < n_c) load_e(c + 1);  // every lane has read its row
        }
        if (g.epi == EPI_GELU_FWD || g.epi == EPI_MUL) {
          if (g.epi == EPI_GELU_FWD) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const float z = v[i], twice = 1.0f + erff(z * 0.70710678118654752440f);  // gelu_f and gelu_prime_f, one erf
              second[i] = 0.5f * twice + z * expf(-0.5f * z * z) * 0.39894228040143267794f;
              v[i] = 0.5f * z * twice;
            }
          }
          free_buffers();
          put_parts(v);
          if (g.epi == EPI_GELU_FWD) put_floats(fbuf, second);
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (g.epi == EPI_GELU_FWD) tma_store_3d(&tmD2, fbuf, col, row0, b);
            tma_store_4d(&tmP, pbuf, col, row0, b, 0);
          }
        } else if (p.direct) {
          if (row0 + lane < g.M) {
            float* D = g.D + b * g.d_sb + (int64_t)(row0 + lane) * g.ldd + col;
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (col + i < g.N) D[i] = v[i];
          }
        } else {
          // plain stores alternate between the two buffers; with E the result replaces it
          const uint32_t buf = !has_e && (c & 1) ? pbuf : fbuf;
          if (!has_e) {
            if (lane == 0) {
              if (c == 0) tma_store_wait_read();  // (the last of the tile before may have gone through either)
              else tma_store_wait_read<1>();
            }
            __syncwarp();
          }
          put_floats(buf, v);
          if (g.relu) {
            free_buffers();
            put_floats(pbuf, second);
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_3d(&tmD, buf, col, row0, b);
            if (g.relu) tma_store_3d(&tmD2, pbuf, col, row0, b);
            if (has_e && c + 1 < n_c) {
              tma_store_wait_read();
              load_e(c + 1);
            }
          }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          sum[0][i] = sum[1][i];
          sum[1][i] = sum[2][i];
        }
      }
    }
    if (lane == 0) {
      tma_store_wait_all();
      if (e_pending) {  // only after an abort: do not leave with a copy into our buffer in flight
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(ebar, e_phase) && global_ns() - t0 < 100000000ull) {
        }
      }
    }
  }

  tc_fence_before();
  leave_together(abort_flag);  // neither CTA leaves (or frees) while its peer may still read its tiles or signal its barriers
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    if (*abort_flag) outlast_copies();
  }
}

// src [rows][4 per_row] -> planes, four floats per thread (one load where src is 16-byte aligned)
template <bool kAligned>
__global__ void split_parts_kernel(const float* __restrict__ src, Planes dst, int64_t n, int per_row) {
  chain_next();
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t row = i / per_row;
  const int c = (int)(i - row * per_row) * 4;
  const float* s = src + row * (4 * (int64_t)per_row) + c;
  const float4 v = kAligned ? __ldcs(reinterpret_cast<const float4*>(s)) : make_float4(s[0], s[1], s[2], s[3]);
  store_parts4(dst.p + row * dst.ld + c, dst.plane, v);
}

}  // namespace

bool tc::map_planes(CUtensorMap* tm, const Planes& P, int cols, int rows, int batch, int box_c, int box_r, CUtensorMapSwizzle swizzle) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch, 3};
  const cuuint64_t strides[3] = {(cuuint64_t)P.ld * 2, (cuuint64_t)(batch > 1 ? P.sb : P.ld * rows) * 2, (cuuint64_t)P.plane * 2};
  const cuuint32_t box[4] = {(cuuint32_t)box_c, (cuuint32_t)box_r, 1, 3}, estr[4] = {1, 1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, P.p, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

void split_parts(Launcher& lc, const float* src, const Planes& dst, int64_t rows, int cols) {
  const int64_t n = rows * (cols / 4);
  const unsigned grid = (unsigned)((n + 255) / 256);
  launch_chained(lc, (uintptr_t)src & 15u ? split_parts_kernel<false> : split_parts_kernel<true>, dim3(grid), 256, 0, 1, src, dst, n, cols / 4);
}

bool parts_fill(int M, int N, int batch) {
  return (int64_t)((M + TILE_M - 1) / TILE_M) * ((N + kMaxTileN - 1) / kMaxTileN) * batch >= sm_count() / 4;
}

bool gemm_parts(Launcher& lc, const PartsGemm& g, int* status_word) {
  Params p;
  p.g = g;
  p.status = status_word;
  p.k_blocks = (g.K + BK - 1) / BK;
  p.m_tiles = (g.M + TILE_M - 1) / TILE_M;
  // The width of a tile: the one whose waves over the SM pairs take the least time.  A block of 32 of K is 12 instructions of
  // n_tile / 2 clocks (narrow ones 40: A is read from shared memory either way) and a tile ends with an epilogue that only the
  // next tile's first blocks run under: 1500 clocks, and 12 a column, 60 where the GELU is formed (from the kernel's times).  Of 7
  // stacks, 64 (256) x 300 to 1024 (2048) x 4000, in each of their products the width chosen so is the fastest of the six or
  // within 4 % of it; a wrong one costs up to 1.9 times (1900 x 520 x 1560, 12 at once: 192 columns 502 us of VJP, 32 863).
  const int pairs = sm_count() / 2;
  int64_t best = 0;
  for (int n = 32; n <= kMaxTileN; n += 32) {
    const int64_t tiles = (int64_t)p.m_tiles * ((g.N + n - 1) / n) * g.batch;
    const int64_t block = 12 * (n / 2 > 40 ? n / 2 : 40);
    const int64_t cost = (tiles + pairs - 1) / pairs * (p.k_blocks * block + 1500 + n * (g.epi == EPI_GELU_FWD ? 60 : 12));
    if (best == 0 || cost <= best) {
      best = cost;
      p.n_tile = n;
    }
  }
  p.n_acc = (int)TMEM_COLS / p.n_tile < kMaxAcc ? (int)TMEM_COLS / p.n_tile : kMaxAcc;
  p.n_tiles = (g.N + p.n_tile - 1) / p.n_tile;
  p.num_tiles = p.m_tiles * p.n_tiles * g.batch;
  const int half_n = p.n_tile / 2;
  p.b_bytes = g.b_mn ? (half_n > 64 ? 2 : 1) * kMnBlock : 3u * half_n * BK * 2;
  p.stages = (int)(kRingBytes / (kABytes + p.b_bytes));
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  p.direct = g.D && ((uintptr_t)g.D & 15u) != 0;
  if (p.direct && g.epi != EPI_STORE) return false;  // (element by element neither E nor the mask is taken along)
  CUtensorMap tmA, tmB, tmD, tmD2, tmE, tmP;
  bool ok = g.a_mn ? map_planes(&tmA, g.A, g.M, g.K, g.batch, 64, BK, CU_TENSOR_MAP_SWIZZLE_128B)
                   : map_planes(&tmA, g.A, g.K, g.M, g.batch, BK, BM, CU_TENSOR_MAP_SWIZZLE_64B);
  ok = ok && (g.b_mn ? map_planes(&tmB, g.B, g.N, g.K, g.batch, 64, BK, CU_TENSOR_MAP_SWIZZLE_128B)
                     : map_planes(&tmB, g.B, g.K, g.N, g.batch, BK, half_n, CU_TENSOR_MAP_SWIZZLE_64B));
  tmD = tmD2 = tmE = tmP = tmA;  // placeholders when unused
  const bool to_parts = g.epi == EPI_GELU_FWD || g.epi == EPI_MUL;
  if (to_parts) ok = ok && map_planes(&tmP, g.Dp, g.N, g.M, g.batch, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
  else if (!p.direct) ok = ok && make_map_epi(&tmD, g.D, true, g.M, g.N, g.batch, g.ldd, g.d_sb);
  if (g.D2) ok = ok && make_map_epi(&tmD2, g.D2, true, g.M, g.N, g.batch, g.ldd2, g.d2_sb);
  if (g.E) ok = ok && make_map_epi(&tmE, g.E, true, g.M, g.N, g.batch, g.lde, g.e_sb);
  if (!ok) return false;
  static PerDevice<bool> attr_done;
  if (!attr_done.here()) {
    if (cudaFuncSetAttribute(gemm_parts_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    attr_done.here() = true;
  }
  if (try_launch_chained(lc, gemm_parts_kernel, dim3(2 * (p.num_tiles < pairs ? p.num_tiles : pairs)), THREADS, SMEM_BYTES, 2, tmA, tmB, tmD,
                         tmD2, tmE, tmP, p) != cudaSuccess)
    return false;
  return true;
}

}  // namespace hbp
