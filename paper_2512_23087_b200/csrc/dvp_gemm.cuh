// Tensor-core contraction C[M,N] (+)= alpha * A[M,K] * B[N,K]^T for sm_100a.
//
// A and B are 16-bit (both bf16 or both f16), row-major with K contiguous; C is
// fp32 row-major.  A persistent kernel, one block per SM, walks 128 x 256 output
// tiles.  Per tile the K dimension is cut in slices of 64: a producer thread
// brings the A (128 x 64) and B (256 x 64) slices into a ring of shared-memory
// stages with TMA tile loads (128-byte swizzle), one thread issues tcgen05.mma
// (M = 128, N = 256, K = 16, four per slice) accumulating in tensor memory, and
// four epilogue warps read the accumulator back with tcgen05.ld, scale it and
// store it.  Two accumulators (2 x 256 TMEM columns) let the epilogue of one
// tile overlap the MMAs of the next.
//
// Every wait on an mbarrier is bounded.  A wait that runs out records a code in
// *status, raises a block-wide abort flag, and every role leaves its loop; the
// block then lets its own copies land, frees its tensor memory and returns.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dvp_common.cuh"

namespace dvp {
namespace gemm {

constexpr int kBM = 128, kBN = 256, kBK = 64;
constexpr int kStages = 4;
constexpr int kUmmaK = 16;
constexpr int kThreads = 192;  // warp 0: TMA, warp 1: MMA, warps 2..5: epilogue
constexpr uint32_t kBytesA = kBM * kBK * 2, kBytesB = kBN * kBK * 2;
constexpr uint32_t kStageBytes = kBytesA + kBytesB;
constexpr uint32_t kTmemCols = 512;
constexpr size_t kSmemBytes = 1024 /*alignment slack*/ + (size_t)kStages * kStageBytes + 256;
constexpr uint32_t kSpinLimit = 1u << 22;

// The tensor core cuts off what does not fit its float32 accumulator, so that terms of one sign lose more the more of them
// one sum takes: relative error of a product of positive numbers 2.35e-5 with K = 4,096, 4.8e-5 with 8,192, 9.6e-5 with
// 16,384.  A launch that asks for it (`chain_k`) makes a tile's K several such sums, one accumulator after the other, and
// adds each to C while the next is formed: the error of as many launches, without their fills and drains.  (Two sums
// kept, added on their way out and stored once: 4 % more time for a call of 4,727 x 2,864 x 12,179 than with one sum, because
// nothing overlaps the stores then.  This way, and with one sum: 1,253 and 1,244 us, 8,192 x 1,024 x 20,011 1,493 and 1,471.)
constexpr int kChainK = 4096;

enum { kErrNone = 0, kErrProducerWait = 11, kErrMmaWaitFull = 12, kErrMmaWaitTmem = 13,
       kErrEpilogueWait = 14 };

struct Params {
  float *C;
  long long ldc;
  int M, N, K;
  float alpha;
  const float *alpha_dev;  // optional device scalar multiplied into alpha
  int accumulate;          // C += instead of C =
  int *status;             // device word, set non-zero when a wait gives up
  int clear_status;        // the word is cleared first (pair kernel); a wait gives up after seconds
  int a_mn_major;          // A is stored transposed, [K, M] with M contiguous (pair kernel only)
  int b_mn_major;          // the same for B, [K, N]
  int split_k;             // pair kernel: each tile's K range is cut into this many units (see range_stride)
  float *row_max;          // optional (pair kernel, no split, no accumulation): row_max[row * row_max_ld + tn]
  long long row_max_ld;    // = the maximum of row `row` of C over the columns of tile column tn
  long long range_stride;  // split_k > 1: 0, the units' results are added to C with atomics (C zeroed or
                           // accumulated into); otherwise K range i goes to C + i * range_stride (elements)
  int early;               // pair kernel: see begin_after
  const float *row_scale;  // optional (pair kernel): row `row` of the product is multiplied by row_scale[row]
  int chain;               // pair kernel: slices of K that are added up in the tensor core (kChainK), and how many such
  int chains;              // sums, each added to C, a unit has
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false when the limit ran out or another role raised the abort flag.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (it > 32) __nanosleep(40);
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x,
                                            int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
      "%4}], [%2];" ::"r"(dst),
      "l"(map), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of
// 128 bytes, groups of 8 rows 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3ffffu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused with swizzle): 16 B
  d |= (uint64_t)(1024 >> 4) << 32;         // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                   // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                   // 128-byte swizzle
  return d;
}

// The same for an MN-major operand (stored [K, MN] with MN contiguous), brought in as
// boxes of 64 K-rows x 64 MN-elements: inside a box a K-row is 128 swizzled bytes, groups
// of 8 K-rows are 1024 bytes apart (stride byte offset), and the next 64 MN-elements
// start one box (8192 bytes) further (leading byte offset).
__device__ __forceinline__ uint64_t smem_desc_sw128_mn(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3ffffu) >> 4);
  d |= (uint64_t)(8192 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor for kind::f16: fp32 accumulate, A and B of format
// `fmt` (0 = f16, 1 = bf16), both K-major, M = 128, N = 256.
__device__ __forceinline__ uint32_t instr_desc(uint32_t fmt) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(kBN >> 3) << 17) |
         ((uint32_t)(kBM >> 4) << 24);
}

__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                     uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
// Both are for whole warps: what lanes store between two reads (rows and columns that end inside a tile) parts them.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
// The registers pass through the wait: nothing may use them before it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[32]) {
  __syncwarp();
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29])
               :
               : "memory");
  asm volatile("" : "+r"(r[30]), "+r"(r[31])::"memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Thirty-two columns of a thread's accumulator row, times alpha, to C.  Every index is a constant: indexed
// by a loop variable the accumulators went through local memory, half of all the bytes the epilogue stored
// (a d_w contraction of 512 tokens x 32,000 x 1,024, which is bound by its epilogue: 68 us then).
//   kStore  C = v     kAdd  C += v by vector reductions in L2: one addend per element and launch, so reruns
//   are bit-identical; loads, additions and stores were 32 dependent round trips a tile
//
// `exchange`: four neighbouring lanes exchange their rows' 32-byte pieces first, so that a store instruction of the
// warp fills 8 whole lines instead of a piece of 32 of them.  With the pieces as they lie a 32,000 x 1,024 C leaves
// the chip at 3.4 TB/s (5.5 in whole lines, with nothing else to do), which bounds products with a short K; the exchange
// goes through the shared-memory path that the MMAs read their operands by, which long ones are bound by.  us without /
// with it, K = 64, 256, 512, 640, 768, 1,024, 2,048: 39.2 / 31.1, 41.5 / 34.8, 46.3 / 42.9, 50.9 / 49.4, 55.9 / 55.6, 63.6 / 67.5,
// 111 / 114.  Rows of 256 bytes by way of shared memory: K = 512 42.4.
constexpr int kExchangeSlices = 8;  // up to this many slices of K in a unit
enum class Out { kStore, kAdd };
// c_own: where the thread's own row (`lane` of the warp's rows) begins; rows: how many of the warp's rows C has.
template <Out kOut>
__device__ __forceinline__ void store_columns(float *c_own, long long ldc, int lane, int rows, const uint32_t (&r)[32],
                                              float alpha, int n_cols, bool exchange) {
  if (n_cols >= 32) {
    float v[4][8];  // v[b]: columns 8 b .. 8 b + 7 of the thread's row
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j >> 3][j & 7] = alpha * __uint_as_float(r[j]);
    // a 4 x 4 transposition of pieces among the lanes 4 g + q: v[k] becomes piece q of row 4 g + k
    if (exchange) {
#pragma unroll
      for (int s = 1; s <= 2; s *= 2) {
        const bool odd = (lane & s) != 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (b & s) continue;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float got = __shfl_xor_sync(0xffffffffu, odd ? v[b][e] : v[b | s][e], s);
            if (odd)
              v[b][e] = got;
            else
              v[b | s][e] = got;
          }
        }
      }
    }
    // piece k of the thread: of its own row, or piece `lane & 3` of row 4 g + k
    const int first = exchange ? lane & ~3 : lane;
    float *c = c_own + (long long)(first - lane) * ldc + (exchange ? 8 * (lane & 3) : 0);
    const long long next = exchange ? ldc : 8;
#pragma unroll
    for (int k = 0; k < 4; ++k, c += next) {
      if (first + (exchange ? k : 0) >= rows) break;
      if constexpr (kOut == Out::kStore) {
        asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(c), "f"(v[k][0]), "f"(v[k][1]),
                     "f"(v[k][2]), "f"(v[k][3]), "f"(v[k][4]), "f"(v[k][5]), "f"(v[k][6]), "f"(v[k][7])
                     : "memory");
      } else {
        asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(c), "f"(v[k][0]), "f"(v[k][1]), "f"(v[k][2]),
                     "f"(v[k][3])
                     : "memory");
        asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(c + 4), "f"(v[k][4]), "f"(v[k][5]),
                     "f"(v[k][6]), "f"(v[k][7])
                     : "memory");
      }
    }
  } else if (lane < rows) {
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j < n_cols) {
        const float v = alpha * __uint_as_float(r[j]);
        if constexpr (kOut == Out::kStore)
          c_own[j] = v;
        else
          atomicAdd(c_own + j, v);
      }
    }
  }
}

struct Shared {
  uint64_t full[kStages], empty[kStages], tmem_full[2], tmem_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};

__global__ void __launch_bounds__(kThreads, 1)
gemm_tn_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const Params p, const uint32_t fmt) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;  // swizzle atoms are 1024-byte aligned
  uint8_t *aligned = smem_raw + (base - smem_u32(smem_raw));
  Shared *sh = reinterpret_cast<Shared *>(aligned + (size_t)kStages * kStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const int tiles_m = (p.M + kBM - 1) / kBM, tiles_n = (p.N + kBN - 1) / kBN;
  const int n_tiles = tiles_m * tiles_n;
  const int k_slices = (p.K + kBK - 1) / kBK;
  // Blocks that run together take consecutive tiles: walk the shorter tile dimension
  // fastest so that they share the operand panel of the longer one through L2.
  const bool m_fastest = tiles_m <= tiles_n;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&sh->tmem_full[b]), 1);
      mbar_init(smem_u32(&sh->tmem_empty[b]), 4);
    }
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {  // one warp allocates the tensor memory of the block
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;
  volatile int *abort_flag = &sh->abort_flag;

  if (warp == 0) {
    // ---------------- producer: TMA loads into the stage ring
    if (lane == 0) {
      uint32_t it = 0;
      for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x) {
        const int tm = m_fastest ? tile % tiles_m : tile / tiles_n;
        const int tn = m_fastest ? tile / tiles_m : tile % tiles_n;
        for (int ks = 0; ks < k_slices; ++ks, ++it) {
          const uint32_t s = it % kStages, round = it / kStages;
          if (round > 0 && !mbar_wait(smem_u32(&sh->empty[s]), (round - 1) & 1, abort_flag)) {
            if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrProducerWait); }
            break;
          }
          const uint32_t bar = smem_u32(&sh->full[s]);
          mbar_expect_tx(bar, kStageBytes);
          const uint32_t dst = base + s * kStageBytes;
          tma_load_2d(dst, &map_a, bar, ks * kBK, tm * kBM);
          tma_load_2d(dst + kBytesA, &map_b, bar, ks * kBK, tn * kBN);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0) {
      const uint32_t idesc = instr_desc(fmt);
      uint32_t it = 0, local_tile = 0;
      for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x, ++local_tile) {
        const uint32_t buf = local_tile & 1, use = local_tile >> 1;
        if (use > 0 && !mbar_wait(smem_u32(&sh->tmem_empty[buf]), (use - 1) & 1, abort_flag)) {
          if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrMmaWaitTmem); }
          break;
        }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + buf * kBN;
        bool ok = true;
        for (int ks = 0; ks < k_slices; ++ks, ++it) {
          const uint32_t s = it % kStages, round = it / kStages;
          if (!mbar_wait(smem_u32(&sh->full[s]), round & 1, abort_flag)) {
            if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrMmaWaitFull); }
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_addr = base + s * kStageBytes, b_addr = a_addr + kBytesA;
          const uint64_t adesc = smem_desc_sw128(a_addr), bdesc = smem_desc_sw128(b_addr);
#pragma unroll
          for (int k = 0; k < kBK / kUmmaK; ++k) {
            // 16 elements of K are 32 bytes inside the 128-byte swizzled row
            const uint64_t step = (uint64_t)((k * kUmmaK * 2) >> 4);
            umma(tmem_d, adesc + step, bdesc + step, idesc, (ks > 0 || k > 0) ? 1u : 0u);
          }
          umma_commit(smem_u32(&sh->empty[s]));  // the stage is free once these MMAs have read it
        }
        if (!ok) break;
        umma_commit(smem_u32(&sh->tmem_full[buf]));  // accumulator complete
      }
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> global
    const int quarter = warp & 3;  // TMEM lanes this warp may read
    const float alpha = p.alpha * (p.alpha_dev ? *p.alpha_dev : 1.f);
    uint32_t local_tile = 0;
    for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x, ++local_tile) {
      const int tm = m_fastest ? tile % tiles_m : tile / tiles_n;
      const int tn = m_fastest ? tile / tiles_m : tile % tiles_n;
      const uint32_t buf = local_tile & 1, use = local_tile >> 1;
      if (!mbar_wait(smem_u32(&sh->tmem_full[buf]), use & 1, abort_flag)) {
        if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrEpilogueWait); }
        break;
      }
      tc_fence_after();
      const int row = tm * kBM + quarter * 32 + lane;
      float *crow = p.C + (long long)row * p.ldc;
#pragma unroll 1
      for (int c0 = 0; c0 < kBN; c0 += 32) {
        uint32_t r[32];
        tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * kBN + c0, r);
        tmem_wait_ld(r);
        const int col = tn * kBN + c0;
        if (col < p.N) {
          if (p.accumulate)
            store_columns<Out::kAdd>(crow + col, p.ldc, lane, p.M - (row - lane), r, alpha, p.N - col, false);
          else
            store_columns<Out::kStore>(crow + col, p.ldc, lane, p.M - (row - lane), r, alpha, p.N - col, false);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh->tmem_empty[buf]));
    }
  }

  // ---------------- teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {
    // give this block's copies in flight time to land before the memory is released
    for (int i = 0; i < 2000; ++i) __nanosleep(500);
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                 : "memory");
  }
}

// ---- the same contraction on pairs of blocks (tcgen05 cta_group::2) ------------------
// Two blocks of a cluster share one 256 x 256 output tile: each holds 128 rows of
// A, 128 of the 256 rows of B, and the 128 x 256 accumulator of its own rows in its
// tensor memory.  One thread of the leader block (cluster rank 0) issues the MMAs for
// both, so each block reads only half of B from shared memory per MMA: this removes
// the shared-memory bandwidth ceiling of the one-block form.  Both blocks' TMA loads
// complete on the leader's "full" barrier; the MMA thread's commits arrive on the
// "empty" and "accumulator full" barriers of both blocks; both blocks' epilogue warps
// arrive on the leader's "accumulator empty" barrier.

constexpr int kPairBM = 256;
constexpr int kStages2 = 6;
constexpr uint32_t kBytesB2 = (kBN / 2) * kBK * 2;
constexpr uint32_t kStageBytes2 = kBytesA + kBytesB2;
constexpr size_t kSmemBytes2 = 1024 + (size_t)kStages2 * kStageBytes2 + 256;

struct Shared2 {
  uint64_t full[kStages2], empty[kStages2], tmem_full[2], tmem_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();  // the aligned forms want the whole warp
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of this block's shared-memory location `local` as seen in block `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
// Hands an accumulator back that this warp has read (tcgen05.wait::ld, tcgen05.fence): nothing in memory passes with it.
// Releasing at cluster scope, the arrival waited until the tile's stores had reached L2, and the next tile's stores did not
// begin before: 32,000 x 1,024 with K = 512 49.4 us, 42.9 this way (K = 64: 37.2 / 33.5).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr)
               : "memory");
}
// TMA tile load whose completion is counted on a barrier that may live in the peer block.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map,
                                                 uint32_t bar_cluster_addr, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(map), "r"(bar_cluster_addr), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive, once these MMAs are done, on the barrier at this offset in both blocks of the pair.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], "
      "%1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}

// kChains: units of several sums (kChainK).  Products of one sum a unit, the others, have a kernel without that: short ones are
// bound by what a tile costs beside its slices (512 x 1,024 x 32,000: 205.7 us a call, 208.1 with one kernel for all).
template <bool kChains>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tn_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                    const Params p, const uint32_t fmt) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *aligned = smem_raw + (base - smem_u32(smem_raw));
  Shared2 *sh = reinterpret_cast<Shared2 *>(aligned + (size_t)kStages2 * kStageBytes2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0 = leader of the pair
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  const int tiles_m = (p.M + kPairBM - 1) / kPairBM, tiles_n = (p.N + kBN - 1) / kBN;
  const int n_tiles = tiles_m * tiles_n;
  const int k_slices = (p.K + kBK - 1) / kBK;
  const bool m_fastest = tiles_m <= tiles_n;
  // work units: every tile once per K range; unit u is tile u % n_tiles of range u / n_tiles
  const int n_units = n_tiles * p.split_k;
  const int k_per = (k_slices + p.split_k - 1) / p.split_k;
  // a pair's accumulators in turn hold the sums of its units, of each one p.chains: from one sum to the next
  const auto next_sum = [&](int &unit, int &sum) {
    if (kChains && ++sum < p.chains) return;
    sum = 0;
    unit += n_pairs;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages2; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);   // the leader's producer, plus the bytes of both blocks
      mbar_init(smem_u32(&sh->empty[s]), 1);  // one commit
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&sh->tmem_full[b]), 1);   // one commit
      mbar_init(smem_u32(&sh->tmem_empty[b]), 8);  // four epilogue warps in each block
    }
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_barrier();  // barriers of both blocks are initialised before anyone signals them
  tc_fence_after();
  begin_after(p.early != 0);
  if (p.clear_status && blockIdx.x == 0 && threadIdx.x == 0) *p.status = 0;
  const uint32_t tmem_base = sh->tmem_base;
  volatile int *abort_flag = &sh->abort_flag;

  if (warp == 0) {
    // ---------------- producer (both blocks): own rows of A, own half of B
    if (lane == 0) {
      uint32_t it = 0;
      for (int unit = pair; unit < n_units && !*abort_flag; unit += n_pairs) {
        const int tile = unit % n_tiles, k_lo = (unit / n_tiles) * k_per;
        const int k_hi = min(k_slices, k_lo + k_per);
        const int tm = m_fastest ? tile % tiles_m : tile / tiles_n;
        const int tn = m_fastest ? tile / tiles_m : tile % tiles_n;
        for (int ks = k_lo; ks < k_hi; ++ks, ++it) {
          const uint32_t s = it % kStages2, round = it / kStages2;
          if (round > 0 && !mbar_wait(smem_u32(&sh->empty[s]), (round - 1) & 1, abort_flag)) {
            if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrProducerWait); }
            break;
          }
          const uint32_t bar_local = smem_u32(&sh->full[s]);
          if (rank == 0) mbar_expect_tx(bar_local, 2 * kStageBytes2);
          const uint32_t bar = map_to_rank(bar_local, 0);
          const uint32_t dst = base + s * kStageBytes2;
          // 128 rows of A or B: one box of 128 x 64 K, or two of 64 K-rows x 64
          const auto load = [&](uint32_t to, const CUtensorMap *map, int mn_major, int row0) {
            if (mn_major) {
              tma_load_2d_pair(to, map, bar, row0, ks * kBK);
              tma_load_2d_pair(to + kBytesA / 2, map, bar, row0 + 64, ks * kBK);
            } else {
              tma_load_2d_pair(to, map, bar, ks * kBK, row0);
            }
          };
          load(dst, &map_a, p.a_mn_major, tm * kPairBM + (int)rank * kBM);
          load(dst + kBytesA, &map_b, p.b_mn_major, tn * kBN + (int)rank * (kBN / 2));
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader block only)
    if (lane == 0 && rank == 0) {
      const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(kBN >> 3) << 17) |
                             ((uint32_t)(kPairBM >> 4) << 24) | (p.a_mn_major ? (1u << 15) : 0u) |
                             (p.b_mn_major ? (1u << 16) : 0u);
      // between two K = 16 steps of an operand: 32 bytes inside a K-major row, 16 K-rows of an MN-major box
      const uint64_t a_step = (p.a_mn_major ? 16u * 128u : (uint32_t)(kUmmaK * 2)) >> 4;
      const uint64_t b_step = (p.b_mn_major ? 16u * 128u : (uint32_t)(kUmmaK * 2)) >> 4;
      uint32_t it = 0, n_sums = 0;
      for (int unit = pair, sum = 0; unit < n_units && !*abort_flag; next_sum(unit, sum), ++n_sums) {
        const int k_lo = (unit / n_tiles) * k_per + (kChains ? sum * p.chain : 0);
        const int k_hi = min(k_slices, k_lo + (kChains ? p.chain : k_per));
        const uint32_t buf = n_sums & 1, use = n_sums >> 1;
        if (use > 0 && !mbar_wait(smem_u32(&sh->tmem_empty[buf]), (use - 1) & 1, abort_flag)) {
          if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrMmaWaitTmem); }
          break;
        }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + buf * kBN;
        bool ok = true;
        for (int ks = k_lo; ks < k_hi; ++ks, ++it) {
          const uint32_t s = it % kStages2, round = it / kStages2;
          if (!mbar_wait(smem_u32(&sh->full[s]), round & 1, abort_flag)) {
            if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrMmaWaitFull); }
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_addr = base + s * kStageBytes2, b_addr = a_addr + kBytesA;
          const uint64_t adesc = p.a_mn_major ? smem_desc_sw128_mn(a_addr) : smem_desc_sw128(a_addr);
          const uint64_t bdesc = p.b_mn_major ? smem_desc_sw128_mn(b_addr) : smem_desc_sw128(b_addr);
#pragma unroll
          for (int k = 0; k < kBK / kUmmaK; ++k)
            umma_pair(tmem_d, adesc + k * a_step, bdesc + k * b_step, idesc, (ks > k_lo || k > 0) ? 1u : 0u);
          umma_commit_pair(smem_u32(&sh->empty[s]));
        }
        if (!ok) break;
        umma_commit_pair(smem_u32(&sh->tmem_full[buf]));
      }
    }
  } else {
    // ---------------- epilogue (both blocks): own 128 rows of the pair's tile
    const int quarter = warp & 3;
    const bool exchange = k_per <= kExchangeSlices;
    const float alpha_all = p.alpha * (p.alpha_dev ? *p.alpha_dev : 1.f);
    uint32_t n_sums = 0;
    for (int unit = pair, sum = 0; unit < n_units; next_sum(unit, sum), ++n_sums) {
      const int tile = unit % n_tiles;
      const int tm = m_fastest ? tile % tiles_m : tile / tiles_n;
      const int tn = m_fastest ? tile / tiles_m : tile % tiles_n;
      const uint32_t buf = n_sums & 1, use = n_sums >> 1;
      // the whole warp goes on or none of it: reading tensor memory and the exchange need every lane
      if (!__all_sync(0xffffffffu, !*abort_flag && mbar_wait(smem_u32(&sh->tmem_full[buf]), use & 1, abort_flag))) {
        if (!*abort_flag) { *abort_flag = 1; atomicExch(p.status, kErrEpilogueWait); }
        break;
      }
      tc_fence_after();
      const int row = tm * kPairBM + (int)rank * kBM + quarter * 32 + lane;
      // a tile's K ranges meet in C by additions, or each range has a matrix of its own
      const bool add_ranges = p.split_k > 1 && p.range_stride == 0;
      float *crow = p.C + (long long)row * p.ldc + (long long)(unit / n_tiles) * p.range_stride;
      const float alpha = alpha_all * ((p.row_scale && row < p.M) ? p.row_scale[row] : 1.f);
      float row_hi = -__builtin_huge_valf();  // maximum of what this thread stores of its row
      const uint32_t tmem_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * kBN;
      // two groups of 32 columns in flight: the next is read from tensor memory while one is stored
      uint32_t ra[32], rb[32];
      auto emit = [&](const uint32_t (&r)[32], int c0) {
        const int col = tn * kBN + c0;
        if (p.row_max && row < p.M) {
          if (col + 32 <= p.N) {
#pragma unroll
            for (int j = 0; j < 32; ++j) row_hi = fmaxf(row_hi, alpha * __uint_as_float(r[j]));
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (col + j < p.N) row_hi = fmaxf(row_hi, alpha * __uint_as_float(r[j]));
          }
        }
        if (col < p.N) {
          if (p.accumulate || add_ranges || (kChains && sum > 0))  // after the thread's own stores of the unit's first sum
            store_columns<Out::kAdd>(crow + col, p.ldc, lane, p.M - (row - lane), r, alpha, p.N - col, exchange);
          else
            store_columns<Out::kStore>(crow + col, p.ldc, lane, p.M - (row - lane), r, alpha, p.N - col, exchange);
        }
      };
      tmem_ld32(tmem_row, ra);
#pragma unroll 1
      for (int c0 = 0; c0 < kBN; c0 += 64) {
        tmem_wait_ld(ra);
        tmem_ld32(tmem_row + c0 + 32, rb);
        emit(ra, c0);
        tmem_wait_ld(rb);
        if (c0 + 64 < kBN) tmem_ld32(tmem_row + c0 + 64, ra);
        emit(rb, c0 + 32);
      }
      if (p.row_max && row < p.M) p.row_max[(long long)row * p.row_max_ld + tn] = row_hi;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(map_to_rank(smem_u32(&sh->tmem_empty[buf]), 0));
    }
  }

  // ---------------- teardown: nobody frees tensor memory the pair still uses
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {
    for (int i = 0; i < 2000; ++i) __nanosleep(500);
  }
  cluster_barrier();
  if (threadIdx.x == 0) end_after(p.early != 0);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                 : "memory");
  }
}

// ---- host side ------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// Tensor map of a row-major [rows, k] 16-bit matrix (row stride ld elements)
// for boxes of box_rows x 64 with the 128-byte swizzle; reads past the extents
// return zeros.
inline bool make_map(CUtensorMap *map, const void *base, long long rows, long long k, long long ld,
                     int box_rows, bool is_bf16) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)k, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, is_bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
            const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The number of K ranges that a cut into `ranges` equal ones (in slices, rounded up) really has.
inline int usable_ranges(int K, int ranges) {
  const int slices = (K + kBK - 1) / kBK;
  const int per = (slices + ranges - 1) / ranges;
  return (slices + per - 1) / per;
}

// K ranges for a product of `tiles` output tiles on `pairs` pairs of blocks, at most `most`: the waves times the
// slices of a unit, plus some 8 slices that a unit cannot overlap (its first loads and last stores), plus the
// traffic of the partial results.  A slice takes about a third of a microsecond.  (512 x 1,024 x 32,000: 8 tiles
// on 74 pairs took 110 us in two ranges each.)
inline int choose_ranges(long long tiles, int K, int pairs, int most, double out_bytes) {
  const int slices = (K + kBK - 1) / kBK;
  int best = 1;
  double best_cost = 1e300;
  for (int r = 1; r <= most && slices >= 4 * r; ++r) {
    if (usable_ranges(K, r) != r) continue;
    const double waves = (double)((tiles * r + pairs - 1) / pairs);
    const double cost = waves * ((slices + r - 1) / r + 8) + (r > 1 ? (r + 1) * out_bytes * 2 / 5e12 / 0.33e-6 : 0.0);
    if (cost < best_cost) {
      best_cost = cost;
      best = r;
    }
  }
  return best;
}

// How the launch follows the one before: in the ordinary way; in the ordinary way as the first of a call's, which the next
// may overlap and which clears the status word; overlapping its end (launch_after); the same without needing its results.
enum class Order { kAlone, kFirst, kAfter, kEarly };

// C[M,N] (+)= alpha * A[M,K] * B[N,K]^T.  lda, ldb multiples of 8; ldc of 8; bases 16-byte
// (A, B) and 32-byte (C) aligned.  Returns a CUDA error code; cudaErrorInvalidValue for
// layouts it cannot take.
inline cudaError_t launch_gemm_tn(const void *A, long long lda, const void *B, long long ldb, float *C,
                                  long long ldc, int M, int N, int K, bool is_bf16, float alpha,
                                  const float *alpha_dev, bool accumulate, int *status, int sm_count,
                                  cudaStream_t stream, bool single_block_tiles = false,
                                  bool a_mn_major = false, int split_k = 1, float *row_max = nullptr,
                                  long long row_max_ld = 0, const float *row_scale = nullptr,
                                  long long range_stride = 0, Order order = Order::kAlone, int chain_k = 0,
                                  bool b_mn_major = false) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  if (lda % 8 || ldb % 8 || ldc % 8 || (uintptr_t)A % 16 || (uintptr_t)B % 16 || (uintptr_t)C % 32)
    return cudaErrorInvalidValue;
  if ((a_mn_major || b_mn_major) && single_block_tiles) return cudaErrorInvalidValue;
  // every K range of a split needs work
  if (single_block_tiles || split_k < 1 || (K + kBK - 1) / kBK < 2 * split_k) split_k = 1;
  if (range_stride != 0) {
    if (usable_ranges(K, split_k) != split_k) return cudaErrorInvalidValue;
  } else {
    split_k = usable_ranges(K, split_k);
  }
  // per-tile row maxima are those of the stored values: only where a tile is stored once, whole
  if (row_max && (single_block_tiles || split_k > 1 || accumulate)) return cudaErrorInvalidValue;
  if (row_scale && single_block_tiles) return cudaErrorInvalidValue;
  const int k_per = ((K + kBK - 1) / kBK + split_k - 1) / split_k;
  // sums of at most chain_k, about one size: none is so short that the one before is still being stored when it ends
  const int most = chain_k > 0 && split_k == 1 ? chain_k / kBK : k_per, n_chains = (k_per + most - 1) / most;
  const int chain = (k_per + n_chains - 1) / n_chains, chains = (k_per + chain - 1) / chain;
  if (row_max && chains > 1) return cudaErrorInvalidValue;
  const bool overlaps = order == Order::kAfter || order == Order::kEarly;
  const int early = order == Order::kEarly || order == Order::kFirst ? 1 : 0, clear = order == Order::kFirst ? 1 : 0;
  Params p{C, ldc, M, N, K, alpha, alpha_dev, accumulate ? 1 : 0, status, clear, a_mn_major ? 1 : 0, b_mn_major ? 1 : 0, split_k,
           row_max, row_max_ld, range_stride, early, row_scale, chain, chains};
  if (split_k > 1 && !accumulate && range_stride == 0) {
    const cudaError_t z = cudaMemset2DAsync(C, (size_t)ldc * 4, 0, (size_t)N * 4, (size_t)M, stream);
    if (z != cudaSuccess) return z;
  }
  CUtensorMap map_a, map_b;
  if (!single_block_tiles) {
    // pairs of blocks on 256 x 256 tiles; a transposed A is [K, M]: its "rows" are K, boxes of 64 x 64; so is a transposed B
    const bool ok_a = a_mn_major ? make_map(&map_a, A, K, M, lda, 64, is_bf16)
                                 : make_map(&map_a, A, M, K, lda, kBM, is_bf16);
    const bool ok_b = b_mn_major ? make_map(&map_b, B, K, N, ldb, 64, is_bf16)
                                 : make_map(&map_b, B, N, K, ldb, kBN / 2, is_bf16);
    if (!ok_a || !ok_b) return cudaErrorInvalidValue;
    auto kernel = chains > 1 ? gemm_tn_pair_kernel<true> : gemm_tn_pair_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes2);
    if (e != cudaSuccess) return e;
    const int tiles = ((M + kPairBM - 1) / kPairBM) * ((N + kBN - 1) / kBN) * split_k;
    int pairs = sm_count / 2;
    if (pairs > tiles) pairs = tiles;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes2;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // No preferred carve-out: with all of an SM's shared memory asked for (34 KB beside this block for blocks of other kernels,
    // 1,792 bytes without), calls hung, once in some 10,000: one cluster of a launch that overlaps the one before did not get
    // past its allocation of tensor memory and its first barrier, while all other blocks that were counted had ended.  Why is
    // not known: the waits before that point (for places, for tensor memory, of the cluster) are the chip's and have no limit, and
    // no kernel that they could wait for was left.  The launches overlap all the same, without the attribute; not overlapping
    // them costs 4 to 7 % of small calls (512 x 1,024 x 32,000 170.5 / 178.0 us, 163 x 416 x 45,277 113.7 / 122.0).
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_after
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlaps ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, map_a, map_b, p, is_bf16 ? 1u : 0u);
  }
  if (!make_map(&map_a, A, M, K, lda, kBM, is_bf16) || !make_map(&map_b, B, N, K, ldb, kBN, is_bf16))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(gemm_tn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemBytes);
  if (e != cudaSuccess) return e;
  const int tiles = ((M + kBM - 1) / kBM) * ((N + kBN - 1) / kBN);
  const int grid = tiles < sm_count ? tiles : sm_count;
  gemm_tn_kernel<<<grid, kThreads, kSmemBytes, stream>>>(map_a, map_b, p, is_bf16 ? 1u : 0u);
  return cudaGetLastError();
}

}  // namespace gemm
}  // namespace dvp
