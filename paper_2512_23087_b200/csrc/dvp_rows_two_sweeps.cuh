// Forward-only pass over stored bfloat16 rows in two sweeps: the inference rows of the fused LM-head entry.
//
// The row kernel (dvp_rows_impl.cuh) forms the masked sum of Def. 5.2 with the full one, under a guess of the
// maximum.  Rows that a linear head gives for random directions have no dominant token and nearly every token in
// the safe set: their coverage Z is 1 up to the rounding of the two sums, so that ln Z is made of those roundings,
// and callers that compare it from call to call get the sums they got before: the full sum online, each thread
// against its own running maximum, then the masked sum over the granules whose maximum reaches the threshold.
// The second sweep costs what the row kernel saves (T = 16,384 x V = 151,936: 2.3 against 1.3 ms beside 58 ms of
// contractions).
//
// Rows that do not start on 32-byte boundaries (an odd vocabulary) had the scalar row kernel, three sweeps with a 2-byte
// load an element, and get its sums for the same reason: 512 partial ones, the i-th over the elements i, i + 512, ...  Here
// a thread has eight neighbouring ones and loads sixteen bytes, and the block is small enough to run beside the first
// contraction.  (us of the kernel by itself, scalar / now: 3,891 x 58,933 500 / 286, 4,727 x 12,179 187 / 94, 767 x 10,474 35 / 24,
// 163 x 45,277 35 / 30.)
#pragma once

#include "dvp_rows_impl.cuh"

namespace dvp {
namespace two_sweeps {

using T = __nv_bfloat16;
constexpr int kElems = Granule<T>::kElems;

// The two bounds of a thread's step are one word: bfloat16 maxima of its granules.
__device__ __forceinline__ void absorb(const Stage<T, 2> &st, LogSum &acc, uint32_t *bound) {
  const float g0 = st.g[0].max(), g1 = st.g[1].max();
  *bound = (uint32_t)bf16_bits_round_up(g0) | ((uint32_t)bf16_bits_round_up(g1) << 16);
  const float cm = fmaxf(fmaxf(kNegInf, g0), g1);
  if (cm > kNegInf) {
    if (cm > acc.m) {
      const float cn = log2_reference(cm);
      acc.s *= ex2(acc.c - cn);  // acc.c = -inf at the start: the factor is 0
      acc.m = cm;
      acc.c = cn;
    }
    const float neg_c = -acc.c;
    float part = 0.f;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      float x[kElems];
      st.g[u].get(x);
#pragma unroll
      for (int j = 0; j < kElems; ++j) part += ex2(fmaf(x[j], kLog2e, neg_c));
    }
    acc.s += part;
  }
}

// The sampled token is left out so that 1 - pi^mp(a) has no cancellation.
__device__ __forceinline__ void masked_sum(const Granule<T> &gr, int g, int a, float tau, float m, SumCount &sc) {
  float x[kElems];
  gr.get(x);
  const int ja = a - g * kElems;  // in [0, kElems) only inside the owner granule
#pragma unroll
  for (int j = 0; j < kElems; ++j) {
    if (x[j] >= tau && x[j] > kNegInf) {  // the fill of a missing granule is never a token
      ++sc.n;
      if (j != ja) sc.s += ex2((x[j] - m) * kLog2e);
    }
  }
}

// Row t, by a block of kBlk threads.
template <int kBlk>
__device__ __forceinline__ void row_of_granules(const RowParams &p, const long long t, float *smem) {
  float *scratch = smem;                                             // 96 floats
  uint16_t *hot_smem = reinterpret_cast<uint16_t *>(smem + 96);      // kHotCap per warp
  uint32_t *bound = reinterpret_cast<uint32_t *>(smem + 96 + (kBlk / 32) * kHotCap / 2);
  const long long id = p.ids ? load_id(p.ids, p.id_is_i32, t) : -1;
  const bool has_id = id >= 0, bad_id = id >= p.V;
  const int a = (has_id && !bad_id) ? (int)id : -1;
  const int V = (int)p.V, tid = (int)threadIdx.x;
  const T *row = reinterpret_cast<const T *>(p.train) + t * p.ld_train;
  const int n_full = V / kElems, n_steps = (n_full + 2 * kBlk - 1) / (2 * kBlk);
  DVP_BOUNDS_BEGIN(p.bounds_status);
  DVP_BOUNDS_SET(n_gran, n_full);
  DVP_BOUNDS_SET(V, V);
  DVP_BOUNDS_SET(n_bound, (long long)n_steps * kBlk);
  DVP_BOUNDS_SET(n_hot, kHotCap);
  DVP_BOUNDS_SYNC();

  LogSum acc = {kNegInf, kNegInf, 0.f};
  if (n_steps > 0) {  // two stages in flight
    Stage<T, 2> s0, s1;
    s0.load_block<kBlk>(row, n_full, 0);
    int step = 0;
    for (; step + 1 < n_steps; step += 2) {
      s1.load_block<kBlk>(row, n_full, step + 1);
      if (DVP_IN(step * kBlk + tid, n_bound, DVP_OOB_BOUND)) absorb(s0, acc, bound + step * kBlk + tid);
      if (step + 2 < n_steps) s0.load_block<kBlk>(row, n_full, step + 2);
      if (DVP_IN((step + 1) * kBlk + tid, n_bound, DVP_OOB_BOUND)) absorb(s1, acc, bound + (step + 1) * kBlk + tid);
    }
    if (step < n_steps && DVP_IN(step * kBlk + tid, n_bound, DVP_OOB_BOUND)) absorb(s0, acc, bound + step * kBlk + tid);
  }
  const int k_tail = n_full * kElems + tid;  // the elements behind the last whole granule, one per thread
  const float x_tail = k_tail < V ? Storage<T>::widen(row[k_tail]) : kNegInf;
  if (x_tail > kNegInf) {
    if (x_tail > acc.m) {
      const float cn = log2_reference(x_tail);
      acc.s *= ex2(acc.c - cn);
      acc.m = x_tail;
      acc.c = cn;
    }
    acc.s += ex2(fmaf(x_tail, kLog2e, -acc.c));
  }
  const LogSum all = block_reduce_logsum(acc, scratch);

  SideStats st;
  st.m = all.m;
  st.lse = lse_from_logsum(all);
  st.sum_c = (double)all.c;
  st.sum_s = all.s;
  st.tau = threshold_f32(all.m, p.log_rho);
  st.z_a = a >= 0 ? Storage<T>::widen(row[a]) : 0.f;
  st.member = a >= 0 && st.z_a >= st.tau;
  st.e_a = st.member ? ex2((st.z_a - st.m) * kLog2e) : 0.f;

  SumCount sc = {0.f, 0};
  if (x_tail >= st.tau && x_tail > kNegInf) {
    ++sc.n;
    if (k_tail != a) sc.s += ex2((x_tail - st.m) * kLog2e);
  }
  // the threshold rounded down to bfloat16 (the list's order is part of the sum's); finite: with rho = 0 the list
  // would name the granules past the end
  const SweepOps<T>::Key key = SweepOps<float>::key(fmaxf(st.tau, -FLT_MAX));
  const HotList hot = build_hot_list<T, kBlk>(bound, n_steps, key, hot_smem);
  if (hot.fits()) {
    const int wbase = tid & ~31, lane = tid & 31;
    for (int q = lane; q < hot.count; q += 64) {
      if (!DVP_IN(q, n_hot, DVP_OOB_HOT)) break;
      const uint32_t e0 = hot.slots[q];
      const bool two = q + 32 < hot.count && DVP_IN(q + 32, n_hot, DVP_OOB_HOT);
      const uint32_t e1 = two ? hot.slots[q + 32] : e0;
      const int g0 = (int)(e0 >> 5) * kBlk + wbase + (int)(e0 & 31);
      const int g1 = (int)(e1 >> 5) * kBlk + wbase + (int)(e1 & 31);
      Granule<T> a0, a1;
      a0.load_whole(row, n_full, g0);
      if (two) a1.load_whole(row, n_full, g1);
      masked_sum(a0, g0, a, st.tau, st.m, sc);
      if (two) masked_sum(a1, g1, a, st.tau, st.m, sc);
    }
  } else {
    for (int step = 0; step < n_steps; ++step) {  // a dense safe set: both loads of a step before either is used
      if (!DVP_IN(step * kBlk + tid, n_bound, DVP_OOB_BOUND)) break;
      const uint32_t b = SweepOps<T>::reach(bound[step * kBlk + tid], key);
      const int g0 = 2 * step * kBlk + tid, g1 = g0 + kBlk;
      Granule<T> a0, a1;
      if (b & 1u) a0.load_whole(row, n_full, g0);
      if (b & 0x10000u) a1.load_whole(row, n_full, g1);
      if (b & 1u) masked_sum(a0, g0, a, st.tau, st.m, sc);
      if (b & 0x10000u) masked_sum(a1, g1, a, st.tau, st.m, sc);
    }
  }
  sc = block_reduce_sumcount(sc, scratch);
  st.s_x = sc.s;
  st.n = sc.n;
  set_mask_mass(st, V, 0, 0.f, a >= 0);
  if (tid == 0) {
    finish_side(p.out_t, t, st, has_id, bad_id);
    if (p.flags)
      p.flags[t] = (uint8_t)((st.member ? DVP_FLAG_IN_TRAIN : 0) | (has_id ? 0 : DVP_FLAG_NO_ID) |
                             (bad_id ? DVP_FLAG_BAD_ID : 0));
  }
  if (p.out_t.mask) write_mask_row<T>(row, V, st.tau, p.out_t.mask + t * ((p.V + 31) / 32), 0, 1);
}
template <int kBlk>
__global__ void __launch_bounds__(kBlk, 1024 / kBlk) dvp_two_sweeps_kernel(const __grid_constant__ RowParams p) {
  extern __shared__ __align__(16) float smem[];
  begin_after(true);  // needs nothing of the fused entry's earlier launches
  row_of_granules<kBlk>(p, blockIdx.x, smem);
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) end_after(true);  // the others leave their place to the next blocks
}

// ---- rows at any alignment ---------------------------------------------------------

constexpr int kSums = 512;  // partial sums of a row

// A row in pieces of kOwn elements, cut at the memory's boundaries: piece c holds the elements kOwn c - mis + (0 .. kOwn
// - 1).  With 512 / kOwn threads, thread j has the pieces j, j + 512 / kOwn, ...: always the same kOwn partial sums.
template <int kOwn>
struct Pieces {
  static constexpr int kPieceBlk = kSums / kOwn, kWords = kOwn / 2;
  struct Words {
    uint32_t w[kWords];
  };
  const T *row;
  int V, mis, lo, hi;  // pieces lo .. hi - 1 are whole

  __device__ __forceinline__ Pieces(const T *r, int V_) : row(r), V(V_) {
    mis = (int)(((uintptr_t)r & (kOwn * sizeof(T) - 1)) / sizeof(T));
    lo = mis ? 1 : 0;
    hi = (int)(((long long)V + mis) / kOwn);
  }
  // f(piece, words, which of its elements are the row's), in ascending order, for the pieces of this thread
  template <typename F>
  __device__ __forceinline__ void each(F f) const {
    constexpr int kAhead = kOwn == 8 ? 8 : 16;  // loads in flight
    const int tid = (int)threadIdx.x;
    if (tid == 0 && lo == 1) ragged(0, f);
    int c = tid < lo ? tid + kPieceBlk : tid;
    for (; c < hi; c += kAhead * kPieceBlk) {
      Words w[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u)
        if (c + u * kPieceBlk < hi && DVP_IN((long long)(c + u * kPieceBlk + 1) * kOwn - mis - 1, V, DVP_OOB_GLOBAL))
          w[u] = load(row + ((long long)(c + u * kPieceBlk) * kOwn - mis));
#pragma unroll
      for (int u = 0; u < kAhead; ++u)
        if (c + u * kPieceBlk < hi) f(c + u * kPieceBlk, w[u], (1u << kOwn) - 1u);
    }
    if (hi >= lo && hi % kPieceBlk == tid && (long long)hi * kOwn - mis < V) ragged(hi, f);
  }
  static __device__ __forceinline__ Words load(const T *p) {
    Words r;
    if constexpr (kOwn == 8) {
      const uint4 v = ld_stream16(p);
      r.w[0] = v.x, r.w[1] = v.y, r.w[2] = v.z, r.w[3] = v.w;
    } else {
      static_assert(kOwn == 2, "pieces of 16 or of 4 bytes");
      asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(r.w[0]) : "l"(p));
    }
    return r;
  }
  template <typename F>
  __device__ __forceinline__ void ragged(int c, F &f) const {
    uint32_t e[kOwn], have = 0;
#pragma unroll
    for (int i = 0; i < kOwn; ++i) {
      const long long k = (long long)c * kOwn - mis + i;
      const bool in = k >= 0 && k < V;
      const T v = in ? row[k] : Storage<T>::narrow(kNegInf);
      e[i] = *reinterpret_cast<const uint16_t *>(&v);
      have |= in ? 1u << i : 0u;
    }
    Words r;
#pragma unroll
    for (int i = 0; i < kWords; ++i) r.w[i] = e[2 * i] | e[2 * i + 1] << 16;
    f(c, r, have);
  }
};

// Pieces of 16 bytes; of 4, with four times the threads, for few rows (163 x 45,277: 30 us, 47 with 64 threads a row).
constexpr int kPieceSmem = 2 * kSums + 64;  // floats
template <int kOwn>
__device__ __forceinline__ void row_of_pieces(const RowParams &p, const long long t, float *smem) {
  constexpr int kPieceBlk = kSums / kOwn;
  using Words = typename Pieces<kOwn>::Words;
  float *part_m = smem, *part_s = smem + kSums, *scratch = smem + 2 * kSums;
  const long long id = p.ids ? load_id(p.ids, p.id_is_i32, t) : -1;
  const bool has_id = id >= 0, bad_id = id >= p.V;
  const int a = (has_id && !bad_id) ? (int)id : -1;
  const int V = (int)p.V, tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T *row = reinterpret_cast<const T *>(p.train) + t * p.ld_train;
  DVP_BOUNDS_BEGIN(p.bounds_status);
  DVP_BOUNDS_SET(V, V);
  DVP_BOUNDS_SYNC();
  const Pieces<kOwn> pieces(row, V);
  const float z_0 = Storage<T>::widen(row[a >= 0 ? a : 0]);
  const uint64_t l2 = pack2(kLog2e, kLog2e);
  auto unpack = [](const Words &w, float (&x)[kOwn]) {
#pragma unroll
    for (int i = 0; i < kOwn / 2; ++i) {
      x[2 * i] = __uint_as_float(w.w[i] << 16);
      x[2 * i + 1] = __uint_as_float(w.w[i] & 0xffff0000u);
    }
  };

  // every partial sum's own maximum, then the sum against it
  __nv_bfloat162 m2[kOwn / 2];
#pragma unroll
  for (int i = 0; i < kOwn / 2; ++i) m2[i] = SweepOps<T>::start(kNegInf);
  pieces.each([&](int, const Words &w, uint32_t) {  // elements that are not the row's are -inf
#pragma unroll
    for (int i = 0; i < kOwn / 2; ++i) m2[i] = __hmax2(m2[i], SweepOps<T>::pair(w.w[i]));
  });
  uint64_t minus[kOwn / 2], sum[kOwn / 2];
#pragma unroll
  for (int i = 0; i < kOwn / 2; ++i) {
    const float lo = Storage<T>::widen(m2[i].x), hi = Storage<T>::widen(m2[i].y);
    minus[i] = pack2(lo > kNegInf ? -lo : 0.f, hi > kNegInf ? -hi : 0.f);  // nothing but -inf: a sum of zeros
    sum[i] = 0;
  }
  pieces.each([&](int, const Words &w, uint32_t) {
    float x[kOwn];
    unpack(w, x);
#pragma unroll
    for (int i = 0; i < kOwn / 2; ++i) {
      float e0, e1;
      unpack2(mul2(add2(pack2(x[2 * i], x[2 * i + 1]), minus[i]), l2), e0, e1);
      sum[i] = add2(sum[i], pack2(ex2(e0), ex2(e1)));
    }
  });
  const int first = kOwn * tid - pieces.mis;  // element of the thread's first partial sum, modulo kSums
#pragma unroll
  for (int i = 0; i < kOwn; ++i) {
    float lo, hi;
    unpack2(sum[i / 2], lo, hi);
    part_m[(first + i) & (kSums - 1)] = Storage<T>::widen(i & 1 ? m2[i / 2].y : m2[i / 2].x);
    part_s[(first + i) & (kSums - 1)] = i & 1 ? hi : lo;
  }
  __syncthreads();
  for (int w = warp; w < kSums / 32; w += kPieceBlk / 32) {
    const MaxSum v = warp_reduce(MaxSum{part_m[w * 32 + lane], part_s[w * 32 + lane]});
    if (lane == 0) {
      scratch[w] = v.m;
      scratch[32 + w] = v.s;
    }
  }
  __syncthreads();
  const MaxSum all = warp_reduce(lane < kSums / 32 ? MaxSum{scratch[lane], scratch[32 + lane]} : MaxSum{kNegInf, 0.f});

  SideStats st;
  st.m = all.m;
  st.lse = (double)all.m + (double)logf(all.s);
  st.sum_c = (double)all.m * (double)kLog2e;
  st.sum_s = all.s;
  st.tau = threshold_f32(all.m, p.log_rho);
  st.z_a = a >= 0 ? z_0 : 0.f;
  st.member = a >= 0 && st.z_a >= st.tau;
  st.e_a = st.member ? ex2((st.z_a - st.m) * kLog2e) : 0.f;

  // the masked sum, without the sampled token
  int n = 0;
#pragma unroll
  for (int i = 0; i < kOwn / 2; ++i) sum[i] = 0;
  const uint64_t minus_m = pack2(-st.m, -st.m);
  pieces.each([&](int c, const Words &w, uint32_t have) {
    const uint32_t ja = (uint32_t)(a - (c * kOwn - pieces.mis));
    const uint32_t add = have & ~(a >= 0 && ja < kOwn ? 1u << ja : 0u);
    float x[kOwn];
    unpack(w, x);
#pragma unroll
    for (int i = 0; i < kOwn / 2; ++i) {
      float e0, e1;
      unpack2(mul2(add2(pack2(x[2 * i], x[2 * i + 1]), minus_m), l2), e0, e1);
      const bool in0 = x[2 * i] >= st.tau && (have >> (2 * i) & 1), in1 = x[2 * i + 1] >= st.tau && (have >> (2 * i + 1) & 1);
      n += (int)in0 + (int)in1;
      // adding zero changes no sum
      sum[i] = add2(sum[i], pack2(in0 && (add >> (2 * i) & 1) ? ex2(e0) : 0.f, in1 && (add >> (2 * i + 1) & 1) ? ex2(e1) : 0.f));
    }
  });
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kOwn; ++i) {
    float lo, hi;
    unpack2(sum[i / 2], lo, hi);
    part_s[(first + i) & (kSums - 1)] = i & 1 ? hi : lo;
  }
  n = __reduce_add_sync(0xffffffffu, n);
  if (lane == 0) reinterpret_cast<int *>(part_m)[warp] = n;
  __syncthreads();
  for (int w = warp; w < kSums / 32; w += kPieceBlk / 32) {
    const SumCount v = warp_reduce(SumCount{part_s[w * 32 + lane], 0});
    if (lane == 0) scratch[w] = v.s;
  }
  __syncthreads();
  st.s_x = warp_reduce(SumCount{lane < kSums / 32 ? scratch[lane] : 0.f, 0}).s;
  st.n = 0;
  for (int w = 0; w < kPieceBlk / 32; ++w) st.n += reinterpret_cast<const int *>(part_m)[w];
  set_mask_mass(st, V, 0, 0.f, a >= 0);
  if (tid == 0) {
    finish_side(p.out_t, t, st, has_id, bad_id);
    if (p.flags)
      p.flags[t] = (uint8_t)((st.member ? DVP_FLAG_IN_TRAIN : 0) | (has_id ? 0 : DVP_FLAG_NO_ID) |
                             (bad_id ? DVP_FLAG_BAD_ID : 0));
  }
  if (p.out_t.mask) write_mask_row<T>(row, V, st.tau, p.out_t.mask + t * ((p.V + 31) / 32), 0, 1);
}
template <int kOwn>
__global__ void __launch_bounds__(kSums / kOwn) dvp_piece_rows_kernel(const __grid_constant__ RowParams p) {
  __shared__ float smem[kPieceSmem];
  begin_after(true);  // needs nothing of the fused entry's earlier launches
  row_of_pieces<kOwn>(p, blockIdx.x, smem);
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) end_after(true);  // the others leave their place to the next blocks
}

template <int kBlk>
static cudaError_t launch_blk(const RowParams &p, size_t smem, cudaStream_t s) {
  auto k = dvp_two_sweeps_kernel<kBlk>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_after(k, (unsigned)p.T, kBlk, smem, s, p);
}

// How a call's rows are swept: in granules by blocks of `threads`, with `smem` bytes; 0: in pieces.
struct Shape {
  int threads;
  size_t smem;
};
static inline Shape shape_of(const RowParams &p) {
  const long long n_gran = (p.V + kElems - 1) / kElems;
  int threads = 256;  // fewer for short rows, so that threads are not idle
  while (threads > 64 && threads >= n_gran) threads /= 2;
  const long long steps = (n_gran + 2 * threads - 1) / (2 * threads);
  const size_t smem = ((size_t)96 + (threads / 32) * kHotCap / 2 + (size_t)steps * threads) * 4;
  if (!aligned32(p.train, p.ld_train, sizeof(T)) || steps * 64 > 65536 || smem > 200 * 1024) return {0, kPieceSmem * 4};
  return {threads, smem};
}

static inline cudaError_t launch(const RowParams &p, cudaStream_t s) {
  const Shape sh = shape_of(p);
  switch (sh.threads) {
    case 0:
      return p.T < 4 * 148 ? launch_after(dvp_piece_rows_kernel<2>, (unsigned)p.T, kSums / 2, 0, s, p)
                           : launch_after(dvp_piece_rows_kernel<8>, (unsigned)p.T, kSums / 8, 0, s, p);
    case 64: return launch_blk<64>(p, sh.smem, s);
    case 128: return launch_blk<128>(p, sh.smem, s);
    default: return launch_blk<256>(p, sh.smem, s);
  }
}

}  // namespace two_sweeps
}  // namespace dvp
