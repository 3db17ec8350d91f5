// Forward-only pass over stored bfloat16 rows in two sweeps: the inference rows of the fused LM-head entry.
//
// The row kernel (dvp_rows_impl.cuh) forms the masked sum of Def. 5.2 with the full one, under a guess of the
// maximum.  Rows that a linear head gives for random directions have no dominant token and nearly every token in
// the safe set: their coverage Z is 1 up to the rounding of the two sums, so that ln Z is made of those roundings,
// and callers that compare it from call to call get the sums they got before: the full sum online, each thread
// against its own running maximum, then the masked sum over the granules whose maximum reaches the threshold.
// The second sweep costs what the row kernel saves (T = 16,384 x V = 151,936: 2.3 against 1.3 ms beside 58 ms of
// contractions).  Rows that do not start on 32-byte boundaries take the scalar row kernel.
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

template <int kBlk>
__global__ void __launch_bounds__(kBlk, 1024 / kBlk) dvp_two_sweeps_kernel(const __grid_constant__ RowParams p) {
  extern __shared__ __align__(16) float smem[];
  float *scratch = smem;                                             // 96 floats
  uint16_t *hot_smem = reinterpret_cast<uint16_t *>(smem + 96);      // kHotCap per warp
  uint32_t *bound = reinterpret_cast<uint32_t *>(smem + 96 + (kBlk / 32) * kHotCap / 2);
  begin_after(true);  // needs nothing of the fused entry's earlier launches
  const long long t = blockIdx.x;
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
  if (blockIdx.x == gridDim.x - 1 && tid == 0) end_after(true);  // the others leave their place to the next blocks
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

static inline cudaError_t launch(const RowParams &p, cudaStream_t s) {
  const long long n_gran = (p.V + kElems - 1) / kElems;
  int threads = 256;  // fewer for short rows, so that threads are not idle
  while (threads > 64 && threads >= n_gran) threads /= 2;
  const long long steps = (n_gran + 2 * threads - 1) / (2 * threads);
  const size_t smem = ((size_t)96 + (threads / 32) * kHotCap / 2 + (size_t)steps * threads) * 4;
  if (!aligned32(p.train, p.ld_train, sizeof(T)) || steps * 64 > 65536 || smem > 200 * 1024) {
    dvp_row_kernel_scalar<T, T><<<(unsigned)p.T, 512, 0, s>>>(p);
    return cudaGetLastError();
  }
  switch (threads) {
    case 64: return launch_blk<64>(p, smem, s);
    case 128: return launch_blk<128>(p, smem, s);
    default: return launch_blk<256>(p, smem, s);
  }
}

}  // namespace two_sweeps
}  // namespace dvp
