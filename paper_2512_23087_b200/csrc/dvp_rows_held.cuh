// Small calls: every row is held in registers.
//
// A call whose rows fit the chip's registers at once is bound by the chain of its phases, not by bytes or instructions.
// The row kernel's chain is long: a guess of the maximum, exchanges while the row streams, a list of what has to be read
// again, the second reading, the sums.  Here a thread loads its granules once, up to five; the maximum passes between
// warps in one exchange, the sums under the threshold that it gives in a second one, and the gradient is formed from what
// the registers hold.  Where a row has several blocks, warps write their results into the shared memory of all of them, so
// that an exchange is one barrier and the reads behind it are local.  The blocks of a token's two rows are one cluster:
// ln pi^mp_infer(a) and the membership pass to the training row's blocks through shared memory, and are waited for where
// they are needed, behind the gradient unless it is weighted.
#pragma once

namespace dvp {
namespace held {

constexpr int kMaxBlk = 512, kMaxWarps = kMaxBlk / 32, kMaxBlocks = 16;

__device__ __forceinline__ void st_cluster(float *local, uint32_t rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr(local, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint64_t *local, uint32_t rank, uint64_t v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cluster_addr(local, rank)), "l"(v) : "memory");
}

// What every warp of the cluster leaves, by its block's rank.
struct Slots {
  float max[kMaxBlocks * kMaxWarps];
  uint64_t sums[kMaxBlocks * kMaxWarps];  // the full sum and the masked one
  float count[kMaxBlocks * kMaxWarps];    // an integer
  float li, member;                       // of the inference row, in the training row's blocks
};

struct Group {
  int blocks, log_parts, log_warps;  // blocks of the cluster; of a row; warps of a block
  // f(slot) for this lane's slots of the row whose blocks begin at rank r0, in a fixed order
  template <typename F>
  __device__ __forceinline__ void each(int r0, F f) const {
    const int n = 1 << (log_parts + log_warps), lane = threadIdx.x & 31;
    for (int i = lane; i < n; i += 32) f((r0 + (i >> log_warps)) * kMaxWarps + (i & ((1 << log_warps) - 1)));
  }
  __device__ __forceinline__ void meet() const {
    if (log_parts > 0) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  }
};

// The statistics of a row from the cluster's slots; z_a: its logit of the sampled token a, if there is one.
template <typename TIn>
__device__ __forceinline__ SideStats stats_from(const Group &grp, const Slots &slots, int r0, float m, const RowParams &p,
                                                bool has_a, float z_a) {
  SideStats st;
  st.m = m;
  st.tau = threshold_of<TIn>(m, p.log_rho, p.mode);
  st.z_a = has_a ? z_a : 0.f;
  st.member = has_a && st.z_a >= st.tau;
  st.e_a = st.member ? ex2((st.z_a - m) * kLog2e) : 0.f;
  const float c = log2_reference(m);
  uint64_t v = 0;  // two zeros
  int n = 0;
  grp.each(r0, [&](int i) {
    v = add2(v, slots.sums[i]);
    n += __float_as_int(slots.count[i]);
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = add2(v, __shfl_xor_sync(0xffffffffu, v, o));
  n = __reduce_add_sync(0xffffffffu, n);
  float all, safe;
  unpack2(v, all, safe);
  if (has_a) all += ex2(fmaf(st.z_a, kLog2e, -c));
  st.lse = 0.0;  // from sum_c and sum_s, by the thread that writes it
  st.sum_c = (double)c;
  st.sum_s = all;
  st.s_x = safe;
  st.n = n + (st.member ? 1 : 0);
  set_mask_mass(st, p.V, p.mode, Storage<TIn>::widen(Storage<TIn>::narrow(p.mask_value)), has_a);
  return st;
}
__device__ __forceinline__ float max_from(const Group &grp, const Slots &slots, int r0) {
  float m = kNegInf;
  grp.each(r0, [&](int i) { m = fmaxf(m, slots.max[i]); });
  return key_value(__reduce_max_sync(0xffffffffu, order_key(m)));
}

// kGran: granules of a row that a thread holds.  `shape`: log2 of the blocks of a row, and kOverInfer where a row has one block
// and the gradient takes the inference rows' place.  (As a flag of the launch: the pointers compared here instead, and the
// shift by an unmasked argument, cost 0.3 us: 64 x 4,096 float32 with the gradient 5.9 / 5.4 us, 148 x 16,000 9.6 / 9.4.)
constexpr int kOverInfer = 16;
template <typename TIn, typename TGrad, Grad kGrad, int kGran>
__global__ void __launch_bounds__(kMaxBlk, 2) dvp_row_kernel_held(const __grid_constant__ RowParams p, const int shape) {
  using Ops = SweepOps<TIn>;
  constexpr int kElems = Granule<TIn>::kElems;
  __shared__ Slots slots;
  __shared__ __align__(16) uint32_t shift_smem[kGrad == Grad::kLoose ? kMaxWarps * kShiftWords : 1];
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5, n_thr = (int)blockDim.x;
  const int log_parts = shape & (kOverInfer - 1), both = p.infer ? 1 : 0, parts = 1 << log_parts;
  const Group grp{parts << both, log_parts, 31 - __clz(n_thr >> 5)};
  const int rank = grp.blocks > 1 ? (int)cluster_rank() : 0, part = rank & (parts - 1), r0 = rank - part;
  const bool second = rank >= parts;  // the inference row's half
  // Blocks write to one another's shared memory once all have begun.  Where a row has one block and the gradient takes the
  // inference row's place, they meet when both rows have been read instead, which no other barrier in front of the gradient
  // says there: the blocks of a longer row meet across the cluster for their maximum, weights wait for the inference row.
  const bool over_infer = kGrad != Grad::kNone && (shape & kOverInfer);
  if (grp.blocks > 1 && !over_infer) cluster_arrive();
  const long long t = blockIdx.x >> (log_parts + both);
  const long long id = p.ids ? load_id(p.ids, p.id_is_i32, t) : -1;
  const TIn *train = reinterpret_cast<const TIn *>(p.train) + t * p.ld_train;
  const TIn *infer = reinterpret_cast<const TIn *>(p.infer) + t * p.ld_infer;
  RowView<TIn> v;
  v.set(second ? infer : train, (int)p.V, part, log_parts);
  DVP_BOUNDS_BEGIN(p.bounds_status);
  DVP_BOUNDS_SET(n_gran, v.n_full);
  DVP_BOUNDS_SET(V, (long long)v.n_full * kElems);
  DVP_BOUNDS_SYNC();
  Granule<TIn> gr[kGran];
#pragma unroll
  for (int u = 0; u < kGran; ++u)
    if (u * n_thr < v.n_full) gr[u].load_whole(v.base, v.n_full, u * n_thr + tid);
  const int k_extra = v.extra();
  const float xe = k_extra < v.V ? Storage<TIn>::widen(v.row[k_extra]) : kNegInf;
  const bool has_id = id >= 0, bad_id = id >= p.V, has_a = has_id && !bad_id;
  const int a = has_a ? (int)id : -1;
  const float z_a = Storage<TIn>::widen(v.row[has_a ? a : 0]);

  // ---- the maximum
  float m = xe;
#pragma unroll
  for (int u = 0; u < kGran; ++u)
    if (u * n_thr < v.n_full) m = fmaxf(m, gr[u].max());
  m = key_value(__reduce_max_sync(0xffffffffu, order_key(m)));
  const int own_slot = rank * kMaxWarps + warp;
  if (grp.blocks > 1 && !over_infer) cluster_wait();  // all blocks have begun
  if (log_parts > 0) {
    if (lane < parts) st_cluster(&slots.max[own_slot], r0 + lane, m);
  } else if (lane == 0) {
    slots.max[own_slot] = m;
  }
  grp.meet();
  if (over_infer) {  // the maximum is one of all that the block's threads hold
    cluster_arrive();
    cluster_wait();
  }
  m = max_from(grp, slots, r0);

  // ---- the sums, without the sampled token
  const float c = log2_reference(m), tau = threshold_of<TIn>(m, p.log_rho, p.mode);
  const typename Ops::Tau tau_p = Ops::threshold(fmaxf(tau, -FLT_MAX));
  const uint64_t l2 = pack2(kLog2e, kLog2e), c2 = pack2(-c, -c);
  const int g_a = v.granule_of(a);
  uint64_t sum = 0;  // two zeros
  float safe = 0.f;
  uint32_t cnt = 0;
#pragma unroll
  for (int u = 0; u < kGran; ++u) {
    if (u * n_thr < v.n_full) {
      Granule<TIn> g = gr[u];
      if (u * n_thr + tid == g_a) {  // the sampled token becomes -inf
        const int ja = v.rel(a) - g_a * kElems;
        constexpr int kPerWord = 4 / (int)sizeof(TIn);
        const TIn fill = Storage<TIn>::narrow(kNegInf);
        uint32_t bits, mask = 0xffffffffu;
        if constexpr (kPerWord == 1) {
          bits = *reinterpret_cast<const uint32_t *>(&fill);
        } else {
          const int sh = 16 * (ja & 1);
          bits = (uint32_t) * reinterpret_cast<const uint16_t *>(&fill) << sh;
          mask = 0xffffu << sh;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i == ja / kPerWord) g.w[i] = (g.w[i] & ~mask) | bits;
      }
      float x[kElems], e[kElems];
      g.get(x);
      uint64_t of_granule = 0;  // added up by themselves first: see Sweep1::absorb
#pragma unroll
      for (int j = 0; j < kElems; j += 2) {
        unpack2(fma2(pack2(x[j], x[j + 1]), l2, c2), e[j], e[j + 1]);
        e[j] = ex2(e[j]);
        e[j + 1] = ex2(e[j + 1]);
        of_granule = add2(of_granule, pack2(e[j], e[j + 1]));
        Ops::masked(g, j / 2, x[j], x[j + 1], e[j], e[j + 1], tau_p, safe, cnt);
      }
      sum = add2(sum, of_granule);
    }
  }
  int n = Ops::count(cnt);
  {
    float s0, s1;
    unpack2(sum, s0, s1);
    // the sum's terms are 2^{z l - c}; those of the definition 2^{(z - m) l}
    safe *= ex2(-fmaf(m, kLog2e, -c));
    s0 += s1;
    if (k_extra != a) {
      s0 += ex2(fmaf(xe, kLog2e, -c));
      if (xe >= tau && xe > kNegInf) {
        ++n;
        safe += ex2((xe - m) * kLog2e);
      }
    }
    sum = pack2(s0, safe);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum = add2(sum, __shfl_xor_sync(0xffffffffu, sum, o));
  n = __reduce_add_sync(0xffffffffu, n);
  if (log_parts > 0) {
    if (lane < parts) {
      st_cluster(&slots.sums[own_slot], r0 + lane, sum);
      st_cluster(&slots.count[own_slot], r0 + lane, __int_as_float(n));
    }
  } else if (lane == 0) {
    slots.sums[own_slot] = sum;
    slots.count[own_slot] = __int_as_float(n);
  }
  grp.meet();

  const SideStats st = stats_from<TIn>(grp, slots, r0, m, p, has_a, z_a);
  const bool weighted = p.weight_kind != DVP_WEIGHT_NONE;
  if (both) {
    if (second && part == 0 && tid < parts) {
      st_cluster(&slots.li, tid, logp_mp_of(st));
      st_cluster(&slots.member, tid, st.member ? 1.f : 0.f);
    }
    cluster_arrive();
  }
  const auto ratio_of = [&] {
    return has_a ? log_ratio_from(p.mode, st.member, logp_mp_of(st), slots.li) : __int_as_float(0x7fc00000);
  };

  // ---- the gradient (row_grad's arithmetic)
  if constexpr (kGrad != Grad::kNone) {
    if (!second) {
      float g = p.upstream[t];
      if (weighted && both) {  // weights need inference rows
        cluster_wait();
        const float w = has_a ? token_weight(ratio_of(), p.weight_kind, p.weight_lo, p.weight_hi) : __int_as_float(0x7fc00000);
        if (w == w) g *= w;
        if (p.weight_out && part == 0 && tid == 0) p.weight_out[t] = w;
      }
      TGrad *grow = reinterpret_cast<TGrad *>(p.grad) + t * p.ld_grad;
      TGrad *gbase = grow + (v.base - v.row);
      const float s_tot = st.s_x + st.e_a + st.s_mask;
      const bool live = st.live;
      const float coef = live ? -g / s_tot : 0.f;
      const float entry_a = st.member ? g * ((st.s_x + st.s_mask) / s_tot) : 0.f;
      const int a_here = live && st.member ? a : -1, g_here = a_here >= 0 ? g_a : -1;
      const float tau_g = live ? fmaxf(tau, -FLT_MAX) : -kNegInf;  // +inf: nothing passes
      if (k_extra < v.V) {
        const float out = xe >= tau_g ? coef * ex2((xe - m) * kLog2e) : 0.f;
        grow[k_extra] = Storage<TGrad>::narrow(k_extra == a_here ? entry_a : out);
      }
      float mc = m, cf = coef;
      if constexpr (kFoldedGrad<TIn, TGrad>) {
        mc = m * kLog2e;
        cf = coef * ex2(-fmaf(m, kLog2e, -mc));
      }
      const uint64_t m2 = pack2(-mc, -mc), cf2 = pack2(cf, cf);
#pragma unroll
      for (int u = 0; u < kGran; ++u) {
        const int gi = u * n_thr + tid, n_here = min(32, v.n_full - (gi - lane));
        if (n_here <= 0 || !DVP_IN((long long)(gi - lane + n_here) * kElems - 1, V, DVP_OOB_GLOBAL)) break;
        const bool hot = live && lane < n_here && gr[u].max() >= tau_g, any = __any_sync(0xffffffffu, hot);
        TGrad *dst = gbase + (size_t)gi * kElems;
        if constexpr (kGrad == Grad::kLoose) {
          constexpr int kWords = kGradWords<TIn, TGrad>;
          uint32_t w[kWords];
#pragma unroll
          for (int i = 0; i < kWords; ++i) w[i] = 0;
          if (hot) grad_words<TIn, TGrad, kFoldedGrad<TIn, TGrad>>(gr[u], tau_g, tau_p, m2, cf2, w);
          store_shifted(w, any, dst - lane * kElems, n_here, shift_smem + warp * kShiftWords);
          __syncwarp();  // the sampled token's entry replaces what a lane of the warp stored there
        } else if (lane < n_here) {
          if (any)
            grad_granule<TIn, TGrad, kFoldedGrad<TIn, TGrad>>(gr[u], dst, tau_g, tau_p, m2, cf2);
          else
            store_zero_granule<TGrad, kElems>(dst);
        }
        if (gi == g_here) grow[a_here] = Storage<TGrad>::narrow(entry_a);
      }
    }
  }

  // ---- per-token results
  if (both && !(kGrad != Grad::kNone && weighted && !second)) cluster_wait();
  const dvp_side_out &out = second ? p.out_i : p.out_t;
  if (part == 0 && tid == 0) {
    SideStats w = st;
    w.lse = lse_from_logsum({st.m, c, st.sum_s});
    (void)finish_side(out, t, w, has_id, bad_id);
    if (!second) {
      if (p.flags)
        p.flags[t] = (uint8_t)((st.member ? DVP_FLAG_IN_TRAIN : 0) | (both && slots.member != 0.f ? DVP_FLAG_IN_INFER : 0) |
                               (has_id ? 0 : DVP_FLAG_NO_ID) | (bad_id ? DVP_FLAG_BAD_ID : 0));
      if (p.log_ratio) p.log_ratio[t] = ratio_of();
    }
  }
  if (out.mask) write_mask_row<TIn>(v.row, v.V, tau, out.mask + t * ((p.V + 31) / 32), part, parts);
}

struct Shape {
  int threads, log_parts, gran;
};
// Is the call one for this kernel, and with how many threads and blocks a row?  Every row's granules have to fit the chip at
// once, 1,024 threads on an SM with four of them, or with five where four are not enough (a few per cent slower where they
// are: 148 x 32,000 with the gradient 12.7 / 13.5 us a call); while it has room, more threads a row are faster.  Clusters are
// begun one after the other, so that many of them cost more than they save: up to 512 tokens, 256 without a gradient; and
// those of several blocks a row take whole SMs of one part of the chip, of which some are left over: up to three quarters of
// the threads.  A row of one policy needs no cluster while one block holds it with three granules a thread.  Device
// us, the row kernel / two or four blocks / one: 30 x 8,200 bfloat16 4.1 / 5.1 / 4.1, 30 x 16,000 4.6 / 5.0 / 4.3, 30 x 24,000 5.9 /
// 5.1 / 4.7, 1 x 7,000 float32 4.2 / 4.6 / 3.7, 30 x 12,001 4.9 / 5.0 / 4.4.  With the gradient two: 12 x 8,200 bfloat16 6.0 / 6.0 / 4.9,
// 30 x 16,000 7.4 / 6.2 / 5.9, 30 x 20,001 8.8 / 6.0 / 6.8.
// Device us, the row kernel / this one (a graph of 20 calls): with the gradient 64 x 4,096 float32 7.4 / 5.2, 300 x 8,000 float16
// 10.9 / 8.1, 400 x 2,100 bfloat16 10.1 / 7.4, 148 x 32,000 15.4 / 11.2, 24 x 100,000 13.9 / 11.8, 8 x 262,144 12.9 / 11.7, 512 x 4,000
// 10.5 / 8.6, weighted 148 x 2,312 float32 7.5 / 5.7;  forward 4 x 20,000 5.7 / 5.3, 256 x 4,000 5.4 / 5.4, 148 x 32,000 11.2 / 8.3,
// 12 x 151,936 11.3 / 8.6; one policy 64 x 30,000 7.9 / 5.3.  Five granules: 16 x 151,936 12.2 / 9.6 and with the gradient 15.5 /
// 13.2, 140 x 40,000 13.1 / 8.9 and 17.8 / 13.4, 250 x 20,000 10.9 / 9.2 and 14.8 / 13.2.  Beyond: with the gradient 1,000 x 2,048 11.3 /
// 12.6, 72 x 50,000 (two blocks a row) 16.2 / 16.5; forward 600 x 4,000 7.5 / 9.9, 72 x 50,000 11.9 / 13.2, 16 x 151,936 in eight
// blocks of four granules 12.1 / 12.4; one policy 500 x 4,000 4.4 / 4.6.  Inside, where the chip is full, as fast: forward 256 x 16,000
// bfloat16 8.4 / 8.4, 240 x 12,500 8.2 / 8.3; slower 256 x 2,100 5.4 / 5.6.
static inline bool shape_of(long long T, bool both, bool grad, long long n_gran, Shape *s) {
  constexpr long long kChip = 148 * 1024, kMost = 8 * kMaxBlk;
  const long long rows = both ? 2 * T : T;
  if (T > (grad ? 512 : 256)) return false;
  for (int gran = 4; gran <= 5; ++gran) {
    long long per_row = 64;  // threads
    while (per_row < kMost && per_row * gran < n_gran) per_row *= 2;
    if (per_row * gran < n_gran || rows * per_row > (per_row > kMaxBlk ? kChip / 4 * 3 : kChip)) continue;
    const bool one_block = !both && n_gran <= (grad ? 2 : 3) * kMaxBlk;
    while (per_row < (one_block ? kMaxBlk : kMost) && 4 * rows * per_row <= kChip && per_row <= n_gran) per_row *= 2;
    s->threads = (int)(per_row < kMaxBlk ? per_row : kMaxBlk);
    s->log_parts = 0;
    while ((long long)s->threads << s->log_parts < per_row) ++s->log_parts;
    s->gran = gran;
    return true;
  }
  return false;
}

template <typename TIn, typename TGrad, Grad kGrad>
static cudaError_t launch(const RowParams &p, const Shape &sh, cudaStream_t s) {
  auto k = sh.gran == 4 ? dvp_row_kernel_held<TIn, TGrad, kGrad, 4> : dvp_row_kernel_held<TIn, TGrad, kGrad, 5>;
  const int log_cluster = sh.log_parts + (p.infer ? 1 : 0);
  if (log_cluster > 3) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.T << log_cluster), 1, 1);
  cfg.blockDim = dim3((unsigned)sh.threads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1u << log_cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = log_cluster > 0 ? 1 : 0;
  const bool over_infer = kGrad != Grad::kNone && sh.log_parts == 0 && p.grad == p.infer;
  return cudaLaunchKernelEx(&cfg, k, p, sh.log_parts | (over_infer ? kOverInfer : 0));
}

}  // namespace held
}  // namespace dvp
