// The row pass of the fused LM-head entry point over one panel of fp32 logits, with the
// normalisation deferred.
//
// The logits contraction leaves every row's maximum (in pieces), so the threshold of
// Def. 5.1 is known before the panel is read and one sweep gives everything: the full sum,
// the masked sum and the count (Def. 5.2), and, written as it goes, the panel
//     P_tk = 2^14 e^{z_tk - m_t}  for k in V_S, k != a_t;   0 otherwise          (float16)
// which is the gradient of Prop. 5.4 up to a factor per row that is known only at the end of
// the row: G_tk = c_t P_tk + 1[k = a_t] q_t with
//     c_t = -g_t / (2^14 s_S,t),   q_t = g_t s_{S\a},t / s_S,t   (= g_t (1 - pi^mp(a_t)), no cancellation).
// The factor goes where it costs nothing: d_hidden_t = c_t (P W)_t + q_t W_a (a row scale in the
// contraction's epilogue, one row of W added), d_w = P^T diag(c) hidden + sum_t q_t e_a hidden_t^T
// (the hidden rows are scaled while they are converted to float16, the 1[k = a] terms are
// added to d_w in a fixed order).  The panel is read once and written once.
#pragma once

#include "dvp_rows_impl.cuh"
#include "dvp_rows_two_sweeps.cuh"

namespace dvp {
namespace panel {

constexpr float kPScale = 16384.f;  // 2^14: P uses float16's normal range for members down to 4e-9 of the maximum

struct PanelParams {
  RowParams row;       // train = the fp32 panel; ids, upstream, T, V, ld_train, log_rho, outputs, weights
  // of the inference rows' pass, or null: ln pi^mp_infer(a) per token, and flags whose DVP_FLAG_IN_TRAIN bit
  // says "a in V'_S"
  const float *logp_mp_i;
  const uint8_t *flags_i;
  const float *row_max;  // the row maxima that the logits contraction left, in pieces: the maximum of row t is
  long long row_max_ld;  // the largest of row_max[t * row_max_ld + i], i < row_max_n
  int row_max_n;
  __half *P;           // [T, ld_p]
  long long ld_p;
  float *row_scale;    // [T] c_t (0 for a row without a gradient): scale of the row in d_hidden's epilogue
  float *hid_scale;    // [T] c_t K, K = 2^14 * scale / 512: scale of the hidden row in d_w's contraction
                       // (|c_t K| < 32, so hidden entries up to 2047 fit float16)
  float *a_coef;       // [T] q_t (0 for a row without a gradient)
  const float *scale;  // device scalar, the power of two taken from max |upstream|
};

struct PanelSums {
  float s_all, s_safe_x;  // sums of e^{z - m}: every token; the safe set without the sampled token
  int n;                  // |V_S|
};

template <bool kWhole>
__device__ __forceinline__ void absorb_panel(const Granule<float> &gr, int g, int V, int a, float m, float tau,
                                             PanelSums &acc, __half *prow) {
  constexpr int kElems = 8;
  float x[kElems];
  gr.get(x);
  const int ja = a - g * kElems;
  float all = 0.f;
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < kElems; j += 2) {
    float o[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float e = ex2((x[j + u] - m) * kLog2e);  // the fill of a ragged last granule is -inf: e = 0
      all += e;
      const bool keep = x[j + u] >= tau && x[j + u] > kNegInf;
      o[u] = 0.f;
      if (keep) {
        ++acc.n;
        if (j + u != ja) {
          acc.s_safe_x += e;
          o[u] = e * kPScale;
        }
      }
    }
    const __half2 h2 = __floats2half2_rn(o[0], o[1]);
    w[j / 2] = *reinterpret_cast<const uint32_t *>(&h2);
  }
  acc.s_all += all;
  if constexpr (kWhole) {
    *reinterpret_cast<uint4 *>(prow + (size_t)g * kElems) = make_uint4(w[0], w[1], w[2], w[3]);
  } else {
    const __half *h = reinterpret_cast<const __half *>(w);
#pragma unroll
    for (int j = 0; j < kElems; ++j) {
      const long long k = (long long)g * kElems + j;
      if (k < V) prow[k] = h[j];
    }
  }
}

// The sums of a row are 512 partial ones, kSets of them a thread: the i-th over the granules i, i + 512, ..., however many
// threads a block has.  Every set has kAhead granules in flight, the first of them while the row's maximum is found.
constexpr int kSums = 512;
template <int kSets, int kAhead>
__device__ __forceinline__ void panel_row(const PanelParams &pp, const long long t, float *scratch) {
  const RowParams &p = pp.row;
  constexpr int kElems = 8, kThreads = kSums / kSets;
  DVP_BOUNDS_BEGIN(p.bounds_status);
  DVP_BOUNDS_SET(n_gran, (p.V + kElems - 1) / kElems);
  DVP_BOUNDS_SET(V, p.V);
  DVP_BOUNDS_SYNC();
  const int V = (int)p.V, tid = (int)threadIdx.x;
  const float *row = reinterpret_cast<const float *>(p.train) + t * p.ld_train;
  __half *prow = pp.P + t * pp.ld_p;
  const int n_full = V / kElems;
  // the logits are not read again, the gradient panel is, by two contractions: L2 keeps the latter (without: 3,891 x 2,752
  // x 58,933 3,894 us a call, 3,710 with; 4,727 x 2,864 x 12,179 1,233 / 1,196)
  auto load_last = [&](Granule<float> &gr, int g) {
    if (DVP_IN((long long)g * kElems + kElems - 1, V, DVP_OOB_GLOBAL)) ld_last32(row + (size_t)g * kElems, gr.w);
  };
  Granule<float> gr[kAhead][kSets];
#pragma unroll
  for (int u = 0; u < kAhead; ++u)
#pragma unroll
    for (int v = 0; v < kSets; ++v)
      if (tid + v * kThreads + u * kSums < n_full) load_last(gr[u][v], tid + v * kThreads + u * kSums);
  const long long id = load_id(p.ids, p.id_is_i32, t);
  const bool has_id = id >= 0, bad_id = id >= p.V;
  const int a = (has_id && !bad_id) ? (int)id : -1;

  const float *pieces = pp.row_max + t * pp.row_max_ld;
  float mx = kNegInf;
  for (int i = tid; i < pp.row_max_n; i += kThreads) mx = fmaxf(mx, pieces[i]);
  const float m = block_reduce_max(mx, scratch);

  SideStats st;
  st.m = m;
  st.tau = threshold_f32(m, p.log_rho);
  const bool has_a = a >= 0;
  st.z_a = has_a ? row[a] : 0.f;
  st.member = has_a && st.z_a >= st.tau;
  st.e_a = st.member ? ex2((st.z_a - m) * kLog2e) : 0.f;

  PanelSums acc[kSets];
#pragma unroll
  for (int v = 0; v < kSets; ++v) acc[v] = {0.f, 0.f, 0};
  for (int g0 = tid; g0 < n_full; g0 += kAhead * kSums) {
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
#pragma unroll
      for (int v = 0; v < kSets; ++v) {
        const int g = g0 + u * kSums + v * kThreads;
        if (g < n_full) absorb_panel<true>(gr[u][v], g, V, a, m, st.tau, acc[v], prow);
        if (g + kAhead * kSums < n_full) load_last(gr[u][v], g + kAhead * kSums);
      }
    }
  }
#pragma unroll
  for (int v = 0; v < kSets; ++v) {
    if (n_full * kElems < V && n_full % kSums == tid + v * kThreads) {  // the ragged last granule
      gr[0][0].load_any(row, V, n_full, n_full);
      absorb_panel<false>(gr[0][0], n_full, V, a, m, st.tau, acc[v], prow);
    }
  }
  {  // the partial sums by warps of 32, then the 16 of those, in a fixed order
    const int lane = tid & 31, warp = tid >> 5;
    constexpr int kParts = kSums / 32;
    __syncthreads();
#pragma unroll
    for (int v = 0; v < kSets; ++v) {
      const SumCount x = warp_reduce(SumCount{acc[v].s_safe_x, acc[v].n});
      const SumCount y = warp_reduce(SumCount{acc[v].s_all, 0});
      if (lane == 0) {
        const int at = warp + v * (kThreads / 32);
        scratch[at] = x.s;
        scratch[32 + at] = y.s;
        scratch[64 + at] = __int_as_float(x.n);
      }
    }
    __syncthreads();
    const SumCount safe = warp_reduce(
        lane < kParts ? SumCount{scratch[lane], __float_as_int(scratch[64 + lane])} : SumCount{0.f, 0});
    const SumCount all = warp_reduce(SumCount{lane < kParts ? scratch[32 + lane] : 0.f, 0});
    st.s_x = safe.s;
    st.n = safe.n;
    st.sum_s = all.s;
  }
  st.lse = (double)m + (double)logf(st.sum_s);
  st.sum_c = (double)m * (double)kLog2e;
  set_mask_mass(st, V, 0, 0.f, has_a);

  if (threadIdx.x == 0) {
    finish_side(p.out_t, t, st, has_id, bad_id);
    const bool in_i = pp.flags_i && (pp.flags_i[t] & DVP_FLAG_IN_TRAIN);
    if (p.flags)
      p.flags[t] = (uint8_t)((st.member ? DVP_FLAG_IN_TRAIN : 0) | (in_i ? DVP_FLAG_IN_INFER : 0) |
                             (has_id ? 0 : DVP_FLAG_NO_ID) | (bad_id ? DVP_FLAG_BAD_ID : 0));
    const float ratio = a >= 0 && pp.logp_mp_i ? log_ratio_of(st.member, in_i, logp_mp_of(st), pp.logp_mp_i[t])
                                               : __int_as_float(0x7fc00000);
    if (p.log_ratio) p.log_ratio[t] = ratio;
    float g = p.upstream[t];
    if (p.weight_kind != DVP_WEIGHT_NONE) {
      const float w = token_weight(ratio, p.weight_kind, p.weight_lo, p.weight_hi);
      if (w == w) g *= w;
      if (p.weight_out) p.weight_out[t] = w;
    }
    // a missing sampled token, or a pruned one, has weight zero: no gradient from this row
    const bool live = st.live && st.member;
    const float s_safe = st.s_x + st.e_a;  // >= 1: the maximum is always in the set
    const float c = live ? -g / (s_safe * kPScale) : 0.f;
    pp.row_scale[t] = c;
    pp.hid_scale[t] = live ? -g * (*pp.scale * (1.f / 512.f)) / s_safe : 0.f;
    pp.a_coef[t] = live ? g * (st.s_x / s_safe) : 0.f;
  }
  if (p.out_t.mask) {  // optional packed membership mask (diagnostic output, plain loads)
    uint32_t *mask_row = p.out_t.mask + t * ((p.V + 31) / 32);
    const int n_words = (V + 31) / 32;
    for (int w = threadIdx.x; w < n_words; w += blockDim.x) {
      uint32_t bits = 0;
      for (int b = 0; b < 32; ++b) {
        const long long k = (long long)w * 32 + b;
        if (k < V && row[k] >= st.tau) bits |= 1u << b;
      }
      mask_row[w] = bits;
    }
  }
}
template <int kSets, int kAhead>
__global__ void __launch_bounds__(kSums / kSets, 2 * kSets) dvp_panel_kernel(const PanelParams pp) {
  __shared__ float scratch[96];
  begin_after();
  panel_row<kSets, kAhead>(pp, blockIdx.x, scratch);
}

// The inference rows and the panel's in one launch, for calls of one panel whose panel rows need nothing of the others: the
// inference rows come first, in the places that the logits contraction's last, partly filled wave leaves, and the panel's
// rows follow without a wave that ends between them.  sum_ranges_kernel forms the log-ratios.  kPieces: inference rows off
// the 32-byte grid.  us a call, two launches / one: 512 x 1,024 x 32,000 184.7 / 169.6, 767 x 1,448 x 10,474 154.7 / 140.4, 163 x
// 416 x 45,277 132.1 / 113.6, 1,200 x 1,024 x 16,000 204.3 / 195.4, 3,000 x 512 x 16,000 304 / 295, 6,000 x 512 x 16,001 640 / 626.  (Four granules a thread in flight in the
// panel's rows instead of two: 2 % more time.)
template <bool kPieces>
__global__ void __launch_bounds__(kSums / 2, 4) dvp_both_rows_kernel(const __grid_constant__ PanelParams pp,
                                                                     const __grid_constant__ RowParams infer) {
  extern __shared__ __align__(16) float smem[];
  const long long b = blockIdx.x;
  if (b < infer.T) {
    begin_after(true);
    if constexpr (kPieces)
      two_sweeps::row_of_pieces<2>(infer, b, smem);
    else
      two_sweeps::row_of_granules<kSums / 2>(infer, b, smem);
  } else {
    begin_after();
    panel_row<2, 1>(pp, b - infer.T, smem);
  }
}

// d_hidden[t, :] = c_t sum_i part_i[t, :] + q_t W[a_t, :], the ranges in order: diag(c) P W from its K ranges and
// the 1[k = a] term, in fp32.  One range: `part` may be d_hidden itself (c_t applied already: scale null).
// `meet`: the two policies' rows meet here (dvp_both_rows_kernel): flags and log-ratios.
struct MeetParams {
  const float *logp_mp_t, *logp_mp_i;
  uint8_t *flags;
  const uint8_t *flags_i;
  float *log_ratio;  // or null
};
__global__ void __launch_bounds__(256) sum_ranges_kernel(const float *part, long long range_stride, long long ld_part,
                                                         int ranges, const float *scale, float *d_hidden,
                                                         long long ld_dh, const __nv_bfloat16 *w, long long ld_w,
                                                         const void *ids, int id_is_i32, const float *a_coef, int H,
                                                         const MeetParams meet) {
  begin_after();
  const unsigned per_row = (unsigned)(H + 1023) / 1024;
  const long long t = blockIdx.x / per_row;
  const int h = (int)((blockIdx.x % per_row) * 1024 + threadIdx.x * 4);
  if (meet.flags_i && h == 0) {
    const uint8_t f = meet.flags[t];
    const bool in_t = f & DVP_FLAG_IN_TRAIN, in_i = meet.flags_i[t] & DVP_FLAG_IN_TRAIN;
    meet.flags[t] = (uint8_t)(f | (in_i ? DVP_FLAG_IN_INFER : 0));
    if (meet.log_ratio)
      meet.log_ratio[t] = f & (DVP_FLAG_NO_ID | DVP_FLAG_BAD_ID)
                              ? __int_as_float(0x7fc00000)
                              : log_ratio_of(in_t, in_i, meet.logp_mp_t[t], meet.logp_mp_i[t]);
  }
  if (h >= H) return;
  const float q = a_coef[t], c = scale ? scale[t] : 1.f;
  const __nv_bfloat16 *wa = q != 0.f ? w + load_id(ids, id_is_i32, t) * ld_w + h : nullptr;
  const float *src = part + t * ld_part + h;
  float *out = d_hidden + t * ld_dh + h;
  if (h + 4 <= H) {  // strides are multiples of 8 elements
    float4 acc = *reinterpret_cast<const float4 *>(src);
    for (int i = 1; i < ranges; ++i) {
      const float4 v = *reinterpret_cast<const float4 *>(src + i * range_stride);
      acc.x += v.x, acc.y += v.y, acc.z += v.z, acc.w += v.w;
    }
    acc.x *= c, acc.y *= c, acc.z *= c, acc.w *= c;
    if (wa) {
      const uint2 raw = *reinterpret_cast<const uint2 *>(wa);
      acc.x = fmaf(q, __uint_as_float(raw.x << 16), acc.x);
      acc.y = fmaf(q, __uint_as_float(raw.x & 0xffff0000u), acc.y);
      acc.z = fmaf(q, __uint_as_float(raw.y << 16), acc.z);
      acc.w = fmaf(q, __uint_as_float(raw.y & 0xffff0000u), acc.w);
    }
    *reinterpret_cast<float4 *>(out) = acc;
  } else {
    for (int j = 0; h + j < H; ++j) {
      float acc = src[j];
      for (int i = 1; i < ranges; ++i) acc += src[i * range_stride + j];
      acc *= c;
      out[j] = wa ? fmaf(q, __bfloat162float(wa[j]), acc) : acc;
    }
  }
}

// d_w[a, :] += sum over the tokens t of the chunk (at most 4096) with a_t = a, in token order, of q_t hidden[t, :].
// One warp per token; the warp of the first token with an id does all tokens with that id, and nobody else adds to that
// row.  A block's eight warps look for theirs among the chunk's ids in shared memory, four to a load; loads go out in
// batches, those of d_w's row among them (reductions in memory instead, 767 x 1,448 x 10,474: 165 us a call, 160 this way).
// With a block a token, which read all ids itself, element by element, the kernel by itself took 15 us (512 x 1,024 x 32,000),
// 46 (767 x 1,448 x 10,474) and 110 (8,192 x 1,024 x 20,011); it takes 8, 16 and 53, of which calls show a part: 206.4 -> 204.9,
// 163.5 -> 160.0 and 1,509 -> 1,477 us.  (Sorting the ids first: 35 to 41 us by itself.  In the epilogue of d_w's contraction:
// 27 us more a call than this, 512 x 1,024 x 32,000.)
constexpr int kIdChunk = 4096;
constexpr int kSampledWarps = 8;
constexpr size_t kSampledSmem = (size_t)kIdChunk * 4 + kSampledWarps * kIdChunk / 8;
__global__ void __launch_bounds__(kSampledWarps * 32)
add_sampled_hidden_kernel(const void *ids, int id_is_i32, const float *a_coef, int n, const __nv_bfloat16 *hidden,
                          long long ld_hidden, float *d_w, long long ld_dw, int H) {
  extern __shared__ __align__(16) int id_of[];  // [kIdChunk], -1: nothing to add
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t *same = reinterpret_cast<uint32_t *>(id_of + kIdChunk) + warp * (kIdChunk / 32);  // bit j: token j has our id
  const int i = (int)blockIdx.x * kSampledWarps + warp;
  // Which token adds what needs only the ids and the panel's coefficients, which were complete before d_w's contraction
  // began: it is found while that ends.  d_w itself is waited for.  (us a call with the wait in front / here: 163 x 416 x 45,277
  // 115.0 / 113.6, 1,200 x 1,024 x 16,000 197.0 / 195.4, 3,000 x 512 x 16,000 301 / 295; 512 x 1,024 x 32,000 173 / 170 and 767 x
  // 1,448 x 10,474 140.4 / 140.4, no more than processes differ.)
  const int n4 = (n + 127) & ~127;
  constexpr int kBlk = kSampledWarps * 32, kLoads = 8;  // all of a batch before the first is stored
  for (int j0 = threadIdx.x; j0 < n4; j0 += kLoads * kBlk) {
    long long of[kLoads];
    float c[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int at = min(j0 + u * kBlk, n - 1);
      of[u] = load_id(ids, id_is_i32, at);
      c[u] = a_coef[at];
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int j = j0 + u * kBlk;
      if (j < n4) id_of[j] = j < n && c[u] != 0.f ? (int)of[u] : -1;
    }
  }
  for (int k = lane; k < kIdChunk / 32; k += 32) same[k] = 0;
  __syncthreads();
  const int a = i < n ? id_of[i] : -1;
  if (a < 0) {
    begin_after();
    return;
  }
  bool earlier = false, later = false;
  for (int j = lane * 4; j < n4; j += 128) {
    const int4 v = *reinterpret_cast<const int4 *>(id_of + j);
    const uint32_t bits = (v.x == a ? 1u : 0u) | (v.y == a ? 2u : 0u) | (v.z == a ? 4u : 0u) | (v.w == a ? 8u : 0u);
    if (bits) {
      if (j < i && bits & ((1u << min(4, i - j)) - 1u)) earlier = true;
      if (j + 3 > i && bits & ~((2u << max(0, i - j)) - (j <= i ? 1u : 2u))) {
        later = true;
        atomicOr(&same[j >> 5], bits << (j & 31));
      }
    }
  }
  if (__any_sync(0xffffffffu, earlier)) {
    begin_after();
    return;
  }
  later = __any_sync(0xffffffffu, later);
  __syncwarp();
  const float q = a_coef[i];
  float *out = d_w + (long long)a * ld_dw;
  const __nv_bfloat16 *own = hidden + (long long)i * ld_hidden;
  // f(t): for the later tokens with this id, in order
  auto others = [&](auto f) {
    for (int k = i >> 5; k < (n + 31) / 32; ++k)
      for (uint32_t m = same[k]; m; m &= m - 1) {
        const int t = k * 32 + __ffs(m) - 1;
        if (t > i) f(t);
      }
  };
  begin_after();
  constexpr int kAhead = 3;  // pieces of 8 columns in flight
  for (int h0 = lane * 8; h0 + 8 <= H; h0 += kAhead * 256) {  // strides are multiples of 8 elements
    uint4 raw[kAhead];
    float was[kAhead][8];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int h = h0 + u * 256;
      if (h + 8 > H) break;
      raw[u] = *reinterpret_cast<const uint4 *>(own + h);
      asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                   : "=f"(was[u][0]), "=f"(was[u][1]), "=f"(was[u][2]), "=f"(was[u][3]), "=f"(was[u][4]), "=f"(was[u][5]),
                     "=f"(was[u][6]), "=f"(was[u][7])
                   : "l"(out + h));
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int h = h0 + u * 256;
      if (h + 8 > H) break;
      float x[8], acc[8];
      Storage<__nv_bfloat16>::unpack(raw[u], x);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = q * x[j];
      if (later)
        others([&](int t) {
          const float c = a_coef[t];
          Storage<__nv_bfloat16>::unpack(*reinterpret_cast<const uint4 *>(hidden + (long long)t * ld_hidden + h), x);
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j] = fmaf(c, x[j], acc[j]);
        });
      asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(out + h), "f"(was[u][0] + acc[0]),
                   "f"(was[u][1] + acc[1]), "f"(was[u][2] + acc[2]), "f"(was[u][3] + acc[3]), "f"(was[u][4] + acc[4]),
                   "f"(was[u][5] + acc[5]), "f"(was[u][6] + acc[6]), "f"(was[u][7] + acc[7])
                   : "memory");
    }
  }
  for (int h = (H & ~7) + lane; h < H; h += 32) {
    float acc = q * __bfloat162float(own[h]);
    if (later) others([&](int t) { acc = fmaf(a_coef[t], __bfloat162float(hidden[(long long)t * ld_hidden + h]), acc); });
    out[h] += acc;
  }
}

}  // namespace panel
}  // namespace dvp
