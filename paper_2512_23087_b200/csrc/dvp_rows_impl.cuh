// Row kernels of Dynamic Vocabulary Pruning for sm_100a.
//
// One thread block (or a cluster of them) owns one row.  The row is streamed from HBM once
// (sweep 1) in 32-byte granules, one DRAM sector per lane and load, two
// pipeline stages deep.  While it streams, every thread adds up what it sees against a
// guess of the row's maximum: the full sum, and the masked sum and count of Def. 5.2
// under the guess's threshold; the maximum of each granule stays in shared memory
// (float32: a bfloat16 upper bound).  Once the row maximum, hence the threshold of
// Def. 5.1, is known, sweep 2 revisits only what came before the guess was the maximum,
// and of it only granules whose bound reaches the threshold.  Sweep 3 (gradient,
// Prop. 5.4) reads the granules with safe tokens again and writes zeros for all the
// others without reading anything.
// With a sparse safe set a row costs one HBM read per logit matrix and one HBM write
// of the gradient; with a dense safe set sweep 3 reads the row a second time.
#pragma once
#include <float.h>
#include <limits.h>

#include <type_traits>

#include "dvp_common.cuh"

namespace dvp {

template <typename T>
struct Pair;
template <>
struct Pair<__nv_bfloat16> {
  using type = __nv_bfloat162;
};
template <>
struct Pair<__half> {
  using type = __half2;
};

// ---- a 32-byte granule of a row, kept packed as loaded ------------------------

template <typename TIn>
struct Granule {
  static constexpr int kElems = 32 / (int)sizeof(TIn);
  uint32_t w[8];

  __device__ __forceinline__ void load(const TIn *p) { ld_stream32(p, w); }

  // Granule `g` of a row of V elements; elements past V read as -inf.
  __device__ __forceinline__ void load_any(const TIn *row, int V, int n_full, int g) {
    // granules past the end of the row are legal here (they read as -inf); what the
    // bounds-checking build verifies is that the vector load below stays inside the row
    if (g < 0 || (g < n_full && !DVP_IN((long long)g * kElems + kElems - 1, V, DVP_OOB_GLOBAL))) {
      (void)DVP_IN(g, n_gran, DVP_OOB_GRANULE);
      const TIn fill = Storage<TIn>::narrow(kNegInf);
      uint32_t f = 0;
      if constexpr (sizeof(TIn) == 4) {
        f = *reinterpret_cast<const uint32_t *>(&fill);
      } else {
        const uint32_t h = *reinterpret_cast<const uint16_t *>(&fill);
        f = h | (h << 16);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = f;
      return;
    }
    if (g < n_full) {
      load(row + (size_t)g * kElems);
    } else {
      __align__(16) TIn tmp[kElems];
#pragma unroll
      for (int j = 0; j < kElems; ++j) {
        const long long k = (long long)g * kElems + j;
        tmp[j] = k < V ? row[k] : Storage<TIn>::narrow(kNegInf);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = reinterpret_cast<const uint32_t *>(tmp)[i];
    }
  }

  // Granule `g` of the row's n_full whole granules; any other index reads as -inf.  The row
  // kernel's sweeps use this one: the elements behind the last whole granule are not theirs (a few
  // threads take them one by one), so no sweep carries the element-wise code of a ragged granule.
  __device__ __forceinline__ void load_whole(const TIn *row, int n_full, int g) {
    if (g < 0 || g >= n_full || !DVP_IN((long long)g * kElems + kElems - 1, V, DVP_OOB_GLOBAL)) {
      if (g < 0) (void)DVP_IN(g, n_gran, DVP_OOB_GRANULE);
      const TIn fill = Storage<TIn>::narrow(kNegInf);
      uint32_t f = 0;
      if constexpr (sizeof(TIn) == 4) {
        f = *reinterpret_cast<const uint32_t *>(&fill);
      } else {
        const uint32_t h = *reinterpret_cast<const uint16_t *>(&fill);
        f = h | (h << 16);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = f;
      return;
    }
    load(row + (size_t)g * kElems);
  }

  __device__ __forceinline__ void get(float *x) const {
    constexpr int kHalf = kElems / 2;
    Storage<TIn>::unpack(make_uint4(w[0], w[1], w[2], w[3]), x);
    Storage<TIn>::unpack(make_uint4(w[4], w[5], w[6], w[7]), x + kHalf);
  }

  __device__ __forceinline__ float max() const {
    if constexpr (sizeof(TIn) == 4) {
      float m = __uint_as_float(w[0]);
#pragma unroll
      for (int i = 1; i < 8; ++i) m = fmaxf(m, __uint_as_float(w[i]));
      return m;
    } else {
      // packed two-at-a-time maxima, then the two halves of the last pair
      using T2 = typename Pair<TIn>::type;
      T2 p[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) p[i] = *reinterpret_cast<const T2 *>(&w[i]);
#pragma unroll
      for (int s = 4; s > 0; s >>= 1)
#pragma unroll
        for (int i = 0; i < s; ++i) p[i] = __hmax2(p[i], p[i + s]);
      return fmaxf(Storage<TIn>::widen(p[0].x), Storage<TIn>::widen(p[0].y));
    }
  }
};

// Upper bound of a float as a bfloat16 bit pattern (round toward +inf).
__device__ __forceinline__ uint16_t bf16_bits_round_up(float v) {
  const uint32_t b = __float_as_uint(v);
  // positive: bump the magnitude unless the low half is zero; negative: truncate
  return (uint16_t)(((b & 0x80000000u) ? b : b + 0xffffu) >> 16);
}
// Largest bfloat16 that is <= v, as a float: comparing the stored upper bounds with
// it flags a superset of the granules whose bound reaches v.
__device__ __forceinline__ float bf16_round_down(float v) {
  const uint32_t b = __float_as_uint(v);
  return __uint_as_float(((b & 0x80000000u) ? b + 0xffffu : b) & 0xffff0000u);
}
template <typename TGrad, int kElems>
__device__ __forceinline__ void store_granule(TGrad *dst, const float *out) {
  constexpr int kBytes = kElems * (int)sizeof(TGrad);
  if constexpr (sizeof(TGrad) == 4) {
#pragma unroll
    for (int i = 0; i < kElems; i += 8) {
      uint32_t w[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = __float_as_uint(out[i + j]);
      st_stream32(dst + i, w);
    }
  } else {
    uint32_t w[kElems / 2];
#pragma unroll
    for (int i = 0; i < kElems / 2; ++i) {
      TGrad lo = Storage<TGrad>::narrow(out[2 * i]), hi = Storage<TGrad>::narrow(out[2 * i + 1]);
      w[i] = (uint32_t) * reinterpret_cast<uint16_t *>(&lo) |
             ((uint32_t) * reinterpret_cast<uint16_t *>(&hi) << 16);
    }
    if constexpr (kBytes == 32) {
      uint32_t v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = w[i];
      st_stream32(dst, v);
    } else {
      static_assert(kBytes == 16, "granule of 8 floats stored as 8 halves");
      st_stream16(dst, make_uint4(w[0], w[1], w[2], w[3]));
    }
  }
}

template <typename TGrad, int kElems>
__device__ __forceinline__ void store_zero_granule(TGrad *dst) {
  constexpr int kBytes = kElems * (int)sizeof(TGrad);
  const uint32_t z[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  if constexpr (kBytes == 64) {
    st_stream32(dst, z);
    st_stream32(reinterpret_cast<char *>(dst) + 32, z);
  } else if constexpr (kBytes == 32) {
    st_stream32(dst, z);
  } else {
    st_stream16(dst, make_uint4(0, 0, 0, 0));
  }
}

// ---- granules that can hold a safe token ----------------------------------------
// Per warp, in the order (slot, lane): entry = ordinal of the granule among the
// warp's granules.  A warp whose hot granules do not fit (a dense safe set)
// walks all of its granules instead, which is then the efficient thing to do.
constexpr int kHotCap = 1024;  // 16-bit entries: slot * 32 + lane stays below 65536 for every row the bounds fit

struct HotList {
  uint16_t *slots;
  int count;  // granules at or above the threshold (may exceed kHotCap)
  __device__ __forceinline__ bool fits() const { return count <= kHotCap; }
};

// Contribution of one granule to the masked sum and the count (Def. 5.2).  tau is finite: no fill passes.
template <typename TIn>
__device__ __forceinline__ void granule_masked_sum(const Granule<TIn> &gr, float tau, float m, SumCount &sc) {
  constexpr int kElems = Granule<TIn>::kElems;
  float x[kElems];
  gr.get(x);
#pragma unroll
  for (int j = 0; j < kElems; ++j) {
    if (x[j] >= tau) {
      ++sc.n;
      sc.s += ex2((x[j] - m) * kLog2e);
    }
  }
}

// Gradient entries of one granule (Prop. 5.4, set fixed), stored to the row.
template <typename TIn, typename TGrad>
__device__ __forceinline__ void granule_grad(const Granule<TIn> &gr, TGrad *grow, int V, int n_full,
                                             int g, int a, float tau, float m, float coef,
                                             float g_a) {
  constexpr int kElems = Granule<TIn>::kElems;
  float x[kElems], out[kElems];
  gr.get(x);
  const int ja = a - g * kElems;
#pragma unroll
  for (int j = 0; j < kElems; ++j) {
    out[j] = x[j] >= tau ? coef * ex2((x[j] - m) * kLog2e) : 0.f;
    if (j == ja) out[j] = g_a;
  }
  // a granule past the end of the row is legal here (a hot list built for a threshold of -inf
  // names them): nothing of it is stored below.  A negative index is not.
  if (g < 0) {
    (void)DVP_IN(g, n_gran, DVP_OOB_GRANULE);
    return;
  }
  if (g < n_full) {
    if (!DVP_IN((long long)g * kElems + kElems - 1, V, DVP_OOB_GLOBAL)) return;
    store_granule<TGrad, kElems>(grow + (size_t)g * kElems, out);
  } else {
#pragma unroll
    for (int j = 0; j < kElems; ++j) {
      const long long k = (long long)g * kElems + j;
      if (k < V) grow[k] = Storage<TGrad>::narrow(out[j]);
    }
  }
}

// One pipeline stage of sweep 1: kStage granules of this thread.
template <typename TIn, int kStage>
struct Stage {
  Granule<TIn> g[kStage];
  // every granule of the step, the elements of a ragged last granule included
  __device__ __forceinline__ void load(const TIn *row, int V, int n_full, int step) {
    const int g0 = step * kStage * (int)blockDim.x + threadIdx.x;
    if ((step + 1) * kStage * (int)blockDim.x <= n_full &&
        DVP_IN(g0 + (kStage - 1) * (int)blockDim.x, n_gran, DVP_OOB_GRANULE)) {
#pragma unroll
      for (int u = 0; u < kStage; ++u)
        g[u].load(row + (size_t)(g0 + u * (int)blockDim.x) * Granule<TIn>::kElems);
    } else {
#pragma unroll
      for (int u = 0; u < kStage; ++u) g[u].load_any(row, V, n_full, g0 + u * (int)blockDim.x);
    }
  }
  // the whole granules of the step only
  template <int kBlk>
  __device__ __forceinline__ void load_block(const TIn *row, int n_full, int step) {
    const int g0 = step * kStage * kBlk + (int)threadIdx.x;
    if ((step + 1) * kStage * kBlk <= n_full && DVP_IN(g0 + (kStage - 1) * kBlk, n_gran, DVP_OOB_GRANULE)) {
      const TIn *p = row + (size_t)g0 * Granule<TIn>::kElems;
#pragma unroll
      for (int u = 0; u < kStage; ++u) g[u].load(p + u * kBlk * Granule<TIn>::kElems);
    } else {
#pragma unroll
      for (int u = 0; u < kStage; ++u) g[u].load_whole(row, n_full, g0 + u * kBlk);
    }
  }
  // granule `hole`, one of this step's, becomes -inf in the thread that holds it
  template <int kBlk>
  __device__ __forceinline__ void punch(int step, int hole) {
    const int u_here = hole - step * kStage * kBlk - (int)threadIdx.x;
#pragma unroll
    for (int u = 0; u < kStage; ++u)
      if (u_here == u * kBlk) g[u].load_whole(nullptr, 0, 0);
    __syncwarp();  // keeps this a branch: predicated, its moves would be issued in every step
  }
};

// ---- sweep 1 ---------------------------------------------------------------------

// Two floats in a 64-bit register pair: one FMA, addition or product for both.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// What depends on the storage type.  The maxima of a step's two granules are one word of shared memory:
// exact, in the storage type, for 2-byte logits; bfloat16 upper bounds for float32.
template <typename TIn>
struct SweepOps {  // 2-byte logits, two at a time
  using T2 = typename Pair<TIn>::type;
  using Max = T2;
  static __device__ __forceinline__ uint32_t bits(T2 v) { return *reinterpret_cast<const uint32_t *>(&v); }
  static __device__ __forceinline__ T2 pair(uint32_t v) { return *reinterpret_cast<const T2 *>(&v); }
  static __device__ __forceinline__ Max start(float v) {
    T2 r;
    r.x = r.y = Storage<TIn>::narrow(v);  // exact: v was stored as TIn
    return r;
  }
  static __device__ __forceinline__ T2 tree(const Granule<TIn> &g) {
    T2 p[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = pair(g.w[i]);
#pragma unroll
    for (int s = 4; s > 0; s >>= 1)
#pragma unroll
      for (int i = 0; i < s; ++i) p[i] = __hmax2(p[i], p[i + s]);
    return p[0];
  }
  // the step's word; raises the running maximum
  static __device__ __forceinline__ uint32_t bounds(const Stage<TIn, 2> &st, Max &mx) {
    const uint32_t a = bits(tree(st.g[0])), b = bits(tree(st.g[1]));
    const T2 w = __hmax2(pair(__byte_perm(a, b, 0x5410)), pair(__byte_perm(a, b, 0x7632)));
    mx = __hmax2(mx, w);
    return bits(w);
  }
  static __device__ __forceinline__ float value(Max m) {
    return fmaxf(Storage<TIn>::widen(m.x), Storage<TIn>::widen(m.y));
  }
  // 0x0000ffff, 0xffff0000: the step's first, second granule may hold a value that reaches the threshold
  using Key = uint32_t;
  static __device__ __forceinline__ Key key(float tau) { return threshold(tau); }
  static __device__ __forceinline__ uint32_t reach(uint32_t word, Key k) { return __hge2_mask(pair(word), pair(k)); }
  static constexpr uint32_t kTop = std::is_same<TIn, __nv_bfloat16>::value ? 0x7f7fu : 0x7bffu;  // largest finite
  // the threshold, rounded up to the storage type: a stored value reaches tau when it reaches that
  using Tau = uint32_t;
  static __device__ __forceinline__ Tau threshold(float tau) {
    T2 t;
    if constexpr (std::is_same<TIn, __nv_bfloat16>::value)
      t.x = __float2bfloat16_ru(tau);
    else
      t.x = __float2half_ru(tau);
    t.y = t.x;
    return bits(t);
  }
  // adds e0, e1 to s where the granule's pair i reaches the threshold and counts them in n (see count())
  static __device__ __forceinline__ void masked(const Granule<TIn> &g, int i, float, float, float e0, float e1, Tau tau,
                                                float &s, uint32_t &n) {
    if constexpr (std::is_same<TIn, __nv_bfloat16>::value)
      asm("{\n\t.reg .pred p, q;\n\tsetp.ge.bf16x2 p|q, %1, %2;\n\t"
          "@p add.f32 %0, %0, %3;\n\t@q add.f32 %0, %0, %4;\n\t}"
          : "+f"(s)
          : "r"(g.w[i]), "r"(tau), "f"(e0), "f"(e1));
    else
      asm("{\n\t.reg .pred p, q;\n\tsetp.ge.f16x2 p|q, %1, %2;\n\t"
          "@p add.f32 %0, %0, %3;\n\t@q add.f32 %0, %0, %4;\n\t}"
          : "+f"(s)
          : "r"(g.w[i]), "r"(tau), "f"(e0), "f"(e1));
    n += __hge2_mask(pair(g.w[i]), pair(tau));
  }
  // A mask has 0xffff in the halves that pass, so that a sum of masks is 0xffff n_lo + 0xffff0000 n_hi
  // = -(n_lo + 2^16 (n_hi - n_lo)) modulo 2^32: exact while both are below 2^16.
  static __device__ __forceinline__ int count(uint32_t cnt) {
    const uint32_t v = 0u - cnt, lo = v & 0xffffu;
    return (int)(lo + (((v >> 16) + lo) & 0xffffu));
  }
};
template <>
struct SweepOps<float> {
  using Max = float;
  static __device__ __forceinline__ Max start(float v) { return v; }
  static __device__ __forceinline__ uint32_t bounds(const Stage<float, 2> &st, Max &mx) {
    const float a = st.g[0].max(), b = st.g[1].max();
    mx = fmaxf(mx, fmaxf(a, b));
    return (uint32_t)bf16_bits_round_up(a) | ((uint32_t)bf16_bits_round_up(b) << 16);
  }
  static __device__ __forceinline__ float value(Max m) { return m; }
  using Key = uint32_t;  // the threshold rounded down to bfloat16, twice
  static __device__ __forceinline__ Key key(float tau) {
    const uint32_t b = __float_as_uint(bf16_round_down(tau));
    return b | (b >> 16);
  }
  static __device__ __forceinline__ uint32_t reach(uint32_t word, Key k) {
    return __hge2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&word), *reinterpret_cast<const __nv_bfloat162 *>(&k));
  }
  static constexpr uint32_t kTop = 0x7f7fu;
  using Tau = float;
  static __device__ __forceinline__ Tau threshold(float tau) { return tau; }
  static __device__ __forceinline__ void masked(const Granule<float> &, int, float x0, float x1, float e0, float e1,
                                                Tau tau, float &s, uint32_t &n) {
    if (x0 >= tau) {
      s += e0;
      ++n;
    }
    if (x1 >= tau) {
      s += e1;
      ++n;
    }
  }
  static __device__ __forceinline__ int count(uint32_t cnt) { return (int)cnt; }
};

// What a thread carries through sweep 1, all without the sampled token: the sum of 2^{z l - c}, c = fl(guess l),
// and the masked sum and count under the threshold of a guess of the row's maximum.
template <typename TIn>
struct Sweep1 {
  using Ops = SweepOps<TIn>;
  typename Ops::Max mx;    // the largest value seen
  typename Ops::Tau tau;   // the guess's threshold
  typename Ops::Key key;   // the same for the bounds
  float guess, c;          // block-uniform
  uint64_t sum;            // two partial sums
  float safe_s;            // masked sum and count over the steps from `first` on
  int safe_n;
  uint32_t cnt;            // counts not yet in safe_n
  int first;

  // the threshold is finite: rho = 0 keeps every finite logit, and the fill of a missing granule never passes
  __device__ __forceinline__ void set_guess(float m, double log_rho, int mode) {
    guess = m;
    c = log2_reference(m);
    const float t = fmaxf(threshold_of<TIn>(m, log_rho, mode), -FLT_MAX);
    tau = Ops::threshold(t);
    key = Ops::key(t);
    safe_s = 0.f;
    safe_n = 0;
    cnt = 0;
  }

  __device__ __forceinline__ void flush_count() {
    safe_n += Ops::count(cnt);
    cnt = 0;
  }

  __device__ __forceinline__ void absorb(const Stage<TIn, 2> &st, uint32_t *bound) {
    const uint32_t word = Ops::bounds(st, mx);
    *bound = word;
    constexpr int kElems = Granule<TIn>::kElems;
    const uint64_t l2 = pack2(kLog2e, kLog2e), c2 = pack2(-c, -c);
    // The step's terms are added up by themselves first: the thread that has met the maximum carries a sum of one or
    // more, where every addition costs half a unit of 2^-23, whatever it adds.  (Term by term: ln Z of 700 rows of
    // 151,936 bfloat16 1.8e-6 off at worst, 8e-7 this way; V = 151,936, forward, T = 8192: 930 / 931 us.)
    uint64_t part = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      float x[kElems], e[kElems];
      st.g[u].get(x);
#pragma unroll
      for (int j = 0; j < kElems; j += 2) {
        unpack2(fma2(pack2(x[j], x[j + 1]), l2, c2), e[j], e[j + 1]);
        e[j] = ex2(e[j]);
        e[j + 1] = ex2(e[j + 1]);
        part = u + j == 0 ? pack2(e[j], e[j + 1]) : add2(part, pack2(e[j], e[j + 1]));
        // 2-byte logits: skipping the masked part where no lane of the warp has a safe token in the granule costs as
        // much as it saves (T = 8192 x V = 151,936: 996 against 986 us forward at 1e-4, 921 / 927 at 1e-3)
        if constexpr (sizeof(TIn) == 2)
          Ops::masked(st.g[u], j / 2, x[j], x[j + 1], e[j], e[j + 1], tau, safe_s, cnt);
      }
      if constexpr (sizeof(TIn) == 4) {  // float32, half as many to a granule: 1885 against 1928 (T = 4096 x V = 262,144)
        if (__any_sync(0xffffffffu, (Ops::reach(word, key) >> (16 * u)) & 1u)) {
#pragma unroll
          for (int j = 0; j < kElems; j += 2)
            Ops::masked(st.g[u], j / 2, x[j], x[j + 1], e[j], e[j + 1], tau, safe_s, cnt);
        }
      }
    }
    sum = add2(sum, part);
  }
};

// ---- thread-block clusters ------------------------------------------------------
// With few tokens a row is split over the blocks of a cluster: block `part` owns a contiguous part of it,
// partial results meet through distributed shared memory.

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The aligned forms want a whole warp at the same instruction, which a branch before them (one thread writing a slot) does
// not leave behind by itself: both bring the warp together first.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void *local, uint32_t rank) {
  uint32_t laddr = (uint32_t)__cvta_generic_to_shared(local), raddr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(raddr) : "r"(laddr), "r"(rank));
  return raddr;
}
__device__ __forceinline__ float ld_cluster_f32(const float *local, uint32_t rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr(local, rank)) : "memory");
  return v;
}
struct RowGroup {
  int parts, part;
  float *slots;  // 6 floats of shared memory, each written once per kernel

  // rank in the cluster of the row's first block: 0, or behind a token's other row
  __device__ __forceinline__ uint32_t first() const { return cluster_rank() & (uint32_t)parts; }

  __device__ __forceinline__ float max(float m) const {
    if (parts == 1) return m;
    if (threadIdx.x == 0) slots[0] = m;
    cluster_arrive();
    cluster_wait();
    float hi = kNegInf;
    const uint32_t r0 = first();
    for (int k = 0; k < parts; ++k) hi = fmaxf(hi, ld_cluster_f32(slots + 0, r0 + k));
    return hi;
  }
  __device__ __forceinline__ void sums(float &all, SumCount &safe) const {
    if (parts == 1) return;
    if (threadIdx.x == 0) {
      slots[1] = all;
      slots[2] = safe.s;
      slots[3] = __int_as_float(safe.n);
    }
    cluster_arrive();
    cluster_wait();
    all = 0.f;
    safe = {0.f, 0};
    const uint32_t r0 = first();
    for (int k = 0; k < parts; ++k) {  // in order: same result in every block
      all += ld_cluster_f32(slots + 1, r0 + k);
      safe.s += ld_cluster_f32(slots + 2, r0 + k);
      safe.n += __float_as_int(ld_cluster_f32(slots + 3, r0 + k));
    }
  }
};

// A row as the sweeps see it.  Granules are cut at the row's own 32-byte boundaries, so that a row may
// start at any element (an odd vocabulary with its rows back to back): `head` elements lie in front of
// the first boundary and, as those behind the last whole granule, are taken one per thread outside the
// sweeps (at most 2 * kElems - 2 of them, fewer than a block has threads).
// Measured against element-wise loads for such rows: float16, T = 1111 x V = 50,021, with the gradient,
// 96 against 338 us; rows on 32-byte boundaries keep their time.
template <typename TIn>
struct RowView {
  const TIn *row;   // element 0
  const TIn *base;  // first element of this block's granules, 32-byte aligned
  int V;
  int head;      // elements in front of the row's first 32-byte boundary
  int n_all;     // whole granules of the row
  int g_first;   // first granule of this block (a cluster's blocks share the granules)
  int n_full;    // whole granules of this block
  bool extras;   // this block takes the elements outside the granules

  __device__ __forceinline__ void set(const TIn *r, int V_, int rank, int log_ranks) {
    constexpr int kElems = Granule<TIn>::kElems;
    row = r;
    V = V_;
    const int mis = (int)(((uintptr_t)r & 31u) / sizeof(TIn));
    head = min(V, mis ? kElems - mis : 0);
    n_all = (V - head) / kElems;
    const int per = (n_all + (1 << log_ranks) - 1) >> log_ranks;
    g_first = min(rank * per, n_all);
    n_full = min(per, n_all - g_first);
    base = r + head + (size_t)g_first * kElems;
    extras = rank == 0;
  }
  // element of the row that this thread takes outside the granules; none when it is >= V
  __device__ __forceinline__ int extra() const {
    const int tid = (int)threadIdx.x;
    return !extras ? V : tid < head ? tid : tid + n_all * Granule<TIn>::kElems;
  }
  // this block's granule that holds element a, -1 when there is none
  __device__ __forceinline__ int granule_of(int a) const {
    const int r = a < 0 ? -1 : rel(a);
    return r >= 0 && r < n_full * Granule<TIn>::kElems ? r / Granule<TIn>::kElems : -1;
  }
  // the same element when sums without the sampled token a are formed: the other elements of its granule
  // g_a count among those outside the granules (threads 32 to 32 + kElems - 1), the token itself is nobody's
  __device__ __forceinline__ int extra_but(int a, int g_a) const {
    const int j = (int)threadIdx.x - 32;
    int k = j < 0 ? extra() : V;
    if (g_a >= 0 && j >= 0 && j < Granule<TIn>::kElems)
      k = head + (g_first + g_a) * Granule<TIn>::kElems + j;
    return k == a ? V : k;
  }
  // element k of the row counted from `base`
  __device__ __forceinline__ int rel(int k) const { return k - head - g_first * Granule<TIn>::kElems; }
};

// A float as an integer of the same order, and back.
__device__ __forceinline__ int order_key(float v) {
  const int b = __float_as_int(v);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_value(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

// Block reductions of the row kernel: two alternating sets of words for maxima (one barrier each), one for
// sums (a maximum's barrier lies between two of them).  Fixed order; every thread gets the result.
constexpr int kMaxWarps = 16, kRedWords = 5 * kMaxWarps;
template <int kBlk>
struct BlockReduce {
  static constexpr int kWarps = kBlk / 32;
  float *words;
  int parity;

  __device__ __forceinline__ float max(float v) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int *slot = reinterpret_cast<int *>(words) + parity * kMaxWarps;
    parity ^= 1;
    const int k = __reduce_max_sync(0xffffffffu, order_key(v));
    if (lane == 0) slot[warp] = k;
    __syncthreads();
    return key_value(__reduce_max_sync(0xffffffffu, slot[lane % kWarps]));
  }
  __device__ __forceinline__ void sums(float &all, SumCount &safe) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *w = words + 2 * kMaxWarps;
    uint64_t v = pack2(all, safe.s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = add2(v, __shfl_xor_sync(0xffffffffu, v, o));
    safe.n = __reduce_add_sync(0xffffffffu, safe.n);
    if (lane == 0) {
      unpack2(v, all, safe.s);
      w[warp] = all;
      w[kMaxWarps + warp] = safe.s;
      w[2 * kMaxWarps + warp] = __int_as_float(safe.n);
    }
    __syncthreads();
    v = pack2(w[lane % kWarps], w[kMaxWarps + lane % kWarps]);
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) v = add2(v, __shfl_xor_sync(0xffffffffu, v, o));
    unpack2(v, all, safe.s);
    safe.n = __reduce_add_sync(0xffffffffu, lane < kWarps ? __float_as_int(w[2 * kMaxWarps + lane]) : 0);
  }
};

// Each thread first gathers the flags of its own granules into a register (16 steps at a time: one packed
// compare per step), then a warp prefix sum hands out list positions: the order of the list is fixed.
template <typename TIn, int kBlk>
__device__ __forceinline__ HotList build_hot_list(const uint32_t *bound, int n_steps,
                                                  typename SweepOps<TIn>::Key key, uint16_t *hot_smem) {
  const int lane = threadIdx.x & 31, tid = threadIdx.x;
  HotList h;
  h.slots = hot_smem + (tid >> 5) * kHotCap;
  h.count = 0;
  __syncwarp();  // the warp's list of an earlier row may still be read
  for (int step0 = 0; step0 < n_steps; step0 += 16) {
    uint32_t acc = 0;  // bit s: first granule of step step0 + s, bit 16 + s: second granule
    const int n = min(16, n_steps - step0);
    for (int s = 0; s < n; ++s) {
      const int wi = (step0 + s) * kBlk + tid;
      const uint32_t w = DVP_IN(wi, n_bound, DVP_OOB_BOUND) ? bound[wi] : 0u;
      acc |= (SweepOps<TIn>::reach(w, key) & 0x00010001u) << s;
    }
    const int cnt = __popc(acc);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    int pos = h.count + incl - cnt;
    while (acc) {
      const int b = __ffs(acc) - 1;
      acc &= acc - 1;
      const int slot = (step0 + (b & 15)) * 2 + (b >> 4);
      if (pos < kHotCap) h.slots[pos] = (uint16_t)(slot * 32 + lane);
      ++pos;
    }
    h.count += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  return h;
}

// Sweep 1 over (a part of) a row.
//
// The first guess of the maximum is the largest of `cand` (a value of the row: the sampled token's, which is
// the maximum in most rows) and of what the first two steps loaded (of the first one alone: T = 8192 x
// V = 151,936 bfloat16 forward 892 against 864 us).  The block's threads exchange their maxima
// every kSyncSteps steps: a larger one becomes the guess, and the masked sum starts again from there
// (`first`).  A value more than kWide above the guess may have overflowed the sum of the steps since the last exchange,
// and what came before is nothing against it (V e^-60): the sweep goes back to that exchange and starts its sums there.
// (Back to the start of the row, heavy-tailed rows without a sampled token took 259 us where they take 210: 2,500 x
// 100,000 bfloat16, both policies.)  All of it happens at fixed places, so that reruns are bit-identical.  `start`: the
// exchange to begin at; `hole`: the granule that reads as -inf (the sampled token's; its bound says that it can hold
// anything); xe: a value outside the granules.
constexpr int kSyncSteps = 4;
constexpr float kWide = 60.f;  // e^60 times the longest row is far from overflow
template <typename TIn, int kBlk>
__device__ __forceinline__ void row_sweep1(const RowView<TIn> &v, int start, int hole, float xe, float cand,
                                           double log_rho, int mode, uint32_t *bound, BlockReduce<kBlk> &red, Sweep1<TIn> &sw) {
  const TIn *row = v.base;
  const int n_full = v.n_full, tid = (int)threadIdx.x;
  const int per_step = 2 * kBlk;
  const int n_steps = (n_full + per_step - 1) / per_step;
  sw.mx = SweepOps<TIn>::start(xe);
  sw.sum = 0;  // two zeros
  sw.first = start;
  sw.set_guess(cand, log_rho, mode);
  const int hole_step = hole >= 0 ? hole / per_step : -1;
  Stage<TIn, 2> s0, s1;
  s0.template load_block<kBlk>(row, n_full, start);
  for (int step = start; step < n_steps; step += 2) {  // two stages in flight
    const bool second = step + 1 < n_steps;
    if (second) s1.template load_block<kBlk>(row, n_full, step + 1);
    if (step == hole_step) s0.template punch<kBlk>(step, hole);
    if (step % kSyncSteps == 0) {
      if (step == 0) {
        (void)SweepOps<TIn>::bounds(s0, sw.mx);
        if (second) (void)SweepOps<TIn>::bounds(s1, sw.mx);
      }
      const float m = red.max(SweepOps<TIn>::value(sw.mx));
      if (m > sw.guess) {
        const bool wide = m - sw.guess > kWide;
        const float f = ex2(sw.c - log2_reference(m));
        sw.sum = wide ? 0 : mul2(sw.sum, pack2(f, f));
        sw.set_guess(m, log_rho, mode);
        sw.first = step;
        if (wide && step > 0) {
          sw.first = step - kSyncSteps;
          s0.template load_block<kBlk>(row, n_full, sw.first);
          step = sw.first - 2;
          continue;
        }
      }
    }
    const int wi = step * kBlk + tid;
    if (DVP_IN(wi, n_bound, DVP_OOB_BOUND)) sw.absorb(s0, bound + wi);  // every thread stays for the exchanges
    if (step + 2 < n_steps) s0.template load_block<kBlk>(row, n_full, step + 2);
    if (second && DVP_IN(wi + kBlk, n_bound, DVP_OOB_BOUND)) {
      if (step + 1 == hole_step) s1.template punch<kBlk>(step + 1, hole);
      sw.absorb(s1, bound + wi + kBlk);
    }
    if ((step & 1023) == 1022) sw.flush_count();
  }
  sw.flush_count();
  if (hole >= 0 && hole % kBlk == tid) {
    const int wi = hole_step * kBlk + tid, sh = (hole / kBlk & 1) * 16;
    if (DVP_IN(wi, n_bound, DVP_OOB_BOUND))
      bound[wi] = (bound[wi] & (0xffff0000u >> sh)) | (SweepOps<TIn>::kTop << sh);
  }
}

// Sweep 2: masked sum and count over the granules of the steps below n_steps (`list` names granules of these
// steps and perhaps of later ones), without granule `hole`.
template <typename TIn, int kBlk>
__device__ __forceinline__ void row_sweep2(const RowView<TIn> &v, int hole, float tau, float m, int n_steps,
                                           typename SweepOps<TIn>::Key key, const uint32_t *bound, const HotList &list, SumCount &sc) {
  const TIn *row = v.base;
  const int n_full = v.n_full;
  const int n_slots = n_steps * 2;
  const int tid = threadIdx.x;
  if (list.fits()) {
    const int wbase = tid & ~31, lane = tid & 31;
    for (int q = lane; q < list.count; q += 64) {
      if (!DVP_IN(q, n_hot, DVP_OOB_HOT)) break;
      const uint32_t e0 = list.slots[q];
      const uint32_t e1 =
          q + 32 < list.count && DVP_IN(q + 32, n_hot, DVP_OOB_HOT) ? list.slots[q + 32] : 0xffffffffu;
      const int g0 = (int)(e0 >> 5) * kBlk + wbase + (int)(e0 & 31);
      const int g1 = (int)(e1 >> 5) * kBlk + wbase + (int)(e1 & 31);
      const bool one = (int)(e0 >> 5) < n_slots && g0 != hole, two = (e1 >> 5) < (uint32_t)n_slots && g1 != hole;
      Granule<TIn> a0, a1;
      if (one) a0.load_whole(row, n_full, g0);
      if (two) a1.load_whole(row, n_full, g1);
      if (one) granule_masked_sum<TIn>(a0, tau, m, sc);
      if (two) granule_masked_sum<TIn>(a1, tau, m, sc);
    }
  } else {
    // a dense safe set: all of the thread's granules, a step's two at a time (both loads before either is used)
    for (int step = 0; step < n_steps; ++step) {
      const int wi = step * kBlk + tid;
      if (!DVP_IN(wi, n_bound, DVP_OOB_BOUND)) break;
      const uint32_t b = SweepOps<TIn>::reach(bound[wi], key);
      const int g0 = 2 * step * kBlk + tid, g1 = g0 + kBlk;
      const bool hot0 = (b & 1u) && g0 != hole, hot1 = (b & 0x10000u) && g1 != hole;
      Granule<TIn> a0, a1;
      if (hot0) a0.load_whole(row, n_full, g0);
      if (hot1) a1.load_whole(row, n_full, g1);
      if (hot0) granule_masked_sum<TIn>(a0, tau, m, sc);
      if (hot1) granule_masked_sum<TIn>(a1, tau, m, sc);
    }
  }
}

// Statistics of one row (this block sweeps its part of it).  `listed`: the caller needs the hot list of the
// whole part.
template <typename TIn, int kBlk>
__device__ __forceinline__ SideStats row_stats(const RowView<TIn> &v, int a, double log_rho, int mode,
                                               float mask_value, bool listed, uint32_t *bound, BlockReduce<kBlk> &red,
                                               const RowGroup &grp, uint16_t *hot_smem, HotList &list) {
  const int n_steps = (v.n_full + 2 * kBlk - 1) / (2 * kBlk);
#ifdef DVP_DEBUG_BOUNDS
  {  // extents of this block's part of the row and of its tables
    __syncthreads();
    DVP_BOUNDS_SET(n_gran, v.n_full);
    DVP_BOUNDS_SET(V, (long long)v.n_full * Granule<TIn>::kElems);
    DVP_BOUNDS_SET(n_bound, (long long)n_steps * kBlk);
    DVP_BOUNDS_SET(n_hot, kHotCap);  // entries of one warp's hot list
    DVP_BOUNDS_SYNC();
  }
#endif
  const bool has_a = a >= 0 && a < v.V;
  const float z_0 = Storage<TIn>::widen(v.row[has_a ? a : 0]);
  const int hole = has_a ? v.granule_of(a) : -1;
  const int k_extra = v.extra_but(has_a ? a : -1, hole);
  const float xe = k_extra < v.V ? Storage<TIn>::widen(v.row[k_extra]) : kNegInf;
  Sweep1<TIn> sw;
  float cand = z_0, m;
  for (int start = 0;; start = (n_steps - 1) / kSyncSteps * kSyncSteps) {
    row_sweep1<TIn, kBlk>(v, start, hole, xe, cand, log_rho, mode, bound, red, sw);
    m = fmaxf(red.max(SweepOps<TIn>::value(sw.mx)), sw.guess);
    if (!(m - sw.guess > kWide) || n_steps == 0) break;
    cand = m;  // the second time it is the maximum
  }
  m = grp.max(m);

  SideStats st;
  st.m = m;
  st.tau = threshold_of<TIn>(m, log_rho, mode);
  st.z_a = has_a ? z_0 : 0.f;
  st.member = has_a && st.z_a >= st.tau;
  st.e_a = st.member ? ex2((st.z_a - st.m) * kLog2e) : 0.f;

  const float c = log2_reference(m);
  float p0, p1;
  unpack2(sw.sum, p0, p1);
  float all = (p0 + p1) * ex2(sw.c - c) + ex2(fmaf(xe, kLog2e, -c));
  SumCount safe = {0.f, 0};
  const bool guessed = sw.guess == m;  // block-uniform
  // the sum's terms are 2^{z l - c}; those of the definition (and of sweep 2) 2^{(z - m) l}
  if (guessed) safe = {sw.safe_s * ex2(-fmaf(m, kLog2e, -c)), sw.safe_n};
  const int n_again = guessed ? sw.first : n_steps;  // steps whose masked sum is still missing
  const typename SweepOps<TIn>::Key key = SweepOps<TIn>::key(fmaxf(st.tau, -FLT_MAX));
  list.slots = hot_smem;
  list.count = 0;
  if (n_again > 0 || listed) list = build_hot_list<TIn, kBlk>(bound, listed ? n_steps : n_again, key, hot_smem);
  if (n_again > 0) row_sweep2<TIn, kBlk>(v, hole, fmaxf(st.tau, -FLT_MAX), m, n_again, key, bound, list, safe);
  if (xe >= st.tau && xe > kNegInf) {
    ++safe.n;
    safe.s += ex2((xe - m) * kLog2e);
  }
  red.sums(all, safe);
  grp.sums(all, safe);
  if (has_a) all += ex2(fmaf(st.z_a, kLog2e, -c));
  st.lse = 0.0;  // from sum_c and sum_s, by the thread that writes it
  st.sum_c = (double)c;
  st.sum_s = all;
  st.s_x = safe.s;
  st.n = safe.n + (st.member ? 1 : 0);
  set_mask_mass(st, v.V, mode, Storage<TIn>::widen(Storage<TIn>::narrow(mask_value)), has_a);
  return st;
}

// The optional packed membership mask of a row (a diagnostic output), shared by the `parts` blocks of the row.  Called at
// the end of the kernel, so that its code lies behind the sweeps'.  A warp takes 1,024 elements at a time, 32 of them to
// an instruction: their votes are one word, and the 32 words are stored together.  A word a thread, read element by
// element by the first block alone, was bound by its 32 dependent strides, the more so the fewer threads a row had: V =
// 151,936 bfloat16, T = 64, both policies' masks: 209 -> 39 us;  float32 1,000 x 8,192: 155 -> 47.
template <typename TIn>
__device__ __forceinline__ void write_mask_row(const TIn *row, int V, float tau, uint32_t *mask_row, int part, int parts) {
  const int lane = threadIdx.x & 31, warps = (int)(blockDim.x >> 5), n_words = (V + 31) / 32;
  for (int w0 = ((int)(threadIdx.x >> 5) * parts + part) * 32; w0 < n_words; w0 += warps * parts * 32) {
    uint32_t mine = 0;  // word w0 + lane
#pragma unroll 8
    for (int b = 0; b < 32; ++b) {
      const long long k = ((long long)w0 + b) * 32 + lane;
      const uint32_t word = __ballot_sync(0xffffffffu, k < V && Storage<TIn>::widen(row[k]) >= tau);
      if (b == lane) mine = word;
    }
    if (w0 + lane < n_words) mask_row[w0 + lane] = mine;
  }
}

// Gradient rows may be stored in granules when each of them starts, with its logits granule, on a
// boundary of the granule's store (32 bytes, or 16 for float32 logits with a 2-byte gradient): elements.
template <typename TIn, typename TGrad>
__host__ __device__ constexpr int grad_align() {
  return Granule<TIn>::kElems < 32 / (int)sizeof(TGrad) ? Granule<TIn>::kElems : 32 / (int)sizeof(TGrad);
}

// 2^{(z - m) l} as 2^{z l - c} 2^{c - m l}, the second factor in the coefficient: one instruction less, and one rounding
// more (float32 entries of 333 x 50,021 logits: relative error 5.9e-8 with it, 5.0e-8 without): the row kernel does so for
// entries of 16 bits, which show it as one in some thousands rounded the other way.  The stand-alone backward does not.
template <typename TIn, typename TGrad>
constexpr bool kFoldedGrad = sizeof(TIn) == 2 && sizeof(TGrad) == 2;

// The words of memory that a granule's gradient entries fill.
template <typename TIn, typename TGrad>
constexpr int kGradWords = Granule<TIn>::kElems * (int)sizeof(TGrad) / 4;

// Gradient entries coef 2^{(z - m) l} of a whole granule (m2: -m twice, coef2: coef twice), zeros below the threshold.
// kFold: coef 2^{z l - m2}, one instruction less for two of them (see kFoldedGrad).
template <typename TIn, typename TGrad, bool kFold>
__device__ __forceinline__ void grad_words(const Granule<TIn> &gr, float tau, typename SweepOps<TIn>::Tau tau_p,
                                           uint64_t m2, uint64_t coef2, uint32_t (&w)[kGradWords<TIn, TGrad>]) {
  constexpr int kElems = Granule<TIn>::kElems;
  constexpr bool by_bits = sizeof(TIn) == 2 && sizeof(TGrad) == 2;  // two entries' comparisons are one
  const uint64_t l2 = pack2(kLog2e, kLog2e);
  float x[kElems];
  gr.get(x);
#pragma unroll
  for (int j = 0; j < kElems; j += 2) {
    float lo, hi;
    unpack2(kFold ? fma2(pack2(x[j], x[j + 1]), l2, m2) : mul2(add2(pack2(x[j], x[j + 1]), m2), l2), lo, hi);
    unpack2(mul2(pack2(ex2(lo), ex2(hi)), coef2), lo, hi);
    if constexpr (!by_bits) {
      lo = x[j] >= tau ? lo : 0.f;
      hi = x[j + 1] >= tau ? hi : 0.f;
    }
    if constexpr (sizeof(TGrad) == 4) {
      w[j] = __float_as_uint(lo);
      w[j + 1] = __float_as_uint(hi);
    } else if constexpr (std::is_same<TGrad, __nv_bfloat16>::value) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
      w[j / 2] = *reinterpret_cast<const uint32_t *>(&h);
    } else {
      const __half2 h = __floats2half2_rn(lo, hi);
      w[j / 2] = *reinterpret_cast<const uint32_t *>(&h);
    }
    if constexpr (by_bits) w[j / 2] &= SweepOps<TIn>::reach(gr.w[j / 2], tau_p);
  }
}
template <typename TIn, typename TGrad, bool kFold>
__device__ __forceinline__ void grad_granule(const Granule<TIn> &gr, TGrad *dst, float tau,
                                             typename SweepOps<TIn>::Tau tau_p, uint64_t m2, uint64_t coef2) {
  constexpr int kWords = kGradWords<TIn, TGrad>;
  uint32_t w[kWords];
  grad_words<TIn, TGrad, kFold>(gr, tau, tau_p, m2, coef2, w);
  if constexpr (kWords == 4) {
    st_stream16(dst, make_uint4(w[0], w[1], w[2], w[3]));
  } else {
#pragma unroll
    for (int i = 0; i < kWords; i += 8) {
      uint32_t v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = w[i + k];
      st_stream32(reinterpret_cast<uint32_t *>(dst) + i, v);
    }
  }
}

// The same for a gradient row that lies differently than its logits row (another row stride or base): the entries of `n`
// neighbouring granules, one a lane from lane 0 on, to `dst`, where those of the first begin, at any alignment of theirs.
// They pass through 512 bytes of the warp's shared memory, so that 32 lanes store 32 neighbouring words, put together from
// the halves of two where 2-byte entries begin at an odd one.  `any`: some lane's granule has a safe token; a lane whose
// granule has none holds zeros.
constexpr int kShiftWords = 128;  // of shared memory, a warp
template <int kWords, typename TGrad>
__device__ __forceinline__ void store_shifted(const uint32_t (&w)[kWords], bool any, TGrad *dst, int n, uint32_t *smem) {
  constexpr int kLanes = 32 * kWords <= kShiftWords ? 32 : kShiftWords / kWords;  // whose entries fit at once
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = 0; h < 32 / kLanes; ++h) {
    const int n_words = min(kLanes, n - h * kLanes) * kWords;
    if (n_words <= 0) break;
    if (any) {
      __syncwarp();  // the words before are stored
      if (lane / kLanes == h) {
        uint32_t *mine = smem + (lane % kLanes) * kWords;
#pragma unroll
        for (int i = 0; i < kWords; i += 4)
          *reinterpret_cast<uint4 *>(mine + i) = make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]);
      }
      __syncwarp();
    }
    uint32_t *out = reinterpret_cast<uint32_t *>(dst) + h * kLanes * kWords;
    if (sizeof(TGrad) == 4 || ((uintptr_t)dst & 3u) == 0) {
#pragma unroll
      for (int k = lane; k < kLanes * kWords; k += 32)
        if (k < n_words) st_stream4(out + k, any ? smem[k] : 0u);
    } else {
      uint16_t *half = reinterpret_cast<uint16_t *>(out);
#pragma unroll
      for (int k = lane; k < kLanes * kWords; k += 32) {
        if (k + 1 < n_words) st_stream4(half + 2 * k + 1, any ? __byte_perm(smem[k], smem[k + 1], 0x5432) : 0u);
        if (k + 1 == n_words) half[2 * k + 1] = any ? (uint16_t)(smem[k] >> 16) : (uint16_t)0;
      }
      if (lane == 0) half[0] = any ? (uint16_t)smem[0] : (uint16_t)0;
    }
  }
}

// Sweep 3 when the gradient row lies differently than its logits row (another row stride or base): zeros first, in the
// gradient row's own 32-byte pieces, then the safe tokens one by one.  (store_shifted for every granule instead, us, 1,000 x
// 100,003 bfloat16 at rho = 1e-4 179 / 187, 5,000 x 20,000 float16 156 / 195; 2,000 x 50,021 at e^-13, where most granules
// have a safe token, 227 / 200; both forms in one kernel cost float16 rows 3 %.)
template <typename TIn, typename TGrad, int kBlk>
__device__ __forceinline__ void row_grad_loose(const RowView<TIn> &v, TGrad *grow, int a, float tau,
                                               typename SweepOps<TIn>::Key key, bool live, float m, float coef,
                                               float g_a, const uint32_t *bound) {
  constexpr int kElems = Granule<TIn>::kElems, kOut = 32 / (int)sizeof(TGrad);
  const int tid = threadIdx.x, n_thr = kBlk;
  const int k0 = v.head + v.g_first * kElems, k1 = k0 + v.n_full * kElems;  // this block's granules, as elements
  TGrad *dst = grow + k0;
  const int n = k1 - k0;
  const int mis = (int)(((uintptr_t)dst & 31u) / sizeof(TGrad));
  const int head = min(n, mis ? kOut - mis : 0), n_vec = (n - head) / kOut;
  const uint32_t z[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  if (tid < head) dst[tid] = Storage<TGrad>::narrow(0.f);
  for (int i = tid; i < n_vec; i += n_thr) st_stream32(dst + head + (size_t)i * kOut, z);
  const int k_rest = head + n_vec * kOut + tid;
  if (k_rest < n) dst[k_rest] = Storage<TGrad>::narrow(0.f);
  __syncthreads();  // the zeros of this block's part are in place before single elements replace them
  if (!live) return;
  for (int i = 0;; ++i) {
    const int g = i * n_thr + tid, wi = (i >> 1) * n_thr + tid;
    if (g >= v.n_full || !DVP_IN(wi, n_bound, DVP_OOB_BOUND)) break;
    if (!((SweepOps<TIn>::reach(bound[wi], key) >> (16 * (i & 1))) & 1u)) continue;
    Granule<TIn> gr;
    gr.load_whole(v.base, v.n_full, g);
    float x[kElems];
    gr.get(x);
    const int ja = a - g * kElems;
#pragma unroll
    for (int j = 0; j < kElems; ++j)
      if (x[j] >= tau)
        dst[(size_t)g * kElems + j] =
            Storage<TGrad>::narrow(j == ja ? g_a : coef * ex2((x[j] - m) * kLog2e));
  }
}

// Sweep 3: gradient of g * ln pi^mp(a) over the row.  Granules without a safe token are written as zeros
// without being read; the others are read again, the next pair while zeros are written and the last one
// is worked on: the reads are scattered and the sweep waits for them.
template <typename TIn, typename TGrad, int kBlk, bool kLoose>
__device__ __forceinline__ void row_grad(const RowView<TIn> &v, TGrad *grow_all, int a_row,
                                         const SideStats &st, float g, const uint32_t *bound,
                                         const HotList &list) {
  constexpr int kElems = Granule<TIn>::kElems;
  const TIn *row = v.base;
  const int n_full = v.n_full;
  TGrad *grow = grow_all + (v.base - v.row);
  const int n_steps = (n_full + 2 * kBlk - 1) / (2 * kBlk);
  const int tid = threadIdx.x;
  const float s_tot = st.s_x + st.e_a + st.s_mask;
  // a missing sampled token, or a pruned one under the -inf semantics, has weight zero:
  // the row is all zeros
  const bool live = st.live;
  const float coef = live ? -g / s_tot : 0.f;
  const float g_a = st.member ? g * ((st.s_x + st.s_mask) / s_tot) : 0.f;
  const int a_here = (live && st.member) ? a_row : -1;
  const bool listed = live && list.fits();
  const float tau = live ? fmaxf(st.tau, -FLT_MAX) : -kNegInf;  // +inf: nothing passes
  const typename SweepOps<TIn>::Key key = SweepOps<TIn>::key(fmaxf(st.tau, -FLT_MAX));

  {  // the elements outside the granules, one per thread
    const int k_extra = v.extra();
    if (k_extra < v.V) {
      const float x = Storage<TIn>::widen(v.row[k_extra]);
      float out = x >= tau ? coef * ex2((x - st.m) * kLog2e) : 0.f;
      if (k_extra == a_here) out = g_a;
      grow_all[k_extra] = Storage<TGrad>::narrow(out);
    }
  }
  // zeros of one step's granules that hold no safe token
  auto zeros = [&](int step) {
    const int wi = step * kBlk + tid;
    if (!DVP_IN(wi, n_bound, DVP_OOB_BOUND)) return;
    const uint32_t b = live ? SweepOps<TIn>::reach(bound[wi], key) : 0u;
    const int g0 = 2 * step * kBlk + tid, g1 = g0 + kBlk;
    if (!(b & 1u) && g0 < n_full && DVP_IN((long long)g0 * kElems + kElems - 1, V, DVP_OOB_GLOBAL))
      store_zero_granule<TGrad, kElems>(grow + (size_t)g0 * kElems);
    if (!(b & 0x10000u) && g1 < n_full && DVP_IN((long long)g1 * kElems + kElems - 1, V, DVP_OOB_GLOBAL))
      store_zero_granule<TGrad, kElems>(grow + (size_t)g1 * kElems);
  };
  float mc = st.m, cf = coef;
  if constexpr (kFoldedGrad<TIn, TGrad>) {
    mc = st.m * kLog2e;
    cf = coef * ex2(-fmaf(st.m, kLog2e, -mc));
  }
  const uint64_t m2 = pack2(-mc, -mc), cf2 = pack2(cf, cf);
  const typename SweepOps<TIn>::Tau tau_p = SweepOps<TIn>::threshold(fmaxf(st.tau, -FLT_MAX));
  const int g_here = a_here >= 0 ? v.granule_of(a_here) : -1;
  if constexpr (kLoose) {
    row_grad_loose<TIn, TGrad, kBlk>(v, grow_all, a_here >= 0 ? v.rel(a_here) : -1, tau, key, live, st.m, coef, g_a, bound);
    return;
  }
  // one granule; the sampled token's entry replaces the one that its granule's store left
  auto emit = [&](const Granule<TIn> &gr, int g) {
    if (!DVP_IN((long long)g * kElems + kElems - 1, V, DVP_OOB_GLOBAL)) return;
    grad_granule<TIn, TGrad, kFoldedGrad<TIn, TGrad>>(gr, grow + (size_t)g * kElems, tau, tau_p, m2, cf2);
    if (g == g_here) grow_all[a_here] = Storage<TGrad>::narrow(g_a);
  };
  int step = 0;
  if (listed) {
    const int wbase = tid & ~31, lane = tid & 31;
    // granule of list position q, -1 behind the end (with rho = 0 a list of float32 granules may name some
    // behind the end of the row)
    auto at = [&](int q) {
      if (q >= list.count || !DVP_IN(q, n_hot, DVP_OOB_HOT)) return -1;
      const uint32_t e = list.slots[q];
      const int g = (int)(e >> 5) * kBlk + wbase + (int)(e & 31);
      return g < n_full ? g : -1;
    };
    Granule<TIn> a0, a1, b0, b1;
    int ga0 = at(lane), ga1 = at(lane + 32);
    if (ga0 >= 0) a0.load_whole(row, n_full, ga0);
    if (ga1 >= 0) a1.load_whole(row, n_full, ga1);
    for (int q = lane; q < list.count; q += 128) {
      const int gb0 = at(q + 64), gb1 = at(q + 96);
      if (gb0 >= 0) b0.load_whole(row, n_full, gb0);
      if (gb1 >= 0) b1.load_whole(row, n_full, gb1);
      if (step < n_steps) zeros(step++);
      if (ga0 >= 0) emit(a0, ga0);
      if (ga1 >= 0) emit(a1, ga1);
      ga0 = at(q + 128);
      ga1 = at(q + 160);
      if (ga0 >= 0) a0.load_whole(row, n_full, ga0);
      if (ga1 >= 0) a1.load_whole(row, n_full, ga1);
      if (step < n_steps) zeros(step++);
      if (gb0 >= 0) emit(b0, gb0);
      if (gb1 >= 0) emit(b1, gb1);
    }
  }
  for (; step < n_steps; ++step) zeros(step);
  if (live && !listed) {
    // a dense safe set: all of the thread's hot granules, a step's two at a time (both loads before either is used)
    for (step = 0; step < n_steps; ++step) {
      const int wi = step * kBlk + tid;
      if (!DVP_IN(wi, n_bound, DVP_OOB_BOUND)) break;
      const uint32_t h = SweepOps<TIn>::reach(bound[wi], key);
      const int g0 = 2 * step * kBlk + tid, g1 = g0 + kBlk;
      const bool hot0 = (h & 1u) && g0 < n_full, hot1 = (h & 0x10000u) && g1 < n_full;
      Granule<TIn> a0, a1;
      if (hot0) a0.load_whole(row, n_full, g0);
      if (hot1) a1.load_whole(row, n_full, g1);
      if (hot0) emit(a0, g0);
      if (hot1) emit(a1, g1);
    }
  }
}

// Shared-memory layout of the row kernel, in 4-byte words: the block reductions, 8 for what blocks of a
// cluster exchange, then the hot lists, then the bounds.
__host__ __device__ inline int smem_words_fixed(int threads) {
  return kRedWords + 8 + (threads / 32) * kHotCap / 2;
}

// The gradient of a launch: none; stored in granules; or with rows that lie differently than the logits'.
enum class Grad { kNone, kGranules, kLoose };

// One row per block, or per cluster of 2^log_parts blocks.  kBlk: threads of a block, 1024 of them on an SM;
// a compile-time constant, because it makes the sweeps' indices immediate operands.
//
// A batch that fills the chip is swept by two launches, one a policy: two copies of the sweeps in one kernel stall on
// instruction fetches, a loop over the two rows spills 460 bytes a thread (rows 12 to 17 % slower), and pairs of blocks in
// a cluster wait for two free places at once (18 % slower with two blocks per SM).  The second launch may begin while the
// last rows of the first are still swept (launch_rows_both says which is first and how the two meet).
//
// Small calls are one launch, a token's two rows in one cluster (kTogether): ln pi^mp_infer(a) and the membership pass
// through shared memory.  Smaller ones, whose rows the chip's registers hold, do not come here (dvp_rows_held.cuh).
//
// kBehind: the inference rows where the training rows come first.  Kernels of their own, because what they do at a row's
// end costs short rows in the kernel that sweeps rows without a gradient in every other order.  us, forward, with it there /
// here: 73,242 x 2,048 bfloat16 356.3 / 352.6, 60,000 x 2,500 float16 355.7 / 352.2, 30,000 x 2,048 float32 165.0 / 163.2.
template <typename TIn, typename TGrad, int kBlk, Grad kGrad, bool kTogether, bool kBehind>
__global__ void __launch_bounds__(kBlk, 1024 / kBlk)
dvp_row_kernel(const __grid_constant__ RowParams p, const long long t0, const int log_parts) {
  extern __shared__ __align__(16) float smem[];
  BlockReduce<kBlk> red{smem, 0};
  uint16_t *hot_smem = reinterpret_cast<uint16_t *>(smem + kRedWords + 8);  // kHotCap per warp
  uint32_t *bound = reinterpret_cast<uint32_t *>(smem + smem_words_fixed(kBlk));

  DVP_BOUNDS_BEGIN(p.bounds_status);
  if (p.order == kOrderFirst) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int both = kTogether;
  const int parts = 1 << log_parts;
  // with both rows of a token in a cluster, the second half of its blocks has the inference row
  auto other_half = [&] { return both && (int)cluster_rank() >= parts; };
  static_assert(!kBehind || (kGrad == Grad::kNone && !kTogether), "the inference rows, in a launch of their own");
  float *slots = smem + kRedWords;
  const RowGroup grp{parts, parts > 1 ? (int)cluster_rank() & (parts - 1) : 0, slots};
  const long long t = t0 + (blockIdx.x >> (log_parts + both));
  const long long id = p.ids ? load_id(p.ids, p.id_is_i32, t) : -1;
  const bool has_id = id >= 0, bad_id = id >= p.V;
  const int a = (has_id && !bad_id) ? (int)id : -1;
  const bool writer = threadIdx.x == 0 && grp.part == 0;
  RowView<TIn> v;
  v.set(other_half() ? reinterpret_cast<const TIn *>(p.infer) + t * p.ld_infer
                      : reinterpret_cast<const TIn *>(p.train) + t * p.ld_train,
        (int)p.V, grp.part, log_parts);
  HotList list;
  SideStats st = row_stats<TIn, kBlk>(v, a, p.log_rho, p.mode, p.mask_value, kGrad == Grad::kGranules && !other_half(),
                                      bound, red, grp, hot_smem, list);
  const bool weighted = p.weight_kind != DVP_WEIGHT_NONE;
  float li = 0.f;
  if (both) {  // ln pi^mp_infer(a) and the membership; and the inference row has been read
    if (other_half() && writer) {
      slots[4] = logp_mp_of(st);
      slots[5] = st.member ? 1.f : 0.f;
    }
    __syncthreads();
    cluster_arrive();
    cluster_wait();
    if (!other_half()) {
      li = ld_cluster_f32(slots + 4, (uint32_t)parts);
      if (writer) {
        slots[4] = li;
        slots[5] = ld_cluster_f32(slots + 5, (uint32_t)parts);
      }
    }
  }
  if (parts > 1 || both) cluster_arrive();  // this block has read the others' slots
  if constexpr (kGrad != Grad::kNone) {
    if (!other_half()) {
      float g = p.upstream[t];
      if (weighted) {
        if (!both) {
          asm volatile("griddepcontrol.wait;" ::: "memory");
          li = load_li(p, t);
        }
        const float w = a < 0 ? __int_as_float(0x7fc00000)
                              : token_weight(log_ratio_from(p.mode, st.member, logp_mp_of(st), li), p.weight_kind,
                                             p.weight_lo, p.weight_hi);
        if (w == w) g *= w;
        if (!both) {
          if (parts > 1) {  // every block of the row has li before the place that holds it is overwritten
            cluster_wait();
            cluster_arrive();
            cluster_wait();
          } else {
            __syncthreads();
          }
        }
        if (p.weight_out && writer) p.weight_out[t] = w;
      }
      row_grad<TIn, TGrad, kBlk, kGrad == Grad::kLoose>(v, reinterpret_cast<TGrad *>(p.grad) + t * p.ld_grad, a, st, g,
                                                        bound, list);
    }
  }
  const bool second_half = other_half();
  const dvp_side_out &out = second_half ? p.out_i : p.out_t;
  if (writer) {
    if (p.order == kOrderSecond && !weighted) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      li = load_li(p, t);
    }
    if (both) li = slots[4];
    st.lse = lse_from_logsum({st.m, (float)st.sum_c, st.sum_s});
    const float own = finish_side(out, t, st, has_id, bad_id);
    if (p.order == kOrderFirst) store_li(p, t, own);
    uint8_t before = 0;  // the other policy's membership
    if (p.flags && !second_half) {
      constexpr uint8_t theirs = kBehind ? DVP_FLAG_IN_TRAIN : DVP_FLAG_IN_INFER;
      before = p.order == kOrderSecond ? p.flags[t] & theirs : both && slots[5] != 0.f ? theirs : 0;
      // the rows of a launch with a gradient are the training rows
      const uint8_t member = kGrad == Grad::kNone && p.side == kSideInfer ? DVP_FLAG_IN_INFER : DVP_FLAG_IN_TRAIN;
      p.flags[t] = (uint8_t)((st.member ? member : 0) | before | (has_id ? 0 : DVP_FLAG_NO_ID) |
                             (bad_id ? DVP_FLAG_BAD_ID : 0));
    }
    if (p.log_ratio && !second_half) {
      float ratio;
      if constexpr (kBehind)  // li is ln pi^mp_train(a)
        ratio = log_ratio_from(p.mode, in_train_by(p.flags, before, li), li, own);
      else
        ratio = log_ratio_from(p.mode, st.member, own, li);
      p.log_ratio[t] = kBehind && p.order == kOrderApart ? (st.member ? 1.f : 0.f)
                       : a < 0                           ? __int_as_float(0x7fc00000)
                                                         : ratio;
    }
    // whoever waits for this launch waits for the one before too
    if (kBehind && p.order == kOrderApart && (blockIdx.x | (parts - 1)) == gridDim.x - 1)
      asm volatile("griddepcontrol.wait;" ::: "memory");
  }
  if (out.mask)
    write_mask_row<TIn>(v.row, v.V, st.tau, out.mask + t * ((p.V + 31) / 32), grp.part, parts);
  // no block may leave while another one can still read its exchange slots
  if (both || (parts > 1 && !(kGrad != Grad::kNone && weighted)))
    cluster_wait();
}

// ---- scalar kernel: any row length --------------------------------------------
// Three plain sweeps per matrix with element-wise loads; used when a row is too long
// for the granule bounds.

template <typename TIn>
__device__ __forceinline__ SideStats row_stats_scalar(const TIn *row, long long V, long long a,
                                                      double log_rho, int mode, float mask_value,
                                                      float *scratch, uint32_t *mask_row) {
  float m = kNegInf;
  for (long long k = threadIdx.x; k < V; k += blockDim.x) m = fmaxf(m, Storage<TIn>::widen(row[k]));
  MaxSum acc = {m, 0.f};
  if (m > kNegInf)
    for (long long k = threadIdx.x; k < V; k += blockDim.x)
      acc.s += ex2((Storage<TIn>::widen(row[k]) - m) * kLog2e);
  const MaxSum all = block_reduce_maxsum(acc, scratch);
  SideStats st;
  st.m = all.m;
  st.lse = (double)all.m + (double)logf(all.s);
  st.sum_c = (double)all.m * (double)kLog2e;
  st.sum_s = all.s;
  st.tau = threshold_of<TIn>(all.m, log_rho, mode);
  const bool has_a = a >= 0 && a < V;
  st.z_a = has_a ? Storage<TIn>::widen(row[a]) : 0.f;
  st.member = has_a && st.z_a >= st.tau;
  st.e_a = st.member ? ex2((st.z_a - st.m) * kLog2e) : 0.f;
  SumCount sc = {0.f, 0};
  for (long long k = threadIdx.x; k < V; k += blockDim.x) {
    const float z = Storage<TIn>::widen(row[k]);
    if (z >= st.tau) {
      ++sc.n;
      if (k != a) sc.s += ex2((z - st.m) * kLog2e);
    }
  }
  const SumCount tot = block_reduce_sumcount(sc, scratch);
  st.s_x = tot.s;
  st.n = tot.n;
  set_mask_mass(st, V, mode, Storage<TIn>::widen(Storage<TIn>::narrow(mask_value)), has_a);
  if (mask_row) {
    const long long n_words = (V + 31) / 32;
    for (long long w = threadIdx.x; w < n_words; w += blockDim.x) {
      uint32_t bits = 0;
      for (int b = 0; b < 32; ++b) {
        const long long k = w * 32 + b;
        if (k < V && Storage<TIn>::widen(row[k]) >= st.tau) bits |= 1u << b;
      }
      mask_row[w] = bits;
    }
  }
  return st;
}

template <typename TIn, typename TGrad>
__global__ void dvp_row_kernel_scalar(const RowParams p) {
  __shared__ float scratch[64];
  const long long t = blockIdx.x;
  const long long id = p.ids ? load_id(p.ids, p.id_is_i32, t) : -1;
  const bool has_id = id >= 0, bad_id = id >= p.V;
  const long long a = (has_id && !bad_id) ? id : -1;

  const TIn *trow = reinterpret_cast<const TIn *>(p.train) + t * p.ld_train;
  const TIn *irow = p.infer ? reinterpret_cast<const TIn *>(p.infer) + t * p.ld_infer : nullptr;
  uint32_t *mask_t = p.out_t.mask ? p.out_t.mask + t * ((p.V + 31) / 32) : nullptr;
  uint32_t *mask_i = p.out_i.mask ? p.out_i.mask + t * ((p.V + 31) / 32) : nullptr;
  const SideStats st =
      row_stats_scalar<TIn>(trow, p.V, a, p.log_rho, p.mode, p.mask_value, scratch, mask_t);
  SideStats si;
  if (irow) si = row_stats_scalar<TIn>(irow, p.V, a, p.log_rho, p.mode, p.mask_value, scratch, mask_i);
  float w = 1.f;
  if (p.weight_kind != DVP_WEIGHT_NONE)
    w = row_weight(p, st, si, a >= 0);  // weights need inference rows
  if (p.weight_out && threadIdx.x == 0) p.weight_out[t] = w;

  if (p.grad) {
    TGrad *grow = reinterpret_cast<TGrad *>(p.grad) + t * p.ld_grad;
    float g = p.upstream[t];
    if (w == w) g *= w;
    const float s_tot = st.s_x + st.e_a + st.s_mask;
    const bool live = st.live;
    const float coef = live ? -g / s_tot : 0.f;
    const float g_a = st.member ? g * ((st.s_x + st.s_mask) / s_tot) : 0.f;
    for (long long k = threadIdx.x; k < p.V; k += blockDim.x) {
      const float z = Storage<TIn>::widen(trow[k]);
      float out = (live && z >= st.tau) ? coef * ex2((z - st.m) * kLog2e) : 0.f;
      if (live && st.member && k == a) out = g_a;
      grow[k] = Storage<TGrad>::narrow(out);
    }
  }

  if (threadIdx.x == 0) {
    const float lt = finish_side(p.out_t, t, st, has_id, bad_id);
    uint8_t flags = (uint8_t)((st.member ? DVP_FLAG_IN_TRAIN : 0) | (has_id ? 0 : DVP_FLAG_NO_ID) |
                              (bad_id ? DVP_FLAG_BAD_ID : 0));
    if (p.infer) {
      const float li = finish_side(p.out_i, t, si, has_id, bad_id);
      if (si.member) flags |= DVP_FLAG_IN_INFER;
      if (p.log_ratio)
        p.log_ratio[t] = !(has_id && !bad_id)              ? __int_as_float(0x7fc00000)
                         : (p.mode & DVP_MODE_FINITE_MASK) ? lt - li
                                                           : log_ratio_of(st.member, si.member, lt, li);
    }
    if (p.flags) p.flags[t] = flags;
  }
}

// ---- stand-alone backward: a streaming map from saved row statistics ---------

// A row is shared by 2^log_parts blocks; nothing passes between them.  Granules are cut as in the row kernel (RowView),
// so that rows may start at any element; kLoose: gradient rows that lie differently (store_shifted).  A step is two
// granules a thread, both loads in flight, the first step's before the row's scalars are read.  Granules of a warp
// without a safe token are written as zeros without an exponential.
template <typename TIn, typename TGrad, bool kLoose>
__global__ void __launch_bounds__(512, 2) dvp_backward_kernel(const __grid_constant__ BackwardParams p, const int log_parts) {
  constexpr int kElems = Granule<TIn>::kElems, kWords = kGradWords<TIn, TGrad>;
  extern __shared__ __align__(16) uint32_t shift_smem[];  // kLoose: kShiftWords a warp
  const long long t = blockIdx.x >> log_parts;
  const int tid = (int)threadIdx.x, n_thr = (int)blockDim.x, lane = tid & 31;
  const TIn *row = reinterpret_cast<const TIn *>(p.train) + t * p.ld_train;
  TGrad *grow = reinterpret_cast<TGrad *>(p.grad) + t * p.ld_grad;
  RowView<TIn> v;
  v.set(row, (int)p.V, (int)blockIdx.x & ((1 << log_parts) - 1), log_parts);
  DVP_BOUNDS_BEGIN(p.bounds_status);
  DVP_BOUNDS_SET(n_gran, v.n_full);
  DVP_BOUNDS_SET(V, (long long)v.n_full * kElems);
  DVP_BOUNDS_SYNC();
  const int n_full = v.n_full;
  Granule<TIn> gr[2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (tid + u * n_thr < n_full) gr[u].load_whole(v.base, n_full, tid + u * n_thr);

  const long long id = load_id(p.ids, p.id_is_i32, t);
  const bool valid = id >= 0 && id < p.V;
  const bool member = (p.flags[t] & DVP_FLAG_IN_TRAIN) && valid;
  // with a finite mask value a pruned sampled token still has a gradient on the kept positions
  const bool live = member || ((p.mode & DVP_MODE_FINITE_MASK) && valid);
  const int a = member ? (int)id : -1;
  const float g = p.upstream[t], m = p.max_t[t];
  const float tau = fmaxf(threshold_of<TIn>(m, p.log_rho, p.mode), -FLT_MAX);
  // e^{z - lse_safe} = e^{z - m} e^{m - lse_safe}; the second factor is 1 / s_safe
  const float coef = live ? -g * ex2((m - p.lse_safe_t[t]) * kLog2e) : 0.f;
  float out_a = 0.f;
  if (member) {
    const float comp = p.comp_mp_t ? p.comp_mp_t[t] : -expm1f(Storage<TIn>::widen(row[a]) - p.lse_safe_t[t]);
    out_a = g * comp;
  }
  const int k_extra = tid < 32 ? v.extra() : v.V;  // V may be close to INT_MAX here
  if (k_extra < v.V) {
    const float x = Storage<TIn>::widen(row[k_extra]);
    const float out = live && x >= tau ? coef * ex2((x - m) * kLog2e) : 0.f;
    grow[k_extra] = Storage<TGrad>::narrow(k_extra == a ? out_a : out);
  }
  const uint64_t m2 = pack2(-m, -m), cf2 = pack2(coef, coef);
  const typename SweepOps<TIn>::Tau tau_p = SweepOps<TIn>::threshold(tau);
  const int g_a = a >= 0 ? v.granule_of(a) : -1;
  TGrad *gbase = grow + (v.base - row);
  // whole warps stay: a lane past the end has nothing to store
  for (int g0 = tid; g0 - lane < n_full; g0 += 2 * n_thr) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int gi = g0 + u * n_thr, n = min(32, n_full - (gi - lane));
      if (n <= 0 || !DVP_IN((long long)(gi - lane + n) * kElems - 1, V, DVP_OOB_GLOBAL)) break;
      const bool hot = live && lane < n && gr[u].max() >= tau, any = __any_sync(0xffffffffu, hot);
      TGrad *dst = gbase + (size_t)gi * kElems;
      if constexpr (kLoose) {
        uint32_t w[kWords];
#pragma unroll
        for (int i = 0; i < kWords; ++i) w[i] = 0;
        if (hot) grad_words<TIn, TGrad, false>(gr[u], tau, tau_p, m2, cf2, w);
        store_shifted(w, any, dst - lane * kElems, n, shift_smem + (tid >> 5) * kShiftWords);
        __syncwarp();  // the sampled token's entry replaces what a lane of the warp stored there
      } else if (lane < n) {
        if (any)
          grad_granule<TIn, TGrad, false>(gr[u], dst, tau, tau_p, m2, cf2);
        else
          store_zero_granule<TGrad, kElems>(dst);
      }
      if (gi == g_a) grow[a] = Storage<TGrad>::narrow(out_a);
      if (gi + 2 * n_thr < n_full) gr[u].load_whole(v.base, n_full, gi + 2 * n_thr);
    }
  }
}


}  // namespace dvp
#include "dvp_rows_held.cuh"
#include "dvp_rows_resident.cuh"
#include "dvp_rows_store.cuh"
namespace dvp {

// ---- host-side launchers, instantiated once per logits type -------------------

static inline bool aligned32(const void *base, long long ld, size_t elem) {
  return base == nullptr || (((uintptr_t)base % 32 == 0) && ((ld * (long long)elem) % 32 == 0));
}

// Do the gradient's granules start on store boundaries wherever the logits' do?
template <typename TIn, typename TGrad>
static inline bool grad_loose(const void *logits, long long ld, const void *grad, long long ld_grad, long long T) {
  constexpr long long kA = grad_align<TIn, TGrad>();
  const long long shift = (long long)((uintptr_t)grad / sizeof(TGrad) % kA) - (long long)((uintptr_t)logits / sizeof(TIn) % kA);
  return shift % kA != 0 || (T > 1 && (ld_grad - ld) % kA != 0);
}

// Does the gradient take the place of (a part of) these logits?
template <typename TIn, typename TGrad>
static inline bool grad_over(const RowParams &p, const void *logits, long long ld) {
  if (!p.grad || !logits) return false;
  const uintptr_t g = (uintptr_t)p.grad, z = (uintptr_t)logits;
  return g < z + (size_t)((p.T - 1) * ld + p.V) * sizeof(TIn) &&
         z < g + (size_t)((p.T - 1) * p.ld_grad + p.V) * sizeof(TGrad);
}

template <typename TIn, typename TGrad, int kBlk, Grad kGrad, bool kTogether, bool kBehind>
static cudaError_t launch_rows_vec(const RowParams &p, long long t0, long long n, int log_parts, size_t smem,
                                   cudaStream_t s) {
  auto k = dvp_row_kernel<TIn, TGrad, kBlk, kGrad, kTogether, kBehind>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  const int log_cluster = log_parts + (kTogether ? 1 : 0);
  cfg.gridDim = dim3((unsigned)(n << log_cluster), 1, 1);
  cfg.blockDim = dim3(kBlk, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  cfg.numAttrs = 0;
  if (log_cluster > 3) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  if (log_cluster > 0) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = 1u << log_cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  // may begin while the first launch ends; not where the gradient overwrites inference rows
  if ((p.order == kOrderSecond || p.order == kOrderApart) && !grad_over<TIn, TGrad>(p, p.infer, p.ld_infer)) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  return cudaLaunchKernelEx(&cfg, k, p, t0, log_parts);
}

template <typename TIn, typename TGrad, Grad kGrad, bool kTogether, bool kBehind = false>
static cudaError_t launch_rows_blk(const RowParams &p, long long t0, long long n, int log_parts, int threads,
                                   size_t smem, cudaStream_t s) {
  switch (threads) {
    case 64:
      if constexpr (kTogether) return cudaErrorInvalidValue;  // not made: launch_rows_both does not ask for it
      return launch_rows_vec<TIn, TGrad, 64, kGrad, false, kBehind>(p, t0, n, log_parts, smem, s);
    case 128: return launch_rows_vec<TIn, TGrad, 128, kGrad, kTogether, kBehind>(p, t0, n, log_parts, smem, s);
    case 256: return launch_rows_vec<TIn, TGrad, 256, kGrad, kTogether, kBehind>(p, t0, n, log_parts, smem, s);
    default: return launch_rows_vec<TIn, TGrad, 512, kGrad, kTogether, kBehind>(p, t0, n, log_parts, smem, s);
  }
}

// Does the gradient lie in the place of the inference rows, row for row?  (Not in other places of theirs.)
template <typename TIn, typename TGrad>
static inline bool grad_over_its_infer_row(const RowParams &p) {
  return p.grad == p.infer && sizeof(TGrad) == sizeof(TIn) && (p.T == 1 || p.ld_grad == p.ld_infer);
}

// Both policies' rows, in one launch, two or three; the second may begin while the first ends.
//
// One launch for calls that fill half of the chip at most, bound by the chain of their phases and by what a launch costs on
// the host.  Most of them go to dvp_rows_held.cuh; left are 257 to 296 short rows without a gradient, and rows that are too
// long for registers.  Device us, two launches / one (a graph of 20 calls): forward 280 x 3,000 bfloat16 6.0 / 5.2, 296 x 3,001
// 6.3 / 5.5, 296 x 1,500 float32 6.0 / 5.3, 260 x 2,048 float16 5.2 / 5.2; with the gradient 4 x 400,000 bfloat16 15.0 / 13.5.  Long
// rows near the line, clusters of 16 blocks, lose by it: 18 x 330,001 bfloat16 20.9 / 21.8 with the gradient, 16.1 / 16.0
// without, 9 x 170,001 float32 13.9 / 16.3 and 11.5 / 12.3, 4 x 262,144 float32 13.6 / 13.9 and 11.5 / 11.0.  Above the line
// clusters wait for free places: forward 400 x 3,000 bfloat16 6.5 / 6.8, 560 x 3,000 7.3 / 7.9, 24 x 330,001 19.0 / 20.2; with the
// gradient 19 x 330,001 19.2 / 20.5, 24 x 330,001 22.8 / 27.1, 12 x 170,001 float32 15.3 / 16.9, 18 x 170,001 19.8 / 26.0.
// Otherwise the rows with a gradient come first: the chip's last wave then has the short rows.  While all rows fit the chip
// at once the inference rows wait for the training rows at their end; in larger batches they would hold their places
// idle, so that neither launch waits for the other and a third one forms the log-ratios and flags (the inference rows'
// membership passes through log_ratio).  us, with the gradient, inference rows first / now: V = 151,936 bfloat16, T = 256
// 72 / 64, 512 122 / 112, 800 177 / 157, 2,048 379 / 358, 4,096 707 / 684; 1,000 x 65,536 99 / 89; float32 1,000 x 50,021
// 129 / 122, 2,000 x 100,000 428 / 418.  (Waiting in larger batches: T = 800 187, 2,048 388.)  The third launch costs some
// 4 us, the last wave of 32,768 bfloat16 rows 40 (5,537 / 5,513); that of float32 rows, which are bound by their bytes
// alone, less than that from some 16 waves on (4,096 x 262,144, 28 waves: 1,892 / 1,897).
// The inference rows come first where the training rows need them, for weights, where the gradient takes their place, and
// without a gradient; and in larger batches where a third launch does not pay or an output that it needs is missing.
//
// Between a first and a second launch ln pi^mp(a) passes through the output that holds it, or through one that the second
// launch writes later: log_ratio, weight_out, or the start of the gradient row (with a single 2-byte gradient element
// there is no room: V = 1, where ln pi^mp(a) is 0).
template <typename TIn, typename TGrad>
static cudaError_t launch_rows_both(const RowParams &p_in, bool loose, int log_parts, int threads, size_t smem,
                                    cudaStream_t s) {
  const bool weighted = p_in.weight_kind != DVP_WEIGHT_NONE;
  const bool over_infer = grad_over<TIn, TGrad>(p_in, p_in.infer, p_in.ld_infer);
  const bool resident = (p_in.T << (log_parts + 1)) * threads <= 148 * 1024;
  auto launch = [&](const RowParams &p, long long t0, long long n, auto together) {
    constexpr bool kTogether = decltype(together)::value;
    return !p.grad ? launch_rows_blk<TIn, TIn, Grad::kNone, kTogether>(p, t0, n, log_parts, threads, smem, s)
           : loose ? launch_rows_blk<TIn, TGrad, Grad::kLoose, kTogether>(p, t0, n, log_parts, threads, smem, s)
                   : launch_rows_blk<TIn, TGrad, Grad::kGranules, kTogether>(p, t0, n, log_parts, threads, smem, s);
  };
  if (p_in.infer && threads > 64 && (p_in.T << (log_parts + 1)) * threads <= 74 * 1024 &&  // 64: less than 128 granules
      (!over_infer || (grad_over_its_infer_row<TIn, TGrad>(p_in) && !p_in.out_i.mask))) {  // masks are written last
    RowParams p = p_in;
    const cudaError_t e = launch(p, 0, p.T, std::true_type{});
    // a cluster of 16 blocks is more than every device (or part of one) takes: two launches then
    if (log_parts < 3 || (e != cudaErrorInvalidClusterSize && e != cudaErrorLaunchOutOfResources)) return e;
    (void)cudaGetLastError();
  }
  const long long per_launch = 0x7fffffffLL >> log_parts;  // a grid holds this many rows
  const bool pays = sizeof(TIn) == 2 || (p_in.T << (log_parts + 1)) * threads <= 16 * 148 * 1024LL;
  const bool train_first = p_in.infer && p_in.grad && !weighted && !over_infer &&
                           (resident || (pays && p_in.log_ratio && p_in.out_t.logp_mp && p_in.out_i.logp_mp));
  for (long long t0 = 0; t0 < p_in.T; t0 += per_launch) {
    const long long n = p_in.T - t0 < per_launch ? p_in.T - t0 : per_launch;
    RowParams p = p_in, q = p_in;  // the training rows' launch, the inference rows'
    p.side = kSideTrain;
    q.side = kSideInfer;
    q.train = p_in.infer;
    q.ld_train = p_in.ld_infer;
    q.out_t = p_in.out_i;
    q.infer = nullptr;
    q.grad = nullptr;
    q.weight_kind = DVP_WEIGHT_NONE;
    RowParams &first = train_first ? p : q, &second = train_first ? q : p;
    cudaError_t e = cudaSuccess;
    if (p_in.infer) {
      first.order = kOrderFirst;
      first.log_ratio = nullptr;
      second.order = train_first && !resident ? kOrderApart : kOrderSecond;
      if (second.order == kOrderApart) {
        second.flags = nullptr;
      } else {
        char *place = reinterpret_cast<char *>(first.out_t.logp_mp ? first.out_t.logp_mp
                                               : p_in.log_ratio    ? p_in.log_ratio
                                                                   : p_in.weight_out);
        p.li_stride = q.li_stride = sizeof(float);
        if (!place && weighted && p_in.V * sizeof(TGrad) >= sizeof(float)) {
          place = reinterpret_cast<char *>(p_in.grad);
          p.li_stride = q.li_stride = p_in.ld_grad * (long long)sizeof(TGrad);
        }
        p.li = q.li = place;
      }
      e = launch(first, t0, n, std::false_type{});
    }
    if (e == cudaSuccess)
      e = train_first ? launch_rows_blk<TIn, TIn, Grad::kNone, false, true>(q, t0, n, log_parts, threads, smem, s)
                      : launch(p, t0, n, std::false_type{});
    if (e == cudaSuccess && second.order == kOrderApart) e = launch_ratio_kernel(p_in, t0, n, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Shared memory one SM can give to `blocks` resident blocks (228 KB per SM, 1 KB of it
// reserved per block), and the most one block may ask for.
static inline size_t smem_per_block(int blocks) {
  const size_t share = (size_t)228 * 1024 / blocks - 1024;
  return share < (size_t)227 * 1024 ? share : (size_t)227 * 1024;
}

// The kernel that keeps the candidates of the safe set on chip (2-byte logits).
template <typename TIn, typename TGrad, int kThreads, int kBlocks, bool kWeighted>
static cudaError_t launch_rows_cs(const RowParams &p, int threads, int n_steps, cudaStream_t s) {
  auto k = cs::dvp_row_kernel_cs<TIn, TGrad, kThreads, kBlocks, kWeighted>;
  if (n_steps > 64) return cudaErrorNotSupported;  // positions are 16 bits
  // as many list entries per warp as the SM's shared memory allows with kBlocks blocks
  // resident, at most every element the warp sees
  const size_t fixed = cs::smem_bytes_cs(threads, 0);
  const size_t budget = smem_per_block(kBlocks * (kThreads / threads));
  const int nwarp = threads / 32;
  long long cap = budget > fixed ? (long long)((budget - fixed) / (4 * (size_t)nwarp)) : 0;
  const long long most = (long long)n_steps * 64 * Granule<TIn>::kElems;
  if (cap > most) cap = most;
  if (cap < 32 * Granule<TIn>::kElems) return cudaErrorNotSupported;
  const size_t smem = cs::smem_bytes_cs(threads, (int)cap);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  k<<<(unsigned)p.T, threads, smem, s>>>(p, n_steps, (int)cap);
  return cudaGetLastError();
}

// Threads of a block and blocks of a row, from the number of rows (both policies') and their length in
// granules.  An SM holds 1,024 threads of the row kernel.
//
// A thread should have about 16 granules: each row costs it some 860 instructions beside the 250 of two
// granules.  Measured, us, with the gradient, for 64 / 128 / 256 / 512 threads: 20,000 x 4,000 float32
// 222 / 266 / 404 / 404; 4,000 x 8,001 float32 91 / 99 / 118 / 185; 8,000 x 20,000 bfloat16 226 at 128 against
// 230 at 64 and 288 at 256; 2,000 x 32,000 float32 173 / 155 / 155 / 175.  Not above `most`, where rows of any
// length run best: 256 for 2-byte logits (V = 151,936: 909 against 1207 at 128), 512 for float32 (V = 262,144:
// 1904 against 2180 at 256).
//
// While all rows fit the chip at once, more threads a row are faster (100 x 20,000 bfloat16: 17.5 at 256
// against 21.5 at 128 and 29.7 at 64); so they are while the rows that come first do, and a thread has four granules (300 x
// 32,000 bfloat16 with the gradient 26.7 -> 22.6; 1,000 x 20,000, which do not fit, 37.1 / 43.2), 2-byte rows up to a few
// more than fit (593 to 608 bfloat16 rows, 128 threads / 256: V = 16,640 29.5 / 27.5 to 30.4 / 29.2, 20,000 31.2 / 30.0 to
// 31.5 / 31.1, 26,000 38.7 / 34.8 to 38.4 / 34.8, 32,000 45.2 / 36.9 to 46.8 / 38.0; 1,185 to 1,216 rows, 64 / 128: V = 8,320
// 32.3 / 27.7, 10,000 33.5 / 30.7, 13,000 41.6 / 35.6, 16,000 47.7 / 36.5; 300 x 27,652 float32 28.3 / 28.9.  The two do not
// meet there yet: 640 rows of 20,000 32.5 / 32.3, of 32,000 47.6 / 39.8).
//
// Then more blocks a row, V = 151,936 bfloat16, 1 / 2 / 4 / 8 blocks: T = 16 forward 36 / 28 / 21 / 19; T = 128 with the
// gradient 57 / 47 / 41.  Blocks that share a row need at least a step and a half of it each (V = 20,000: 13 / 15), without
// a gradient two and a half where they fill more than half of the chip (100 x 32,000 12.4 / 14.1).
//
// With the gradient they pay also beyond the chip, the further the longer a thread's part of a row is, because the last
// wave is shorter.  us, 1 block / 2, at about 2, 3.5, 4.7 and 6.9 times the chip: 64 granules a thread (V = 262,144) 101 / 74,
// 203 / 180, 264 / 237, 358 / 331; 37 (V = 151,936) 64 / 50, 117 / 113, 146 / 146, 198 / 200; 24 (V = 100,000 float32) 57 / 55, 80 / 79,
// 114 / 126; with weights 37 granules 171 / 164 at 4.7, 24 91 / 86 at 3.5; 12 (V = 50,021) 29 / 31 at 1.4.  2 blocks / 4 at 2, 2.7
// and 4: 64 granules 74 / 68, 90 / 81, 113 / 111; 37 50 / 49, 56 / 58, 75 / 81; 24 28 / 30 at 1.7.
// Without a gradient only very long rows gain by it: V = 262,144 140 / 130 and 196 / 169 at 3.5 and 4.7 times the chip;
// V = 151,936 65 / 81 and 77 / 88 at 2.7 and 3.5, V = 100,000 float32 44 / 55 at 2.7.
struct RowShape {
  int threads, log_parts;
};
// `first`: the rows, of `rows`, that are swept first (with weights taken like without, so that their statistics are the same).
static inline RowShape choose_shape(long long rows, long long first, long long n_gran, int most, bool grad) {
  const long long chip = 148 * 1024, nearly = most == 256 ? 152 * 1024 : chip;  // 256: 2-byte rows
  RowShape s = {64, 0};
  while (s.threads < most && 16LL * s.threads < n_gran) s.threads *= 2;
  while (s.threads < most && 2 * rows * s.threads <= chip && n_gran >= 2 * s.threads) s.threads *= 2;
  while (s.threads < most && 2 * first * s.threads <= nearly && n_gran >= 8 * s.threads) s.threads *= 2;
  while (s.log_parts < 3) {
    const int lp = s.log_parts + 1;
    const long long per = n_gran >> lp, total = (rows << lp) * s.threads, steps = n_gran / s.threads;
    const long long least = grad || 2 * total <= chip ? 3 : 5;
    // total / chip: at most steps / 6, but 8 (2 blocks), or steps / 16 (4); steps / 12 or / 24 without a gradient
    const long long scale = grad ? (lp == 1 ? 6 : 16) : 6 << lp;
    const bool beyond =
        lp < 3 && steps >= (grad ? 20 : 48) && total * scale <= steps * chip && total <= 8 * chip;
    if (per < least * s.threads || !(total <= chip || beyond)) break;
    s.log_parts = lp;
  }
  return s;
}

template <typename TIn, typename TGrad>
static cudaError_t launch_rows(const RowParams &p, uint32_t hint, cudaStream_t s) {
  constexpr int kElems = Granule<TIn>::kElems;
  int threads = hint & 0xffff, stage = (hint >> 16) & 0xff, cluster = (hint >> 24) & 0xff;
  const int stage_hint = stage;
  // stage byte 0x11: the kernel that keeps the row in shared memory; 0x1e: the same with
  // block 0's first copy withheld (self-test of the wait limit)
  if (stage == 0x11 || stage == 0x1e) {
    const bool ok16 = aligned32(p.train, p.ld_train, sizeof(TIn)) &&
                      aligned32(p.infer, p.ld_infer, sizeof(TIn)) &&
                      aligned32(p.grad, p.ld_grad, sizeof(TGrad));
    const cudaError_t e =
        ok16 ? res::launch_resident<TIn, TGrad>(p, s, stage == 0x1e) : cudaErrorNotSupported;
    if (e != cudaErrorNotSupported) return e;
    cluster = 0;  // rows it cannot take: the streaming kernel below
  }
  stage = 2;  // two granules per thread and pipeline stage
  const bool vec_ok = aligned32(p.train, p.ld_train, sizeof(TIn)) &&
                      aligned32(p.infer, p.ld_infer, sizeof(TIn)) &&
                      aligned32(p.grad, p.ld_grad, sizeof(TGrad));
  const bool loose = p.grad && grad_loose<TIn, TGrad>(p.train, p.ld_train, p.grad, p.ld_grad, p.T);
  const long long n_gran_row = (p.V + kElems - 1) / kElems;
  const bool weighted = p.weight_kind != DVP_WEIGHT_NONE;
  const bool store_kernel = sizeof(TIn) == 2 && (stage_hint == 3 || stage_hint == 4);
  int log_parts = 0;
  if (threads == 0 && cluster == 0 && !store_kernel) {
    const bool over_infer = grad_over<TIn, TGrad>(p, p.infer, p.ld_infer);
    held::Shape sh;
    if (held::shape_of(p.T, p.infer != nullptr, p.grad != nullptr, n_gran_row, &sh) &&
        (!over_infer || (grad_over_its_infer_row<TIn, TGrad>(p) && !p.out_i.mask))) {  // masks are written last
      const cudaError_t e = !p.grad ? held::launch<TIn, TIn, Grad::kNone>(p, sh, s)
                            : loose ? held::launch<TIn, TGrad, Grad::kLoose>(p, sh, s)
                                    : held::launch<TIn, TGrad, Grad::kGranules>(p, sh, s);
      // a cluster of 16 blocks is more than every device (or part of one) takes
      if (sh.log_parts < 3 || (e != cudaErrorInvalidClusterSize && e != cudaErrorLaunchOutOfResources)) return e;
      (void)cudaGetLastError();
    }
  }
  if (threads == 0 && cluster == 0 && !store_kernel) {
    const RowShape sh = choose_shape(p.T * (p.infer ? 2 : 1), p.T * (p.infer && !p.grad ? 2 : 1), n_gran_row,
                                     sizeof(TIn) == 4 ? 512 : 256, p.grad != nullptr);
    threads = sh.threads;
    log_parts = sh.log_parts;
  } else {
    if (threads == 0) threads = sizeof(TIn) == 4 ? 512 : 256;
    log_parts = cluster == 8 ? 3 : cluster == 4 ? 2 : cluster == 2 ? 1 : 0;
    while (log_parts > 0 && (n_gran_row >> log_parts) < 256) --log_parts;
    int pow2 = 64;  // the largest of 64, 128, 256 and 512 threads that is not above the choice
    while (2 * pow2 <= threads) pow2 *= 2;
    threads = pow2;
    while (threads > 64 && threads >= n_gran_row >> log_parts) threads /= 2;
  }
  const int parts = 1 << log_parts;
  const long long n_gran = (n_gran_row + parts - 1) / parts;  // granules per block
  const long long per = (long long)stage * threads;
  const size_t smem = (size_t)smem_words_fixed(threads) * 4 +
                      (size_t)((n_gran + per - 1) / per) * threads * 4;
  // 16-bit hot-list entries hold slot * 32 + lane: very long rows swept by few threads
  // would not fit them
  const bool hot_ok = ((n_gran + per - 1) / per) * stage * 32 <= 65536;
  if constexpr (sizeof(TIn) == 2) {
    // stage byte 3 or 4: the kernel that keeps the candidates of the safe set on chip, with
    // three or four resident blocks per SM (measured slower than the kernel below; kept for
    // comparison)
    if (store_kernel && vec_ok && parts == 1 && threads <= 256) {
      const int n_steps = (int)((n_gran + per - 1) / per);
      cudaError_t e;
      if (weighted)
        e = launch_rows_cs<TIn, TGrad, 256, 3, true>(p, threads, n_steps, s);
      else if (stage_hint == 3)
        e = launch_rows_cs<TIn, TGrad, 256, 3, false>(p, threads, n_steps, s);
      else
        e = launch_rows_cs<TIn, TGrad, 256, 4, false>(p, threads, n_steps, s);
      if (e != cudaErrorNotSupported) return e;
    }
  }
  // Weights with no output to pass ln pi^mp_infer(a) through (launch_rows_both) and a gradient in place of logits that
  // it would be written over: both rows of a token in one block.
  const bool no_place = weighted && !p.out_i.logp_mp && !p.log_ratio && !p.weight_out &&
                        (grad_over<TIn, TGrad>(p, p.train, p.ld_train) || grad_over<TIn, TGrad>(p, p.infer, p.ld_infer));
  if (hot_ok && smem <= 200 * 1024 && !no_place) {
    return launch_rows_both<TIn, TGrad>(p, loose, log_parts, threads, smem, s);
  }
  dvp_row_kernel_scalar<TIn, TGrad><<<(unsigned)p.T, 512, 0, s>>>(p);
  return cudaGetLastError();
}

template <typename TIn>
static cudaError_t launch_rows_g(const RowParams &p, int grad_dtype, uint32_t hint, cudaStream_t s) {
  switch (grad_dtype) {
    case DVP_F32: return launch_rows<TIn, float>(p, hint, s);
    case DVP_BF16: return launch_rows<TIn, __nv_bfloat16>(p, hint, s);
    default: return launch_rows<TIn, __half>(p, hint, s);
  }
}

// Threads: up to eight granules each (64 / 128 / 256 threads, us: 20,000 x 4,001 bfloat16 57 / 68 / 98, 10,000 x 2,500 with
// float32 entries 30 / 35 / 47, 3,130 x 7,488 float16 15.3 / 17.8 / 18.6, 10,400 x 21,440 bfloat16 144 / 140 / 140).  Blocks of a row:
// as many as bring some 16 warps to every SM (four times its 1,024 threads' worth of rows are enough), while each has a
// step or more.
template <typename TIn, typename TGrad>
static cudaError_t launch_bwd(const BackwardParams &p, uint32_t hint, cudaStream_t s) {
  const long long n_gran = p.V / Granule<TIn>::kElems;
  int threads = hint & 0xffff, log_parts = 0;
  if (threads == 0) {
    threads = 64;
    while (threads < 256 && n_gran > 8 * threads) threads *= 2;
  }
  while (log_parts < 10 && (p.T << log_parts) * threads < 4 * 148 * 1024 && n_gran >> (log_parts + 1) >= 2 * threads)
    ++log_parts;
  const bool loose = grad_loose<TIn, TGrad>(p.train, p.ld_train, p.grad, p.ld_grad, p.T);
  const unsigned grid = (unsigned)(p.T << log_parts);
  if (loose)
    dvp_backward_kernel<TIn, TGrad, true><<<grid, threads, threads / 32 * kShiftWords * 4, s>>>(p, log_parts);
  else
    dvp_backward_kernel<TIn, TGrad, false><<<grid, threads, 0, s>>>(p, log_parts);
  return cudaGetLastError();
}

template <typename TIn>
static cudaError_t launch_bwd_g(const BackwardParams &p, int grad_dtype, uint32_t hint,
                                cudaStream_t s) {
  switch (grad_dtype) {
    case DVP_F32: return launch_bwd<TIn, float>(p, hint, s);
    case DVP_BF16: return launch_bwd<TIn, __nv_bfloat16>(p, hint, s);
    default: return launch_bwd<TIn, __half>(p, hint, s);
  }
}

}  // namespace dvp
